"""The block solver's shared-memory layout: every array ends at or before the next one, for every
string class and form of sigma.  Host arithmetic (block_layout.cuh compiled on its own)."""

import math
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GLOBAL, TILED, LIST = 0, 1, 2

PROGRAM = """
#include "block_layout.cuh"
#include <cstdio>
using namespace mbe;
int main()
{
    int n, k, ns, r, form, rdm;
    while (scanf("%d %d %d %d %d %d", &n, &k, &ns, &r, &form, &rdm) == 6) {
        if (form < 0) form = sigma_form(n, ns);
        const BlockMem S = block_mem(n, form, ns, r, rdm);
        const GemmShape f = gemm_shape<float>(n, ns, r), d = gemm_shape<double>(n, ns, r);
        const DigitShape g = digit_shape(n, ns, r);
        printf("%d %d %d %d %d %d %d %d %d %d %d %d %d %d %d %d %d %d %d %d", form, v32_stride(form, n * (n + 1) / 2), S.off_V32,
               S.off_red, S.off_hd, S.off_list, S.off_c, S.off_T, S.bytes, S.digits, list_stride(ns), f.fst, f.pst, f.cst, f.g,
               d.g, g.bytes, g.cs, LIST_STAGE, DIGITS);
        printf(" %d %d %d %d\\n", S.off_h, S.off_V64, S.off_G, S.off_g1);
    }
}
"""
FIELDS = ("form v32 off_V32 off_red off_hd off_list off_c off_T bytes digits list_stride fst pst cst gf gd digit_bytes "
          "digit_cs stage DIGITS off_h off_V64 off_G off_g1").split()


@pytest.fixture(scope="module")
def layouts(tmp_path_factory):
    from paper_1910_03527_gb300 import _build
    d = tmp_path_factory.mktemp("layout")
    src, exe = d / "layout.cu", d / "layout"
    src.write_text(PROGRAM)
    subprocess.run([_build.nvcc(), *_build.ARCH, "-std=c++17", "-O0", "-I" + _build.INCLUDE, "-I" + _build.CSRC, str(src),
                    "-o", str(exe)], check=True, capture_output=True)
    cases = [(n, k, math.comb(n, k), k * (n - k + 1), form, rdm)
             for n in range(2, 17) for k in range(1, n) for form in (-1, GLOBAL) for rdm in (0, 1)]
    out = subprocess.run([str(exe)], input="\n".join(" ".join(map(str, c)) for c in cases), capture_output=True, text=True,
                         check=True).stdout.split("\n")
    return [(c, dict(zip(FIELDS, map(int, line.split())))) for c, line in zip(cases, out)]


def test_every_array_ends_before_the_next(layouts):
    assert len(layouts) == 480 and {s["form"] for _, s in layouts} == {GLOBAL, TILED, LIST}
    for (n, k, ns, r, _, rdm), s in layouts:
        P, where, form = n * (n + 1) // 2, (n, k, s["form"], rdm), s["form"]
        assert s["off_h"] + 8 * n * n <= s["off_V64"], where
        assert s["off_V64"] + (0 if form == LIST else 8 * P * P) <= s["off_V32"], where
        assert s["v32"] >= P and s["off_V32"] + 4 * P * s["v32"] <= s["off_red"], where
        assert s["off_red"] + 8 * 32 * 24 <= s["off_G"], where
        assert s["off_g1"] + 8 * n * n <= s["off_hd"], where
        if form == LIST:
            assert s["off_list"] + 4 * ns * (k * (n - k) + 1) <= s["off_c"], where
            assert s["off_c"] + 4 * ns * s["list_stride"] <= s["off_T"] and s["list_stride"] >= ns, where
            assert s["off_T"] + s["stage"] <= s["bytes"], where
        if form == TILED:
            assert s["pst"] == s["v32"] and s["off_hd"] + 8 * ns <= s["off_list"], where
            assert s["off_list"] + 2 * ns * (r | 1) <= s["off_c"], where
            c32 = (4 * ns * s["fst"] + 15) // 16 * 16 + 8 * P * s["pst"] + 4 * ns * r
            c64 = s["digit_bytes"] if s["digits"] else 8 * ns * s["cst"]
            assert s["off_c"] + max(c32, c64) <= s["off_T"], where
            hs = 2 * s["DIGITS"] * 16 * s["digit_cs"] if s["digits"] else 0
            assert s["off_T"] + max(4 * s["gf"] * P * s["cst"], 8 * s["gd"] * P * s["cst"], hs) <= s["bytes"], where
        if rdm and n <= 10:
            assert s["off_c"] + 8 * 33 * (n * n + 1) <= s["bytes"], where
