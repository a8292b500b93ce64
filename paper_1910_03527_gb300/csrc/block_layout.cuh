#pragma once
// Shared memory and workspace of the block solver: where the arrays of one tuple lie, for every
// form of sigma.  Host and device; casci_block.cu has the kernels.
#include "casci_dev.cuh"
#include "digits.cuh"

namespace mbe {

constexpr int BLOCK_THREADS = 512;  // one block per SM: 128 registers a thread, up to 227 KB
constexpr int GEMM_MAX_N = 9;       // orbitals up to which sigma is the tiled product
constexpr int GEMM_T_BYTES = 48 * 1024;
constexpr int LIST_STAGE = 16 * 1024;  // bytes of Hs staged by SIGMA_LIST
constexpr int LIST_MAX_NS = 128;    // strings up to which larger orbital counts keep c in shared memory

// Forms of sigma: c in global memory and both lists walked per element; the tiled product; c and
// V in shared memory and the off-diagonal lists walked (10-16 orbitals with few strings).
enum { SIGMA_GLOBAL = 0, SIGMA_TILED = 1, SIGMA_LIST = 2 };
__host__ __device__ inline int sigma_form(int n, int ns)
{
    return n <= GEMM_MAX_N ? SIGMA_TILED : ns <= LIST_MAX_NS ? SIGMA_LIST : SIGMA_GLOBAL;
}

// Row stride of the float32 V of a form, the only one that its readers and writers use: pairs
// padded to 6 for the tiles, to an odd number for gathers by rows.
__host__ __device__ inline int v32_stride(int form, int P)
{
    return form == SIGMA_TILED ? (P + 5) / 6 * 6 : form == SIGMA_LIST ? P | 1 : P;
}

// Per-block slot of the workspace.
struct BlockSlot {
    size_t off_V, off_W, off_x, off_t, off_diag, off_Hs64, off_Hs32, off_x2, off_x0, off_full, off_V64, off_U, vec, bytes;
};

__host__ __device__ inline int hs_stride(int ns) { return (ns + 3) / 4 * 4; }

__host__ __device__ inline BlockSlot block_slot(int n, int ns)
{
    BlockSlot L;
    size_t o = 0;
    const size_t vec = ((size_t)ns * (ns + 1) / 2 * 8 + 255) & ~(size_t)255;
    const size_t mat = ((size_t)ns * hs_stride(ns) * 8 + 255) & ~(size_t)255;
    L.vec = vec;
    L.off_V = o; o += vec * MMAX;
    L.off_W = o; o += vec * MMAX;
    L.off_x = o; o += vec;
    L.off_t = o; o += vec;
    L.off_diag = o; o += vec;
    L.off_x2 = o; o += vec;
    L.off_x0 = o; o += vec;
    L.off_Hs64 = o; o += mat;
    L.off_Hs32 = o; o += mat / 2;
    L.off_full = o; o += mat;  // the product C Hs, or the whole coefficient matrix
    // SIGMA_LIST: the float64 V, and sums of V over each string's orbitals
    const size_t P = (size_t)n * (n + 1) / 2, list = sigma_form(n, ns) == SIGMA_LIST ? 1 : 0;
    L.off_V64 = o; o += list * ((P * P * 8 + 255) & ~(size_t)255);
    L.off_U = o; o += list * ((ns * P * 4 + 255) & ~(size_t)255);
    L.bytes = o;
    return L;
}

// Shapes of the tiled sigma of one string class.
struct GemmShape {
    int cst;        // row stride of T and of the fixed-point c (strings, padded to 4)
    int fst;        // row stride of the float32 c (not a multiple of 32: its columns are written too)
    int pst;        // row stride of the float32 V (v32_stride)
    int rs;         // row stride of the lists
    int nj, np, tiles;  // string and pair groups, tiles per alpha string
    int g;          // alpha strings per stage
};

template <typename T>
__host__ __device__ inline GemmShape gemm_shape(int n, int ns, int r)
{
    GemmShape s;
    const int P = n * (n + 1) / 2, tp = sizeof(T) == 8 ? 3 : 6, tj = sizeof(T) == 8 ? 4 : 8;
    s.cst = hs_stride(ns);
    s.fst = s.cst % 32 == 0 ? s.cst + 4 : s.cst;
    if (s.fst % 8) s.fst += 4;  // (whole tiles of 8)
    if (s.fst % 32 == 0) s.fst += 8;
    s.pst = v32_stride(SIGMA_TILED, P);
    s.rs = r | 1;
    s.np = (P + tp - 1) / tp;
    s.nj = (s.cst + tj - 1) / tj;
    s.tiles = s.np * s.nj;
    s.g = BLOCK_THREADS / s.tiles;
    const int fit = (n < GEMM_MAX_N ? 2 : 1) * GEMM_T_BYTES / (P * s.cst * (int)sizeof(T));
    if (s.g > fit) s.g = fit;
    if (s.g > ns) s.g = ns;
    if (s.g > 1) s.g &= ~1;  // (strings are taken in pairs)
    if (s.g < 1) s.g = 1;
    return s;
}

// Float64 operands of the tiled sigma as digits (sigma_digits), from off_c on.
constexpr int DIGITS_SMEM = 226 * 1024;  // used where all of the block's shared memory fits in this
struct DigitShape {
    int c8, cs, vs, mt;  // tiles of 8 strings; row strides (16-bit words) of c and V; tiles of 16 pairs
    int g;               // strings per round: as many as the float32 T has room for
    int off_v, off_l, off_rows, bytes;
};

__host__ __device__ inline DigitShape digit_shape(int n, int ns, int r)
{
    DigitShape d;
    const int P = n * (n + 1) / 2;
    const GemmShape a = gemm_shape<float>(n, ns, r), b = gemm_shape<double>(n, ns, r);
    d.g = a.g / 2 > b.g ? a.g / 2 : b.g;
    if (d.g > 1) d.g &= ~1;
    d.c8 = (ns + 7) / 8;
    d.cs = 8 * (d.c8 | 1);  // (odd multiples of 16 bytes: the 8 rows of a matrix in different banks)
    d.mt = (P + 15) / 16;
    d.vs = d.mt * 16 + 8;
    d.off_v = 2 * DIGITS * (ns + 1) * d.cs;  // (row ns of c is zero)
    d.off_l = d.off_v + 2 * DIGITS * P * d.vs;
    d.off_rows = al16(d.off_l + 2 * ns * ((r + 15) / 16 * 16));
    d.bytes = d.off_rows + 8 * d.g * (d.cs + d.mt * 16);
    return d;
}

// Row stride of the float32 c of SIGMA_LIST
__host__ __device__ inline int list_stride(int ns)
{
    const int s = (ns + 7) / 8 * 8;  // (whole tiles of the same-spin product)
    return s % 32 == 0 ? s + 8 : s;
}

struct BlockMem {  // dynamic shared memory
    int off_A, off_pp, off_h, off_V64, off_V32, off_red, off_G, off_J, off_ev, off_y, off_yp, off_r, off_misc,
        off_hd, off_list, off_c, off_T, off_g1, bytes, digits;
};

// The tiled sigma's lists, c and T; the lists and c of SIGMA_LIST; else those are absent.
// rdm: density matrices follow the solve.
__host__ __device__ inline BlockMem block_mem(int n, int form, int ns, int r, int rdm, int digits = 1)
{
    BlockMem S;
    S.digits = form == SIGMA_TILED ? digits : 0;
    const int P = n * (n + 1) / 2;
    const bool gemm = form == SIGMA_TILED;
    int o = 0;
    S.off_A = o; o = al16(o + 4 * MBE_MAX_STRING_ORB);
    S.off_pp = o; o = al16(o + 4 * P);
    S.off_h = o; o = al16(o + 8 * n * n);
    S.off_V64 = o; o = al16(o + (form == SIGMA_LIST ? 0 : 8 * P * P));  // (SIGMA_LIST: in the slot)
    S.off_V32 = o; o = al16(o + 4 * P * v32_stride(form, P));
    S.off_red = o; o = al16(o + 8 * 32 * KRED);
    S.off_G = o; o = al16(o + 8 * MMAX * MMAX);
    S.off_J = o; o = al16(o + 4 * 4 * MMAX * MMAX);
    S.off_ev = o; o = al16(o + 4 * MMAX);
    S.off_y = o; o = al16(o + 8 * MMAX);
    S.off_yp = o; o = al16(o + 8 * MMAX);
    S.off_r = o; o = al16(o + 8 * MMAX);
    S.off_misc = o; o = al16(o + 8 * 4);
    S.off_g1 = o; o = al16(o + 8 * n * n);
    S.off_hd = o; o = al16(o + (gemm ? 8 * ns : 0));
    S.off_list = o; o = al16(o + (gemm ? 2 * ns * (r | 1) : form == SIGMA_LIST ? 4 * ns * (r + 1) : 0));
    S.off_c = o;
    if (form == SIGMA_LIST) o = al16(o + 4 * ns * list_stride(ns));
    const int stage = form == SIGMA_LIST ? LIST_STAGE : 0;
    if (gemm) {
        // fixed point: c; float32: c, V twice over with both signs, list offsets (see sigma_gemm)
        const GemmShape a = gemm_shape<float>(n, ns, r);
        const int f = al16(4 * ns * a.fst) + 8 * P * a.pst + 4 * ns * r;
        const int c = S.digits ? digit_shape(n, ns, r).bytes : 8 * ns * a.cst;
        o = al16(o + (f > c ? f : c));
    }
    S.off_T = o;
    if (gemm) {
        const GemmShape a = gemm_shape<float>(n, ns, r), b = gemm_shape<double>(n, ns, r);
        const int ta = a.g * P * a.cst * 4, tb = b.g * P * b.cst * 8;
        const int th = S.digits ? 2 * DIGITS * 16 * digit_shape(n, ns, r).cs : 0;  // (16 rows of Hs)
        o = al16(o + (ta > tb ? ta > th ? ta : th : tb > th ? tb : th));
    }
    o = al16(o + stage);
    // the density matrices' vectors lie over c and T
    const int d = rdm ? S.off_c + 8 * 33 * (n * n + 1) : 0;
    S.bytes = al16(o > d ? o : d);
    return S.digits && S.bytes > DIGITS_SMEM ? block_mem(n, form, ns, r, rdm, 0) : S;
}

}  // namespace mbe
