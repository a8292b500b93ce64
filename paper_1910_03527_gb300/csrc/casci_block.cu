// a2-a7, the block solver: one tuple CASCI beyond the warp solvers per thread block.
//
// The Davidson's vectors lie in one spin-flip sector and are kept as their Ns (Ns + 1) / 2
// elements with Ia <= Ib (orthonormal basis of the sector, as in casci_sector.cuh), in a
// per-block slot of the workspace: half of the memory traffic of the vector algebra, which
// with the sigma below is what bounds a tuple of 8 or 9 orbitals (46 vectors of up to 32 KB
// in float32 per block do not fit in L2 for all blocks).
//
// sigma up to 9 orbitals (at most 126 strings): the whole coefficient matrix c sits in shared
// memory, and per alpha string Ia the opposite-spin term is a dense product and a gather,
//     T[p][J] = sum_x s_x V[p_x][p] c[J_x][J],   sigma[Ia][Ib] = sum_y s_y T[p_y][J_y].
// The product is register-tiled in float32 (8 strings x 6 pairs per thread, see gemm_tile), where the
// double loop over both lists gathers three values for every multiply-add; it does 2 P / R = 3.6
// times more of them at 9 orbitals, but near the rate of the pipe.  In float64, where a
// multiply-add costs 74 float32 ones, the product is one of exact digits on the tensor cores
// (sigma_digits), or, where those do not fit in shared memory, of 55-bit fixed-point numbers in
// two limbs (three wide integer multiply-adds per term).  Cycles per phase of an iteration, before
// and after each step: the float32 product 595 -> 390 thousand at 9 orbitals, the float64 one
// 782 -> 317 thousand at 8.
// From 10 orbitals with at most 128 strings, c and V in shared memory and sorted lists (sigma_list);
// beyond, c does not fit, and sigma walks both lists per element.
#include "block_layout.cuh"
#include "casci_sector.cuh"
#include "digits.cuh"

namespace mbe {

// The block's dynamic shared memory.  Named by its symbol wherever it is read: through a pointer
// kept in a struct the compiler loses the address space, and the tiled product took twice as
// many instructions (generic loads with 64-bit addresses).
__device__ __forceinline__ char *block_shared()
{
    extern __shared__ __align__(16) char smem[];
    return smem;
}

struct BlockProblem {
    Problem pb;       // N: packed elements; diag: packed
    int form;         // of sigma
    const float *U;   // SIGMA_LIST: U[I][p] = sum over the orbitals q of string I of V[qq][p]
    bool bad;         // an element of V or Hs is not finite (float64 sigma: fixed point cannot hold it)
    int E;            // fixed-point exponent: 2^E is above the elements of V and (off-diagonal) Hs
    int Eh;           // the same with the diagonal of H: the unit of residuals (0 if H is zero)
    BlockMem S;
    double *full;     // [Ns][stride] scratch of the slot
};

__device__ __forceinline__ uint64_t dup2(float v)
{
    const uint64_t u = __float_as_uint(v);
    return u << 32 | u;
}

// The packed vector v as the whole matrix [Ns][ld] (elements with Ia != Ib scaled back).
template <typename T>
__device__ inline void expand_full(const Problem &pb, const T *v, T *full, int ld)
{
    int ia = 0, ib = 0;
    tri_advance(ia, ib, threadIdx.x, pb.Ns);
    for (int h = threadIdx.x; h < pb.N; h += blockDim.x) {
        const T c = ia == ib ? v[h] : (T)0.70710678118654752 * v[h];
        full[ia * ld + ib] = c;
        full[ib * ld + ia] = pb.sector > 0 ? c : -c;
        tri_advance(ia, ib, blockDim.x, pb.Ns);
    }
}

// M = C Hs for the float32 product: 8 x 4 tiles, c from shared memory by its rows (C[i][J] is
// sgn C[J][i]), Hs in chunks of rows through shared memory (buf: bytes of it that are free; Hs is
// larger than what is left of L1, and one row of it per step left the warps waiting for L2).
// Ends without a barrier.
__device__ inline void same_spin(const Problem &pb, int ld, int fst, const float *c, const float *Hs, float *M, char *buf,
                                 int bytes)
{
    const int nj = ld / 4, ni = (pb.Ns + 7) / 8, tid = threadIdx.x, nt = blockDim.x;
    const int rows = min(pb.Ns, bytes / (4 * ld));
    float *hs = (float *)buf;
    for (int q0 = 0; q0 < ni * nj; q0 += nt) {
        const int q = q0 + tid, i0 = q / nj * 8, j0 = (q - q / nj * nj) * 4;
        const bool on = q < ni * nj;
        const int i1 = i0 + 4 < fst ? i0 + 4 : i0;  // (past the last string: not stored)
        uint64_t a[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) a[i][j] = 0ull;
        for (int J0 = 0; J0 < pb.Ns; J0 += rows) {
            const int jn = min(rows, pb.Ns - J0);
            __syncthreads();
#pragma unroll 4
            for (int e = tid; e < jn * nj; e += nt) ((float4 *)hs)[e] = ((const float4 *)(Hs + J0 * ld))[e];
            __syncthreads();
            if (on)
#pragma unroll 2
                for (int J = 0; J < jn; ++J) {
                    const float4 h = *(const float4 *)(hs + J * ld + j0);
                    const ulonglong2 c0 = *(const ulonglong2 *)(c + (J0 + J) * fst + i0),
                                     c1 = *(const ulonglong2 *)(c + (J0 + J) * fst + i1);
                    const uint64_t cc[4] = {c0.x, c0.y, c1.x, c1.y};
                    const uint64_t hh[4] = {dup2(h.x), dup2(h.y), dup2(h.z), dup2(h.w)};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) ffma2(a[i][j], cc[i], hh[j]);
                }
        }
        const float sg = pb.sector > 0 ? 1.f : -1.f;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (on && i0 + i < pb.Ns) {
                float4 o;
                const int h = 32 * (i & 1);
                o.x = sg * __uint_as_float((uint32_t)(a[i >> 1][0] >> h));
                o.y = sg * __uint_as_float((uint32_t)(a[i >> 1][1] >> h));
                o.z = sg * __uint_as_float((uint32_t)(a[i >> 1][2] >> h));
                o.w = sg * __uint_as_float((uint32_t)(a[i >> 1][3] >> h));
                *(float4 *)(M + (i0 + i) * ld + j0) = o;
            }
    }
}

// The same on integers (Hs without its diagonal): 2 x 2 tiles, one int64 per element.
__device__ inline void same_spin(const Problem &pb, int ld, int, const int2 *c, const int2 *Hs, long long *M, char *, int)
{
    const int nt = ld / 2;
    for (int q = threadIdx.x; q < nt * nt; q += blockDim.x) {
        const int i0 = q / nt * 2, j0 = (q - q / nt * nt) * 2;
        const int2 *c0 = c + i0 * ld, *c1 = c + (i0 + 1 < pb.Ns ? i0 + 1 : i0) * ld;
        long long h00 = 0, h01 = 0, h10 = 0, h11 = 0, l00 = 0, l01 = 0, l10 = 0, l11 = 0;
#pragma unroll 2
        for (int J = 0; J < pb.Ns; ++J) {
            const int4 h = *(const int4 *)(Hs + J * ld + j0);
            const int2 a = c0[J], b = c1[J];
            h00 += (long long)a.x * h.x; l00 += (long long)a.x * h.y; l00 += (long long)a.y * h.x;
            h01 += (long long)a.x * h.z; l01 += (long long)a.x * h.w; l01 += (long long)a.y * h.z;
            h10 += (long long)b.x * h.x; l10 += (long long)b.x * h.y; l10 += (long long)b.y * h.x;
            h11 += (long long)b.x * h.z; l11 += (long long)b.x * h.w; l11 += (long long)b.y * h.z;
        }
        const long long half = 1LL << 27;
        if (i0 < pb.Ns) {
            M[i0 * ld + j0] = h00 + ((l00 + half) >> 28);
            M[i0 * ld + j0 + 1] = h01 + ((l01 + half) >> 28);
        }
        if (i0 + 1 < pb.Ns) {
            M[(i0 + 1) * ld + j0] = h10 + ((l10 + half) >> 28);
            M[(i0 + 1) * ld + j0 + 1] = h11 + ((l11 + half) >> 28);
        }
    }
}

// One tile of T in float32: 8 strings x 6 pairs, two strings per instruction (fma.rn.f32x2).  A
// 16-byte shared load takes four cycles of the SM's load path even when all lanes read the same
// address, so the tile is chosen for few bytes per multiply-add: 56 for 48 (at 4 x 6 with V
// stored twice over, 64 for 24, the load path was the bound).
__device__ __forceinline__ void gemm_tile(const Problem &pb, const GemmShape &s, const uint32_t *la, const char *c,
                                          const char *V, int j0, int pg, float *T)
{
    uint64_t a[6][4];
#pragma unroll
    for (int k = 0; k < 6; ++k)
#pragma unroll
        for (int i = 0; i < 4; ++i) a[k][i] = 0ull;
    c += 4 * j0;
    V += 24 * pg;
#pragma unroll 2
    for (int x = 0; x < pb.R; ++x) {
        const uint32_t e = la[x];
        const ulonglong2 *cp = (const ulonglong2 *)(c + ((e & 0xffffu) << 4));
        const ulonglong2 c0 = cp[0], c1 = cp[1];
        const float2 *v = (const float2 *)(V + (e >> 16 << 3));
        const float2 v0 = v[0], v1 = v[1], v2 = v[2];
        const float vv[6] = {v0.x, v0.y, v1.x, v1.y, v2.x, v2.y};
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const uint64_t d = dup2(vv[k]);
            ffma2(a[k][0], d, c0.x);
            ffma2(a[k][1], d, c0.y);
            ffma2(a[k][2], d, c1.x);
            ffma2(a[k][3], d, c1.y);
        }
    }
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (pg * 6 + k < pb.P) {
            float *t = T + (pg * 6 + k) * s.cst + j0;
            *(ulonglong2 *)t = make_ulonglong2(a[k][0], a[k][1]);
            if (j0 + 4 < s.cst) *(ulonglong2 *)(t + 4) = make_ulonglong2(a[k][2], a[k][3]);
        }
}

// One tile of T in fixed point: 4 strings x 3 pairs.
__device__ __forceinline__ void gemm_tile(const Problem &pb, const GemmShape &s, const uint16_t *la, const int2 *c,
                                          const int2 *V, int j0, int pg, long long *T)
{
    long long hi[4][3], lo[4][3];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) hi[i][k] = lo[i][k] = 0;
    const int p0 = pg * 3, p1 = min(p0 + 1, pb.P - 1), p2 = min(p0 + 2, pb.P - 1);
#pragma unroll 1
    for (int x = 0; x < pb.R; ++x) {
        const int e = la[x], m = -(e & 1);
        const int4 c01 = *(const int4 *)(c + (e >> 7) * s.cst + j0), c23 = *(const int4 *)(c + (e >> 7) * s.cst + j0 + 2);
        const int2 *v = V + ((e >> 1) & 63) * pb.P;
        const int ch[4] = {c01.x, c01.z, c23.x, c23.z}, cl[4] = {c01.y, c01.w, c23.y, c23.w};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            int2 w = v[k == 0 ? p0 : k == 1 ? p1 : p2];
            w.x = (w.x ^ m) - m;
            w.y = (w.y ^ m) - m;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                hi[i][k] += (long long)w.x * ch[i];
                lo[i][k] += (long long)w.x * cl[i];
                lo[i][k] += (long long)w.y * ch[i];
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
        if (p0 + k < pb.P)
#pragma unroll
            for (int i = 0; i < 4; ++i) T[(p0 + k) * s.cst + j0 + i] = hi[i][k] + ((lo[i][k] + (1LL << 27)) >> 28);
}

// The strings are taken from both ends of the list, so that each pair of them has Ns + 1 elements
// with Ia <= Ib.
__device__ __forceinline__ int tail_string(int Ns, int i) { return i & 1 ? Ns - 1 - (i >> 1) : i >> 1; }

// sigma of the elements of gc strings from their T and the same-spin terms M.
template <typename T, typename A>
__device__ __forceinline__ void gather_strings(const BlockProblem &B, const GemmShape &s, const A *Tm, const A *M, int I0, int gc,
                                               const T *src, T *dst)
{
    constexpr bool F64 = sizeof(T) == 8;
    const Problem &pb = B.pb;
    const int Ns = pb.Ns, tid = threadIdx.x, nt = blockDim.x, R = pb.R, sgn = pb.sector;
    const uint16_t *list = (const uint16_t *)(block_shared() + B.S.off_list);
    const double *hd = (const double *)(block_shared() + B.S.off_hd);
    const int n1 = Ns + 1, ne = (gc + 1) / 2 * n1;
    int split = 0;  // 2^split threads per element, where they fit
    while (split < 3 && (ne << (split + 1)) <= nt) ++split;
    for (int q0 = 0; q0 < ne << split; q0 += nt) {
        const int q = q0 + tid, el = q >> split, pr = el / n1, r = el - pr * n1;
        const int first = tail_string(Ns, I0 + 2 * pr), len = Ns - first;  // elements of the pair's first string
        const int g = 2 * pr + (r < len ? 0 : 1), Ia = r < len ? first : tail_string(Ns, I0 + g), Ib = Ia + r - (r < len ? 0 : len);
        const bool on = g < gc && Ib < Ns, last = on && (q & ((1 << split) - 1)) == 0;
        // (the same-spin terms come from L2: asked for before the walk over the list)
        const A m0 = last ? M[Ia * s.cst + Ib] : (A)0, m1 = last ? M[Ib * s.cst + Ia] : (A)0;
        A acc = 0;
        if (on) {
            const A *t = Tm + g * pb.P * s.cst;
            const uint16_t *lb = list + Ib * s.rs;
#pragma unroll 4
            for (int y = q & ((1 << split) - 1); y < R; y += 1 << split) {
                const int e = lb[y];
                const A v = t[((e >> 1) & 63) * s.cst + (e >> 7)];
                acc += e & 1 ? -v : v;
            }
        }
        for (int o = 1; o < 1 << split; o <<= 1) acc += __shfl_xor_sync(FULL, acc, o);
        if (last) {
            const int h = Ia * Ns - Ia * (Ia - 1) / 2 + Ib - Ia;
            acc += m0 + (sgn > 0 ? m1 : -m1);
            T v;
            if constexpr (F64) {
                v = fma(hd[Ia] + hd[Ib], src[h], (double)acc * (pow2(B.E - 54) * (Ia == Ib ? 1.0 : 1.4142135623730951)));
                if (B.bad) v = __longlong_as_double(0x7ff8000000000000LL);
            } else {
                v = Ia == Ib ? acc : 1.41421356f * acc;
            }
            dst[h] = sgn < 0 && Ia == Ib ? (T)0 : v;
        }
    }
}

// float64 sigma of a packed sector vector with the products on the tensor cores, in exact digits
// (digits.cuh: 32 multiply-adds per clock and SM, where three wide integer ones per product reach
// 7).  T per alpha string Ia as mma.sync tiles of 16 pairs x 8 strings: the rows of V and c that
// the off-diagonal replacements name are gathered by ldmatrix, the signs are flipped in c's
// fragments, and the k diagonal replacements, all of which keep J = Ia, enter as one row, their
// sum U of V, in integers: k (n - k) <= 16 list entries up to 8 orbitals, one mma step.  The sums
// of up to 32 products stay within 2^22, so the accumulators start at 1.5 * 2^23 and hold
// their integers in the low bits.  A warp takes a run of consecutive tiles.  Tm: [P][cst]
// per string as in sigma_gemm, the same units; the rest of sigma is that of sigma_gemm.
__device__ __noinline__ void sigma_digits(const BlockProblem &B, const double *src, double *dst)
{
    const Problem &pb = B.pb;
    const int n = pb.n, P = pb.P, Ns = pb.Ns, R = pb.R, sgn = pb.sector, tid = threadIdx.x, nt = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const DigitShape d = digit_shape(n, Ns, R);
    GemmShape s = gemm_shape<double>(n, Ns, R);
    s.g = d.g;
    char *at = block_shared() + B.S.off_c;
    uint16_t *cd = (uint16_t *)at, *vd = (uint16_t *)(at + d.off_v), *off = (uint16_t *)(at + d.off_l);
    int2 *rows = (int2 *)(at + d.off_rows);  // per string of a round: its row of c, and U
    const int rst = d.cs + d.mt * 16;
    long long *Tm = (long long *)(block_shared() + B.S.off_T), *M = (long long *)B.full;
    const uint16_t *list = (const uint16_t *)(block_shared() + B.S.off_list);
    const int2 *Vf = (const int2 *)(block_shared() + B.S.off_V64), *Hf = (const int2 *)pb.Hs64;
    const int cplane = (Ns + 1) * d.cs, vplane = P * d.vs, ro = pb.k * (n - pb.k), nks = (ro + 15) / 16, kx = 16 * nks;
    const double one = 36028797018963968.0, root = 0.70710678118654752 * 36028797018963968.0;  // 2^55
    auto joined = [](int2 f) { return ((long long)f.x << 28) + f.y; };
    {
        int ia = 0, ib = 0;
        tri_advance(ia, ib, tid, Ns);
        for (int h = tid; h < pb.N; h += nt) {
            uint16_t f[DIGITS];
            to_digits(__double2ll_rn(src[h] * (ia == ib ? one : root)), f);
#pragma unroll
            for (int i = 0; i < DIGITS; ++i) {
                cd[i * cplane + ia * d.cs + ib] = f[i];
                cd[i * cplane + ib * d.cs + ia] = sgn > 0 ? f[i] : f[i] ^ 0x8000;
            }
            tri_advance(ia, ib, nt, Ns);
        }
        const int pad = d.cs - Ns;
        for (int q = tid; q < Ns * pad + d.cs; q += nt) {
            const int to = q < Ns * pad ? q / pad * d.cs + Ns + q % pad : Ns * d.cs + q - Ns * pad;
#pragma unroll
            for (int i = 0; i < DIGITS; ++i) cd[i * cplane + to] = 0;
        }
        for (int q = tid; q < vplane; q += nt) {
            const int x = q / d.vs, y = q - x * d.vs;
            uint16_t f[DIGITS];
            to_digits(y < P ? joined(Vf[x * P + y]) : 0, f);
#pragma unroll
            for (int i = 0; i < DIGITS; ++i) vd[i * vplane + q] = f[i];
        }
        for (int I = tid; I < Ns; I += nt) {
            int to = 0;
            for (int x = 0; x < R; ++x) {
                const int e = list[I * s.rs + x];
                if (e >> 7 != I) off[I * kx + to++] = (uint16_t)e;
            }
            for (; to < kx; ++to) off[I * kx + to] = (uint16_t)(Ns << 7);
        }
    }
    auto stage_rows = [&](int I0) {
        for (int q = tid; q < min(s.g, Ns - I0) * rst; q += nt) {
            const int g = q / rst, x = q - g * rst, Ia = tail_string(Ns, I0 + g);
            int2 f = make_int2(0, 0);
            if (x < Ns) {
                const int lo = min(Ia, x), hi = max(Ia, x);
                f = to_fixed(src[lo * Ns - lo * (lo - 1) / 2 + hi - lo], Ia == x ? one : root);
                if (sgn < 0 && x < Ia) f = make_int2(-f.x, -f.y);
            } else if (x >= d.cs && x - d.cs < P) {
                for (uint32_t m = pb.str[Ia]; m; m &= m - 1u) {
                    const int2 v = Vf[pair_index(__ffs((int)m) - 1, __ffs((int)m) - 1) * P + x - d.cs];
                    f.x += v.x;
                    f.y += v.y;
                }
            }
            rows[q] = f;
        }
    };
    stage_rows(0);
    // same-spin terms: M = c Hs, the digits of Hs made in chunks of rows where T will be
    const int hr = min(min((Ns + 15) / 16 * 16, 128), (B.S.bytes - B.S.off_T) / (2 * DIGITS * d.cs) / 16 * 16);
    uint16_t *hs = (uint16_t *)Tm;
    for (int J0 = 0; J0 < Ns; J0 += hr) {
        const int jn = min(hr, (Ns - J0 + 15) / 16 * 16), hplane = jn * d.cs;
        __syncthreads();
        for (int q = tid; q < hplane; q += nt) {
            const int J = J0 + q / d.cs, j = q % d.cs;
            uint16_t f[DIGITS];
            to_digits(J < Ns && j < s.cst ? joined(Hf[J * s.cst + j]) : 0, f);
#pragma unroll
            for (int i = 0; i < DIGITS; ++i) hs[i * hplane + q] = f[i];
        }
        __syncthreads();
        for (int t = warp; t < (Ns + 15) / 16 * d.c8; t += nw) {
            const int m = t / d.c8, jt = t - m * d.c8;
            // (rows and columns of c beyond Ns are whatever digits follow: such rows are not
            // stored, such columns meet zeros of Hs)
            const uint32_t aa = shared_u32(cd + (m * 16 + (lane & 15)) * d.cs + (lane >> 4) * 8 + J0);
            const uint32_t ba = shared_u32(hs + (lane & 15) * d.cs + jt * 8);
            float acc[DIGITS][4];
#pragma unroll
            for (int i = 0; i < DIGITS; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
#pragma unroll 1
            for (int k = 0; k < jn; k += 16) {
                uint32_t bf[DIGITS][2];
#pragma unroll
                for (int j = 0; j < DIGITS; ++j) ldsm_x2_trans(bf[j], ba + 2 * (j * hplane + k * d.cs));
#pragma unroll
                for (int i = 0; i < DIGITS; ++i) {
                    uint32_t af[4];
                    ldsm_x4(af, aa + 2 * (i * cplane + k));
#pragma unroll
                    for (int j = 0; i + j < DIGITS; ++j) mma_bf16(acc[i + j], af, bf[j][0], bf[j][1]);
                }
            }
            const int i = m * 16 + (lane >> 2), j = jt * 8 + (lane & 3) * 2;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (i + 8 * h < Ns && j < s.cst) {
                    longlong2 *o = (longlong2 *)(M + (i + 8 * h) * s.cst + j);
                    const longlong2 old = J0 ? *o : make_longlong2(0, 0);
                    *o = make_longlong2(old.x + join_digits(acc, 2 * h), old.y + join_digits(acc, 2 * h + 1));
                }
        }
    }
    __syncthreads();  // (Hs was staged over T)
    for (int I0 = 0; I0 < Ns; I0 += s.g) {
        const int gc = min(s.g, Ns - I0), tiles = gc * d.mt * d.c8, last = (warp + 1) * tiles / nw;
        int now = -1, g = 0, m = 0;
        uint32_t aa[2] = {0, 0}, ba[2] = {0, 0}, flip[2][2] = {{0, 0}, {0, 0}};
        for (int t = warp * tiles / nw; t < last; ++t) {
            const int gm = t / d.c8, jt = t - gm * d.c8;
            if (gm != now) {
                now = gm;
                g = gm / d.mt;
                m = gm - g * d.mt;
                const uint16_t *l = off + tail_string(Ns, I0 + g) * kx;
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    if (k < nks) {
                        ba[k] = shared_u32(cd + (l[16 * k + (lane & 15)] >> 7) * d.cs);
                        aa[k] = shared_u32(vd + (l[16 * k + (lane & 7) + (lane >> 4) * 8] >> 1 & 63) * d.vs + m * 16 + (lane >> 3 & 1) * 8);
                        const uint16_t *x = l + 16 * k + (lane & 3) * 2;
                        flip[k][0] = (x[0] & 1u) << 15 | (x[1] & 1u) << 31;
                        flip[k][1] = (x[8] & 1u) << 15 | (x[9] & 1u) << 31;
                    }
            }
            float acc[DIGITS][4];
#pragma unroll
            for (int i = 0; i < DIGITS; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 12582912.f;
            uint32_t av = aa[0], bv = ba[0] + 16 * jt, f0 = flip[0][0], f1 = flip[0][1];
#pragma unroll 1
            for (int k = 0; k < nks; ++k) {
                uint32_t bf[DIGITS][2];
#pragma unroll
                for (int j = 0; j < DIGITS; ++j) {
                    ldsm_x2_trans(bf[j], bv + 2 * j * cplane);
                    bf[j][0] ^= f0;
                    bf[j][1] ^= f1;
                }
#pragma unroll
                for (int i = 0; i < DIGITS; ++i) {
                    uint32_t af[4];
                    ldsm_x4_trans(af, av + 2 * i * vplane);
#pragma unroll
                    for (int j = 0; i + j < DIGITS; ++j) mma_bf16(acc[i + j], af, bf[j][0], bf[j][1]);
                }
                av = aa[1];
                bv = ba[1] + 16 * jt;
                f0 = flip[1][0];
                f1 = flip[1][1];
            }
            const int p0 = m * 16 + (lane >> 2), J = jt * 8 + (lane & 3) * 2;
            const int4 cr = *(const int4 *)(rows + g * rst + J);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int p = p0 + 8 * h;
                if (p >= P || J >= s.cst) continue;
                const int2 u = rows[g * rst + d.cs + p];
                long long v[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    // (the joins of two sums fit in 32 bits, and the offsets cancel modulo 2^32)
                    auto pair = [&](int i) {
                        return (int)((__float_as_uint(acc[i][2 * h + e]) << 8) + __float_as_uint(acc[i + 1][2 * h + e]) -
                                     0x4b400000u * 257u);
                    };
                    const int rest = ((int)(__float_as_uint(acc[6][2 * h + e]) - 0x4b400000u) + 128) >> 8;
                    const int cx = e ? cr.z : cr.x, cy = e ? cr.w : cr.y;
                    long long lo = 1LL << 27;
                    lo += (long long)u.x * cy;
                    lo += (long long)u.y * cx;
                    v[e] = ((long long)pair(0) << 32) + (long long)pair(2) * 65536 + pair(4) + rest;
                    v[e] += (long long)u.x * cx + (lo >> 28);
                }
                *(longlong2 *)(Tm + (g * P + p) * s.cst + J) = make_longlong2(v[0], v[1]);
            }
        }
        __syncthreads();  // (also orders M, written above, before its first use)
        gather_strings<double>(B, s, Tm, M, I0, gc, src, dst);
        if (I0 + s.g < Ns) stage_rows(I0 + s.g);
        __syncthreads();
    }
}

// sigma of a packed sector vector, tiled product.
template <typename T>
__device__ __noinline__ void sigma_gemm(const BlockProblem &B, const T *src, T *dst)
{
    constexpr bool F64 = sizeof(T) == 8;
    using E = typename std::conditional<F64, int2, float>::type;       // elements of c and V
    using A = typename std::conditional<F64, long long, float>::type;  // sums
    const Problem &pb = B.pb;
    const int Ns = pb.Ns, tid = threadIdx.x, nt = blockDim.x, R = pb.R, sgn = pb.sector;
    const GemmShape s = gemm_shape<T>(pb.n, Ns, R);
    E *c = (E *)(block_shared() + B.S.off_c);
    A *Tm = (A *)(block_shared() + B.S.off_T);
    const uint16_t *list = (const uint16_t *)(block_shared() + B.S.off_list);
    const double *hd = (const double *)(block_shared() + B.S.off_hd);
    A *M = (A *)B.full;
    const int cld = F64 ? s.cst : s.fst;
    // float32: behind c, V with both signs (rows 2 pair + neg), and the lists as offsets of the
    // rows of c (low half, in units of 16 bytes) and V (high half, 8 bytes)
    char *Vd = block_shared() + B.S.off_c + al16(4 * Ns * s.fst);
    uint32_t *list32 = (uint32_t *)(Vd + 8 * pb.P * s.pst);
    {
        int ia = 0, ib = 0;
        tri_advance(ia, ib, tid, Ns);
        for (int h = tid; h < pb.N; h += nt) {
            if constexpr (F64) {
                const int2 f = to_fixed(src[h], ia == ib ? 36028797018963968.0 : 0.70710678118654752 * 36028797018963968.0);
                c[ia * cld + ib] = f;
                c[ib * cld + ia] = sgn > 0 ? f : make_int2(-f.x, -f.y);
            } else {
                const float f = ia == ib ? src[h] : 0.70710678118654752f * src[h];
                c[ia * cld + ib] = f;
                c[ib * cld + ia] = sgn > 0 ? f : -f;
            }
            tri_advance(ia, ib, nt, Ns);
        }
        for (int q = tid; q < Ns * (cld - Ns); q += nt) c[q / (cld - Ns) * cld + Ns + q % (cld - Ns)] = E{};
        if constexpr (!F64) {
            const float *V32 = (const float *)(block_shared() + B.S.off_V32);
            for (int q = tid; q < pb.P * s.pst; q += nt) {
                const int x = q / s.pst, y = q - x * s.pst;
                ((float *)Vd)[2 * x * s.pst + y] = V32[q];
                ((float *)Vd)[(2 * x + 1) * s.pst + y] = -V32[q];
            }
            for (int q = tid; q < Ns * R; q += nt) {
                const int e = list[q / R * s.rs + q % R];
                list32[q] = (uint32_t)((e >> 7) * (s.fst / 4)) | (uint32_t)((e & 127) * (s.pst / 2)) << 16;
            }
        }
    }
    __syncthreads();
    same_spin(pb, s.cst, cld, c, F64 ? (const E *)pb.Hs64 : (const E *)pb.Hs32, M, (char *)Tm,
              s.g * pb.P * s.cst * (int)sizeof(A));
    if constexpr (!F64) __syncthreads();  // (Hs was staged over T)
    for (int I0 = 0; I0 < Ns; I0 += s.g) {
        const int gc = min(s.g, Ns - I0);
        for (int q = tid; q < gc * s.tiles; q += nt) {
            const int g = q / s.tiles, r = q - g * s.tiles, pg = r / s.nj, jj = r - pg * s.nj, Ia = tail_string(Ns, I0 + g);
            if constexpr (F64)
                gemm_tile(pb, s, list + Ia * s.rs, c, (const int2 *)(block_shared() + B.S.off_V64), 4 * jj, pg,
                          Tm + g * pb.P * s.cst);
            else
                gemm_tile(pb, s, list32 + Ia * R, (const char *)c, Vd, 8 * jj, pg, Tm + g * pb.P * s.cst);
        }
        __syncthreads();  // (also orders M, written above, before its first use)
        gather_strings<T>(B, s, Tm, M, I0, gc, src, dst);
        __syncthreads();
    }
}

// Float32 sigma of 10-16 orbitals with few strings: c and V in shared memory, one element per
// thread.  The diagonal replacements are summed beforehand (U), so that k (n - k) entries of
// each list are left, and each string's entries are sorted by sign: (k (n - k))^2 multiply-adds
// per element instead of R^2 (676 for 1,521 at 13 electron pairs in 15 orbitals), two shared
// gathers each; four entries of Ib share the decoding of one of Ia.
__device__ __noinline__ void sigma_list(const BlockProblem &B, const float *src, float *dst)
{
    const Problem &pb = B.pb;
    const BlockMem &S = B.S;
    char *smem = block_shared();
    const int Ns = pb.Ns, P = pb.P, tid = threadIdx.x, nt = blockDim.x, sgn = pb.sector, ld = list_stride(Ns), vs = v32_stride(SIGMA_LIST, P);
    const int ro = pb.k * (pb.n - pb.k);  // entries; word ro of a list holds the number of positive ones
    float *c = (float *)(smem + S.off_c);
    const char *V = smem + S.off_V32;
    const uint32_t *list = (const uint32_t *)(smem + S.off_list);
    float *M = (float *)B.full;
    {
        int ia = 0, ib = 0;
        tri_advance(ia, ib, tid, Ns);
        for (int h = tid; h < pb.N; h += nt) {
            const float f = ia == ib ? src[h] : 0.70710678118654752f * src[h];
            c[ia * ld + ib] = f;
            c[ib * ld + ia] = sgn > 0 ? f : -f;
            tri_advance(ia, ib, nt, Ns);
        }
        for (int q = tid; q < Ns * (ld - Ns); q += nt) c[q / (ld - Ns) * ld + Ns + q % (ld - Ns)] = 0.f;
    }
    __syncthreads();
    same_spin(pb, hs_stride(Ns), ld, c, pb.Hs32, M, smem + S.off_T, LIST_STAGE);
    __syncthreads();
    int ia = 0, ib = 0;
    tri_advance(ia, ib, tid, Ns);
    for (int h = tid; h < pb.N; h += nt) {
        const uint32_t *la = list + ia * (ro + 1), *lb = list + ib * (ro + 1);
        const float *Ua = B.U + ia * P, *Ub = B.U + ib * P;
        const int ap = la[ro], bp = lb[ro];
        float acc = 0.f;
        // both replacements off the diagonal; a list word is 4 pair | (4 ld J) << 12
        for (int y0 = 0; y0 < ro; y0 += 4) {
            const char *v[4], *cc[4];
            float s[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t e = lb[y0 + i < ro ? y0 + i : ro - 1];
                v[i] = V + (e & 0xfffu) * vs;            // row pair(e)
                cc[i] = (const char *)c + (e >> 12) / ld;  // column J(e)
                s[i] = 0.f;
            }
#pragma unroll 2
            for (int x = 0; x < ap; ++x) {
                const uint32_t e = la[x], p = e & 0xfffu, j = e >> 12;
#pragma unroll
                for (int i = 0; i < 4; ++i) s[i] = fmaf(*(const float *)(v[i] + p), *(const float *)(cc[i] + j), s[i]);
            }
#pragma unroll 2
            for (int x = ap; x < ro; ++x) {
                const uint32_t e = la[x], p = e & 0xfffu, j = e >> 12;
#pragma unroll
                for (int i = 0; i < 4; ++i) s[i] = fmaf(-*(const float *)(v[i] + p), *(const float *)(cc[i] + j), s[i]);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (y0 + i < ro) acc += y0 + i < bp ? s[i] : -s[i];
        }
        // one of them on the diagonal, then both
        float one = 0.f;
        for (int x = 0; x < ro; ++x) {
            const uint32_t a = la[x], b = lb[x];
            const float u = Ub[(a & 0xfffu) >> 2] * *(const float *)((const char *)(c + ib) + (a >> 12));
            const float w = Ua[(b & 0xfffu) >> 2] * *(const float *)((const char *)(c + ia * ld) + (b >> 12) / ld);
            one += x < ap ? u : -u;
            one += x < bp ? w : -w;
        }
        float dd = 0.f;
        for (uint32_t m = pb.str[ib]; m; m &= m - 1u) {
            const int q = __ffs((int)m) - 1;
            dd += Ua[pair_index(q, q)];
        }
        acc += one + dd * c[ia * ld + ib];
        const float mt = M[ib * hs_stride(Ns) + ia];
        acc += M[ia * hs_stride(Ns) + ib] + (sgn > 0 ? mt : -mt);
        dst[h] = ia == ib ? (sgn > 0 ? acc : 0.f) : 1.41421356f * acc;
        tri_advance(ia, ib, nt, Ns);
    }
    __syncthreads();
}

// sigma of a packed sector vector; ends with a barrier.
template <typename T>
__device__ __noinline__ void sigma_block(const BlockProblem &B, const T *src, T *dst)
{
    const Problem &pb = B.pb;
    const bool done = B.form == SIGMA_TILED || (B.form == SIGMA_LIST && sizeof(T) == 4);  // but for the penalty
    if (B.form == SIGMA_TILED) {
        bool digits = false;
        if constexpr (sizeof(T) == 8) {
            digits = B.S.digits;
            if (digits) sigma_digits(B, src, dst);
        }
        if (!digits) sigma_gemm<T>(B, src, dst);
    }
    if constexpr (sizeof(T) == 4)
        if (B.form == SIGMA_LIST) sigma_list(B, src, dst);
    if (done && pb.s2mu == 0.0) return;
    T *full = (T *)B.full;
    expand_full<T>(pb, src, full, pb.Ns);
    __syncthreads();
    int ia = 0, ib = 0;
    tri_advance(ia, ib, threadIdx.x, pb.Ns);
    for (int h = threadIdx.x; h < pb.N; h += blockDim.x) {
        T v = (T)0;
        if (!(pb.sector < 0 && ia == ib)) {
            if (!done) {
                if constexpr (sizeof(T) == 4)
                    v = sigma_elem_ashared<T>(pb, pb.V32, pb.Hs32, full, ia, ib);
                else
                    v = sigma_elem<T>(pb, pb.V64, pb.Hs64, full, ia * pb.Ns + ib);
            }
            if (pb.s2mu != 0.0) v += (T)pb.s2mu * s2_elem<T, T>(pb, full, ia, ib);
            if (ia != ib) v *= (T)1.4142135623730951;
        }
        dst[h] = done ? dst[h] + v : v;
        tri_advance(ia, ib, blockDim.x, pb.Ns);
    }
    __syncthreads();
}

// Lowest eigenpair of the m x m symmetric Rayleigh matrix G (shared memory, float64, row
// stride MMAX) by the whole block.  warm: the last call was on the leading (m - 1) x (m - 1) part
// of G; in its eigenbasis an arrow matrix is left, whose eigenvalues are the roots of a secular
// equation (one lane each) and whose eigenvectors have a closed form, with the couplings recomputed
// from the roots, which keeps them orthogonal (Gu and Eisenstat, SIAM J. Matrix Anal. Appl. 16,
// 172, 1995).  Otherwise a float32 Jacobi on G - G00 I in round-robin order, m / 2 disjoint
// rotations at a time (60-90 thousand cycles where the arrow takes 19, or 33 in
// float64).  In float64 then two Newton steps in that
// eigenbasis, z = y - sum_{k != 0} e_k (e_k . r) / (theta_k - theta),  r = G y - theta y,
// theta = y.G y, which make the lowest pair float64-accurate; in float32 one (one warp).
// All float32 work is on (G - G00 I) 2^-e, e from its largest element, so that neither its squares
// nor the absolute floors below depend on the unit of the integrals; ev is kept in that unit, e
// (which may change from call to call) in misc[1].
// Output: y[0..m) (unit norm), y2 (the second lowest, which seeds the thick restart), and
// misc[0] = theta; ends with a barrier.
template <bool REFINE>
__device__ __noinline__ void small_eig_block(const BlockMem &S, int m, bool warm)
{
    char *smem = block_shared();
    const double *G = (const double *)(smem + S.off_G);
    float *buf = (float *)(smem + S.off_J), *ev = (float *)(smem + S.off_ev);
    double *y = (double *)(smem + S.off_y), *y2 = (double *)(smem + S.off_yp), *r = (double *)(smem + S.off_r),
           *misc = (double *)(smem + S.off_misc);
    __shared__ float2 rot[MMAX + 1];
    const int tid = threadIdx.x, i = tid / MMAX, j = tid - i * MMAX, lane = tid & 31;
    const bool on = i < m && j < m;
    const double shift = G[0];
    int top = lane < m ? high_word(G[lane * MMAX + lane] - shift) : 0;  // (in every warp)
    for (int q = lane; q < m * MMAX; q += 32)
        if (q % MMAX < q / MMAX) top = max(top, high_word(G[q]));
    top = __reduce_max_sync(FULL, top);
    const int e2 = top == 0 ? 0 : max(-1000, min(1000, (top >> 20) - 1023));
    const double down = pow2(-e2), up = pow2(e2);
    float *A = buf, *E = buf + MMAX * MMAX, *A2 = buf + 2 * MMAX * MMAX, *E2 = buf + 3 * MMAX * MMAX;
    if (warm) {
        // half a warp per pole or root, its lanes share the terms of every sum
        const int q = m - 1, half = tid >> 4, l0 = tid & 15;
        const bool work = half < MMAX;  // (whole warps)
        float *sd = A2, *sb = sd + MMAX, *sp = sb + MMAX, *st = sp + MMAX, *sn = st + MMAX;  // poles, couplings, a root's
                                                                                            // pole and offset, norms
        auto sum16 = [](float v) {
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
            return v;
        };
        auto over = [](float x, float y) {  // x / y, y a normal number
            float r;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y));
            return x * r;
        };
        auto gap = [&](int k, int l) { return (sp[k] - sd[l]) + st[k]; };  // root k - pole l
        if (work) {
            float b = 0.f;  // the new row in the last basis
            for (int k = l0; k < q; k += 16) b += half < q ? E[k * MMAX + half] * (float)(G[k * MMAX + q] * down) : 0.f;
            b = sum16(b);
            if (l0 == 0) sb[half] = b;
        }
        __syncthreads();
        // the arrow matrix: diagonal d = ev, row b, corner a
        const float a = (float)((G[q * MMAX + q] - shift) * down);
        const float unit = (float)pow2(max(-126, min(126, (int)misc[1] - e2)));  // of the last ev
        float b = lane < q ? sb[lane] : 0.f, d = lane < q ? ev[lane] * unit : 0.f;  // (in every warp)
        float scale = fmaxf(fabsf(a), fmaxf(fabsf(d), fabsf(b)));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) scale = fmaxf(scale, __shfl_xor_sync(FULL, scale, o));
        // poles apart by a rounding error of the matrix; couplings nonzero, their squares in float32's
        // range (and no larger: those of an anchored basis to x0 are of the size of its residual, and
        // whatever is added to them bounds the residual that a refinement can reach)
        const float eps = fmaxf(1.2e-7f * scale, 1e-15f);
        if (lane < q && fabsf(b) < 1e-17f) b = copysignf(1e-17f, b);
        d = lane < q ? d - lane * 2.f * eps : -3e38f;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float u = __shfl_up_sync(FULL, d, o);
            if (lane >= o && lane < q) d = fmaxf(d, u);
        }
        d += lane * 2.f * eps;
        const float nb = sqrtf(warp_sum(b * b)) * 1.001f;
        if (tid < q) sd[tid] = d;
        __syncthreads();  // (sb has been read)
        if (tid < q) sb[tid] = b;
        __syncthreads();
        if (work) {
            const int l1 = l0 + 16;
            const float d0 = l0 < q ? sd[l0] : 0.f, b0 = l0 < q ? sb[l0] * sb[l0] : 0.f;
            const float d1 = l1 < q ? sd[l1] : 0.f, b1 = l1 < q ? sb[l1] * sb[l1] : 0.f;
            auto secular = [&](float pole, float t) {  // falls from pole to pole
                float f = l0 < q ? over(b0, (d0 - pole) - t) : 0.f;
                if (l1 < q) f += over(b1, (d1 - pole) - t);
                return ((a - pole) - t) - sum16(f);
            };
            // root `half` lies between poles half - 1 and half: as a distance from the nearer one, by
            // bisection on its bits
            const int k = min(half, q), lp = max(k - 1, 0), rp = min(k, q - 1);
            const float mid2 = 0.5f * (sd[rp] - sd[lp]);
            const float fm = secular(sd[lp], mid2 > 0.f ? mid2 : nb);
            const bool left = k == q || (k > 0 && !(fm > 0.f));
            const float pole = sd[left ? lp : rp];
            const float lim = k == 0 ? fmaxf(pole - a, 0.f) + nb : k == q ? fmaxf(a - pole, 0.f) + nb : mid2;
            int lo = 0x00800000, hi = max(__float_as_int(lim), lo);
#pragma unroll 1
            for (int it = 0; it < 31; ++it) {
                const int mid = lo + ((hi - lo) >> 1);
                const float t = __int_as_float(mid);
                if ((secular(pole, left ? t : -t) > 0.f) == left)
                    lo = mid;
                else
                    hi = mid;
            }
            if (l0 == 0 && half <= q) {
                sp[half] = pole;
                st[half] = left ? __int_as_float(hi) : -__int_as_float(hi);
            }
        }
        __syncthreads();
        float bh = 0.f;
        if (work) {
            // the couplings whose arrow matrix has exactly these roots
            float p = 1.f;
            for (int l = l0; l < q; l += 16)
                if (half < q) p *= l == half ? -gap(l, half) * gap(l + 1, half) : over(gap(l < half ? l : l + 1, half), sd[l] - sd[half]);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) p *= __shfl_xor_sync(FULL, p, o);
            bh = half < q ? copysignf(sqrtf(fmaxf(p, 0.f)), sb[half]) : 0.f;
        }
        __syncthreads();
        if (work && l0 == 0 && half < q) sb[half] = bh;
        __syncthreads();
        if (work) {
            float z = 0.f;
            for (int l = l0; l < q; l += 16)
                if (half <= q) {
                    const float v = over(sb[l], gap(half, l));
                    z += v * v;
                }
            z = sum16(z);
            if (l0 == 0 && half <= q) {
                sn[half] = rsqrtf(1.f + z);
                ev[half] = sp[half] + st[half];
            }
        }
        __syncthreads();
        if (on) A[tid] = sn[j] * (i < q ? over(sb[i], gap(j, i)) : 1.f);
        __syncthreads();
        float e = 0.f;
        if (on) {
            if (i < q)
                for (int l = 0; l < q; ++l) e += E[i * MMAX + l] * A[l * MMAX + j];
            else
                e = A[tid];
        }
        __syncthreads();
        if (on) E[tid] = e;
        __syncthreads();
    }
    if (!warm) {
        if (on) {
            A[tid] = (float)((G[i * MMAX + j] - (i == j ? shift : 0.0)) * down);
            E[tid] = i == j ? 1.0f : 0.0f;
        }
        __syncthreads();
    }
    const int M = m + (m & 1);  // an odd matrix gets an idle partner
    for (int sweep = 0; sweep < 10 && m > 1 && !warm; ++sweep) {
        float dia = 0.f;
        bool big = false;
        if (on) {
            for (int k = 0; k < m; ++k) dia += A[k * MMAX + k] * A[k * MMAX + k];
            const float a = A[tid];
            big = i != j && a * a > 1e-14f * dia && fabsf(a) > 1e-18f;
        }
        if (!__syncthreads_or(big)) break;
        for (int step = 0; step < M - 1; ++step) {
            auto partner = [&](int u) {
                if (u == M - 1) return step;
                if (u == step) return M - 1;
                const int v = 2 * step - u;
                return v < 0 ? v + M - 1 : v >= M - 1 ? v - (M - 1) : v;
            };
            // the rotations of the step, one lane each: coefficients of a row itself and of its partner
            if (tid < M) {
                const int v = partner(tid);
                if (tid < v) {
                    float c = 1.f, sn = 0.f;
                    const float apq = v < m ? A[tid * MMAX + v] : 0.f;
                    if (fabsf(apq) >= 1e-36f) {
                        // (fast division and root: a rotation that is off by a rounding error leaves
                        // that much for the next sweep)
                        const float th = __fdividef(A[v * MMAX + v] - A[tid * MMAX + tid], 2.0f * apq), q = th * th + 1.0f;
                        float t = q < 1e30f ? __fdividef(1.0f, fabsf(th) + q * rsqrtf(q)) : 0.5f / fabsf(th);
                        if (th < 0.0f) t = -t;
                        c = rsqrtf(t * t + 1.0f);
                        sn = t * c;
                    }
                    rot[tid] = make_float2(c, -sn);
                    rot[v] = make_float2(c, sn);
                }
            }
            __syncthreads();
            if (on) {
                const int pi = partner(i), pj = partner(j);
                const float2 ri = rot[i], rj = rot[j];
                const int ui = pi < m ? pi : i, uj = pj < m ? pj : j;
                const float a0 = rj.x * A[i * MMAX + j] + rj.y * A[i * MMAX + uj];
                const float a1 = rj.x * A[ui * MMAX + j] + rj.y * A[ui * MMAX + uj];
                A2[tid] = pi == j ? 0.0f : ri.x * a0 + ri.y * a1;
                E2[tid] = rj.x * E[i * MMAX + j] + rj.y * E[i * MMAX + uj];
            }
            __syncthreads();
            float *z = A;
            A = A2;
            A2 = z;
            z = E;
            E = E2;
            E2 = z;
        }
    }
    if (!warm) {
        // eigenvalues in ascending order, into ev and the place of E
        int *rank = (int *)rot;
        if (tid < m) {
            const float x = A[tid * MMAX + tid];
            int r = 0;
            for (int k = 0; k < m; ++k) {
                const float v = A[k * MMAX + k];
                r += v < x || (v == x && k < tid) ? 1 : 0;
            }
            rank[tid] = min(r, m - 1);
            ev[min(r, m - 1)] = x;
        }
        const float e = on ? E[tid] : 0.f;
        __syncthreads();
        E = buf + MMAX * MMAX;
        if (on) E[i * MMAX + rank[j]] = e;
        __syncthreads();
    }
    if (tid < 32) {
        constexpr int bi = 0;
        if (lane < m) {
            y[lane] = (double)E[lane * MMAX];
            y2[lane] = m > 1 ? (double)E[lane * MMAX + 1] : 0.0;
        }
        __syncwarp();
        double theta = shift + (double)ev[0] * up;
        __syncwarp();
        if (!REFINE) {
            // one such step in float32, which also takes out what the warm starts have gathered in E
            float row[MMAX];
            const double own = lane < m ? G[lane * MMAX + lane] - shift : 0.0;
#pragma unroll
            for (int k = 0; k < MMAX; ++k)
                row[k] = lane < m && k < m ? (float)((k == lane ? own : G[lane * MMAX + k]) * down) : 0.f;
            float yi = lane < m ? E[lane * MMAX + bi] : 0.f;
            float th = 0.f;
#pragma unroll 1
            for (int step = 0; step < 2; ++step) {
                float g = 0.f;
#pragma unroll
                for (int k = 0; k < MMAX; ++k) g += row[k] * __shfl_sync(FULL, yi, k);
                th = warp_sum(yi * g) / warp_sum(yi * yi);
                if (step == 1) break;
                const float ri = g - th * yi;
                float ck = 0.f;
                for (int k = 0; k < m; ++k) ck += (lane < m ? E[k * MMAX + lane] : 0.f) * __shfl_sync(FULL, ri, k);
                const float den = lane < m ? ev[lane] - th : 0.f;
                ck = lane != bi && fabsf(den) > 1e-30f ? ck / den : 0.f;
                float z = yi;
                for (int k = 0; k < m; ++k) z -= (lane < m ? E[lane * MMAX + k] : 0.f) * __shfl_sync(FULL, ck, k);
                yi = z * rsqrtf(warp_sum(z * z));
            }
            if (lane < m) y[lane] = (double)yi;
            theta = shift + (double)th * up;
        }
        if (REFINE) {
            for (int step = 0; step < 2; ++step) {
                double g = 0.0, yi = (lane < m) ? y[lane] : 0.0;
                if (lane < m)
                    for (int k = 0; k < m; ++k) g += G[lane * MMAX + k] * y[k];
                double yy = warp_sum(yi * yi), ygy = warp_sum(yi * g);
                theta = ygy / yy;
                if (lane < m) r[lane] = g - theta * yi;
                __syncwarp();
                // coefficient of eigenvector k (lane k)
                double ck = 0.0;
                if (lane < m && lane != bi) {
                    for (int k = 0; k < m; ++k) ck += (double)E[k * MMAX + lane] * r[k];
                    double den = shift + (double)ev[lane] * up - theta;
                    ck = (fabs(den) > 1e-300) ? ck / den : 0.0;
                }
                __syncwarp();
                if (lane < m) r[lane] = ck;  // reuse r for the coefficients
                __syncwarp();
                double z = yi;
                if (lane < m)
                    for (int k = 0; k < m; ++k) z -= (double)E[lane * MMAX + k] * r[k];
                double zz = warp_sum(z * z);
                if (lane < m) y[lane] = z / sqrt(zz);
                __syncwarp();
            }
            double g = 0.0, yi = (lane < m) ? y[lane] : 0.0;
            if (lane < m)
                for (int k = 0; k < m; ++k) g += G[lane * MMAX + k] * y[k];
            theta = warp_sum(yi * g);
        }
        if (lane == 0) {
            misc[0] = theta;
            misc[1] = (double)e2;
        }
    }
    __syncthreads();
}

// Sums of K values over the block; every thread gets the totals.  Two barriers.
template <int K, typename T>
__device__ __forceinline__ void block_sums(T (&v)[K], T *red)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int i = 0; i < K; ++i) v[i] = warp_sum(v[i]);
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < K; ++i) red[w * KRED + i] = v[i];
    __syncthreads();
    T *tot = red + 31 * KRED;
    if (w < K) {
        const T s = warp_sum(lane < nw ? red[lane * KRED + w] : (T)0);
        if (lane == 0) tot[w] = s;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < K; ++i) v[i] = tot[i];
}

// The same for the first k <= KRED of the values of v, which end up in tot[0..k) (shared).  A
// warp folds the values and its lanes at the same time: 31 exchanges, after which lane i holds
// the sum of value i.
template <typename T>
__device__ __forceinline__ const T *block_sums_many(T (&v)[32], int k, T *red)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {
        const bool up = lane & m;
#pragma unroll
        for (int i = 0; i < m; ++i) {
            const T send = up ? v[i] : v[i + m];
            const T keep = up ? v[i + m] : v[i];
            v[i] = keep + __shfl_xor_sync(FULL, send, m);
        }
    }
    if (lane < KRED) red[w * KRED + lane] = v[0];
    __syncthreads();
    T *tot = red + 31 * KRED;
    for (int i = w; i < k; i += nw) {
        const T s = warp_sum(lane < nw ? red[lane * KRED + i] : (T)0);
        if (lane == 0) tot[i] = s;
    }
    __syncthreads();
    return tot;
}

// The vectors are read and written 16 bytes at a time; the elements between N and the next
// multiple of 16 bytes are zero in every vector (one in the diagonal).
template <typename T>
struct alignas(16) Pack {
    static constexpr int L = 16 / sizeof(T);
    T e[L];
};

// One Davidson phase in precision T on packed sector vectors.  V, W: MMAX vectors each,
// leading dimension ld (elements).
// Plain: x is the start vector in, the unit Ritz vector out.  Anchored (T =
// float, anch): V[0] = x0 and W[0] = r0 = (H - shift) x0 are given (see struct
// Anchor), every other basis vector is a correction whose image is the float32
// sigma minus shift times it, the Ritz value is that of H - shift, the coupling
// of x0 to a vector v is formed as v.r0, a thick restart keeps x0 and the
// corrections of the two lowest Ritz vectors, and x returns the correction d of
// the Ritz vector x0 + d.  steer: iterations without a 10% residual drop that end
// the phase (0: none).
template <typename T>
__device__ __noinline__ PhaseOut davidson_block(const BlockProblem &B, T *Vp, T *Wp, size_t ld_, T *xp, T *tp, double tol,
                                                int min_iter, int max_iter, int steer, double shift = 0.0,
                                                bool anchored = false, int mmax = MMAX)
{
    using K = Pack<T>;
    bool anch = anchored;
    constexpr int VL = K::L;
    const Problem &pb = B.pb;
    const BlockMem &S = B.S;
    char *smem = block_shared();
    const int tid = threadIdx.x, nt = blockDim.x, N = (pb.N + VL - 1) / VL;  // packs
    const size_t ld = ld_ / VL;
    K *V = (K *)Vp, *W = (K *)Wp, *x = (K *)xp, *tx = (K *)tp;
    T *red = (T *)(smem + S.off_red);
    double *G = (double *)(smem + S.off_G);
    double *ys = (double *)(smem + S.off_y);
    double *y2s = (double *)(smem + S.off_yp);
    double *misc = (double *)(smem + S.off_misc);
    PhaseOut o;
    o.nsig = 0;
    o.status = MBE_STATUS_OK;
    o.dnorm = 0.0;
    const T shT = (T)shift, shT_lo = (T)(shift - (double)shT);
    // float32 residuals are squared in the unit 2^Eh and the corrections kept near |r| 2^-Eh (the floor
    // of the preconditioner's denominator is 1e-4 in any unit): integrals of 1e-18 would underflow
    const int Ec = sizeof(T) == 8 ? 0 : max(-100, min(100, B.Eh));
    const T per_unit = (T)pow2(-Ec), unit = (T)pow2(Ec), lift = (T)pow2(Ec < -13 ? -13 - Ec : 0);
    T v1[1], v2[2];
    auto dot = [&](const K &a, const K &b, T s) {
#pragma unroll
        for (int l = 0; l < VL; ++l) s = fma(a.e[l], b.e[l], s);
        return s;
    };
    auto axpy = [&](T a, const K &b, K &c) {
#pragma unroll
        for (int l = 0; l < VL; ++l) c.e[l] = fma(a, b.e[l], c.e[l]);
    };
    auto scale = [&](T a, K *c) {
        for (int d = tid; d < N; d += nt) {
            K q = c[d];
#pragma unroll
            for (int l = 0; l < VL; ++l) q.e[l] *= a;
            c[d] = q;
        }
    };
    if (!anch) {
        v1[0] = 0;
        for (int d = tid; d < N; d += nt) v1[0] = dot(x[d], x[d], v1[0]);
        block_sums(v1, red);
        const T inv = (T)1 / sqrt(v1[0]);
        for (int d = tid; d < N; d += nt) {
            K q = x[d];
#pragma unroll
            for (int l = 0; l < VL; ++l) q.e[l] *= inv;
            V[d] = q;
        }
        __syncthreads();
        sigma_block<T>(B, (const T *)V, (T *)W);
        ++o.nsig;
        v1[0] = 0;
        for (int d = tid; d < N; d += nt) v1[0] = dot(V[d], W[d], v1[0]);
        block_sums(v1, red);
        if (tid == 0) G[0] = (double)v1[0];
    } else if (tid == 0) {
        G[0] = 0.0;  // x0.r0 = 0: shift is x0's Rayleigh quotient
    }
    __syncthreads();
    int m = 1, warm = 0;
    double theta = 0.0;
    T rn = 0;
    T best = (T)3e38;
    int stall = 0;
    for (int it = 0;; ++it) {
        anch = opaque(anchored);
        small_eig_block<sizeof(T) == 8>(S, m, opaque(warm));
        warm = 1;
        theta = misc[0];
        const T th = (T)theta;
        K *tdst = (m < mmax) ? V + (size_t)m * ld : tx;
        v2[0] = v2[1] = 0;
        for (int d = tid; d < N; d += nt) {
            K xs, hs, td;
#pragma unroll
            for (int l = 0; l < VL; ++l) xs.e[l] = hs.e[l] = 0;
#pragma unroll 4
            for (int i = 0; i < m; ++i) {
                const T yi = (T)ys[i];
                axpy(yi, V[(size_t)i * ld + d], xs);
                axpy(yi, W[(size_t)i * ld + d], hs);
            }
#pragma unroll
            for (int l = 0; l < VL; ++l) {
                const T r = hs.e[l] - th * xs.e[l], ru = r * per_unit;
                v2[0] += ru * ru;
                T den = (T)(pb.diag[d * VL + l] - shift) - th;
                if (fabs(den) < (T)1e-4) den = den >= (T)0 ? (T)1e-4 : (T)-1e-4;
                td.e[l] = r * lift / den;
                v2[1] += td.e[l] * td.e[l];
            }
            tdst[d] = td;
        }
        block_sums(v2, red);
        rn = sqrt(v2[0]) * unit;
        const T t0n = sqrt(v2[1]);
        if (!isfinite(rn) || !isfinite(theta)) {
            o.status = MBE_STATUS_NONFINITE;
            break;
        }
        if (rn <= (T)tol && it >= min_iter) break;
        if (it >= max_iter) {
            o.status = MBE_STATUS_MAXITER;
            break;
        }
        if (steer) {
            if (rn < (T)0.9 * best) {
                best = rn;
                stall = 0;
            } else if (++stall >= steer) {
                break;
            }
        }
        if (m == mmax) {
            // Thick restart on the two lowest Ritz vectors (orthogonal by construction, so W
            // stays consistent with H V); anchored: V[0] = x0, W[0] = r0 stay and the
            // corrections of the two go to V[1], V[2] (both orthogonal to x0).
            const int b = anch ? 1 : 0;
            K *V0 = V + b * ld, *W0 = W + b * ld, *V1 = V0 + ld, *W1 = W0 + ld;
            v1[0] = 0;
            for (int d = tid; d < N; d += nt) {
                K u1, w1, u2, w2;
#pragma unroll
                for (int l = 0; l < VL; ++l) u1.e[l] = w1.e[l] = u2.e[l] = w2.e[l] = 0;
#pragma unroll 2
                for (int i = b; i < mmax; ++i) {
                    const K vi = V[(size_t)i * ld + d], wi = W[(size_t)i * ld + d];
                    axpy((T)ys[i], vi, u1);
                    axpy((T)ys[i], wi, w1);
                    axpy((T)y2s[i], vi, u2);
                    axpy((T)y2s[i], wi, w2);
                }
                V0[d] = u1;
                W0[d] = w1;
                V1[d] = u2;
                W1[d] = w2;
                v1[0] = dot(u1, u1, v1[0]);
            }
            block_sums(v1, red);
            const T n0 = sqrt(v1[0]);
            if (anch) {
                scale((T)1 / n0, V0);
                scale((T)1 / n0, W0);
            }
            for (int pass = 0; pass < 2; ++pass) {
                v1[0] = 0;
                for (int d = tid; d < N; d += nt) v1[0] = dot(V0[d], V1[d], v1[0]);
                block_sums(v1, red);
                for (int d = tid; d < N; d += nt) {
                    K q = V1[d], w = W1[d];
                    axpy(-v1[0], V0[d], q);
                    axpy(-v1[0], W0[d], w);
                    V1[d] = q;
                    W1[d] = w;
                }
            }
            v1[0] = 0;
            for (int d = tid; d < N; d += nt) v1[0] = dot(V1[d], V1[d], v1[0]);
            block_sums(v1, red);
            const T nn = sqrt(v1[0]);
            const bool keep = nn > (anch ? (T)1e-3 : (T)0.5);
            if (keep) {
                scale((T)1 / nn, V1);
                scale((T)1 / nn, W1);
            }
            T q[5] = {0, 0, 0, 0, 0};
            for (int d = tid; d < N; d += nt) {
                const K a0 = V0[d], b0 = W0[d];
                q[0] = dot(a0, b0, q[0]);
                if (anch) q[1] = dot(W[d], a0, q[1]);  // x0.(A u1) as u1.r0
                if (keep) {
                    const K a1 = V1[d], b1 = W1[d];
                    q[2] = dot(a0, b1, q[2]);
                    q[3] = dot(a1, b1, q[3]);
                    if (anch) q[4] = dot(W[d], a1, q[4]);
                }
            }
            block_sums(q, red);
            if (tid == 0) {
                G[b * MMAX + b] = (double)q[0];
                if (anch) G[1] = G[MMAX] = (double)q[1];
                if (keep) {
                    G[b * MMAX + b + 1] = G[(b + 1) * MMAX + b] = (double)q[2];
                    G[(b + 1) * MMAX + b + 1] = (double)q[3];
                    if (anch) G[2] = G[2 * MMAX] = (double)q[4];
                }
                // the Ritz vector in the new basis
                ys[b] = anch ? (double)n0 : 1.0;
                ys[b + 1] = 0.0;
            }
            m = b + (keep ? 2 : 1);
            warm = 0;
        }
        // Correction: orthogonalise against V[0..m) into V[m]; a second pass when the first
        // one cancelled (less than half of |t|^2 left; with more left, one pass is orthogonal
        // to within a few rounding errors), and in float64 near the end of what it can reach, where
        // those few add up in the residual (integrals of 5: 95% of the (8,4) tuples got to 1e-13
        // with two passes, 76% without).
        const bool twice = sizeof(T) == 8 && rn < (T)1e-12 * (T)pow2(B.Eh);
        K *tv = V + (size_t)m * ld;
        const K *tsrc = (tdst == tx) ? tx : tv;
        T tn = t0n;
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            const K *src = pass == 0 ? tsrc : tv;
            T v[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = 0;
            for (int d = tid; d < N; d += nt) {
                const K td = src[d];
#pragma unroll
                for (int i = 0; i < MMAX; ++i)
                    if (i < m) v[i] = dot(V[(size_t)i * ld + d], td, v[i]);
            }
            const T *tot = block_sums_many(v, m, red);
            T c[MMAX];
#pragma unroll
            for (int i = 0; i < MMAX; ++i) c[i] = i < m ? -tot[i] : (T)0;
            v1[0] = 0;
            for (int d = tid; d < N; d += nt) {
                K td = src[d];
#pragma unroll
                for (int i = 0; i < MMAX; ++i)
                    if (i < m) axpy(c[i], V[(size_t)i * ld + d], td);
                tv[d] = td;
                v1[0] = dot(td, td, v1[0]);
            }
            __syncthreads();  // (tot is read before the next sums)
            block_sums(v1, red);
            const T before = tn;
            tn = sqrt(v1[0]);
            if (tn >= (T)0.70710678 * before && !twice) break;
        }
        if (!(tn > (T)1e-12 * t0n) || !(tn > (T)0)) {
            // The correction lies in the current basis: nothing left to add.
            if (!steer && rn > (T)tol) o.status = MBE_STATUS_MAXITER;
            break;
        }
        scale((T)1 / tn, tv);
        __syncthreads();
        K *wv = W + (size_t)m * ld;
        sigma_block<T>(B, (const T *)tv, (T *)wv);
        ++o.nsig;
        T v[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = 0;
        for (int d = tid; d < N; d += nt) {
            K wd = wv[d];
            const K td = tv[d];
            if (anch) {
#pragma unroll
                for (int l = 0; l < VL; ++l) wd.e[l] = (wd.e[l] - shT * td.e[l]) - shT_lo * td.e[l];
                wv[d] = wd;
            }
#pragma unroll
            for (int i = 0; i < MMAX; ++i)
                if (i < m) v[i] = dot(V[(size_t)i * ld + d], wd, v[i]);
            v[MMAX] = dot(td, wd, v[MMAX]);
            if (anch) v[MMAX + 1] = dot(W[d], td, v[MMAX + 1]);  // x0.(A t) as t.r0
        }
        const T *tot = block_sums_many(v, MMAX + 2, red);
        if (tid <= m) {
            const double g = tid == m ? (double)tot[MMAX] : anch && tid == 0 ? (double)tot[MMAX + 1] : (double)tot[tid];
            G[tid * MMAX + m] = G[m * MMAX + tid] = g;
        }
        __syncthreads();
        ++m;
    }
    // the Ritz vector; anchored: its correction d, scaled so that x0 keeps coefficient 1
    __syncthreads();
    const T inv0 = anch ? (T)(1.0 / ys[0]) : (T)1;
    v1[0] = 0;
    for (int d = tid; d < N; d += nt) {
        K u;
#pragma unroll
        for (int l = 0; l < VL; ++l) u.e[l] = 0;
#pragma unroll 4
        for (int i = anch ? 1 : 0; i < m; ++i) axpy((T)ys[i] * inv0, V[(size_t)i * ld + d], u);
        x[d] = u;
        v1[0] = dot(u, u, v1[0]);
    }
    block_sums(v1, red);
    if (anch) o.dnorm = (double)sqrt(v1[0]);
    o.lambda = theta;
    o.rnorm = (double)rn;
    return o;
}

// Element h of the sector's start vector in the packed basis (see sector_guess).
__device__ inline double block_guess(int ia, int ib, int Ns, int h, int g, int sgn)
{
    const double z = GUESS_NOISE * guess_noise(ia * Ns + ib);
    if (ia == ib) return sgn > 0 ? z + (h == g ? 2.0 : 0.0) : 0.0;
    return 1.4142135623730951 * (z + (h == g ? 1.0 : 0.0));
}

template <typename T>
__device__ inline void write_guess(const Problem &pb, int g, T *x)
{
    int ia = 0, ib = 0;
    tri_advance(ia, ib, threadIdx.x, pb.Ns);
    for (int h = threadIdx.x; h < pb.N; h += blockDim.x) {
        x[h] = (T)block_guess(ia, ib, pb.Ns, h, g, pb.sector);
        tri_advance(ia, ib, blockDim.x, pb.Ns);
    }
}

// a2, a4: h_eff, V, Hs (Slater-Condon elements) and the packed diagonal, and for the tiled
// sigma the lists, the padded float32 V and the fixed-point V and Hs (over the float64 ones).
__device__ void block_setup(const BatchArgs &a, BlockProblem &B, const ClassInfo &ci)
{
    Problem &pb = B.pb;
    const int tid = threadIdx.x, nt = blockDim.x, n = pb.n, P = pb.P, norb = a.norb, Ns = pb.Ns, st = pb.HSS;
    double *red = (double *)(block_shared() + B.S.off_red);
    for (int e = tid; e < P; e += nt) {
        int p = 0;
        while ((p + 1) * (p + 2) / 2 <= e) ++p;
        ((short *)pb.pp)[2 * e] = (short)p;
        ((short *)pb.pp)[2 * e + 1] = (short)(e - p * (p + 1) / 2);
    }
    for (int e = tid; e < n * n; e += nt) {
        const int x = e / n, y = e - x * n, gp = pb.A[x], gq = pb.A[y];
        double v = a.F[gp * norb + gq];
        for (int c = 0; c < n; ++c) {
            const int gi = pb.A[c];
            if (a.occ[gi])
                v -= 2.0 * a.eri[eri_index(norb, gp, gq, gi, gi)] - a.eri[eri_index(norb, gp, gi, gi, gq)];
        }
        pb.h[e] = v;
    }
    __syncthreads();
    const int vs = v32_stride(B.form, P);
    double big = 0.0;
    bool bad = false;
    for (int e = tid; e < P * vs; e += nt) {
        const int x = e / vs, y = e - x * vs;
        double v = 0.0;
        if (y < P) {
            const int p = pb.pp[2 * x], q = pb.pp[2 * x + 1], r = pb.pp[2 * y], s = pb.pp[2 * y + 1];
            v = a.eri[eri_index(norb, pb.A[p], pb.A[q], pb.A[r], pb.A[s])];
            pb.V64[x * P + y] = v;
            big = fmax(big, fabs(v));
            bad = bad || !isfinite(v);
        }
        pb.V32[e] = (float)v;
    }
    if (B.form == SIGMA_LIST) {
        // off-diagonal replacements, the positive ones first, then their number
        uint32_t *list = (uint32_t *)(block_shared() + B.S.off_list);
        const int ro = pb.k * (n - pb.k), ld = list_stride(Ns);
        for (int I = tid; I < Ns; I += nt) {
            int at = 0, positive = 0;
            for (int neg = 0; neg < 2; ++neg) {
                for (int x = 0; x < pb.R; ++x) {
                    const int t = ci.table[I * pb.R + x];
                    if (entry_J(t) != I && entry_neg(t) == neg)
                        list[I * (ro + 1) + at++] = (uint32_t)(4 * entry_pair(t)) | (uint32_t)(4 * ld * entry_J(t)) << 12;
                }
                if (neg == 0) positive = at;
            }
            list[I * (ro + 1) + ro] = (uint32_t)positive;
        }
    }
    if (B.form == SIGMA_TILED) {
        uint16_t *list = (uint16_t *)(block_shared() + B.S.off_list);
        const int rs = pb.R | 1;
        for (int e = tid; e < Ns * pb.R; e += nt) {
            const int t = ci.table[e], I = e / pb.R;
            list[I * rs + e - I * pb.R] = (uint16_t)(entry_J(t) << 7 | (t & 127));
        }
    }
    __syncthreads();
    auto H = [&](int p, int q) { return pb.h[p * n + q]; };
    auto V = [&](int p, int q, int r, int s) { return pb.V64[pair_index(p, q) * P + pair_index(r, s)]; };
    double *hd = (double *)(block_shared() + B.S.off_hd);
    {
        int ia = 0, ib = 0;
        tri_advance(ia, ib, tid, Ns);
        for (int h = tid; h < pb.N; h += nt) {
            const double v = string_element(pb.str[ia], pb.str[ib], H, V);
            pb.Hs64[ia * st + ib] = pb.Hs64[ib * st + ia] = v;
            pb.Hs32[ia * st + ib] = pb.Hs32[ib * st + ia] = (float)v;
            if (ia != ib) big = fmax(big, fabs(v));
            bad = bad || !isfinite(v);
            tri_advance(ia, ib, nt, Ns);
        }
        for (int q = tid; q < Ns * (st - Ns); q += nt) {
            const int at = q / (st - Ns) * st + Ns + q % (st - Ns);
            pb.Hs64[at] = 0.0;
            pb.Hs32[at] = 0.f;
        }
    }
    B.bad = __syncthreads_or(bad);
    int top = 0;
    if (B.form == SIGMA_LIST)
        for (int e = tid; e < Ns * P; e += nt) {
            const int I = e / P, p = e - I * P;
            double u = 0.0;
            for (uint32_t m = pb.str[I]; m; m &= m - 1u) u += pb.V64[pair_index(__ffs((int)m) - 1, __ffs((int)m) - 1) * P + p];
            ((float *)B.U)[e] = (float)u;
        }
    {
        int ia = 0, ib = 0;
        tri_advance(ia, ib, tid, Ns);
        for (int h = tid; h < pb.N; h += nt) {
            double v = pb.Hs64[ia * st + ia] + pb.Hs64[ib * st + ib];
            for (uint32_t sa = pb.str[ia]; sa; sa &= sa - 1u) {
                const int p = __ffs((int)sa) - 1;
                for (uint32_t sb = pb.str[ib]; sb; sb &= sb - 1u) v += V(p, p, __ffs((int)sb) - 1, __ffs((int)sb) - 1);
            }
            v += pb.s2mu * __popc(pb.str[ia] & ~pb.str[ib]);
            pb.diag[h] = v;
            top = max(top, high_word(v));
            tri_advance(ia, ib, nt, Ns);
        }
        if (tid < (4 - pb.N % 4) % 4) pb.diag[pb.N + tid] = 1.0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_xor_sync(FULL, big, o));
    top = __reduce_max_sync(FULL, top);
    if ((tid & 31) == 0) {
        red[tid >> 5] = big;
        red[32 + (tid >> 5)] = (double)top;
    }
    __syncthreads();
    big = (tid & 31) < (nt >> 5) ? red[tid & 31] : 0.0;
    top = (tid & 31) < (nt >> 5) ? max((int)red[32 + (tid & 31)], high_word(big)) : 0;
    B.E = fixed_exponent(high_word(big));
    B.Eh = __reduce_max_sync(FULL, top) == 0 ? 0 : fixed_exponent(top);
    if (B.form == SIGMA_TILED) {
        const double scale = pow2(55 - B.E);
        int2 *Vf = (int2 *)pb.V64, *Hf = (int2 *)pb.Hs64;
        for (int e = tid; e < P * P; e += nt) Vf[e] = to_fixed(pb.V64[e], scale);
        for (int e = tid; e < Ns * st; e += nt) {
            const int I = e / st;
            const double v = pb.Hs64[e];
            if (e - I * st == I) hd[I] = v;
            Hf[e] = e - I * st == I ? make_int2(0, 0) : to_fixed(v, scale);
        }
    }
    __syncthreads();
}

// Spin-free density matrices of the packed unit vector x and their share of the gradients: the
// Gram matrix of the vectors E_rs c (see sector_rdm), 32 elements of all of them in shared
// memory at a time, the entries of the Gram matrix in registers.
__device__ __noinline__ void block_rdm(const BatchArgs &a, const BlockProblem &B, const double *x, double w)
{
    constexpr int GE = 11;  // entries per thread: (n^2 + 1)(n^2 + 2) / 2 of them up to 10 orbitals
    const Problem &pb = B.pb;
    const int tid = threadIdx.x, nt = blockDim.x, n = pb.n, n2 = n * n, Ns = pb.Ns, lane = tid & 31;
    const bool two = a.grad_eri != nullptr;
    const int first = two ? 0 : n2 * (n2 + 1) / 2, ng = n2 * (n2 + 1) / 2 + n2;  // (without c.c)
    double *D = (double *)(block_shared() + B.S.off_c), *g1 = (double *)(block_shared() + B.S.off_g1), *c = B.full;
    expand_full<double>(pb, x, c, Ns);
    double gram[GE];
    int uv[GE];
#pragma unroll
    for (int i = 0; i < GE; ++i) {
        const int q = first + tid + nt * i;
        int v = (int)((sqrtf(8.f * q + 1.f) - 1.f) * 0.5f);
        while ((v + 1) * (v + 2) / 2 <= q) ++v;
        while (v * (v + 1) / 2 > q) --v;
        uv[i] = q < ng ? v << 8 | (q - v * (v + 1) / 2) : -1;
        gram[i] = 0.0;
    }
    __syncthreads();
    const uint32_t full = (1u << n) - 1u;
    int ia = 0, ib = 0;
    tri_advance(ia, ib, lane, Ns);
    // <I| E_rs = s <J| with |J> = s E_sr |I>: r occupied in I, s empty or r itself
    auto entry = [&](int I, uint32_t st, int r, int s) {
        const int at = __popc(st & ((1u << r) - 1u)) * (n - pb.k + 1) + __popc(~st & full & ((1u << s) - 1u)) + (r < s ? 1 : 0);
        return pb.tab[I * pb.RS + at];
    };
    for (int h0 = 0; h0 < pb.N; h0 += 32) {
        const bool on = h0 + lane < pb.N;
        const int i = on ? ia : 0, j = on ? ib : 0;
        const double wt = !on ? 0.0 : i == j ? 1.0 : 1.4142135623730951;
        const uint32_t sa = pb.str[i], sb = pb.str[j];
        for (int rs = tid >> 5; rs <= n2; rs += nt >> 5) {
            double v = 0.0;
            if (rs == n2) {
                v = c[i * Ns + j];
            } else {
                const int r = rs / n, s = rs - r * n;
                if ((sa >> r & 1u) && (r == s || !(sa >> s & 1u))) {
                    const int q = entry(i, sa, r, s);
                    v = flip_if(c[entry_J(q) * Ns + j], entry_neg(q));
                }
                if ((sb >> r & 1u) && (r == s || !(sb >> s & 1u))) {
                    const int q = entry(j, sb, r, s);
                    v += flip_if(c[i * Ns + entry_J(q)], entry_neg(q));
                }
            }
            D[rs * 33 + lane] = wt * v;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < GE; ++q)
            if (uv[q] >= 0) {
                const double *du = D + (uv[q] & 255) * 33, *dv = D + (uv[q] >> 8) * 33;
                double s = gram[q];
#pragma unroll 8
                for (int h = 0; h < 32; ++h) s = fma(du[h], dv[h], s);
                gram[q] = s;
            }
        __syncthreads();
        tri_advance(ia, ib, 32, Ns);
    }
#pragma unroll
    for (int q = 0; q < GE; ++q)
        if (uv[q] >= 0 && uv[q] >> 8 == n2) g1[uv[q] & 255] = gram[q];
    __syncthreads();
    for (int e = tid; e < n2; e += nt) {
        const int p = e / n, q = e - p * n;
        rdm_one_body(a, pb.A, n, p, q, w * (g1[e] - ((p == q && a.occ[pb.A[p]]) ? 2.0 : 0.0)));
    }
    if (two)
#pragma unroll
        for (int q = 0; q < GE; ++q)
            if (uv[q] >= 0 && uv[q] >> 8 != n2) rdm_two_body(a, pb.A, n, uv[q] & 255, uv[q] >> 8, gram[q], g1, w);
    __syncthreads();
}

__global__ void __launch_bounds__(BLOCK_THREADS, 1) k_casci_block(BatchArgs a, int bucket)
{
    char *smem = block_shared();
    const int n = a.n, P = n * (n + 1) / 2, tid = threadIdx.x, nt = blockDim.x;
    __shared__ unsigned long long s_pos;
    char *slot = a.scratch + (size_t)blockIdx.x * a.slot_bytes;
    const int64_t begin = a.bucket_off[bucket];
    const int64_t cnt = a.bucket_off[bucket + 1] - begin;
    int *A = (int *)smem;
    for (;;) {
        if (tid == 0) s_pos = atomicAdd(&a.counters[bucket], 1ULL);
        __syncthreads();
        const unsigned long long pos = s_pos;
        __syncthreads();
        if ((int64_t)pos >= cnt) break;
        const int64_t t = a.perm[begin + (int64_t)pos];
        if (tid == 0) build_A(a, t, A);
        __syncthreads();
        int k = 0;
        uint32_t mphi = 0;
        for (int i = 0; i < n; ++i)
            if (a.occ[A[i]]) {
                ++k;
                mphi |= 1u << i;
            }
        const ClassInfo ci = a.cls[k];
        const BlockSlot L = block_slot(n, ci.ns);
        BlockProblem B;
        B.form = a.tiled ? sigma_form(n, ci.ns) : SIGMA_GLOBAL;
        B.S = block_mem(n, B.form, ci.ns, ci.r, a.rdm);
        B.U = (const float *)(slot + L.off_U);
        B.E = B.Eh = 0;
        B.full = (double *)(slot + L.off_full);
        const BlockMem &S = B.S;
        Problem &pb = B.pb;
        pb.n = n;
        pb.P = P;
        pb.k = k;
        pb.Ns = ci.ns;
        pb.N = ci.ns * (ci.ns + 1) / 2;
        pb.R = ci.r;
        pb.RS = ci.r;
        pb.HSS = hs_stride(ci.ns);
        pb.str = ci.strings;
        pb.tab = ci.table;
        pb.A = A;
        pb.pp = (const short *)(smem + S.off_pp);
        pb.h = (double *)(smem + S.off_h);
        pb.hp = nullptr;
        pb.V64 = (double *)(B.form == SIGMA_LIST ? slot + L.off_V64 : smem + S.off_V64);
        pb.V32 = (float *)(smem + S.off_V32);
        pb.Hs64 = (double *)(slot + L.off_Hs64);
        pb.Hs32 = (float *)(slot + L.off_Hs32);
        pb.diag = (double *)(slot + L.off_diag);
        pb.c = nullptr;
        const bool mixed = a.precision == MBE_PREC_MIXED;
        pb.s2mu = a.s2mu;
        block_setup(a, B, ci);
        const int iphi = string_rank(mphi);
        const double ephi = pb.diag[iphi * pb.Ns - iphi * (iphi - 1) / 2];
        if (pb.N == 1) {
            if (tid == 0) store_result(a, t, pb.diag[0] - ephi - a.e_ref_corr, MBE_STATUS_OK, 0, 0);
            __syncthreads();
            continue;
        }
        double *red = (double *)(smem + S.off_red);
        // start vectors: the lowest diagonal element (ties -> lowest index), and for
        // the P = -1 sector the lowest one with Ia != Ib
        double best = 1e300, best_o = 1e300;
        int bi = 0x7fffffff, bj = 0x7fffffff;
        {
            int ia = 0, ib = 0;
            tri_advance(ia, ib, tid, pb.Ns);
            for (int d = tid; d < pb.N; d += nt) {
                const double v = pb.diag[d];
                if (v < best) {
                    best = v;
                    bi = d;
                }
                if (ia != ib && v < best_o) {
                    best_o = v;
                    bj = d;
                }
                tri_advance(ia, ib, nt, pb.Ns);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            double ov = __shfl_xor_sync(FULL, best, o);
            int oi = __shfl_xor_sync(FULL, bi, o);
            if (ov < best || (ov == best && oi < bi)) {
                best = ov;
                bi = oi;
            }
            ov = __shfl_xor_sync(FULL, best_o, o);
            oi = __shfl_xor_sync(FULL, bj, o);
            if (ov < best_o || (ov == best_o && oi < bj)) {
                best_o = ov;
                bj = oi;
            }
        }
        __syncthreads();
        if ((tid & 31) == 0) {
            red[tid >> 5] = best;
            red[32 + (tid >> 5)] = best_o;
            ((int *)(red + 64))[tid >> 5] = bi;
            ((int *)(red + 64))[32 + (tid >> 5)] = bj;
        }
        __syncthreads();
        best = red[0];
        best_o = red[32];
        bi = ((int *)(red + 64))[0];
        bj = ((int *)(red + 64))[32];
        for (int w = 1; w < (nt >> 5); ++w) {
            double ov = red[w];
            int oi = ((int *)(red + 64))[w];
            if (ov < best || (ov == best && oi < bi)) {
                best = ov;
                bi = oi;
            }
            ov = red[32 + w];
            oi = ((int *)(red + 64))[32 + w];
            if (ov < best_o || (ov == best_o && oi < bj)) {
                best_o = ov;
                bj = oi;
            }
        }
        // The padding of the vectors (see Pack) is zero, and every operation on packs keeps it
        // so; the float32 one is also overwritten by float64 vectors in the same place.
        auto zero_padding = [&](bool f32) {
            const int pad = f32 ? (4 - pb.N % 4) % 4 : pb.N % 2;
            for (int q = tid; q < (2 * MMAX + 2) * pad; q += nt) {
                const int v = q / pad, l = q - v * pad;
                char *base = slot + (v < MMAX ? L.off_V + v * L.vec : v < 2 * MMAX ? L.off_W + (v - MMAX) * L.vec
                                                              : v == 2 * MMAX ? L.off_x : L.off_t);
                if (f32) ((float *)base)[pb.N + l] = 0.f; else ((double *)base)[pb.N + l] = 0.0;
            }
        };
        zero_padding(false);
        __syncthreads();
        double *x64 = (double *)(slot + L.off_x), *x2 = (double *)(slot + L.off_x2);
        float *x32 = (float *)(slot + L.off_x);
        double *V64 = (double *)(slot + L.off_V), *W64 = (double *)(slot + L.off_W), *t64 = (double *)(slot + L.off_t);
        float *V32 = (float *)V64, *W32 = (float *)W64, *t32 = (float *)t64;
        double lam = 0.0;
        int status = MBE_STATUS_OK, n64 = 0, n32 = 0, won = 1;
        bool degen = false;
        // one copy of the sector's Davidson: two inlined copies, both hot on an SM,
        // overflow the instruction cache and slow every phase of every warp
#pragma unroll 1
        for (int sector = 0; sector < 2; ++sector) {
            if (sector == 1 && (pb.Ns < 2 || status != MBE_STATUS_OK || a.even_only)) break;
            const int g = sector == 0 ? bi : bj;
            if (sector == 1 && a.rdm)
                for (int d = tid; d < pb.N; d += nt) x2[d] = x64[d];
            __syncthreads();  // (the float32 padding zeroed below lies inside x64)
            pb.sector = sector == 0 ? 1 : -1;
            if (mixed) zero_padding(true);
            __syncthreads();
            bool lose = false, refined = false;
            if (mixed) {
                write_guess<float>(pb, g, x32);
                __syncthreads();
                // the second sector: a pass to SECTOR_TOL, then one to tol_switch if undecided
                PhaseOut o32;
                for (int pass = 0; pass < 1 + sector; ++pass) {
                    const double tl = (sector == 0 || pass == 1) ? a.tol_switch : SECTOR_TOL;
                    o32 = davidson_block<float>(B, V32, W32, L.vec / 4, x32, t32, tl, 0, a.max_iter, BLOCK_STALL, 0.0,
                                                false, a.block_basis);
                    n32 += o32.nsig;
                    if (sector == 1)
                        lose = o32.status == MBE_STATUS_NONFINITE ||
                               sector_loses(o32.lambda, o32.rnorm, lam, a.tol_switch);
                    if (lose || o32.status == MBE_STATUS_NONFINITE) break;
                }
                const bool finite = o32.status != MBE_STATUS_NONFINITE;
                double *x0 = (double *)(slot + L.off_x0);
                if (!lose && finite) {
                    // Anchored refinement (struct Anchor): a float64 sigma of the float64
                    // anchor x0, then the float32 Davidson on H - theta0 with x0 as its
                    // first basis vector; x0 <- (x0 + d) / |x0 + d| after each pass, re-anchoring
                    // while the residual stays above tol.
                    for (int d = tid; d < pb.N; d += nt) x0[d] = (double)x32[d];
                    __syncthreads();
                    bool done = false, bad = false;
                    double lam_s = 0.0;
                    for (int anc = 0; anc < BLOCK_ANCHORS && !done && !bad; ++anc) {
                        // (the image over the basis, of which nothing is kept between anchors)
                        double *s0 = W64 + (MMAX / 2) * (L.vec / 8);
                        sigma_block<double>(B, x0, s0);
                        ++n64;
                        double q[2] = {0.0, 0.0};
                        for (int d = tid; d < pb.N; d += nt) {
                            q[0] += x0[d] * s0[d];
                            q[1] += x0[d] * x0[d];
                        }
                        block_sums(q, red);
                        const double th = q[0] / q[1], inv = 1.0 / sqrt(q[1]);
                        for (int d = tid; d < pb.N; d += nt) {
                            V32[d] = (float)(x0[d] * inv);
                            W32[d] = (float)((s0[d] - th * x0[d]) * inv);
                        }
                        __syncthreads();
                        zero_padding(true);  // (s0 lay over one W)
                        __syncthreads();
                        PhaseOut o = davidson_block<float>(B, V32, W32, L.vec / 4, x32, t32, a.tol, a.min_fp64, a.max_iter,
                                                           BLOCK_ANCHOR_STALL, th, true, a.block_basis);
                        n32 += o.nsig;
                        lam_s = th + o.lambda;
                        bad = o.status == MBE_STATUS_NONFINITE;
                        done = !bad && o.rnorm <= a.tol && o.dnorm <= MIX_DMAX;
                        // x0 <- x0 + d as a unit vector: |d| may be anything until a pass is accepted,
                        // and the fixed-point sigma holds elements of at most 1
                        if (!bad) {
                            double nn[1] = {0.0};
                            for (int d = tid; d < pb.N; d += nt) {
                                const double v = x0[d] * inv + (double)x32[d];
                                x0[d] = v;
                                nn[0] += v * v;
                            }
                            block_sums(nn, red);
                            const double unit = 1.0 / sqrt(nn[0]);
                            for (int d = tid; d < pb.N; d += nt) x0[d] *= unit;
                        }
                        __syncthreads();
                    }
                    // the refined vector (or the start of the float64 fallback) as x64
                    if (bad)
                        write_guess<double>(pb, g, x64);
                    else
                        for (int d = tid; d < pb.N; d += nt) x64[d] = x0[d];
                    __syncthreads();
                    if (done) {
                        refined = true;
                        if (sector == 1) degen = status == MBE_STATUS_OK && fabs(lam_s - lam) <= DEGEN_TOL;
                        if (sector == 0 || lam_s < lam) {
                            lam = lam_s;
                            status = MBE_STATUS_OK;
                            won = pb.sector;
                        } else {
                            lose = true;
                        }
                    }
                } else if (finite) {
                    for (int d = tid; d < pb.N; d += nt) x0[d] = (double)x32[d];
                    __syncthreads();
                    for (int d = tid; d < pb.N; d += nt) x64[d] = x0[d];
                    __syncthreads();
                } else {
                    write_guess<double>(pb, g, x64);
                    __syncthreads();
                }
            } else {
                write_guess<double>(pb, g, x64);
                __syncthreads();
                if (sector == 1) {
                    PhaseOut o1 = davidson_block<double>(B, V64, W64, L.vec / 8, x64, t64, SECTOR_TOL, 0, a.max_iter,
                                                         BLOCK_STALL, 0.0, false, a.block_basis);
                    n64 += o1.nsig;
                    lose = o1.status == MBE_STATUS_NONFINITE || sector_loses(o1.lambda, o1.rnorm, lam, 0.0);
                }
            }
            if (!lose && !refined) {
                PhaseOut o64 = davidson_block<double>(B, V64, W64, L.vec / 8, x64, t64, a.tol, mixed ? a.min_fp64 : 0,
                                                      a.max_iter, 0, 0.0, false, a.block_basis);
                n64 += o64.nsig;
                if (sector == 0) {
                    lam = o64.lambda;
                    status = o64.status;
                } else {
                    degen = o64.status == MBE_STATUS_OK && status == MBE_STATUS_OK && fabs(o64.lambda - lam) <= DEGEN_TOL;
                    lose = o64.status == MBE_STATUS_NONFINITE || !(o64.lambda < lam);
                    if (!lose) {
                        lam = o64.lambda;
                        status = o64.status;
                        won = -1;
                    }
                }
            }
            if (lose && a.rdm) {
                __syncthreads();
                for (int d = tid; d < pb.N; d += nt) x64[d] = x2[d];
            }
            __syncthreads();
        }
        if (tid == 0) {
            double e = status == MBE_STATUS_NONFINITE ? __longlong_as_double(0x7ff8000000000000LL)
                                                      : lam - ephi - a.e_ref_corr;
            store_result(a, t, e, with_degeneracy(status, degen), n64, n32);
        }
        __syncthreads();
        if (a.rdm) {
            pb.sector = won;
            block_rdm(a, B, x64, a.weights ? a.weights[t] : 1.0);
        }
    }
}

// small_eig_block on a Rayleigh matrix in global memory (the large-CAS solver's).  col: its new last
// column, put in first (m values, or NULL).  basis: the eigenbasis and eigenvalues of the
// last call, read if warm ([MMAX + 1][MMAX], then their unit's exponent), replaced.
__global__ void __launch_bounds__(416) k_small_eig(double *Gd, int m, const double *col, int warm, BlockMem S, float *basis, double *ys,
                                                   double *y2s, double *misc)
{
    const int tid = threadIdx.x;
    double *G = (double *)(block_shared() + S.off_G);
    float *E = (float *)(block_shared() + S.off_J) + MMAX * MMAX, *ev = (float *)(block_shared() + S.off_ev);
    if (col && tid < m) Gd[tid * MMAX + m - 1] = Gd[(m - 1) * MMAX + tid] = col[tid];
    __syncthreads();
    if (tid < MMAX * MMAX) {
        G[tid] = Gd[tid];
        if (warm) E[tid] = basis[tid];
    }
    if (warm && tid < MMAX) ev[tid] = basis[MMAX * MMAX + tid];
    double *unit = (double *)(block_shared() + S.off_misc) + 1;
    if (warm && tid == 0) *unit = (double)basis[(MMAX + 1) * MMAX];
    __syncthreads();
    small_eig_block<true>(S, m, warm);
    if (tid < MMAX * MMAX) basis[tid] = E[tid];
    if (tid < MMAX) basis[MMAX * MMAX + tid] = ev[tid];
    if (tid == 0) basis[(MMAX + 1) * MMAX] = (float)*unit;
    if (tid < m) {
        ys[tid] = ((double *)(block_shared() + S.off_y))[tid];
        y2s[tid] = ((double *)(block_shared() + S.off_yp))[tid];
    }
    if (tid == 0) misc[0] = *(double *)(block_shared() + S.off_misc);
}

int launch_small_eig(cudaStream_t st, double *Gd, int m, const double *col, int warm, float *basis, double *ys, double *y2s,
                     double *misc)
{
    const BlockMem S = block_mem(2, SIGMA_GLOBAL, 1, 1, 0);
    k_small_eig<<<1, 416, S.bytes, st>>>(Gd, m, col, warm, S, basis, ys, y2s, misc);
    MBE_CU(cudaGetLastError());
    return MBE_OK;
}

// Shared memory and slot size of a bucket's block launch (the classes `in`); a.tiled is cleared
// when the shared-memory forms of sigma do not fit.
int block_grid(mbe_ctx *ctx, BatchArgs &a, const bool (&in)[MBE_MAX_STRING_ORB + 1], int rdm, int *grid, size_t *smem,
               size_t *slot)
{
    for (a.tiled = 1; a.tiled >= 0; --a.tiled) {
        *smem = *slot = 0;
        for (int k = 0; k <= a.n; ++k)
            if (in[k]) {
                const int form = a.tiled ? sigma_form(a.n, a.cls[k].ns) : SIGMA_GLOBAL;
                *smem = std::max(*smem, (size_t)block_mem(a.n, form, a.cls[k].ns, a.cls[k].r, rdm).bytes);
                *slot = std::max(*slot, block_slot(a.n, a.cls[k].ns).bytes);
            }
        if (*smem <= ctx->smem_optin - 1024) break;  // (some static shared memory besides)
    }
    MBE_CHECK(a.tiled >= 0, MBE_EUNSUPPORTED, "casci_batch: block solver needs %zu B shared memory", *smem);
    MBE_CU(allow_smem(k_casci_block, ctx->smem_optin));
    *grid = (int)std::min<int64_t>(ctx->sm_count, a.n_tuples);
    return MBE_OK;
}

int launch_block(mbe_ctx *ctx, const BatchArgs &a, int b, int grid, size_t smem)
{
    k_casci_block<<<grid, BLOCK_THREADS, smem, ctx->stream>>>(a, b);
    MBE_CU(cudaGetLastError());
    return MBE_OK;
}

}  // namespace mbe
