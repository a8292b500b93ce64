// ------------------------------------------------------------------ single large active space
//
// One CASCI over a large active space (up to 16 orbitals, 165.6M determinants
// at (16e,16o)), spread over the whole GPU:
//   * set-up: h_eff, packed V (one block); the one-spin Hamiltonian Hs by the Slater-Condon
//     rules over the grid as a dense Ns x Ns matrix, then compressed to CSR (each row holds
//     the strings connected by at most a double replacement);
//   * sigma = (Hs x 1) c + (1 x Hs) c + opposite-spin term.  In float64 up to 14 orbitals all of
//     it is products of exact digits on the tensor cores (large_digits.cu); above, with few strings and
//     for operands that digits do not suit, the direct
//     double loop over the alpha and beta replacement lists (one thread per determinant, V in
//     shared memory) and row-streamed sparse products C' = Hs C, the beta one applied to the
//     transposed coefficient matrix and added back transposed.  In float32 the opposite-spin
//     term is, per alpha string, a dense product on the tensor cores followed by a scatter
//     (large_tc.cu), and the sparse products take slabs of c from shared memory;
//   * inside the Davidson every vector lies in one spin-flip sector,
//     c[Ia][Ib] = sgn c[Ib][Ia], and is kept packed (LargeDav); the beta same-spin term is
//     sgn times the transpose of the alpha one (one sparse product and a transposing add);
//   * Davidson: the tuple solvers' algorithm (MLARGE-vector basis, thick restart
//     on the two lowest Ritz vectors, float32 phase then float64 phase) with its
//     vector algebra in grid-wide kernels, the projected eigenproblem in one
//     block, and the host reading back two norms per iteration to decide convergence.

#include "casci_sector.cuh"
#include "large_digits.cuh"

using namespace mbe;


namespace mbe {

constexpr int MLARGE = 12;      // Davidson basis of the large solver (<= MMAX)
constexpr int LARGE_STALL = 20; // iterations without a 10% residual drop that end the sector-deciding pass
constexpr int LARGE_ANCHORS = 8;         // anchored refinements before the float64 fallback
constexpr int LARGE_ANCHOR_STALL = 30;   // iterations without a 10% drop before re-anchoring
constexpr int LRED = MLARGE + 2;  // values per grid reduction
constexpr int LARGE_THREADS = 256;
constexpr int SIGMA_THREADS = 512;

struct LargeCas {
    int n, P, k, Ns, R;
    int64_t N;
    const uint32_t *str;
    const int32_t *tab;
    double *V;      // [P*P]
    float *V32;     // [P*P]
    double *h;      // [P] h_eff
    short *pp;      // [2P]
    double *Hd;     // dense Hs [Ns*Ns] (set-up only)
    int64_t *roff;  // CSR [Ns+1]
    int32_t *col;   // CSR [nnz]
    double *val;    // CSR [nnz]
    float *val32;   // CSR [nnz]
    double *diag;   // [N]
    int64_t nnz;
    const int32_t *tabT;  // beta lists transposed: tabT[y * Ns + J] = tab[J * R + y]
};


struct LargeSetupArgs {
    int norb;
    const double *eri;
    const double *F;
    const uint8_t *occ;
    int A[MBE_MAX_STRING_ORB];
};

// One block: pair table, h_eff, V over packed pairs (float64 and float32).
__global__ void __launch_bounds__(CTA_THREADS) k_large_setup(LargeSetupArgs a, LargeCas L)
{
    __shared__ int A[MBE_MAX_STRING_ORB];
    __shared__ double h[MBE_MAX_STRING_ORB * MBE_MAX_STRING_ORB];
    const int n = L.n, P = L.P, norb = a.norb;
    if (threadIdx.x < n) A[threadIdx.x] = a.A[threadIdx.x];
    for (int e = threadIdx.x; e < P; e += blockDim.x) {
        int p = 0;
        while ((p + 1) * (p + 2) / 2 <= e) ++p;
        L.pp[2 * e] = (short)p;
        L.pp[2 * e + 1] = (short)(e - p * (p + 1) / 2);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        int x = e / n, y = e - x * n;
        int gp = A[x], gq = A[y];
        double v = a.F[gp * norb + gq];
        for (int c = 0; c < n; ++c) {
            int gi = A[c];
            if (a.occ[gi])
                v -= 2.0 * a.eri[eri_index(norb, gp, gq, gi, gi)] - a.eri[eri_index(norb, gp, gi, gi, gq)];
        }
        h[e] = v;
    }
    for (int e = threadIdx.x; e < P * P; e += blockDim.x) {
        int x = e / P, y = e - x * P;
        int p = L.pp[2 * x], q = L.pp[2 * x + 1], r = L.pp[2 * y], s = L.pp[2 * y + 1];
        double v = a.eri[eri_index(norb, A[p], A[q], A[r], A[s])];
        L.V[e] = v;
        L.V32[e] = (float)v;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < P; e += blockDim.x) L.h[e] = h[L.pp[2 * e] * n + L.pp[2 * e + 1]];
}

// Dense Hs by the Slater-Condon rules, one element per thread (a row per block), V in shared
// memory: 25 us at 12 orbitals.  (One thread per column multiplying out sum E_pq E_rs took
// 0.8 ms at 12 orbitals and 1.4 ms at 14: 924 and 3,432 threads with R^2 dependent updates.)
__global__ void __launch_bounds__(256) k_large_hs(LargeCas L)
{
    extern __shared__ __align__(16) char smem[];
    double *Vs = (double *)smem, *hs = Vs + L.P * L.P;
    for (int e = threadIdx.x; e < L.P * L.P; e += blockDim.x) Vs[e] = L.V[e];
    for (int e = threadIdx.x; e < L.P; e += blockDim.x) hs[e] = L.h[e];
    __syncthreads();
    auto H = [&](int p, int q) { return hs[pair_index(p, q)]; };
    auto V = [&](int p, int q, int r, int s) { return Vs[pair_index(p, q) * L.P + pair_index(r, s)]; };
    for (int I = blockIdx.x; I < L.Ns; I += gridDim.x) {
        const uint32_t sI = L.str[I];
        for (int J = threadIdx.x; J < L.Ns; J += blockDim.x) {
            const uint32_t sJ = L.str[J];
            double v = 0.0;
            if (__popc(sI ^ sJ) <= 4) v = string_element(sI, sJ, H, V);
            L.Hd[(size_t)I * L.Ns + J] = v;
        }
    }
}

// Non-zeros per row (one warp per row), for the CSR offsets.
__global__ void k_large_hs_count(LargeCas L, int32_t *cnt)
{
    int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (row >= L.Ns) return;
    const double *hr = L.Hd + (size_t)row * L.Ns;
    int c = 0;
    for (int base = 0; base < L.Ns; base += 32) {
        int j = base + lane;
        bool nz = j < L.Ns && hr[j] != 0.0;
        c += __popc(__ballot_sync(FULL, nz));
    }
    if (lane == 0) cnt[row] = c;
}

__global__ void k_large_hs_fill(LargeCas L, const int64_t *off)
{
    int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (row >= L.Ns) return;
    const double *hr = L.Hd + (size_t)row * L.Ns;
    int64_t pos = off[row];
    if (lane == 0) L.roff[row] = pos;
    if (row == L.Ns - 1 && lane == 0) L.roff[L.Ns] = off[L.Ns];
    for (int base = 0; base < L.Ns; base += 32) {
        int j = base + lane;
        double v = (j < L.Ns) ? hr[j] : 0.0;
        unsigned m = __ballot_sync(FULL, v != 0.0);
        if (v != 0.0) {
            int64_t at = pos + __popc(m & ((1u << lane) - 1u));
            L.col[at] = j;
            L.val[at] = v;
            L.val32[at] = (float)v;
        }
        pos += __popc(m);
    }
}

// Diagonal of H, a row per block: V's part of a string is the sum of two table entries, one for
// its lower and one for its upper 8 orbitals (the double loop over both strings' orbitals took
// 1.1 ms at 14 orbitals).
__global__ void __launch_bounds__(256) k_large_diag(LargeCas L)
{
    __shared__ double u[16], part[2][256];
    const int Ns = L.Ns, P = L.P, tid = threadIdx.x;
    for (int ia = blockIdx.x; ia < Ns; ia += gridDim.x) {
        __syncthreads();
        if (tid < 16) {
            double v = 0.0;
            if (tid < L.n)
                for (uint32_t s = L.str[ia]; s; s &= s - 1)
                    v += L.V[pair_index(__ffs((int)s) - 1, __ffs((int)s) - 1) * P + pair_index(tid, tid)];
            u[tid] = v;
        }
        __syncthreads();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            double v = 0.0;
            for (uint32_t s = tid; s; s &= s - 1) v += u[8 * h + __ffs((int)s) - 1];
            part[h][tid] = v;
        }
        __syncthreads();
        const double ha = L.Hd[(size_t)ia * Ns + ia];
        for (int ib = tid; ib < Ns; ib += blockDim.x) {
            const uint32_t s = L.str[ib];
            L.diag[(size_t)ia * Ns + ib] = ha + L.Hd[(size_t)ib * Ns + ib] + (part[0][s & 255] + part[1][s >> 8]);
        }
    }
}

// Opposite-spin part of sigma in float64, one thread per determinant:
//     sigma[Ia][Ib] = sum_{x in list(Ia)} s_x sum_{y in list(Ib)} s_y V[p_x][p_y] c[J_x][J_y]
// (written, not accumulated). The beta lists are read through the transposed
// table, so a warp's 32 consecutive Ib load 32 consecutive words.
// SECTOR: c lies in the spin-flip sector sgn (c[Ia][Ib] = sgn c[Ib][Ia]), so only
// the elements with Ia <= Ib are computed, walking the upper triangle row by
// row, and each is mirrored, sigma[Ib][Ia] = sgn sigma[Ia][Ib] (the diagonal of
// the odd sector vanishes).  Otherwise every element, in row-major order.
template <bool SECTOR>
__global__ void __launch_bounds__(SIGMA_THREADS) k_large_ab64(LargeCas L, const double *__restrict__ c,
                                                               double *__restrict__ sigma, int sgn,
                                                               const unsigned long long *digits)
{
    extern __shared__ __align__(16) char smem[];
    if (digits && digits_usable(digits)) return;
    double *Vs = (double *)smem;
    const int P = L.P, Ns = L.Ns, R = L.R;
    for (int e = threadIdx.x; e < P * P; e += blockDim.x) Vs[e] = L.V[e];
    __syncthreads();
    const int64_t count = SECTOR ? (int64_t)Ns * (Ns + 1) / 2 : L.N;
    for (int64_t h = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; h < count; h += (int64_t)gridDim.x * blockDim.x) {
        int ia, ib;
        if (SECTOR) {
            // row ia of the upper triangle starts at ia Ns - ia (ia - 1) / 2
            const double b2 = 2.0 * Ns + 1.0;
            ia = (int)((b2 - sqrt(b2 * b2 - 8.0 * (double)h)) * 0.5);
            auto start = [&](int64_t r) { return r * Ns - r * (r - 1) / 2; };
            while (ia > 0 && start(ia) > h) --ia;
            while (ia + 1 < Ns && start(ia + 1) <= h) ++ia;
            ib = ia + (int)(h - start(ia));
            if (sgn < 0 && ia == ib) {
                sigma[(int64_t)ia * Ns + ib] = 0.0;
                continue;
            }
        } else {
            ia = (int)(h / Ns);
            ib = (int)(h - (int64_t)ia * Ns);
        }
        double acc0 = 0.0, acc1 = 0.0;
        const int32_t *ta = L.tab + (size_t)ia * R;
        const int32_t *tb = L.tabT + ib;
        for (int x = 0; x < R; ++x) {
            const int ea = ta[x];
            const double *vrow = Vs + entry_pair(ea) * P;
            const double *cr = c + (int64_t)entry_J(ea) * Ns;
            double s0 = 0.0, s1 = 0.0;
            int y = 0;
            for (; y + 1 < R; y += 2) {
                const int e0 = tb[(size_t)y * Ns], e1 = tb[(size_t)(y + 1) * Ns];
                s0 = fma(flip_if(vrow[entry_pair(e0)], entry_neg(e0)), cr[entry_J(e0)], s0);
                s1 = fma(flip_if(vrow[entry_pair(e1)], entry_neg(e1)), cr[entry_J(e1)], s1);
            }
            if (y < R) {
                const int e0 = tb[(size_t)y * Ns];
                s0 = fma(flip_if(vrow[entry_pair(e0)], entry_neg(e0)), cr[entry_J(e0)], s0);
            }
            const double s = s0 + s1;
            if (x & 1) acc1 += flip_if(s, entry_neg(ea)); else acc0 += flip_if(s, entry_neg(ea));
        }
        const double v = acc0 + acc1;
        sigma[(int64_t)ia * Ns + ib] = v;
        if (SECTOR && ia < ib) sigma[(int64_t)ib * Ns + ia] = sgn > 0 ? v : -v;
    }
}

// Same-spin part, row-streamed: out[I][K] += sum_e val[e] X[col[e]][K] over the
// CSR row I of Hs, for a block of SS_ROWS rows and a tile of SS_TK columns per
// work item. Column tiles are the outer work index, so the CTAs in flight share
// one slab of X in L2. With TRANS the result is added at out[K][I] (X is the
// transposed coefficient matrix and the product is C Hs^T).
constexpr int SS_ROWS = 32, SS_TK = 256, SS_THREADS = 256;

// STORE: out[I][K] = (Hs X)[I][K] instead of adding it (TRANS false only).
template <typename T, bool TRANS, bool STORE = false>
__global__ void __launch_bounds__(SS_THREADS) k_large_ss(LargeCas L, const T *__restrict__ X,
                                                          double *__restrict__ sigma,
                                                          const unsigned long long *digits)
{
    extern __shared__ __align__(16) char smem[];
    if (digits && digits_usable(digits)) return;
    T *out = (T *)smem;  // [SS_ROWS][SS_TK + 1]
    const int Ns = L.Ns, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const T *val = sizeof(T) == 8 ? (const T *)L.val : (const T *)L.val32;
    const int nrb = (Ns + SS_ROWS - 1) / SS_ROWS, nct = (Ns + SS_TK - 1) / SS_TK;
    for (int item = blockIdx.x; item < nrb * nct; item += gridDim.x) {
        const int ct = item / nrb, rb = item - ct * nrb;
        const int I0 = rb * SS_ROWS, K0 = ct * SS_TK;
        for (int r = w; r < SS_ROWS; r += SS_THREADS / 32) {
            const int I = I0 + r;
            T acc[SS_TK / 32];
#pragma unroll
            for (int j = 0; j < SS_TK / 32; ++j) acc[j] = 0;
            if (I < Ns) {
                const int64_t e1 = L.roff[I + 1];
                for (int64_t e = L.roff[I]; e < e1; ++e) {
                    const T v = val[e];
                    const T *xr = X + (size_t)L.col[e] * Ns + K0 + lane;
#pragma unroll
                    for (int j = 0; j < SS_TK / 32; ++j)
                        if (K0 + lane + 32 * j < Ns) acc[j] = fma(v, xr[32 * j], acc[j]);
                }
            }
#pragma unroll
            for (int j = 0; j < SS_TK / 32; ++j) out[r * (SS_TK + 1) + lane + 32 * j] = acc[j];
        }
        __syncthreads();
        for (int i = threadIdx.x; i < SS_ROWS * SS_TK; i += SS_THREADS) {
            const int r = TRANS ? (i & (SS_ROWS - 1)) : i / SS_TK;
            const int k = TRANS ? i / SS_ROWS : (i & (SS_TK - 1));
            const int I = I0 + r, K = K0 + k;
            if (I < Ns && K < Ns) {
                const size_t at = TRANS ? (size_t)K * Ns + I : (size_t)I * Ns + K;
                if (STORE)
                    sigma[at] = (double)out[r * (SS_TK + 1) + k];
                else
                    sigma[at] += (double)out[r * (SS_TK + 1) + k];
            }
        }
        __syncthreads();
    }
}

// The same in float32 while a slab of TK columns of X fits in shared memory (up to 14 orbitals):
// there the rows of X are gathered from shared memory instead of L2, whose rate bounded
// k_large_ss (11.5 of ~12 TB/s): 334 -> 57 us at 12 orbitals; at 14, where only 16 columns fit
// and half of the paired rows share banks, 2.0 -> 1.65 ms (the shared-memory pipe).  A row of Hs per TK / 4 lanes, four columns a lane, the entries
// loaded one per lane and handed round; the padding of the last ones reads a row of zeros.  Work
// items are slabs x blocks of rows.
constexpr int SLAB_THREADS = 1024;

template <int TK, bool TRANS, bool STORE>
__global__ void __launch_bounds__(SLAB_THREADS) k_large_ss_slab(LargeCas L, const float *__restrict__ X,
                                                                double *__restrict__ sigma, int blocks)
{
    extern __shared__ __align__(16) char smem[];
    constexpr int LPR = TK / 4, RPW = 32 / LPR;
    float *slab = (float *)smem;  // [Ns + 1][TK]
    const int Ns = L.Ns, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, l = lane % LPR;
    const int nslab = (Ns + TK - 1) / TK, per = ((Ns + blocks - 1) / blocks + RPW - 1) / RPW * RPW;
    for (int item = blockIdx.x; item < nslab * blocks; item += gridDim.x) {
        const int K0 = item / blocks * TK, b = item % blocks;
        __syncthreads();  // the last slab is done with
#pragma unroll 8
        for (int q = threadIdx.x; q < (Ns + 1) * TK; q += SLAB_THREADS) {
            const int J = q / TK, K = K0 + q % TK;
            slab[q] = J < Ns && K < Ns ? X[(size_t)J * Ns + K] : 0.f;
        }
        __syncthreads();
        const int I1 = min((b + 1) * per, Ns);
        for (int r = b * per + warp * RPW; r < I1; r += SLAB_THREADS / 32 * RPW) {
            const int I = r + lane / LPR;
            const int64_t e0 = I < I1 ? L.roff[I] : 0;
            const int n = I < I1 ? (int)(L.roff[I + 1] - e0) : 0;
            const int most = __reduce_max_sync(FULL, n);
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
            int col = l < n ? L.col[e0 + l] : Ns;
            float val = l < n ? L.val32[e0 + l] : 0.f;
            for (int e = 0; e < most; e += LPR) {
                const int cc = col;
                const float cv = val;
                const int next = e + LPR + l;
                col = next < n ? L.col[e0 + next] : Ns;
                val = next < n ? L.val32[e0 + next] : 0.f;
#pragma unroll
                for (int i = 0; i < LPR; ++i) {
                    const int J = __shfl_sync(FULL, cc, i, LPR);
                    const float v = __shfl_sync(FULL, cv, i, LPR);
                    const float4 x = *(const float4 *)(slab + J * TK + 4 * l);
                    a0 = fmaf(v, x.x, a0);
                    a1 = fmaf(v, x.y, a1);
                    a2 = fmaf(v, x.z, a2);
                    a3 = fmaf(v, x.w, a3);
                }
            }
            const float out[4] = {a0, a1, a2, a3};
            if (I < I1)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int K = K0 + 4 * l + j;
                    if (K >= Ns) continue;
                    double *o = sigma + (TRANS ? (size_t)K * Ns + I : (size_t)I * Ns + K);
                    if (STORE)
                        *o = (double)out[j];
                    else
                        *o += (double)out[j];
                }
        }
    }
}

// Launch shape of k_large_ss_slab: columns per slab (0: none fits), row blocks that fill the last
// wave best (a slab's load counted as 2% of a whole product with it).
static int slab_columns(size_t smem_optin, int Ns)
{
    for (int tk = 32; tk >= 16; tk /= 2)
        if ((size_t)(Ns + 1) * tk * 4 + 1024 <= smem_optin) return tk;
    return 0;
}
static int slab_blocks(int sm_count, int Ns, int tk)
{
    const int nslab = (Ns + tk - 1) / tk;
    int best = 1;
    double cost = 1e300;
    for (int b = 1; b <= 16 && b * 32 <= Ns + 31; ++b) {
        const double c = (double)((nslab * b + sm_count - 1) / sm_count) * (1.0 / b + 0.02);
        if (c < cost) {
            cost = c;
            best = b;
        }
    }
    return best;
}

// sigma += A + sgn A^T for an Ns x Ns matrix A (32 x 32 tiles through shared
// memory): the same-spin terms of a vector in the spin-flip sector sgn, whose
// beta term is sgn times the transpose of the alpha term A = Hs C.
__global__ void k_sym_add(const double *__restrict__ A, int Ns, int sgn, double *__restrict__ sigma,
                          const unsigned long long *digits)
{
    if (digits && digits_usable(digits)) return;
    __shared__ double tile[32][33];
    const int nt = (Ns + 31) / 32;
    for (int64_t t = blockIdx.x; t < (int64_t)nt * nt; t += gridDim.x) {
        const int bi = (int)(t / nt), bj = (int)(t - (int64_t)bi * nt);
        // tile[x][r] = A[bj*32 + r][bi*32 + x], read row-wise (coalesced)
        for (int r = threadIdx.y; r < 32; r += blockDim.y) {
            const int i = bj * 32 + r, j = bi * 32 + threadIdx.x;
            tile[threadIdx.x][r] = (i < Ns && j < Ns) ? A[(size_t)i * Ns + j] : 0.0;
        }
        __syncthreads();
        for (int r = threadIdx.y; r < 32; r += blockDim.y) {
            const int i = bi * 32 + r, j = bj * 32 + threadIdx.x;
            if (i < Ns && j < Ns) {
                const size_t at = (size_t)i * Ns + j;
                const double at_t = tile[r][threadIdx.x];  // A[j][i]
                sigma[at] += A[at] + (sgn > 0 ? at_t : -at_t);
            }
        }
        __syncthreads();
    }
}

// out = in^T for an Ns x Ns matrix, 32 x 32 tiles through shared memory.
template <typename T>
__global__ void k_large_transpose(const T *__restrict__ in, int Ns, T *__restrict__ out, const unsigned long long *digits)
{
    if (digits && digits_usable(digits)) return;
    __shared__ T tile[32][33];
    const int nt = (Ns + 31) / 32;
    for (int64_t t = blockIdx.x; t < (int64_t)nt * nt; t += gridDim.x) {
        const int bi = (int)(t / nt), bj = (int)(t - (int64_t)bi * nt);
        for (int r = threadIdx.y; r < 32; r += blockDim.y) {
            const int i = bi * 32 + r, j = bj * 32 + threadIdx.x;
            if (i < Ns && j < Ns) tile[r][threadIdx.x] = in[(size_t)i * Ns + j];
        }
        __syncthreads();
        for (int r = threadIdx.y; r < 32; r += blockDim.y) {
            const int j = bj * 32 + r, i = bi * 32 + threadIdx.x;
            if (i < Ns && j < Ns) out[(size_t)j * Ns + i] = tile[threadIdx.x][r];
        }
        __syncthreads();
    }
}

// tabT[y * Ns + J] = tab[J * R + y] (the beta lists of the float64 opposite-spin term)
__global__ void k_large_tables(LargeCas L, int32_t *tabT)
{
    for (int J = blockIdx.x * blockDim.x + threadIdx.x; J < L.Ns; J += gridDim.x * blockDim.x)
        for (int y = 0; y < L.R; ++y) tabT[(size_t)y * L.Ns + J] = L.tab[(size_t)J * L.R + y];
}

// ---- grid-wide vector algebra of the large Davidson (all float64)

// out[i] = sum of v[i] over the grid, i < K (fixed order): each block's sums to partial, and the
// block that finishes last (ticket, back at 0 afterwards) adds them up.
template <int L>
__device__ __forceinline__ void grid_sums(double (&v)[L], int K, double *partial, unsigned *ticket, double *out)
{
    __shared__ double red[32 * L];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int i = 0; i < L; ++i)
        if (i < K) v[i] = warp_sum(v[i]);
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < L; ++i)
            if (i < K) red[w * L + i] = v[i];
    __syncthreads();
    if (threadIdx.x < K) {
        double s = 0.0;
        for (int j = 0; j < nw; ++j) s += red[j * L + threadIdx.x];
        __stcg(partial + (size_t)blockIdx.x * K + threadIdx.x, s);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int i = w; i < K; i += nw) {
        double s = 0.0;
        for (int b = lane; b < gridDim.x; b += 32) s += __ldcg(partial + (size_t)b * K + i);
        s = warp_sum(s);
        if (lane == 0) out[i] = s;
    }
}

// Whether the second orthogonalisation pass is needed: the first one left less than half of
// |t|^2 (with more left, one pass is orthogonal to within a few rounding errors).
__device__ __forceinline__ bool cancelled(const double *left, const double *t2) { return !(*left >= 0.5 * *t2); }

// out[i] = sum_d A_i[d] * u[d], i < K; A_i = A + i*ld.  Bound by the FP64 pipe.  left, t2: of a
// second pass, see cancelled.
__global__ void __launch_bounds__(LARGE_THREADS) k_multidot(const double *A, size_t ld, int K, const double *u,
                                                            int64_t N, double *partial, unsigned *ticket, double *out,
                                                            const double *left, const double *t2)
{
    if (left && !cancelled(left, t2)) return;
    double v[LRED];
#pragma unroll
    for (int i = 0; i < LRED; ++i) v[i] = 0.0;
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < N; d += (int64_t)gridDim.x * blockDim.x) {
        const double ud = u[d];
#pragma unroll
        for (int i = 0; i < LRED; ++i)
            if (i < K) v[i] += A[i * ld + d] * ud;
    }
    grid_sums(v, K, partial, ticket, out);
}

// u -= sum_{i<K} coef[i] A_i and out = |u|^2.  A second pass that is not needed only passes the
// norm on.
__global__ void __launch_bounds__(LARGE_THREADS) k_orthogonalise(const double *A, size_t ld, int K, const double *coef,
                                                                 int64_t N, double *u, double *partial, unsigned *ticket,
                                                                 double *out, const double *left, const double *t2)
{
    if (left && !cancelled(left, t2)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *out = *left;
        return;
    }
    double cf[MLARGE], v[1] = {0.0};
#pragma unroll
    for (int i = 0; i < MLARGE; ++i) cf[i] = (i < K) ? coef[i] : 0.0;
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < N; d += (int64_t)gridDim.x * blockDim.x) {
        double s = u[d];
#pragma unroll
        for (int i = 0; i < MLARGE; ++i)
            if (i < K) s -= cf[i] * A[i * ld + d];
        u[d] = s;
        v[0] += s * s;
    }
    grid_sums(v, 1, partial, ticket, out);
}

// x = V y, hx = W y, r = hx - theta x, t = r / clamp(diag - theta); out = |r|^2, |t|^2.
__global__ void __launch_bounds__(LARGE_THREADS) k_ritz(const double *V, const double *W, size_t ld, int m,
                                                        const double *ys, const double *misc, const double *diag,
                                                        double shift, int64_t N, double *x, double *hx, double *t,
                                                        double *partial, unsigned *ticket, double *out)
{
    const double th = misc[0];
    double y[MLARGE];
#pragma unroll
    for (int i = 0; i < MLARGE; ++i) y[i] = (i < m) ? ys[i] : 0.0;
    double v2[2] = {0.0, 0.0};
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < N; d += (int64_t)gridDim.x * blockDim.x) {
        double xs = 0.0, hs = 0.0;
#pragma unroll
        for (int i = 0; i < MLARGE; ++i)
            if (i < m) {
                xs += y[i] * V[i * ld + d];
                hs += y[i] * W[i * ld + d];
            }
        x[d] = xs;
        hx[d] = hs;
        double r = hs - th * xs;
        double den = (diag[d] - shift) - th;
        if (fabs(den) < 1e-4) den = den >= 0.0 ? 1e-4 : -1e-4;
        double td = r / den;
        t[d] = td;
        v2[0] += r * r;
        v2[1] += td * td;
    }
    grid_sums(v2, 2, partial, ticket, out);
}

// u -= sum_{i<K} coef[i] A_i and ub -= sum coef[i] B_i, coefficients read on the device.
__global__ void k_subtract(const double *A, const double *B, size_t ld, int K, const double *coef, int64_t N,
                           double *u, double *ub)
{
    double cf[LRED];
#pragma unroll
    for (int i = 0; i < LRED; ++i) cf[i] = (i < K) ? coef[i] : 0.0;
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < N; d += (int64_t)gridDim.x * blockDim.x) {
        double s = u[d], sb = ub[d];
#pragma unroll
        for (int i = 0; i < LRED; ++i)
            if (i < K) {
                s -= cf[i] * A[i * ld + d];
                sb -= cf[i] * B[i * ld + d];
            }
        u[d] = s;
        ub[d] = sb;
    }
}

// u = src * scale(norm2), scale = 1/sqrt(norm2[0]); optional second vector.
__global__ void k_scale_copy(const double *src, const double *src2, const double *norm2, int64_t N, double *u,
                             double *u2)
{
    const double s = 1.0 / sqrt(norm2[0]);
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < N; d += (int64_t)gridDim.x * blockDim.x) {
        u[d] = src[d] * s;
        if (u2) u2[d] = src2[d] * s;
    }
}

__global__ void k_to_float(const double *src, int64_t N, float *dst)
{
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < N; d += (int64_t)gridDim.x * blockDim.x)
        dst[d] = (float)src[d];
}

__global__ void k_copy2(const double *a, const double *b, int64_t N, double *ca, double *cb)
{
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < N; d += (int64_t)gridDim.x * blockDim.x) {
        ca[d] = a[d];
        cb[d] = b[d];
    }
}

// Row of element h of a packed sector vector (the upper triangle row by row, row i starting at
// i Ns - i (i - 1) / 2).
__device__ __forceinline__ int64_t packed_at(int Ns, int i, int j) { return (int64_t)i * Ns - (int64_t)i * (i - 1) / 2 + j - i; }

// Tiles of 32 x 32 on and above the diagonal of an Ns x Ns matrix, one per block and step.
template <typename F>
__device__ __forceinline__ void upper_tiles(int Ns, F f)
{
    const int nt = (Ns + 31) / 32;
    for (int64_t t = blockIdx.x; t < (int64_t)nt * nt; t += gridDim.x) {
        const int bi = (int)(t / nt), bj = (int)(t - (int64_t)bi * nt);
        if (bi > bj) continue;
        __syncthreads();
        f(bi * 32, bj * 32);
    }
}

constexpr double ROOT_HALF = 0.70710678118654752440, ROOT_2 = 1.41421356237309504880;

// full = the coefficient matrix of a packed vector v of the sector sgn; norm2: v is divided by
// its norm first, in place.
template <typename T>
__global__ void k_unpack(double *v, const double *norm2, int Ns, int sgn, T *full)
{
    __shared__ T tile[32][33];
    const double s = norm2 ? 1.0 / sqrt(*norm2) : 1.0;
    upper_tiles(Ns, [&](int i0, int j0) {
        for (int r = threadIdx.y; r < 32; r += blockDim.y) {
            const int i = i0 + r, j = j0 + threadIdx.x;
            if (i > j || j >= Ns) continue;
            double x = v[packed_at(Ns, i, j)];
            if (norm2) v[packed_at(Ns, i, j)] = x *= s;
            const T c = (T)(i == j ? x : ROOT_HALF * x);
            full[(size_t)i * Ns + j] = c;
            tile[r][threadIdx.x] = c;
        }
        __syncthreads();
        for (int r = threadIdx.y; r < 32; r += blockDim.y) {
            const int i = i0 + threadIdx.x, j = j0 + r;
            if (i < j && j < Ns) full[(size_t)j * Ns + i] = sgn > 0 ? tile[threadIdx.x][r] : -tile[threadIdx.x][r];
        }
    });
}

// The packed form of the sector's part of S + A + sgn A^T (A: may be NULL), less shift v (v: may be
// NULL): S and its mirror image are averaged, since its rounding is not symmetric and would let the
// other sector's lower states leak in.
__global__ void k_pack(const double *__restrict__ S, const double *__restrict__ A, int Ns, int sgn, const double *v,
                       double shift, double *__restrict__ out)
{
    __shared__ double tile[32][33];
    auto at = [&](int i, int j) { return 0.5 * S[(size_t)i * Ns + j] + (A ? A[(size_t)i * Ns + j] : 0.0); };
    upper_tiles(Ns, [&](int i0, int j0) {
        for (int r = threadIdx.y; r < 32; r += blockDim.y) {
            const int j = j0 + r, i = i0 + threadIdx.x;
            tile[threadIdx.x][r] = i <= j && j < Ns ? at(j, i) : 0.0;
        }
        __syncthreads();
        for (int r = threadIdx.y; r < 32; r += blockDim.y) {
            const int i = i0 + r, j = j0 + threadIdx.x;
            if (i > j || j >= Ns) continue;
            double x = at(i, j) + (sgn > 0 ? tile[r][threadIdx.x] : -tile[r][threadIdx.x]);
            if (i == j)
                x = sgn > 0 ? x : 0.0;
            else
                x *= ROOT_2;
            const int64_t h = packed_at(Ns, i, j);
            out[h] = v ? x - shift * v[h] : x;
        }
    });
}

// start vector (packed): lowest diagonal element (index given) + fixed admixture
__global__ void k_large_guess(const int64_t *best, int Ns, int sgn, double *x)
{
    const SectorGuess sg{(int)best[0], sgn};
    for (int i = blockIdx.x; i < Ns; i += gridDim.x)
        for (int j = i + threadIdx.x; j < Ns; j += blockDim.x)
            x[packed_at(Ns, i, j)] = i == j && sgn < 0 ? 0.0 : (i == j ? 1.0 : ROOT_2) * sector_guess(i * Ns + j, Ns, sg);
}

// the packed vector's elements of the diagonal of H
__global__ void k_pack_diag(const double *diag, int Ns, double *out)
{
    for (int i = blockIdx.x; i < Ns; i += gridDim.x)
        for (int j = i + threadIdx.x; j < Ns; j += blockDim.x) out[packed_at(Ns, i, j)] = diag[(size_t)i * Ns + j];
}

// index of the smallest diagonal element (ties -> lowest index), optionally
// among the determinants with Ia != Ib only; one block
__global__ void k_argmin(const double *diag, int64_t N, int Ns, int open_only, int64_t *out)
{
    __shared__ double bv[32];
    __shared__ int64_t bix[32];
    double best = 1e300;
    int64_t bi = INT64_MAX;
    for (int64_t d = threadIdx.x; d < N; d += blockDim.x) {
        if (open_only && d / Ns == d % Ns) continue;
        double v = diag[d];
        if (v < best || (v == best && d < bi)) {
            best = v;
            bi = d;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        double ov = __shfl_xor_sync(FULL, best, o);
        int64_t oi = __shfl_xor_sync(FULL, bi, o);
        if (ov < best || (ov == best && oi < bi)) {
            best = ov;
            bi = oi;
        }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) {
        bv[w] = best;
        bix[w] = bi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int j = 1; j < (int)(blockDim.x >> 5); ++j)
            if (bv[j] < best || (bv[j] == best && bix[j] < bi)) {
                best = bv[j];
                bi = bix[j];
            }
        out[0] = bi;
    }
}

// Bookkeeping of G on the device.
__global__ void k_set_g2(double *Gd, const double *dots, int two)
{
    if (threadIdx.x == 0) {
        Gd[0] = dots[0];
        if (two) {
            Gd[1] = Gd[MMAX] = dots[1];
            Gd[MMAX + 1] = dots[2];
        }
    }
}

}  // namespace mbe

namespace mbe {

struct LargePlan {
    LargeCas L;
    int grid_ab64, grid_ss64, grid_ss32, grid_vec, grid_tr;
    size_t smem_ab64, smem_ss64, smem_ss32;
    void *cT;      // transposed coefficients (room for N float64)
    DigitsArgs dg;  // float64 sigma on the tensor cores
    int dg_chunk;   // 0: not used
    int slab_tk, slab_blocks;  // k_large_ss_slab (0: k_large_ss)
    uint32_t *tc_lists;        // of large_ab_tc
};


// Strings from which the float64 sigma is made of digits (six launches more than the plain kernels):
// in casci_sigma_large 5 of 10 orbitals (Ns = 252) 1002 -> 262 us, (6, 3) with 20 strings 185 -> 158,
// (6, 2) with 15 147 -> 155, (5, 2) with 10 126 -> 152; inside casci_solve, where the set-up is
// paid once, 12 strings 5.83 -> 5.74 and 18.2 -> 16.5 ms, 10 strings 3.64 -> 3.85 ms.
constexpr int DIGITS_SIGMA_NS = 16, DIGITS_SOLVE_NS = 11;

// Sets up one large CAS; the dense Hs may live in `dense_at` (e.g. the Davidson
// basis region, unused during set-up). `fp32` adds the float32 sigma's tables, and `fp64` the
// digits' from that many strings on (0: never).
static int large_setup(mbe_ctx *ctx, int norb, const double *h1, const double *eri, const uint8_t *occ, int n_cas,
                       const int32_t *cas_orbs, Bump &bump, double *dense_at, bool fp32, int fp64, LargePlan *plan,
                       int *k_out, int64_t *dphi_out)
{
    MBE_CHECK(n_cas >= 1 && n_cas <= MBE_MAX_STRING_ORB && n_cas <= norb, MBE_EUNSUPPORTED,
              "large CASCI: n_cas %d outside 1..%d", n_cas, MBE_MAX_STRING_ORB);
    std::vector<int> A(cas_orbs, cas_orbs + n_cas);
    std::sort(A.begin(), A.end());
    for (int i = 0; i < n_cas; ++i)
        MBE_CHECK(A[i] >= 0 && A[i] < norb && (i == 0 || A[i] != A[i - 1]), MBE_EINVAL,
                  "large CASCI: active orbital %d out of range or repeated", A[i]);
    std::vector<uint8_t> occ_h(norb);
    MBE_CU(cudaMemcpyAsync(occ_h.data(), occ, norb, cudaMemcpyDeviceToHost, ctx->stream));
    MBE_CU(cudaStreamSynchronize(ctx->stream));
    int k = 0;
    uint32_t mphi = 0;
    for (int i = 0; i < n_cas; ++i)
        if (occ_h[A[i]]) {
            ++k;
            mphi |= 1u << i;
        }
    const StringTable *st = nullptr;
    int rc = get_table(ctx, n_cas, k, &st);
    if (rc) return rc;
    LargeCas &L = plan->L;
    L.n = n_cas;
    L.P = n_cas * (n_cas + 1) / 2;
    L.k = k;
    L.Ns = (int)st->ns;
    L.R = st->r;
    L.N = st->ns * st->ns;
    L.str = st->strings;
    L.tab = st->table;
    const int P = L.P;
    const int64_t conn = 1 + (int64_t)k * (n_cas - k) + binom(k, 2) * binom(n_cas - k, 2);
    double *F = bump.take<double>((size_t)norb * norb);
    L.V = bump.take<double>((size_t)P * P);
    L.V32 = bump.take<float>((size_t)P * P);
    L.h = bump.take<double>(P);
    L.pp = bump.take<short>(2 * P);
    L.roff = bump.take<int64_t>((size_t)L.Ns + 1);
    L.col = bump.take<int32_t>((size_t)L.Ns * conn);
    L.val = bump.take<double>((size_t)L.Ns * conn);
    L.val32 = bump.take<float>((size_t)L.Ns * conn);
    L.diag = bump.take<double>((size_t)L.N);
    int32_t *cnt = bump.take<int32_t>((size_t)L.Ns);
    int64_t *off = bump.take<int64_t>((size_t)L.Ns + 1);
    int32_t *tabT = bump.take<int32_t>((size_t)L.R * L.Ns);
    L.tabT = tabT;
    plan->cT = bump.take<double>((size_t)L.N);  // float32 or float64 use
    L.Hd = dense_at ? dense_at : bump.take<double>((size_t)L.Ns * L.Ns);
    plan->tc_lists = fp32 ? (uint32_t *)bump.take<char>(large_tc_list_bytes(ctx->smem_optin, P, L.Ns, L.R)) : nullptr;
    plan->dg_chunk = fp64 > 0 && L.Ns >= fp64 ? large_digits_chunk(ctx->smem_optin, P, L.Ns, L.R) : 0;
    double *hd = nullptr;
    if (plan->dg_chunk) {
        DigitsArgs &g = plan->dg;
        g.P = P;
        g.Ns = L.Ns;
        g.R = L.R;
        g.nsp = (L.Ns + 63) / 64 * 64;
        g.n = 0;
        g.tab = L.tab;
        g.tabT = L.tabT;
        g.V = L.V;
        g.hd = hd = bump.take<double>((size_t)L.Ns);
        g.inv = bump.take<int32_t>((size_t)P * g.nsp);
        g.maxb = bump.take<unsigned long long>(4);
        g.planes = bump.take<uint16_t>((size_t)DIGITS * L.Ns * g.nsp);
        g.hplanes = bump.take<uint16_t>((size_t)DIGITS * L.Ns * g.nsp);
    }
    // (all of the above fits: the caller sized the workspace with large_bytes)
    k_core_fock<<<(norb * norb + 127) / 128, 128, 0, ctx->stream>>>(norb, h1, eri, occ, F);
    LargeSetupArgs sa;
    memset(&sa, 0, sizeof(sa));
    for (int i = 0; i < n_cas; ++i) sa.A[i] = A[i];
    sa.norb = norb;
    sa.eri = eri;
    sa.occ = occ;
    sa.F = F;
    k_large_setup<<<1, CTA_THREADS, 0, ctx->stream>>>(sa, L);
    const size_t smem_hs = (size_t)(P * P + P) * 8;
    MBE_CU(allow_smem(k_large_hs, ctx->smem_optin));
    k_large_hs<<<std::min(L.Ns, ctx->sm_count * 4), 256, smem_hs, ctx->stream>>>(L);
    const unsigned wgrid = (unsigned)(((int64_t)L.Ns * 32 + 255) / 256);
    k_large_hs_count<<<wgrid, 256, 0, ctx->stream>>>(L, cnt);
    k_scan_counts<<<1, 256, 0, ctx->stream>>>(cnt, L.Ns, off);
    k_large_hs_fill<<<wgrid, 256, 0, ctx->stream>>>(L, off);
    k_large_diag<<<ctx->sm_count * 8, 256, 0, ctx->stream>>>(L);
    k_large_tables<<<(L.Ns + 255) / 256, 256, 0, ctx->stream>>>(L, tabT);
    MBE_CU(cudaGetLastError());
    ctx->launches += 8;
    if (fp32) {
        if ((rc = large_tc_lists(ctx->stream, ctx->smem_optin, P, L.Ns, L.R, L.tab, plan->tc_lists))) return rc;
        ++ctx->launches;
    }
    if (plan->dg_chunk) {
        rc = large_digits_setup(ctx->stream, ctx->sm_count, plan->dg, L.Hd, hd);
        if (rc) return rc;
        ctx->launches += 4;
    }
    *k_out = k;
    int iphi = string_rank(mphi);
    *dphi_out = (int64_t)iphi * L.Ns + iphi;
    // launch shapes
    plan->smem_ab64 = (size_t)P * P * 8;
    MBE_CHECK(plan->smem_ab64 <= ctx->smem_optin, MBE_EUNSUPPORTED, "large CASCI: V needs %zu B shared memory",
              plan->smem_ab64);
    MBE_CU(allow_smem(k_large_ab64<false>, ctx->smem_optin));
    MBE_CU(allow_smem(k_large_ab64<true>, ctx->smem_optin));
    int b = 0;
    MBE_CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_large_ab64<false>, SIGMA_THREADS, plan->smem_ab64));
    plan->grid_ab64 = ctx->sm_count * (b > 0 ? b : 1);
    plan->smem_ss64 = (size_t)SS_ROWS * (SS_TK + 1) * 8;
    plan->smem_ss32 = (size_t)SS_ROWS * (SS_TK + 1) * 4;
    MBE_CU(allow_smem(k_large_ss<double, false>, ctx->smem_optin));
    MBE_CU(allow_smem(k_large_ss<double, true>, ctx->smem_optin));
    MBE_CU(allow_smem(k_large_ss<double, false, true>, ctx->smem_optin));
    MBE_CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_large_ss<double, false>, SS_THREADS, plan->smem_ss64));
    plan->grid_ss64 = ctx->sm_count * (b > 0 ? b : 1);
    MBE_CU(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_large_ss<float, false>, SS_THREADS, plan->smem_ss32));
    plan->grid_ss32 = ctx->sm_count * (b > 0 ? b : 1);
    plan->slab_tk = slab_columns(ctx->smem_optin, L.Ns);
    plan->slab_blocks = plan->slab_tk ? slab_blocks(ctx->sm_count, L.Ns, plan->slab_tk) : 0;
    plan->grid_tr = ctx->sm_count * 8;
    plan->grid_vec = ctx->sm_count * 4;
    return MBE_OK;
}

// Workspace bytes of large_setup (and the dense Hs unless aliased).
static size_t large_bytes(const mbe_ctx *ctx, int norb, int n, int k, bool dense_separate, bool fp32, int fp64)
{
    const int64_t ns = binom(n, k), N = ns * ns;
    const int P = n * (n + 1) / 2;
    const int64_t conn = 1 + (int64_t)k * (n - k) + binom(k, 2) * binom(n - k, 2);
    size_t b = align256((size_t)norb * norb * 8) + align256((size_t)P * P * 8) + align256((size_t)P * P * 4) +
               align256(P * 8) + align256(2 * P * 2) + align256((ns + 1) * 8) + align256(ns * conn * 4) +
               align256(ns * conn * 8) + align256(ns * conn * 4) + align256(N * 8) + align256(ns * 4) +
               align256((ns + 1) * 8) + 4096;
    b += align256((size_t)k * (n - k + 1) * ns * 4) + align256((size_t)N * 8);
    if (dense_separate) b += align256((size_t)ns * ns * 8);
    if (fp32) b += align256(large_tc_list_bytes(ctx->smem_optin, P, (int)ns, k * (n - k + 1)));
    if (fp64 > 0 && ns >= fp64 && large_digits_chunk(ctx->smem_optin, P, (int)ns, k * (n - k + 1))) {
        const size_t nsp = (size_t)(ns + 63) / 64 * 64;
        b += align256(ns * 8) + align256(P * nsp * 4) + 256 + 2 * align256((size_t)DIGITS * ns * nsp * 2);
    }
    return b;
}

template <bool TRANS, bool STORE>
static int large_ss_slab(mbe_ctx *ctx, const LargePlan &pl, const float *X, double *out)
{
    const int Ns = pl.L.Ns, items = (Ns + pl.slab_tk - 1) / pl.slab_tk * pl.slab_blocks;
    const int grid = std::min(items, ctx->sm_count), smem = (Ns + 1) * pl.slab_tk * 4;
    auto launch = [&](auto *kernel) -> int {
        MBE_CU(allow_smem(kernel, ctx->smem_optin));
        kernel<<<grid, SLAB_THREADS, smem, ctx->stream>>>(pl.L, X, out, pl.slab_blocks);
        return MBE_OK;
    };
    return pl.slab_tk == 32 ? launch(k_large_ss_slab<32, TRANS, STORE>) : launch(k_large_ss_slab<16, TRANS, STORE>);
}

// sigma = H c: the opposite-spin term written first, then Hs C added, then C Hs^T
// added through the transposed copy of c.
template <typename T>
static int large_sigma_launch(mbe_ctx *ctx, const LargePlan &pl, const T *c, double *sigma, int order_tag,
                              int sgn = 0, double *packed = nullptr, const double *v = nullptr, double shift = 0.0)
{
    TimedLaunch tl(ctx, order_tag, 2, sizeof(T) == 8 ? 64 : 32);
    const int Ns = pl.L.Ns;
    const unsigned long long *digits = nullptr;
    if (sizeof(T) == 8) {
        if (pl.dg_chunk) {
            DigitsArgs g = pl.dg;
            g.c = (const double *)c;
            g.sigma = sigma;
            const int rc = large_sigma_digits(ctx->stream, ctx->sm_count, ctx->smem_optin, g, pl.dg_chunk);
            if (rc) return rc;
            ctx->launches += g.n ? 6 : 4;
            digits = pl.dg.maxb;  // the kernels below return at once, unless digits_usable() says no
        }
        if (sgn == 0)
            k_large_ab64<false><<<pl.grid_ab64, SIGMA_THREADS, pl.smem_ab64, ctx->stream>>>(pl.L, (const double *)c,
                                                                                          sigma, 0, digits);
        else
            k_large_ab64<true><<<pl.grid_ab64, SIGMA_THREADS, pl.smem_ab64, ctx->stream>>>(pl.L, (const double *)c,
                                                                                         sigma, sgn, digits);
    } else {
        // the dense product on the tensor cores (large_tc.cu)
        const int rc = large_ab_tc(ctx->stream, ctx->sm_count, ctx->smem_optin, pl.L.P, pl.L.Ns, pl.L.R, pl.L.tab,
                                   pl.tc_lists, pl.L.V32, (const float *)c, sigma, ctx->dev_err);
        if (rc) return rc;
    }
    if (sizeof(T) == 4 && pl.slab_tk) {
        if (sgn == 0) {
            float *cT = (float *)pl.cT;
            int rc = large_ss_slab<false, false>(ctx, pl, (const float *)c, sigma);
            k_large_transpose<float><<<pl.grid_tr, dim3(32, 8), 0, ctx->stream>>>((const float *)c, Ns, cT, nullptr);
            if (!rc) rc = large_ss_slab<true, false>(ctx, pl, cT, sigma);
            if (rc) return rc;
        } else {
            double *A = (double *)pl.cT;
            const int rc = large_ss_slab<false, true>(ctx, pl, (const float *)c, A);
            if (rc) return rc;
            k_pack<<<pl.grid_tr, dim3(32, 8), 0, ctx->stream>>>(sigma, A, Ns, sgn, v, shift, packed);
        }
        MBE_CU(cudaGetLastError());
        ctx->launches += sgn == 0 ? 4 : 3;
        return tl.done();
    }
    const int grid_ss = sizeof(T) == 8 ? pl.grid_ss64 : pl.grid_ss32;
    const size_t smem_ss = sizeof(T) == 8 ? pl.smem_ss64 : pl.smem_ss32;
    if (sgn == 0) {
        T *cT = (T *)pl.cT;
        k_large_ss<T, false><<<grid_ss, SS_THREADS, smem_ss, ctx->stream>>>(pl.L, c, sigma, digits);
        k_large_transpose<T><<<pl.grid_tr, dim3(32, 8), 0, ctx->stream>>>(c, Ns, cT, digits);
        k_large_ss<T, true><<<grid_ss, SS_THREADS, smem_ss, ctx->stream>>>(pl.L, cT, sigma, digits);
    } else {
        // c in the sector sgn: the beta same-spin term is sgn times the transpose
        // of the alpha one, so one product (into the spare buffer) and a
        // transposing add replace the second product and the transpose of c
        double *A = (double *)pl.cT;
        k_large_ss<T, false, true><<<grid_ss, SS_THREADS, smem_ss, ctx->stream>>>(pl.L, c, A, digits);
        if (sizeof(T) == 8) {
            k_sym_add<<<pl.grid_tr, dim3(32, 8), 0, ctx->stream>>>(A, Ns, sgn, sigma, digits);
            ++ctx->launches;
        }
        k_pack<<<pl.grid_tr, dim3(32, 8), 0, ctx->stream>>>(sigma, sizeof(T) == 8 ? nullptr : A, Ns, sgn, v, shift, packed);
    }
    MBE_CU(cudaGetLastError());
    ctx->launches += sgn == 0 ? 4 : 3;
    return tl.done();
}

}  // namespace mbe

extern "C" int casci_sigma_large(mbe_ctx *ctx, int norb, const double *h1, const double *eri, const uint8_t *occ,
                                 int n_cas, const int32_t *cas_orbs, int precision, const double *c,
                                 double *sigma, double *diag)
{
    MBE_CHECK(ctx && h1 && eri && occ && cas_orbs && c && sigma, MBE_EINVAL, "casci_sigma_large: NULL argument");
    MBE_CHECK(norb >= 1 && norb <= MBE_MAX_NORB, MBE_EINVAL, "casci_sigma_large: norb %d", norb);
    MBE_CHECK(precision == MBE_PREC_FP64 || precision == MBE_PREC_MIXED, MBE_EINVAL,
              "casci_sigma_large: precision %d", precision);
    MBE_CU(cudaSetDevice(ctx->device));
    // occupation count first (sizes depend on it)
    std::vector<uint8_t> occ_h(norb);
    MBE_CU(cudaMemcpyAsync(occ_h.data(), occ, norb, cudaMemcpyDeviceToHost, ctx->stream));
    MBE_CU(cudaStreamSynchronize(ctx->stream));
    MBE_CHECK(n_cas >= 1 && n_cas <= MBE_MAX_STRING_ORB && n_cas <= norb, MBE_EUNSUPPORTED,
              "casci_sigma_large: n_cas %d outside 1..%d", n_cas, MBE_MAX_STRING_ORB);
    int k0 = 0;
    for (int i = 0; i < n_cas; ++i) k0 += (cas_orbs[i] >= 0 && cas_orbs[i] < norb && occ_h[cas_orbs[i]]) ? 1 : 0;
    const int64_t N = binom(n_cas, k0) * binom(n_cas, k0);
    const bool fp32 = precision == MBE_PREC_MIXED;
    const int fp64 = fp32 ? 0 : DIGITS_SIGMA_NS;  // (a float32 sigma needs no digits)
    size_t bytes = large_bytes(ctx, norb, n_cas, k0, true, fp32, fp64) + (fp32 ? align256(N * 4) : 0);
    void *ws = nullptr;
    int rc = workspace(ctx, bytes, &ws);
    if (rc) return rc;
    Bump bump(ws);
    LargePlan pl;
    int k = 0;
    int64_t dphi = 0;
    rc = large_setup(ctx, norb, h1, eri, occ, n_cas, cas_orbs, bump, nullptr, fp32, fp64, &pl, &k, &dphi);
    if (rc) return rc;
    if (diag) MBE_CU(cudaMemcpyAsync(diag, pl.L.diag, N * 8, cudaMemcpyDeviceToDevice, ctx->stream));
    if (precision == MBE_PREC_FP64) {
        pl.dg.n = n_cas;  // (a caller's vector may have any spread; inside the eigensolver the norm of the error counts)
        return large_sigma_launch<double>(ctx, pl, c, sigma, n_cas);
    }
    float *c32 = bump.take<float>((size_t)N);
    k_to_float<<<pl.grid_vec, 256, 0, ctx->stream>>>(c, N, c32);
    ++ctx->launches;
    rc = large_sigma_launch<float>(ctx, pl, c32, sigma, n_cas);
    if (rc) return rc;
    return check_dev_err(ctx);  // the tensor-core product reports a wait that ran out
}

namespace mbe {

// x2 = V y2, hx2 = W y2 over the first m basis vectors
__global__ void k_lincomb2(const double *V, const double *W, size_t ld, int m, const double *ys, int64_t N,
                           double *x2, double *hx2)
{
    double y[MLARGE];
#pragma unroll
    for (int i = 0; i < MLARGE; ++i) y[i] = (i < m) ? ys[i] : 0.0;
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < N; d += (int64_t)gridDim.x * blockDim.x) {
        double xs = 0.0, hs = 0.0;
#pragma unroll
        for (int i = 0; i < MLARGE; ++i)
            if (i < m) {
                xs += y[i] * V[i * ld + d];
                hs += y[i] * W[i * ld + d];
            }
        x2[d] = xs;
        hx2[d] = hs;
    }
}

// w -= shift * v  (the image of a correction under H - theta0)
__global__ void k_shift_image(const double *v, double shift, int64_t N, double *w)
{
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < N; d += (int64_t)gridDim.x * blockDim.x)
        w[d] -= shift * v[d];
}

// Thick restart that keeps the anchor V[0], W[0]: u1 = sum_{i>=1} y_i V_i and
// u2 = sum_{i>=1} y2_i V_i (the corrections of the two lowest Ritz vectors) and
// their images.
__global__ void k_anchor_restart(const double *V, const double *W, size_t ld, int m, const double *ys,
                                 const double *y2s, int64_t N, double *u1, double *w1, double *u2, double *w2)
{
    double y[MLARGE], y2[MLARGE];
#pragma unroll
    for (int i = 0; i < MLARGE; ++i) {
        y[i] = (i >= 1 && i < m) ? ys[i] : 0.0;
        y2[i] = (i >= 1 && i < m) ? y2s[i] : 0.0;
    }
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < N; d += (int64_t)gridDim.x * blockDim.x) {
        double a = 0.0, b = 0.0, c = 0.0, e = 0.0;
#pragma unroll
        for (int i = 1; i < MLARGE; ++i) {
            const double v = V[i * ld + d], w = W[i * ld + d];
            a += y[i] * v;
            b += y[i] * w;
            c += y2[i] * v;
            e += y2[i] * w;
        }
        u1[d] = a;
        w1[d] = b;
        u2[d] = c;
        w2[d] = e;
    }
}

// G entries of the anchored restart basis {V0, V1, V2} from dots = [W0.V1, V1.W1,
// W0.V2, V1.W2, V2.W2] (G00 kept); two = 0 when V2 was dropped.
__global__ void k_set_g3(double *Gd, const double *dots, int two)
{
    if (threadIdx.x == 0) {
        Gd[1] = Gd[MMAX] = dots[0];
        Gd[MMAX + 1] = dots[1];
        if (two) {
            Gd[2] = Gd[2 * MMAX] = dots[2];
            Gd[MMAX + 2] = Gd[2 * MMAX + 1] = dots[3];
            Gd[2 * MMAX + 2] = dots[4];
        }
    }
}

struct LargeDav {
    // vectors are packed: the elements Ia <= Ib of a sector vector, those with Ia != Ib times
    // sqrt 2 (half the work of the vector algebra, which the FP64 pipe bounds, and of its memory)
    double *V, *W, *x, *hx, *t, *x2, *hx2, *xs, *diag, *partial, *dots, *Gd, *ys, *y2s, *misc;
    double *full, *S;  // coefficient matrix (also as float32) and sigma of the sigma in work
    unsigned *ticket;
    float *basis;  // of launch_small_eig
    int64_t *best;
    int64_t N;  // packed elements
    size_t ld;
    int nblk;
};
// places in LargeDav::dots besides the sums of a call: |r|^2, |t|^2; |u|^2 after one pass and two
constexpr int DOT_R = 24, DOT_T = 25, DOT_U1 = 26, DOT_U2 = 27;

static void dot_to(mbe_ctx *ctx, const LargeDav &D, const double *A, int K, const double *u, double *out,
                   const double *left = nullptr)
{
    k_multidot<<<D.nblk, LARGE_THREADS, 0, ctx->stream>>>(A, D.ld, K, u, D.N, D.partial, D.ticket, out, left, D.dots + DOT_T);
    ++ctx->launches;
}

// wout = (H - shift) vin, both packed; norm2: vin is normalised first, in place.
template <typename T>
static int large_apply(mbe_ctx *ctx, const LargePlan &pl, const LargeDav &D, double *vin, const double *norm2, double *wout,
                       int sgn, double shift)
{
    k_unpack<T><<<pl.grid_tr, dim3(32, 8), 0, ctx->stream>>>(vin, norm2, pl.L.Ns, sgn, (T *)D.full);
    ++ctx->launches;
    return large_sigma_launch<T>(ctx, pl, (const T *)D.full, D.S, pl.L.n, sgn, wout, shift != 0.0 ? vin : nullptr, shift);
}

// One Davidson phase on the large space (T = sigma arithmetic).  D.x: start
// vector in, Ritz vector out.
// Anchored (anchor != NULL, T = float; see struct Anchor): D.x is the anchor x0;
// one float64 sigma gives theta0 = x0.Hx0 and the exact image W0 = (H - theta0) x0
// of V0 = x0; every later basis vector is a correction whose image is the float32
// sigma minus theta0 times it; the coupling of x0 to V_m is formed as W0.V_m; a
// thick restart keeps V0; *lambda returns theta0 + mu, *anchor_y0 the coefficient
// of x0 in the Ritz vector (which is left in D.x, float64).
template <typename T>
static int large_phase(mbe_ctx *ctx, const LargePlan &pl, const LargeDav &D, int sgn, double tol, int min_iter,
                       int max_iter, int steer, double *lambda, double *rnorm, int *nsig, int *status,
                       int *nsig64 = nullptr, double *anchor_y0 = nullptr)
{
    const int64_t N = D.N;
    const size_t ld = D.ld;
    cudaStream_t st = ctx->stream;
    const int g = pl.grid_vec;
    const bool anch = sizeof(T) == 4 && anchor_y0 != nullptr;
    double h3[4];
    *nsig = 0;
    *status = MBE_STATUS_OK;
    int rc;
    double shift = 0.0;
    dot_to(ctx, D, D.x, 1, D.x, D.dots);
    k_scale_copy<<<g, 256, 0, st>>>(D.x, nullptr, D.dots, N, D.V, nullptr);
    ++ctx->launches;
    if (anch) {
        if ((rc = large_apply<double>(ctx, pl, D, D.V, nullptr, D.W, sgn, 0.0))) return rc;
        ++*nsig64;
        dot_to(ctx, D, D.W, 1, D.V, D.dots);
        MBE_CU(cudaMemcpyAsync(&shift, D.dots, 8, cudaMemcpyDeviceToHost, st));
        MBE_CU(cudaStreamSynchronize(st));
        k_shift_image<<<g, 256, 0, st>>>(D.V, shift, N, D.W);
        ++ctx->launches;
    } else {
        if ((rc = large_apply<T>(ctx, pl, D, D.V, nullptr, D.W, sgn, 0.0))) return rc;
        ++*nsig;
    }
    dot_to(ctx, D, D.W, 1, D.V, D.dots);
    k_set_g2<<<1, 32, 0, st>>>(D.Gd, D.dots, 0);
    ++ctx->launches;
    int m = 1;
    double best = 3e38;
    int stall = 0;
    const double *col = nullptr;  // the new column of G
    int warm = 0;                 // G grew by it since the last eigenproblem
    for (int it = 0;; ++it) {
        if ((rc = launch_small_eig(st, D.Gd, m, col, warm, D.basis, D.ys, D.y2s, D.misc))) return rc;
        warm = 1;
        double *tdst = (m < MLARGE) ? D.V + (size_t)m * ld : D.t;
        k_ritz<<<D.nblk, LARGE_THREADS, 0, st>>>(D.V, D.W, ld, m, D.ys, D.misc, D.diag, shift, N, D.x, D.hx, tdst,
                                                 D.partial, D.ticket, D.dots + DOT_R);
        ctx->launches += 2;
        int herr = 0;
        MBE_CU(cudaMemcpyAsync(h3, D.dots + DOT_R, 16, cudaMemcpyDeviceToHost, st));
        MBE_CU(cudaMemcpyAsync(h3 + 2, D.misc, 8, cudaMemcpyDeviceToHost, st));
        MBE_CU(cudaMemcpyAsync(h3 + 3, D.ys, 8, cudaMemcpyDeviceToHost, st));
        MBE_CU(cudaMemcpyAsync(&herr, ctx->dev_err, sizeof(int), cudaMemcpyDeviceToHost, st));
        MBE_CU(cudaStreamSynchronize(st));
        if (herr) return check_dev_err(ctx);
        const double rn = sqrt(h3[0]), t0n = sqrt(h3[1]);
        *lambda = shift + h3[2];
        *rnorm = rn;
        if (anch) *anchor_y0 = h3[3];
        if (!std::isfinite(rn) || !std::isfinite(h3[2])) {
            *status = MBE_STATUS_NONFINITE;
            break;
        }
        if (rn <= tol && it >= min_iter) break;
        if (it >= max_iter) {
            *status = MBE_STATUS_MAXITER;
            break;
        }
        if (steer) {
            if (rn < 0.9 * best) {
                best = rn;
                stall = 0;
            } else if (++stall >= steer) {
                break;
            }
        }
        double *u = D.V + (size_t)m * ld;
        if (m == MLARGE && anch) {
            // keep V0 = x0, W0 = r0; V1, V2: corrections of the two lowest Ritz vectors
            // (D.t holds the new correction; D.x, D.hx are recomputed by the next k_ritz)
            k_anchor_restart<<<g, 256, 0, st>>>(D.V, D.W, ld, m, D.ys, D.y2s, N, D.x2, D.hx2, D.x, D.hx);
            k_copy2<<<g, 256, 0, st>>>(D.x2, D.hx2, N, D.V + ld, D.W + ld);
            ctx->launches += 2;
            dot_to(ctx, D, D.V + ld, 1, D.V + ld, D.dots);
            k_scale_copy<<<g, 256, 0, st>>>(D.V + ld, D.W + ld, D.dots, N, D.V + ld, D.W + ld);
            k_copy2<<<g, 256, 0, st>>>(D.x, D.hx, N, D.V + 2 * ld, D.W + 2 * ld);
            ctx->launches += 2;
            for (int pass = 0; pass < 2; ++pass) {
                dot_to(ctx, D, D.V + ld, 1, D.V + 2 * ld, D.dots);
                k_subtract<<<g, 256, 0, st>>>(D.V + ld, D.W + ld, ld, 1, D.dots, N, D.V + 2 * ld, D.W + 2 * ld);
                ++ctx->launches;
            }
            dot_to(ctx, D, D.V + 2 * ld, 1, D.V + 2 * ld, D.dots);
            MBE_CU(cudaMemcpyAsync(h3, D.dots, 8, cudaMemcpyDeviceToHost, st));
            MBE_CU(cudaStreamSynchronize(st));
            const int two = sqrt(h3[0]) > 1e-3 ? 1 : 0;
            if (two) {
                k_scale_copy<<<g, 256, 0, st>>>(D.V + 2 * ld, D.W + 2 * ld, D.dots, N, D.V + 2 * ld, D.W + 2 * ld);
                ++ctx->launches;
            }
            dot_to(ctx, D, D.W, 1, D.V + ld, D.dots);               // W0.V1
            dot_to(ctx, D, D.V + ld, 1, D.W + ld, D.dots + 1);      // V1.W1
            if (two) {
                dot_to(ctx, D, D.W, 1, D.V + 2 * ld, D.dots + 2);   // W0.V2
                dot_to(ctx, D, D.V + ld, 1, D.W + 2 * ld, D.dots + 3);  // V1.W2
                dot_to(ctx, D, D.V + 2 * ld, 1, D.W + 2 * ld, D.dots + 4);  // V2.W2
            }
            k_set_g3<<<1, 32, 0, st>>>(D.Gd, D.dots, two);
            ++ctx->launches;
            m = 2 + two;
            warm = 0;
            u = D.V + (size_t)m * ld;
            MBE_CU(cudaMemcpyAsync(u, D.t, (size_t)N * 8, cudaMemcpyDeviceToDevice, st));
        } else if (m == MLARGE) {
            // thick restart on the two lowest Ritz vectors (orthogonal by construction)
            k_lincomb2<<<g, 256, 0, st>>>(D.V, D.W, ld, m, D.y2s, N, D.x2, D.hx2);
            k_copy2<<<g, 256, 0, st>>>(D.x, D.hx, N, D.V, D.W);
            k_copy2<<<g, 256, 0, st>>>(D.x2, D.hx2, N, D.V + ld, D.W + ld);
            ctx->launches += 3;
            for (int pass = 0; pass < 2; ++pass) {
                dot_to(ctx, D, D.V, 1, D.V + ld, D.dots);
                k_subtract<<<g, 256, 0, st>>>(D.V, D.W, ld, 1, D.dots, N, D.V + ld, D.W + ld);
                ++ctx->launches;
            }
            dot_to(ctx, D, D.V + ld, 1, D.V + ld, D.dots);
            k_scale_copy<<<g, 256, 0, st>>>(D.V + ld, D.W + ld, D.dots, N, D.V + ld, D.W + ld);
            dot_to(ctx, D, D.W, 2, D.V, D.dots);
            dot_to(ctx, D, D.W + ld, 1, D.V + ld, D.dots + 2);
            k_set_g2<<<1, 32, 0, st>>>(D.Gd, D.dots, 1);
            ctx->launches += 2;
            m = 2;
            warm = 0;
            u = D.V + (size_t)m * ld;
            MBE_CU(cudaMemcpyAsync(u, D.t, (size_t)N * 8, cudaMemcpyDeviceToDevice, st));
        }
        for (int pass = 0; pass < 2; ++pass) {
            const double *left = pass ? D.dots + DOT_U1 : nullptr;
            dot_to(ctx, D, D.V, m, u, D.dots, left);
            k_orthogonalise<<<D.nblk, LARGE_THREADS, 0, st>>>(D.V, ld, m, D.dots, N, u, D.partial, D.ticket,
                                                              D.dots + (pass ? DOT_U2 : DOT_U1), left, D.dots + DOT_T);
            ++ctx->launches;
        }
        MBE_CU(cudaMemcpyAsync(h3, D.dots + DOT_U2, 8, cudaMemcpyDeviceToHost, st));
        MBE_CU(cudaStreamSynchronize(st));
        const double tn = sqrt(h3[0]);
        if (!(tn > 1e-12 * t0n) || !(tn > 0.0)) {
            if (!steer && rn > tol) *status = MBE_STATUS_MAXITER;
            break;
        }
        if ((rc = large_apply<T>(ctx, pl, D, u, D.dots + DOT_U2, D.W + (size_t)m * ld, sgn, anch ? shift : 0.0))) return rc;
        ++*nsig;
        dot_to(ctx, D, D.V, m + 1, D.W + (size_t)m * ld, D.dots);
        if (anch) dot_to(ctx, D, D.W, 1, u, D.dots);  // x0.(A u) as u.r0
        col = D.dots;
        ++m;
    }
    return MBE_OK;
}

}  // namespace mbe

extern "C" int casci_solve(mbe_ctx *ctx, int norb, const double *h1, const double *eri, const uint8_t *occ,
                           int n_cas, const int32_t *cas_orbs, const mbe_opts *opts, double *result,
                           int32_t *info, double *cvec)
{
    MBE_CHECK(ctx && h1 && eri && occ && cas_orbs && result && info, MBE_EINVAL, "casci_solve: NULL argument");
    MBE_CHECK(norb >= 1 && norb <= MBE_MAX_NORB, MBE_EINVAL, "casci_solve: norb %d", norb);
    MBE_CHECK(n_cas >= 1 && n_cas <= MBE_MAX_STRING_ORB && n_cas <= norb, MBE_EUNSUPPORTED,
              "casci_solve: n_cas %d outside 1..%d", n_cas, MBE_MAX_STRING_ORB);
    mbe_opts o;
    if (opts) o = *opts; else mbe_default_opts(&o);
    MBE_CHECK(o.precision == MBE_PREC_FP64 || o.precision == MBE_PREC_MIXED, MBE_EINVAL,
              "casci_solve: unknown precision %d", o.precision);
    MBE_CHECK(o.tol > 0 && o.tol_switch > 0 && o.max_iter >= 1 && o.fp64_final_iters >= 0 &&
                  (o.sectors == MBE_SECTORS_BOTH || o.sectors == MBE_SECTORS_EVEN), MBE_EINVAL,
              "casci_solve: bad options");
    MBE_CHECK(o.s2_penalty == 0.0, MBE_EUNSUPPORTED, "casci_solve: the S^2 penalty is not supported for one large CAS");
    MBE_CU(cudaSetDevice(ctx->device));
    std::vector<uint8_t> occ_h(norb);
    MBE_CU(cudaMemcpyAsync(occ_h.data(), occ, norb, cudaMemcpyDeviceToHost, ctx->stream));
    MBE_CU(cudaStreamSynchronize(ctx->stream));
    int k0 = 0;
    for (int i = 0; i < n_cas; ++i) k0 += (cas_orbs[i] >= 0 && cas_orbs[i] < norb && occ_h[cas_orbs[i]]) ? 1 : 0;
    const int64_t N = binom(n_cas, k0) * binom(n_cas, k0);
    const int64_t ns0 = binom(n_cas, k0);
    LargeDav D;
    D.N = ns0 * (ns0 + 1) / 2;
    const size_t vec = align256((size_t)D.N * 8);
    D.ld = vec / 8;
    D.nblk = ctx->sm_count * 4;
    const bool mixed = o.precision == MBE_PREC_MIXED;
    size_t bytes = large_bytes(ctx, norb, n_cas, k0, false, mixed, DIGITS_SOLVE_NS) + vec * (2 * MLARGE + 7) + 2 * align256((size_t)N * 8) +
                   align256((size_t)D.nblk * LRED * 8) + 8 * 256 + 8192;
    void *ws = nullptr;
    int rc = workspace(ctx, bytes, &ws);
    if (rc) return rc;
    Bump bump(ws);
    D.V = bump.take<double>(D.ld * MLARGE);
    D.W = bump.take<double>(D.ld * MLARGE);
    D.x = bump.take<double>(D.ld);
    D.hx = bump.take<double>(D.ld);
    D.t = bump.take<double>(D.ld);
    D.x2 = bump.take<double>(D.ld);
    D.hx2 = bump.take<double>(D.ld);
    D.xs = bump.take<double>(D.ld);
    D.diag = bump.take<double>(D.ld);
    D.full = bump.take<double>((size_t)N);
    D.S = bump.take<double>((size_t)N);
    D.ticket = bump.take<unsigned>(1);
    D.basis = bump.take<float>((MMAX + 1) * MMAX + 1);
    D.partial = bump.take<double>((size_t)D.nblk * LRED);
    D.dots = bump.take<double>(32);
    D.Gd = bump.take<double>(MMAX * MMAX);
    D.ys = bump.take<double>(MMAX);
    D.y2s = bump.take<double>(MMAX);
    D.misc = bump.take<double>(8);
    D.best = bump.take<int64_t>(4);
    LargePlan pl;
    int k = 0;
    int64_t dphi = 0;
    // The dense one-spin Hamiltonian of the set-up lives in the (not yet used) basis region.
    rc = large_setup(ctx, norb, h1, eri, occ, n_cas, cas_orbs, bump, D.V, mixed, DIGITS_SOLVE_NS, &pl, &k, &dphi);
    if (rc) return rc;
    const int Ns = pl.L.Ns;
    k_argmin<<<1, 1024, 0, ctx->stream>>>(pl.L.diag, N, Ns, 0, D.best);
    k_argmin<<<1, 1024, 0, ctx->stream>>>(pl.L.diag, N, Ns, 1, D.best + 1);
    k_pack_diag<<<std::min(Ns, ctx->sm_count * 8), 256, 0, ctx->stream>>>(pl.L.diag, Ns, D.diag);
    MBE_CU(cudaMemsetAsync(D.ticket, 0, sizeof(unsigned), ctx->stream));
    ctx->launches += 3;
    double lam = 0.0, rn = 0.0;
    int n32 = 0, n64 = 0, st = 0;
    int won = 1;
    bool degen = false;
    // the two spin-flip sectors (see sector_guess); each runs the float32 phase
    // (mixed mode) and the float64 phase; the second sector first runs a float64
    // pass to the residual SECTOR_TOL only and stops there when sector_loses
    for (int sector = 0; sector < 2; ++sector) {
        if (sector == 1 && (Ns < 2 || st != MBE_STATUS_OK || o.sectors == MBE_SECTORS_EVEN)) break;
        const int sgn = sector == 0 ? 1 : -1;
        if (sector == 1) MBE_CU(cudaMemcpyAsync(D.xs, D.x, (size_t)D.N * 8, cudaMemcpyDeviceToDevice, ctx->stream));
        k_large_guess<<<std::min(Ns, ctx->sm_count * 8), 256, 0, ctx->stream>>>(D.best + sector, Ns, sgn, D.x);
        ++ctx->launches;
        double l = 0.0, r = 0.0;
        int s64 = 0, s32 = 0, ss = MBE_STATUS_OK;
        bool lose = false, refined = false;
        if (mixed) {
            // float32 phase (tensor-core sigma), then anchored refinements (struct
            // Anchor): one float64 sigma per anchor, float32 sigmas for the
            // corrections; the second sector is decided once its residual reaches
            // SECTOR_TOL. A refinement that fails hands over to the float64 phase.
            int n = 0;
            rc = large_phase<float>(ctx, pl, D, sgn, o.tol_switch, 0, o.max_iter, 3, &l, &r, &n, &ss);
            if (rc) return rc;
            s32 += n;
            bool decided = sector == 0;
            if (ss == MBE_STATUS_NONFINITE) {
                k_large_guess<<<std::min(Ns, ctx->sm_count * 8), 256, 0, ctx->stream>>>(D.best + sector, Ns, sgn, D.x);
                ++ctx->launches;
            } else {
                for (int anc = 0; anc < LARGE_ANCHORS && !lose && !refined; ++anc) {
                    const double tgt = decided ? o.tol : SECTOR_TOL;
                    double y0 = 1.0;
                    int n64a = 0;
                    n = 0;
                    rc = large_phase<float>(ctx, pl, D, sgn, tgt, decided ? o.fp64_final_iters : 0, o.max_iter,
                                            LARGE_ANCHOR_STALL, &l, &r, &n, &ss, &n64a, &y0);
                    if (rc) return rc;
                    s32 += n;
                    s64 += n64a;
                    if (ss == MBE_STATUS_NONFINITE) break;
                    if (!decided && r <= SECTOR_TOL) {
                        decided = true;
                        lose = sector_loses(l, r, lam, 0.0);
                        continue;
                    }
                    const double dn = sqrt(std::max(0.0, 1.0 - y0 * y0)) / std::max(fabs(y0), 1e-300);
                    refined = decided && r <= o.tol && dn <= MIX_DMAX;
                }
            }
        } else if (sector == 1) {
            // a float64 pass from the start vector to SECTOR_TOL decides
            int n = 0;
            rc = large_phase<double>(ctx, pl, D, sgn, SECTOR_TOL, 0, o.max_iter, LARGE_STALL, &l, &r, &n, &ss);
            if (rc) return rc;
            s64 += n;
            lose = ss == MBE_STATUS_NONFINITE || sector_loses(l, r, lam, 0.0);
        }
        if (refined) ss = MBE_STATUS_OK;
        if (!lose && !refined) {
            int n = 0;
            rc = large_phase<double>(ctx, pl, D, sgn, o.tol, (mixed && sector == 0) ? o.fp64_final_iters : 0,
                                     o.max_iter, 0, &l, &r, &n, &ss);
            if (rc) return rc;
            s64 += n;
        }
        n64 += s64;
        n32 += s32;
        if (sector == 0) {
            lam = l;
            rn = r;
            st = ss;
        } else if (!lose && ss != MBE_STATUS_NONFINITE && l < lam) {
            degen = degen || (ss == MBE_STATUS_OK && st == MBE_STATUS_OK && fabs(l - lam) <= DEGEN_TOL);
            lam = l;
            rn = r;
            st = ss;
            won = sgn;
        } else {
            degen = degen || (!lose && ss == MBE_STATUS_OK && st == MBE_STATUS_OK && fabs(l - lam) <= DEGEN_TOL);
            MBE_CU(cudaMemcpyAsync(D.x, D.xs, (size_t)D.N * 8, cudaMemcpyDeviceToDevice, ctx->stream));
        }
    }
    double ephi = 0.0;
    MBE_CU(cudaMemcpyAsync(&ephi, pl.L.diag + dphi, 8, cudaMemcpyDeviceToHost, ctx->stream));
    if (cvec) {
        k_unpack<double><<<pl.grid_tr, dim3(32, 8), 0, ctx->stream>>>(D.x, nullptr, Ns, won, cvec);
        MBE_CU(cudaGetLastError());
        ++ctx->launches;
    }
    MBE_CU(cudaStreamSynchronize(ctx->stream));
    result[0] = lam;
    result[1] = lam - ephi;
    result[2] = rn;
    info[0] = with_degeneracy(st, degen);
    info[1] = n64;
    info[2] = n32;
    return MBE_OK;
}
