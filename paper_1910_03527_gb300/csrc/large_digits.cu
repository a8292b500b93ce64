// The float64 sigma of one large active space on the tensor cores.
//
//     sigma[Ia][Ib] = sum_{x in list(Ia)} s_x sum_{y in list(Ib)} s_y V[p_x][p_y] c[J_x][J_y]
//                     + (Hs c + c Hs)[Ia][Ib]
//
// A float64 multiply-add runs on 1.67 lanes per clock and SM here, and the plain kernels stood at
// 95% of that (4.3 ms at 12 orbitals).  The products are made of exact ones of 8-bit digits
// instead (the Ozaki scheme: Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 95, 2012): V, Hs
// and c as fixed-point numbers of 55 bits and sign below their largest elements, in seven signed
// digits of base 256, each exact in bfloat16.  The products of digits i of one and j of the other
// operand with the same i + j = d add up in one float32 accumulator, exactly (at most 1,023 of
// them, each at most 2^14); the pairs with i + j > 7, below 2^-61 of the largest term, are left
// out: 34 products of mma.sync.m16n8k16.  The eight sums of an element are joined in a 64-bit
// integer and rounded to 2^-54 of the largest term.  (28 products, without i + j = 7, took 1.33 ms
// at 12 orbitals where these take 1.41, but their errors were those of the pairs left out, 2.4 times
// as large.)
// The error is a fraction of the operands' largest elements, where that of a float64 sum is a
// fraction of its own terms: a caller's vector is looked at first (k_digits_near).
//
// Opposite-spin term, per alpha string Ia: a dense product T[p][J] = sum_x (s_x V[p_x][p])
// c[J_x][J] and a scatter, sigma[Ia][K] += s T[p][J] for every E_p |J> = s |K>, in three 21-bit
// parts (32-bit shared atomics, exact in any order).  One CTA per SM, persistent over Ia; the
// digits of the signed V columns stay in shared memory, the rows of c come in chunks of strings
// by cp.async from planes of digits (made once per vector), two buffers.  A warp takes 16 pairs
// x 8 strings at a time: per 16 list entries 14 ldmatrix for 34 mma.
// Same-spin terms: Hs (symmetric, its diagonal kept out and added in float64: it would set the
// scale) and c as dense matrices of digits.
//
// casci_sigma_large in float64, with its set-up, against the plain kernels: 12 orbitals 5.6 -> 1.5 ms;
// largest error against 64-bit sums there 3.6e-16 of the largest element, 6.0e-16 before.
#include <algorithm>

#include "common.cuh"
#include "large_digits.cuh"

namespace mbe {

constexpr int DG_THREADS = 640;  // 20 warps: the 5 x 8 tiles of 12 orbitals in two rounds
// Row strides in 16-bit words are odd multiples of 8 so that the 8 rows of an ldmatrix matrix lie
// in different banks.

// Sums kept: the digit pairs with i + j < DIGIT_SUMS.
constexpr int DIGIT_SUMS = DIGITS + 1;

// The sums of an element, joined (in units of 256^7, as join_digits).
__device__ __forceinline__ long long join_sums(const float (&acc)[DIGIT_SUMS][4], int e)
{
    long long s = (long long)__float2int_rn(acc[0][e]);
#pragma unroll
    for (int d = 1; d < DIGITS - 1; ++d) s = s * 256 + __float2int_rn(acc[d][e]);
    const int rest = __float2int_rn(acc[DIGITS - 1][e]) + ((__float2int_rn(acc[DIGITS][e]) + 128) >> 8);
    return s + ((rest + 128) >> 8);
}

struct DigitsShape {
    int mt, kp, as, off_b, off_row, off_jx, bytes;
};

static __host__ __device__ inline DigitsShape digits_shape(int P, int Ns, int R, int chunk)
{
    DigitsShape s;
    s.mt = (P + 15) / 16;
    s.kp = (R + 15) / 16 * 16;
    s.as = s.kp + 8;
    s.off_b = DIGITS * s.mt * 16 * s.as * 2;
    s.off_row = s.off_b + 2 * DIGITS * s.kp * (chunk + 8) * 2;
    s.off_jx = s.off_row + 12 * Ns;
    s.bytes = (s.off_jx + 4 * s.kp + 15) / 16 * 16;
    return s;
}

// 64 strings per chunk up to 13 orbitals, 32 at 14; at 15 the row of sigma alone takes 77 KB.
int large_digits_chunk(size_t smem_optin, int P, int Ns, int R)
{
    if (R < 1 || R > 80) return 0;
    for (int chunk = 64; chunk >= 32; chunk /= 2)
        if ((size_t)digits_shape(P, Ns, R, chunk).bytes + 1024 <= smem_optin) return chunk;
    return 0;
}

// The largest element of an Ns x Ns matrix, the diagonal left out (and copied to diag) if asked.
__global__ void k_digits_max(const double *__restrict__ M, int64_t rows, int cols, double *diag, unsigned long long *out)
{
    const int64_t N = rows * cols;
    unsigned long long big = 0;
    for (int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; d < N; d += (int64_t)gridDim.x * blockDim.x) {
        const double v = M[d];
        if (diag && d % (cols + 1) == 0) {
            diag[d / (cols + 1)] = v;
            continue;
        }
        const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
        big = b > big ? b : big;
    }
    __syncwarp();
    max_bits(big, out);
}

// Whether digits are as accurate as float64 sums for every element of the result.  They round V, Hs
// and c to fixed fractions of their largest elements, float64 sums each term to a fraction of itself,
// so digits are the more accurate ones where the sums are not made of small terms only: the R^2
// elements of c that an element of sigma adds up must average EVEN_C of the largest (first, the sums
// over the beta lists; then those over the alpha lists), the elements of V EVEN_V of its largest, and
// Hs must not exceed n max|V|.  Otherwise (a converged CI vector, say, whose elements fall with the
// excitation) usable[3] is set, and the plain float64 kernels answer.  Errors in units of 2^-53 sum
// |V| |c|, root mean square (largest) over 1,400 elements of 10 orbitals, plain and by digits:
// normal c 0.75 (4.0) and 0.34 (1.2); c falling by 3 per excitation 0.63 (3.3) and 33 (300).  The two
// passes over c take 45 us at 12 orbitals.
constexpr double EVEN_C = 1.0 / 12, EVEN_V = 1.0 / 40;

__global__ void __launch_bounds__(256) k_digits_near(DigitsArgs a, float *near)
{
    extern __shared__ __align__(128) unsigned char smem[];
    float *row = (float *)smem;
    if (!digits_in_range(a.maxb)) return;
    const int Ns = a.Ns;
    const double scale = pow2d(-bits_exponent(a.maxb[2]));
    for (int I = blockIdx.x; I < Ns; I += gridDim.x) {
        __syncthreads();
        for (int K = threadIdx.x; K < Ns; K += blockDim.x) row[K] = (float)fabs(a.c[(size_t)I * Ns + K] * scale);
        __syncthreads();
        for (int K = threadIdx.x; K < Ns; K += blockDim.x) {
            float v = 0.f;
            for (int y = 0; y < a.R; ++y) v += row[entry_J(a.tabT[(size_t)y * Ns + K])];
            near[(size_t)I * Ns + K] = v;
        }
    }
}

// (The last block looks at the integrals.)
__global__ void __launch_bounds__(256) k_digits_even(DigitsArgs a, const float *near)
{
    if (!digits_in_range(a.maxb)) return;
    const int Ns = a.Ns, last = gridDim.x - 1;
    if (blockIdx.x == last) {
        __shared__ float part[8];
        const double vscale = pow2d(-bits_exponent(a.maxb[0]));
        float v = 0.f;
        for (int q = threadIdx.x; q < a.P * a.P; q += blockDim.x) v += (float)fabs(a.V[q] * vscale);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < 8; ++w) v += part[w];
            const double top = __longlong_as_double((long long)a.maxb[0]), hs = __longlong_as_double((long long)a.maxb[1]);
            if (!(v >= EVEN_V * a.P * a.P * top * vscale) || !(hs <= a.n * top)) a.maxb[3] = 1ull;
        }
        return;
    }
    const double top = __longlong_as_double((long long)a.maxb[2]) * pow2d(-bits_exponent(a.maxb[2]));
    const float least = (float)(EVEN_C * a.R * a.R * top);
    bool even = true;
    for (int I = blockIdx.x; I < Ns; I += last) {
        const int32_t *ta = a.tab + (size_t)I * a.R;
        for (int K = threadIdx.x; K < Ns; K += blockDim.x) {
            float v = 0.f;
            for (int x = 0; x < a.R; ++x) v += near[(size_t)entry_J(ta[x]) * Ns + K];
            even = even && v >= least;
        }
    }
    if (!even) a.maxb[3] = 1ull;
}

// Planes of digits of an Ns x Ns matrix, rows padded to nsp with zeros; skip: the diagonal as 0.
// usable: of all operands, or NULL (the planes are made in any case).
__global__ void k_digits_planes(const double *__restrict__ M, int Ns, int nsp, int skip, const unsigned long long *big,
                                const unsigned long long *usable, uint16_t *planes)
{
    if (usable && !digits_usable(usable)) return;
    const double scale = pow2d(55 - bits_exponent(*big));
    const size_t plane = (size_t)Ns * nsp;
    for (int I = blockIdx.x; I < Ns; I += gridDim.x)
        for (int J = threadIdx.x; J < nsp; J += blockDim.x) {
            uint16_t d[DIGITS];
            to_digits(J < Ns && !(skip && I == J) ? __double2ll_rn(M[(size_t)I * Ns + J] * scale) : 0, d);
#pragma unroll
            for (int i = 0; i < DIGITS; ++i) planes[i * plane + (size_t)I * nsp + J] = d[i];
        }
}

// inv[p][J] = K << 1 | neg for E_p |J> = s |K>, else -1 (set beforehand)
__global__ void k_digits_inverse(const int32_t *tab, int Ns, int nsp, int R, int32_t *inv)
{
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < Ns * R; q += gridDim.x * blockDim.x) {
        const int J = q / R, e = tab[q];
        inv[(size_t)entry_pair(e) * nsp + J] = entry_J(e) << 1 | entry_neg(e);
    }
}

// sigma[Ia][K] = opposite-spin term + (hd[Ia] + hd[K]) c[Ia][K]
template <int DG_CHUNK>
__global__ void __launch_bounds__(DG_THREADS, 1) k_large_ab_digits(DigitsArgs a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int DG_BS = DG_CHUNK + 8;
    if (!digits_usable(a.maxb)) return;
    const int P = a.P, Ns = a.Ns, R = a.R, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const DigitsShape S = digits_shape(P, Ns, R, DG_CHUNK);
    uint16_t *A = (uint16_t *)smem, *B = (uint16_t *)(smem + S.off_b);
    int *row = (int *)(smem + S.off_row), *jx = (int *)(smem + S.off_jx);
    const int nchunk = (Ns + DG_CHUNK - 1) / DG_CHUNK, bplane = S.kp * DG_BS, aplane = S.mt * 16 * S.as;
    const size_t plane = (size_t)Ns * a.nsp;
    const double vscale = pow2d(55 - bits_exponent(a.maxb[0]));
    const double unit = pow2d(bits_exponent(a.maxb[0]) + bits_exponent(a.maxb[2]) - 54);
    // the rows of B beyond the list are zero in both buffers
    for (int q = tid; q < 2 * DIGITS * (S.kp - R) * DG_BS; q += DG_THREADS) {
        const int pl = q / ((S.kp - R) * DG_BS), r = q - pl * (S.kp - R) * DG_BS;
        B[pl * bplane + R * DG_BS + r] = 0;
    }
    for (int Ia = blockIdx.x; Ia < Ns; Ia += gridDim.x) {
        const int32_t *ta = a.tab + (size_t)Ia * R;
        __syncthreads();  // the last row is written, its operands are free
        for (int x = tid; x < R; x += DG_THREADS) jx[x] = entry_J(ta[x]);
        for (int q = tid; q < 3 * Ns; q += DG_THREADS) row[q] = 0;
        for (int q = tid; q < S.mt * 16 * S.kp; q += DG_THREADS) {
            const int x = q / (S.mt * 16), p = q - x * S.mt * 16;  // (V is read along its rows)
            long long f = 0;
            if (x < R && p < P) {
                const int e = ta[x];
                f = __double2ll_rn(a.V[entry_pair(e) * P + p] * vscale);
                if (entry_neg(e)) f = -f;
            }
            uint16_t d[DIGITS];
            to_digits(f, d);
#pragma unroll
            for (int i = 0; i < DIGITS; ++i) A[i * aplane + p * S.as + x] = d[i];
        }
        __syncthreads();
        auto fetch = [&](int chunk) {
            uint16_t *buf = B + (chunk & 1) * DIGITS * bplane;
            for (int q = tid; q < DIGITS * R * (DG_CHUNK / 8); q += DG_THREADS) {
                const int s = q % (DG_CHUNK / 8), r = q / (DG_CHUNK / 8), i = r / R, x = r - i * R;
                const uint16_t *src = a.planes + i * plane + (size_t)jx[x] * a.nsp + chunk * DG_CHUNK + 8 * s;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(shared_u32(buf + i * bplane + x * DG_BS + 8 * s)),
                             "l"(src)
                             : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        fetch(0);
        for (int ch = 0; ch < nchunk; ++ch) {
            if (ch + 1 < nchunk) fetch(ch + 1);
            if (ch + 1 < nchunk)
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            else
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            const uint16_t *buf = B + (ch & 1) * DIGITS * bplane;
            for (int t = warp; t < S.mt * (DG_CHUNK / 8); t += DG_THREADS / 32) {
                const int mt = t / (DG_CHUNK / 8), nt = t - mt * (DG_CHUNK / 8);
                int to[4];  // where the tile's elements go (asked for before the product)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int p = mt * 16 + (lane >> 2) + (e >> 1) * 8, J = ch * DG_CHUNK + nt * 8 + (lane & 3) * 2 + (e & 1);
                    to[e] = p < P && J < Ns ? a.inv[(size_t)p * a.nsp + J] : -1;
                }
                float acc[DIGIT_SUMS][4];
#pragma unroll
                for (int d = 0; d < DIGIT_SUMS; ++d) acc[d][0] = acc[d][1] = acc[d][2] = acc[d][3] = 0.f;
                const uint32_t aa = shared_u32(A + (mt * 16 + (lane & 15)) * S.as + (lane >> 4) * 8);
                const uint32_t ba = shared_u32(buf + (lane & 15) * DG_BS + nt * 8);
#pragma unroll 1
                for (int k = 0; k < S.kp; k += 16) {
                    uint32_t bf[DIGITS][2];
#pragma unroll
                    for (int j = 0; j < DIGITS; ++j) ldsm_x2_trans(bf[j], ba + 2 * (j * bplane + k * DG_BS));
                    uint32_t af[2][4];
                    ldsm_x4(af[0], aa + 2 * k);
#pragma unroll
                    for (int i = 0; i < DIGITS; ++i) {
                        if (i + 1 < DIGITS) ldsm_x4(af[(i + 1) & 1], aa + 2 * ((i + 1) * aplane + k));
#pragma unroll
                        for (int j = 0; j < DIGITS && i + j < DIGIT_SUMS; ++j) mma_bf16(acc[i + j], af[i & 1], bf[j][0], bf[j][1]);
                    }
                }
                // scatter
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (to[e] < 0) continue;
                    long long s = join_sums(acc, e);
                    if (to[e] & 1) s = -s;
                    int *r = row + (to[e] >> 1);
                    atomicAdd(r, (int)(s & 0x1fffff));
                    atomicAdd(r + Ns, (int)(s >> 21 & 0x1fffff));
                    atomicAdd(r + 2 * Ns, (int)(s >> 42));
                }
            }
            __syncthreads();  // the buffer is free for the chunk after the next
        }
        const double ha = a.hd[Ia];
        for (int K = tid; K < Ns; K += DG_THREADS) {
            const long long low = row[K] + ((long long)row[Ns + K] << 21);
            const double t = fma((double)row[2 * Ns + K], 4398046511104.0, (double)low);  // 2^42
            a.sigma[(size_t)Ia * Ns + K] = fma(ha + a.hd[K], a.c[(size_t)Ia * Ns + K], t * unit);
        }
    }
}

// sigma += Hs c + c Hs without the diagonal of Hs: one 64 x 32 tile per CTA, two CTAs per SM, a
// warp 16 x 16 of it, the two products one after the other along 2 Ns in chunks of 32 by cp.async,
// two buffers.  The float32 sums are joined and added in float64 every 128 steps.  Dense, although
// 72% of Hs is zero at 12 orbitals (86% at 14): the sparse float64 products take five times as
// long there.
constexpr int GM_M = 64, GM_N = 32, GM_K = 32, GM_THREADS = 256, GM_S = 40;
constexpr int GM_BUF = DIGITS * (GM_M + GM_K) * GM_S;  // 16-bit words of one buffer

__global__ void __launch_bounds__(GM_THREADS, 2) k_large_ss_digits(DigitsArgs a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    if (!digits_usable(a.maxb)) return;
    uint16_t *buf = (uint16_t *)smem;
    const int Ns = a.Ns, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ntn = (Ns + GM_N - 1) / GM_N, ntm = (Ns + GM_M - 1) / GM_M, nk = (Ns + GM_K - 1) / GM_K;
    const size_t plane = (size_t)Ns * a.nsp;
    const double unit = pow2d(bits_exponent(a.maxb[1]) + bits_exponent(a.maxb[2]) - 54);
    const int wm = warp >> 1, wn = warp & 1;
    for (int t = blockIdx.x; t < ntm * ntn; t += gridDim.x) {
        const int I0 = t / ntn * GM_M, K0 = (t - t / ntn * ntn) * GM_N;
        auto fetch = [&](int ch) {
            const uint16_t *left = ch < nk ? a.hplanes : a.planes, *right = ch < nk ? a.planes : a.hplanes;
            const int k0 = (ch < nk ? ch : ch - nk) * GM_K;
            uint16_t *A = buf + (ch & 1) * GM_BUF, *B = A + DIGITS * GM_M * GM_S;
            // (a chunk of 8 columns lies below nsp; rows from Ns on are filled with zeros)
            for (int q = tid; q < DIGITS * GM_M * (GM_K / 8); q += GM_THREADS) {
                const int s = q % (GM_K / 8), r = q / (GM_K / 8), i = r / GM_M, m = r % GM_M, in = I0 + m < Ns;
                const uint16_t *src = left + i * plane + (size_t)(in ? I0 + m : 0) * a.nsp + k0 + 8 * s;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(shared_u32(A + r * GM_S + 8 * s)),
                             "l"(src), "r"(in ? 16 : 0)
                             : "memory");
            }
            for (int q = tid; q < DIGITS * GM_K * (GM_N / 8); q += GM_THREADS) {
                const int s = q % (GM_N / 8), r = q / (GM_N / 8), i = r / GM_K, k = r % GM_K, in = k0 + k < Ns;
                const uint16_t *src = right + i * plane + (size_t)(in ? k0 + k : 0) * a.nsp + K0 + 8 * s;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(shared_u32(B + r * GM_S + 8 * s)),
                             "l"(src), "r"(in ? 16 : 0)
                             : "memory");
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        float acc[2][DIGIT_SUMS][4];
        double sum[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                sum[h][e] = 0.0;
#pragma unroll
                for (int d = 0; d < DIGIT_SUMS; ++d) acc[h][d][e] = 0.f;
            }
        __syncthreads();  // the last tile's buffers are free
        fetch(0);
        for (int ch = 0; ch < 2 * nk; ++ch) {
            if (ch + 1 < 2 * nk) {
                fetch(ch + 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            const uint16_t *A = buf + (ch & 1) * GM_BUF, *B = A + DIGITS * GM_M * GM_S;
            const uint32_t aa = shared_u32(A + (wm * 16 + (lane & 15)) * GM_S + (lane >> 4) * 8);
            const uint32_t ba = shared_u32(B + (lane & 15) * GM_S + wn * 16 + (lane >> 4) * 8);
#pragma unroll 1
            for (int k = 0; k < GM_K; k += 16) {
                uint32_t bf[DIGITS][4];
#pragma unroll
                for (int j = 0; j < DIGITS; ++j) ldsm_x4_trans(bf[j], ba + 2 * (j * GM_K + k) * GM_S);
                uint32_t af[2][4];
                ldsm_x4(af[0], aa + 2 * k);
#pragma unroll
                for (int i = 0; i < DIGITS; ++i) {
                    if (i + 1 < DIGITS) ldsm_x4(af[(i + 1) & 1], aa + 2 * ((i + 1) * GM_M * GM_S + k));
#pragma unroll
                    for (int j = 0; j < DIGITS && i + j < DIGIT_SUMS; ++j) {
                        mma_bf16(acc[0][i + j], af[i & 1], bf[j][0], bf[j][1]);
                        mma_bf16(acc[1][i + j], af[i & 1], bf[j][2], bf[j][3]);
                    }
                }
            }
            if ((ch & 3) == 3 || ch == 2 * nk - 1) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        sum[h][e] += (double)join_sums(acc[h], e);
#pragma unroll
                        for (int d = 0; d < DIGIT_SUMS; ++d) acc[h][d][e] = 0.f;
                    }
            }
            __syncthreads();  // the buffer is free for the chunk after the next
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int I = I0 + wm * 16 + (lane >> 2) + (e >> 1) * 8, K = K0 + wn * 16 + h * 8 + (lane & 3) * 2 + (e & 1);
                if (I < Ns && K < Ns) {
                    double *o = a.sigma + (size_t)I * Ns + K;
                    *o = fma(sum[h][e], unit, *o);
                }
            }
    }
}

int large_sigma_digits(cudaStream_t st, int sm_count, size_t smem_optin, const DigitsArgs &a, int chunk)
{
    const DigitsShape S = digits_shape(a.P, a.Ns, a.R, chunk);
    const int smem_ss = 2 * GM_BUF * 2, rows = std::min(a.Ns, sm_count * 8);
    MBE_CU(cudaMemsetAsync(a.maxb + 2, 0, 2 * 8, st));
    k_digits_max<<<rows, 256, 0, st>>>(a.c, a.Ns, a.Ns, nullptr, a.maxb + 2);
    if (a.n) {  // (the sums lie where the planes will)
        k_digits_near<<<rows, 256, std::max(a.Ns, 32) * 4, st>>>(a, (float *)a.planes);
        k_digits_even<<<rows + 1, 256, 0, st>>>(a, (const float *)a.planes);
    }
    k_digits_planes<<<rows, 256, 0, st>>>(a.c, a.Ns, a.nsp, 0, a.maxb + 2, a.maxb, a.planes);
    if (chunk == 64) {
        MBE_CU(allow_smem(k_large_ab_digits<64>, smem_optin));
        k_large_ab_digits<64><<<std::min(sm_count, a.Ns), DG_THREADS, S.bytes, st>>>(a);
    } else {
        MBE_CU(allow_smem(k_large_ab_digits<32>, smem_optin));
        k_large_ab_digits<32><<<std::min(sm_count, a.Ns), DG_THREADS, S.bytes, st>>>(a);
    }
    MBE_CU(allow_smem(k_large_ss_digits, smem_optin));
    const int tiles = (a.Ns + GM_M - 1) / GM_M * ((a.Ns + GM_N - 1) / GM_N);
    k_large_ss_digits<<<std::min(tiles, sm_count * 2), GM_THREADS, smem_ss, st>>>(a);
    MBE_CU(cudaGetLastError());
    return MBE_OK;
}

int large_digits_setup(cudaStream_t st, int sm_count, const DigitsArgs &a, const double *Hs, double *hd)
{
    const int rows = std::min(a.Ns, sm_count * 8);
    MBE_CU(cudaMemsetAsync(a.maxb, 0, 4 * 8, st));
    MBE_CU(cudaMemsetAsync(a.inv, 0xff, (size_t)a.P * a.nsp * 4, st));
    k_digits_max<<<1, 1024, 0, st>>>(a.V, a.P, a.P, nullptr, a.maxb);
    k_digits_max<<<rows, 256, 0, st>>>(Hs, a.Ns, a.Ns, hd, a.maxb + 1);
    k_digits_planes<<<rows, 256, 0, st>>>(Hs, a.Ns, a.nsp, 1, a.maxb + 1, nullptr, a.hplanes);
    k_digits_inverse<<<(a.Ns * a.R + 255) / 256, 256, 0, st>>>(a.tab, a.Ns, a.nsp, a.R, a.inv);
    MBE_CU(cudaGetLastError());
    return MBE_OK;
}

}  // namespace mbe
