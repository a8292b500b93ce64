#pragma once
// a2-a7 for tuples of 2-6 orbitals: the sector solvers, one tuple per warp.
//
// A kernel is compiled per string class (n, k).  Two things follow from that:
//   * every Davidson vector lies in one spin-flip sector, c[Ia][Ib] = sgn c[Ib][Ia],
//     and is kept as its Ns (Ns + 1) / 2 elements with Ia <= Ib in an orthonormal
//     basis of the sector (off-diagonal elements scaled by sqrt 2, so that plain dot
//     products are those of the whole vector): 7 register slots per lane at (6, 3)
//     instead of 13, and half of the vector algebra;
//   * the replacement lists of one spin are compile-time constants.  A lane owns one
//     beta string Ib and, for each entry y of Ib's list, reads the row J_y of c and the
//     row p_y of V once and forms its share of all Ns elements sigma[*][Ib] with the
//     alpha lists unrolled: at (6, 3), 240 fused multiply-adds on registers for 21
//     shared-memory loads, where a loop over both lists needs three dependent loads
//     (entry, V, c) and a sign flip for every multiply-add.
// The element count is not halved (all Ia, not only Ia <= Ib): the unrolled lists
// need the same Ia in every lane.  The same-spin terms ride along as M = C Hs of the
// lane's own row, and one symmetrisation at the end gives
//     sigma[Ia][Ib] = A[Ia][Ib] + sgn A[Ib][Ia],   A = 1/2 (alpha-beta term) + sgn M^T.
#include <utility>

#include "casci_dev.cuh"

namespace mbe {

// ------------------------------------------------------------------ string classes at compile time

template <int N_, int K_>
struct Cls {
    static constexpr int n = N_, k = K_;
    static constexpr int choose(int a, int b)
    {
        int c = 1;
        for (int i = 1; i <= b; ++i) c = c * (a - b + i) / i;
        return b < 0 || b > a ? 0 : c;
    }
    static constexpr int NS = choose(n, k), R = k * (n - k + 1), P = n * (n + 1) / 2;
    static constexpr int NH = NS * (NS + 1) / 2, DH = (NH + 31) / 32;
    static constexpr int PT = P * (P + 1) / 2;  // packed V
    static constexpr int PH = (P + 1) / 2, NSH = (NS + 1) / 2;
    // row stride of float and int64 Ns x Ns scratch: 16-byte rows whose starts spread over the banks
    static constexpr int NSP = (NS + 3) / 4 * 4 % 16 == 0 ? (NS + 3) / 4 * 4 + 4 : (NS + 3) / 4 * 4;
    // lanes per beta string; 20 strings leave 12 lanes, which take a third of the lists (see rounds())
    static constexpr bool HELP = NS == 20;
    static constexpr int L = HELP ? 2 : 32 / NS;  // partial results per element

    static __host__ __device__ constexpr uint32_t str(int i)  // i-th string in ascending order
    {
        uint32_t s = (1u << k) - 1u;
        for (; i > 0; --i) {
            const uint32_t c = s & (0u - s), r = s + c;
            s = (((r ^ s) >> 2) / c) | r;
        }
        return s;
    }
    static __host__ __device__ constexpr int bits(uint32_t s)
    {
        int c = 0;
        for (; s; s &= s - 1u) ++c;
        return c;
    }
    static __host__ __device__ constexpr int rank(uint32_t s)
    {
        int i = 0;
        while (str(i) != s) ++i;
        return i;
    }
    // e_ab |I> = s |J> for the pair {a >= b}, e_ab = E_ab + E_ba (E_aa if a == b): J, or -1
    static __host__ __device__ constexpr int target(int I, int a, int b)
    {
        const uint32_t s = str(I);
        const bool oa = (s >> a) & 1u, ob = (s >> b) & 1u;
        if (a == b) return oa ? I : -1;
        return oa == ob ? -1 : rank(s ^ (1u << a) ^ (1u << b));
    }
    static __host__ __device__ constexpr bool negative(int I, int a, int b)
    {
        return a != b && (bits(str(I) & ((1u << a) - 1u) & ~((2u << b) - 1u)) & 1);
    }
    static __host__ __device__ constexpr int pair_hi(int p)
    {
        int a = 0;
        while ((a + 1) * (a + 2) / 2 <= p) ++a;
        return a;
    }
    static __host__ __device__ constexpr int pair_lo(int p) { return p - pair_hi(p) * (pair_hi(p) + 1) / 2; }
};

template <int I>
struct Const {
    static constexpr int value = I;
    __host__ __device__ constexpr operator int() const { return I; }
};
template <class F, int... I>
__device__ __forceinline__ void static_for_(F f, std::integer_sequence<int, I...>)
{
    (f(Const<I>{}), ...);
}
template <int COUNT, class F>
__device__ __forceinline__ void static_for(F f)
{
    static_for_(f, std::make_integer_sequence<int, COUNT>{});
}

// v, hidden from the optimiser.  A condition that never changes inside the Davidson loop
// (plain or anchored, the sector's sign) makes the compiler write one copy of the loop for each
// of its values, sigma included; on an SM all copies are hot, and the instruction cache is what
// these kernels wait for.
__device__ __forceinline__ int opaque(int v)
{
    asm volatile("" : "+r"(v));
    return v;
}

// ------------------------------------------------------------------ block-wide tables

// Tables of the class, built once per block: the replacement lists (J << 8 | pair << 1
// | neg), the packed triangles of string pairs (Ia <= Ib, row-major) and of orbital-pair
// pairs (x >= y), and the orbitals of each pair.
template <class C>
struct SectorTables {
    uint16_t list[C::NS * C::R];
    uchar2 tri[C::NH];
    uchar2 ptri[C::PT];
    uchar2 pq[C::P];
    uint32_t str[C::NS];
};

template <class C>
__device__ void build_tables(SectorTables<C> &T, const ClassInfo &ci)
{
#pragma unroll 1
    for (int i = threadIdx.x; i < C::NS * C::R; i += blockDim.x) {
        const int e = ci.table[i];
        T.list[i] = (uint16_t)(entry_J(e) << 8 | (e & 0xff));
    }
#pragma unroll 1
    for (int i = threadIdx.x; i < C::NS; i += blockDim.x) {
        T.str[i] = ci.strings[i];
#pragma unroll 1
        for (int j = i; j < C::NS; ++j)
            T.tri[i * C::NS - i * (i - 1) / 2 + j - i] = make_uchar2((unsigned char)i, (unsigned char)j);
    }
#pragma unroll 1
    for (int x = threadIdx.x; x < C::P; x += blockDim.x) {
        const int a = C::pair_hi(x);
        T.pq[x] = make_uchar2((unsigned char)a, (unsigned char)(x - a * (a + 1) / 2));
#pragma unroll 1
        for (int y = 0; y <= x; ++y) T.ptri[x * (x + 1) / 2 + y] = make_uchar2((unsigned char)x, (unsigned char)y);
    }
    __syncthreads();
}

// ------------------------------------------------------------------ per-tuple set-up

// One element of the one-spin string Hamiltonian by the Slater-Condon rules, from
// h(p, q) and V(p, q, r, s) = (pq|rs): at most k^2 additions, where multiplying out
// sum E_pq E_rs takes R^2 per column.
template <class H, class VF>
__host__ __device__ inline double string_element(uint32_t I, uint32_t J, H h, VF V)
{
    auto low = [](uint32_t s) {
        int b = 0;
#ifdef __CUDA_ARCH__
        b = __ffs((int)s) - 1;
#else
        while (!(s >> b & 1u)) ++b;
#endif
        return b;
    };
    auto odd = [](uint32_t s) {
        int c = 0;
#ifdef __CUDA_ARCH__
        c = __popc(s) & 1;
#else
        for (; s; s &= s - 1u) c ^= 1;
#endif
        return c;
    };
    auto between = [](int a, int b) {
        const int lo = a < b ? a : b, hi = a < b ? b : a;
        return ((1u << hi) - 1u) & ~((2u << lo) - 1u);
    };
    uint32_t from = I & ~J, to = J & ~I;
    double v = 0.0;
    if (from == 0u) {
#pragma unroll 1
        for (uint32_t a = I; a; a &= a - 1u) {
            const int p = low(a);
            v += h(p, p);
#pragma unroll 1
            for (uint32_t b = a & (a - 1u); b; b &= b - 1u) {
                const int q = low(b);
                v += V(p, p, q, q) - V(p, q, p, q);
            }
        }
        return v;
    }
    const int p = low(from), a = low(to);
    from &= from - 1u;
    to &= to - 1u;
    int neg = odd(I & between(p, a));
    if (from == 0u) {
        v = h(p, a);
#pragma unroll 1
        for (uint32_t c = I & J; c; c &= c - 1u) {
            const int r = low(c);
            v += V(p, a, r, r) - V(p, r, r, a);
        }
        return neg ? -v : v;
    }
    const int q = low(from), b = low(to);
    from &= from - 1u;
    if (from != 0u) return 0.0;
    neg ^= odd((I ^ (1u << p) ^ (1u << a)) & between(q, b));
    v = V(p, a, q, b) - V(p, b, q, a);
    return neg ? -v : v;
}

// Fixed-point form of a float64 value for the integer sigma: v = (hi 2^28 + lo) 2^(E - 55),
// |v| <= 2^E, with |hi| <= 2^27 and -2^27 <= lo < 2^27.
__device__ inline int2 to_fixed(double v, double scale)
{
    const long long f = __double2ll_rn(v * scale);
    const int hi = (int)((f + (1LL << 27)) >> 28);
    return make_int2(hi, (int)(f - ((long long)hi << 28)));
}

// 2^e as a double (e within the normal range)
__device__ inline double pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// |v|'s high word: ordered like |v| (a warp's double fmax is 19 cycles of the FP64 pipe).
__device__ inline int high_word(double v) { return __double2hiint(v) & 0x7fffffff; }

// Exponent E of the fixed-point scale: 2^E is the power of two above the warp's largest value,
// from its high words.
__device__ inline int fixed_exponent(int hi)
{
    const int E = (__reduce_max_sync(FULL, hi) >> 20) - 1022;
    return E < -900 ? -900 : E > 900 ? 900 : E;
}

struct SectorStart {
    int g, go;      // packed index of the lowest diagonal element, and of the lowest with Ia != Ib
    double ephi;    // diagonal element of Phi_A
};

// A warp's tuple: h_eff, V and Hs in float64, the diagonal.  Vp [PT], Hsp [NH] and hd [NS]
// (the diagonal of Hs) stay; h and diag are scratch.
template <class C>
__device__ SectorStart sector_setup(const BatchArgs &a, const SectorTables<C> &T, const int *A, double *Vp, double *Hsp,
                                    double *hd, double *h, double *dsum, double *diag)
{
    const int lane = threadIdx.x & 31;
    const size_t norb = a.norb;
#pragma unroll 2
    for (int e = lane; e < C::PT; e += 32) {
        const uchar2 xy = T.ptri[e], pq = T.pq[xy.x], rs = T.pq[xy.y];
        Vp[e] = a.eri[eri_index(a.norb, A[pq.x], A[pq.y], A[rs.x], A[rs.y])];
    }
    uint32_t mphi = 0;
#pragma unroll
    for (int i = 0; i < C::n; ++i)
        if (a.occ[A[i]]) mphi |= 1u << i;
    __syncwarp();
    if (lane < C::P) {
        const int p = T.pq[lane].x, q = T.pq[lane].y;
        double v = a.F[A[p] * norb + A[q]];
#pragma unroll 1
        for (uint32_t m = mphi; m; m &= m - 1u) {
            const int i = __ffs((int)m) - 1;
            v -= 2.0 * Vp[tri_index(lane, pair_index(i, i))] - Vp[tri_index(pair_index(p, i), pair_index(i, q))];
        }
        h[lane] = v;
    }
#pragma unroll 1
    for (int e = lane; e < C::NS * C::n; e += 32) {  // sum_{p in I} (pp|qq)
        const int I = e / C::n, q = e - I * C::n;
        double v = 0.0;
#pragma unroll 1
        for (uint32_t m = T.str[I]; m; m &= m - 1u) {
            const int p = __ffs((int)m) - 1;
            v += Vp[tri_index(pair_index(p, p), pair_index(q, q))];
        }
        dsum[e] = v;
    }
    __syncwarp();
    auto hf = [&](int p, int q) { return h[pair_index(p, q)]; };
    auto Vf = [&](int p, int q, int r, int s) { return Vp[tri_index(pair_index(p, q), pair_index(r, s))]; };
#pragma unroll 1
    for (int e = lane; e < C::NH; e += 32) {
        const uchar2 ij = T.tri[e];
        const double v = string_element(T.str[ij.x], T.str[ij.y], hf, Vf);
        Hsp[e] = v;
        if (ij.x == ij.y) hd[ij.x] = v;
    }
    __syncwarp();
    // (compared as integers that are ordered like the values: a warp's float64 comparison holds the
    // FP64 pipe for 19 cycles)
    auto ordered = [](double v) {
        const long long b = __double_as_longlong(v);
        return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
    };
    long long best = ordered(1e300), best_o = best;
    SectorStart st;
    st.g = st.go = 0x7fffffff;
#pragma unroll 1
    for (int e = lane; e < C::NH; e += 32) {
        const uchar2 ij = T.tri[e];
        double v = hd[ij.x] + hd[ij.y];
#pragma unroll 1
        for (uint32_t m = T.str[ij.y]; m; m &= m - 1u) v += dsum[ij.x * C::n + __ffs((int)m) - 1];
        diag[e] = v;
        const long long u = ordered(v);
        if (u < best) {
            best = u;
            st.g = e;
        }
        if (ij.x != ij.y && u < best_o) {
            best_o = u;
            st.go = e;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {  // the lowest element, ties to the lowest index
        long long ov = __shfl_xor_sync(FULL, best, o);
        int oi = __shfl_xor_sync(FULL, st.g, o);
        if (ov < best || (ov == best && oi < st.g)) {
            best = ov;
            st.g = oi;
        }
        ov = __shfl_xor_sync(FULL, best_o, o);
        oi = __shfl_xor_sync(FULL, st.go, o);
        if (ov < best_o || (ov == best_o && oi < st.go)) {
            best_o = ov;
            st.go = oi;
        }
    }
    if (st.g > C::NH) st.g = 0;  // (a diagonal without finite elements)
    if (st.go > C::NH) st.go = 1;
    __syncwarp();
    const int iphi = string_rank(mphi);
    st.ephi = diag[iphi * C::NS - iphi * (iphi - 1) / 2];
    return st;
}

// Element e of a sector's start vector in the packed basis (see sector_guess).
template <class C, typename T>
__device__ inline T packed_guess(uchar2 ij, int e, int g, int sgn)
{
    const T z = (T)GUESS_NOISE * (T)guess_noise(ij.x * C::NS + ij.y);
    if (ij.x == ij.y) return sgn > 0 ? z + (e == g ? (T)2 : (T)0) : (T)0;
    return (T)1.4142135623730951 * (z + (e == g ? (T)1 : (T)0));
}

// ------------------------------------------------------------------ sigma, float32

// Walks this lane's share of the list entries y of its beta strings and of the rows J of
// Hs.  ab(Ib, y) and row(Ib, J) add to the accumulators, flush(Ib, part) stores and clears
// them.  With 20 strings, lanes 0-19 take the entries 0-7 of their own string, and lanes
// 20-31 the entries 8-11 of strings 0-11, then of 12-19: 8 rounds instead of the 12 that
// 20 lanes alone would need.  Otherwise L lanes share each string.
template <class C, class AB, class ROW, class FLUSH>
__device__ __forceinline__ void sector_rounds(AB ab, ROW row, FLUSH flush)
{
    const int lane = threadIdx.x & 31;
    if constexpr (C::HELP) {
        const bool main = lane < C::NS;
#pragma unroll 1
        for (int ph = 0; ph < 2; ++ph) {
            const int Ib = main ? lane : lane - C::NS + 12 * ph;
            if (Ib < C::NS) {
#pragma unroll 1
                for (int r = 0; r < 4; ++r) {
                    ab(Ib, (main ? 4 * ph : 8) + r);
                    row(Ib, main ? 8 * ph + 2 * r : 16 + r);
                    if (main) row(Ib, 8 * ph + 2 * r + 1);
                }
                if (!main) flush(Ib, 1);
            }
        }
        if (main) flush(lane, 0);
    } else {
        const int part = lane / C::NS, Ib = lane - part * C::NS;
        if (part < C::L) {
#pragma unroll 1
            for (int y = part; y < C::R; y += C::L) ab(Ib, y);
#pragma unroll 1
            for (int J = part; J < C::NS; J += C::L) row(Ib, J);
            flush(Ib, part);
        }
    }
}

// Position of c[J][m] in the coefficient matrix: columns m in pairs, so that one 8-byte load
// per column pair reads neighbouring words for neighbouring J.
template <class C>
__device__ __forceinline__ int c_at(int J, int m) { return ((m >> 1) * C::NS + J) * 2 + (m & 1); }

// Two float32 values in one register pair, for fma.rn.f32x2: one instruction for two
// multiply-adds (the rate of the pipe is the same, but these kernels wait for instructions).
__device__ __forceinline__ uint64_t pack2(float x, float y)
{
    return (uint64_t)__float_as_uint(y) << 32 | __float_as_uint(x);
}
__device__ __forceinline__ float2 unpack2(uint64_t v)
{
    return make_float2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
}
__device__ __forceinline__ void ffma2(uint64_t &d, uint64_t a, uint64_t b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// sector_rounds for the float32 sigma, which takes list entries and rows of Hs two at a time:
// ab(Ib, y) does entries y and y + 1 (y + 1 = R: the zero row), row(Ib, j) rows 2j and 2j + 1.
template <class C, class AB, class ROW, class FLUSH>
__device__ __forceinline__ void sector_rounds2(AB ab, ROW row, FLUSH flush)
{
    const int lane = threadIdx.x & 31;
    if constexpr (C::HELP) {
        const bool main = lane < C::NS;
#pragma unroll 1
        for (int ph = 0; ph < 2; ++ph) {
            const int Ib = main ? lane : lane - C::NS + 12 * ph;
            if (Ib < C::NS) {
#pragma unroll 1
                for (int r = 0; r < 2; ++r) {
                    ab(Ib, (main ? 4 * ph : 8) + 2 * r);
                    row(Ib, main ? 4 * ph + 2 * r : 8 + r);
                    if (main) row(Ib, 4 * ph + 2 * r + 1);
                }
                if (!main) flush(Ib, 1);
            }
        }
        if (main) flush(lane, 0);
    } else {
        const int part = lane / C::NS, Ib = lane - part * C::NS;
        if (part < C::L) {
#pragma unroll 1
            for (int y = 2 * part; y < C::R; y += 2 * C::L) ab(Ib, y);
#pragma unroll 1
            for (int j = part; j < C::NSH; j += C::L) row(Ib, j);
            flush(Ib, part);
        }
    }
}

// sigma of the packed vector t.  cm: c[J][m] at m NS + J.  Vs: [P][2P + 1], 1/2 V with rows (of
// the second index) 2 pair + neg, the sign applied, and a zero row.  Hs2: [NSH][NSP] pairs of
// rows of Hs.
template <class C>
__device__ __forceinline__ void sigma_sector(const SectorTables<C> &Tb, const float *Vs, const float2 *Hs2, float *cm,
                                             float *S, int sgn, const float (&t)[C::DH], float (&out)[C::DH])
{
    constexpr int VR = 2 * C::P + 1;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < C::DH; ++j) {
        const int e = lane + 32 * j;
        if (e < C::NH) {
            const uchar2 ij = Tb.tri[e];
            const float v = ij.x == ij.y ? t[j] : 0.70710678f * t[j];
            cm[ij.y * C::NS + ij.x] = v;
            cm[ij.x * C::NS + ij.y] = (float)sgn * v;
        }
    }
    __syncwarp();
    uint64_t acc[C::NS];
#pragma unroll
    for (int i = 0; i < C::NS; ++i) acc[i] = 0ull;
    const int flip = (1 - sgn) >> 1;  // (row J_y is read as column J_y: sgn times it)
    sector_rounds2<C>(
        [&](int Ib, int y) {
            const int e0 = Tb.list[Ib * C::R + y], J0 = e0 >> 8, row0 = (e0 & 255) ^ flip;
            int J1 = 0, row1 = 2 * C::P;
            if (C::R % 2 == 0 || y + 1 < C::R) {
                const int e1 = Tb.list[Ib * C::R + y + 1];
                J1 = e1 >> 8;
                row1 = (e1 & 255) ^ flip;
            }
            uint64_t c[C::NS];
#pragma unroll
            for (int m = 0; m < C::NS; ++m) c[m] = pack2(cm[m * C::NS + J0], cm[m * C::NS + J1]);
            static_for<C::P>([&](auto p) {
                const float v0 = Vs[p * VR + row0], v1 = Vs[p * VR + row1];
                const uint64_t v = pack2(v0, v1), w = pack2(-v0, -v1);
                static_for<C::NS>([&](auto I) {
                    constexpr int a = C::pair_hi(decltype(p)::value), b = C::pair_lo(decltype(p)::value);
                    constexpr int Jx = C::target(decltype(I)::value, a, b);
                    if constexpr (Jx >= 0) ffma2(acc[I], C::negative(decltype(I)::value, a, b) ? w : v, c[Jx]);
                });
            });
        },
        [&](int Ib, int j) {
            const int J1 = 2 * j + 1 < C::NS ? 2 * j + 1 : 2 * j;
            const uint64_t c = pack2((float)sgn * cm[2 * j * C::NS + Ib], (float)sgn * cm[J1 * C::NS + Ib]);
            const ulonglong2 *hs = (const ulonglong2 *)(Hs2 + j * C::NSP);
#pragma unroll
            for (int i = 0; i < (C::NS + 1) / 2; ++i) {
                const ulonglong2 v = hs[i];
                ffma2(acc[2 * i], c, v.x);
                if (2 * i + 1 < C::NS) ffma2(acc[2 * i + 1 < C::NS ? 2 * i + 1 : 0], c, v.y);
            }
        },
        [&](int Ib, int part) {
            float *s = S + (part * C::NS + Ib) * C::NSP;
#pragma unroll
            for (int i = 0; i < C::NS; ++i) {
                const float2 v = unpack2(acc[i]);
                s[i] = v.x + v.y;
                acc[i] = 0ull;
            }
        });
    __syncwarp();
#pragma unroll
    for (int j = 0; j < C::DH; ++j) {
        const int e = lane + 32 * j;
        out[j] = 0.f;
        if (e < C::NH) {
            const uchar2 ij = Tb.tri[e];
            float u = 0.f, w = 0.f;
#pragma unroll
            for (int p = 0; p < C::L; ++p) {
                u += S[(p * C::NS + ij.y) * C::NSP + ij.x];
                w += S[(p * C::NS + ij.x) * C::NSP + ij.y];
            }
            const float v = fmaf((float)sgn, w, u);  // (zero on the diagonal of the odd sector)
            out[j] = ij.x == ij.y ? v : 1.41421356f * v;
        }
    }
    __syncwarp();
}

// ------------------------------------------------------------------ sigma of an anchor, integers

// H x0 of an anchor to float64 accuracy on the integer pipe.  A float64 multiply-add costs
// about 12 times a wide integer one here (1.67 against 18-23 lanes per clock and SM, measured with
// operands that change), so V and Hs are kept as 55-bit fixed-point numbers in two limbs (to_fixed)
// and the anchor as integers c 2^28 (it may be any vector near the float32 one: r0 belongs to the
// integer one): each term is two 32 x 32 + 64 -> 64 bit multiply-adds, exact.  The sums
// cannot overflow: by Cauchy-Schwarz the absolute terms of one element add up to at most
// (12 * 3 + 9) |c| |V|max < 2^5.5 * 2^28 * 2^27 for a unit vector (a list of 12 entries holds
// its own string 3 times, every other string once).  The result is rounded once, to 2^-55 of
// the largest element of V and Hs.  Taken once or twice per tuple, so the loops are kept rolled:
// unrolled like the float32 sigma they were 37 KB of code for the same number of instructions.  The diagonal of Hs
// is left to the caller (it would set the scale).
template <class C>
__device__ __forceinline__ void sigma_anchor(const SectorTables<C> &Tb, const int2 *Vf, const int2 *Hsf, const int *cm,
                                             long long *S, int sgn)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int h = lane; h < C::NH; h += 32) {
        const uchar2 ij = Tb.tri[h];
        long long hi = 0, lo = 0;
        const uint16_t *la = Tb.list + ij.x * C::R, *lb = Tb.list + ij.y * C::R;
#pragma unroll 1
        for (int x = 0; x < C::R; ++x) {
            const int ea = la[x];
            const int2 *v = Vf + ((ea & 255) >> 1) * C::P;
            const int *c = cm + (ea >> 8) * C::NS;
#pragma unroll 2
            for (int y = 0; y < C::R; ++y) {
                const int eb = lb[y], m = -((ea ^ eb) & 1);
                const int2 w = v[(eb & 255) >> 1];
                const int q = (c[eb >> 8] ^ m) - m;
                hi += (long long)w.x * q;
                lo += (long long)w.y * q;
            }
        }
#pragma unroll 2
        for (int J = 0; J < C::NS; ++J) {  // (Hs C)[Ia][Ib] + (C Hs)[Ia][Ib], without the diagonal of Hs
            const int r = min(ij.x, J), s = max(ij.x, J), t = min(ij.y, J), u = max(ij.y, J);
            const int2 a = Hsf[r * C::NS - r * (r - 1) / 2 + s - r], b = Hsf[t * C::NS - t * (t - 1) / 2 + u - t];
            const int p = cm[J * C::NS + ij.y], q = cm[ij.x * C::NS + J];
            hi += (long long)a.x * p;
            lo += (long long)a.y * p;
            hi += (long long)b.x * q;
            lo += (long long)b.y * q;
        }
        S[h] = hi + ((lo + (1LL << 27)) >> 28);
    }
    __syncwarp();
}

// Sums of the K (a power of two) values over the warp; every lane gets all totals.  Each
// step halves the values that a lane carries, so K = 8 takes 9 additions instead of 40.
template <int K, typename T>
__device__ __forceinline__ void warp_sum_n(T (&v)[K])
{
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int m = K / 2; m >= 1; m >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < m; ++i) {
            const T send = up ? v[i] : v[i + m];
            const T keep = up ? v[i + m] : v[i];
            v[i] = keep + __shfl_xor_sync(FULL, send, o);
        }
        o >>= 1;
    }
#pragma unroll
    for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(FULL, v[0], o);
    const T s = v[0];
    // value i was kept by the lanes whose leading bits spell i
#pragma unroll
    for (int i = 0; i < K; ++i) v[i] = __shfl_sync(FULL, s, i * (32 / K));
}

// ------------------------------------------------------------------ Davidson on packed sector vectors

// The warp solver's Davidson (davidson_warp, plain and anchored) on packed vectors; sigma(t,
// ht) forms the image of t.  The dot products of a stage are reduced together, and the second
// orthogonalisation pass is taken only when the first one cancelled (less than half of |t|^2
// left; with more left, one pass is orthogonal to within a few rounding errors).
template <class C, class SIGMA>
__device__ __forceinline__ PhaseOut davidson_sector(SIGMA sigma, const float *dg, float (&x)[C::DH], double tol,
                                                    int min_iter, int max_iter, const Anchor &an, bool anchored)
{
    constexpr int DH = C::DH;
    const int lane = threadIdx.x & 31;
    const float *x0s = an.x0, *r0s = an.r0;
    const float shift = an.shift, shift_lo = an.shift_lo, x0x0 = an.x0x0;  // (shift 0 when plain)
    float hx[DH], p[DH], hp[DH], t[DH], ht[DH], x0[DH], r0[DH];
    PhaseOut o;
    o.nsig = 0;
    o.status = MBE_STATUS_OK;
    o.dnorm = 0.0;
    float lam = 0.f;
    int first = opaque(!anchored);
#pragma unroll
    for (int j = 0; j < DH; ++j) p[j] = hp[j] = hx[j] = 0.f;
    if (!anchored) {
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < DH; ++j) s += x[j] * x[j];
        s = warp_sum(s);
        const float inv = 1.f / sqrtf(s);
#pragma unroll
        for (int j = 0; j < DH; ++j) t[j] = x[j] = x[j] * inv;
    } else {
#pragma unroll
        for (int j = 0; j < DH; ++j) x[j] = 0.f;
    }
    bool have_p = false;
    float best = 3e38f, rn = 0.f, xx = 1.f;
    int stall = 0;
    for (int it = 0;;) {
        const bool anch = opaque(anchored);
        if (!first) {
            float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // |r|^2, x.t, p.t, |t|^2, |x|^2
#pragma unroll
            for (int j = 0; j < DH; ++j) {
                const int e = lane + 32 * j;
                t[j] = x0[j] = 0.f;
                if (e < C::NH) {
                    float r0j = 0.f;
                    if (anch) {
                        x0[j] = x0s[e];
                        r0j = r0s[e];
                    }
                    const float xj = x0[j] + x[j], r = (r0j + hx[j]) - lam * xj;
                    float den = dg[e] - shift - lam;
                    if (fabsf(den) < 1e-4f) den = den >= 0.f ? 1e-4f : -1e-4f;
                    t[j] = __fdividef(r, den);
                    v[0] += r * r;
                    v[1] += xj * t[j];
                    v[2] += p[j] * t[j];
                    v[3] += t[j] * t[j];
                    v[4] += xj * xj;
                }
            }
            warp_sum_n<8>(v);
            rn = sqrtf(v[0]);
            if (!isfinite(rn) || !isfinite(lam)) {
                o.status = MBE_STATUS_NONFINITE;
                break;
            }
            if (rn <= (float)tol && it >= min_iter) break;
            if (it >= max_iter) {
                o.status = MBE_STATUS_MAXITER;
                break;
            }
            if (rn < 0.9f * best) {
                best = rn;
                stall = 0;
            } else if (++stall >= 3) {
                break;
            }
            if (anch) xx = v[4];
            // orthonormalise t against x and p
            float ax = v[1] / xx, ap = v[2], tt = 0.f;
#pragma unroll
            for (int j = 0; j < DH; ++j) {
                t[j] -= ax * (x0[j] + x[j]) + ap * p[j];
                tt += t[j] * t[j];
            }
            tt = warp_sum(tt);
            if (!(tt >= 0.5f * v[3])) {
                float w[2] = {0.f, 0.f};
#pragma unroll
                for (int j = 0; j < DH; ++j) {
                    w[0] += (x0[j] + x[j]) * t[j];
                    w[1] += p[j] * t[j];
                }
                warp_sum_n<2>(w);
                ax = w[0] / xx;
                ap = w[1];
                tt = 0.f;
#pragma unroll
                for (int j = 0; j < DH; ++j) {
                    t[j] -= ax * (x0[j] + x[j]) + ap * p[j];
                    tt += t[j] * t[j];
                }
                tt = warp_sum(tt);
            }
            const float tn = sqrtf(tt);
            if (anch ? !(tn > 1e-4f * sqrtf(v[3])) : !(tn > tiny_norm<float>())) break;  // nothing left to add
            const float tinv = 1.f / tn;
#pragma unroll
            for (int j = 0; j < DH; ++j) t[j] *= tinv;
        }
        sigma(t, ht);
        ++o.nsig;
        if (first) {
            float xh = 0.f;
#pragma unroll
            for (int j = 0; j < DH; ++j) {
                hx[j] = ht[j];
                xh += x[j] * ht[j];
            }
            lam = warp_sum(xh);
            first = opaque(0);
            continue;
        }
        ++it;
        // G = [x p t]^T A [x p t]; a coupling x.(A v) is formed as v.r0 + d.(A v)
        float g[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < DH; ++j) {
            const int e = lane + 32 * j;
            r0[j] = anch && e < C::NH ? r0s[e] : 0.f;
            ht[j] = (ht[j] - shift * t[j]) - shift_lo * t[j];
            g[0] += x[j] * (2.f * r0[j] + hx[j]);
            g[1] += p[j] * r0[j] + x[j] * hp[j];
            g[2] += t[j] * r0[j] + x[j] * ht[j];
            g[3] += p[j] * hp[j];
            g[4] += p[j] * ht[j];
            g[5] += t[j] * ht[j];
        }
        warp_sum_n<8>(g);
        float G[3][3];
        const float sx = anch ? 1.f / sqrtf(xx) : 1.f;
        G[0][0] = g[0] * sx * sx;
        G[0][1] = G[1][0] = g[1] * sx;
        G[0][2] = G[2][0] = g[2] * sx;
        G[1][1] = g[3];
        G[1][2] = G[2][1] = g[4];
        G[2][2] = g[5];
        float y[3];
        eig3<float>(G, have_p, y);
        const float y0 = y[0] * sx, y1 = y[1], y2 = y[2];
        const float w2 = y1 * y1 + y2 * y2;
        float q0 = -w2 * y0, q1 = y1 - w2 * y1, q2 = y2 - w2 * y2;
        const float zn = sqrtf(q0 * q0 * xx + q1 * q1 + q2 * q2);
        have_p = zn > (anch ? 1e-30f : tiny_norm<float>() * 1e-3f);
        const float zi = have_p ? 1.f / zn : 0.f;
        q0 *= zi;
        q1 *= zi;
        q2 *= zi;
        float n[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < DH; ++j) {
            const int e = lane + 32 * j;
            x0[j] = anch && e < C::NH ? x0s[e] : 0.f;
            const float nx = y0 * x[j] + y1 * p[j] + y2 * t[j];
            const float nhx = y0 * hx[j] + y1 * hp[j] + y2 * ht[j];
            p[j] = q0 * (x0[j] + x[j]) + q1 * p[j] + q2 * t[j];
            hp[j] = q0 * (r0[j] + hx[j]) + q1 * hp[j] + q2 * ht[j];
            x[j] = nx;
            hx[j] = nhx;
            n[0] += nx * nx;
            n[1] += nx * nhx;
            n[2] += nx * r0[j];
            n[3] += nx * x0[j];
        }
        warp_sum_n<4>(n);
        float sc;
        if (anch) {
            sc = 1.f / y0;
            // mu = (x.Ax) / (x.x), x = x0 + sc nx, A x = r0 + sc A nx, x0.r0 = 0
            lam = (sc * 2.f * n[2] + sc * sc * n[1]) / (x0x0 + sc * 2.f * n[3] + sc * sc * n[0]);
            o.dnorm = (double)(fabsf(sc) * sqrtf(n[0]));
        } else {
            sc = 1.f / sqrtf(n[0]);
            lam = n[1] / n[0];
        }
#pragma unroll
        for (int j = 0; j < DH; ++j) {
            x[j] *= sc;
            hx[j] *= sc;
        }
    }
    o.lambda = (double)lam;
    o.rnorm = (double)rn;
    return o;
}

// ------------------------------------------------------------------ mixed kernel

// Shared memory of one warp of the mixed sector solver.
template <class C>
struct SectorMixed {
    int2 Vf[C::P * C::P];  // float64 V (packed) during set-up, then fixed point
    long long Hsf[C::NH];  // float64 Hs during set-up, then fixed point (off-diagonal)
    double hd[C::NS];      // diagonal of Hs
    union {                // sigma partial sums; set-up scratch
        alignas(16) float S[C::L * C::NS * C::NSP];
        long long S64[C::NH];
        struct {
            double diag[C::NH], h[C::P];
        } su;
    } s;
    union {
        alignas(16) float cm[2 * C::NSH * C::NS];
        int cmi[2 * C::NSH * C::NS];
        double dsum[C::NS * C::n];
    } c;
    alignas(16) float2 Hs2[C::NSH * C::NSP];  // rows of Hs in pairs
    float Vs[C::P * (2 * C::P + 1)];          // 1/2 V, both signs
    float dg[C::NH];
    union {
        struct {
            float x0[C::NH], r0[C::NH];
        };
        double Vp[C::PT];  // set-up: float64 V
    };
    int A[8];
};

constexpr int SECTOR_WARPS = 4;  // most warps per block (mbe_tuning.warp_warps)

// Mixed precision (see k_casci_warp_mixed for the method: float32 Davidson, anchored
// refinements), one warp per tuple of the class (n, k).
template <class C>
__device__ __forceinline__ void sector_mixed_tuples(const BatchArgs &a, int bucket)
{
    extern __shared__ __align__(16) char smem[];
    SectorTables<C> &T = *(SectorTables<C> *)smem;
    SectorMixed<C> &W = ((SectorMixed<C> *)(smem + al16((int)sizeof(SectorTables<C>))))[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    build_tables<C>(T, a.cls[C::k]);
    const int64_t begin = a.bucket_off[bucket];
    const int64_t cnt = a.bucket_off[bucket + 1] - begin;
    for (;;) {
        unsigned long long pos = 0;
        if (lane == 0) pos = atomicAdd(&a.counters[bucket], 1ULL);
        pos = __shfl_sync(FULL, pos, 0);
        if ((int64_t)pos >= cnt) break;
        const int64_t t = a.perm[begin + (int64_t)pos];
        if (lane == 0) build_A(a, t, W.A);
        __syncwarp();
        double *Vp = W.Vp, *Hsp = (double *)W.Hsf;
        const SectorStart st =
            sector_setup<C>(a, T, W.A, Vp, Hsp, W.hd, W.s.su.h, W.c.dsum, W.s.su.diag);
        int vmax = 0;
#pragma unroll 1
        for (int e = lane; e < C::PT; e += 32) {
            const uchar2 xy = T.ptri[e];
            const double v = Vp[e];
            const float f = 0.5f * (float)v;
            constexpr int VR = 2 * C::P + 1;
            float *s = W.Vs + xy.y * VR + 2 * xy.x;
            s[0] = f;
            s[1] = -f;
            s = W.Vs + xy.x * VR + 2 * xy.y;
            s[0] = f;
            s[1] = -f;
            vmax = max(vmax, high_word(v));
        }
#pragma unroll 1
        for (int e = lane; e < C::NH; e += 32) {
            const uchar2 ij = T.tri[e];
            const double v = Hsp[e];
            float *hs = (float *)W.Hs2;
            hs[((ij.x >> 1) * C::NSP + ij.y) * 2 + (ij.x & 1)] = (float)v;
            hs[((ij.y >> 1) * C::NSP + ij.x) * 2 + (ij.y & 1)] = (float)v;
            if (ij.x != ij.y) vmax = max(vmax, high_word(v));
            W.dg[e] = (float)W.s.su.diag[e];
        }
        for (int p = lane; p < C::P; p += 32) W.Vs[p * (2 * C::P + 1) + 2 * C::P] = 0.f;
        if (C::NS & 1)  // the last row's partner
            for (int i = lane; i < C::NS; i += 32) W.Hs2[(C::NSH - 1) * C::NSP + i].y = 0.f;
        const int E = fixed_exponent(vmax);
        const double scale = pow2(55 - E);
        __syncwarp();
#pragma unroll 1
        for (int e = lane; e < C::PT; e += 32) {
            const uchar2 xy = T.ptri[e];
            W.Vf[xy.x * C::P + xy.y] = W.Vf[xy.y * C::P + xy.x] = to_fixed(Vp[e], scale);
        }
#pragma unroll 1
        for (int e = lane; e < C::NH; e += 32) {
            const uchar2 ij = T.tri[e];
            ((int2 *)W.Hsf)[e] = ij.x == ij.y ? make_int2(0, 0) : to_fixed(Hsp[e], scale);
        }
        __syncwarp();  // the float64 diagonal is dead from here
        int n32 = 0, n64 = 0;
        bool redo = false, degen = false;
        double lam = 0.0, lam32 = 0.0;
        // one copy of the sector's Davidson: two inlined copies, both hot on an SM,
        // overflow the instruction cache and slow every phase of every warp
#pragma unroll 1
        for (int sector = opaque(0); sector < 2 && !redo; ++sector) {
            if (sector == 1 && a.even_only) break;
            const int sgn = opaque(sector == 0 ? 1 : -1), g = sector == 0 ? st.g : st.go;
            float xv[C::DH];
#pragma unroll
            for (int j = 0; j < C::DH; ++j) {
                const int e = lane + 32 * j;
                xv[j] = e < C::NH ? packed_guess<C, float>(T.tri[e], e, g, sgn) : 0.f;
            }
            auto sigma = [&](const float(&tv)[C::DH], float(&out)[C::DH]) {
                sigma_sector<C>(T, W.Vs, W.Hs2, W.c.cm, W.s.S, sgn, tv, out);
            };
            // plain float32 passes (the first sector one to tol_switch; the second one
            // to SECTOR_TOL, then tol_switch, decided against the first's float32
            // eigenvalue), then anchored refinements; one call site of the Davidson
            int passes = 0, anchors = 0;
            bool lose = false, fail = false, done = false;
            double th = 0.0, lam_s = 0.0;
            Anchor an{W.x0, W.r0, 0.f, 0.f, 1.f};
            for (;;) {
                const bool anchored = opaque(anchors) > 0;
                const double tl = anchored ? a.tol : ((sector == 0 || passes == 1) ? a.tol_switch : SECTOR_TOL);
                const PhaseOut o = davidson_sector<C>(sigma, W.dg, xv, tl, anchored ? a.min_fp64 : 0, a.max_iter, an,
                                                      anchored);
                n32 += o.nsig;
                if (!anchored) {
                    const bool finite = o.status != MBE_STATUS_NONFINITE;
                    if (sector == 0) {
                        lam32 = o.lambda;
                        if (!finite) {
                            fail = true;
                            break;
                        }
                    } else {
                        lose = !finite || sector_loses(o.lambda, o.rnorm, lam32, a.tol_switch);
                        if (lose) break;
                    }
                    ++passes;
                    if (sector == 1 && passes < 2) continue;
                } else {
                    lam_s = th + o.lambda;
                    if (o.status == MBE_STATUS_NONFINITE) {
                        fail = true;
                        break;
                    }
                    if (o.rnorm <= a.tol && o.dnorm <= MIX_DMAX) {
                        done = true;
                        break;
                    }
                    if (anchors >= MIX_ANCHORS) {
                        fail = true;
                        break;
                    }
                    // stalled short of tol: re-anchor at x0 + d
#pragma unroll
                    for (int j = 0; j < C::DH; ++j) {
                        const int e = lane + 32 * j;
                        xv[j] = e < C::NH ? W.x0[e] + xv[j] : 0.f;
                    }
                }
                // Anchor: xv rounded to integers c 2^28 (|c| <= 1: a unit vector), its image
                // from the integer sigma, theta0, and x0 and r0 = (H - theta0) x0 in float32.
                // x0 itself enters the refinement only multiplied by mu or in the
                // orthogonalisation, so its float32 rounding is of second order; r0 belongs
                // to the integer vector exactly.
                float nn = 0.f;
#pragma unroll
                for (int j = 0; j < C::DH; ++j) nn += xv[j] * xv[j];
                const float inv = 1.f / sqrtf(warp_sum(nn));
#pragma unroll
                for (int j = 0; j < C::DH; ++j) {
                    const int e = lane + 32 * j;
                    if (e < C::NH) {
                        const uchar2 ij = T.tri[e];
                        const float f = xv[j] * inv * (ij.x == ij.y ? 268435456.f : 0.70710678f * 268435456.f);
                        const int q = __float2int_rn(fminf(fmaxf(f, -268435456.f), 268435456.f));
                        W.c.cmi[ij.x * C::NS + ij.y] = q;
                        W.c.cmi[ij.y * C::NS + ij.x] = sgn * q;
                    }
                }
                __syncwarp();
                sigma_anchor<C>(T, W.Vf, (const int2 *)W.Hsf, W.c.cmi, W.s.S64, sgn);
                ++n64;
                double xs = 0.0, xx = 0.0;
                double s0[C::DH], c0[C::DH];
#pragma unroll
                for (int j = 0; j < C::DH; ++j) {
                    const int e = lane + 32 * j;
                    s0[j] = c0[j] = 0.0;
                    if (e < C::NH) {
                        const uchar2 ij = T.tri[e];
                        const double wt = ij.x == ij.y ? 1.0 : 1.4142135623730951;
                        c0[j] = (double)W.c.cmi[ij.x * C::NS + ij.y] * (wt * pow2(-28));
                        s0[j] = fma(W.hd[ij.x] + W.hd[ij.y], c0[j], ij.x == ij.y && sgn < 0 ? 0.0 : (double)W.s.S64[e] * (wt * pow2(E - 55)));
                        xs = fma(c0[j], s0[j], xs);
                        xx = fma(c0[j], c0[j], xx);
                    }
                }
                xs = warp_sum(xs);
                xx = warp_sum(xx);
                th = xs / xx;
#pragma unroll
                for (int j = 0; j < C::DH; ++j) {
                    const int e = lane + 32 * j;
                    if (e < C::NH) {
                        W.x0[e] = (float)c0[j];
                        W.r0[e] = (float)(s0[j] - th * c0[j]);
                    }
                }
                __syncwarp();
                an.shift = (float)th;
                an.shift_lo = (float)(th - (double)an.shift);
                an.x0x0 = (float)xx;
                ++anchors;
            }
            if (sector == 0) {
                if (fail || !done) redo = true;
                lam = lam_s;
            } else if (!lose) {
                if (fail || !done) redo = true;
                degen = fabs(lam_s - lam) <= DEGEN_TOL;
                if (lam_s < lam) lam = lam_s;
            }
            __syncwarp();
        }
        if (lane == 0) {
            if (redo) {
                a.pstate[2 * t] = PS_REDO;
                a.pstate[2 * t + 1] = n32;
            } else {
                a.pstate[2 * t] = PS_DONE;
                store_result(a, t, lam - st.ephi - a.e_ref_corr, with_degeneracy(MBE_STATUS_OK, degen), n64, n32);
            }
        }
        __syncwarp();
    }
}

template <class C>
__global__ void __launch_bounds__(SECTOR_WARPS * 32, C::DH > 4 ? 3 : 4) k_sector_mixed(BatchArgs a, int bucket)
{
    sector_mixed_tuples<C>(a, bucket);
}

// Whether a bucket has more than `least` tuples left, for the whole block (a barrier).
__device__ __forceinline__ bool bucket_open(const BatchArgs &a, const unsigned long long *counters, int bucket, unsigned least)
{
    const unsigned long long cnt = (unsigned long long)(a.bucket_off[bucket + 1] - a.bucket_off[bucket]);
    return __syncthreads_or(threadIdx.x == 0 && *(const volatile unsigned long long *)(counters + bucket) + least < cnt);
}

// Two classes in one launch (buckets b and b + 1): the first half of the blocks starts with the first
// class, the second half with the second (so that every SM gets both), and a block whose own class is
// done goes on with the other one where more is left than that one's blocks take in a round (fewer
// would only crowd on some SMs: 600 tuples of one class in float64 289 -> 351 us).
template <class C0, class C1>
__global__ void __launch_bounds__(SECTOR_WARPS * 32, 4) k_sector_mixed_pair(BatchArgs a, int b)
{
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        const unsigned half = gridDim.x / 2, second = (blockIdx.x >= half) != (pass == 1);
        if (!bucket_open(a, a.counters, b + second, pass ? half * (blockDim.x >> 5) : 0)) continue;
        if (second)
            sector_mixed_tuples<C1>(a, b + 1);
        else
            sector_mixed_tuples<C0>(a, b);
    }
}

}  // namespace mbe
