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
    for (int i = threadIdx.x; i < C::NS * C::R; i += blockDim.x) {
        const int e = ci.table[i];
        T.list[i] = (uint16_t)(entry_J(e) << 8 | (e & 0xff));
    }
    for (int i = threadIdx.x; i < C::NS; i += blockDim.x) {
        T.str[i] = ci.strings[i];
        for (int j = i; j < C::NS; ++j)
            T.tri[i * C::NS - i * (i - 1) / 2 + j - i] = make_uchar2((unsigned char)i, (unsigned char)j);
    }
    for (int x = threadIdx.x; x < C::P; x += blockDim.x) {
        const int a = C::pair_hi(x);
        T.pq[x] = make_uchar2((unsigned char)a, (unsigned char)(x - a * (a + 1) / 2));
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
        for (; s; s &= s - 1u) c ^= 1;
        return c;
    };
    auto between = [](int a, int b) {
        const int lo = a < b ? a : b, hi = a < b ? b : a;
        return ((1u << hi) - 1u) & ~((2u << lo) - 1u);
    };
    uint32_t from = I & ~J, to = J & ~I;
    double v = 0.0;
    if (from == 0u) {
        for (uint32_t a = I; a; a &= a - 1u) {
            const int p = low(a);
            v += h(p, p);
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

// Exponent E of the fixed-point scale: 2^E is the power of two above the warp's largest v.
__device__ inline int fixed_exponent(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(FULL, v, o));
    const int E = (int)((__double_as_longlong(v) >> 52) & 0x7ff) - 1022;
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
#pragma unroll 4
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
        for (uint32_t m = mphi; m; m &= m - 1u) {
            const int i = __ffs((int)m) - 1;
            v -= 2.0 * Vp[tri_index(lane, pair_index(i, i))] - Vp[tri_index(pair_index(p, i), pair_index(i, q))];
        }
        h[lane] = v;
    }
    for (int e = lane; e < C::NS * C::n; e += 32) {  // sum_{p in I} (pp|qq)
        const int I = e / C::n, q = e - I * C::n;
        double v = 0.0;
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
    double best = 1e300, best_o = 1e300;
    SectorStart st;
    st.g = st.go = 0x7fffffff;
#pragma unroll 1
    for (int e = lane; e < C::NH; e += 32) {
        const uchar2 ij = T.tri[e];
        double v = hd[ij.x] + hd[ij.y];
        for (uint32_t m = T.str[ij.y]; m; m &= m - 1u) v += dsum[ij.x * C::n + __ffs((int)m) - 1];
        diag[e] = v;
        if (v < best) {
            best = v;
            st.g = e;
        }
        if (ij.x != ij.y && v < best_o) {
            best_o = v;
            st.go = e;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {  // the lowest element, ties to the lowest index
        double ov = __shfl_xor_sync(FULL, best, o);
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

// Writes the packed sector vector t as the full coefficient matrix.
template <class C, typename T>
__device__ __forceinline__ void expand(const SectorTables<C> &Tb, const T (&t)[C::DH], int sgn, T *cm)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < C::DH; ++j) {
        const int e = lane + 32 * j;
        if (e < C::NH) {
            const uchar2 ij = Tb.tri[e];
            const T v = ij.x == ij.y ? t[j] : (T)0.70710678118654752 * t[j];
            cm[c_at<C>(ij.x, ij.y)] = v;
            cm[c_at<C>(ij.y, ij.x)] = sgn > 0 ? v : -v;
        }
    }
}

// V2: [PH][2P] pairs of columns of 1/2 V, rows 2 pair + neg with the sign applied.
template <class C>
__device__ __forceinline__ void sigma_sector(const SectorTables<C> &Tb, const float2 *V2, const float *Hs, float *cm,
                                             float *S, int sgn, const float (&t)[C::DH], float (&out)[C::DH])
{
    const int lane = threadIdx.x & 31;
    expand<C, float>(Tb, t, sgn, cm);
    __syncwarp();
    const float2 *cm2 = (const float2 *)cm;
    float acc[C::NSP];
#pragma unroll
    for (int i = 0; i < C::NSP; ++i) acc[i] = 0.f;
    sector_rounds<C>(
        [&](int Ib, int y) {
            // (row J_y read as column J_y: sgn times it)
            const int e = Tb.list[Ib * C::R + y], J = e >> 8, row = (e & 255) ^ (sgn < 0 ? 1 : 0);
            float c[2 * C::NSH];
#pragma unroll
            for (int m = 0; m < C::NSH; ++m) {
                const float2 v = cm2[m * C::NS + J];
                c[2 * m] = v.x;
                c[2 * m + 1] = v.y;
            }
            static_for<C::PH>([&](auto ph) {
                const float2 v2 = V2[ph * 2 * C::P + row];
                static_for<2>([&](auto half) {
                    constexpr int p = 2 * decltype(ph)::value + decltype(half)::value;
                    if constexpr (p < C::P) {
                        const float v = decltype(half)::value ? v2.y : v2.x;
                        static_for<C::NS>([&](auto I) {
                            constexpr int a = C::pair_hi(p), b = C::pair_lo(p);
                            constexpr int Jx = C::target(decltype(I)::value, a, b);
                            if constexpr (Jx >= 0) {
                                if constexpr (C::negative(decltype(I)::value, a, b))
                                    acc[I] = fmaf(-v, c[Jx], acc[I]);
                                else
                                    acc[I] = fmaf(v, c[Jx], acc[I]);
                            }
                        });
                    }
                });
            });
        },
        [&](int Ib, int J) {
            float c = cm[c_at<C>(Ib, J)];
            c = sgn > 0 ? c : -c;
            const float4 *hs = (const float4 *)(Hs + J * C::NSP);
#pragma unroll
            for (int i = 0; i < C::NSP / 4; ++i) {
                if (4 * i >= C::NS) break;
                const float4 v = hs[i];
                acc[4 * i] = fmaf(c, v.x, acc[4 * i]);
                acc[4 * i + 1] = fmaf(c, v.y, acc[4 * i + 1]);
                acc[4 * i + 2] = fmaf(c, v.z, acc[4 * i + 2]);
                acc[4 * i + 3] = fmaf(c, v.w, acc[4 * i + 3]);
            }
        },
        [&](int Ib, int part) {
            float4 *s = (float4 *)(S + (part * C::NS + Ib) * C::NSP);
#pragma unroll
            for (int i = 0; i < C::NSP / 4; ++i) {
                s[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
                acc[4 * i] = acc[4 * i + 1] = acc[4 * i + 2] = acc[4 * i + 3] = 0.f;
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
            const float v = sgn > 0 ? u + w : u - w;
            out[j] = ij.x == ij.y ? (sgn > 0 ? v : 0.f) : 1.41421356f * v;
        }
    }
    __syncwarp();
}

// ------------------------------------------------------------------ sigma of an anchor, integers

// H x0 of an anchor to float64 accuracy on the integer pipe.  A float64 multiply-add costs
// about 36 times a wide integer one here (1.67 against 60 lanes per clock and SM, measured),
// so V and Hs are kept as 55-bit fixed-point numbers in two limbs (to_fixed) and the anchor
// as integers c 2^28: each term is two 32 x 32 + 64 -> 64 bit multiply-adds, exact.  The sums
// cannot overflow: by Cauchy-Schwarz the absolute terms of one element add up to at most
// (12 * 3 + 5) |c| |V|max < 2^5.4 * 2^28 * 2^27 for a unit vector (a list of 12 entries holds
// its own string 3 times, every other string once).  The result is rounded once, to 2^-55 of
// the largest element of V and Hs.  The diagonal of Hs
// is left to the caller (it would set the scale).
template <class C>
__device__ __forceinline__ void sigma_anchor(const SectorTables<C> &Tb, const int2 *Vf, const int2 *Hsf, const int *cm,
                                             long long *S, int sgn)
{
    const int lane = threadIdx.x & 31;
    const int2 *cm2 = (const int2 *)cm;
    constexpr int ST = C::NS | 1;
    if (lane < C::NS) {
        const int Ib = lane;
        long long hi[C::NS], lo[C::NS];
#pragma unroll
        for (int i = 0; i < C::NS; ++i) hi[i] = lo[i] = 0;
#pragma unroll 1
        for (int y = 0; y < C::R; ++y) {
            const int e = Tb.list[Ib * C::R + y], J = e >> 8, pr = (e & 255) >> 1, m = -((e & 1) ^ (sgn < 0 ? 1 : 0));
            int c[2 * C::NSH];
#pragma unroll
            for (int i = 0; i < C::NSH; ++i) {
                const int2 v = cm2[i * C::NS + J];
                c[2 * i] = (v.x ^ m) - m;
                c[2 * i + 1] = (v.y ^ m) - m;
            }
            static_for<C::P>([&](auto p) {
                const int2 v = Vf[tri_index(pr, p)];
                static_for<C::NS>([&](auto I) {
                    constexpr int a = C::pair_hi(decltype(p)::value), b = C::pair_lo(decltype(p)::value);
                    constexpr int Jx = C::target(decltype(I)::value, a, b);
                    if constexpr (Jx >= 0) {
                        constexpr bool neg = C::negative(decltype(I)::value, a, b);
                        hi[I] += (long long)(neg ? -v.x : v.x) * c[Jx];
                        lo[I] += (long long)(neg ? -v.y : v.y) * c[Jx];
                    }
                });
            });
        }
#pragma unroll 1
        for (int J = 0; J < C::NS; ++J) {
            int c = cm[c_at<C>(Ib, J)];
            c = sgn > 0 ? c : -c;
            static_for<C::NS>([&](auto I) {
                const int r = J < I ? J : (int)I, s = J < I ? (int)I : J;
                const int2 v = Hsf[r * C::NS - r * (r - 1) / 2 + s - r];
                hi[I] += (long long)v.x * c;
                lo[I] += (long long)v.y * c;
            });
        }
#pragma unroll
        for (int i = 0; i < C::NS; ++i) S[Ib * ST + i] = hi[i] + ((lo[i] + (1LL << 27)) >> 28);
    }
    __syncwarp();
}

// ------------------------------------------------------------------ Davidson on packed sector vectors

// The warp solver's Davidson (davidson_warp, plain and anchored) on packed vectors; sigma(t,
// ht) forms the image of t.
template <class C, class SIGMA>
__device__ __forceinline__ PhaseOut davidson_sector(SIGMA sigma, const float *dg, float (&x)[C::DH], double tol,
                                                    int min_iter, int max_iter, const Anchor *an)
{
    constexpr int DH = C::DH;
    const int lane = threadIdx.x & 31;
    const bool anch = an != nullptr;
    const float *x0s = anch ? an->x0 : nullptr, *r0s = anch ? an->r0 : nullptr;
    const float shift = anch ? an->shift : 0.f, shift_lo = anch ? an->shift_lo : 0.f;
    const float x0x0 = anch ? an->x0x0 : 0.f;
    float hx[DH], p[DH], hp[DH], t[DH], ht[DH], x0[DH], r0[DH];
    PhaseOut o;
    o.nsig = 0;
    o.status = MBE_STATUS_OK;
    o.dnorm = 0.0;
    float lam = 0.f;
    bool first = !anch;
#pragma unroll
    for (int j = 0; j < DH; ++j) p[j] = hp[j] = hx[j] = 0.f;
    if (!anch) {
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
        if (!first) {
            float rr = 0.f, t0n = 0.f;
#pragma unroll
            for (int j = 0; j < DH; ++j) {
                const int e = lane + 32 * j;
                t[j] = x0[j] = r0[j] = 0.f;
                if (e < C::NH) {
                    if (anch) {
                        x0[j] = x0s[e];
                        r0[j] = r0s[e];
                    }
                    const float r = (r0[j] + hx[j]) - lam * (x0[j] + x[j]);
                    rr += r * r;
                    float den = dg[e] - shift - lam;
                    if (fabsf(den) < 1e-4f) den = den >= 0.f ? 1e-4f : -1e-4f;
                    t[j] = r / den;
                    t0n += t[j] * t[j];
                }
            }
            rn = sqrtf(warp_sum(rr));
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
            if (anch) {
                float s = 0.f;
#pragma unroll
                for (int j = 0; j < DH; ++j) {
                    const float xj = x0[j] + x[j];
                    s += xj * xj;
                }
                t0n = sqrtf(warp_sum(t0n));
                xx = warp_sum(s);
            }
            // orthonormalise t against x and p (two passes)
#pragma unroll 1
            for (int pass = 0; pass < 2; ++pass) {
                float ax = 0.f, ap = 0.f;
#pragma unroll
                for (int j = 0; j < DH; ++j) {
                    ax += (x0[j] + x[j]) * t[j];
                    ap += p[j] * t[j];
                }
                ax = warp_sum(ax) / xx;
                ap = warp_sum(ap);
#pragma unroll
                for (int j = 0; j < DH; ++j) t[j] -= ax * (x0[j] + x[j]) + ap * p[j];
            }
            float tt = 0.f;
#pragma unroll
            for (int j = 0; j < DH; ++j) tt += t[j] * t[j];
            const float tn = sqrtf(warp_sum(tt));
            if (anch ? !(tn > 1e-4f * t0n) : !(tn > tiny_norm<float>())) break;  // nothing left to add
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
            first = false;
            continue;
        }
        ++it;
        // G = [x p t]^T A [x p t]; a coupling x.(A v) is formed as v.r0 + d.(A v)
        float g00 = 0.f, g01 = 0.f, g02 = 0.f, g11 = 0.f, g12 = 0.f, g22 = 0.f;
#pragma unroll
        for (int j = 0; j < DH; ++j) {
            const int e = lane + 32 * j;
            r0[j] = anch && e < C::NH ? r0s[e] : 0.f;
            if (anch) ht[j] = (ht[j] - shift * t[j]) - shift_lo * t[j];
            g00 += x[j] * (2.f * r0[j] + hx[j]);
            g01 += p[j] * r0[j] + x[j] * hp[j];
            g02 += t[j] * r0[j] + x[j] * ht[j];
            g11 += p[j] * hp[j];
            g12 += p[j] * ht[j];
            g22 += t[j] * ht[j];
        }
        float G[3][3];
        const float sx = anch ? 1.f / sqrtf(xx) : 1.f;
        G[0][0] = warp_sum(g00) * sx * sx;
        G[0][1] = G[1][0] = warp_sum(g01) * sx;
        G[0][2] = G[2][0] = warp_sum(g02) * sx;
        G[1][1] = warp_sum(g11);
        G[1][2] = G[2][1] = warp_sum(g12);
        G[2][2] = warp_sum(g22);
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
        float nxx = 0.f, nxh = 0.f, nxr = 0.f, nx0 = 0.f;
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
            nxx += nx * nx;
            nxh += nx * nhx;
            nxr += nx * r0[j];
            nx0 += nx * x0[j];
        }
        nxx = warp_sum(nxx);
        nxh = warp_sum(nxh);
        float sc;
        if (anch) {
            nxr = warp_sum(nxr);
            nx0 = warp_sum(nx0);
            sc = 1.f / y0;
            // mu = (x.Ax) / (x.x), x = x0 + sc nx, A x = r0 + sc A nx, x0.r0 = 0
            lam = (sc * 2.f * nxr + sc * sc * nxh) / (x0x0 + sc * 2.f * nx0 + sc * sc * nxx);
            o.dnorm = (double)(fabsf(sc) * sqrtf(nxx));
        } else {
            sc = 1.f / sqrtf(nxx);
            lam = nxh / nxx;
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
    long long Vf[C::PT];   // float64 V during set-up, then fixed point (1/2 V)
    long long Hsf[C::NH];  // float64 Hs during set-up, then fixed point (off-diagonal)
    double hd[C::NS];      // diagonal of Hs
    union {                // sigma partial sums; set-up scratch
        alignas(16) float S[C::L * C::NS * C::NSP];
        long long S64[C::NS * (C::NS | 1)];
        struct {
            double diag[C::NH], h[C::P];
        } su;
    } s;
    union {
        alignas(16) float cm[2 * C::NSH * C::NS];
        int cmi[2 * C::NSH * C::NS];
        double dsum[C::NS * C::n];
    } c;
    alignas(16) float Hs32[C::NS * C::NSP];
    float2 V2[C::PH * 2 * C::P];
    float dg[C::NH], x0[C::NH], r0[C::NH];
    int A[8];
};

constexpr int SECTOR_WARPS = 4;  // most warps per block (mbe_tuning.warp_warps)

// Mixed precision (see k_casci_warp_mixed for the method: float32 Davidson, anchored
// refinements), one warp per tuple of the class (n, k).
template <class C>
__global__ void __launch_bounds__(SECTOR_WARPS * 32, C::DH > 4 ? 3 : 4) k_sector_mixed(BatchArgs a, int bucket)
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
        double *Vp = (double *)W.Vf, *Hsp = (double *)W.Hsf;
        const SectorStart st =
            sector_setup<C>(a, T, W.A, Vp, Hsp, W.hd, W.s.su.h, W.c.dsum, W.s.su.diag);
        double vmax = 0.0;
        for (int e = lane; e < C::PT; e += 32) {
            const uchar2 xy = T.ptri[e];
            const double v = 0.5 * Vp[e];
            const float f = (float)v;
            float *col = (float *)&W.V2[(xy.y >> 1) * 2 * C::P] + (xy.y & 1);
            col[4 * xy.x] = f;
            col[4 * xy.x + 2] = -f;
            col = (float *)&W.V2[(xy.x >> 1) * 2 * C::P] + (xy.x & 1);
            col[4 * xy.y] = f;
            col[4 * xy.y + 2] = -f;
            vmax = fmax(vmax, fabs(v));
        }
        for (int e = lane; e < C::NH; e += 32) {
            const uchar2 ij = T.tri[e];
            const double v = Hsp[e];
            W.Hs32[ij.x * C::NSP + ij.y] = W.Hs32[ij.y * C::NSP + ij.x] = (float)v;
            if (ij.x != ij.y) vmax = fmax(vmax, fabs(v));
            W.dg[e] = (float)W.s.su.diag[e];
        }
        const int E = fixed_exponent(vmax);
        const double scale = pow2(55 - E);
        __syncwarp();
        for (int e = lane; e < C::PT; e += 32) ((int2 *)W.Vf)[e] = to_fixed(0.5 * Vp[e], scale);
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
        for (int sector = 0; sector < 2 && !redo; ++sector) {
            if (sector == 1 && a.even_only) break;
            const int sgn = sector == 0 ? 1 : -1, g = sector == 0 ? st.g : st.go;
            float xv[C::DH];
#pragma unroll
            for (int j = 0; j < C::DH; ++j) {
                const int e = lane + 32 * j;
                xv[j] = e < C::NH ? packed_guess<C, float>(T.tri[e], e, g, sgn) : 0.f;
            }
            auto sigma = [&](const float(&tv)[C::DH], float(&out)[C::DH]) {
                sigma_sector<C>(T, W.V2, W.Hs32, W.c.cm, W.s.S, sgn, tv, out);
            };
            // plain float32 passes (the first sector one to tol_switch; the second one
            // to SECTOR_TOL, then tol_switch, decided against the first's float32
            // eigenvalue), then anchored refinements; one call site of the Davidson
            int passes = 0, anchors = 0;
            bool lose = false, fail = false, done = false;
            double th = 0.0, lam_s = 0.0;
            Anchor an{W.x0, W.r0, 0.f, 0.f, 1.f};
            for (;;) {
                const bool anchored = anchors > 0;
                const double tl = anchored ? a.tol : ((sector == 0 || passes == 1) ? a.tol_switch : SECTOR_TOL);
                const PhaseOut o = davidson_sector<C>(sigma, W.dg, xv, tl, anchored ? a.min_fp64 : 0, a.max_iter,
                                                      anchored ? &an : nullptr);
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
                        W.c.cmi[c_at<C>(ij.x, ij.y)] = q;
                        W.c.cmi[c_at<C>(ij.y, ij.x)] = sgn > 0 ? q : -q;
                    }
                }
                __syncwarp();
                sigma_anchor<C>(T, (const int2 *)W.Vf, (const int2 *)W.Hsf, W.c.cmi, W.s.S64, sgn);
                ++n64;
                double xs = 0.0, xx = 0.0;
                double s0[C::DH], c0[C::DH];
#pragma unroll
                for (int j = 0; j < C::DH; ++j) {
                    const int e = lane + 32 * j;
                    s0[j] = c0[j] = 0.0;
                    if (e < C::NH) {
                        const uchar2 ij = T.tri[e];
                        constexpr int ST = C::NS | 1;
                        const long long u = W.s.S64[ij.y * ST + ij.x], w = W.s.S64[ij.x * ST + ij.y];
                        const double wt = ij.x == ij.y ? 1.0 : 1.4142135623730951;
                        c0[j] = (double)W.c.cmi[c_at<C>(ij.x, ij.y)] * (wt * pow2(-28));
                        s0[j] = fma(W.hd[ij.x] + W.hd[ij.y], c0[j], (double)(sgn > 0 ? u + w : u - w) * (wt * pow2(E - 55)));
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

}  // namespace mbe
