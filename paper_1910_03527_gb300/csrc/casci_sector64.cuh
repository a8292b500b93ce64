#pragma once
// The float64 sector solver (see casci_sector.cuh): float64 mode, the tuples that the mixed
// solver hands back, and the density matrices of the adjoint.
//
// A float64 multiply-add runs on 1.67 lanes per clock and SM here, a wide integer one
// (32 x 32 + 64 -> 64 bits) with operands that change on 18-23.  sigma is therefore formed in
// 55-bit fixed point: the unit vector and V each in two limbs (to_fixed), three integer
// multiply-adds per term (hi hi, hi lo, lo hi; lo lo, at most 2^-56 of the largest element of V
// and Hs, is left out) in 64-bit sums, the low ones rounded to 2^-54 once per partial sum.
// The diagonal of Hs is added in float64.  The error is a fraction of the largest element where a
// float64 sum's is one of its own terms, which an eigenpair does not see: the same tuples reach residuals
// of 1e-12 to 1e-14, and energies and gradients of the timed expansions are as far from 64 bits as
// with float64 sums.  What is left for the float64 pipe is the Davidson's vector algebra, which
// bounds the kernel: about 40 operations per packed element and iteration.
#include "casci_sector.cuh"

namespace mbe {

// Shared memory of one warp.
template <class C>
struct Sector64 {
    union {
        struct {
            int2 Vf[C::P * C::P];                      // 1/2 V, fixed point
            alignas(16) int2 Hsf[C::NS * C::NSP];      // Hs without its diagonal, fixed point
            union {
                long long S[C::L * C::NS * (C::NS | 1)];  // partial sums of sigma
                struct {
                    double Vp[C::PT], Hsp[C::NH], h[C::P], dsum[C::NS * C::n];
                } su;
            } u;
        } s;
        struct {  // density matrices: 32 elements of every E_rs c, and of c
            double D[(C::n * C::n + 1) * 33];
            double g1[C::n * C::n];
        } r;
    } m;
    union {
        alignas(16) int4 ci[C::NSH * C::NS];  // coefficients in fixed point, columns in pairs (c_at)
        double c[C::NS * C::NS];              // float64 coefficients (density matrices)
    } c;
    double hd[C::NS], dg[C::NH], x2[C::NH];
    int A[8];
};

template <class C>
__device__ __forceinline__ void sigma_sector64(const SectorTables<C> &Tb, Sector64<C> &W, int E, int sgn,
                                               const double (&t)[C::DH], double (&out)[C::DH])
{
    constexpr int ST = C::NS | 1;
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < C::DH; ++j) {
        const int e = lane + 32 * j;
        if (e < C::NH) {
            const uchar2 ij = Tb.tri[e];
            const double w = ij.x == ij.y ? 36028797018963968.0 : 0.70710678118654752 * 36028797018963968.0;  // 2^55
            const int2 f = to_fixed(t[j], w);
            int2 *ci = (int2 *)W.c.ci;
            ci[c_at<C>(ij.x, ij.y)] = f;
            ci[c_at<C>(ij.y, ij.x)] = make_int2(sgn * f.x, sgn * f.y);
        }
    }
    __syncwarp();
    long long hi[C::NS], lo[C::NS];
#pragma unroll
    for (int i = 0; i < C::NS; ++i) hi[i] = lo[i] = 0;
    sector_rounds<C>(
        [&](int Ib, int y) {
            const int e = Tb.list[Ib * C::R + y], J = e >> 8, pr = (e & 255) >> 1, m = -((e & 1) ^ ((1 - sgn) >> 1));
            int ch[2 * C::NSH], cl[2 * C::NSH];
#pragma unroll
            for (int i = 0; i < C::NSH; ++i) {
                const int4 v = W.c.ci[i * C::NS + J];
                ch[2 * i] = (v.x ^ m) - m;
                cl[2 * i] = (v.y ^ m) - m;
                ch[2 * i + 1] = (v.z ^ m) - m;
                cl[2 * i + 1] = (v.w ^ m) - m;
            }
            static_for<C::P>([&](auto p) {
                const int2 v = W.m.s.Vf[p * C::P + pr];
                static_for<C::NS>([&](auto I) {
                    constexpr int a = C::pair_hi(decltype(p)::value), b = C::pair_lo(decltype(p)::value);
                    constexpr int Jx = C::target(decltype(I)::value, a, b);
                    if constexpr (Jx >= 0) {
                        constexpr bool neg = C::negative(decltype(I)::value, a, b);
                        const int vh = neg ? -v.x : v.x, vl = neg ? -v.y : v.y;
                        hi[I] += (long long)vh * ch[Jx];
                        lo[I] += (long long)vh * cl[Jx];
                        lo[I] += (long long)vl * ch[Jx];
                    }
                });
            });
        },
        [&](int Ib, int J) {
            int2 c = ((const int2 *)W.c.ci)[c_at<C>(Ib, J)];
            c = make_int2(sgn * c.x, sgn * c.y);
            const int4 *hs = (const int4 *)(W.m.s.Hsf + J * C::NSP);
#pragma unroll
            for (int i = 0; i < C::NSP / 2; ++i) {
                if (2 * i >= C::NS) break;
                const int4 v = hs[i];
                hi[2 * i] += (long long)v.x * c.x;
                lo[2 * i] += (long long)v.x * c.y;
                lo[2 * i] += (long long)v.y * c.x;
                if (2 * i + 1 < C::NS) {
                    hi[2 * i + 1] += (long long)v.z * c.x;
                    lo[2 * i + 1] += (long long)v.z * c.y;
                    lo[2 * i + 1] += (long long)v.w * c.x;
                }
            }
        },
        [&](int Ib, int part) {
#pragma unroll
            for (int i = 0; i < C::NS; ++i) {
                W.m.s.u.S[(part * C::NS + Ib) * ST + i] = hi[i] + ((lo[i] + (1LL << 27)) >> 28);
                hi[i] = lo[i] = 0;
            }
        });
    __syncwarp();
    const double unit = pow2(E - 54);
#pragma unroll
    for (int j = 0; j < C::DH; ++j) {
        const int e = lane + 32 * j;
        out[j] = 0.0;
        if (e < C::NH) {
            const uchar2 ij = Tb.tri[e];
            long long u = 0, w = 0;
#pragma unroll
            for (int p = 0; p < C::L; ++p) {
                u += W.m.s.u.S[(p * C::NS + ij.y) * ST + ij.x];
                w += W.m.s.u.S[(p * C::NS + ij.x) * ST + ij.y];
            }
            const double wt = ij.x == ij.y ? unit : 1.4142135623730951 * unit;
            out[j] = fma(W.hd[ij.x] + W.hd[ij.y], t[j], (double)(u + sgn * w) * wt);
        }
    }
    __syncwarp();
}

// davidson_warp<double> on packed vectors, with fewer float64 operations: the dot products
// of a stage are reduced together, the second orthogonalisation pass is taken only when the
// first one cancelled (less than half of |t|^2 left; with more left, one pass is orthogonal
// to within a few rounding errors), the reciprocal of the preconditioner is a float32 one
// with a Newton step (relative error 4e-15), and x is rescaled only when its norm has drifted.
template <class C, class SIGMA>
__device__ __forceinline__ PhaseOut davidson_sector64(SIGMA sigma, const double *dg, double (&x)[C::DH], double tol,
                                                      int min_iter, int max_iter, bool steered)
{
    constexpr int DH = C::DH;
    const int lane = threadIdx.x & 31;
    double hx[DH], p[DH], hp[DH], t[DH], ht[DH];
    PhaseOut o;
    o.nsig = 0;
    o.status = MBE_STATUS_OK;
    o.dnorm = 0.0;
    double lam = 0.0, rn = 0.0, best = 1e300;
    int stall = 0;
    int first = opaque(1);
    bool have_p = false;
    {
        double s = 0.0;
#pragma unroll
        for (int j = 0; j < DH; ++j) s = fma(x[j], x[j], s);
        s = inv_sqrt64(warp_sum(s));
#pragma unroll
        for (int j = 0; j < DH; ++j) {
            t[j] = x[j] = x[j] * s;
            p[j] = hp[j] = hx[j] = 0.0;
        }
    }
    for (int it = 0;;) {
        const bool steer = opaque(steered);
        if (!first) {
            double v[4] = {0.0, 0.0, 0.0, 0.0};  // |r|^2, x.t, p.t, |t|^2
#pragma unroll
            for (int j = 0; j < DH; ++j) {
                const int e = lane + 32 * j;
                t[j] = 0.0;
                if (e < C::NH) {
                    const double r = fma(-lam, x[j], hx[j]);
                    double den = dg[e] - lam;
                    if (fabs(den) < 1e-4) den = den >= 0.0 ? 1e-4 : -1e-4;
                    const double y = (double)(1.0f / (float)den);
                    t[j] = r * fma(y, fma(-den, y, 1.0), y);
                    v[0] = fma(r, r, v[0]);
                    v[1] = fma(x[j], t[j], v[1]);
                    v[2] = fma(p[j], t[j], v[2]);
                    v[3] = fma(t[j], t[j], v[3]);
                }
            }
            warp_sum_n<4>(v);
            rn = sqrt(v[0]);
            if (!isfinite(rn) || !isfinite(lam)) {
                o.status = MBE_STATUS_NONFINITE;
                break;
            }
            if (rn <= tol && it >= min_iter) break;
            if (it >= max_iter) {
                o.status = MBE_STATUS_MAXITER;
                break;
            }
            if (steer) {
                if (rn < 0.9 * best) {
                    best = rn;
                    stall = 0;
                } else if (++stall >= 3) {
                    break;
                }
            }
            double tt = 0.0;
#pragma unroll
            for (int j = 0; j < DH; ++j) {
                t[j] = fma(-v[1], x[j], fma(-v[2], p[j], t[j]));
                tt = fma(t[j], t[j], tt);
            }
            tt = warp_sum(tt);
            if (!(tt >= 0.5 * v[3])) {
                double w[2] = {0.0, 0.0};
#pragma unroll
                for (int j = 0; j < DH; ++j) {
                    w[0] = fma(x[j], t[j], w[0]);
                    w[1] = fma(p[j], t[j], w[1]);
                }
                warp_sum_n<2>(w);
                tt = 0.0;
#pragma unroll
                for (int j = 0; j < DH; ++j) {
                    t[j] = fma(-w[0], x[j], fma(-w[1], p[j], t[j]));
                    tt = fma(t[j], t[j], tt);
                }
                tt = warp_sum(tt);
            }
            const double tn = sqrt(tt);
            if (!(tn > tiny_norm<double>())) {
                // The correction lies in span{x, p}: nothing left to add.
                if (!steer && rn > tol) o.status = MBE_STATUS_MAXITER;
                break;
            }
            const double tinv = div64(1.0, tn);
#pragma unroll
            for (int j = 0; j < DH; ++j) t[j] *= tinv;
        }
        sigma(t, ht);
        ++o.nsig;
        if (first) {
            double xh = 0.0;
#pragma unroll
            for (int j = 0; j < DH; ++j) {
                hx[j] = ht[j];
                xh = fma(x[j], ht[j], xh);
            }
            lam = warp_sum(xh);
            first = opaque(0);
            continue;
        }
        ++it;
        // G = [x p t]^T H [x p t], x.Hx the Ritz value
        double g[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int j = 0; j < DH; ++j) {
            g[0] = fma(x[j], hp[j], g[0]);
            g[1] = fma(x[j], ht[j], g[1]);
            g[2] = fma(p[j], hp[j], g[2]);
            g[3] = fma(p[j], ht[j], g[3]);
            g[4] = fma(t[j], ht[j], g[4]);
        }
        warp_sum_n<8>(g);
        double G[3][3];
        G[0][0] = lam;
        G[0][1] = G[1][0] = g[0];
        G[0][2] = G[2][0] = g[1];
        G[1][1] = g[2];
        G[1][2] = G[2][1] = g[3];
        G[2][2] = g[4];
        double y[3];
        eig3<double>(G, have_p, y);
        const double w2 = y[1] * y[1] + y[2] * y[2];
        double q0 = -w2 * y[0], q1 = y[1] - w2 * y[1], q2 = y[2] - w2 * y[2];
        const double zn = sqrt(q0 * q0 + q1 * q1 + q2 * q2);
        have_p = zn > tiny_norm<double>() * 1e-3;
        const double zi = have_p ? div64(1.0, zn) : 0.0;
        q0 *= zi;
        q1 *= zi;
        q2 *= zi;
        double n[2] = {0.0, 0.0};
#pragma unroll
        for (int j = 0; j < DH; ++j) {
            const double nx = fma(y[0], x[j], fma(y[1], p[j], y[2] * t[j]));
            const double nhx = fma(y[0], hx[j], fma(y[1], hp[j], y[2] * ht[j]));
            p[j] = fma(q0, x[j], fma(q1, p[j], q2 * t[j]));
            hp[j] = fma(q0, hx[j], fma(q1, hp[j], q2 * ht[j]));
            x[j] = nx;
            hx[j] = nhx;
            n[0] = fma(nx, nx, n[0]);
            n[1] = fma(nx, nhx, n[1]);
        }
        warp_sum_n<2>(n);
        lam = div64(n[1], n[0]);
        if (!(fabs(n[0] - 1.0) <= 4e-15)) {
            const double sc = inv_sqrt64(n[0]);
#pragma unroll
            for (int j = 0; j < DH; ++j) {
                x[j] *= sc;
                hx[j] *= sc;
            }
        }
    }
    o.lambda = lam;
    o.rnorm = rn;
    return o;
}

// Spin-free density matrices of the sector vector x and their share of the gradients.
// <c| E_pq E_rs |c> = (E_qp c).(E_rs c), so the 2-RDM is the Gram matrix of the n^2 vectors
// E_rs c (all in c's own sector: half of the elements), formed 32 elements at a time: each
// lane fills one element of every vector, then owns a share of the Gram matrix.  No atomics
// but the final ones, where walking the lists from every determinant takes 4 R^2 of them.
template <class C>
__device__ __noinline__ void sector_rdm(const BatchArgs &a, const SectorTables<C> &Tb, Sector64<C> &W, int sgn,
                                        const double (&x)[C::DH], double w)
{
    constexpr int n = C::n, n2 = n * n, NV = n2 + 1, NG = NV * (NV + 1) / 2, GE = (NG + 31) / 32;
    const int lane = threadIdx.x & 31;
    double *D = W.m.r.D, *c = W.c.c;
#pragma unroll
    for (int j = 0; j < C::DH; ++j) {
        const int e = lane + 32 * j;
        if (e < C::NH) {
            const uchar2 ij = Tb.tri[e];
            const double v = ij.x == ij.y ? x[j] : 0.70710678118654752 * x[j];
            c[ij.x * C::NS + ij.y] = v;
            c[ij.y * C::NS + ij.x] = sgn > 0 ? v : -v;
        }
    }
    __syncwarp();
    const bool two = a.grad_eri != nullptr;
    double gram[GE];
#pragma unroll
    for (int i = 0; i < GE; ++i) gram[i] = 0.0;
#pragma unroll 1
    for (int j = 0; j < C::DH; ++j) {
        const int e = lane + 32 * j;
        const uchar2 ij = Tb.tri[e < C::NH ? e : 0];
        const double wt = e < C::NH ? (ij.x == ij.y ? 1.0 : 1.4142135623730951) : 0.0;
        const uint32_t sa = Tb.str[ij.x], sb = Tb.str[ij.y];
        constexpr uint32_t full = (1u << n) - 1u;
        // <I| E_rs = s <J| with |J> = s E_sr |I>: r occupied in I, s empty or r itself
        auto entry = [&](int I, uint32_t st, int r, int s) {
            const int at = __popc(st & ((1u << r) - 1u)) * (n - C::k + 1) + __popc(~st & full & ((1u << s) - 1u)) +
                           (r < s ? 1 : 0);
            return (int)Tb.list[I * C::R + at];
        };
#pragma unroll 1
        for (int rs = 0; rs < n2; ++rs) {
            const int r = rs / n, s = rs - r * n;
            double v = 0.0;
            if ((sa >> r & 1u) && (r == s || !(sa >> s & 1u))) {
                const int q = entry(ij.x, sa, r, s);
                v = flip_if(c[(q >> 8) * C::NS + ij.y], q & 1);
            }
            if ((sb >> r & 1u) && (r == s || !(sb >> s & 1u))) {
                const int q = entry(ij.y, sb, r, s);
                v += flip_if(c[ij.x * C::NS + (q >> 8)], q & 1);
            }
            D[rs * 33 + lane] = wt * v;
        }
        D[n2 * 33 + lane] = wt * c[ij.x * C::NS + ij.y];
        __syncwarp();
#pragma unroll
        for (int i = 0; i < GE; ++i) {
            const int q = lane + 32 * i;
            // row v of the triangle (v >= u); the last row holds c itself: gamma
            int v = (int)((sqrtf(8.f * q + 1.f) - 1.f) * 0.5f);
            v += (v + 1) * (v + 2) / 2 <= q ? 1 : 0;
            v -= v * (v + 1) / 2 > q ? 1 : 0;
            const int u = q - v * (v + 1) / 2;
            if (q < NG && u < n2 && (two || v == n2)) {
                double s = gram[i];
#pragma unroll 8
                for (int h = 0; h < 32; ++h) s = fma(D[u * 33 + h], D[v * 33 + h], s);
                gram[i] = s;
            }
        }
        __syncwarp();
    }
    double *g1 = W.m.r.g1;
#pragma unroll
    for (int i = 0; i < GE; ++i) {
        const int q = lane + 32 * i;
        if (q < NG && q >= n2 * (n2 + 1) / 2 && q < NG - 1) g1[q - n2 * (n2 + 1) / 2] = gram[i];
    }
    __syncwarp();
    const int *A = W.A;
    for (int e = lane; e < n2; e += 32) {
        const int p = e / n, q = e - p * n;
        rdm_one_body(a, A, n, p, q, w * (g1[e] - ((p == q && a.occ[A[p]]) ? 2.0 : 0.0)));
    }
    if (!two) return;
#pragma unroll
    for (int i = 0; i < GE; ++i) {
        const int g = lane + 32 * i;
        int v = (int)((sqrtf(8.f * g + 1.f) - 1.f) * 0.5f);
        v += (v + 1) * (v + 2) / 2 <= g ? 1 : 0;
        v -= v * (v + 1) / 2 > g ? 1 : 0;
        const int u = g - v * (v + 1) / 2;
        if (v >= n2 || u >= n2) continue;
        rdm_two_body(a, A, n, u, v, gram[i], g1, w);
    }
    __syncwarp();
}

// One warp per tuple of the class (n, k); REDO: only the tuples that the mixed solver
// flagged.  Density matrices when a.rdm is set.
template <class C, bool REDO>
__device__ __forceinline__ void sector64_tuples(const BatchArgs &a, int bucket)
{
    extern __shared__ __align__(16) char smem[];
    SectorTables<C> &T = *(SectorTables<C> *)smem;
    Sector64<C> &W = ((Sector64<C> *)(smem + al16((int)sizeof(SectorTables<C>))))[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    build_tables<C>(T, a.cls[C::k]);
    const int64_t begin = a.bucket_off[bucket];
    const int64_t cnt = a.bucket_off[bucket + 1] - begin;
    for (;;) {
        unsigned long long pos = 0;
        if (lane == 0) pos = atomicAdd(&(REDO ? a.counters2 : a.counters)[bucket], 1ULL);
        pos = __shfl_sync(FULL, pos, 0);
        if ((int64_t)pos >= cnt) break;
        const int64_t t = a.perm[begin + (int64_t)pos];
        if (REDO && a.pstate[2 * t] != PS_REDO) continue;
        if (lane == 0) build_A(a, t, W.A);
        __syncwarp();
        double *Vp = W.m.s.u.su.Vp, *Hsp = W.m.s.u.su.Hsp;
        const SectorStart st = sector_setup<C>(a, T, W.A, Vp, Hsp, W.hd, W.m.s.u.su.h, W.m.s.u.su.dsum, W.dg);
        int vmax = 0;
        bool bad = false;
#pragma unroll 1
        for (int e = lane; e < C::PT; e += 32) {
            const int hi = high_word(Vp[e]);
            vmax = max(vmax, hi - 0x00100000);  // (of 1/2 V)
            bad = bad || hi >= 0x7ff00000;
        }
#pragma unroll 1
        for (int e = lane; e < C::NH; e += 32) {
            const uchar2 ij = T.tri[e];
            const int hi = high_word(Hsp[e]);
            if (ij.x != ij.y) vmax = max(vmax, hi);
            bad = bad || hi >= 0x7ff00000;
        }
        const int E = fixed_exponent(vmax);
        const double scale = pow2(55 - E);
#pragma unroll 1
        for (int e = lane; e < C::PT; e += 32) {
            const uchar2 xy = T.ptri[e];
            W.m.s.Vf[xy.x * C::P + xy.y] = W.m.s.Vf[xy.y * C::P + xy.x] = to_fixed(Vp[e], 0.5 * scale);
        }
#pragma unroll 1
        for (int e = lane; e < C::NH; e += 32) {
            const uchar2 ij = T.tri[e];
            const int2 f = ij.x == ij.y ? make_int2(0, 0) : to_fixed(Hsp[e], scale);
            W.m.s.Hsf[ij.x * C::NSP + ij.y] = W.m.s.Hsf[ij.y * C::NSP + ij.x] = f;
        }
        __syncwarp();
        // an element that is not finite has no fixed-point form: make the image not finite
        if (__any_sync(FULL, bad) && lane < C::NS) W.hd[lane] = __longlong_as_double(0x7ff8000000000000LL);
        __syncwarp();
        double x[C::DH];
        double lam = 0.0;
        int status = MBE_STATUS_OK, n64 = 0, won = 1;
        bool degen = false;
        const int n32 = REDO ? a.pstate[2 * t + 1] : 0;  // the mixed solver's float32 work
#pragma unroll 1
        for (int sector = opaque(0); sector < 2; ++sector) {
            if (sector == 1 && (status != MBE_STATUS_OK || a.even_only)) break;
            const int sgn = opaque(sector == 0 ? 1 : -1), g = sector == 0 ? st.g : st.go;
#pragma unroll
            for (int j = 0; j < C::DH; ++j) {
                const int e = lane + 32 * j;
                if (sector == 1 && a.rdm && e < C::NH) W.x2[e] = x[j];
                x[j] = e < C::NH ? packed_guess<C, double>(T.tri[e], e, g, sgn) : 0.0;
            }
            auto sigma = [&](const double(&tv)[C::DH], double(&out)[C::DH]) {
                sigma_sector64<C>(T, W, E, sgn, tv, out);
            };
            // the second sector's first pass (to SECTOR_TOL) decides whether it is refined;
            // one call site keeps the kernel within the instruction cache
            bool lose = false;
#pragma unroll 1
            for (int pass = opaque(sector == 1 ? 0 : 1); pass < 2 && !lose; ++pass) {
                const bool decide = pass == 0;
                const PhaseOut o = davidson_sector64<C>(sigma, W.dg, x, decide ? SECTOR_TOL : a.tol, 0, a.max_iter, decide);
                n64 += o.nsig;
                if (decide) {
                    lose = o.status == MBE_STATUS_NONFINITE || sector_loses(o.lambda, o.rnorm, lam, 0.0);
                } else if (sector == 0) {
                    lam = o.lambda;
                    status = o.status;
                } else {
                    degen = o.status == MBE_STATUS_OK && fabs(o.lambda - lam) <= DEGEN_TOL;
                    lose = o.status == MBE_STATUS_NONFINITE || !(o.lambda < lam);
                    if (!lose) {
                        lam = o.lambda;
                        status = o.status;
                        won = -1;
                    }
                }
            }
            if (lose && a.rdm) {
#pragma unroll
                for (int j = 0; j < C::DH; ++j) {
                    const int e = lane + 32 * j;
                    x[j] = e < C::NH ? W.x2[e] : 0.0;
                }
            }
            __syncwarp();
        }
        if (lane == 0) {
            const double e = status == MBE_STATUS_NONFINITE ? __longlong_as_double(0x7ff8000000000000LL)
                                                            : lam - st.ephi - a.e_ref_corr;
            store_result(a, t, e, with_degeneracy(status, degen), n64, n32);
        }
        if (a.rdm) sector_rdm<C>(a, T, W, won, x, a.weights ? a.weights[t] : 1.0);
        __syncwarp();
    }
}

template <class C, bool REDO>
__global__ void __launch_bounds__(SECTOR_WARPS * 32, C::DH > 4 ? 2 : 3) k_sector64(BatchArgs a, int bucket)
{
    sector64_tuples<C, REDO>(a, bucket);
}

// Two classes in one launch, as k_sector_mixed_pair.
template <class C0, class C1, bool REDO>
__global__ void __launch_bounds__(SECTOR_WARPS * 32, 3) k_sector64_pair(BatchArgs a, int b)
{
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        const unsigned half = gridDim.x / 2, second = (blockIdx.x >= half) != (pass == 1);
        if (!bucket_open(a, REDO ? a.counters2 : a.counters, b + second, pass ? half * (blockDim.x >> 5) : 0)) continue;
        if (second)
            sector64_tuples<C1, REDO>(a, b + 1);
        else
            sector64_tuples<C0, REDO>(a, b);
    }
}

}  // namespace mbe
