// Wilson hop on block fixed-point numbers, for the FP64 outer residual.
//
// A GB300 SM issues two FP64 multiply-adds per cycle and 64 32-bit integer
// ones, so the link products of the outer step run on the integer pipe:
// a site's 12 complex components are 64-bit integers q with one exponent E
// per site, value q 2^E, |q| <= 2^56; a link entry is u = w 2^(k-57) with
// |w| <= 2^57 and one k per link.  Both are cut into two signed
// digits, q = q1 2^29 + q0 with q0 in [-2^28, 2^28), and
//   (w q) 2^-57 = 2 w1 q1 + (w1 q0 + w0 q1) 2^-28 + w0 q0 2^-57
// is summed exactly in two 64-bit accumulators (three 32 x 32 -> 64
// multiply-adds per real product) but for the last term, below 1/2.
//
// Accuracy: converted from doubles, the largest |q| of a site and the largest
// |w| of a link are at least 2^55 and 2^56, so a component within a factor 8 of
// its site's largest keeps all 53 bits and a smaller one is rounded at 2^-57 of
// the largest; an entry of a link within a factor 16 of the link's largest keeps
// all its bits.  A hop adds its eight products at the exponent of the largest
// (site exponent plus link exponent), about a unit of 2^-56 of that for each.
// Its output (t64) keeps that exponent, also where the sum cancelled.  So errors
// are small against the largest neighbour, not against each component: a result
// far below its site's others has fewer right bits than in FP64 (1e-6 of them:
// nine digits), and on links that leave the colours apart (U = 1) it has.
// Where links mix them, FP64 rounds its sums at 2^-53 of the largest term too.
// Errors against a 64-bit mantissa, root mean square over 8^3 x 16, kappa 0.12,
// x the solution for one random source, FP64 hop -> this: links exp(0.3 i H) by
// site norm 4.3e-17 -> 5.8e-18, by component 3.4e-16 -> 6.5e-17; U = 1 by site
// norm 3.1e-17 -> 8.7e-18.
#pragma once

#include "pt_common.cuh"

#define FX_ZERO (-(1 << 20))     // exponent of a site without a nonzero component
#define FX_BAD (1 << 22)         // of a site or link with a NaN or an infinity (FX_BAD + FX_ZERO is bad too)

struct FxC { long long re, im; };

// q of the double v at a site whose largest biased exponent is em; `up` = bits
// gained over the 53 of the largest (3: |q| < 2^56; links 4: |w| < 2^57)
__host__ __device__ __forceinline__ long long fx_quant(long long b, int em, int up) {
    int e = (int)((b >> 52) & 0x7ff);
    long long m = b & 0xfffffffffffffLL;
    if (e) m |= 0x10000000000000LL;
    else e = 1;
    const int sh = e - em + up;
    long long r;
    if (sh >= 0) r = m << sh;
    else if (sh > -56) r = (m + (1LL << (-sh - 1))) >> -sh;
    else r = 0;
    return b < 0 ? -r : r;
}

// a site's 12 components to fixed point; returns its exponent
__device__ __forceinline__ int fx_site(const Cx<double> (&v)[12], FxC (&q)[12]) {
    unsigned mx = 0, lo = 0;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        mx = max(mx, (unsigned)__double2hiint(v[c].re) & 0x7fffffffu);
        mx = max(mx, (unsigned)__double2hiint(v[c].im) & 0x7fffffffu);
        lo |= (unsigned)__double2loint(v[c].re) | (unsigned)__double2loint(v[c].im);
    }
    const int em = max((int)(mx >> 20), 1);
#pragma unroll
    for (int c = 0; c < 12; ++c) {
        q[c].re = fx_quant(__double_as_longlong(v[c].re), em, 3);
        q[c].im = fx_quant(__double_as_longlong(v[c].im), em, 3);
    }
    if (em == 2047) return FX_BAD;
    return (mx | lo) ? em - 1078 : FX_ZERO;
}

// 2^E (0 below the normal range, NaN for FX_BAD)
__device__ __forceinline__ double fx_pow2(int E) {
    if (E >= FX_BAD / 2) return __longlong_as_double(0x7ff8000000000000LL);
    if (E < -1022) return 0.0;
    return __longlong_as_double((long long)(min(E, 1024) + 1023) << 52);
}

// two signed digits of a 64-bit integer below 2^59
__host__ __device__ __forceinline__ void fx_digits(long long h, int &h1, int &h0) {
    h1 = (int)((h + (1LL << 28)) >> 29);
    h0 = ((int)((unsigned)h << 3)) >> 3;
}

// h 2^-d, rounded (0 <= d <= 62)
__device__ __forceinline__ long long fx_down(long long h, int d) {
    return (h + ((1LL << d) >> 1)) >> d;
}

// sum of three complex products u h (or conj(u) h: conj = -1, else 0), digits
// of u and h as (re1, re0, im1, im0)
__device__ __forceinline__ FxC fx_dot3(const int4 (&u)[3], const int4 (&h)[3], int conj) {
    long long r1 = 0, r2 = 0, i1 = 0, i2 = 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const int a1 = u[b].x, a0 = u[b].y, c1 = (u[b].z ^ conj) - conj, c0 = (u[b].w ^ conj) - conj;
        const int n1 = -c1, n0 = -c0;
        r1 += (long long)a1 * h[b].x;
        r1 += (long long)n1 * h[b].z;
        i1 += (long long)a1 * h[b].z;
        i1 += (long long)c1 * h[b].x;
        r2 += (long long)a1 * h[b].y;
        r2 += (long long)a0 * h[b].x;
        r2 += (long long)n1 * h[b].w;
        r2 += (long long)n0 * h[b].z;
        i2 += (long long)a1 * h[b].w;
        i2 += (long long)a0 * h[b].z;
        i2 += (long long)c1 * h[b].y;
        i2 += (long long)c0 * h[b].x;
    }
    FxC o;
    o.re = 2 * r1 + ((r2 + (1LL << 27)) >> 28);
    o.im = 2 * i1 + ((i2 + (1LL << 27)) >> 28);
    return o;
}

__device__ __forceinline__ FxC fx_add(FxC a, FxC b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ FxC fx_sub(FxC a, FxC b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ FxC fx_i(FxC a) { return {-a.im, a.re}; }
// a + s b, s = +1 or -1 (known where it is inlined)
__device__ __forceinline__ FxC fx_pm(FxC a, FxC b, int s) { return s > 0 ? fx_add(a, b) : fx_sub(a, b); }

// The projections of spin_project and spin_accumulate on integers, sg = -1
// forward, +1 backward.
template <int MU, int SG>
__device__ __forceinline__ void fx_project(const FxC (&ps)[4][3], FxC (&h)[2][3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (MU == 0) {
            h[0][a] = fx_pm(ps[0][a], fx_i(ps[3][a]), -SG);
            h[1][a] = fx_pm(ps[1][a], fx_i(ps[2][a]), -SG);
        } else if (MU == 1) {
            h[0][a] = fx_pm(ps[0][a], ps[3][a], -SG);
            h[1][a] = fx_pm(ps[1][a], ps[2][a], SG);
        } else if (MU == 2) {
            h[0][a] = fx_pm(ps[0][a], fx_i(ps[2][a]), -SG);
            h[1][a] = fx_pm(ps[1][a], fx_i(ps[3][a]), SG);
        } else {
            h[0][a] = fx_pm(ps[0][a], ps[2][a], SG);
            h[1][a] = fx_pm(ps[1][a], ps[3][a], SG);
        }
    }
}
template <int MU, int SG>
__device__ __forceinline__ void fx_accumulate(const FxC (&u)[2][3], FxC (&acc)[4][3]) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        acc[0][a] = fx_add(acc[0][a], u[0][a]);
        acc[1][a] = fx_add(acc[1][a], u[1][a]);
        if (MU == 0) {
            acc[2][a] = fx_pm(acc[2][a], fx_i(u[1][a]), SG);
            acc[3][a] = fx_pm(acc[3][a], fx_i(u[0][a]), SG);
        } else if (MU == 1) {
            acc[2][a] = fx_pm(acc[2][a], u[1][a], SG);
            acc[3][a] = fx_pm(acc[3][a], u[0][a], -SG);
        } else if (MU == 2) {
            acc[2][a] = fx_pm(acc[2][a], fx_i(u[0][a]), SG);
            acc[3][a] = fx_pm(acc[3][a], fx_i(u[1][a]), -SG);
        } else {
            acc[2][a] = fx_pm(acc[2][a], u[0][a], SG);
            acc[3][a] = fx_pm(acc[3][a], u[1][a], SG);
        }
    }
}

// a field of fixed-point sites: three components at each of four addresses
struct FxField {
    const longlong2 *p[4];
    const int *e;
};
// links: digits [4][9][N] and exponents [4][N], by site or in even-odd order
struct FxLinks {
    const int4 *u;
    const int *k;
};

// (H psi)(x) at site idx: the integers in acc, the exponent returned (FX_ZERO:
// all zero, FX_BAD: a NaN or infinity among the neighbours or links).  EO: idx
// has parity par, f is the half field of the other parity and the links are in
// even-odd order; else f is a full field and the links by site.  The eight
// directions share one copy of the products in a loop: unrolled, the 6400
// instructions of a hop were fetched from beyond the instruction cache (3.3 of
// 6.8 stall cycles per instruction).
template <bool EO>
__device__ __forceinline__ int fx_hop(const Geom &g, const FxField &f, const FxLinks &U, int antip, int par, int idx,
                                      const int x[4], FxC (&acc)[4][3]) {
    const size_t N = (size_t)g.N;
    const int Ne = EO ? g.N >> 1 : g.N;
    constexpr int half = EO ? 1 : 0;
    // entries of the links U_mu(x) and U_mu(y) in one of the nine arrays of a direction
    const int own = EO ? par * Ne + (idx >> 1) : idx, other = EO ? (1 - par) * Ne : 0;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int a = 0; a < 3; ++a) acc[s][a] = FxC{0, 0};
    int E = FX_ZERO;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        const int yf = nb_fwd(g, idx, x, mu) >> half, yb = nb_bwd(g, idx, x, mu) >> half;
        E = max(E, max(f.e[yf] + U.k[mu * N + own], f.e[yb] + U.k[mu * N + other + yb]));
    }
    if (E >= FX_BAD / 2) return FX_BAD;
    if (E <= FX_ZERO / 2) return FX_ZERO;
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
        int y;
        bool neg = false;
        switch (k) {
            case 0: y = nb_fwd(g, idx, x, 0); break;
            case 1: y = nb_bwd(g, idx, x, 0); break;
            case 2: y = nb_fwd(g, idx, x, 1); break;
            case 3: y = nb_bwd(g, idx, x, 1); break;
            case 4: y = nb_fwd(g, idx, x, 2); break;
            case 5: y = nb_bwd(g, idx, x, 2); break;
            case 6: y = nb_fwd(g, idx, x, 3); neg = antip && x[3] == g.D[3] - 1; break;
            default: y = nb_bwd(g, idx, x, 3); neg = antip && x[3] == 0;
        }
        const bool bwd = k & 1;
        const int yh = y >> half;
        FxC ps[4][3], h[2][3], uh[2][3];
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const longlong2 v = f.p[c / 3][(size_t)(c % 3) * Ne + yh];
            ps[c / 3][c % 3] = FxC{v.x, v.y};
        }
        const int l = bwd ? other + yh : own;
        const int d = min(E - f.e[yh] - U.k[(k >> 1) * N + l], 62);
        switch (k) {
            case 0: fx_project<0, -1>(ps, h); break;
            case 1: fx_project<0, 1>(ps, h); break;
            case 2: fx_project<1, -1>(ps, h); break;
            case 3: fx_project<1, 1>(ps, h); break;
            case 4: fx_project<2, -1>(ps, h); break;
            case 5: fx_project<2, 1>(ps, h); break;
            case 6: fx_project<3, -1>(ps, h); break;
            default: fx_project<3, 1>(ps, h);
        }
        int4 hd[2][3];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                fx_digits(fx_down(h[q][a].re, d), hd[q][a].x, hd[q][a].y);
                fx_digits(fx_down(h[q][a].im, d), hd[q][a].z, hd[q][a].w);
            }
        // U_mu(x) by rows, or the conjugate of U_mu(x - mu) by columns
        const int4 *Uk = U.u + (size_t)(k >> 1) * 9 * N + l;
        const size_t sa = (bwd ? 1 : 3) * N, sb = (bwd ? 3 : 1) * N;
        const int conj = bwd ? -1 : 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            int4 u[3];
#pragma unroll
            for (int b = 0; b < 3; ++b) u[b] = Uk[a * sa + b * sb];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uh[q][a] = fx_dot3(u, hd[q], conj);
                if (neg) uh[q][a] = FxC{-uh[q][a].re, -uh[q][a].im};
            }
        }
        switch (k) {
            case 0: fx_accumulate<0, -1>(uh, acc); break;
            case 1: fx_accumulate<0, 1>(uh, acc); break;
            case 2: fx_accumulate<1, -1>(uh, acc); break;
            case 3: fx_accumulate<1, 1>(uh, acc); break;
            case 4: fx_accumulate<2, -1>(uh, acc); break;
            case 5: fx_accumulate<2, 1>(uh, acc); break;
            case 6: fx_accumulate<3, -1>(uh, acc); break;
            default: fx_accumulate<3, 1>(uh, acc);
        }
    }
    return E;
}

// bring the integers below 2^56 again; returns the exponent that goes with them
__device__ __forceinline__ int fx_normalise(FxC (&q)[4][3], int E) {
    unsigned long long mx = 0;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            mx |= (unsigned long long)(q[s][a].re < 0 ? ~q[s][a].re : q[s][a].re);
            mx |= (unsigned long long)(q[s][a].im < 0 ? ~q[s][a].im : q[s][a].im);
        }
    // rounding up may reach 2^56 itself: aim one bit lower
    const int d = max(0, 64 - __clzll((long long)mx) - 55);
    if (E == FX_ZERO || E >= FX_BAD) return E;
    if (d)
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int a = 0; a < 3; ++a) q[s][a] = FxC{fx_down(q[s][a].re, d), fx_down(q[s][a].im, d)};
    return E + d;
}

// ---- link digits and exponents, one thread per link: by site, or in the
// even-odd link order (EO: site s of an array at parity N/2 + s/2)
template <bool EO>
__global__ void k_fx_links(Geom g, const double2 *__restrict__ src, int4 *__restrict__ dst, int *__restrict__ kexp) {
    const int N = g.N;
    const int64_t total = (int64_t)4 * N;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t mu = t / N;
        const int s = (int)(t - mu * N);
        int o = s;
        if (EO) {
            int x[4];
            site_coords(g, s, x);
            o = ((x[0] + x[1] + x[2] + x[3]) & 1) * (N >> 1) + (s >> 1);
        }
        double2 v[9];
        int em = 1;
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            v[c] = src[(mu * 9 + c) * N + s];
            em = max(em, (__double2hiint(v[c].x) & 0x7fffffff) >> 20);
            em = max(em, (__double2hiint(v[c].y) & 0x7fffffff) >> 20);
        }
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            int4 d;
            fx_digits(fx_quant(__double_as_longlong(v[c].x), em, 4), d.x, d.y);
            fx_digits(fx_quant(__double_as_longlong(v[c].y), em, 4), d.z, d.w);
            dst[(mu * 9 + c) * N + o] = d;
        }
        kexp[mu * N + o] = em == 2047 ? FX_BAD : em - 1022;
    }
}
