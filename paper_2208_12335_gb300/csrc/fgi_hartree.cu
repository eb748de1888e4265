// The step upstream of the grid integration: the Hartree potential of the
// density on the grid, v_H(r) = int n(r') / |r - r'| dr', by the multipole
// method of Becke & Dickson (1988) and Delley (1990), which the NAO method
// uses for the electrostatic potential (the paper's Fig. 4 caption notes that
// this potential was not yet accelerated on GPUs).
//
//  1. k_hartree_moments: a warp per (atom a, radial shell k), over its points p
//     (listed once at set-up),
//       rho~_a,lm(r_k) = sum_p (w_p / (r_k^3 ln q)) n_p A_lm(rhat_p)
//     (w_p / (r_k^3 ln q) is the partitioned angular weight; A_lm = Y_lm / K_lm
//     the unnormalised harmonics).  Harmonics and sums of l >= 1 are double-float
//     (about 2^-45 relative), offsets, w_p n_p, the sum for l = 0 and the final scale FP64:
//     GB300's FP64 pipe has 1/64 of the FP32 rate.
//  2. k_hartree_radial (FP64): a warp per (atom, l, m), lanes along the shells, the
//     radial Poisson equation
//       V(r) = 4 pi/(2l+1) [r^-(l+1) int_0^r rho r'^(l+2) dr' + r^l int_r^inf rho r'^(1-l) dr']
//     with the partial integrals in x = ln r interval by interval, each by the
//     integral of the cubic through its four nearest shells, plus
//     rho(r_0) r_0^(l+3)/(l+3) inside the first shell; Q_lm = the whole inner
//     integral (the exterior multipole moments).  Stored with K_lm^2 folded in
//     (Y_lm Y_lm-weighted sums become A_lm sums): l = 0 in FP64 (V) and as a
//     double-float (Q, in a packed per-atom record with the atom's position),
//     l >= 1 in FP32.
//  3. k_hartree_eval: per point, over the atoms of its system, V_a,lm at the
//     distance times Y_lm of the direction: 4-point Lagrange interpolation in
//     the fractional shell index inside the grid (l = 0 as a double-float:
//     the interpolating cubic of each interval stored in f = x - k, and
//     f = ln(d / r_k) / ln q from an atanh series; FP64 for coarse grids),
//     4 pi/(2l+1) Q_lm / d^(l+1) beyond the last shell (l = 0 as a
//     double-float: offset, distance and 1/d from the double-float point and
//     atom positions), V(r_0) (d/r_0)^l inside the first shell.  The l >= 1
//     terms (angular functions, their coefficients and sums) are FP32: each
//     carries a relative error of a few FP32 roundings of the l >= 1 part,
//     against the FP64 pipe's 1/64 rate on GB300.  The sum over atoms is a
//     double-float.
#include "fgi_dd.cuh"
#include "fgi_hartree.h"
#include "fgi_ylm.cuh"

namespace fgi {

namespace {

constexpr int kL = (kHartreeLmax + 1) * (kHartreeLmax + 1);  // stride of the FP64 moment rows
constexpr int kLf = kL - 1;                                     // stride of the FP32 l >= 1 rows
// 2/3 and 2/5 as double-floats (compile-time)
constexpr float kTwoThirdHi = (float)(2.0 / 3.0), kTwoThirdLo = (float)(2.0 / 3.0 - (double)kTwoThirdHi);
constexpr float kTwoFifthHi = (float)(2.0 / 5.0), kTwoFifthLo = (float)(2.0 / 5.0 - (double)kTwoFifthHi);

struct HartreeTabs {
    double *rho;      // [n_shells][kL]    unnormalised moments
    double *Vd;       // [n_shells][kL]    scratch: inner part of V
    double *F;        // [n_shells][kL]    scratch: inner integrand
    float4 *rec;      // [n_atoms][3]      position (double-float), (last radius)^2, 4 pi K_00^2 Q_00
    float4 *rk;       // [n_shells]        r_k and 1/r_k as double-floats
    float4 *c0;       // [n_shells][2]     V_00 on interval k as a cubic in f (double-floats a0..a3)
    double *V0;       // [n_shells]        K_00^2 V_00
    float *Vf;        // [n_shells][kLf]   K_lm^2 V_lm, l >= 1
    float *Qf;        // [n_atoms][kLf]    4 pi/(2l+1) K_lm^2 Q_lm, l >= 1
};

size_t al256(size_t b) { return (b + 255) & ~(size_t)255; }

HartreeTabs carve(const HartreeDev &H, void *ws)
{
    char *b = (char *)ws;
    HartreeTabs T;
    T.rho = (double *)b;
    b += al256(sizeof(double) * kL * (size_t)H.n_shells);
    T.Vd = (double *)b;
    b += al256(sizeof(double) * kL * (size_t)H.n_shells);
    T.F = (double *)b;
    b += al256(sizeof(double) * kL * (size_t)H.n_shells);
    T.rec = (float4 *)b;
    b += al256(sizeof(float4) * 3 * (size_t)H.n_atoms);
    T.rk = (float4 *)b;
    b += al256(sizeof(float4) * (size_t)H.n_shells);
    T.c0 = (float4 *)b;
    b += al256(sizeof(float4) * 2 * (size_t)H.n_shells);
    T.V0 = (double *)b;
    b += al256(sizeof(double) * (size_t)H.n_shells);
    T.Vf = (float *)b;
    b += al256(sizeof(float) * kLf * (size_t)H.n_shells);
    T.Qf = (float *)b;
    return T;
}

__device__ __forceinline__ df dfa(df a, df b)      // sum of two double-floats (absolute accuracy)
{
    df s = df_two_sum(a.hi, b.hi);
    s.lo += a.lo + b.lo;
    return df_fast_two_sum(s.hi, s.lo);
}

__device__ __forceinline__ df dfa_f(df a, float b)
{
    df s = df_two_sum(a.hi, b);
    s.lo += a.lo;
    return df_fast_two_sum(s.hi, s.lo);
}

__device__ __forceinline__ df df_sqr(df a)
{
    df p = df_two_prod(a.hi, a.hi);
    p.lo = fmaf(2.0f * a.hi, a.lo, p.lo);
    return df_fast_two_sum(p.hi, p.lo);
}

// 1/sqrt(a) from y ~ rsqrtf(a.hi) by one Newton step with a double-float residual
__device__ __forceinline__ df df_rsqrt(df a, float y)
{
    const df ay2 = df_mul(a, df_two_prod(y, y));   // ~ 1
    const float e = (1.0f - ay2.hi) - ay2.lo;
    return df_fast_two_sum(y, y * (0.5f * e));
}

__device__ __forceinline__ double ipow(double r, int n)      // r^n, 0 <= n <= 9
{
    double p = 1.0;
    for (int i = 0; i < n; i++) p *= r;
    return p;
}

// acc += a b (double-floats; acc's low part a plain FP32 sum)
__device__ __forceinline__ void df_fma_acc(df &acc, df a, df b)
{
    df p = df_two_prod(a.hi, b.hi);
    p.lo = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, p.lo));
    const df t = df_two_sum(acc.hi, p.hi);
    acc.hi = t.hi;
    acc.lo += t.lo + p.lo;
}

// Sum of v[0 .. n) over the 32 lanes: each step halves the values a lane
// holds; lane's values end up as v[0 .. ceil(n/32)) = sums off .. of the n,
// those below lim.
template <int N, int MASK>
__device__ __forceinline__ void warp_sum_split(df *v, int &off, int &lim)
{
    if constexpr (MASK > 0) {
        constexpr int H = (N + 1) / 2;
        const bool upper = (threadIdx.x & MASK) != 0;
#pragma unroll
        for (int q = 0; q < H; q++) {
            const df b = q + H < N ? v[q + H < N ? q + H : 0] : df{0.f, 0.f};
            const float sh = upper ? v[q].hi : b.hi, sl = upper ? v[q].lo : b.lo;
            const float kh = upper ? b.hi : v[q].hi, kl = upper ? b.lo : v[q].lo;
            const df t = df_two_sum(kh, __shfl_xor_sync(0xffffffffu, sh, MASK));
            v[q].hi = t.hi;
            v[q].lo = t.lo + (kl + __shfl_xor_sync(0xffffffffu, sl, MASK));
        }
        if (upper) off += H;
        else lim = min(lim, off + H);
        warp_sum_split<H, MASK / 2>(v, off, lim);
    }
}

// Exponent field of a double, and a float 2^e (zero below FP32's range)
__device__ __forceinline__ int exp_field(double x) { return (int)((unsigned)__double2hiint(x) >> 20) & 0x7FF; }
__device__ __forceinline__ float pow2f(int e) { return e < -126 ? 0.f : __int_as_float((e + 127) << 23); }

// x 2^(1023 - e) as a double-float, for a field e not below x's own (or by at most
// 40), in integers: the leading 24 bits of x are the high part, the other 29
// the low part.  Zero where |x| is 2^126 times smaller than 2^(e - 1023).  Infinity and
// NaN give NaN.  (A conversion each way and a subtraction in FP64 would take
// the pipe that has 1/64 of the FP32 rate.)
__device__ __forceinline__ df df_scaled(double x, int e)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int f = (int)(hi >> 20) & 0x7FF, q = f - e;
    if (f == 0x7FF) return {__int_as_float(0x7FFFFFFF), 0.f};
    if (f == 0 || q < -126) return {0.f, 0.f};
    const unsigned sign = hi & 0x80000000u;
    const float h = __uint_as_float(sign | (unsigned)(q + 127) << 23 | (__funnelshift_l(lo, hi, 3) & 0x7FFFFFu));
    const float l = __uint2float_rn(lo & 0x1FFFFFFFu) * pow2f(q - 52);
    return df_fast_two_sum(h, sign ? -l : l);
}

// One warp per (atom, shell).  (A thread per point with FP64 harmonics and
// (l_max + 1)^2 FP64 atomics was bound by the FP64 pipe: 250-atom cluster, 7.3 M
// points, l_max 6, 3.30 ms; now 0.62 ms.)  The monopole's sum stays FP64: the
// l = 0 terms are all there is at l_max 0, and the others end in FP32.
//
// The offsets are differences in FP64 and w n a product in FP64; both become
// double-floats relative to a power of two (the largest component's; that of the
// warp's largest |w n| so far), so that neither an atom far from the origin nor
// the range of FP32 costs any of the 48 bits.  (Offsets from double-float positions and
// w n as a pair of FP32 numbers: 0.52 ms.)
template <int LMAX>
__global__ void __launch_bounds__(128) k_hartree_moments(DevPlan P, HartreeDev H, const double *n, double *rho)
{
    constexpr int L = (LMAX + 1) * (LMAX + 1);
    constexpr int kHeadroom = 40;                                      // binades w n may grow before the sums are scaled
    const long long bin = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (bin >= H.n_shells) return;
    const long long i0 = H.bin_off[bin], i1 = H.bin_off[bin + 1];
    df acc[L];
#pragma unroll
    for (int q = 0; q < L; q++) acc[q] = df{0.f, 0.f};
    double mono = 0.0;
    int ew = 0;                                                        // the sums hold w n 2^(1023 - ew)
    const int a = H.bin_atom[bin];
    const double ax = P.atom_xyz[3 * a], ay = P.atom_xyz[3 * a + 1], az = P.atom_xyz[3 * a + 2];
    for (long long ib = i0; ib < i1; ib += 32) {
        const bool has = ib + lane < i1;
        const long long p = H.order[has ? ib + lane : i0];
        const double dx = P.px[p] - ax, dy = P.py[p] - ay, dz = P.pz[p] - az;
        const int ed = max(exp_field(dx), max(exp_field(dy), exp_field(dz)));
        // a point on the nucleus has no direction
        const bool live = has && ed > 0;
        const double wn = live ? P.pw[p] * n[p] : 0.0;
        mono += wn;
        if (LMAX == 0) continue;
        const int fw = exp_field(wn);
        const int top = (int)__reduce_max_sync(0xffffffffu, fw == 0x7FF ? 0u : (unsigned)fw);
        if (top > ew + kHeadroom || ew == 0) {                         // the same for the whole warp
            const float down = ew == 0 ? 0.f : pow2f(ew - top);
#pragma unroll
            for (int q = 1; q < L; q++) acc[q] = df{acc[q].hi * down, acc[q].lo * down};
            ew = top;
        }
        if (!live) continue;
        df x = df_scaled(dx, ed), y = df_scaled(dy, ed), z = df_scaled(dz, ed);
        const df d2 = dfa(dfa(df_sqr(x), df_sqr(y)), df_sqr(z));
        const df ir = df_rsqrt(d2, rsqrtf(d2.hi));
        x = df_mul(x, ir);
        y = df_mul(y, ir);
        z = df_mul(z, ir);
        df cm = df_scaled(wn, ew), sm{0.f, 0.f};                   // w n Re, Im (x + i y)^m
        float pmm = 1.f;
#pragma unroll
        for (int m = 0; m <= LMAX; m++) {
            if (m > 0) {
                const df c = dfa(df_mul(cm, x), df_mul(df{-sm.hi, -sm.lo}, y));
                sm = dfa(df_mul(cm, y), df_mul(sm, x));
                cm = c;
                pmm *= (float)(2 * m - 1);                          // Pbar_m^m, exact
            }
            df p2{0.f, 0.f}, p1{pmm, 0.f};
#pragma unroll
            for (int l = m; l <= LMAX; l++) {
                df pl = p1;
                if (l == m + 1) {
                    pl = df_mul_f(z, (float)(2 * m + 1) * pmm);
                } else if (l > m + 1) {
                    // 1/(l-m) as a double-float
                    constexpr double one = 1.0;
                    const double iv = one / (double)(l - m);
                    const df inv{(float)iv, (float)(iv - (double)(float)iv)};
                    const df u = df_mul(df_mul_f(z, (float)(2 * l - 1)), p1);
                    pl = df_mul(dfa(u, df_mul_f(p2, -(float)(l + m - 1))), inv);
                }
                if (l > m) {
                    p2 = p1;
                    p1 = pl;
                }
                if (l > 0) df_fma_acc(acc[l * l + l + m], pl, cm);
                if (m > 0) df_fma_acc(acc[l * l + l - m], pl, sm);
            }
        }
    }
    int off = 0, lim = L;
    warp_sum_split<L, 16>(acc, off, lim);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mono += __shfl_xor_sync(0xffffffffu, mono, o);
    double scale = 0.0;
    if (i0 < i1) {
        const HartreeRad g = H.rad[a];
        const double rk = g.r0 * exp(g.lnq * (double)(bin - H.rad_off[a]));
        scale = 1.0 / (rk * rk * rk * g.lnq);
    }
    const double unit = __hiloint2double(ew << 20, 0);                 // 2^(ew - 1023)
#pragma unroll
    for (int q = 0; q < (L + 31) / 32; q++)
        if (off + q < lim)
            rho[bin * kL + off + q] = (off + q == 0 ? mono : ((double)acc[q].hi + (double)acc[q].lo) * unit) * scale;
}

__device__ __forceinline__ double warp_scan_up(double v, int lane)       // inclusive, towards higher lanes
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

__device__ __forceinline__ double warp_scan_down(double v, int lane)     // inclusive, towards lower lanes
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_down_sync(0xffffffffu, v, o);
        if (lane + o < 32) v += u;
    }
    return v;
}

constexpr int kRadShells = 256;         // shells the radial equation keeps in shared memory
constexpr int kRadWarps = 4;            // warps a CTA

// The radial equation of atom a for one (l, m) by one warp, lanes along the
// shells: the partial integrals as warp scans.  F and V: n doubles each of
// the warp's own, `st` apart (shared memory, or the global scratch of an atom
// with more shells than that).
template <int l, class Radius>
__device__ void radial_lm(const DevPlan &P, const HartreeRad &g, int a, int mi, long long o, const HartreeTabs &T,
                          const Radius &rk, double *F, double *V, int st)
{
    const int lane = threadIdx.x & 31, n = g.nrad;
    const double h24 = g.lnq / 24.0;
    const double *rho = T.rho + o * kL + l * l + mi;
    // the integrands per dx = dr / r: f = rho r^(l+3) (inner), g = rho r^(2-l) (outer, over f)
    for (int k = lane; k < n; k += 32) F[k * st] = rho[k * kL] * ipow(rk(k), l + 3);
    __syncwarp();
    // integral over interval [k, k+1] of the cubic through the nearest four samples (n >= 4)
    auto seg = [&](int k) {
        auto v = [&](int j) { return F[j * st]; };
        if (k == 0) return h24 * (9.0 * v(0) + 19.0 * v(1) - 5.0 * v(2) + v(3));
        if (k == n - 2) return h24 * (v(n - 4) - 5.0 * v(n - 3) + 19.0 * v(n - 2) + 9.0 * v(n - 1));
        return h24 * (13.0 * (v(k) + v(k + 1)) - (v(k - 1) + v(k + 2)));
    };
    // 4 pi/(2l+1), times K_lm^2 for the two unnormalised harmonics (moment, evaluation)
    double pref = 0.0;
#pragma unroll
    for (int m = 0; m < 2 * l + 1; m++)
        if (m == mi) pref = 4.0 * 3.14159265358979323846 / (2.0 * l + 1.0) * ylm_norm2(l, m - l);
    double carry = F[0] / (double)(l + 3);
    // inner integrals, forward: the inner part of V
    for (int k0 = 0; k0 < n; k0 += 32) {
        const int k = k0 + lane;
        const double ir = 1.0 / ipow(rk(min(k, n - 1)), l + 1);
        const double iin = carry + warp_scan_up(k > 0 && k < n ? seg(k - 1) : 0.0, lane);
        if (k < n) V[k * st] = pref * iin * ir;
        carry = __shfl_sync(0xffffffffu, iin, 31);
    }
    if (lane == 0) {
        if (l == 0) {
            const float *aa = P.atom_dd + 6 * a;
            const df q = df_from_double(pref * carry);
            T.rec[3 * a] = make_float4(aa[0], aa[1], aa[2], aa[3]);
            T.rec[3 * a + 1] = make_float4(aa[4], aa[5], g.rmax2_hi, g.rmax2_lo);
            T.rec[3 * a + 2] = make_float4(q.hi, q.lo, 0.f, 0.f);
        } else {
            T.Qf[(long long)a * kLf + l * l + mi - 1] = (float)(pref * carry);
        }
    }
    __syncwarp();
    for (int k = lane; k < n; k += 32) {
        const double r = rk(k), rg = l <= 2 ? ipow(r, 2 - l) : 1.0 / ipow(r, l - 2);
        F[k * st] = rho[k * kL] * rg;
    }
    __syncwarp();
    // outer integrals, backward; V = inner + outer part, stored once
    carry = 0.0;
    for (int k0 = (n - 1) / 32 * 32; k0 >= 0; k0 -= 32) {
        const int k = k0 + lane;
        const double rl = ipow(rk(min(k, n - 1)), l);
        const double iout = carry + warp_scan_down(k < n - 1 ? seg(k) : 0.0, lane);
        if (k < n) {
            const double v = V[k * st] + pref * iout * rl;
            if (l == 0) T.V0[o + k] = v;
            else T.Vf[(o + k) * kLf + l * l + mi - 1] = (float)v;
        }
        carry = __shfl_sync(0xffffffffu, iout, 0);
    }
}

// One warp per (atom, l, m), the warps of a CTA on one atom; the warp with
// l = 0 also packs the atom's records for the evaluation.
//
// Bound by latency and by the FP64 unit (two lanes a clock and SM): an
// exponential a shell, once a CTA, and chains of FP64 sums.  A warp per
// (atom, l) with its 2l+1 functions side by side in global scratch kept a few
// SMs busy and the others idle: 67 -> 19 us for 3 atoms, l_max 4; 79 -> 24
// for 64 atoms; 300 -> 184 for 250 atoms, l_max 6.  One warp a CTA gives the
// same for the small systems and 244 us for 250 atoms.
__global__ void __launch_bounds__(32 * kRadWarps) k_hartree_radial(DevPlan P, HartreeDev H, int l_max, HartreeTabs T)
{
    __shared__ double rs[kRadShells], sF[kRadWarps][kRadShells], sV[kRadWarps][kRadShells];
    const int nlm = (l_max + 1) * (l_max + 1), per = (nlm + kRadWarps - 1) / kRadWarps;
    const int a = blockIdx.x / per, warp = threadIdx.x >> 5, lm = (blockIdx.x - a * per) * kRadWarps + warp;
    const int lane = threadIdx.x & 31;
    const HartreeRad g = H.rad[a];
    const int n = g.nrad;
    const long long o = H.rad_off[a];
    const bool smem = n <= kRadShells;
    if (smem)
        for (int k = threadIdx.x; k < n; k += blockDim.x) rs[k] = g.r0 * exp(g.lnq * (double)k);
    __syncthreads();
    if (lm >= nlm) return;
    int l = 0;
    while ((l + 1) * (l + 1) <= lm) l++;
    const int m = lm - l * l;
    auto rk = [&](int k) { return smem ? rs[k] : g.r0 * exp(g.lnq * (double)k); };
    double *F = smem ? sF[warp] : T.F + o * kL + lm, *V = smem ? sV[warp] : T.Vd + o * kL + lm;
    const int st = smem ? 1 : kL;
    switch (l) {
    case 0: radial_lm<0>(P, g, a, m, o, T, rk, F, V, st); break;
    case 1: radial_lm<1>(P, g, a, m, o, T, rk, F, V, st); return;
    case 2: radial_lm<2>(P, g, a, m, o, T, rk, F, V, st); return;
    case 3: radial_lm<3>(P, g, a, m, o, T, rk, F, V, st); return;
    case 4: radial_lm<4>(P, g, a, m, o, T, rk, F, V, st); return;
    case 5: radial_lm<5>(P, g, a, m, o, T, rk, F, V, st); return;
    default: radial_lm<6>(P, g, a, m, o, T, rk, F, V, st); return;
    }
    __syncwarp();
    // the shells' radii, and V_00 on each interval k as the cubic through
    // shells i0 .. i0+3 (i0 = k - 1 clamped to [0, n-4]) in f = x - k,
    // x = ln(r / r_0) / ln q: a_m = p^(m)(o) / m! with o = k - i0 and
    // p(t) = V_i0 + t D1 + t(t-1)/2 D2 + t(t-1)(t-2)/6 D3 (forward differences)
    for (int k = lane; k < n; k += 32) {
        const double r = rk(k);
        const df rh = df_from_double(r), ri = df_from_double(1.0 / r);
        T.rk[o + k] = make_float4(rh.hi, rh.lo, ri.hi, ri.lo);
    }
    for (int k = lane; k + 1 < n; k += 32) {
        const int i0 = k - 1 < 0 ? 0 : (k - 1 > n - 4 ? n - 4 : k - 1);
        const double t = (double)(k - i0);
        const double *v = T.V0 + o + i0;
        const double D1 = v[1] - v[0], D2 = v[2] - 2.0 * v[1] + v[0], D3 = v[3] - 3.0 * v[2] + 3.0 * v[1] - v[0];
        const df a0 = df_from_double(v[k - i0]);
        const df a1 = df_from_double(D1 + (2.0 * t - 1.0) * 0.5 * D2 + (3.0 * t * t - 6.0 * t + 2.0) * (1.0 / 6.0) * D3);
        const df a2 = df_from_double(0.5 * (D2 + (t - 1.0) * D3));
        const df a3 = df_from_double(D3 * (1.0 / 6.0));
        T.c0[2 * (o + k)] = make_float4(a0.hi, a0.lo, a1.hi, a1.lo);
        T.c0[2 * (o + k) + 1] = make_float4(a2.hi, a2.lo, a3.hi, a3.lo);
    }
}

// A row of 48 FP32 coefficients, or the first of it, in 32-byte loads: a load
// costs the L1 a look-up for each lane whose row differs, whatever its width.
template <int N>
__device__ __forceinline__ void load_row(const float *p, float *v)
{
#pragma unroll
    for (int j = 0; j < (N + 7) / 8; j++)
        asm("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=f"(v[8 * j]), "=f"(v[8 * j + 1]), "=f"(v[8 * j + 2]), "=f"(v[8 * j + 3]), "=f"(v[8 * j + 4]),
              "=f"(v[8 * j + 5]), "=f"(v[8 * j + 6]), "=f"(v[8 * j + 7])
            : "l"(p + 8 * j));
}

// CTA per batch, thread per point; the atoms of the batch's system.  Bound by
// the FP32 pipe (about 330 operations a pair of a point and a far atom at l_max
// 6).  Two far atoms at a time in packed FP32 pairs issued a fifth fewer
// instructions and took as long; six CTAs an SM instead of four: 250-atom
// cluster, l_max 6, 28.9 -> 27.2 ms.
template <int LMAX>
__global__ void __launch_bounds__(128, 6) k_hartree_eval(DevPlan P, HartreeDev H, HartreeTabs T, double *vh)
{
    constexpr int L = (LMAX + 1) * (LMAX + 1);
    const DevBatch B = P.batches[blockIdx.x];
    const long long a0 = H.sys_atom0[B.sys], a1 = H.sys_atom0[B.sys + 1];
    for (int i = threadIdx.x; i < B.np; i += blockDim.x) {
        const long long p = B.pt0 + i;
        const float *pp = P.pts_dd + 6 * p;
        const df px{pp[0], pp[1]}, py{pp[2], pp[3]}, pz{pp[4], pp[5]};
        df acc{0.f, 0.f};
        for (long long a = a0; a < a1; a++) {
            const float4 r0 = T.rec[3 * a], r1 = T.rec[3 * a + 1];
            const df dx = dfa(px, df{-r0.x, -r0.y}), dy = dfa(py, df{-r0.z, -r0.w}), dz = dfa(pz, df{-r1.x, -r1.y});
            const df d2 = dfa(dfa(df_sqr(dx), df_sqr(dy)), df_sqr(dz));
            const float ri = d2.hi > 0.f ? rsqrtf(d2.hi) : 0.f;
            float A[L];
            if constexpr (LMAX > 0) ylm_unnormalised<LMAX, float>(dx.hi * ri, dy.hi * ri, dz.hi * ri, A);
            float part = 0.f;
            if (d2.hi > r1.z || (d2.hi == r1.z && d2.lo >= r1.w)) {
                // beyond the last shell: the exterior multipoles
                const float4 r2 = T.rec[3 * a + 2];
                acc = dfa(acc, df_mul(df{r2.x, r2.y}, df_rsqrt(d2, ri)));
                if constexpr (LMAX > 0) {
                    constexpr int NQ4 = (L - 1 + 3) / 4;
                    float q[NQ4 * 4];
                    const float4 *q4 = reinterpret_cast<const float4 *>(T.Qf + a * kLf);
#pragma unroll
                    for (int j = 0; j < NQ4; j++) {
                        const float4 u = q4[j];
                        q[4 * j] = u.x;
                        q[4 * j + 1] = u.y;
                        q[4 * j + 2] = u.z;
                        q[4 * j + 3] = u.w;
                    }
                    float rl = ri * ri;                              // 1/d^(l+1), l = 1
#pragma unroll
                    for (int l = 1; l <= LMAX; l++) {
                        float s = 0.f;
#pragma unroll
                        for (int m = -l; m <= l; m++) s = fmaf(q[l * l + l + m - 1], A[l * l + l + m], s);
                        part = fmaf(s, rl, part);
                        rl *= ri;
                    }
                }
            } else {
                const HartreeRad g = H.rad[a];
                const long long o = H.rad_off[a];
                const float4 R0 = T.rk[o];
                const df r02 = df_sqr(df{R0.x, R0.y});
                if (d2.hi < r02.hi || (d2.hi == r02.hi && d2.lo <= r02.lo)) {
                    // inside the first shell: V(r_0) (d / r_0)^l
                    acc = dfa(acc, df_from_double(T.V0[o]));
                    if constexpr (LMAX > 0) {
                        const float sr = d2.hi * ri * g.inv_r0;
                        const float *vf = T.Vf + o * kLf;
                        float sl = sr;
#pragma unroll
                        for (int l = 1; l <= LMAX; l++) {
                            float s = 0.f;
#pragma unroll
                            for (int m = -l; m <= l; m++) s = fmaf(vf[l * l + l + m - 1], A[l * l + l + m], s);
                            part = fmaf(s, sl, part);
                            sl *= sr;
                        }
                    }
                } else {
                    // between shells: interval k (r_k <= d < r_k+1), f = ln(d / r_k) / ln q
                    int k, i0;
                    float t;
                    if (g.df_log) {
                        // double-float: k from an FP32 estimate of x = ln(d / r_0) / ln q,
                        // corrected against the radii; ln(d / r_k) = 2 atanh(s),
                        // s = u / (2 + u), u = d / r_k - 1 < q - 1:
                        // 2 s + s z (2/3 + z (2/5 + z R(z))), z = s^2, with the terms
                        // to s^5 as double-floats and R = 2/7 + 2/9 z + ... + 2/19 z^6
                        // in FP32 (ln q <= 0.6 keeps s <= 0.3; the FP32 part's rounding
                        // and the first dropped term, 2 s^21 / 21, together stay below
                        // 6e-12 in ln(d / r_k))
                        const df d = df_sqrt(d2);
                        k = (int)floorf((__logf(d.hi) - g.ln_r0_f) * g.inv_lnq_f);
                        k = k < 0 ? 0 : (k > g.nrad - 2 ? g.nrad - 2 : k);
                        float4 Rk = T.rk[o + k];
                        if (k > 0 && (d.hi < Rk.x || (d.hi == Rk.x && d.lo < Rk.y))) {
                            k--;
                            Rk = T.rk[o + k];
                        } else if (k < g.nrad - 2) {
                            const float4 R1 = T.rk[o + k + 1];
                            if (!(d.hi < R1.x || (d.hi == R1.x && d.lo < R1.y))) {
                                k++;
                                Rk = R1;
                            }
                        }
                        const df u = dfa(df_mul(d, df{Rk.z, Rk.w}), df{-1.f, 0.f});
                        const df sv = df_mul(u, df_rcp(dfa(u, df{2.f, 0.f})));
                        const df z = df_sqr(sv);
                        float rz = 2.f / 19.f;
                        rz = fmaf(rz, z.hi, 2.f / 17.f);
                        rz = fmaf(rz, z.hi, 2.f / 15.f);
                        rz = fmaf(rz, z.hi, 2.f / 13.f);
                        rz = fmaf(rz, z.hi, 2.f / 11.f);
                        rz = fmaf(rz, z.hi, 2.f / 9.f);
                        rz = fmaf(rz, z.hi, 2.f / 7.f);
                        df ser = dfa_f(df{kTwoFifthHi, kTwoFifthLo}, z.hi * rz);     // 2/5 + z R
                        ser = dfa(df{kTwoThirdHi, kTwoThirdLo}, df_mul(z, ser));     // 2/3 + z (...)
                        const df ln1p = dfa(df{2.f * sv.hi, 2.f * sv.lo}, df_mul(sv, df_mul(z, ser)));
                        const df f = df_mul(ln1p, df{g.inv_lnq_hi, g.inv_lnq_lo});
                        // V_00 = a0 + f (a1 + f (a2 + f a3)) on interval k
                        const float4 c01 = T.c0[2 * (o + k)], c23 = T.c0[2 * (o + k) + 1];
                        df pv = dfa(df{c23.x, c23.y}, df_mul(f, df{c23.z, c23.w}));
                        pv = dfa(df{c01.z, c01.w}, df_mul(f, pv));
                        pv = dfa(df{c01.x, c01.y}, df_mul(f, pv));
                        acc = dfa(acc, pv);
                        i0 = k - 1 < 0 ? 0 : (k - 1 > g.nrad - 4 ? g.nrad - 4 : k - 1);
                        t = (float)(k - i0) + f.hi;
                    } else {
                        // coarse radial grids: FP64 logarithm and Lagrange weights
                        const double dd2 = (double)d2.hi + (double)d2.lo;
                        const double *v0 = T.V0 + o;
                        const double x = (0.5 * log(dd2) - g.ln_r0) * g.inv_lnq;
                        i0 = (int)floor(x) - 1;
                        i0 = i0 < 0 ? 0 : (i0 > g.nrad - 4 ? g.nrad - 4 : i0);
                        const double td = x - (double)i0;
                        const double w0 = -(td - 1.0) * (td - 2.0) * (td - 3.0) * (1.0 / 6.0);
                        const double w1 = td * (td - 2.0) * (td - 3.0) * 0.5;
                        const double w2 = -td * (td - 1.0) * (td - 3.0) * 0.5;
                        const double w3 = td * (td - 1.0) * (td - 2.0) * (1.0 / 6.0);
                        acc = dfa(acc, df_from_double(w0 * v0[i0] + w1 * v0[i0 + 1] + w2 * v0[i0 + 2] + w3 * v0[i0 + 3]));
                        t = (float)td;
                        k = 0;
                    }
                    (void)k;
                    if constexpr (LMAX > 0) {
                        // l >= 1: Lagrange weights at nodes t = 0, 1, 2, 3 (shells i0 .. i0+3), FP32
                        const float f0 = -(t - 1.f) * (t - 2.f) * (t - 3.f) * (1.f / 6.f);
                        const float f1 = t * (t - 2.f) * (t - 3.f) * 0.5f;
                        const float f2 = -t * (t - 1.f) * (t - 3.f) * 0.5f;
                        const float f3 = t * (t - 1.f) * (t - 2.f) * (1.f / 6.f);
                        const float *vf = T.Vf + (o + i0) * kLf;
                        // eight coefficients of the four rows at a time, in pairs
                        const pk w0 = pk_dup(f0), w1 = pk_dup(f1), w2 = pk_dup(f2), w3 = pk_dup(f3);
#pragma unroll
                        for (int q8 = 0; q8 < L - 1; q8 += 8) {
                            float v0[8], v1[8], v2[8], v3[8];
                            load_row<8>(vf + q8, v0);
                            load_row<8>(vf + kLf + q8, v1);
                            load_row<8>(vf + 2 * kLf + q8, v2);
                            load_row<8>(vf + 3 * kLf + q8, v3);
#pragma unroll
                            for (int q = 0; q < 8; q += 2) {
                                if (q8 + q >= L - 1) break;
                                const pk v = fma2(w3, pk_make(v3[q], v3[q + 1]),
                                                  fma2(w2, pk_make(v2[q], v2[q + 1]),
                                                       fma2(w0, pk_make(v0[q], v0[q + 1]),
                                                            w1 * pk_make(v1[q], v1[q + 1]))));
                                const float2 u = pk_get(v);
                                part = fmaf(u.x, A[q8 + q + 1], part);
                                if (q8 + q + 1 < L - 1) part = fmaf(u.y, A[q8 + q + 2 < L ? q8 + q + 2 : 0], part);
                            }
                        }
                    }
                }
            }
            acc = dfa_f(acc, part);
        }
        vh[p] = (double)acc.hi + (double)acc.lo;
    }
}

}  // namespace

HartreeRad hartree_rad(double r_min, double ln_q, int n_rad)
{
    HartreeRad g{};
    g.r0 = r_min;
    g.lnq = ln_q;
    g.inv_lnq = 1.0 / ln_q;
    g.ln_r0 = std::log(r_min);
    const double rmax = r_min * std::exp(ln_q * (double)(n_rad - 1));
    const double r2 = rmax * rmax;
    const df d = df_from_double(r2);
    // a normalised pair: hi the nearest float, lo the remainder rounded
    g.rmax2_hi = d.hi;
    g.rmax2_lo = d.lo;
    g.inv_r0 = (float)(1.0 / r_min);
    g.nrad = n_rad;
    const df il = df_from_double(1.0 / ln_q);
    g.inv_lnq_hi = il.hi;
    g.inv_lnq_lo = il.lo;
    g.ln_r0_f = (float)std::log(r_min);
    g.inv_lnq_f = (float)(1.0 / ln_q);
    g.df_log = ln_q <= 0.6 ? 1 : 0;
    return g;
}

size_t hartree_ws_bytes(const HartreeDev &H)
{
    return 3 * al256(sizeof(double) * kL * (size_t)H.n_shells) + al256(sizeof(float4) * 3 * (size_t)H.n_atoms) +
           al256(sizeof(float4) * (size_t)H.n_shells) + al256(sizeof(float4) * 2 * (size_t)H.n_shells) +
           al256(sizeof(double) * (size_t)H.n_shells) +
           al256(sizeof(float) * kLf * (size_t)H.n_shells) +
           al256(sizeof(float) * kLf * (size_t)H.n_atoms);
}

cudaError_t launch_hartree(const DevPlan &P, const HartreeDev &H, int n_batch, int l_max,
                           const double *n, double *vh, double *ws, cudaStream_t s)
{
    const HartreeTabs T = carve(H, ws);
    cudaError_t e = cudaSuccess;
    if (H.n_shells > 0) {
        const unsigned grid = (unsigned)((H.n_shells + 3) / 4);
        switch (l_max) {
        case 0: k_hartree_moments<0><<<grid, 128, 0, s>>>(P, H, n, T.rho); break;
        case 1: k_hartree_moments<1><<<grid, 128, 0, s>>>(P, H, n, T.rho); break;
        case 2: k_hartree_moments<2><<<grid, 128, 0, s>>>(P, H, n, T.rho); break;
        case 3: k_hartree_moments<3><<<grid, 128, 0, s>>>(P, H, n, T.rho); break;
        case 4: k_hartree_moments<4><<<grid, 128, 0, s>>>(P, H, n, T.rho); break;
        case 5: k_hartree_moments<5><<<grid, 128, 0, s>>>(P, H, n, T.rho); break;
        default: k_hartree_moments<6><<<grid, 128, 0, s>>>(P, H, n, T.rho); break;
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (H.n_atoms > 0) {
        const int nlm = (l_max + 1) * (l_max + 1), per = (nlm + kRadWarps - 1) / kRadWarps;
        k_hartree_radial<<<(unsigned)(H.n_atoms * per), 32 * kRadWarps, 0, s>>>(P, H, l_max, T);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (n_batch > 0) {
        switch (l_max) {
        case 0: k_hartree_eval<0><<<n_batch, 128, 0, s>>>(P, H, T, vh); break;
        case 1: k_hartree_eval<1><<<n_batch, 128, 0, s>>>(P, H, T, vh); break;
        case 2: k_hartree_eval<2><<<n_batch, 128, 0, s>>>(P, H, T, vh); break;
        case 3: k_hartree_eval<3><<<n_batch, 128, 0, s>>>(P, H, T, vh); break;
        case 4: k_hartree_eval<4><<<n_batch, 128, 0, s>>>(P, H, T, vh); break;
        case 5: k_hartree_eval<5><<<n_batch, 128, 0, s>>>(P, H, T, vh); break;
        default: k_hartree_eval<6><<<n_batch, 128, 0, s>>>(P, H, T, vh); break;
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace fgi
