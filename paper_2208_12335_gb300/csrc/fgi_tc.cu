// Tensor-core path for sm_103a: basis evaluation into swizzled BF16 operand
// images, the H contraction h_b = Phi_b^T diag(w v) Phi_b on tcgen05 (or
// s Psi_b^T Psi_b with Psi = Phi sqrt|w v| where w v has one sign s) with a
// fixed-point scatter into H, the D_b gather, and the density contraction
// n_p = sum_j (D_b Phi_b^T)_jp phi_j(p) on tcgen05.
//
// Precision: every value x entering a contraction is split into three BF16
// terms x = x0 + x1 + x2: x0 a fixed-point digit on a power-of-two grid per
// row (H) or per point (density), chosen so that every partial sum of
// x0*y0 products is exact in FP32, and x1, x2 the BF16 split of the
// remainder.  H and the density accumulate the 8 products of combined
// order <= 3 except x2*y2; x0*y0 has its own FP32
// accumulator in tensor memory, the others a second one.  Cross-batch sums:
// H in 2^-40 fixed point (int64 atomics, deterministic), the density in
// FP64.  n_split = 1 keeps x0*y0 only (plain BF16).
#include <cuda_bf16.h>

#include <algorithm>
#include <climits>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/fgi.h"
#include "fgi_basis.cuh"
#include "fgi_bounds.h"
#include "fgi_dd.cuh"
#include "fgi_index.cuh"
#include "fgi_tc.h"

namespace fgi {

namespace {

// ------------------------------------------------------------ PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

constexpr uint64_t kWaitLimitNs = 2000000000ull;   // 2 s: a wait that long means a bug

// Bounded wait on an mbarrier phase (time-out: kStatusTimeout), with a CTA-wide abort flag: once any wait of the CTA has
// timed out, every later wait fails at once, so that the roles finish their
// loops quickly with unchanged control flow (no named barrier is skipped).
__device__ __forceinline__ bool mbar_wait_a(uint64_t *bar, uint32_t parity, int *status, volatile int *abort)
{
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort) return false;
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (*abort) return false;
        if (global_ns() - t0 > kWaitLimitNs) {
            *abort = 1;
            atomicOr(status, kStatusTimeout);
            return false;
        }
    }
    return true;
}

// At the end of a role: wait, as long at most, for what it has itself in flight (bulk
// copies, MMAs), whatever the abort flag says: shared and tensor memory are
// given up when the CTA leaves, also after a time-out.
__device__ __forceinline__ bool mbar_drain(uint64_t *bar, uint32_t parity)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait(bar, parity))
        if (global_ns() - t0 > kWaitLimitNs) return false;
    return true;
}

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// add to a global 64-bit word where pred holds, without a branch
__device__ __forceinline__ void red_add_if(bool pred, unsigned long long addr, long long x)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t"
                 "@p red.relaxed.gpu.global.add.u64 [%0], %1;\n\t}" ::"l"(addr), "l"(x), "r"((int)pred)
                 : "memory");
}

// the largest of m, |a|, |b|; NaN when one of them is
__device__ __forceinline__ float max_abs_nan(float m, float a, float b)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(fabsf(a)), "f"(fabsf(b)));
    return r;
}

__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)),
                 "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// one lane of a converged warp
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// 32 lanes x 32 consecutive 32-bit columns: thread (lane) gets its row's 32 values
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float *v)
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
          "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
          "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
          "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 32; i++) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float *v)
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, 128-byte swizzle (tcgen05 format: version 1).
// K-major: rows of 64 BF16 (128 B), 8-row atoms of 1 KB; sbo = atom stride.
// MN-major: lbo = stride between 64-element MN atoms, sbo = stride between
// 8-row K groups.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}

// Instruction descriptor: kind::f16, BF16 x BF16 -> F32, dense.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn, bool b_mn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// --------------------------------------------------------------- splitting
// byte offset (plane 0) of the 16-byte unit (row r, 8-column group g) inside
// chunk (blk, c); a chunk's three planes follow each other
__device__ __forceinline__ long long unit_offset(int blk, int nchunk, int c, int r, int g)
{
    return (long long)(blk * nchunk + c) * kChunkStride + r * 128 + ((g ^ (r & 7)) << 4);
}

// Adding and subtracting it rounds |x| < 2^22 to the nearest integer (ties to even)
constexpr float kRoundMagic = 12582912.f;            // 1.5 * 2^23

// Normalisation constants of the real spherical harmonics as double-floats.
#define FGI_DF_CONST(c) {(float)(c), (float)((c) - (double)(float)(c))}
__constant__ float2 kYlmC[10] = {
    FGI_DF_CONST(0.28209479177387814),  // l0
    FGI_DF_CONST(0.4886025119029199),   // l1
    FGI_DF_CONST(1.0925484305920792),   // l2: xy, yz, xz
    FGI_DF_CONST(0.31539156525252005),  // l2: 2z^2 - x^2 - y^2
    FGI_DF_CONST(0.5462742152960396),   // l2: x^2 - y^2
    FGI_DF_CONST(0.5900435899266435),   // l3: y(3x^2 - y^2), x(x^2 - 3y^2)
    FGI_DF_CONST(2.890611442640554),    // l3: xyz
    FGI_DF_CONST(0.4570457994644658),   // l3: y(4z^2 - x^2 - y^2), x(...)
    FGI_DF_CONST(0.3731763325901154),   // l3: z(2z^2 - 3x^2 - 3y^2)
    FGI_DF_CONST(1.445305721320277)};   // l3: z(x^2 - y^2)
#undef FGI_DF_CONST

// r^l Y_lm = C_lm * Q_lm(x, y, z): Q with small integer coefficients (FP32),
// the constant index into kYlmC.
__device__ __forceinline__ void ylm_poly_f32(int l, float x, float y, float z, float *Q, int *ci)
{
    if (l == 0) {
        Q[0] = 1.f; ci[0] = 0;
    } else if (l == 1) {
        Q[0] = y; Q[1] = z; Q[2] = x;
        ci[0] = ci[1] = ci[2] = 1;
    } else if (l == 2) {
        Q[0] = x * y; Q[1] = y * z; Q[2] = 2.f * z * z - x * x - y * y; Q[3] = x * z; Q[4] = x * x - y * y;
        ci[0] = 2; ci[1] = 2; ci[2] = 3; ci[3] = 2; ci[4] = 4;
    } else {
        const float q = 4.f * z * z - x * x - y * y;
        Q[0] = y * (3.f * x * x - y * y); Q[1] = x * y * z; Q[2] = y * q;
        Q[3] = z * (2.f * z * z - 3.f * x * x - 3.f * y * y); Q[4] = x * q; Q[5] = z * (x * x - y * y);
        Q[6] = x * (x * x - 3.f * y * y);
        ci[0] = 5; ci[1] = 6; ci[2] = 7; ci[3] = 8; ci[4] = 7; ci[5] = 9; ci[6] = 5;
    }
}

// two FP32 values rounded to BF16, lo in the low half
__device__ __forceinline__ uint32_t pack2_bf16(float lo, float hi)
{
    const __nv_bfloat162 w = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&w);
}

// Split with a fixed-point leading term: x0 = m * unit, m = rint(x / unit),
// unit = 2^(e-7) with 2^e >= the row's largest |x|, so |m| <= 128 and every
// product x0*y0 of a row pair is an integer multiple of unit_x*unit_y not
// exceeding 2^14 in units; a sum of up to 1024 of them (a batch) is exact in
// FP32 whatever the accumulator's rounding.  The remainder x - x0 is split
// relative to itself into two BF16 terms.  x.hi - x0 is exact: x0 is a
// multiple of unit, and unit >= ulp(x.hi) because |x.hi| <= 2^e (1 + 2^-12)
// and unit = 2^(e - bits), bits <= 8.

// Power-of-two scale 2^(b-e) and unit 2^(e-b) for a row whose largest |x|
// is mx: |x| * scale <= 2^b.  b digit bits keep the exact sum: 2^(2b) times
// the contraction depth must not exceed 2^24.  Rows below 1e-30 (negligible
// against any stored value) put everything in the remainder terms.
__device__ __forceinline__ int fixed_bits(int depth)
{
    int b = 7;
    while (b > 1 && ((long long)depth << (2 * b)) > (1ll << 24)) b--;
    return b;
}

// Leading-digit width: 8 bits when the row's sum S = sum|x|/2^e <= 200 (then
// every row-pair sum stays below 65536 S + 128 K < 2^24 for K <= 8192),
// otherwise the width that keeps depth x 2^(2b) <= 2^24.
__device__ __forceinline__ void fixed_scale_adaptive(float mx, float sum, int depth, float &scale, float &unit)
{
    if (!(mx > 1e-30f)) {
        scale = 0.f;
        unit = 0.f;
        return;
    }
    int e;
    frexpf(mx * (1.f + 1.f / 4096.f), &e);
    const float S = ldexpf(sum, -e) * 1.001f;
    const int bits = (S <= 200.f) ? 8 : fixed_bits(depth);
    scale = ldexpf(1.f, bits - e);
    unit = ldexpf(1.f, e - bits);
}


// FP32 u(d)/d^(l+1) for the first passes, which only take maxima and sums
// of |phi| from it (a relative error of a few ulp is far inside the 2^-12
// margin of the fixed-point grids); inv_d = 1/d, computed once per point.
// tab: the radial's interval-0 entry (hi coefficients), entries `step` float4 apart.
__device__ __forceinline__ float radial_over_d_f32(const DevRadial &R, const float4 *tab, int step, float d,
                                                   float inv_d)
{
    if (d >= R.rcut_f) return 0.f;
    if (d < 1e-12f) return R.l == 0 ? __ldg(tab).y * R.inv_h_hi : 0.f;
    const float s = d * R.inv_h_hi;
    int k = (int)s;
    if (k > R.nk - 2) k = R.nk - 2;
    const float t = s - (float)k;
    const float4 c = __ldg(tab + (long long)k * step);
    const float u = c.x + t * (c.y + t * (c.z + t * c.w));
    const float i2 = inv_d * inv_d;
    const float ip = R.l == 0 ? inv_d : (R.l == 1 ? i2 : (R.l == 2 ? i2 * inv_d : i2 * i2));
    return u * ip;
}

// Interval-0 entry of shell sh's spline and the distance between interval
// entries: the species' interleaved table when its shells share one grid.
__device__ __forceinline__ const float4 *spline_tab(const DevPlan &P, const DevSpecies &S, const DevRadial &R, int sh,
                                                    int &step)
{
    if (S.shared_grid) {
        step = 2 * S.n_shell;
        return P.scoef + S.scoef_off + 2 * sh;
    }
    step = 2;
    return P.coef_dd + 2 * R.coef_off;
}

// ----------------------------------------- basis evaluation, two points a lane
// A warp evaluates every function of one atom at the 64 points of a chunk, two
// neighbouring points a lane in packed FP32 pairs (half the issue slots, which
// bound the kernels), and hands each pair of values straight to an emitter
// (split + one 32-bit store a plane into the operand image): values never pass
// through shared memory, and a warp stores whole 128-byte image rows.  The
// geometry (offset, distance, 1/d^(l+1)) is double-float once per (point,
// atom); the radial factor once per shell, times the per-point scale of each
// image; the angular polynomial FP32.

// One value split on its row's or point's grid (as above; NSPLIT 1:
// plain BF16) and stored as one 16-bit BF16 per plane
template <int NSPLIT>
__device__ __forceinline__ void store_value(uint8_t *dst, df x, float scale, float unit)
{
    if (NSPLIT == 3) {
        // the rounding to an integer as an addition (the FRND
        // unit has a sixteenth of the FADD rate): |x scale| <= 2^8, far inside
        // 2^22.  x0 has at most 9 significant bits, 8 below a power of two: its
        // BF16 form is the upper half of the word.
        const float x0 = (fmaf(x.hi, scale, kRoundMagic) - kRoundMagic) * unit;
        const float d = x.hi - x0;
        const __nv_bfloat16 b = __float2bfloat16_rn(d);
        const __nv_bfloat16 c = __float2bfloat16_rn((d - __bfloat162float(b)) + x.lo);
        *reinterpret_cast<unsigned short *>(dst) = (unsigned short)(__float_as_uint(x0) >> 16);
        *reinterpret_cast<unsigned short *>(dst + kChunkBytes) = __bfloat16_as_ushort(b);
        *reinterpret_cast<unsigned short *>(dst + 2 * kChunkBytes) = __bfloat16_as_ushort(c);
    } else {
        *reinterpret_cast<unsigned short *>(dst) = __bfloat16_as_ushort(__float2bfloat16_rn(x.hi));
    }
}

// The same for the values hi - nlo of two neighbouring points (scale and unit a
// pair too): one 32-bit store a plane
template <int NSPLIT>
__device__ __forceinline__ void store_pair(uint8_t *dst, pk hi, pk nlo, pk scale, pk unit)
{
    if (NSPLIT == 3) {
        const pk x0 = (fma2(hi, scale, pk_dup(kRoundMagic)) + pk_dup(-kRoundMagic)) * unit;
        const pk d = hi - x0;
        const float2 xf = pk_get(x0), df_ = pk_get(d);
        const uint32_t b = pack2_bf16(df_.x, df_.y);
        const pk e = (d - pk_make(__uint_as_float(b << 16), __uint_as_float(b & 0xFFFF0000u))) - nlo;
        const float2 ef = pk_get(e);
        *reinterpret_cast<uint32_t *>(dst) = __byte_perm(__float_as_uint(xf.x), __float_as_uint(xf.y), 0x7632);
        *reinterpret_cast<uint32_t *>(dst + kChunkBytes) = b;
        *reinterpret_cast<uint32_t *>(dst + 2 * kChunkBytes) = pack2_bf16(ef.x, ef.y);
    } else {
        const float2 hf = pk_get(hi);
        *reinterpret_cast<uint32_t *>(dst) = pack2_bf16(hf.x, hf.y);
    }
}

template <int NSPLIT>
__device__ __forceinline__ void store_zero(uint8_t *dst)
{
#pragma unroll
    for (int pl = 0; pl < NSPLIT; pl++) *reinterpret_cast<unsigned short *>(dst + pl * kChunkBytes) = 0;
}

// Ratios of the other normalisation constants of an l shell to its first
// (the spline tables of the basis kernels hold u times the first constant):
// l = 2: C(2z^2-x^2-y^2)/C(xy) = 1/(2 sqrt 3); l = 3: C(z(x^2-y^2))/C(y(3x^2-y^2))
// = sqrt 6 (C(xyz) is twice that), sqrt(3/5) and sqrt(2/5).
#define FGI_DF_CONST(c) {(float)(c), (float)((c) - (double)(float)(c))}
__constant__ float2 kYlmRatio[4] = {
    FGI_DF_CONST(0.28867513459481287),   // 1/(2 sqrt 3)
    FGI_DF_CONST(2.449489742783178),     // sqrt 6
    FGI_DF_CONST(0.7745966692414834),    // sqrt(3/5)
    FGI_DF_CONST(0.6324555320336759)};   // sqrt(2/5)
#undef FGI_DF_CONST

// r^l Y_lm / C_l (C_l the first constant of the shell) = K_g * Q_m: Q in
// FP32 with the exact factors 2 and 1/2 folded in, g the index of the
// ratio K (0: K = 1).
template <int L>
__device__ __forceinline__ void ylm_poly_unit(float x, float y, float z, float *Q, int *g)
{
    if (L == 0) {
        Q[0] = 1.f; g[0] = 0;
    } else if (L == 1) {
        Q[0] = y; Q[1] = z; Q[2] = x;
        g[0] = g[1] = g[2] = 0;
    } else if (L == 2) {
        Q[0] = x * y; Q[1] = y * z; Q[2] = fmaf(-y, y, fmaf(2.f * z, z, -(x * x))); Q[3] = x * z;
        Q[4] = 0.5f * fmaf(x, x, -(y * y));
        g[0] = 0; g[1] = 0; g[2] = 1; g[3] = 0; g[4] = 0;
    } else {
        const float xx = x * x, q = fmaf(-y, y, fmaf(4.f * z, z, -xx));
        Q[0] = y * fmaf(-y, y, (3.f * x) * x);
        Q[1] = 2.f * ((x * y) * z);
        Q[2] = y * q;
        Q[3] = z * fmaf(-(3.f * y), y, fmaf(2.f * z, z, -((3.f * x) * x)));
        Q[4] = x * q;
        Q[5] = z * fmaf(-y, y, xx);
        Q[6] = x * fmaf(-(3.f * y), y, xx);
        g[0] = 0; g[1] = 1; g[2] = 2; g[3] = 3; g[4] = 2; g[5] = 1; g[6] = 0;
    }
}

// the 2l+1 values of one shell for NIMG radial factors rk[k] (= C_l
// u/d^(l+1) times the image's per-point scale), handed to the emitter as
// unnormalised double-floats (the split uses hi + lo only)
template <int L, int NIMG, class Emit>
__device__ __forceinline__ void emit_shell_lane(const df *rk, float x, float y, float z, int f0, int f_lo, int f_hi,
                                                Emit &emit)
{
    constexpr int NM = 2 * L + 1;
    constexpr int NG = L < 2 ? 1 : (L == 2 ? 2 : 4);
    constexpr int G0 = L == 2 ? 0 : 1;               // first kYlmRatio entry of groups 1..
    if constexpr (L == 0) {                          // the angular factor is 1
        if (f0 >= f_lo && f0 < f_hi) emit(f0, rk);
        return;
    }
    float Q[NM];
    int gi[7];
    ylm_poly_unit<L>(x, y, z, Q, gi);
    df rc[NIMG][NG];
#pragma unroll
    for (int k = 0; k < NIMG; k++) {
        rc[k][0] = rk[k];
#pragma unroll
        for (int c = 1; c < NG; c++)
            rc[k][c] = df_mul(rk[k], df{kYlmRatio[G0 + c - 1].x, kYlmRatio[G0 + c - 1].y});
    }
    const bool whole = f0 >= f_lo && f0 + NM <= f_hi;
#pragma unroll
    for (int m = 0; m < NM; m++) {
        const int fm = f0 + m;
        if (!whole && (fm < f_lo || fm >= f_hi)) continue;
        df val[NIMG];
#pragma unroll
        for (int k = 0; k < NIMG; k++) val[k] = df_mul_f_raw(rc[k][gi[m]], Q[m]);
        emit(fm, val);
    }
}

// the same polynomials for two points, rounding for rounding
template <int L>
__device__ __forceinline__ void ylm_poly_unit2(pk x, pk y, pk z, pk *Q, int *g)
{
    if (L == 1) {
        Q[0] = y; Q[1] = z; Q[2] = x;
        g[0] = g[1] = g[2] = 0;
    } else if (L == 2) {
        const pk two = pk_dup(2.f), half = pk_dup(0.5f);
        Q[0] = x * y; Q[1] = y * z;
        Q[2] = fma2(-y, y, fma2(two * z, z, -(x * x)));
        Q[3] = x * z;
        Q[4] = half * fma2(x, x, -(y * y));
        g[0] = 0; g[1] = 0; g[2] = 1; g[3] = 0; g[4] = 0;
    } else {
        const pk two = pk_dup(2.f), three = pk_dup(3.f), four = pk_dup(4.f);
        const pk xx = x * x;
        const pk q = fma2(-y, y, fma2(four * z, z, -xx));
        Q[0] = y * fma2(-y, y, (three * x) * x);
        Q[1] = two * ((x * y) * z);
        Q[2] = y * q;
        Q[3] = z * fma2(-(three * y), y, fma2(two * z, z, -((three * x) * x)));
        Q[4] = x * q;
        Q[5] = z * fma2(-y, y, xx);
        Q[6] = x * fma2(-(three * y), y, xx);
        g[0] = 0; g[1] = 1; g[2] = 2; g[3] = 3; g[4] = 2; g[5] = 1; g[6] = 0;
    }
}

// a point's or an atom's coordinates as double-floats (24 bytes, 8-byte aligned)
struct Dd3 {
    float2 x, y, z;
};
__device__ __forceinline__ Dd3 load_dd3(const float *p)
{
    const float2 *q = reinterpret_cast<const float2 *>(p);
    return Dd3{__ldg(q), __ldg(q + 1), __ldg(q + 2)};
}

// FP32 difference of two positions (from the double-floats)
__device__ __forceinline__ float3 offset_f32(const Dd3 &p, const Dd3 &a)
{
    return make_float3((p.x.x - a.x.x) + (p.x.y - a.x.y), (p.y.x - a.y.x) + (p.y.y - a.y.y),
                       (p.z.x - a.z.x) + (p.z.y - a.z.y));
}

// One interval of a shell's spline: c0..c3 and the low parts of c0 and c1.
// The 32-byte entry in one load: the lanes' intervals differ, so a load costs
// the L1 one tag look-up per lane, and two 16-byte loads cost two.  (These
// look-ups, with those of the bounds below, kept the L1 60 % busy beside an
// issue rate of 64 %.  One load an entry, one for four shells' bounds and the
// lanes without divergence: 64-atom Si cluster, 1.11 M points, H images 3.75
// -> 2.68 ms, density images 2.62 -> 1.84 ms; 75-atom cluster with f shells,
// two images a batch, 6.57 -> 3.72 ms.)
struct SplineEntry {
    float4 h;
    float2 l;
};
__device__ __forceinline__ SplineEntry load_entry(const float4 *p)
{
    SplineEntry e;
    asm("{\n\t.reg .f32 u0, u1;\n\t"
        "ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,u0,u1}, [%6];\n\t}"
        : "=f"(e.h.x), "=f"(e.h.y), "=f"(e.h.z), "=f"(e.h.w), "=f"(e.l.x), "=f"(e.l.y)
        : "l"(p));
    return e;
}

// u = c0 + t c1 + t^2 (c2 + t c3) at t + tl: c0 + t c1 in double-float
__device__ __forceinline__ df spline_value(const SplineEntry &e, float t, float tl)
{
    const df lin = df_two_prod(t, e.h.y);
    const float lin_lo = fmaf(t, e.l.y, fmaf(tl, e.h.y, lin.lo));
    const float quad = (t * t) * fmaf(t, e.h.w, e.h.z);
    const df uu = df_two_sum(e.h.x, lin.hi);
    return df_two_sum(uu.hi, uu.lo + ((e.l.x + lin_lo) + quad));
}

// Every function [f_lo, f_hi) of atom `atom` (species S, shell table sh_tab
// indexed from S.shell0) at the point pp (has: there is one), for any
// species and any point: each shell's own knots, and the point at the
// nucleus.  emit(f, val[NIMG]) receives phi times the image's scale (SCALED
// false: image 0 unscaled); emit0(f) a value that is zero in every image.
template <int NIMG, bool SCALED, class Emit, class Emit0>
__device__ __forceinline__ void eval_atom_general(const float4 *coef, const DevSpecies &S, const DevShell *sh_tab,
                                                  const Dd3 &aa, const Dd3 &pp, bool has, int f_lo, int f_hi,
                                                  const df *scale, Emit &emit, Emit0 &emit0)
{
    const df zero{0.f, 0.f};
    const float3 o = offset_f32(pp, aa);
    const float rcs = (float)S.rcut * 1.00001f;
    if (!has || o.x * o.x + o.y * o.y + o.z * o.z > rcs * rcs) {
        for (int f = f_lo; f < f_hi; f++) emit0(f);
        return;
    }
    const df x = df_sub_sloppy(df{pp.x.x, pp.x.y}, df{aa.x.x, aa.x.y});
    const df y = df_sub_sloppy(df{pp.y.x, pp.y.y}, df{aa.y.x, aa.y.y});
    const df z = df_sub_sloppy(df{pp.z.x, pp.z.y}, df{aa.z.x, aa.z.y});
    const df d2 = df_add_sloppy(df_add_sloppy(df_mul(x, x), df_mul(y, y)), df_mul(z, z));
    const bool origin = d2.hi < 1e-24f;                 // d < 1e-12
    df d = zero, i0 = zero;
    if (!origin) {
        i0 = df_rsqrt(d2);
        d = df_mul(d2, i0);
    }
    float grid_hi = -1.f, grid_lo = 0.f, t = 0.f, tl = 0.f;
    int grid_nk = -1, kk = 0, sh = 0;
    df pw = i0;
    auto shells_of_l = [&](auto lc) {
        constexpr int L = decltype(lc)::value;
        constexpr int NM = 2 * L + 1;
        const int end = sh + S.nl[L];
        if (L > 0) pw = df_mul(pw, i0);
        for (; sh < end; sh++) {
            const DevShell R = sh_tab[S.shell0 + sh];
            const int f = R.fn0;
            if (f + NM <= f_lo || f >= f_hi) continue;
            if (!(d.hi < R.rcut_f) || (origin && L > 0)) {
                const int m0 = max(f, f_lo), m1 = min(f + NM, f_hi);
                for (int m = m0; m < m1; m++) emit0(m);
                continue;
            }
            df rk[NIMG];
            if (origin) {                               // the l = 0 limit C_0 c1/h
                const SplineEntry e = load_entry(coef + 2 * R.coef_off);
                const df u = df_mul(df{e.h.y, e.l.y}, df{R.inv_h_hi, R.inv_h_lo});
#pragma unroll
                for (int k = 0; k < NIMG; k++) rk[k] = (SCALED || k > 0) ? df_mul(u, scale[k]) : u;
            } else {
                if (R.inv_h_hi != grid_hi || R.inv_h_lo != grid_lo || R.nk != grid_nk) {
                    grid_hi = R.inv_h_hi;
                    grid_lo = R.inv_h_lo;
                    grid_nk = R.nk;
                    const df s2 = df_mul(d, df{R.inv_h_hi, R.inv_h_lo});
                    kk = (int)floorf(s2.hi);
                    kk = max(0, min(kk, R.nk - 2));
                    t = s2.hi - (float)kk;
                    tl = s2.lo;
                }
                const df u = spline_value(load_entry(coef + 2 * (R.coef_off + kk)), t, tl);
#pragma unroll
                for (int k = 0; k < NIMG; k++) rk[k] = df_mul(u, (SCALED || k > 0) ? df_mul(pw, scale[k]) : pw);
            }
            emit_shell_lane<L, NIMG>(rk, x.hi, y.hi, z.hi, f, f_lo, f_hi, emit);
        }
    };
    shells_of_l(std::integral_constant<int, 0>{});
    if (S.lmax >= 1) shells_of_l(std::integral_constant<int, 1>{});
    if (S.lmax >= 2) shells_of_l(std::integral_constant<int, 2>{});
    if (S.lmax >= 3) shells_of_l(std::integral_constant<int, 3>{});
}

// two points' coordinates as pairs of double-floats
struct Dd3x2 {
    df2 x, y, z;
};
__device__ __forceinline__ Dd3x2 pair_dd3(const Dd3 &a, const Dd3 &b)
{
    return Dd3x2{{pk_make(a.x.x, b.x.x), pk_make(a.x.y, b.x.y)},
                 {pk_make(a.y.x, b.y.x), pk_make(a.y.y, b.y.y)},
                 {pk_make(a.z.x, b.z.x), pk_make(a.z.y, b.z.y)}};
}

// The same for a warp together (one atom, two points a lane: p0, p1 their
// coordinates, has0, has1 whether there are such points).  Warps whose points
// are all beyond the species' cutoff call zero_all() and clear their part of
// the image with 16-byte stores.  Where the species' shells share one knot grid
// (and no point sits on the nucleus) the lanes run one path without
// divergence: a point beyond the cutoff multiplies by zero instead of
// branching, and the interval and its fraction are found once.  emit2(f, hi, nlo)
// receives the pair of values hi[k] - nlo[k] of image k: the low parts are kept
// negated from the radial factor on, which saves the packed negations and
// changes no rounding.  The operations of a value are those of the general
// path, in its order.
//
// What bounds it is instruction issue, then the L1's look-ups: two points a lane
// halve the FP32 instructions a point (f32x2) and fill four bytes a store where
// one filled two.  The 64-atom Si cluster's density images 1.84 -> 1.66 ms, 64
// molecules' (9.0 M points) images 15.7 -> 13.9 ms with the preparation below.
// Loading the next shell's coefficients ahead costs registers that a third CTA
// an SM is worth more of: 2.14 -> 2.06 ms of H images without it.
template <int NIMG, bool SCALED, class Emit2, class General, class Zero>
__device__ __forceinline__ void eval_atom_warp(const DevPlan &P, const DevSpecies &S, const DevShell *sh_tab,
                                               const Dd3 &aa, const Dd3x2 &pp, bool has0, bool has1, int f_lo,
                                               int f_hi, const df2 *scale, Emit2 &emit2, General &general,
                                               Zero &zero_all)
{
    // beyond the species' largest cutoff every value is zero (FP32 distance,
    // relative error ~1e-7, against the cutoff with a 1e-5 margin)
    const df2 ax{pk_dup(-aa.x.x), pk_dup(-aa.x.y)}, ay{pk_dup(-aa.y.x), pk_dup(-aa.y.y)}, az{pk_dup(-aa.z.x), pk_dup(-aa.z.y)};
    const pk ox = (pp.x.hi + ax.hi) + (pp.x.lo + ax.lo), oy = (pp.y.hi + ay.hi) + (pp.y.lo + ay.lo),
             oz = (pp.z.hi + az.hi) + (pp.z.lo + az.lo);
    const float2 o2 = pk_get(fma2(oz, oz, fma2(oy, oy, ox * ox)));
    const float rcs = (float)S.rcut * 1.00001f;
    const bool in0 = has0 && o2.x <= rcs * rcs, in1 = has1 && o2.y <= rcs * rcs;
    if (__all_sync(0xffffffffu, !in0 && !in1)) {
        zero_all();
        return;
    }
    // (the density's kernel gains from leaving here; H's, whose general path is a call,
    // from looking once: the 75-atom cluster's H 4.83 ms, 4.90 with the look here)
    if (NIMG == 1 && !SCALED && !S.shared_grid) {
        general();
        return;
    }
    // offset from the atom (the rounding of the low parts differs from point
    // to point), d^2 (terms of one sign), 1/d from a refined rsqrtf, d = d^2/d
    const df2 x = df2_add_sloppy(pp.x, ax), y = df2_add_sloppy(pp.y, ay), z = df2_add_sloppy(pp.z, az);
    const df2 d2 = df2_add_sloppy(df2_add_sloppy(df2_mul(x, x), df2_mul(y, y)), df2_mul(z, z));
    const float2 d2h = pk_get(d2.hi);
    if (!S.shared_grid || __any_sync(0xffffffffu, (in0 && d2h.x < 1e-24f) || (in1 && d2h.y < 1e-24f))) {
        general();
        return;
    }
    const df2 i0 = df2_rsqrt(d2);
    const df2 d = df2_mul(d2, i0);
    const float rcut = sh_tab[S.shell0].rcut_f;
    const float2 dh = pk_get(d.hi);
    const bool live0 = in0 && dh.x < rcut, live1 = in1 && dh.y < rcut;
    const df2 sd = df2_mul(d, {pk_dup(S.inv_h_hi), pk_dup(S.inv_h_lo)});
    const float2 sh2 = pk_get(sd.hi);
    const int k0 = live0 ? max(0, min((int)floorf(sh2.x), S.nk - 2)) : 0;
    const int k1 = live1 ? max(0, min((int)floorf(sh2.y), S.nk - 2)) : 0;
    const float2 tl2 = pk_get(sd.lo);
    // a point that is not live: t = 0 on interval 0, times ip = 0
    const pk t = pk_make(live0 ? sh2.x - (float)k0 : 0.f, live1 ? sh2.y - (float)k1 : 0.f);
    const pk nt = -t, ntl = pk_make(live0 ? -tl2.x : 0.f, live1 ? -tl2.y : 0.f), tt = t * t;
    // and the polynomials of offset 0: those of a far point overflow FP32 (f shells
    // from 7e12 Bohr on), and zero times infinity is not zero
    const float2 xh = pk_get(x.hi), yh = pk_get(y.hi), zh = pk_get(z.hi);
    const pk qx = pk_make(live0 ? xh.x : 0.f, live1 ? xh.y : 0.f), qy = pk_make(live0 ? yh.x : 0.f, live1 ? yh.y : 0.f),
             qz = pk_make(live0 ? zh.x : 0.f, live1 ? zh.y : 0.f);
    const float4 *tab = P.scoefn + S.scoef_off;
    const float4 *c0 = tab + 2 * ((long long)k0 * S.n_shell), *c1 = tab + 2 * ((long long)k1 * S.n_shell);
    int sh = 0;
    df2 pw = i0;                                        // 1/d^(l+1)
    auto shells_of_l = [&](auto lc) {
        constexpr int L = decltype(lc)::value;
        constexpr int NM = 2 * L + 1;
        constexpr int NG = L < 2 ? 1 : (L == 2 ? 2 : 4);
        constexpr int G0 = L == 2 ? 0 : 1;              // first kYlmRatio entry of groups 1..
        const int end = sh + S.nl[L];
        if (L > 0) pw = df2_mul(pw, i0);
        if (sh == end) return;
        df2 ip[NIMG], nip[NIMG];                        // times each image's scale; and negated
#pragma unroll
        for (int k = 0; k < NIMG; k++) {
            const df2 v = (SCALED || k > 0) ? df2_mul(pw, scale[k]) : pw;
            const float2 vh = pk_get(v.hi), vl = pk_get(v.lo);
            ip[k] = df2{pk_make(live0 ? vh.x : 0.f, live1 ? vh.y : 0.f), pk_make(live0 ? vl.x : 0.f, live1 ? vl.y : 0.f)};
            nip[k] = df2{-ip[k].hi, -ip[k].lo};
        }
        pk Q[NM];
        int gi[7];
        if constexpr (L > 0) ylm_poly_unit2<L>(qx, qy, qz, Q, gi);
        for (; sh < end; sh++) {
            const SplineEntry a = load_entry(c0 + 2 * sh), b = load_entry(c1 + 2 * sh);
            const int f = sh_tab[S.shell0 + sh].fn0;
            if (f + NM <= f_lo || f >= f_hi) continue;
            // u = c0 + t c1 + t^2 (c2 + t c3), c0 + t c1 in double-float (spline_value)
            const pk h1 = pk_make(a.h.y, b.h.y), lin = t * h1;
            const pk nlin_lo = fma2(nt, pk_make(a.l.y, b.l.y), fma2(ntl, h1, fma2(nt, h1, lin)));
            const pk quad = tt * fma2(t, pk_make(a.h.w, b.h.w), pk_make(a.h.z, b.h.z));
            const df2 u1 = df2_two_sum(pk_make(a.h.x, b.h.x), lin);
            const df2 u = df2_two_sum(u1.hi, u1.lo + ((pk_make(a.l.x, b.l.x) - nlin_lo) + quad));
            pk rh[NIMG][NG], nrh[NIMG][NG], nrl[NIMG][NG];   // radial factors: high, -high, -low
#pragma unroll
            for (int k = 0; k < NIMG; k++) {
                const pk p = u.hi * ip[k].hi;
                const pk nlo = fma2(u.hi, nip[k].lo, fma2(u.lo, nip[k].hi, fma2(u.hi, nip[k].hi, p)));
                rh[k][0] = p - nlo;
                nrl[k][0] = nlo + (rh[k][0] - p);
#pragma unroll
                for (int c = 1; c < NG; c++) {
                    const float2 K = kYlmRatio[G0 + c - 1];
                    const pk kh = pk_dup(K.x), kl = pk_dup(K.y), pc = rh[k][0] * kh;
                    // -(rh kl + (rl kh + (rh kh - pc)))
                    const pk nl = fma2(-rh[k][0], kl, fma2(nrl[k][0], kh, fma2(-rh[k][0], kh, pc)));
                    rh[k][c] = pc - nl;
                    nrl[k][c] = nl + (rh[k][c] - pc);
                }
#pragma unroll
                for (int c = 0; c < NG; c++) nrh[k][c] = -rh[k][c];
            }
            if constexpr (L == 0) {                     // the angular factor is 1
                pk hi[NIMG], nlo[NIMG];
#pragma unroll
                for (int k = 0; k < NIMG; k++) {
                    hi[k] = rh[k][0];
                    nlo[k] = nrl[k][0];
                }
                emit2(f, hi, nlo);
            } else {
                const bool whole = f >= f_lo && f + NM <= f_hi;
#pragma unroll
                for (int m = 0; m < NM; m++) {
                    if (!whole && (f + m < f_lo || f + m >= f_hi)) continue;
                    pk hi[NIMG], nlo[NIMG];
#pragma unroll
                    for (int k = 0; k < NIMG; k++) {    // df_mul_f_raw
                        hi[k] = rh[k][gi[m]] * Q[m];
                        nlo[k] = fma2(nrl[k][gi[m]], Q[m], fma2(nrh[k][gi[m]], Q[m], hi[k]));
                    }
                    emit2(f + m, hi, nlo);
                }
            }
        }
    };
    shells_of_l(std::integral_constant<int, 0>{});
    if (S.lmax >= 1) shells_of_l(std::integral_constant<int, 1>{});
    if (S.lmax >= 2) shells_of_l(std::integral_constant<int, 2>{});
    if (S.lmax >= 3) shells_of_l(std::integral_constant<int, 3>{});
}

// the species' shells for one CTA: shared memory when they fit
constexpr int kMaxShellsSmem = 64;
__device__ __forceinline__ const DevShell *stage_shells(const DevPlan &P, DevShell *smem)
{
    if (P.n_shells > kMaxShellsSmem) return P.shells;
    for (int i = threadIdx.x; i < P.n_shells; i += blockDim.x) smem[i] = P.shells[i];
    return smem;                                    // valid after the caller's next __syncthreads
}

// swizzled place of point column group g16 = g << 4 in row r of a chunk
__device__ __forceinline__ uint32_t row_offset(uint32_t r, uint32_t g16) { return r * 128u + (((r << 4) ^ g16) & 0x70u); }

// One atom's functions [f_lo, f_hi) at the points of chunk c by the general path,
// a point a lane: 64 consecutive bytes of a row a store.  (Every second point a
// lane wrote half sectors: 64 atoms, shells on knots of their own, potential of both
// signs, H 5.15 -> 4.58 ms with the rest below.)  A function of its own, for its
// registers would cost the path on shared knots.
template <int NIMG, int NSPLIT>
__device__ __noinline__ void h_image_general(const float4 *coef, const DevSpecies *species, const DevShell *sh_tab,
                                             const float *atom, const float *pts, int np, int c, int rb, int f_lo,
                                             int f_hi, uint8_t *c0, uint8_t *c1, const float2 *wvs,
                                             const float4 (*fsc)[128])
{
    const DevSpecies S = *species;
    const Dd3 aa = load_dd3(atom);
#pragma unroll 1
    for (int kg = threadIdx.x & 31; kg < 64; kg += 32) {
        const int pg = c * 64 + kg;
        const bool has = pg < np;
        const Dd3 q = load_dd3(pts + 6 * (has ? pg : 0));
        const float2 s2 = has ? wvs[pg] : make_float2(0.f, 0.f);
        df sc[NIMG];
#pragma unroll
        for (int k = 0; k < NIMG; k++) sc[k] = df{s2.x, s2.y};
        const uint32_t g16 = (uint32_t)(kg >> 3) << 4, hb = (uint32_t)(kg & 7) * 2u;
        auto emit = [&](int f, const df *val) {
            const int r = rb + f;
            const uint32_t off = row_offset((uint32_t)r, g16) + hb;
#pragma unroll
            for (int k = 0; k < NIMG; k++) {
                const float4 su = fsc[NIMG == 1 ? 1 : k][r];
                store_value<NSPLIT>((k == 0 ? c0 : c1) + off, val[k], su.x, su.z);
            }
        };
        auto emit0 = [&](int f) {
            const uint32_t off = row_offset((uint32_t)(rb + f), g16) + hb;
#pragma unroll
            for (int k = 0; k < NIMG; k++) store_zero<NSPLIT>((k == 0 ? c0 : c1) + off);
        };
        eval_atom_general<NIMG, NIMG == 1>(coef, S, sh_tab, aa, q, has, f_lo, f_hi, sc, emit, emit0);
    }
}

// H images of one 128-row block: warp tasks (atom of the block, 64-point
// chunk).  NIMG 1: psi = phi sqrt|w v| on the second grid set; NIMG 2: phi
// (first set) and w v phi (second set) into two images.
template <int NIMG, int NSPLIT>
__device__ __forceinline__ void h_image_lanes(const DevPlan &P, const DevBatch &B, const TcBatch &T,
                                              const DevAct *act, const DevShell *sh_tab, int I, int e0, int ne,
                                              uint8_t *img0, uint8_t *img1, const float2 *wvs,
                                              const float4 (*fsc)[128])
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    const int r0 = I * 128;
    const uint32_t g16 = (uint32_t)(lane >> 2) << 4, pb = (uint32_t)(lane & 3) * 4u;
    for (int task = warp; task < ne * T.nc; task += nwarp) {
        const int eq = task / T.nc, c = task - eq * T.nc;
        const DevAct A = act[e0 + eq];
        const DevSpecies S = P.species[P.atom_species[A.atom]];
        const int f_lo = max(0, r0 - A.fn_loc), f_hi = min(S.n_fn, r0 + 128 - A.fn_loc);
        const int p = c * 64 + 2 * lane;
        const bool has0 = p < B.np, has1 = p + 1 < B.np;
        const Dd3 q0 = load_dd3(P.pts_dd + 6 * (B.pt0 + (has0 ? p : 0)));
        const Dd3 q1 = load_dd3(P.pts_dd + 6 * (B.pt0 + (has1 ? p + 1 : 0)));
        const Dd3 aa = load_dd3(P.atom_dd + 6 * A.atom);
        const float2 s0 = has0 ? wvs[p] : make_float2(0.f, 0.f), s1 = has1 ? wvs[p + 1] : make_float2(0.f, 0.f);
        df2 scale[NIMG];
#pragma unroll
        for (int k = 0; k < NIMG; k++) scale[k] = df2{pk_make(s0.x, s1.x), pk_make(s0.y, s1.y)};
        const int rb = A.fn_loc - r0;
        uint8_t *const c0 = img0 + (long long)(I * T.nc_alloc + c) * kChunkStride;
        uint8_t *const c1 = img1 + (long long)(I * T.nc_alloc + c) * kChunkStride;
        auto emit2 = [&](int f, const pk *hi, const pk *nlo) {
            const int r = rb + f;
            const uint32_t off = row_offset((uint32_t)r, g16) + pb;
#pragma unroll
            for (int k = 0; k < NIMG; k++) {
                const float4 su = fsc[NIMG == 1 ? 1 : k][r];
                store_pair<NSPLIT>((k == 0 ? c0 : c1) + off, hi[k], nlo[k], pk_make(su.x, su.y), pk_make(su.z, su.w));
            }
        };
        auto general = [&]() {
            h_image_general<NIMG, NSPLIT>(P.coef_ddn, P.species + P.atom_species[A.atom], sh_tab, P.atom_dd + 6 * A.atom,
                                          P.pts_dd + 6 * B.pt0, B.np, c, rb, f_lo, f_hi, c0, c1, wvs, fsc);
        };
        // the chunk's columns of rows rb + [f_lo, f_hi): eight 16-byte units a row and plane
        auto zero_all = [&]() {
            for (int u = lane; u < (f_hi - f_lo) * 8; u += 32) {
                const uint32_t off = row_offset((uint32_t)(rb + f_lo + (u >> 3)), (uint32_t)(u & 7) << 4);
#pragma unroll
                for (int k = 0; k < NIMG; k++)
#pragma unroll
                    for (int pl = 0; pl < NSPLIT; pl++)
                        *reinterpret_cast<uint4 *>((k == 0 ? c0 : c1) + off + pl * kChunkBytes) =
                            make_uint4(0u, 0u, 0u, 0u);
            }
        };
        eval_atom_warp<NIMG, NIMG == 1>(P, S, sh_tab, aa, pair_dd3(q0, q1), has0, has1, f_lo, f_hi, scale, emit2,
                                        general, zero_all);
    }
}

// ------------------------------------- preparation of the H images (K0)
// CTA per super-batch: the sign of w v, the images' scale of every point, the
// digit grid (scale, unit) of every function in both images, and the
// descriptors of the row blocks.  A kernel of its own: these passes want many
// small warps in flight, the evaluation few with many registers, and a
// super-batch's atoms and points are looked at once instead of once a row
// block.  H images with it and two points a lane: 64-atom Si cluster, 1.11 M
// points, 2.73 -> 1.85 ms (0.25 of it here), 75-atom cluster with f shells,
// two images a batch, 3.80 -> 2.9 ms (0.49 here).
constexpr int kPhiThreads = 256;

// Knot interval of distance d from below (against FP32 rounding of d) for the
// suffix bounds of |u(r)/r|, or -1 beyond the cutoff
__device__ __forceinline__ int knot_below(float d, float rcut_f, float inv_h, int nk)
{
    if (!(d < rcut_f * 1.00001f)) return -1;
    return min(max((int)(d * 0.999999f * inv_h), 0), nk - 2);
}

__device__ __forceinline__ float warp_sum(float s)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

__device__ __forceinline__ float warp_max(float m)                   // m >= 0
{
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));
}

// digit grid of function f (row of its block) in image `set`
__device__ __forceinline__ void put_grid(HGrid *grids, int set, int f, float mx, float sum, int depth)
{
    float sc, un;
    fixed_scale_adaptive(mx, sum, depth, sc, un);
    grids[f >> 7].s[set][f & 127] = make_float2(sc, un);
}

// lane m: the grid of function m of a shell (first function f0 in the batch) from
// the bound of its radial factor and of the factor's sum, times max |Y_lm|
__device__ __forceinline__ void put_shell_grid(const DevPlan &P, HGrid *grids, int set, int l, int f0, float m, float s,
                                               int depth, int lane)
{
    if (lane > 2 * l) return;
    const float yl = __ldg(P.rbound + l * l + lane);
    put_grid(grids, set, f0 + lane, m > 0.f ? fminf(m * yl, 1.0e30f) : 0.f, fminf(s * 1.0001f * yl, 1.0e30f), depth);
}

// Sum over the warp of twelve values at once: lane L receives the sum of value
// L / 2 (zero beyond).  Each step adds across one lane bit and hands half of the
// values to the other lane: 16 shuffles where twelve sums take 60, every sum in
// the order of warp_sum.
__device__ __forceinline__ float warp_sums12(const float *v, int lane)
{
    float a[8], b[4], c[2];
    const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4, h1 = lane & 2;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const float lo = v[j], hi = j < 4 ? v[8 + j] : 0.f;
        a[j] = (h4 ? hi : lo) + __shfl_xor_sync(0xffffffffu, h4 ? lo : hi, 16);
    }
#pragma unroll
    for (int j = 0; j < 4; j++)
        b[j] = (h3 ? a[4 + j] : a[j]) + __shfl_xor_sync(0xffffffffu, h3 ? a[j] : a[4 + j], 8);
#pragma unroll
    for (int j = 0; j < 2; j++)
        c[j] = (h2 ? b[2 + j] : b[j]) + __shfl_xor_sync(0xffffffffu, h2 ? b[j] : b[2 + j], 4);
    float d = (h1 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, h1 ? c[0] : c[1], 2);
    return d + __shfl_xor_sync(0xffffffffu, d, 1);
}

// The maxima of twelve values (>= 0) in the same places
__device__ __forceinline__ float warp_maxs12(const float *v, int lane)
{
    float r = 0.f;
#pragma unroll
    for (int j = 0; j < 12; j++) {
        const float m = warp_max(v[j]);
        if (lane >> 1 == j) r = m;
    }
    return r;
}

// Grids of one atom's functions by a warp from the interleaved table bounds: per
// point one look-up of the suffix bounds of |u(r)/r| serves four shells, times
// sqrt|w v| (psi) or |w v| (w v phi) of the point; the maximum over the points
// times max |Y_lm| bounds each row, and the same products summed over the
// points bound the row sums, so that rows whose sum allows it keep an 8-bit
// digit.  MIXED: also |phi| itself (set 0), which only batches with both signs
// use.  The grids themselves are found a function a lane: a shell at a time
// (2l+1 lanes of 32, after its own reductions) that part took as long as the
// points: the preparation 0.46 -> 0.25 ms for the 64-atom Si cluster, 0.67 ->
// 0.49 for the 75-atom cluster, 1.34 -> 1.17 for 64 molecules.
template <bool MIXED>
__device__ __forceinline__ void atom_grids(const DevPlan &P, const DevBatch &B, const DevAct &A, const DevSpecies &S,
                                           const DevShell *sh_tab, const Dd3 *pts, const float *wvf, HGrid *grids,
                                           int depth)
{
    const int lane = threadIdx.x & 31;
    const Dd3 aa = load_dd3(P.atom_dd + 6 * A.atom);
    const float rcut = sh_tab[S.shell0].rcut_f;
    for (int q0 = 0; 4 * q0 < S.n_shell; q0 += 3) {                // twelve shells a pass
        const int nq = min(3, (S.n_shell + 3) / 4 - q0);
        const float *bt = P.sbound + S.sbound_off + 4 * q0;
        float m0[12], m1[12], s0[12], s1[12];
#pragma unroll
        for (int j = 0; j < 12; j++) m0[j] = m1[j] = s0[j] = s1[j] = 0.f;
        for (int p = lane; p < B.np; p += 32) {
            const float3 o = offset_f32(pts[p], aa);
            const int ki = knot_below(sqrtf(o.x * o.x + o.y * o.y + o.z * o.z), rcut, S.inv_h_hi, S.nk);
            if (ki < 0) continue;
            const float4 *row = reinterpret_cast<const float4 *>(bt + (long long)ki * S.sbound_stride);
            const float w = wvf[p];
#pragma unroll
            for (int q = 0; q < 3; q++) {
                if (q >= nq) break;
                const float4 t4 = __ldg(row + q);
                const float t[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const float tw = t[j] * w;
                    m1[4 * q + j] = fmaxf(m1[4 * q + j], tw);
                    s1[4 * q + j] += tw;
                    if (MIXED) {
                        m0[4 * q + j] = fmaxf(m0[4 * q + j], t[j]);
                        s0[4 * q + j] += t[j];
                    }
                }
            }
        }
        __syncwarp();
        // lane 2 j: shell j of the pass
        const float a1 = warp_maxs12(m1, lane), b1 = warp_sums12(s1, lane);
        float a0 = 0.f, b0 = 0.f;
        if (MIXED) {
            a0 = warp_maxs12(m0, lane);
            b0 = warp_sums12(s0, lane);
        }
        // function i in the order of the shell table (by l): its shell and m
        for (int i0 = 0; i0 < S.n_fn; i0 += 32) {
            int i = i0 + lane, sh = 0, l = 0;
            for (; l < kMaxL; l++) {
                const int nf = S.nl[l] * (2 * l + 1);
                if (i < nf) break;
                i -= nf;
                sh += S.nl[l];
            }
            const int q = i / (2 * l + 1), m = i - q * (2 * l + 1), j = sh + q - 4 * q0;
            const bool mine = i0 + lane < S.n_fn && j >= 0 && j < 12;
            const int src = 2 * max(0, min(j, 11));
            const float mx1 = __shfl_sync(0xffffffffu, a1, src), sm1 = __shfl_sync(0xffffffffu, b1, src);
            float mx0 = 0.f, sm0 = 0.f;
            if (MIXED) {
                mx0 = __shfl_sync(0xffffffffu, a0, src);
                sm0 = __shfl_sync(0xffffffffu, b0, src);
            }
            if (mine) {
                const int f = A.fn_loc + sh_tab[S.shell0 + sh + q].fn0 + m;
                const float yl = __ldg(P.rbound + l * l + m);
                put_grid(grids, 1, f, mx1 > 0.f ? fminf(mx1 * yl, 1.0e30f) : 0.f, fminf(sm1 * 1.0001f * yl, 1.0e30f), depth);
                if (MIXED)
                    put_grid(grids, 0, f, mx0 > 0.f ? fminf(mx0 * yl, 1.0e30f) : 0.f, fminf(sm0 * 1.0001f * yl, 1.0e30f),
                             depth);
            }
        }
    }
}

// The same for any species, each shell on its own table, four shells a look at the
// points
__device__ __forceinline__ void atom_grids_general(const DevPlan &P, const DevBatch &B, const DevAct &A,
                                                   const DevSpecies &S, const DevShell *sh_tab, const Dd3 *pts,
                                                   const float *wvf, HGrid *grids, int depth)
{
    const int lane = threadIdx.x & 31;
    const Dd3 aa = load_dd3(P.atom_dd + 6 * A.atom);
    for (int sh0 = 0; sh0 < S.n_shell; sh0 += 4) {
        const DevShell *sh = sh_tab + S.shell0 + sh0;
        const int ns = min(4, S.n_shell - sh0);
        float m0[4], m1[4], s0[4], s1[4];
#pragma unroll
        for (int j = 0; j < 4; j++) m0[j] = m1[j] = s0[j] = s1[j] = 0.f;
        for (int p = lane; p < B.np; p += 32) {
            const float3 o = offset_f32(pts[p], aa);
            const float d = sqrtf(o.x * o.x + o.y * o.y + o.z * o.z), w = wvf[p];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                if (j >= ns) break;
                const int ki = knot_below(d, sh[j].rcut_f, sh[j].inv_h_hi, sh[j].nk);
                if (ki < 0) continue;
                const float t = __ldg(P.rbound + sh[j].bound_off + ki), tw = t * w;
                m0[j] = fmaxf(m0[j], t);
                m1[j] = fmaxf(m1[j], tw);
                s0[j] += t;
                s1[j] += tw;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            if (j >= ns) break;
            const float a0 = warp_max(m0[j]), a1 = warp_max(m1[j]), b0 = warp_sum(s0[j]), b1 = warp_sum(s1[j]);
            put_shell_grid(P, grids, 0, sh[j].l, A.fn_loc + sh[j].fn0, a0, b0, depth, lane);
            put_shell_grid(P, grids, 1, sh[j].l, A.fn_loc + sh[j].fn0, a1, b1, depth, lane);
        }
    }
}

// The exact maxima and sums of |phi| and |w v phi| (or |psi|) over the points,
// in FP32 (bound_grids 0 and 1)
__device__ __forceinline__ void atom_grids_exact(const DevPlan &P, const DevBatch &B, const DevAct &A, const DevSpecies &S,
                                                 const Dd3 *pts, const float *wvf, HGrid *grids, int depth)
{
    const int lane = threadIdx.x & 31;
    const float *aa = P.atom_dd + 6 * A.atom;
    const float ax = aa[0] + aa[1], ay = aa[2] + aa[3], az = aa[4] + aa[5];
    int f = A.fn_loc;
    for (int sh = 0; sh < S.n_shell; sh++) {
        const DevRadial R = P.radials[P.shell_rad[S.shell0 + sh]];
        const int nm = 2 * R.l + 1;
        int tstep;
        const float4 *tab = spline_tab(P, S, R, sh, tstep);
        float mx[7], sm[7], mxw[7], smw[7];
#pragma unroll
        for (int m = 0; m < 7; m++) mx[m] = sm[m] = mxw[m] = smw[m] = 0.f;
        for (int p = lane; p < B.np; p += 32) {
            const Dd3 pp = pts[p];
            const float x = (pp.x.x + pp.x.y) - ax, y = (pp.y.x + pp.y.y) - ay, z = (pp.z.x + pp.z.y) - az;
            const float d = sqrtf(x * x + y * y + z * z);
            const float rad = radial_over_d_f32(R, tab, tstep, d, __frcp_rn(d));
            if (rad == 0.f) continue;
            float Q[7];
            int ci[7];
            ylm_poly_f32(R.l, x, y, z, Q, ci);
            const float wvp = wvf[p];
#pragma unroll
            for (int m = 0; m < 7; m++) {
                if (m >= nm) break;
                const float a = fminf(fabsf(rad * kYlmC[ci[m]].x * Q[m]), 1.0e30f);
                const float aw = fminf(a * wvp, 1.0e30f);
                mx[m] = fmaxf(mx[m], a);
                sm[m] += a;
                mxw[m] = fmaxf(mxw[m], aw);
                smw[m] += aw;
            }
        }
#pragma unroll
        for (int m = 0; m < 7; m++) {
            if (m >= nm) break;
            const float a = warp_max(mx[m]), aw = warp_max(mxw[m]), s1 = warp_sum(sm[m]), s2 = warp_sum(smw[m]);
            if (lane == 0) {
                put_grid(grids, 0, f + m, a, s1, depth);
                put_grid(grids, 1, f + m, aw, s2, depth);
            }
        }
        f += nm;
    }
}

// The descriptor of one row block for the H scatter (threads 0 .. 127, a row
// each; e0 the first of the block's ne active atoms)
__device__ __forceinline__ void write_hblock(const DevPlan &P, const DevBatch &B, const DevAct *act, int r0, int r, int e0,
                                             int ne, HBlock *out)
{
    const int f = r0 + r;
    long long base = 0;
    int li = 0, slot = 0;
    if (f < B.nfn) {
        slot = find_act(act + e0, ne, f);
        const DevAct A = act[e0 + slot];
        li = f - A.fn_loc;
        base = P.rowptr[P.atom_fn0[A.atom] + li] - li;
    }
    out->base[r] = base;
    out->li[r] = (unsigned short)li;
    out->slot[r] = (unsigned char)slot;
    if (r < ne) out->loc[r] = P.atom_loc[act[e0 + r].atom];
    if (r == 0) {
        out->pair_off = P.sys_pair_off[B.sys];
        out->nat = P.sys_nat[B.sys];
        out->nslot = ne;
        out->n = min(128, B.nfn - r0);
    }
}

__global__ void __launch_bounds__(kPhiThreads, 4) k_h_prep(DevPlan P, const TcBatch *tb, int b0, uint8_t *ws, const double *v,
                                                        int fixed, int bound, int *bsign, unsigned int *counter)
{
    __shared__ Dd3 pts[kMaxBatchPoints];
    __shared__ float wvf[kMaxBatchPoints];           // |w v| or its root per point (FP32)
    __shared__ DevShell shs[kMaxShellsSmem];
    if (blockIdx.x == 0 && threadIdx.x == 0) *counter = 0u;       // of the contraction that follows
    const int b = b0 + blockIdx.x;
    const DevBatch B = P.batches[b];
    if (B.np <= 0 || B.nfn <= 0) return;
    const TcBatch T = tb[b];
    const DevAct *act = P.act + B.act0;
    const DevShell *sh_tab = stage_shells(P, shs);
    // sign of w v over the batch: one sign s (or zero) everywhere lets H use a
    // single image psi = phi sqrt|w v| for both operands, H = s psi^T psi;
    // mixed signs keep the phi and w v phi images
    bool pos = false, neg = false, bad = false;
    for (int p = threadIdx.x; p < B.np; p += blockDim.x) {
        const double vv = v[B.pt0 + p], wv = P.pw[B.pt0 + p] * vv;
        pos |= wv > 0.0;
        neg |= wv < 0.0;
        bad |= !isfinite(vv);
        pts[p] = load_dd3(P.pts_dd + 6 * (B.pt0 + p));
    }
    if (bad) atomicOr(P.status, kStatusNonFinite);
    pos = __syncthreads_or(pos) != 0;
    neg = __syncthreads_or(neg) != 0;
    const int sgn = (pos && neg) ? 0 : (neg ? -1 : 1);
    if (threadIdx.x == 0) bsign[b] = sgn;
    // the per-point scale of the images, sqrt|w v| (psi) or w v (mixed signs),
    // and its size for the grids
    HGrid *grids = reinterpret_cast<HGrid *>(ws + T.hgrid);
    float2 *wvs = reinterpret_cast<float2 *>(ws + T.hscale);
    const float up = bound ? 1.f + 1.f / 1048576.f : 1.f;
    for (int p = threadIdx.x; p < B.np; p += blockDim.x) {
        const double s = P.pw[B.pt0 + p] * v[B.pt0 + p];
        df sd = df_from_double(sgn != 0 ? fabs(s) : s);
        if (sgn != 0) sd = df_sqrt(sd);
        wvs[p] = make_float2(sd.hi, sd.lo);
        const float a = fabsf((float)s) * up;
        wvf[p] = fminf(sgn != 0 ? sqrtf(a) * up : a, 1.0e30f);
    }
    for (int q = threadIdx.x; q < T.nrb * 128; q += blockDim.x) {
        const int r0 = q & ~127, rend = min(r0 + 128, B.nfn);
        const int e0 = find_act(act, B.n_act, r0), e1 = find_act(act, B.n_act, rend - 1);
        write_hblock(P, B, act, r0, q & 127, e0, e1 - e0 + 1, reinterpret_cast<HBlock *>(ws + T.hblock) + (q >> 7));
    }
    if (!fixed) return;
    __syncthreads();
    const int warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5, depth = T.nc * 64;
    for (int e = warp; e < B.n_act; e += nwarp) {
        const DevAct A = act[e];
        const DevSpecies S = P.species[P.atom_species[A.atom]];
        if (!bound) atom_grids_exact(P, B, A, S, pts, wvf, grids, depth);
        else if (S.sbound_stride == 0) atom_grids_general(P, B, A, S, sh_tab, pts, wvf, grids, depth);
        else if (sgn != 0) atom_grids<false>(P, B, A, S, sh_tab, pts, wvf, grids, depth);
        else atom_grids<true>(P, B, A, S, sh_tab, pts, wvf, grids, depth);
    }
}

// -------------------------------------------- basis -> operand images (K1)
// CTA per (batch, 128-row block): every function of the block is evaluated, two
// points a lane, and the split planes of psi = phi sqrt|w v| (batches where w v
// has one sign) or of phi and w v phi (mixed signs) are written on the grids of
// the preparation.
//
// The radial factor N_lm u(d)/d^(l+1) -- shared by all angular points of a
// radial shell, so its rounding would be systematic -- is evaluated in
// double-float from a double-float spline table and double-float
// coordinates; only the angular polynomial Q_lm(x, y, z) is FP32 (its
// rounding varies from point to point).
//
// Three CTAs an SM (80 registers, of which 96 bytes a thread spill): two take 2.28 ms
// where three take 2.06 and four (64 registers, more spilled) 2.08.
__global__ void __launch_bounds__(kPhiThreads, 3) k_tc_phi(DevPlan P, const TcBatch *tb, const WorkItem *items,
                                                uint8_t *ws, int fixed, const int *bsign)
{
    __shared__ float2 wvs[kMaxBatchPoints];         // per-point image scale (double-float)
    __shared__ DevShell shs[kMaxShellsSmem];
    __shared__ float4 fsc[2][128];                   // per row: scale twice, unit twice
    const WorkItem it = items[blockIdx.x];
    const DevBatch B = P.batches[it.batch];
    const TcBatch T = tb[it.batch];
    const int I = it.ti;
    const int r0 = I * 128;
    const DevAct *act = P.act + B.act0;
    const int rend = min(r0 + 128, B.nfn);
    const int e0 = find_act(act, B.n_act, r0);
    const int e1 = find_act(act, B.n_act, rend - 1);
    const int ne = e1 - e0 + 1;
    uint8_t *phi_img = ws + T.img_phi;
    uint8_t *a_img = ws + T.img_aux;
    const DevShell *sh_tab = stage_shells(P, shs);
    const int sgn = bsign[it.batch];
    for (int p = threadIdx.x; p < B.np; p += blockDim.x) wvs[p] = reinterpret_cast<const float2 *>(ws + T.hscale)[p];
    if (fixed) {
        const HGrid *g = reinterpret_cast<const HGrid *>(ws + T.hgrid) + I;
        for (int q = threadIdx.x; q < 256; q += blockDim.x) {
            const float2 su = g->s[q >> 7][q & 127];
            fsc[q >> 7][q & 127] = make_float4(su.x, su.x, su.y, su.y);
        }
    }
    __syncthreads();
    uint8_t *img1 = sgn == 0 ? a_img : phi_img;
    if (sgn != 0) {
        if (fixed) h_image_lanes<1, 3>(P, B, T, act, sh_tab, I, e0, ne, phi_img, img1, wvs, fsc);
        else h_image_lanes<1, 1>(P, B, T, act, sh_tab, I, e0, ne, phi_img, img1, wvs, fsc);
    } else {
        if (fixed) h_image_lanes<2, 3>(P, B, T, act, sh_tab, I, e0, ne, phi_img, img1, wvs, fsc);
        else h_image_lanes<2, 1>(P, B, T, act, sh_tab, I, e0, ne, phi_img, img1, wvs, fsc);
    }
    // rows past n_b in the last block stay as they are: a row or column of a
    // product depends on its own operand row alone, and the scatter leaves
    // those out (the padding of the points is zero)
}

// The density's image of one 64-point chunk: a warp an active atom, two
// neighbouring points a lane (the same for all of the warp's atoms), every
// function of the atom, split on the points' grids.
template <int NSPLIT>
__device__ __forceinline__ void density_image_lanes(const DevPlan &P, const DevBatch &B, const TcBatch &T,
                                                    const DevAct *act, const DevShell *sh_tab, int c, uint8_t *phi_img,
                                                    const float2 *csc)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    const int k = 2 * lane, p = c * 64 + k;
    const bool has0 = p < B.np, has1 = p + 1 < B.np;
    const Dd3 q0 = load_dd3(P.pts_dd + 6 * (B.pt0 + (has0 ? p : 0)));
    const Dd3 q1 = load_dd3(P.pts_dd + 6 * (B.pt0 + (has1 ? p + 1 : 0)));
    const Dd3x2 pp = pair_dd3(q0, q1);
    const float2 s0 = NSPLIT == 3 ? csc[k] : make_float2(0.f, 0.f), s1 = NSPLIT == 3 ? csc[k + 1] : make_float2(0.f, 0.f);
    const pk sc = pk_make(s0.x, s1.x), un = pk_make(s0.y, s1.y);
    uint8_t *const img = phi_img + (long long)c * kChunkStride;
    const uint32_t g16 = (uint32_t)(lane >> 2) << 4, pb = (uint32_t)(lane & 3) * 4u;
    const uint32_t blk = (uint32_t)T.nc_alloc * kChunkStride - 128u * 128u;   // a row block, less its rows' offsets
    for (int e = warp; e < B.n_act; e += nwarp) {
        const DevAct A = act[e];
        const DevSpecies S = P.species[P.atom_species[A.atom]];
        const Dd3 aa = load_dd3(P.atom_dd + 6 * A.atom);
        auto place = [&](int f, uint32_t g) {
            const uint32_t rg = (uint32_t)(A.fn_loc + f);
            return (rg >> 7) * blk + row_offset(rg, g);
        };
        auto emit2 = [&](int f, const pk *hi, const pk *nlo) {
            store_pair<NSPLIT>(img + place(f, g16) + pb, hi[0], nlo[0], sc, un);
        };
        auto general = [&]() {                       // a point a lane, 64 consecutive bytes of a row a store
#pragma unroll
            for (int kg = lane; kg < 64; kg += 32) {
                const int pg = c * 64 + kg;
                const bool has = pg < B.np;
                const Dd3 q = load_dd3(P.pts_dd + 6 * (B.pt0 + (has ? pg : 0)));
                const float2 su = NSPLIT == 3 ? csc[kg] : make_float2(0.f, 0.f);
                const uint32_t gg16 = (uint32_t)(kg >> 3) << 4, hb = (uint32_t)(kg & 7) * 2u;
                auto emit = [&](int f, const df *val) { store_value<NSPLIT>(img + place(f, gg16) + hb, val[0], su.x, su.y); };
                auto emit0 = [&](int f) { store_zero<NSPLIT>(img + place(f, gg16) + hb); };
                eval_atom_general<1, false>(P.coef_ddn, S, sh_tab, aa, q, has, 0, S.n_fn, nullptr, emit, emit0);
            }
        };
        // the chunk's columns of the atom's rows: eight 16-byte units a row and plane
        auto zero_all = [&]() {
            for (int u = lane; u < S.n_fn * 8; u += 32) {
                const uint32_t off = place(u >> 3, (uint32_t)(u & 7) << 4);
#pragma unroll
                for (int pl = 0; pl < NSPLIT; pl++)
                    *reinterpret_cast<uint4 *>(img + off + pl * kChunkBytes) = make_uint4(0u, 0u, 0u, 0u);
            }
        };
        eval_atom_warp<1, false>(P, S, sh_tab, aa, pp, has0, has1, 0, S.n_fn, (const df2 *)nullptr, emit2, general,
                                 zero_all);
    }
}

// What the column bounds need of an active atom
struct ColAtom {
    Dd3 pos;
    float rcut, inv_h;                               // cutoff with its margin; of the species' knot grid
    int nk, species;
    long long cbound;                                // first of its (maximum, sum) bounds, -1: none
};
constexpr int kColAtoms = 128;                       // staged at a time

// CTA per (batch, 64-point chunk c): the phi image for the density.  The
// density contracts over functions, so the fixed-point grid of the leading
// term is per point (column): first bounds of the largest |phi_i(p)| and of
// their sum over all of the batch's functions (FP32), then the values.
//
// The bounds of a column take one 8-byte look-up an atom (the species' maximum
// and sum over its shells and m at the knot), the atoms' tables are staged in
// shared memory.  With look-ups of four shells and a chain of table loads an
// atom the bounds took a quarter of the kernel: 64 molecules (9.0 M points),
// images 13.9 -> 12.7 ms (H's included); the 64-atom Si cluster 1.66 -> 1.43 ms.
__global__ void __launch_bounds__(kPhiThreads, 3) k_tc_phi_cols(DevPlan P, const TcBatch *tb, const WorkItem *items,
                                                     uint8_t *ws, int n_split, int bound, unsigned int *counter)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) *counter = 0u;       // of the contraction that follows
    __shared__ float colmax[kPhiThreads / 64][64], colsum[kPhiThreads / 64][64];
    __shared__ float2 csc[64];                       // per point: scale, unit
    __shared__ ColAtom ca[kColAtoms];
    __shared__ DevShell shs[kMaxShellsSmem];
    const WorkItem it = items[blockIdx.x];
    const DevBatch B = P.batches[it.batch];
    const TcBatch T = tb[it.batch];
    const int c = it.ti;
    const DevAct *act = P.act + B.act0;
    uint8_t *phi_img = ws + T.img_phi;
    const bool fixed = n_split == 3;
    const DevShell *sh_tab = stage_shells(P, shs);
    if (fixed) {
        // one column of the chunk and every fourth active atom per thread: the
        // column's coordinates load once and its maximum and sum stay in
        // registers
        const int k = threadIdx.x & 63, part = threadIdx.x >> 6, p = c * 64 + k;
        const Dd3 pp = load_dd3(P.pts_dd + 6 * (B.pt0 + min(p, B.np - 1)));
        float mxc = 0.f, smc = 0.f;
        for (int e0 = 0; e0 < B.n_act; e0 += kColAtoms) {
            const int ne = min(kColAtoms, B.n_act - e0);
            __syncthreads();
            if (threadIdx.x < ne) {
                const int atom = act[e0 + threadIdx.x].atom, sp = P.atom_species[atom];
                const DevSpecies &S = P.species[sp];
                ca[threadIdx.x] = ColAtom{load_dd3(P.atom_dd + 6 * atom), (float)S.rcut * 1.00001f, S.inv_h_hi, S.nk, sp,
                                          bound ? S.cbound_off : -1ll};
            }
            __syncthreads();
            for (int e = part; e < ne; e += kPhiThreads / 64) {
                const ColAtom &A = ca[e];
                const float3 o = offset_f32(pp, A.pos);
                const float d = sqrtf(o.x * o.x + o.y * o.y + o.z * o.z);
                if (d > A.rcut) continue;                          // every shell is zero here
                float mx = 0.f, sm = 0.f;
                if (A.cbound >= 0) {
                    if (!(d < A.rcut)) continue;                   // knot_below, one knot grid
                    const int ki = min(max((int)(d * 0.999999f * A.inv_h), 0), A.nk - 2);
                    const float2 b = __ldg(P.cbound + A.cbound + ki);
                    mx = b.x;
                    sm = b.y;
                } else if (bound) {
                    // a shell at a time from its own table, the knot index taken
                    // from below against FP32 rounding of d
                    const DevSpecies &S = P.species[A.species];
                    for (int sh = 0; sh < S.n_shell; sh++) {
                        const DevShell R = sh_tab[S.shell0 + sh];
                        const int ki = knot_below(d, R.rcut_f, R.inv_h_hi, R.nk);
                        if (ki < 0) continue;
                        const float tb = __ldg(P.rbound + R.bound_off + ki);
                        float y = 0.f;
                        for (int m = 0; m <= 2 * R.l; m++) y = fmaxf(y, __ldg(P.rbound + R.l * R.l + m));
                        mx = fmaxf(mx, fminf(tb * y, 1.0e30f));
                        sm += fminf(tb * ylm_sum_bound(R.l), 1.0e30f);
                    }
                } else {
                    const DevSpecies &S = P.species[A.species];
                    const float inv_d = __frcp_rn(d);
                    for (int sh = 0; sh < S.n_shell; sh++) {
                        const DevRadial R = P.radials[P.shell_rad[S.shell0 + sh]];
                        int tstep;
                        const float4 *tab = spline_tab(P, S, R, sh, tstep);
                        const float rad = radial_over_d_f32(R, tab, tstep, d, inv_d);
                        float Q[7];
                        int ci[7];
                        ylm_poly_f32(R.l, o.x, o.y, o.z, Q, ci);
#pragma unroll
                        for (int m = 0; m < 7; m++) {
                            if (m >= 2 * R.l + 1) break;
                            const float a = fabsf(rad * kYlmC[ci[m]].x * Q[m]);
                            mx = fmaxf(mx, a);
                            sm += a;
                        }
                    }
                    if (!(mx < 1.0e30f)) mx = 1.0e30f;
                }
                if (!(sm < 1.0e30f)) sm = 1.0e30f;
                mxc = fmaxf(mxc, mx);
                smc += sm;
            }
        }
        colmax[part][k] = mxc;
        colsum[part][k] = smc;
        __syncthreads();
        if (threadIdx.x < 64) {
            float sc, un;
            const float mx = fmaxf(fmaxf(colmax[0][k], colmax[1][k]), fmaxf(colmax[2][k], colmax[3][k]));
            const float sm = (colsum[0][k] + colsum[1][k]) + (colsum[2][k] + colsum[3][k]);
            fixed_scale_adaptive(mx, sm, T.nkc * 64, sc, un);
            csc[k] = make_float2(sc, un);
        }
    }
    __syncthreads();
    if (fixed) density_image_lanes<3>(P, B, T, act, sh_tab, c, phi_img, csc);
    else density_image_lanes<1>(P, B, T, act, sh_tab, c, phi_img, csc);
    // rows from n_b to the end of the contraction's last 16-deep step: zeros
    const int nplanes = fixed ? 3 : 1;
    for (int u = threadIdx.x; u < (-B.nfn & 15) * 8; u += blockDim.x) {
        const int rg = B.nfn + (u >> 3), g = u & 7;
        const long long off = unit_offset(rg >> 7, T.nc_alloc, c, rg & 127, g);
        for (int pl = 0; pl < nplanes; pl++)
            *reinterpret_cast<uint4 *>(phi_img + off + pl * kChunkBytes) = make_uint4(0u, 0u, 0u, 0u);
    }
}

// FP32 value -> signed fixed point with unit 2^-40.  With t = v 2^8,
// h = rint(t) and f = t - h (exact, |f| <= 1/2), the value is
// h 2^32 + trunc(f 2^32): two 32-bit conversions instead of 64-bit shifts.
// The bits below 2^-40 are dropped toward zero (f = +1/2 exactly saturates
// the low word, an error of one unit).  |v| must stay below 2^22; larger or
// non-finite values set *bad.

__device__ __forceinline__ long long f32_to_fix(float v, bool &bad)
{
    const float t = v * 256.f;
    bad |= !(fabsf(t) < 1073741824.f);                 // 2^30; also catches NaN
    const float h = rintf(t);
    const float f = t - h;
    const int hi = __float2int_rz(h);
    const int lo = __float2int_rz(f * 4294967296.f);
    return (long long)hi * 4294967296ll + (long long)lo;
}

// h[k] = (accumulate ? h[k] : 0) + acc[k] 2^-40
__global__ void k_fix_to_h(const long long *acc, double *h, long long n, int accumulate)
{
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const double v = (double)acc[k] * 0x1p-40;
        h[k] = accumulate ? h[k] + v : v;
    }
}

// ----------------------------------------------- H contraction on tcgen05 (K2)
// Persistent: one CTA per SM takes tiles (batch, I, J), I <= J, from a shared
// counter; each tile is 128 x 128 outputs with K = the batch's points in
// chunks of 64, computed transposed (A = phi of block J, B = w v phi of block
// I).  One warp (one lane) fetches tiles ahead, publishes them in a small tile
// ring and streams operand chunks into a shared-memory ring with bulk copies;
// one (one lane) issues the MMAs into one of two tensor-memory accumulator
// sets (acc0 + acc1, 256 columns each); two groups of eight warps, one for each
// set, drain and scatter the upper triangle into the fixed-point H
// accumulator, so the scatter of one tile overlaps the MMAs of the next.  A
// warp's lanes hold 32 consecutive functions j, so the atomics for one column
// i land on consecutive values of row i.
//
// The counter keeps the tiles in flight next to each other in the list: with a
// fixed stride the CTAs drift apart over ~90 super-batches, whose operands
// outgrow L2 (17 GB read from DRAM for 4.7 GB of images in the 64-atom Si
// cluster's density).  Prefetching the next tile's operands into L2 was
// measured 1-3 % slower and is not done.
// Two groups of eight epilogue warps, one for each accumulator set: a group's
// table look-ups and drain of one tile overlap the other group's and the MMAs.
constexpr int kGroupWarps = 8, kGroupThreads = 32 * kGroupWarps;
constexpr int kWarpProducer = 2 * kGroupWarps, kWarpMma = kWarpProducer + 1;
constexpr int kThreadsTc = 32 * (kWarpMma + 1);
// Ring of operand chunks, A and B of 64 contraction steps each.  Four stages of
// 32 (64-byte rows) are slower, 64-atom Si cluster: H 3.15 -> 3.44 ms, density
// 3.57 -> 3.84: a stage boundary costs the MMA warp about 220 clocks that the
// queue behind it does not hide.
constexpr int kStages = 2;
constexpr int kOperandBytes = kChunkStride;      // three planes
constexpr int kStageBytes = 2 * kOperandBytes;
// split products kept in the density: combined order <= 3 except x2*y2 (8 of
// 9), as in H; the order-3 pair x1*y2, x2*y1 is about 2^-27 of the leading
// product, which over ~10^3 functions is no longer far below the 1e-7
// relative bound on n
constexpr int kDensityOrder = 3;

// One tile, resolved by the producer so that the other roles have no chain of
// dependent global loads.
struct TileInfo {
    int ti, tj;                                  // H: blocks I, J; density: point tile m, block J.  ti < 0: no more tiles
    int np, nfn;                                 // points and functions of the batch
    int nc, nkc, nc_alloc;                       // see TcBatch
    int sign;                                    // H: of w v over the batch
    long long img_phi, img_e, part_row;          // density
    long long pad;
};
constexpr int kTiles = 4;                        // tile ring
constexpr int kPairSlots = 32;                   // atoms of a block in the pair table

// An H tile's rows and columns as the epilogue needs them: the descriptors of
// blocks I and J (HBlock, written with the operand images).
struct HTile {
    HBlock i, j;
};

// Scatter tables of one group: for column i the address of the first stored
// value of row i less i's index in its atom; for a pair of atoms (of I, of J)
// the byte offset from there to atom(j)'s run, 0 for the same atom, negative
// where the pair is not stored.
struct HColumn {
    unsigned long long base;
    int pair_row;                                // first entry of the column's atom in pair
    int pad;
};
struct HTables {
    HColumn col[128];
    int pair[kPairSlots * kPairSlots];
};

struct TcRing {
    uint64_t full[kStages], empty[kStages];
    uint64_t tfull[2], tempty[2];                // accumulator sets
    uint64_t nfull[kTiles], nempty[kTiles];      // tile ring
    TileInfo tile[kTiles];
    uint32_t tmem;
    int abort;
    int go[2];                                   // per group: the tile's entry holds a tile
};

__device__ __forceinline__ uint8_t *align1024(uint8_t *p)
{
    return reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(p) + 1023) & ~(uintptr_t)1023);
}

// named barrier of one group of epilogue warps
__device__ __forceinline__ void group_sync(int group)
{
    asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kGroupThreads) : "memory");
}

__device__ __forceinline__ void ring_init(TcRing *S)
{
    for (int s = 0; s < kStages; s++) {
        mbar_init(&S->full[s], 1);
        mbar_init(&S->empty[s], 1);
    }
    for (int b = 0; b < 2; b++) {
        mbar_init(&S->tfull[b], 1);
        mbar_init(&S->tempty[b], kGroupThreads);
    }
    for (int e = 0; e < kTiles; e++) {
        mbar_init(&S->nfull[e], 1);
        mbar_init(&S->nempty[e], 2);             // the MMA warp and the tile's epilogue group
    }
    S->abort = 0;
    fence_mbar_init();
}

// The operand ring: stage n % kStages holds the n-th chunk, in the order the
// producer and the MMA warp both walk.  Producer: room for chunk n (false:
// timed out).
__device__ __forceinline__ bool stage_wait_empty(TcRing *S, uint32_t n, int *status)
{
    return n < kStages || mbar_wait_a(&S->empty[n % kStages], (n / kStages - 1) & 1, status, &S->abort);
}

__device__ __forceinline__ bool stage_wait_full(TcRing *S, uint32_t n, int *status)
{
    return mbar_wait_a(&S->full[n % kStages], (n / kStages) & 1, status, &S->abort);
}

// Producer, at the end: do not leave while one of its n copies may still be landing
__device__ __forceinline__ void ring_drain(TcRing *S, uint32_t n)
{
    for (uint32_t q = (n > kStages ? n - kStages : 0); q < n; q++) mbar_drain(&S->full[q % kStages], (q / kStages) & 1);
}

// ---- tile ring: entry lt % kTiles holds this CTA's lt-th tile, drained by
// group lt % 2
//
// Producer side: the next tiles of the shared list, their tables loading while
// the tile before them streams.  A CTA holds three tiles of the list at a time; its
// first three are a grid apart and the counter gives the rest, so that a list
// shorter than that is spread evenly.  (With the first three from the counter too, the first
// CTAs to arrive took three each and the others none: a water molecule's H, 32
// tiles, 55.6 -> 43.3 us.)
struct TileFetch {
    const WorkItem *items;
    const TcBatch *tb;
    const DevBatch *batches;
    const int *bsign;                            // H only
    unsigned int *counter;
    unsigned int n_items;
    WorkItem it;                                 // current tile and its tables
    TcBatch T;
    int np, nfn, sign;
    bool have;
    WorkItem it1;                                // the next tile
    bool have1;
    unsigned int idx2;                           // index of the one after it
};

__device__ __forceinline__ void fetch_tables(TileFetch &F)
{
    if (!F.have) return;
    F.T = F.tb[F.it.batch];
    F.np = F.batches[F.it.batch].np;
    F.nfn = F.batches[F.it.batch].nfn;
    F.sign = F.bsign ? F.bsign[F.it.batch] : 0;
}

__device__ __forceinline__ WorkItem fetch_item(const TileFetch &F, unsigned int k, bool &have)
{
    have = k < F.n_items;
    return have ? F.items[k] : WorkItem{0, 0, 0};
}

__device__ __forceinline__ void fetch_start(TileFetch &F)
{
    F.idx2 = blockIdx.x + 2 * gridDim.x;
    F.it = fetch_item(F, blockIdx.x, F.have);
    F.it1 = fetch_item(F, blockIdx.x + gridDim.x, F.have1);
    fetch_tables(F);
}

// the following tile becomes the current one
__device__ __forceinline__ void fetch_next(TileFetch &F)
{
    F.it = F.it1;
    F.have = F.have1;
    F.it1 = fetch_item(F, F.idx2, F.have1);
    F.idx2 = 3 * gridDim.x + atomicAdd(F.counter, 1u);
    fetch_tables(F);
}

__device__ __forceinline__ bool tile_wait_empty(TcRing *S, uint32_t lt, int *status)
{
    return lt < kTiles || mbar_wait_a(&S->nempty[lt % kTiles], (lt / kTiles - 1) & 1, status, &S->abort);
}

__device__ __forceinline__ bool tile_wait_full(TcRing *S, uint32_t lt, int *status)
{
    return mbar_wait_a(&S->nfull[lt % kTiles], (lt / kTiles) & 1, status, &S->abort);
}

// Producer, after its last tile (lt of them): an end mark for each group; returns
// how many places of the ring they took
__device__ __forceinline__ uint32_t tiles_end(TcRing *S, uint32_t lt, int *status)
{
    for (uint32_t k = 0; k < 2; k++) {
        if (!tile_wait_empty(S, lt + k, status)) return k;
        S->tile[(lt + k) % kTiles].ti = -1;
        mbar_arrive(&S->nfull[(lt + k) % kTiles]);
    }
    return 2;
}

// Epilogue group: its next tile; false at the end (or after a time-out) for
// all of the group's threads alike, so that none skips a named barrier
__device__ __forceinline__ bool group_next_tile(TcRing *S, uint32_t lt, int group, int tid, int *status)
{
    if (tid == 0) S->go[group] = tile_wait_full(S, lt, status) && S->tile[lt % kTiles].ti >= 0;
    group_sync(group);
    // every thread looks at the barrier itself: it orders the tile's copies before its reads
    return S->go[group] != 0 && tile_wait_full(S, lt, status);
}

// Issue the split products of the first nks 16-deep steps of a 64-deep chunk:
// every product of combined order <= ORDER except x2*y2; x0*y0 alone in
// accumulator 0.  The plane and k-step offsets are added to the descriptors'
// address field (addr >> 4, no carry out of it inside shared memory).
// The tensor pipe holds few MMAs in its queue, so what its warp does between
// them shows: the whole warp walks the loops and one lane issues, which leaves
// the descriptors in uniform registers (40 instead of 50 cycles an MMA, 64 the
// pipe needs), and a stage has one barrier each way.  Without epilogues a
// 64-deep chunk takes 2252 cycles this way, 2048 of them the pipe's, and took
// 2880 with one lane in divergent code and a barrier an operand.
// first: the chunk opens the item (the first product into each accumulator
// overwrites it).
// The planes of the first operand go slowest.  It is A (K-major) for H; for the
// density (PHI_A) it is B and the second operand, read as MN-major, is A, so
// that the points lie along the lanes of the accumulators.
template <int NSPLIT, int ORDER, bool PHI_A>
__device__ __forceinline__ void mma_chunk(uint32_t acc_base, const uint8_t *sm1, const uint8_t *sm2, uint32_t idesc,
                                          bool first, int nks)
{
    uint64_t d1 = desc_sw128(smem_u32(sm1), 16, 1024);
    uint64_t d2 = PHI_A ? desc_sw128(smem_u32(sm2), 8192, 1024) : desc_sw128(smem_u32(sm2), 16, 1024);
#pragma unroll 1
    for (int ks = 0; ks < nks; ks++) {
        if (elect_one()) {
#pragma unroll
            for (int p1 = 0; p1 < NSPLIT; p1++) {
#pragma unroll
                for (int p2 = 0; p2 < NSPLIT; p2++) {
                    if (p1 + p2 > ORDER || (p1 == 2 && p2 == 2)) continue;
                    const int acc = (p1 + p2 == 0) ? 0 : 1;
                    const bool opens = acc == 0 || (p1 == 0 && p2 == 1);
                    const uint64_t e1 = d1 + (uint64_t)((p1 * kChunkBytes) >> 4), e2 = d2 + (uint64_t)((p2 * kChunkBytes) >> 4);
                    tc_mma(acc_base + acc * 128, PHI_A ? e2 : e1, PHI_A ? e1 : e2, idesc,
                           (opens && first && ks == 0) ? 0u : 1u);
                }
            }
        }
        d1 += 32 >> 4;
        d2 += (PHI_A ? 2048 : 32) >> 4;
    }
}

__global__ void __launch_bounds__(kThreadsTc, 1) k_tc_h(DevPlan P, const TcBatch *tb, const WorkItem *items,
                                                        int n_items, const uint8_t *ws, unsigned long long *hfix,
                                                        int n_split, const int *bsign, unsigned int *counter)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = align1024(smem_raw);
    HTile *htile = reinterpret_cast<HTile *>(sm + kStages * kStageBytes);       // [kTiles]
    HTables *tables = reinterpret_cast<HTables *>(htile + kTiles);            // [2]
    TcRing *S = reinterpret_cast<TcRing *>(tables + 2);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) ring_init(S);
    if (warp == kWarpMma) {
        tmem_alloc(&S->tmem, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S->tmem;
    const uint32_t chunk = (uint32_t)n_split * kChunkBytes;

    // A = phi rows of block J (TMEM lanes), B = w v phi rows of block I (TMEM
    // columns): the transposed tile, so that the scatter of one column i by the
    // 32 lanes of a warp hits consecutive values of row i.  Batches where w v has
    // one sign hold psi = phi sqrt|w v| in the phi image, which then serves as
    // both operands; their diagonal tiles need one chunk for the two.
    if (warp == kWarpProducer) {
        if (lane == 0) {
            uint32_t n = 0, lt = 0;
            bool ok = true;
            TileFetch F{};
            F.items = items;
            F.tb = tb;
            F.batches = P.batches;
            F.bsign = bsign;
            F.counter = counter;
            F.n_items = (unsigned int)n_items;
            for (fetch_start(F); F.have && ok; lt++) {
                const WorkItem it = F.it;
                const TcBatch T = F.T;
                const bool same = F.sign != 0 && it.ti == it.tj;
                if (!(ok = tile_wait_empty(S, lt, P.status))) break;
                const int e = (int)(lt % kTiles);
                TileInfo &I = S->tile[e];
                I.ti = it.ti;
                I.tj = it.tj;
                I.np = F.np;
                I.nfn = F.nfn;
                I.nc = T.nc;
                I.sign = F.sign;
                mbar_expect_tx(&S->nfull[e], 2 * (uint32_t)sizeof(HBlock));
                const HBlock *hb = reinterpret_cast<const HBlock *>(ws + T.hblock);
                bulk_g2s(&htile[e].i, hb + it.ti, sizeof(HBlock), &S->nfull[e]);
                bulk_g2s(&htile[e].j, hb + it.tj, sizeof(HBlock), &S->nfull[e]);
                const uint8_t *a_img = ws + T.img_phi + (long long)it.tj * T.nc_alloc * kChunkStride;
                const uint8_t *b_img = ws + (F.sign != 0 ? T.img_phi : T.img_aux) + (long long)it.ti * T.nc_alloc * kChunkStride;
                fetch_next(F);
                for (int c = 0; c < T.nc; c++) {
                    if (!(ok = stage_wait_empty(S, n, P.status))) break;
                    const uint32_t q = n++ % kStages;
                    uint8_t *dst = sm + q * kStageBytes;
                    mbar_expect_tx(&S->full[q], same ? chunk : 2 * chunk);
                    bulk_g2s(dst, a_img + (long long)c * kChunkStride, chunk, &S->full[q]);
                    if (!same) bulk_g2s(dst + kOperandBytes, b_img + (long long)c * kChunkStride, chunk, &S->full[q]);
                }
            }
            const uint32_t marks = ok ? tiles_end(S, lt, P.status) : 0;
            ring_drain(S, n);
            // nor while a tile's descriptors may (those of older tiles and those in
            // the places of the marks have been read)
            for (uint32_t q = lt + marks > kTiles ? lt + marks - kTiles : 0; q < lt; q++)
                mbar_drain(&S->nfull[q % kTiles], (q / kTiles) & 1);
        }
        __syncwarp();
    } else if (warp == kWarpMma) {
        uint32_t n = 0;
        uint32_t lt = 0;
        bool ok = true;
        for (; ok && __all_sync(0xffffffffu, tile_wait_full(S, lt, P.status)); lt++) {
            const int e = (int)(lt % kTiles);
            const int ti = S->tile[e].ti, tj = S->tile[e].tj, np = S->tile[e].np, nfn = S->tile[e].nfn, nc = S->tile[e].nc;
            const bool same = S->tile[e].sign != 0 && ti == tj;
            if (ti < 0) break;
            __syncwarp();
            if (elect_one()) mbar_arrive(&S->nempty[e]);
            // the columns of the last block end at n_b
            const uint32_t idesc = idesc_bf16(128, min(128, (nfn - ti * 128 + 15) & ~15), false, false);
            const uint32_t buf = lt & 1, use = lt >> 1;
            ok = use == 0 || mbar_wait_a(&S->tempty[buf], (use - 1) & 1, P.status, &S->abort);
            tc_fence_after();
            for (int c = 0; c < nc; c++, n++) {
                ok = __all_sync(0xffffffffu, ok && stage_wait_full(S, n, P.status));
                if (!ok) break;
                // steps past the batch's points would add zeros
                const int nks = min(4, (np - c * 64 + 15) >> 4);
                const uint8_t *a_sm = sm + (n % kStages) * kStageBytes, *b_sm = same ? a_sm : a_sm + kOperandBytes;
                if (n_split == 3)
                    mma_chunk<3, 3, false>(tmem + buf * 256, a_sm, b_sm, idesc, c == 0, nks);
                else
                    mma_chunk<1, 0, false>(tmem + buf * 256, a_sm, b_sm, idesc, c == 0, nks);
                if (elect_one()) tc_commit(&S->empty[n % kStages]);
            }
            if (elect_one()) tc_commit(&S->tfull[buf]);
        }
        // the last commit covers every MMA before it
        if (lt > 0) mbar_drain(&S->tfull[(lt - 1) & 1], ((lt - 1) >> 1) & 1);
        __syncwarp();
    } else {
        // Warp w of a group: TMEM lanes 32 (w % 4) .. + 31 (functions j of block
        // J), columns 64 (w / 4) .. + 63 (functions i of block I).  Bound by the
        // instructions of the conversion to fixed point (about 20 a value).
        const int group = warp >> 3, quad = warp & 3, half = (warp >> 2) & 1;
        const int tid = threadIdx.x & (kGroupThreads - 1), r = quad * 32 + lane;
        HTables &H = tables[group];
        const uint32_t acc_base = tmem + group * 256 + ((uint32_t)(quad * 32) << 16);
        bool bad = false;
        for (uint32_t lt = group; group_next_tile(S, lt, group, tid, P.status); lt += 2) {
            const int e = (int)(lt % kTiles);
            const int ti = S->tile[e].ti, tj = S->tile[e].tj;
            const HBlock &bi = htile[e].i, &bj = htile[e].j;
            const int ncol = bi.n, ni = bi.nslot, nj = bj.nslot;
            const float scale = S->tile[e].sign < 0 ? -256.f : 256.f;    // H = -psi^T psi
            const int *pp_sys = P.pairpos + bi.pair_off;
            const long long nat = bi.nat;
            const bool tab = ni <= kPairSlots && nj <= kPairSlots;
            if (tid < 128)
                H.col[tid] = HColumn{(unsigned long long)__cvta_generic_to_global(hfix + bi.base[tid]),
                                     bi.slot[tid] * kPairSlots, 0};
            if (tab) {
                for (int q = tid; q < ni * kPairSlots; q += kGroupThreads) {
                    const int a = q / kPairSlots, b = q % kPairSlots;
                    if (b >= nj) continue;
                    const int pp = bi.loc[a] == bj.loc[b] ? 0 : __ldg(pp_sys + bi.loc[a] * nat + bj.loc[b]);
                    H.pair[q] = pp < 0 ? INT_MIN : 8 * pp;
                }
            }
            // this lane's function j
            const int sj = bj.slot[r], lj = 8 * bj.li[r], locj = bj.loc[sj];
            const bool inj = r < bj.n;
            group_sync(group);
            const bool ok = mbar_wait_a(&S->tfull[group], (lt >> 1) & 1, P.status, &S->abort);
            tc_fence_after();
            // (i, j) is stored for i <= j: only diagonal tiles cross that line
            const int rlim = !inj ? -1 : ti == tj ? r : 127;
            for (int cq = 0; cq < 2; cq++) {
                const int c0 = 64 * half + 32 * cq;
                if (c0 >= ncol) break;
                float a0[32], a1[32];
                tmem_ld32(acc_base + c0, a0);
                if (n_split > 1) tmem_ld32(acc_base + 128 + c0, a1);
                else
#pragma unroll
                    for (int q = 0; q < 32; q++) a1[q] = 0.f;
                tmem_wait_ld();
                if (!ok) continue;
                if (ncol - c0 < 32) {
                    // columns past n_b hold what was there before: products of stale image
                    // rows, an earlier tile's values or none at all
#pragma unroll
                    for (int q = 0; q < 32; q++) {
                        a0[q] = c0 + q < ncol ? a0[q] : 0.f;
                        a1[q] = c0 + q < ncol ? a1[q] : 0.f;
                    }
                }
                float size = 0.f;
#pragma unroll
                for (int q = 0; q < 32; q++) size = max_abs_nan(size, a0[q], a1[q]);
                if (!inj) size = 0.f;              // a row past n_b
                if (tab && !__any_sync(0xffffffffu, !(size < 16384.f))) {
                    // v 2^8 = h + f with h its rounding (by an addition, the FRND unit
                    // is slow), f exact: h 2^32 + f 2^32 in units of 2^-40, the sign of
                    // the batch in the factor
#pragma unroll
                    for (int q = 0; q < 32; q++) {
                        const int il = c0 + q;
                        const HColumn col = H.col[il];
                        const int off = H.pair[col.pair_row + sj];
                        const float h0 = fmaf(a0[q], scale, kRoundMagic), h1 = fmaf(a1[q], scale, kRoundMagic);
                        const float f0 = fmaf(a0[q], scale, -(h0 - kRoundMagic)), f1 = fmaf(a1[q], scale, -(h1 - kRoundMagic));
                        // the words of kRoundMagic + h less those of kRoundMagic
                        const int hi = (int)(__float_as_uint(h0) + __float_as_uint(h1) - 2u * 0x4B400000u);
                        const long long fx = (((long long)hi << 32) + __float2int_rz(f0 * 4294967296.f)) +
                                             __float2int_rz(f1 * 4294967296.f);
                        red_add_if(off >= 0 && il <= rlim && fx != 0, col.base + (unsigned int)(off + lj), fx);
                    }
                    continue;
                }
                // values of 2^14 Ha and more (or not finite), or more atoms than the
                // pair table holds
                const float sgn = scale * 0.00390625f;
#pragma unroll
                for (int q = 0; q < 32; q++) {
                    const int il = c0 + q;
                    if (il > rlim || il >= ncol) continue;
                    const int loci = bi.loc[bi.slot[il]];
                    const int pp = loci == locj ? 0 : __ldg(pp_sys + loci * nat + locj);
                    const long long fx = f32_to_fix(a0[q] * sgn, bad) + f32_to_fix(a1[q] * sgn, bad);
                    red_add_if(pp >= 0 && fx != 0, H.col[il].base + 8ll * pp + lj, fx);
                }
            }
            tc_fence_before();
            mbar_arrive(&S->tempty[group]);
            group_sync(group);                     // the tables may be filled again
            if (tid == 0) mbar_arrive(&S->nempty[e]);
        }
        if (bad) atomicOr(P.status, kStatusNonFinite);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kWarpMma) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------- D_b gather (K3a)
// CTA per (batch, 128-row block J): D(j, i) for local functions j (rows) and
// i (columns) from the stored upper triangle, split into BF16 planes as a
// K-major swizzled image.  In the split mode the leading term is fixed-point
// on a per-row grid (the density contracts over i), found by a first pass
// over the row block.
// D values as double-floats (once per density call; nnz elements), and for
// every function g the largest |D_gi| and the sum of |D_gi| over its full
// symmetric row: bounds (valid for every batch) for the fixed-point grid of
// the gathered rows.  One warp per row of the stored upper triangle.
__global__ void k_to_df(const double *x, float2 *out, const long long *rowptr, const int *fn_sys,
                        const long long *sys_val0, const long long *sys_nnz, long long n_fn, unsigned int *gmax,
                        float *gsum)
{
    const int lane = threadIdx.x & 31;
    const long long warp0 = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long g = warp0; g < n_fn; g += nwarps) {
        const int s = fn_sys[g];
        const long long k0 = rowptr[g];
        const long long k1 = (g + 1 < n_fn && fn_sys[g + 1] == s) ? rowptr[g + 1] : sys_val0[s] + sys_nnz[s];
        float mx = 0.f, sm = 0.f;
        for (long long k = k0 + lane; k < k1; k += 32) {
            const df v = df_from_double(x[k]);
            out[k] = make_float2(v.hi, v.lo);
            float a = fabsf(v.hi);
            if (!(a < 1.0e30f)) a = 1.0e30f;
            mx = fmaxf(mx, a);
            sm += a;
        }
        mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sm += __shfl_xor_sync(0xffffffffu, sm, o);
        if (lane == 0) {
            atomicMax(gmax + g, __float_as_uint(mx));
            atomicAdd(gsum + g, sm);
        }
    }
}

constexpr int kGatherActSmem = 512;     // active atoms of a batch the gather stages in shared memory

// the column side of the symmetric rows: value (g, j), j > g, bounds row j
__global__ void k_d_colbounds(const float2 *v, const int *col_of, long long nnz, unsigned int *gmax, float *gsum)
{
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < nnz; k += (long long)gridDim.x * blockDim.x) {
        const int j = col_of[k];
        if (j < 0) continue;                       // diagonal entries are counted once
        float a = fabsf(v[k].x);
        if (!(a < 1.0e30f)) a = 1.0e30f;
        atomicMax(gmax + j, __float_as_uint(a));
        atomicAdd(gsum + j, a);
    }
}

// Row j of the gather: with li_j its index in its atom, `base` = (first stored
// value of row j) - li_j.  A stored value (j, i) with i >= j lies at base +
// [start of atom(i)'s run in the row, 0 for j's own atom] + li_i; one with
// i < j in row i at (row i's base) + [start of atom(j)'s run] + li_j.
struct GatherRow {
    long long base;
    int atom, loc, li, pad;
};

// Bound by the latency and sectors of the loads of D.  One warp walks 16 rows,
// a lane owns two neighbouring columns of the 64-column chunk: a row's loads
// are the consecutive stored values of its runs, and its three stores are
// whole 128-byte rows of the image.  The offset of a (row atom, column) pair
// is looked up once per row atom; four rows' loads are in flight together.
// (Eight values a thread, its loads 64 bytes apart and a table search a value,
// took 300 issue slots a value: 64-atom Si cluster, 1368 super-batches, 3.2 ms;
// now 0.8 ms, the full G of the adjoint 5.2 -> 1.5 ms.)
template <int NSPLIT>
__global__ void __launch_bounds__(256) k_tc_gather_d(DevPlan P, const TcBatch *tb, const WorkItem *items,
                                                     uint8_t *ws, const float2 *ddv, const unsigned int *gmax,
                                                     const float *gsum, float offdiag_scale, int full)
{
    const WorkItem it = items[blockIdx.x];
    const DevBatch B = P.batches[it.batch];
    const TcBatch T = tb[it.batch];
    const int J = it.ti;
    __shared__ GatherRow row[128];
    __shared__ float2 rsc[128];                      // per row: scale, unit
    __shared__ int4 sact[kGatherActSmem];            // per active atom: fn_loc, atom, loc, first global fn
    const DevAct *act = P.act + B.act0;
    const int *pp_sys = P.pairpos + P.sys_pair_off[B.sys];
    const long long nat = P.sys_nat[B.sys];
    const bool staged = B.n_act <= kGatherActSmem;
    if (staged) {
        for (int e = threadIdx.x; e < B.n_act; e += blockDim.x) {
            const DevAct A = act[e];
            sact[e] = make_int4(A.fn_loc, A.atom, P.atom_loc[A.atom], (int)P.atom_fn0[A.atom]);
        }
    }
    __syncthreads();
    // entry e of the active atoms, and the last one that starts at or before l
    auto entry = [&](int e) -> int4 {
        if (staged) return sact[e];
        const DevAct A = act[e];
        return make_int4(A.fn_loc, A.atom, P.atom_loc[A.atom], (int)P.atom_fn0[A.atom]);
    };
    auto find = [&](int l) -> int {
        int lo = 0, hi = B.n_act - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((staged ? sact[mid].x : act[mid].fn_loc) <= l) lo = mid; else hi = mid - 1;
        }
        return lo;
    };
    if (threadIdx.x < 128) {
        const int j = J * 128 + threadIdx.x;
        GatherRow g{0, -1, 0, 0, 0};
        float sc = 0.f, un = 0.f;
        if (j < B.nfn) {
            const int4 a = entry(find(j));
            g.li = j - a.x;
            g.atom = a.y;
            g.loc = a.z;
            const long long gi = (long long)a.w + g.li;
            g.base = P.rowptr[gi] - g.li;
            if (NSPLIT == 3) fixed_scale_adaptive(__uint_as_float(gmax[gi]), gsum[gi], T.nkc * 64, sc, un);
        }
        row[threadIdx.x] = g;
        rsc[threadIdx.x] = make_float2(sc, un);
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t g16 = (uint32_t)(lane >> 2) << 4, cb = (uint32_t)(lane & 3) * 4u;
    uint8_t *img = ws + T.img_aux + (long long)J * T.nkc * kChunkStride;
    // D is symmetric: block row J holds only the chunks i >= 128 J, the
    // diagonal block halved (n = 2 sum_J phi_J . E_J, exact in binary); in
    // full (the adjoint's G Phi) every chunk, nothing halved
    for (int kc = full ? 0 : 2 * J; kc < T.nkc; kc++) {
        const float blk = (!full && kc < 2 * J + 2) ? 0.5f : 1.f;
        const int i0 = kc * 64 + 2 * lane;
        int catom[2], cloc[2], cli[2];
        long long cbase[2] = {0, 0};                 // row i's base, for values below the diagonal
        bool cin[2];
        int e = find(min(i0, B.nfn - 1));
#pragma unroll
        for (int c = 0; c < 2; c++) {
            const int i = i0 + c;
            cin[c] = i < B.nfn;
            if (c == 1 && cin[1] && e + 1 < B.n_act && (staged ? sact[e + 1].x : act[e + 1].fn_loc) <= i) e++;
            const int4 a = entry(e);
            catom[c] = a.y;
            cloc[c] = a.z;
            cli[c] = i - a.x;
            if (cin[c] && kc < 2 * J + 2) cbase[c] = P.rowptr[(long long)a.w + cli[c]] - cli[c];
        }
        int cur = -2;                                // the row atom of up/low/ok
        long long up[2] = {0, 0}, low[2] = {0, 0};
        bool ok[2] = {false, false};
        for (int rb = warp * 16; rb < warp * 16 + 16; rb += 4) {
            float2 v[4][2];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const GatherRow g = row[rb + q];
                const int j = J * 128 + rb + q;
                if (g.atom != cur) {                 // the same for the whole warp
                    cur = g.atom;
#pragma unroll
                    for (int c = 0; c < 2; c++) {
                        int pp = 0;
                        if (cur >= 0 && cin[c] && catom[c] != cur)
                            pp = catom[c] > cur ? __ldg(pp_sys + g.loc * nat + cloc[c])
                                                : __ldg(pp_sys + cloc[c] * nat + g.loc);
                        ok[c] = cur >= 0 && cin[c] && pp >= 0;
                        up[c] = pp + cli[c];
                        low[c] = cbase[c] + pp;
                    }
                }
#pragma unroll
                for (int c = 0; c < 2; c++) {
                    v[q][c] = make_float2(0.f, 0.f);
                    const long long k = i0 + c >= j ? g.base + up[c] : low[c] + g.li;
                    if (ok[c]) v[q][c] = __ldg(ddv + k);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int r = rb + q, j = J * 128 + r;
                const float2 su = rsc[r];
                uint32_t w0, w1 = 0, w2 = 0;
                if (NSPLIT == 3) {
                    float x0[2], d[2], lo[2];
#pragma unroll
                    for (int c = 0; c < 2; c++) {
                        const float s = (i0 + c == j ? 1.f : offdiag_scale) * blk;
                        const float hi = v[q][c].x * s;
                        lo[c] = v[q][c].y * s;
                        x0[c] = rintf(hi * su.x) * su.y;
                        d[c] = hi - x0[c];
                    }
                    w0 = pack2_bf16(x0[0], x0[1]);
                    w1 = pack2_bf16(d[0], d[1]);
                    w2 = pack2_bf16((d[0] - __uint_as_float(w1 << 16)) + lo[0],
                                    (d[1] - __uint_as_float(w1 & 0xFFFF0000u)) + lo[1]);
                } else {
                    w0 = pack2_bf16(v[q][0].x * ((i0 == j ? 1.f : offdiag_scale) * blk),
                                    v[q][1].x * ((i0 + 1 == j ? 1.f : offdiag_scale) * blk));
                }
                uint8_t *dst = img + (long long)kc * kChunkStride + row_offset((uint32_t)r, g16) + cb;
                *reinterpret_cast<uint32_t *>(dst) = w0;
                if (NSPLIT == 3) {
                    *reinterpret_cast<uint32_t *>(dst + kChunkBytes) = w1;
                    *reinterpret_cast<uint32_t *>(dst + 2 * kChunkBytes) = w2;
                }
            }
        }
    }
}

// ------------------------------------------------- density on tcgen05 (K3b)
// Persistent, with the roles, the rings and the tile counter of the H
// contraction, over the items (batch, 128-point tile m, 128-function block J),
// J ascending so the longest contractions come first:
// E[p][j] = sum_{i >= 128 J} phi_i(p) D'[j][i] over the upper block
// triangle of the symmetric D (D' = D with its diagonal block halved;
// A = phi image read as MN-major, B = D image, K-major) accumulates in one of
// two tensor-memory sets while a group of warps finishes an earlier item: the
// partial density sum_{j in J} E[p][j] phi_j(p) in double-float, a thread its
// own point p (tensor-memory lane) and half of the j, one row of 128 doubles
// per item.  Many items per batch keep the CTAs on few batches at a
// time, so the D and phi images are read from L2.  k_density_sum then forms
// n_p = 2 sum_J partial_J(p).
//
// ADJ (the adjoint's E = G Phi): every function chunk of the full G image,
// and each thread also stores its point's E (acc0 + acc1 in FP32; rows of
// points) for the position gradient.
template <bool ADJ>
__global__ void __launch_bounds__(kThreadsTc, 1) k_tc_density(DevPlan P, const TcBatch *tb, const WorkItem *items,
                                                              int n_items, const uint8_t *ws, double *part,
                                                              int n_split, uint8_t *ws_e, unsigned int *counter)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sm = align1024(smem_raw);
    TcRing *S = reinterpret_cast<TcRing *>(sm + kStages * kStageBytes);
    __shared__ double red[2][2][128];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) ring_init(S);
    if (warp == kWarpMma) {
        tmem_alloc(&S->tmem, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S->tmem;
    const uint32_t chunk = (uint32_t)n_split * kChunkBytes;

    if (warp == kWarpProducer) {
        if (lane == 0) {
            uint32_t n = 0, lt = 0;
            bool ok = true;
            TileFetch F{};
            F.items = items;
            F.tb = tb;
            F.batches = P.batches;
            F.counter = counter;
            F.n_items = (unsigned int)n_items;
            for (fetch_start(F); F.have && ok; lt++) {
                const TcBatch T = F.T;
                const int m = F.it.ti, J = F.it.tj;
                if (!(ok = tile_wait_empty(S, lt, P.status))) break;
                TileInfo &I = S->tile[lt % kTiles];
                I.ti = m;
                I.tj = J;
                I.np = F.np;
                I.nfn = F.nfn;
                I.nkc = T.nkc;
                I.nc_alloc = T.nc_alloc;
                I.img_phi = T.img_phi;
                I.img_e = T.img_e;
                I.part_row = T.part0 + (long long)J * (T.nc_alloc / 2) + m;
                mbar_arrive(&S->nfull[lt % kTiles]);
                fetch_next(F);
                const uint8_t *d_img = ws + T.img_aux + (long long)J * T.nkc * kChunkStride, *phi_img = ws + T.img_phi;
                // a last tile of at most 64 points has one column chunk
                const int halves = 2 * m + 1 < T.nc ? 2 : 1;
                for (int kc = ADJ ? 0 : 2 * J; kc < T.nkc; kc++) {
                    if (!(ok = stage_wait_empty(S, n, P.status))) break;
                    const uint32_t q = n++ % kStages;
                    uint8_t *dst = sm + q * kStageBytes;
                    mbar_expect_tx(&S->full[q], chunk + (uint32_t)(n_split * halves * 8192));
                    bulk_g2s(dst, d_img + (long long)kc * kChunkStride, chunk, &S->full[q]);
                    for (int c2 = 0; c2 < halves; c2++)
                        for (int s = 0; s < n_split; s++)
                            bulk_g2s(dst + kOperandBytes + s * kChunkBytes + c2 * 8192,
                                     phi_img + (long long)((kc >> 1) * T.nc_alloc + 2 * m + c2) * kChunkStride +
                                         s * kChunkBytes + (kc & 1) * 8192,
                                     8192, &S->full[q]);
                }
            }
            if (ok) tiles_end(S, lt, P.status);
            ring_drain(S, n);
        }
        __syncwarp();
    } else if (warp == kWarpMma) {
        uint32_t n = 0;
        uint32_t lt = 0;
        bool ok = true;
        for (; ok && __all_sync(0xffffffffu, tile_wait_full(S, lt, P.status)); lt++) {
            const int e = (int)(lt % kTiles);
            const int m = S->tile[e].ti, J = S->tile[e].tj, nfn = S->tile[e].nfn, nkc = S->tile[e].nkc;
            if (m < 0) break;
            __syncwarp();
            if (elect_one()) mbar_arrive(&S->nempty[e]);
            // the columns of the last block end at n_b
            const uint32_t idesc = idesc_bf16(128, min(128, (nfn - J * 128 + 15) & ~15), true, false);
            const uint32_t buf = lt & 1, use = lt >> 1;
            ok = use == 0 || mbar_wait_a(&S->tempty[buf], (use - 1) & 1, P.status, &S->abort);
            tc_fence_after();
            const int kc0 = ADJ ? 0 : 2 * J;
            for (int kc = kc0; kc < nkc; kc++, n++) {
                ok = __all_sync(0xffffffffu, ok && stage_wait_full(S, n, P.status));
                if (!ok) break;
                // steps past the batch's functions would add zeros
                const int nks = min(4, (nfn - kc * 64 + 15) >> 4);
                const uint8_t *a_sm = sm + (n % kStages) * kStageBytes, *b_sm = a_sm + kOperandBytes;
                if (n_split == 3)
                    mma_chunk<3, kDensityOrder, true>(tmem + buf * 256, a_sm, b_sm, idesc, kc == kc0, nks);
                else
                    mma_chunk<1, 0, true>(tmem + buf * 256, a_sm, b_sm, idesc, kc == kc0, nks);
                if (elect_one()) tc_commit(&S->empty[n % kStages]);
            }
            if (elect_one()) tc_commit(&S->tfull[buf]);
        }
        // the last commit covers every MMA before it
        if (lt > 0) mbar_drain(&S->tfull[(lt - 1) & 1], ((lt - 1) >> 1) & 1);
        __syncwarp();
    } else {
        // Warp w of a group: TMEM lanes 32 (w % 4) .. + 31 (points of the tile),
        // columns 64 (w / 4) .. + 63 (functions j of the block), eight at a time.
        // Bound by its instructions, about 17 a value of E in packed pairs of j.
        // (With the functions along the lanes, the sum over them took a butterfly
        // of selects and shuffles and 37 instructions a value: the epilogue alone
        // needed 6.4 of the 7.4 ms of 64 molecules' density.)
        const int group = warp >> 3, quad = warp & 3, half = (warp >> 2) & 1;
        const int tid = threadIdx.x & (kGroupThreads - 1), pl = quad * 32 + lane;
        const uint32_t acc_base = tmem + group * 256 + ((uint32_t)(quad * 32) << 16) + 64 * half;
        const uint32_t g16 = (uint32_t)((pl >> 3) & 7) << 4, pb = (uint32_t)(pl & 7) * 2u;
        for (uint32_t lt = group; group_next_tile(S, lt, group, tid, P.status); lt += 2) {
            const TileInfo T = S->tile[lt % kTiles];
            const int m = T.ti, J = T.tj;
            const int nj = min(64, T.nfn - J * 128 - 64 * half);     // this warp's functions
            // phi of rows 64 half + .. at this thread's point, in row order: row r at
            // r 128 + its swizzled unit, the planes a chunk's bytes apart
            const uint8_t *row = ws + T.img_phi + (long long)(J * T.nc_alloc + 2 * m + (pl >> 6)) * kChunkStride +
                                 64 * half * 128 + pb;
            unsigned short w[2][8][3];
            auto load_phi = [&](int piece, unsigned short (*v)[3]) {
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    const uint8_t *src = row + piece * 1024 + row_offset(q, g16);
#pragma unroll
                    for (int sp = 0; sp < 3; sp++)
                        v[q][sp] = sp < n_split ? *reinterpret_cast<const unsigned short *>(src + sp * kChunkBytes) : 0;
                }
            };
            if (nj > 0) load_phi(0, w[0]);
            if (nj > 8) load_phi(1, w[1]);
            const bool ok = mbar_wait_a(&S->tfull[group], (lt >> 1) & 1, P.status, &S->abort);
            tc_fence_after();
            pk s2 = pk_dup(0.f), c2 = pk_dup(0.f);       // sums over even and odd j
            auto piece_sum = [&](int piece, unsigned short (*v)[3]) {
                float hi[8], lo[8];
                tmem_ld8(acc_base + 8 * piece, hi);
                if (n_split > 1) tmem_ld8(acc_base + 128 + 8 * piece, lo);
                else
#pragma unroll
                    for (int q = 0; q < 8; q++) lo[q] = 0.f;
                tmem_wait_ld();
                if (ADJ && ok) {
                    float *dst = reinterpret_cast<float *>(ws_e + T.img_e) +
                                 (long long)(J * 128 + 64 * half + 8 * piece) * T.nc_alloc * 64 + m * 128 + pl;
#pragma unroll
                    for (int q = 0; q < 8; q++)
                        if (8 * piece + q < nj) dst[(long long)q * T.nc_alloc * 64] = hi[q] + lo[q];
                }
                // E phi in double-float: e = acc0 + acc1, phi = f0 + (f1 + f2).  The inner
                // sum is never larger than a non-zero f0; its rounding, 2^-25 of f1, is
                // far below what f2 itself leaves out (2^-18 of f1).  The products are
                // summed with their errors, the low parts in FP32: about 2^-42 of the
                // terms.  Rows past n_b up to the next 16 are zero in both images.
#pragma unroll
                for (int q = 0; q < 8; q += 2) {
                    auto term = [&](int sp) {
                        return pk_make(__uint_as_float((uint32_t)v[q][sp] << 16), __uint_as_float((uint32_t)v[q + 1][sp] << 16));
                    };
                    const df2 ph = df2_fast_two_sum(term(0), term(1) + term(2));
                    const df2 e = df2_two_sum(pk_make(hi[q], hi[q + 1]), pk_make(lo[q], lo[q + 1]));
                    const pk pr = e.hi * ph.hi;
                    const pk pl2 = fma2(e.lo, ph.hi, fma2(e.hi, ph.lo, fma2(e.hi, ph.hi, -pr)));
                    const df2 t = df2_two_sum(s2, pr);
                    s2 = t.hi;
                    c2 = c2 + (t.lo + pl2);
                }
            };
#pragma unroll 1
            for (int piece = 0; 8 * piece < nj; piece += 2) {
                piece_sum(piece, w[0]);
                if (8 * (piece + 2) < nj) load_phi(piece + 2, w[0]);
                if (8 * (piece + 1) < nj) {
                    piece_sum(piece + 1, w[1]);
                    if (8 * (piece + 3) < nj) load_phi(piece + 3, w[1]);
                }
            }
            tc_fence_before();
            mbar_arrive(&S->tempty[group]);              // accumulator set may be reused
            const float2 sf = pk_get(s2), cf = pk_get(c2);
            red[group][half][pl] = ((double)sf.x + (double)sf.y) + ((double)cf.x + (double)cf.y);
            // item complete: this block's partial density at the tile's 128 points
            group_sync(group);
            if (tid == 0) mbar_arrive(&S->nempty[lt % kTiles]);
            if (tid < 128) part[T.part_row * 128 + tid] = ok ? red[group][0][tid] + red[group][1][tid] : 0.0;
            group_sync(group);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kWarpMma) tmem_dealloc(tmem, 512);
}

// n_p = 2 sum_J part[J][p] over the batch's function blocks, in J order
// (deterministic); one CTA of 128 threads per (batch, point tile).
__global__ void __launch_bounds__(128) k_density_sum(DevPlan P, const TcBatch *tb, const WorkItem *items,
                                                    const double *part, double *n_out, double factor)
{
    const WorkItem it = items[blockIdx.x];
    const DevBatch B = P.batches[it.batch];
    const TcBatch T = tb[it.batch];
    const int p = it.ti * 128 + threadIdx.x;
    if (p >= B.np) return;
    const long long nt = T.nc_alloc / 2;
    double s = 0.0;
    for (int J = 0; J < T.nrb; J++) s += part[(T.part0 + J * nt + it.ti) * 128 + threadIdx.x];
    n_out[B.pt0 + p] = factor * s;
}

// What the position gradient needs of a shell (in the species' own order) and
// of an active atom
struct AdjShell {
    int l, nk, coef_off;
    float rcut_f, inv_h;
};
struct AdjAtom {
    Dd3 pos;
    float rlim, rcut_f;                              // the species' cutoff with its margin; of the shared knots
    float inv_h;
    int nk, shared, shell0, n_shell, fn_loc, atom;
    const float4 *tab;                               // shared knots: interval 0 of the species' splines
};
constexpr int kAdjAtoms = 64;                        // staged at a time

__device__ __forceinline__ AdjShell adj_shell_entry(const DevPlan &P, int i)
{
    const DevRadial &R = P.radials[P.shell_rad[i]];
    return AdjShell{R.l, R.nk, (int)R.coef_off, R.rcut_f, R.inv_h_hi};
}

// Two points' P = r^l Y_lm and its gradient: add(m, Y_m, G_m, mask) for every m, mask the
// components of the gradient that are not zero
template <int L, class Add>
__device__ __forceinline__ void adj_angular(pk x, pk y, pk z, Add &&add)
{
    const pk no = pk_dup(0.f);
    auto g3 = [&](int m, pk Y, pk gx, pk gy, pk gz, int mask) {
        const pk G[3] = {gx, gy, gz};
        add(m, Y, G, mask);
    };
    if constexpr (L == 0) {
        g3(0, pk_dup(0.28209479177387814f), no, no, no, 0);
    } else if constexpr (L == 1) {
        const pk c = pk_dup(0.4886025119029199f);
        g3(0, c * y, no, c, no, 2);
        g3(1, c * z, no, no, c, 4);
        g3(2, c * x, c, no, no, 1);
    } else if constexpr (L == 2) {
        constexpr float fb = 0.31539156525252005f, fc = 0.5462742152960396f;
        const pk a = pk_dup(1.0925484305920792f), b = pk_dup(fb), c = pk_dup(fc);
        const pk ax = a * x, ay = a * y, az = a * z, xx = x * x, yy = y * y;
        g3(0, ax * y, ay, ax, no, 3);
        g3(1, ay * z, no, az, ay, 6);
        g3(2, b * (fma2(pk_dup(2.f) * z, z, -xx) - yy), pk_dup(-2.f * fb) * x, pk_dup(-2.f * fb) * y, pk_dup(4.f * fb) * z,
           7);
        g3(3, ax * z, az, no, ax, 5);
        g3(4, c * (xx - yy), pk_dup(2.f * fc) * x, pk_dup(-2.f * fc) * y, no, 3);
    } else {
        constexpr float f3 = 0.5900435899266435f, f2 = 2.890611442640554f, f1 = 0.4570457994644658f,
                        f0 = 0.3731763325901154f, f2b = 1.445305721320277f;
        const pk c3 = pk_dup(f3), c2 = pk_dup(f2), c1 = pk_dup(f1), c0 = pk_dup(f0), c2b = pk_dup(f2b);
        const pk xx = x * x, yy = y * y, y3 = pk_dup(3.f) * y, txx = (pk_dup(3.f) * x) * x;
        const pk fz = pk_dup(4.f) * z, zx = fma2(fz, z, -xx), q = zx - yy, dxy = xx - yy;
        const pk c2x = c2 * x;
        g3(0, (c3 * y) * (txx - yy), (pk_dup(6.f * f3) * x) * y, pk_dup(3.f * f3) * dxy, no, 3);
        g3(1, (c2x * y) * z, (c2 * y) * z, c2x * z, c2x * y, 7);
        g3(2, (c1 * y) * q, (pk_dup(-2.f * f1) * x) * y, c1 * fma2(-y3, y, zx), (pk_dup(8.f * f1) * y) * z, 7);
        g3(3, (c0 * z) * fma2(-y3, y, fma2(pk_dup(2.f) * z, z, -txx)), (pk_dup(-6.f * f0) * x) * z,
           (pk_dup(-6.f * f0) * y) * z, c0 * fma2(-y3, y, fma2(pk_dup(6.f) * z, z, -txx)), 7);
        g3(4, (c1 * x) * q, c1 * (fma2(fz, z, -txx) - yy), (pk_dup(-2.f * f1) * x) * y, (pk_dup(8.f * f1) * x) * z, 7);
        g3(5, (c2b * z) * dxy, (pk_dup(2.f * f2b) * x) * z, (pk_dup(-2.f * f2b) * y) * z, c2b * dxy, 7);
        g3(6, (c3 * x) * fma2(-y3, y, xx), pk_dup(3.f * f3) * dxy, (pk_dup(-6.f * f3) * x) * y, no, 3);
    }
}

// Two points' place in an atom's shells
struct AdjPair {
    float d[2];
    bool live[2];
    pk x, y, z, n[3], inv;
    pk t;                                            // on the species' knots: fraction of the interval
    const float4 *c[2];                              // and the interval's splines
};

// the run of shells of one l that starts at sh (SHARED: all on the species' knots
// and with its cutoff): sums over their functions of E_i grad phi_i
template <int L, bool SHARED>
__device__ __forceinline__ void adj_run(const AdjAtom &A, const AdjShell *sh_tab, const DevPlan &P, const AdjPair &q,
                                        int &sh, const float *&Erow, long long Pa, pk *gr)
{
    constexpr int NM = 2 * L + 1;
    pk ipl = q.inv;                                     // 1/d^(l+1)
#pragma unroll
    for (int i = 0; i < L; i++) ipl = ipl * q.inv;
    AdjShell R;
    if (!SHARED) R = sh_tab ? sh_tab[A.shell0 + sh] : adj_shell_entry(P, A.shell0 + sh);
    do {
        pk t = q.t, ih = pk_dup(A.inv_h);
        const float4 *c0 = q.c[0] + 2 * sh, *c1 = q.c[1] + 2 * sh;
        bool in0 = true, in1 = true;
        if (!SHARED) {
            in0 = q.live[0] && q.d[0] < R.rcut_f;
            in1 = q.live[1] && q.d[1] < R.rcut_f;
            const float a0 = q.d[0] * R.inv_h, a1 = q.d[1] * R.inv_h;
            const int k0 = in0 ? min((int)a0, R.nk - 2) : 0, k1 = in1 ? min((int)a1, R.nk - 2) : 0;
            t = pk_make(__fsub_rn(a0, (float)k0), __fsub_rn(a1, (float)k1));
            ih = pk_dup(R.inv_h);
            c0 = P.coef_dd + 2 * ((long long)R.coef_off + k0);
            c1 = P.coef_dd + 2 * ((long long)R.coef_off + k1);
        }
        const float4 a = __ldg(c0), b = __ldg(c1);
        pk e[NM];
#pragma unroll
        for (int m = 0; m < NM; m++) {
            const float2 v = __ldg(reinterpret_cast<const float2 *>(Erow + m * Pa));
            e[m] = pk_make(v.x, v.y);
        }
        Erow += NM * Pa;
        const pk w = pk_make(a.w, b.w), zc = pk_make(a.z, b.z), yc = pk_make(a.y, b.y);
        const pk u = fma2(t, fma2(t, fma2(t, w, zc), yc), pk_make(a.x, b.x));
        const pk dq = fma2(t, fma2(pk_dup(2.f), zc, (pk_dup(3.f) * t) * w), yc);
        pk g = u * ipl, gp = fma2(pk_dup(-(float)(L + 1)) * u, q.inv, dq * ih) * ipl;
        if (!SHARED) {
            const float2 gv = pk_get(g), pv = pk_get(gp);
            g = pk_make(in0 ? gv.x : 0.f, in1 ? gv.y : 0.f);
            gp = pk_make(in0 ? pv.x : 0.f, in1 ? pv.y : 0.f);
        }
        adj_angular<L>(q.x, q.y, q.z, [&](int m, pk Ym, const pk *Gm, int mask) {
            const pk am = gp * Ym;
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const pk v = (mask >> c & 1) ? fma2(am, q.n[c], g * Gm[c]) : am * q.n[c];
                gr[c] = fma2(e[m], v, gr[c]);
            }
        });
        sh++;
        if (sh == A.n_shell) break;
        R = sh_tab ? sh_tab[A.shell0 + sh] : adj_shell_entry(P, A.shell0 + sh);
    } while (R.l == L);
}

template <bool SHARED>
__device__ __forceinline__ void adj_atom(const AdjAtom &A, const AdjShell *sh_tab, const DevPlan &P, const AdjPair &q,
                                         const float *Erow, long long Pa, pk *gr)
{
    for (int sh = 0; sh < A.n_shell;) {
        switch ((sh_tab ? sh_tab[A.shell0 + sh] : adj_shell_entry(P, A.shell0 + sh)).l) {
        case 0: adj_run<0, SHARED>(A, sh_tab, P, q, sh, Erow, Pa, gr); break;
        case 1: adj_run<1, SHARED>(A, sh_tab, P, q, sh, Erow, Pa, gr); break;
        case 2: adj_run<2, SHARED>(A, sh_tab, P, q, sh, Erow, Pa, gr); break;
        default: adj_run<3, SHARED>(A, sh_tab, P, q, sh, Erow, Pa, gr); break;
        }
    }
}

// distance (x^2 and y^2 are shared with the polynomials and rounded before the sum)
__device__ __forceinline__ float adj_dist(const float3 &o)
{
    return sqrtf(fmaf(o.z, o.z, __fadd_rn(__fmul_rn(o.x, o.x), __fmul_rn(o.y, o.y))));
}

// Position gradient of the adjoint on CUDA cores (FP32): CTA per (batch,
// 64-point chunk), a warp an active atom, two neighbouring points a lane in
// packed pairs.  The lane forms sum_{i on the atom} grad phi_i(p) . E_i(p) from
// the E rows the contraction stored, times -2 w_p v_p; the warp sums each half
// of its 64 points and adds the atom's three components to dR (FP64 atomics).
//   grad phi = g'(d) (r/d) P(r) + g(d) grad P(r),  g = u/d^(l+1),
//   g' = u'/d^(l+1) - (l+1) u/d^(l+2),  P = r^l Y_lm (a polynomial in x, y, z)
// The rows of E are read once, in 256-byte pieces.  What bounds it is the
// latency of those loads: a point a lane, with the species' and shells' tables
// found through a chain of dependent look-ups a shell, took 3.1 ms where the
// atoms and shells staged in shared memory and two points a lane take 1.26
// (64-atom Si cluster, 1.11 M points; 3.1 GB of E, 0.45 ms at the measured
// copy rate); 0.38 -> 0.17 ms for a molecule of 30 atoms.  Four CTAs an SM: two
// and three are slower (1.9, 1.6 ms), and so are six (1.55); four keep 64 registers a
// thread and spill 124 bytes.
__global__ void __launch_bounds__(256, 4) k_tc_adj_grad(DevPlan P, const TcBatch *tb, const WorkItem *items,
                                                     const uint8_t *ws, const double *v, double *dR)
{
    __shared__ AdjAtom at[kAdjAtoms];
    __shared__ AdjShell shs[kMaxShellsSmem];
    const WorkItem it = items[blockIdx.x];
    const DevBatch B = P.batches[it.batch];
    const TcBatch T = tb[it.batch];
    const DevAct *act = P.act + B.act0;
    const float *E = reinterpret_cast<const float *>(ws + T.img_e);
    const long long Pa = (long long)T.nc_alloc * 64;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    const AdjShell *sh_tab = P.n_shells <= kMaxShellsSmem ? shs : nullptr;
    if (sh_tab)
        for (int i = threadIdx.x; i < P.n_shells; i += blockDim.x) shs[i] = adj_shell_entry(P, i);
    const int p = it.ti * 64 + 2 * lane;
    const bool has0 = p < B.np, has1 = p + 1 < B.np;
    const Dd3 q0 = load_dd3(P.pts_dd + 6 * (B.pt0 + (has0 ? p : 0)));
    const Dd3 q1 = load_dd3(P.pts_dd + 6 * (B.pt0 + (has1 ? p + 1 : 0)));
    const float w0 = has0 ? (float)(-2.0 * P.pw[B.pt0 + p] * v[B.pt0 + p]) : 0.f;
    const float w1 = has1 ? (float)(-2.0 * P.pw[B.pt0 + p + 1] * v[B.pt0 + p + 1]) : 0.f;
    for (int e0 = 0; e0 < B.n_act; e0 += kAdjAtoms) {
        const int ne = min(kAdjAtoms, B.n_act - e0);
        __syncthreads();
        if (threadIdx.x < ne) {
            const DevAct D = act[e0 + threadIdx.x];
            const DevSpecies &S = P.species[P.atom_species[D.atom]];
            at[threadIdx.x] = AdjAtom{load_dd3(P.atom_dd + 6 * D.atom), (float)S.rcut * 1.00001f, (float)S.rcut, S.inv_h_hi,
                                      S.nk, S.shared_grid, S.shell0, S.n_shell, D.fn_loc, D.atom,
                                      P.scoef + S.scoef_off};
        }
        __syncthreads();
        for (int e = warp; e < ne; e += nwarp) {
            const AdjAtom &A = at[e];
            const float3 o0 = offset_f32(q0, A.pos), o1 = offset_f32(q1, A.pos);
            AdjPair q;
            q.d[0] = adj_dist(o0);
            q.d[1] = adj_dist(o1);
            q.live[0] = has0 && q.d[0] > 1e-12f && q.d[0] < A.rlim;
            q.live[1] = has1 && q.d[1] > 1e-12f && q.d[1] < A.rlim;
            if (!__any_sync(0xffffffffu, q.live[0] || q.live[1])) continue;
            const float i0 = 1.f / q.d[0], i1 = 1.f / q.d[1];
            q.x = pk_make(o0.x, o1.x);
            q.y = pk_make(o0.y, o1.y);
            q.z = pk_make(o0.z, o1.z);
            q.inv = pk_make(i0, i1);
            q.n[0] = q.x * q.inv;
            q.n[1] = q.y * q.inv;
            q.n[2] = q.z * q.inv;
            const float *Erow = E + (long long)A.fn_loc * Pa + p;
            pk gr[3] = {pk_dup(0.f), pk_dup(0.f), pk_dup(0.f)};
            if (A.shared) {
                q.live[0] = q.live[0] && q.d[0] < A.rcut_f;
                q.live[1] = q.live[1] && q.d[1] < A.rcut_f;
                const float a0 = q.d[0] * A.inv_h, a1 = q.d[1] * A.inv_h;
                const int k0 = q.live[0] ? min((int)a0, A.nk - 2) : 0, k1 = q.live[1] ? min((int)a1, A.nk - 2) : 0;
                q.t = pk_make(__fsub_rn(a0, (float)k0), __fsub_rn(a1, (float)k1));
                q.c[0] = A.tab + 2ll * k0 * A.n_shell;
                q.c[1] = A.tab + 2ll * k1 * A.n_shell;
                adj_atom<true>(A, sh_tab, P, q, Erow, Pa, gr);
            } else {
                q.t = pk_dup(0.f);
                q.c[0] = q.c[1] = P.coef_dd;
                adj_atom<false>(A, sh_tab, P, q, Erow, Pa, gr);
            }
            float s0[3], s1[3];
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const float2 r = pk_get(gr[c]);
                s0[c] = q.live[0] ? r.x * w0 : 0.f;
                s1[c] = q.live[1] ? r.y * w1 : 0.f;
            }
            // sums over 32 points each: lanes 0 .. 15 hold the first half's,
            // 16 .. 31 the second's; the lanes' pairs are taken apart at the
            // first step (bit 3: the first or the second of a pair)
            const bool up = lane & 8;
            float r[3];
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const float mine = up ? s1[c] : s0[c];
                r[c] = mine + __shfl_xor_sync(0xffffffffu, up ? s0[c] : s1[c], 8);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1)
#pragma unroll
                for (int c = 0; c < 3; c++) r[c] += __shfl_xor_sync(0xffffffffu, r[c], o);
#pragma unroll
            for (int c = 0; c < 3; c++) r[c] += __shfl_xor_sync(0xffffffffu, r[c], 8);
            const int c = lane & 15;
            if (c < 3 && (r[0] != 0.f || r[1] != 0.f || r[2] != 0.f))
                atomicAdd(dR + 3 * A.atom + c, (double)(c == 0 ? r[0] : c == 1 ? r[1] : r[2]));
        }
    }
}

// Dynamic shared memory of the tcgen05 kernels: the two-stage ring (about
// 200 KB) keeps one CTA per SM, which holds all 512 tensor-memory columns.
size_t smem_tc(int n_split)
{
    (void)n_split;
    return 1024 + (size_t)kStages * kStageBytes + sizeof(TcRing);
}

size_t smem_tc_h() { return smem_tc(3) + kTiles * sizeof(HTile) + 2 * sizeof(HTables); }
static_assert(1024 + kStages * kStageBytes + sizeof(TcRing) + kTiles * sizeof(HTile) + 2 * sizeof(HTables) <= 232448,
              "the H contraction's shared memory");

bool attrs_set = false;

cudaError_t set_attrs()
{
    if (attrs_set) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_tc_h, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_tc_h());
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_tc_density<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_tc(3));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_tc_density<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_tc(3));
    if (e != cudaSuccess) return e;
    attrs_set = true;
    return cudaSuccess;
}

}  // namespace

// ==================================================================== host
// Super-batches: runs of consecutive batches of one system (the batcher
// emits spatial neighbours consecutively), merged while the points stay
// within sb_points and the union of active atoms carries at most
// sb_growth times the functions of the largest member.  Every sum of the
// method is over points, so any grouping of points gives the same H and n;
// merging cuts the per-batch scatter, D gather and tile overheads.
static void build_super_batches(TcPlan &t, const TcPlanInput &in, int sb_points, double sb_growth)
{
    t.sb.clear();
    t.sact.clear();
    t.sb_first.clear();
    std::vector<int> uni, tmp;
    int b = 0;
    while (b < in.n_batch) {
        t.sb_first.push_back(b);
        const DevBatch &B0 = in.batches[b];
        uni.clear();
        for (int e = 0; e < B0.n_act; e++) uni.push_back(in.act[B0.act0 + e].atom);
        int np = B0.np, maxfn = B0.nfn, b2 = b + 1;
        while (sb_points > 0 && b2 < in.n_batch && in.batches[b2].sys == B0.sys &&
               np + in.batches[b2].np <= sb_points) {
            const DevBatch &Bn = in.batches[b2];
            tmp.clear();
            size_t i = 0;
            int e = 0;
            while (i < uni.size() || e < Bn.n_act) {
                const int a = e < Bn.n_act ? in.act[Bn.act0 + e].atom : 1 << 30;
                const int u = i < uni.size() ? uni[i] : 1 << 30;
                if (u == a) { tmp.push_back(u); i++; e++; }
                else if (u < a) { tmp.push_back(u); i++; }
                else { tmp.push_back(a); e++; }
            }
            long long nfn = 0;
            for (int a : tmp) nfn += in.atom_nfn[a];
            const int mx = std::max(maxfn, Bn.nfn);
            if (nfn > sb_growth * mx || nfn > kMaxBatchFns) break;
            uni.swap(tmp);
            np += Bn.np;
            maxfn = mx;
            b2++;
        }
        DevBatch S{};
        S.pt0 = B0.pt0;
        S.np = np;
        S.sys = B0.sys;
        S.act0 = (int)t.sact.size();
        S.n_act = (int)uni.size();
        int fl = 0;
        for (int a : uni) {
            t.sact.push_back(DevAct{a, fl});
            fl += in.atom_nfn[a];
        }
        S.nfn = fl;
        t.sb.push_back(S);
        b = b2;
    }
    t.sb_first.push_back(in.n_batch);
}

int tc_build(TcPlan &t, const TcPlanInput &in, std::string *err)
{
    tc_free(t);
    build_super_batches(t, in, std::min(in.sb_points, kMaxBatchPoints), std::max(1.0, in.sb_growth));
    const int n_sb = (int)t.sb.size();
    t.batches.assign(n_sb, TcBatch{});
    t.sb_rank.assign(n_sb, -1);
    t.items.clear();
    t.waves.clear();
    size_t cap = (size_t)24 << 30;   // workloads up to ~24 GB of operand images run as one wave
    if (in.wave_mb > 0) cap = (size_t)in.wave_mb << 20;
    if (const char *e = getenv("FGI_TC_WAVE_MB")) cap = (size_t)std::max(1L, atol(e)) << 20;
    t.wave_cap = cap;
    // per-batch image geometry and footprint (3 planes always reserved)
    std::vector<size_t> foot(n_sb, 0);
    for (int b = 0; b < n_sb; b++) {
        const DevBatch &B = t.sb[b];
        TcBatch &T = t.batches[b];
        T.nrb = (B.nfn + 127) / 128;
        T.nc = (B.np + 63) / 64;
        T.nc_alloc = (T.nc + 1) / 2 * 2;
        T.nkc = (B.nfn + 63) / 64;
        T.plane_phi = (long long)T.nrb * T.nc_alloc * kChunkBytes;
        T.plane_d = (long long)T.nrb * T.nkc * kChunkBytes;
        foot[b] = 3 * (size_t)T.plane_phi + 3 * (size_t)std::max(T.plane_phi, T.plane_d);
        T.hblock = T.hgrid = T.hscale = -1;
        T.img_e = -1;
        if (in.with_e) foot[b] += 2 * (size_t)T.plane_phi;     // E in FP32: twice a BF16 plane
    }
    t.bound_grids = in.bound_grids;
    size_t max_ws = 0, max_all = 0;
    TcWave w;
    size_t off = 0;
    auto close_wave = [&](int b_end) {
        w.nb = b_end - w.b0;
        if (w.nb <= 0) return;
        max_ws = std::max(max_ws, off);
        t.waves.push_back(w);
    };
    // each wave: the batches' images, then their partial densities (one row
    // of 128 doubles per (point tile, function block))
    long long part = 0;
    auto part_rows = [&](int b) { return (long long)(t.batches[b].nc_alloc / 2) * t.batches[b].nrb; };
    // H: the row blocks' descriptors and grids and the points' scales of a batch
    // go behind its two images where the room for D is larger, else to the end
    // of the wave (at most 2.6 % of the images), outside the wave's budget
    std::vector<int> at_end;
    auto desc_bytes = [&](const TcBatch &T) {
        return ((size_t)T.nrb * (sizeof(HBlock) + sizeof(HGrid)) + (size_t)T.nc * 512 + 1023) / 1024 * 1024;
    };
    auto place_desc = [&](TcBatch &T, size_t at) {
        T.hblock = (long long)at;
        T.hgrid = T.hblock + (long long)T.nrb * (long long)sizeof(HBlock);
        T.hscale = T.hgrid + (long long)T.nrb * (long long)sizeof(HGrid);
    };
    auto finish_wave = [&](int b_end) {
        w.part_off = (off + 1023) / 1024 * 1024;
        off = w.part_off + (size_t)part * 128 * sizeof(double);
        close_wave(b_end);
        size_t at = (off + 1023) / 1024 * 1024;
        for (int b : at_end) {
            place_desc(t.batches[b], at);
            at += desc_bytes(t.batches[b]);
        }
        max_all = std::max(max_all, at_end.empty() ? off : at);
        at_end.clear();
    };
    for (int b = 0; b < n_sb; b++) {
        const size_t pb = (size_t)part_rows(b) * 128 * sizeof(double);
        if (b > w.b0 && off + foot[b] + pb + (size_t)part * 1024 + 1024 > cap) {
            finish_wave(b);
            w = TcWave{};
            w.b0 = b;
            off = 0;
            part = 0;
        }
        TcBatch &T = t.batches[b];
        T.img_phi = (long long)off;
        T.img_aux = (long long)(off + 3 * (size_t)T.plane_phi);
        if (in.for_h) {
            if (6 * (size_t)T.plane_phi + desc_bytes(T) <= foot[b]) place_desc(T, off + 6 * (size_t)T.plane_phi);
            else at_end.push_back(b);
        }
        if (in.with_e) T.img_e = (long long)(off + 3 * (size_t)T.plane_phi + 3 * (size_t)std::max(T.plane_phi, T.plane_d));
        T.part0 = part;
        part += part_rows(b);
        off += foot[b];
    }
    finish_wave(n_sb);
    {
        size_t n_items = 0;   // the six lists below, for one allocation
        for (int b = 0; b < n_sb; b++) {
            if (t.sb[b].np <= 0 || t.sb[b].nfn <= 0) continue;
            const size_t nrb = (size_t)t.batches[b].nrb, nca = (size_t)t.batches[b].nc_alloc;
            n_items += 2 * nrb + nrb * (nrb + 1) / 2 + nca + nca / 2 + nrb * (nca / 2);
        }
        t.items.reserve(n_items);
    }
    for (TcWave &wv : t.waves) {
        // longest first: the wave's batches by contraction cost P n^2, each
        // batch's items kept together (they share image tiles in L2); the
        // persistent kernels take them in this order, so the small items land last
        std::vector<int> ord;
        for (int b = wv.b0; b < wv.b0 + wv.nb; b++)
            if (t.sb[b].np > 0 && t.sb[b].nfn > 0) ord.push_back(b);
        auto cost = [&](int b) { return (double)t.sb[b].np * t.sb[b].nfn * t.sb[b].nfn; };
        std::stable_sort(ord.begin(), ord.end(), [&](int a, int b) { return cost(a) > cost(b); });
        for (size_t r = 0; r < ord.size(); r++) t.sb_rank[ord[r]] = (int)r;
        wv.phi0 = (long long)t.items.size();
        for (int b : ord)
            for (int I = 0; I < t.batches[b].nrb; I++) t.items.push_back(WorkItem{b, (short)I, 0});
        wv.nphi = (long long)t.items.size() - wv.phi0;
        wv.h0 = (long long)t.items.size();
        for (int b : ord)
            for (int I = 0; I < t.batches[b].nrb; I++)
                for (int J = I; J < t.batches[b].nrb; J++) t.items.push_back(WorkItem{b, (short)I, (short)J});
        wv.nh = (long long)t.items.size() - wv.h0;
        wv.g0 = (long long)t.items.size();
        for (int b : ord)
            for (int J = 0; J < t.batches[b].nrb; J++) t.items.push_back(WorkItem{b, (short)J, 0});
        wv.ng = (long long)t.items.size() - wv.g0;
        wv.pc0 = (long long)t.items.size();
        for (int b : ord)
            for (int c = 0; c < t.batches[b].nc; c++) t.items.push_back(WorkItem{b, (short)c, 0});
        wv.npc = (long long)t.items.size() - wv.pc0;
        wv.d0 = (long long)t.items.size();
        for (int b : ord)
            for (int mt = 0; mt < t.batches[b].nc_alloc / 2; mt++) t.items.push_back(WorkItem{b, (short)mt, 0});
        wv.nd = (long long)t.items.size() - wv.d0;
        // MMA items: J ascending (the longest contractions first), every point tile
        wv.e0 = (long long)t.items.size();
        for (int b : ord)
            for (int J = 0; J < t.batches[b].nrb; J++)
                for (int mt = 0; mt < t.batches[b].nc_alloc / 2; mt++)
                    t.items.push_back(WorkItem{b, (short)mt, (short)J});
        wv.ne = (long long)t.items.size() - wv.e0;
        for (int b = wv.b0; b < wv.b0 + wv.nb; b++) {
            const double P = t.sb[b].np, n = t.sb[b].nfn;
            wv.phi_flops += 30.0 * P * n;
            wv.phi_bytes += 32.0 * P + 12.0 * P * n;
            wv.h_flops += P * n * (n + 1.0);
            wv.h_bytes += 16.0 * n * (n + 1) / 2 + 12.0 * P * n;
            // symmetric D: the upper block triangle (about half of n^2)
            wv.n_flops += P * n * (n + 1.0) + 2.0 * P * n;
            wv.n_bytes += 3.0 * n * n + 6.0 * P * n + 16.0 * P;
            wv.g_bytes += 7.0 * n * n;
        }
    }
    // scratch before the images: the fixed-point H accumulator, or the
    // double-float copy of D followed by the per-function bounds of D
    t.nnz = in.nnz;
    t.n_fn = in.n_fn;
    t.bound_off = ((size_t)in.nnz * 8 + 255) / 256 * 256;
    t.sign_off = (t.bound_off + 8 * (size_t)in.n_fn + 255) / 256 * 256;
    // the contraction's tile counter in scratch of the other call: H has no bounds
    // of D, the density no signs of w v
    t.counter_off = in.for_h ? t.bound_off : t.sign_off;
    t.img_base = (t.sign_off + 4 * (size_t)n_sb + 1023) / 1024 * 1024;
    t.ws_images = t.img_base + max_ws + 1024;
    t.ws_bytes = t.img_base + std::max(max_ws, max_all) + 1024;
    // items must not be empty for the device copy
    if (!in.host_only) {
        const size_t nb_bytes = t.batches.size() * sizeof(TcBatch);
        const size_t ni_bytes = t.items.size() * sizeof(WorkItem);
        const size_t sb_bytes = t.sb.size() * sizeof(DevBatch);
        const size_t sa_bytes = t.sact.size() * sizeof(DevAct);
        auto al = [](size_t x) { return (x + 255) / 256 * 256; };
        const size_t tot = al(nb_bytes) + al(ni_bytes) + al(sb_bytes) + al(sa_bytes) + 256;
        cudaError_t e = cudaMalloc(&t.d_mem, tot);
        if (e != cudaSuccess) {
            t.d_mem = nullptr;
            *err = std::string("tensor-core plan: cudaMalloc failed: ") + cudaGetErrorString(e);
            return FGI_ERR_NOMEM;
        }
        char *base = (char *)t.d_mem;
        if (nb_bytes) cudaMemcpy(base, t.batches.data(), nb_bytes, cudaMemcpyHostToDevice);
        const size_t ioff = ((nb_bytes + 255) / 256) * 256;
        if (ni_bytes) cudaMemcpy(base + ioff, t.items.data(), ni_bytes, cudaMemcpyHostToDevice);
        t.d_batches = (const TcBatch *)base;
        t.d_items = (const WorkItem *)(base + ioff);
        const size_t soff = ioff + al(ni_bytes), aoff = soff + al(sb_bytes);
        if (sb_bytes) cudaMemcpy(base + soff, t.sb.data(), sb_bytes, cudaMemcpyHostToDevice);
        if (sa_bytes) cudaMemcpy(base + aoff, t.sact.data(), sa_bytes, cudaMemcpyHostToDevice);
        t.d_sb = (const DevBatch *)(base + soff);
        t.d_sact = (const DevAct *)(base + aoff);
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&t.num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (t.num_sms <= 0) t.num_sms = 1;
        e = set_attrs();
        if (e != cudaSuccess) {
            *err = std::string("tensor-core plan: cudaFuncSetAttribute: ") + cudaGetErrorString(e);
            return FGI_ERR_CUDA;
        }
    }
    t.built = true;
    return FGI_OK;
}

void tc_free(TcPlan &t)
{
    if (t.d_mem) cudaFree(t.d_mem);
    t.d_mem = nullptr;
    t.d_batches = nullptr;
    t.d_items = nullptr;
    t.built = false;
}

size_t tc_workspace_bytes(const TcPlan &t) { return t.ws_bytes; }

cudaError_t tc_launch_phi(const TcPlan &t, const DevPlan &P, const TcWave &w, const double *v, void *ws,
                          int n_split, cudaStream_t s)
{
    if (w.nphi <= 0) return cudaSuccess;
    const int fixed = n_split == 3 ? 1 : 0;             // the split mode's fixed-point leading term
    uint8_t *img = (uint8_t *)ws + t.img_base;
    int *bsign = reinterpret_cast<int *>((uint8_t *)ws + t.sign_off);
    k_h_prep<<<(unsigned)w.nb, kPhiThreads, 0, s>>>(P, t.d_batches, w.b0, img, v, fixed, t.bound_grids >= 2 ? 1 : 0,
                                                    bsign, reinterpret_cast<unsigned int *>((uint8_t *)ws + t.counter_off));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_tc_phi<<<(unsigned)w.nphi, kPhiThreads, 0, s>>>(P, t.d_batches, t.d_items + w.phi0, img, fixed, bsign);
    return cudaGetLastError();
}

cudaError_t tc_launch_phi_cols(const TcPlan &t, const DevPlan &P, const TcWave &w, void *ws, int n_split,
                               cudaStream_t s)
{
    if (w.npc <= 0) return cudaSuccess;
    k_tc_phi_cols<<<(unsigned)w.npc, kPhiThreads, 0, s>>>(P, t.d_batches, t.d_items + w.pc0,
                                                           (uint8_t *)ws + t.img_base, n_split,
                                                           t.bound_grids >= 1 ? 1 : 0,
                                                           reinterpret_cast<unsigned int *>((uint8_t *)ws + t.counter_off));
    return cudaGetLastError();
}

cudaError_t tc_launch_h(const TcPlan &t, const DevPlan &P, const TcWave &w, const void *ws, int n_split,
                        cudaStream_t s)
{
    if (w.nh <= 0) return cudaSuccess;
    const int grid = (int)std::min<long long>(w.nh, t.num_sms);
    k_tc_h<<<grid, kThreadsTc, smem_tc_h(), s>>>(P, t.d_batches, t.d_items + w.h0, (int)w.nh,
                                                (const uint8_t *)ws + t.img_base, (unsigned long long *)ws, n_split,
                                                reinterpret_cast<const int *>((const uint8_t *)ws + t.sign_off),
                                                (unsigned int *)((const uint8_t *)ws + t.counter_off));
    return cudaGetLastError();
}

cudaError_t tc_launch_fix_to_h(const TcPlan &t, const void *ws, double *h, long long nnz, int accumulate,
                               cudaStream_t s)
{
    (void)t;
    if (nnz <= 0) return cudaSuccess;
    k_fix_to_h<<<1216, 256, 0, s>>>((const long long *)ws, h, nnz, accumulate);
    return cudaGetLastError();
}

cudaError_t tc_launch_gather_d(const TcPlan &t, const DevPlan &P, const TcWave &w, double offdiag_scale,
                               void *ws, int n_split, cudaStream_t s, bool full)
{
    if (w.ng <= 0) return cudaSuccess;
    const char *base = (const char *)ws;
    auto kernel = n_split == 3 ? k_tc_gather_d<3> : k_tc_gather_d<1>;
    kernel<<<(unsigned)w.ng, 256, 0, s>>>(P, t.d_batches, t.d_items + w.g0, (uint8_t *)ws + t.img_base,
                                          (const float2 *)base, (const unsigned int *)(base + t.bound_off),
                                          (const float *)(base + t.bound_off + 4 * t.n_fn), (float)offdiag_scale,
                                          full ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t tc_launch_to_df(const TcPlan &t, const DevPlan &P, const double *x, void *ws, const long long *sys_val0,
                            const long long *sys_nnz, const int *fn_sys, cudaStream_t s)
{
    if (t.nnz <= 0) return cudaSuccess;
    char *base = (char *)ws;
    unsigned int *gmax = (unsigned int *)(base + t.bound_off);
    float *gsum = (float *)(base + t.bound_off + 4 * t.n_fn);
    cudaError_t e = cudaMemsetAsync(gmax, 0, 8 * (size_t)t.n_fn, s);
    if (e != cudaSuccess) return e;
    k_to_df<<<1216, 256, 0, s>>>(x, (float2 *)base, P.rowptr, fn_sys, sys_val0, sys_nnz, t.n_fn, gmax, gsum);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_d_colbounds<<<1216, 256, 0, s>>>((const float2 *)base, P.col_glob, t.nnz, gmax, gsum);
    return cudaGetLastError();
}

cudaError_t tc_launch_density(const TcPlan &t, const DevPlan &P, const TcWave &w, const void *ws, double *n,
                              int n_split, cudaStream_t s)
{
    if (w.nd <= 0) return cudaSuccess;
    double *part = reinterpret_cast<double *>((uint8_t *)const_cast<void *>(ws) + t.img_base + w.part_off);
    const int grid = (int)std::min<long long>(w.ne, t.num_sms);
    k_tc_density<false><<<grid, kThreadsTc, smem_tc(3), s>>>(P, t.d_batches, t.d_items + w.e0, (int)w.ne,
                                                             (const uint8_t *)ws + t.img_base, part, n_split,
                                                             nullptr,
                                                             (unsigned int *)((const uint8_t *)ws + t.counter_off));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_density_sum<<<(unsigned)w.nd, 128, 0, s>>>(P, t.d_batches, t.d_items + w.d0, part, n, 2.0);
    return cudaGetLastError();
}

cudaError_t tc_launch_adjoint(const TcPlan &t, const DevPlan &P, const TcWave &w, const void *ws, const double *v,
                              double *dv, double *dR, int n_split, cudaStream_t s)
{
    if (w.nd <= 0) return cudaSuccess;
    if (!t.batches.empty() && t.batches[w.b0].img_e < 0) return cudaErrorInvalidValue;   // no room for E
    uint8_t *img = (uint8_t *)const_cast<void *>(ws) + t.img_base;
    double *part = reinterpret_cast<double *>(img + w.part_off);
    const int grid = (int)std::min<long long>(w.ne, t.num_sms);
    k_tc_density<true><<<grid, kThreadsTc, smem_tc(3), s>>>(P, t.d_batches, t.d_items + w.e0, (int)w.ne, img, part,
                                                            n_split, img,
                                                            (unsigned int *)((const uint8_t *)ws + t.counter_off));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_density_sum<<<(unsigned)w.nd, 128, 0, s>>>(P, t.d_batches, t.d_items + w.d0, part, dv, 1.0);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_tc_adj_grad<<<(unsigned)w.npc, 256, 0, s>>>(P, t.d_batches, t.d_items + w.pc0, img, v, dR);
    return cudaGetLastError();
}

// Self-test of the failure path: one CTA waits on an mbarrier that nothing
// completes.  The bounded wait gives up after kWaitLimitNs and records the
// time-out in the status word, as a stalled pipeline would; no fault, no hang.
// Then a copy is started and drained with the abort flag set, as a role does that leaves
// after a time-out; if the drain gives up, the status becomes another error.
__device__ __align__(128) unsigned char g_selftest_src[kChunkBytes];

__global__ void k_wait_selftest(int *status)
{
    __shared__ __align__(128) unsigned char dst[kChunkBytes];
    __shared__ uint64_t bar, copied;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_init(&copied, 1);
        abort_flag = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        mbar_wait_a(&bar, 0, status, &abort_flag);
        mbar_expect_tx(&copied, kChunkBytes);
        bulk_g2s(dst, g_selftest_src, kChunkBytes, &copied);
        if (!mbar_drain(&copied, 0)) atomicExch(status, kStatusBadIndex);
    }
}

cudaError_t tc_launch_wait_selftest(int *status, cudaStream_t s)
{
    k_wait_selftest<<<1, 32, 0, s>>>(status);
    return cudaGetLastError();
}

}  // namespace fgi
