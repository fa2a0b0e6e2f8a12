// Fused smoothing-proximal-gradient iteration for sm_103a: one launch runs
// `niter` iterations for every volume of a context.
//
// Per voxel v the launch computes, from x_k, d_k = x_k - x_{k-1}, b, w, om1,
// omtv (Sec. 2.1 Eq. 12, 16, 17, 20, 21; Sec. 2.2 Eq. 28 data term):
//   (Dy)_a = [v_a >= 1] ((x_k[v] - x_k[v-e_a]) + beta (d[v] - d[v-e_a]))       Eq. 12 on y
//   p_a    = omtv_v (Dy)_a / max(mu, |Dy_v|)                                   Eq. 16, weighted
//   div    = sum_a p_a[v] - p_a[v+e_a]                                          Eq. 17
//   g      = w ((x_k - b) + beta d) + lambda_tv div                             grad f(y)
//   delta  = beta d - tau g,  z = x_k + delta                                   Eq. 20
//   x_{k+1} = 0 if |z| < t else x_k + (delta - t sign z),  t = tau lambda_l1 om1   Eq. 21
// and, when the step is recorded, the three sums of F(x_k) (data, l1, TV).
//
// y = x_k + beta d is never rounded on its own: differences and the data
// residual are formed from x_k and d separately, and the update is added to
// x_k once, so each iteration commits a single float32 rounding per voxel.
// Two storage forms of the extrapolation pair (template flag XD):
//  - XD = false: x_k and x_{k-1} are stored (three rotating buffers) and
//    d = x_k - x_{k-1} is formed in registers;
//  - XD = true: x_k and the increment d_k are stored (two ping-pong pairs);
//    the kernel writes x_{k+1} = x_k + inc and d_{k+1} = inc, where inc is
//    the float32 increment before it is added to x_k. The momentum term then
//    never sees the rounding of x, which keeps a float32 solve within ~1e-6
//    of exact arithmetic at the cost of one more 4-byte write per voxel.
//
// Data movement: a CTA owns an x-y tile (TX = 32*VX by TY voxels) and marches
// over z. Each z-step's inputs arrive by TMA (cp.async.bulk.tensor) into one
// of S shared-memory stages, tracked by an mbarrier: x_k and x_{k-1} (or d_k) with a
// one-voxel x-y halo (the box starts 4 elements left of the tile so the
// innermost coordinate stays 16-byte aligned), omtv with a +1 halo, and b, w,
// om1 of the plane being written. Plane z's p is computed while plane z-1 is
// written, so each voxel's inputs are read from HBM once per iteration; the
// halo rows come from L2 because neighbouring tiles march the same planes at
// the same time. Warp r of TY computes row r; one extra warp computes the +y
// halo row and the +x halo column. p_y crosses warps through a 3-deep shared
// ring, p_x through a lane shuffle; p_z and the z-1 values stay in registers.
//
// Several iterations per launch (niter > 1, a cooperative launch): the
// iterations are separated by a barrier over the grid's CTAs instead of a
// kernel boundary. A launch per iteration paid, on the critical path of a
// small volume, launch latency, a chain of five dependent loads (device state,
// schedule, item, descriptor, extrapolation weight) before the first copy
// could start, and the last CTA's objective sums and state update before the
// next launch could read the state. Here the schedule's items are held in
// shared memory, the extrapolation index is counted, and the objective partials of
// every iteration are kept ([niter][nitems]) and reduced after the last one
// by all CTAs together (a warp per iteration and volume). The copies of an
// item's first planes are issued while the previous item's last ones are
// computed, and of an iteration's first planes those that no iteration writes
// before the barrier. An iteration with the objective, one per launch
// (replayed from a graph) -> many per launch -> items in shared memory (the
// barrier drops L1, and the chain schedule, item, descriptor from L2 delayed
// the first copies) and copies before the barrier -> missing neighbours by
// address (16 selects fewer among 360 instructions of a 4-voxel plane step),
// same tiles but for the first: 28 x 32 x 40 9.7 -> 5.4 -> 5.1 -> 4.8 us, 64^3 11.3
// -> 7.6 -> 7.0 -> 6.9, 128^3 18.6 -> 14.1 -> 13.5 -> 13.2, 101 x 147 x 183 30.7 ->
// 20.8 -> 20.0 -> 19.8, 180^3 57.6 -> 43.3 -> 41.3 -> 40.4, 256^3 86.8 -> 81.5 ->
// 79.7 -> 78.7, 512^3 618.4 -> 617.2 -> 614.1 -> 606.6; 24 volumes of 96^3 .. 256^3
// (the last three) 777 -> 767 -> 755. These are of launches of up to 10 ms; with
// the 2 ms that a launch may take (for other contexts' sake, spg_api.cu) the
// longest iterations take 0.6-0.9 % more. (With the producer's position in shared memory instead of
// the item's registers the long marches lost: 623.6 at 512^3, 1128 for the
// batch: its warp is the last to arrive at every plane's barrier.)
#pragma once

#include <cuda_bf16.h>

#include "spg_ff.cuh"
#include "spg_internal.h"

namespace spg {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int kItemCache = 16;  // work items of a CTA held in its shared memory

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, int count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ long long global_ns()
{
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait: false when `limit_ns` passed without the phase completing.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, long long limit_ns)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = global_ns();
    for (;;) {
        for (int i = 0; i < 32; i++)
            if (mbar_try_wait(bar, parity)) return true;
        if (global_ns() - t0 > limit_ns) return false;
    }
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int x, int y, int z,
                                            uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// Index checks of the checked build (compiled with -DSPG_CHECK, in place of
// a memory checker): SPG_GUARD(st, cond, code) is `true` in the production
// build; in the checked build a false `cond` records SPG_ECHECK and `code` in
// the device state and the guarded access is skipped.
#ifdef SPG_CHECK
__device__ __noinline__ void check_failed(DevState *st, unsigned code)
{
    atomicCAS(&st->err, 0, (int)SPG_ECHECK);
    atomicCAS(&st->err_info, 0u, code);
}
#define SPG_GUARD(st, cond, code) ((cond) ? true : (::spg::check_failed((st), (code)), false))
#else
#define SPG_GUARD(st, cond, code) true
#endif

// Compensated float32 accumulator (Kahan): per-thread objective sums.
struct KSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v)
    {
        float y = v - c;
        float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ ff::FF value() const { return {s, -c}; }
};

// Packed float32 pairs (sm_100 and later issue one instruction for two
// lanes' worth of add, multiply or fused multiply-add). Each lane rounds to
// nearest exactly as the scalar operation does, so the results are bitwise
// those of the scalar code; only the issue slots are halved.
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b rounded once: the product b * (-1) is exact
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// Barrier of the TY row warps (named barrier 1; the halo warp takes no part).
template <int TY>
__device__ __forceinline__ void row_warps_sync()
{
    asm volatile("bar.sync 1, %0;" ::"n"(32 * TY) : "memory");
}

// Two compensated (Kahan) float32 accumulators advanced together.
struct KSum2 {
    float2 s = make_float2(0.f, 0.f), c = make_float2(0.f, 0.f);
    __device__ __forceinline__ void add(float2 v)
    {
        const float2 y = sub2(v, c);
        const float2 t = add2(s, y);
        c = sub2(sub2(t, s), y);
        s = t;
    }
    __device__ __forceinline__ ff::FF value_x() const { return {s.x, -c.x}; }
    __device__ __forceinline__ ff::FF value_y() const { return {s.y, -c.y}; }
};

// Phase A of one z-step at a thread's VX voxels of plane z: the weighted
// clipped gradient p = omtv (Dy) / max(mu, |Dy|) (Eq. 12, 16) and, with REC,
// the weighted smoothed norm omtv h_mu(D x_k) (Eq. 14) summed into *tsum.
// xl, ld: x_k and d at the voxel left of the first one; xu, du: the row
// above; xz, dz: the plane below. Pairs of voxels go through the packed
// operations; the differences along x (operands one register apart) stay
// scalar.
template <int VX, bool REC>
__device__ __forceinline__ void phase_a(const float (&xc)[VX], const float (&dc)[VX], const float (&xu)[VX],
                                        const float (&du)[VX], const float (&xz)[VX], const float (&dz)[VX],
                                        const float (&om)[VX], float xl, float ld, float beta, float inv_mu,
                                        float half_inv_mu, float half_mu, float mu2, float (&pc)[3][VX],
                                        float *tsum)
{
    if constexpr (VX % 2 == 0) {
        float ex[VX], exd[VX];
#pragma unroll
        for (int i = 0; i < VX; i++) {
            ex[i] = xc[i] - (i ? xc[i - 1] : xl);
            exd[i] = dc[i] - (i ? dc[i - 1] : ld);
        }
        const float2 B = dup2(beta);
        float2 ts = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < VX / 2; q++) {
            const int i = 2 * q;
            const float2 X = make_float2(xc[i], xc[i + 1]), D = make_float2(dc[i], dc[i + 1]);
            const float2 EX = make_float2(ex[i], ex[i + 1]);
            const float2 EY = sub2(X, make_float2(xu[i], xu[i + 1]));
            const float2 EZ = sub2(X, make_float2(xz[i], xz[i + 1]));
            const float2 AX = fma2(B, make_float2(exd[i], exd[i + 1]), EX);
            const float2 AY = fma2(B, sub2(D, make_float2(du[i], du[i + 1])), EY);
            const float2 AZ = fma2(B, sub2(D, make_float2(dz[i], dz[i + 1])), EZ);
            const float2 S2 = fma2(AX, AX, fma2(AY, AY, mul2(AZ, AZ)));
            const float2 SC = mul2(make_float2(om[i], om[i + 1]),
                                   make_float2(fminf(inv_mu, rsqrtf(S2.x)), fminf(inv_mu, rsqrtf(S2.y))));
            const float2 P0 = mul2(AX, SC), P1 = mul2(AY, SC), P2 = mul2(AZ, SC);
            pc[0][i] = P0.x; pc[0][i + 1] = P0.y;
            pc[1][i] = P1.x; pc[1][i + 1] = P1.y;
            pc[2][i] = P2.x; pc[2][i + 1] = P2.y;
            if constexpr (REC) {
                const float2 Q = fma2(EX, EX, fma2(EY, EY, mul2(EZ, EZ)));
                const float2 HQ = mul2(Q, dup2(half_inv_mu));
                const float2 HL = fma2(Q, make_float2(rsqrtf(Q.x), rsqrtf(Q.y)), dup2(-half_mu));
                const float2 H = make_float2(Q.x <= mu2 ? HQ.x : HL.x, Q.y <= mu2 ? HQ.y : HL.y);
                ts = fma2(make_float2(om[i], om[i + 1]), H, ts);
            }
        }
        if constexpr (REC) *tsum = ts.x + ts.y;
    } else {
        float t = 0.f;
#pragma unroll
        for (int i = 0; i < VX; i++) {
            const float lx = i ? xc[i - 1] : xl;
            const float l_d = i ? dc[i - 1] : ld;
            const float ex = xc[i] - lx, ey = xc[i] - xu[i], ez = xc[i] - xz[i];
            const float ax = fmaf(beta, dc[i] - l_d, ex);
            const float ay = fmaf(beta, dc[i] - du[i], ey);
            const float az = fmaf(beta, dc[i] - dz[i], ez);
            const float s2 = fmaf(ax, ax, fmaf(ay, ay, az * az));
            const float sc = om[i] * fminf(inv_mu, rsqrtf(s2));
            pc[0][i] = ax * sc;
            pc[1][i] = ay * sc;
            pc[2][i] = az * sc;
            if constexpr (REC) {
                const float q = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
                const float h = q <= mu2 ? q * half_inv_mu : fmaf(q, rsqrtf(q), -half_mu);
                t = fmaf(om[i], h, t);
            }
        }
        if constexpr (REC) *tsum = t;
    }
}

// Phase B at a thread's VX voxels of plane z-1: divergence (Eq. 17), data
// gradient, gradient step and weighted soft-threshold (Eq. 20-21). Writes the
// new iterate `out` and the increment `inc`; with REC adds the data and l1
// terms of F(x_k) into dl (x: data, y: l1), with DOT the restart product
// (y - x+).(x+ - x) into *rsum. pxr: p_x of the voxel right of the last one.
template <int VX, bool REC, bool DOT, bool FOURIER>
__device__ __forceinline__ void phase_b(const float (&pp)[3][VX], float pxn, const float (&pyd)[VX],
                                        const float (&pz)[VX], const float (&xz)[VX], const float (&dz)[VX],
                                        const float (&bb)[VX], const float (&ww)[VX], const float (&oo)[VX],
                                        float beta, float tau, float lam_tv, float tl1, float (&out)[VX],
                                        float (&inc)[VX], float2 *dl, float *rsum)
{
    if constexpr (VX % 2 == 0) {
        float dxx[VX];
#pragma unroll
        for (int i = 0; i < VX; i++) dxx[i] = pp[0][i] - (i < VX - 1 ? pp[0][i + 1] : pxn);
        const float2 B = dup2(beta), NT = dup2(-tau), LT = dup2(lam_tv), TL = dup2(tl1);
        float2 d2 = make_float2(0.f, 0.f), l2 = make_float2(0.f, 0.f);
        float r = 0.f;
#pragma unroll
        for (int q = 0; q < VX / 2; q++) {
            const int i = 2 * q;
            const float2 XZ = make_float2(xz[i], xz[i + 1]), DZ = make_float2(dz[i], dz[i + 1]);
            const float2 DIV = add2(add2(make_float2(dxx[i], dxx[i + 1]),
                                         sub2(make_float2(pp[1][i], pp[1][i + 1]), make_float2(pyd[i], pyd[i + 1]))),
                                    sub2(make_float2(pp[2][i], pp[2][i + 1]), make_float2(pz[i], pz[i + 1])));
            const float2 BB = make_float2(bb[i], bb[i + 1]);
            const float2 RES = sub2(XZ, BB);
            const float2 GD = FOURIER ? BB : mul2(make_float2(ww[i], ww[i + 1]), fma2(B, DZ, RES));
            const float2 G = fma2(LT, DIV, GD);
            const float2 DL = fma2(B, DZ, mul2(NT, G));
            const float2 ZZ = add2(XZ, DL);
            const float2 T = mul2(TL, make_float2(oo[i], oo[i + 1]));
            const float2 CS = make_float2(copysignf(T.x, ZZ.x), copysignf(T.y, ZZ.y));
            const float2 IN0 = sub2(DL, CS);
            const float2 IN = make_float2(fabsf(ZZ.x) < T.x ? -XZ.x : IN0.x, fabsf(ZZ.y) < T.y ? -XZ.y : IN0.y);
            const float2 OUT = add2(XZ, IN);
            out[i] = OUT.x; out[i + 1] = OUT.y;
            inc[i] = IN.x; inc[i + 1] = IN.y;
            if constexpr (DOT) {
                r = fmaf(fmaf(beta, DZ.x, -IN.x), IN.x, r);
                r = fmaf(fmaf(beta, DZ.y, -IN.y), IN.y, r);
            }
            if constexpr (REC) {
                if constexpr (!FOURIER) d2 = fma2(mul2(make_float2(ww[i], ww[i + 1]), RES), RES, d2);
                l2 = fma2(make_float2(oo[i], oo[i + 1]), make_float2(fabsf(XZ.x), fabsf(XZ.y)), l2);
            }
        }
        if constexpr (REC) *dl = make_float2(d2.x + d2.y, l2.x + l2.y);
        if constexpr (DOT) *rsum = r;
    } else {
        float dsum = 0.f, lsum = 0.f, r = 0.f;
#pragma unroll
        for (int i = 0; i < VX; i++) {
            const float pxr = (i < VX - 1) ? pp[0][i + 1] : pxn;
            const float div = (pp[0][i] - pxr) + (pp[1][i] - pyd[i]) + (pp[2][i] - pz[i]);
            const float res = xz[i] - bb[i];
            const float gdat = FOURIER ? bb[i] : ww[i] * fmaf(beta, dz[i], res);
            const float g = fmaf(lam_tv, div, gdat);
            const float delta = fmaf(beta, dz[i], -tau * g);
            const float zz = xz[i] + delta;
            const float t = tl1 * oo[i];
            inc[i] = fabsf(zz) < t ? -xz[i] : delta - copysignf(t, zz);
            out[i] = xz[i] + inc[i];
            if constexpr (DOT) r = fmaf(fmaf(beta, dz[i], -inc[i]), inc[i], r);
            if constexpr (REC) {
                if constexpr (!FOURIER) dsum = fmaf(ww[i] * res, res, dsum);
                lsum = fmaf(oo[i], fabsf(xz[i]), lsum);
            }
        }
        if constexpr (REC) *dl = make_float2(dsum, lsum);
        if constexpr (DOT) *rsum = r;
    }
}

template <int VX>
__device__ __forceinline__ void ld_vec(const float *p, float (&v)[VX])
{
    if constexpr (VX == 4) {
        float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else if constexpr (VX == 2) {
        float2 t = *reinterpret_cast<const float2 *>(p);
        v[0] = t.x; v[1] = t.y;
    } else {
        v[0] = p[0];
    }
}

template <int VX>
__device__ __forceinline__ void st_vec(float *p, const float (&v)[VX])
{
    if constexpr (VX == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else if constexpr (VX == 2) {
        *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
    } else {
        p[0] = v[0];
    }
}

__device__ __forceinline__ float bf16_bits_to_f32(uint32_t h) { return __uint_as_float(h << 16); }

// Load VX data values stored as float32 or bfloat16 (raw bits widened exactly).
template <int VX, bool BF16>
__device__ __forceinline__ void ld_data(const unsigned char *tile, int idx, float (&v)[VX])
{
    if constexpr (!BF16) {
        ld_vec<VX>(reinterpret_cast<const float *>(tile) + idx, v);
    } else {
        const uint16_t *t = reinterpret_cast<const uint16_t *>(tile) + idx;
        // the low half moves up by 16 bits, the high half is masked in place
        if constexpr (VX == 4) {
            uint2 u = *reinterpret_cast<const uint2 *>(t);
            v[0] = __uint_as_float(u.x << 16); v[1] = __uint_as_float(u.x & 0xffff0000u);
            v[2] = __uint_as_float(u.y << 16); v[3] = __uint_as_float(u.y & 0xffff0000u);
        } else if constexpr (VX == 2) {
            uint32_t u = *reinterpret_cast<const uint32_t *>(t);
            v[0] = __uint_as_float(u << 16); v[1] = __uint_as_float(u & 0xffff0000u);
        } else {
            v[0] = bf16_bits_to_f32(t[0]);
        }
    }
}

struct StateSnap {
    int cur, k_round, hist_count, last;
    long long k_total;
    int rec0, pad;  // k_total modulo the recording interval at the launch's first iteration
};

template <int VX, int TY, int S, bool BF16>
struct Cfg {
    static constexpr int TX = 32 * VX;
    static constexpr int XW = TX + 8, XH = TY + 2;   // x tiles: origin (x0-4, y0-1)
    static constexpr int OW = TX + 4, OH = TY + 1;   // omtv tile: origin (x0, y0)
    static constexpr int ES = BF16 ? 2 : 4;
    static constexpr int XT_BYTES = XW * XH * 4;
    static constexpr int OM_BYTES = OW * OH * 4;
    static constexpr int BW_BYTES = TX * TY * ES;
    static constexpr int O1_BYTES = TX * TY * 4;
    static constexpr int al(int n) { return (n + 127) / 128 * 128; }
    static constexpr int OFF_XK = 0;
    static constexpr int OFF_XM = OFF_XK + al(XT_BYTES);
    static constexpr int OFF_OM = OFF_XM + al(XT_BYTES);
    static constexpr int OFF_B = OFF_OM + al(OM_BYTES);
    static constexpr int OFF_W = OFF_B + al(BW_BYTES);
    static constexpr int OFF_O1 = OFF_W + al(BW_BYTES);
    static constexpr int STAGE = OFF_O1 + al(O1_BYTES);
    static constexpr int OFF_PY = S * STAGE;                  // 3 x (TY+1) x TX floats
    static constexpr int OFF_HX = OFF_PY + al(3 * (TY + 1) * TX * 4);  // 3 x 32 floats
    static constexpr int OFF_RED = OFF_HX + 3 * 32 * 4;       // 32 x 4 doubles
    static constexpr int OFF_BAR = OFF_RED + 32 * 4 * 8;      // S mbarriers
    static constexpr int OFF_ST = OFF_BAR + al(S * 8);        // state snapshot
    static constexpr int OFF_KM = OFF_ST + 128;               // extrapolation index per item (restart)
    static constexpr int OFF_IT = OFF_KM + kMaxCtaItems * 4;  // the CTA's first items
    static constexpr int TOTAL = OFF_IT + kItemCache * (int)sizeof(WorkItem) + 128;  // + alignment slack
    static_assert(sizeof(StateSnap) <= 64 && sizeof(WorkItem) <= 64, "state snapshot and next item share 128 bytes");
    static constexpr int THREADS = 32 * (TY + 1);
    static_assert(TY + 1 <= 32, "reduction scratch sized for at most 32 warps");
    static_assert(TY <= 32, "halo column handled by one lane per row");
};

// Producer (one thread): stage contents for step j of work item W, i.e.
// plane z = z0-1+j of x_k (buffer ia) and of x_{k-1} or d_k (buffer ib), both
// with halo, and of omtv, and plane z-1 of b, w and om1. Steps 0 and 1 skip
// what they do not consume. In two parts: what no iteration writes, with the
// stage's byte count (it can be fetched before the iterate is final), and the
// iterate.
template <class C, int S, bool LOADW>
__device__ __forceinline__ void issue_fixed(unsigned char *sm, uint64_t *bars, const TmapSet *tm, const WorkItem &W,
                                            unsigned gstep, int j)
{
    const int s = (int)((gstep + (unsigned)j) % S);
    unsigned char *base = sm + s * C::STAGE;
    const int z = W.z0 - 1 + j;
    const bool need_om = j >= 1, need_bwo = j >= 2;
    const uint32_t bytes = 2 * C::XT_BYTES + (need_om ? C::OM_BYTES : 0) +
                           (need_bwo ? (LOADW ? 2 : 1) * C::BW_BYTES + C::O1_BYTES : 0);
    mbar_arrive_expect_tx(&bars[s], bytes);
    if (need_om) tma_load_3d(base + C::OFF_OM, &tm->omtv, W.x0, W.y0, z, &bars[s]);
    if (need_bwo) {
        tma_load_3d(base + C::OFF_B, &tm->b, W.x0, W.y0, z - 1, &bars[s]);
        if (LOADW) tma_load_3d(base + C::OFF_W, &tm->w, W.x0, W.y0, z - 1, &bars[s]);
        tma_load_3d(base + C::OFF_O1, &tm->om1, W.x0, W.y0, z - 1, &bars[s]);
    }
}

template <class C, int S>
__device__ __forceinline__ void issue_iterate(unsigned char *sm, uint64_t *bars, const TmapSet *tm, const WorkItem &W,
                                              int ia, int ib, unsigned gstep, int j)
{
    const int s = (int)((gstep + (unsigned)j) % S);
    unsigned char *base = sm + s * C::STAGE;
    // below the first plane: that plane itself, whose difference is then zero (Eq. 12)
    const int z = max(W.z0 - 1 + j, 0);
    tma_load_3d(base + C::OFF_XK, &tm->x[ia], W.x0 - 4, W.y0 - 1, z, &bars[s]);
    tma_load_3d(base + C::OFF_XM, &tm->x[ib], W.x0 - 4, W.y0 - 1, z, &bars[s]);
}

// Shared-memory carve-up of one CTA.
struct Smem {
    unsigned char *sm;
    uint64_t *bars;
    float *py_ring;
    float *hx_ring;
    double *red;
    StateSnap *snap;
    WorkItem *next;  // the item after the current one (producer lane only)
    WorkItem *items; // the CTA's first kItemCache items
    int *kmom;  // restart: extrapolation index of each of the CTA's items
};

// Pipeline bookkeeping of one CTA (issued: producer lane only).
struct Pipe {
    unsigned gstep;       // steps consumed so far
    unsigned iter_first;  // first step of the current iteration
    unsigned issued;      // steps issued so far
    unsigned drain_from;  // first step that may be pending after an abort
};

// One work item: plane-by-plane march over [z0, z1) of one x-y tile.
// REC adds the three sums of F(x_k) (data, l1, TV) for the item, written to
// `part`. kmom: the volume's extrapolation index in this iteration; tm: the
// iteration's tensor maps (of every volume); has_next: the CTA has another item
// in this iteration (*sh.next), whose first planes the producer fetches while
// this item's last ones are computed. The copies of the iteration's first S
// steps are issued by the caller. Ends with a barrier over the CTA
// after the item's last stores to the iterate; the sums go to `part` behind it
// (with DOT before a further barrier), so a reader in another CTA needs one more.
// Returns true when a barrier wait gave up (the CTA then stops).
template <int VX, int TY, int S, bool BF16, bool XD, bool REC, bool DOT, bool FOURIER>
__device__ __forceinline__ bool run_item(const StepParams &P, const Smem &sh, Pipe &pp_, const WorkItem &W,
                                         bool has_next, double *part, int kmom, const TmapSet *tm, int ia, int ib,
                                         float *xout_base, float *dout_base)
{
    using C = Cfg<VX, TY, S, BF16>;
    constexpr int TX = C::TX, XW = C::XW, OW = C::OW;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool main_warp = warp < TY;
    const int r = warp;  // tile row of this warp (r == TY: the +y halo row)
    const VolDesc V = P.vols[W.vol];
    const int nsteps = (W.z1 - W.z0) + 2;
    const float beta = SPG_GUARD(P.st, kmom >= 0 && kmom < P.beta_len, 2u) ? P.beta[kmom] : 0.f;
    const float beta_next = (FOURIER && kmom + 1 < P.beta_len) ? P.beta[kmom + 1] : 0.f;
    // (per volume: restarts reset a volume's extrapolation index)
    const float tau = V.tau, lam_tv = V.lambda_tv, tl1 = V.tau * V.lambda_l1;
    const float inv_mu = 1.0f / V.mu, half_inv_mu = 0.5f / V.mu, half_mu = 0.5f * V.mu;
    const float mu2 = V.mu * V.mu;
    const unsigned g0 = pp_.gstep;

    // the TMA producer is lane 0 of the halo warp, which has no write phase
    const bool producer = (warp == TY) && (lane == 0);
    // Producer: copies of the CTA's plane step d steps into this item, or
    // past its end into the next one's (an item has at least 3 steps, so d
    // never reaches a third item).
    static_assert(S <= 4, "the producer runs at most 3 steps ahead");
    auto issue = [&](int d) {
        if (d < nsteps) {
            const TmapSet *t = tm + W.vol;
            issue_fixed<C, S, !FOURIER>(sh.sm, sh.bars, t, W, g0, d);
            issue_iterate<C, S>(sh.sm, sh.bars, t, W, ia, ib, g0, d);
        } else if (has_next) {
            const WorkItem N = *sh.next;
            const TmapSet *t = tm + N.vol;
            issue_fixed<C, S, !FOURIER>(sh.sm, sh.bars, t, N, g0 + (unsigned)nsteps, d - nsteps);
            issue_iterate<C, S>(sh.sm, sh.bars, t, N, ia, ib, g0 + (unsigned)nsteps, d - nsteps);
        } else {
            return;
        }
        pp_.issued++;
    };

    // registers carried across z-steps
    float xz[VX], dz[VX];         // x_k and d on plane z-1, own columns
    float pp[3][VX];              // p on plane z-1, own columns
    float cxz = 0.f, cdz = 0.f;   // +x halo column values on plane z-1
#pragma unroll
    for (int i = 0; i < VX; i++) {
        xz[i] = 0.f;
        dz[i] = 0.f;
        pp[0][i] = pp[1][i] = pp[2][i] = 0.f;
    }
    KSum2 kdl;            // objective sums: data (x) and l1 (y)
    KSum kt, kr;          // TV sum and (DOT) the restart test <y - x+, x+ - x>

    const int gy = W.y0 + r;
    const int gx0 = W.x0 + VX * lane;
    const bool col_lane = (warp == TY) && (lane < TY);
    const bool gy_in = gy < V.ny;

    // Outside the volume the TMA boxes read zeros, so omtv, b, w and om1 are 0
    // there and p and every objective term vanish without per-voxel masks.
    // The zero differences on the first column, row and plane (Eq. 12) are
    // made by substituting the voxel itself for its missing neighbour, by where
    // the neighbour is read (its own row or column, the first plane twice)
    // rather than by selecting between loaded values: 16 of the 360 instructions
    // of a 4-voxel plane step.
    const int row_off = (r + 1) * XW + 4 + VX * lane;                           // own row
    const int up_off = (gy == 0 ? r + 1 : r) * XW + 4 + VX * lane;              // row y - 1
    const int left_off = (r + 1) * XW + (W.x0 == 0 ? 4 : 3);                    // column x0 - 1 (lane 0)
    const int col_off = (lane + 1) * XW + TX + 4;                               // +x halo column
    const int col_up_off = (W.y0 + lane == 0 ? lane + 1 : lane) * XW + TX + 4;  // and its row y - 1
    bool aborted = false;
    // output offset of plane z-1 = W.z0 - 2 + j, advanced by one plane per step
    const long long plane_elems = (long long)V.ny * V.pitch;
    long long o = V.off + ((long long)(W.z0 - 2) * V.ny + gy) * V.pitch + gx0;
    int slot = 0, slot_prev = 2;  // j % 3 and (j - 1) % 3 (p_y and p_x halo rings)
#pragma unroll 2
    for (int j = 0; j < nsteps; j++) {
        const int s = (int)((g0 + j) % S);
        const uint32_t parity = (uint32_t)(((g0 + j) / S) & 1);
        const unsigned char *base = sh.sm + s * C::STAGE;
        const float *XK = reinterpret_cast<const float *>(base + C::OFF_XK);
        const float *XM = reinterpret_cast<const float *>(base + C::OFF_XM);
        const float *OM = reinterpret_cast<const float *>(base + C::OFF_OM);
        const int z = W.z0 - 1 + j;

        const bool ok = mbar_wait(&sh.bars[s], parity, P.timeout_ns);

        // ---- A: p on plane z at this thread's columns ----
        float xc[VX] = {}, mc[VX] = {}, xu[VX] = {}, mu_[VX] = {}, dc[VX];
        if (SPG_GUARD(P.st, up_off >= 0 && up_off <= row_off && row_off + VX <= XW * C::XH, 3u)) {
            ld_vec<VX>(XK + row_off, xc);
            ld_vec<VX>(XM + row_off, mc);
            ld_vec<VX>(XK + up_off, xu);
            ld_vec<VX>(XM + up_off, mu_);
        }
        float xl = __shfl_up_sync(FULL, xc[VX - 1], 1);
        float ml = __shfl_up_sync(FULL, mc[VX - 1], 1);
        if (lane == 0) {
            xl = XK[left_off];
            ml = XM[left_off];
        }
#pragma unroll
        for (int i = 0; i < VX; i++) dc[i] = XD ? mc[i] : xc[i] - mc[i];
        float pc[3][VX];
        if (j >= 1) {
            float om[VX] = {};
            if (SPG_GUARD(P.st, r * OW + VX * (lane + 1) <= OW * C::OH, 5u)) ld_vec<VX>(OM + r * OW + VX * lane, om);
            float tsum = 0.f;
            float dup_[VX];
#pragma unroll
            for (int i = 0; i < VX; i++) dup_[i] = XD ? mu_[i] : xu[i] - mu_[i];
            phase_a<VX, REC>(xc, dc, xu, dup_, xz, dz, om, xl, XD ? ml : xl - ml, beta, inv_mu, half_inv_mu,
                             half_mu, mu2, pc, &tsum);
            if constexpr (REC) {
                if (main_warp && z < W.z1) kt.add(tsum);
            }
            // +x halo column (only p_x is consumed), one lane per tile row
            if (col_lane && SPG_GUARD(P.st, col_off < XW * C::XH && lane * OW + TX < OW * C::OH, 4u)) {
                const float cx = XK[col_off], cm = XM[col_off];
                const float cxl = XK[col_off - 1], cml = XM[col_off - 1];
                const float cxu = XK[col_up_off], cmu = XM[col_up_off];
                const float cd = XD ? cm : cx - cm;
                const int hx = W.x0 + TX, hy = W.y0 + lane;
                // the operations of phase_a, so that a voxel's result does not depend
                // on where the tiles' borders lie
                const float ax = fmaf(beta, cd - (XD ? cml : cxl - cml), cx - cxl);
                const float ay = fmaf(beta, cd - (XD ? cmu : cxu - cmu), cx - cxu);
                const float az = fmaf(beta, cd - cdz, cx - cxz);
                const float s2 = fmaf(ax, ax, fmaf(ay, ay, az * az));
                const bool in = hx < V.nx && hy < V.ny && z < V.nz;
                const float sc = in ? OM[lane * OW + TX] * fminf(inv_mu, rsqrtf(s2)) : 0.f;
                sh.hx_ring[slot * 32 + lane] = ax * sc;
            }
            if (SPG_GUARD(P.st, r <= TY && slot == j % 3 && (slot * (TY + 1) + r) * TX + VX * (lane + 1) <= 3 * (TY + 1) * TX, 6u))
                st_vec<VX>(sh.py_ring + (slot * (TY + 1) + r) * TX + VX * lane, pc[1]);
        } else {
#pragma unroll
            for (int i = 0; i < VX; i++) pc[0][i] = pc[1][i] = pc[2][i] = 0.f;
        }
        if (col_lane) {
            const float cx = XK[col_off], cm = XM[col_off];
            cxz = cx;
            cdz = XD ? cm : cx - cm;
        }

        if (__syncthreads_or(ok ? 0 : 1)) {
            aborted = true;
            pp_.drain_from = g0 + j;
            break;
        }
        // refill the stage of the step before this one (of this item or of the
        // one before), which every warp has finished with
        if (producer && g0 + j != pp_.iter_first) issue(j - 1 + S);

        // ---- B: write plane z-1 ----
        if (main_warp && j >= 2) {
            const int zo = z - 1;
            float bb[VX] = {}, ww[VX] = {}, oo[VX] = {}, pyd[VX] = {};
            if (SPG_GUARD(P.st, r < TY && r * TX + VX * (lane + 1) <= TX * TY, 7u)) {
                ld_data<VX, BF16>(base + C::OFF_B, r * TX + VX * lane, bb);
                if constexpr (!FOURIER) ld_data<VX, BF16>(base + C::OFF_W, r * TX + VX * lane, ww);
                ld_vec<VX>(reinterpret_cast<const float *>(base + C::OFF_O1) + r * TX + VX * lane, oo);
                ld_vec<VX>(sh.py_ring + ((slot_prev * (TY + 1)) + r + 1) * TX + VX * lane, pyd);
            }
            float pxn = __shfl_down_sync(FULL, pp[0][0], 1);
            if (lane == 31) pxn = sh.hx_ring[slot_prev * 32 + r];
            float out[VX], inc[VX];
            float2 dl = make_float2(0.f, 0.f);
            float rsum = 0.f;
            phase_b<VX, REC, DOT, FOURIER>(pp, pxn, pyd, pc[2], xz, dz, bb, ww, oo, beta, tau, lam_tv, tl1, out, inc,
                                           &dl, &rsum);
            if constexpr (REC) kdl.add(dl);
            if constexpr (DOT) kr.add(rsum);
            if (gy_in && gx0 < V.pitch &&
                SPG_GUARD(P.st, zo >= 0 && zo < V.nz && gx0 + VX <= V.pitch &&
                          o == V.off + ((long long)zo * V.ny + gy) * V.pitch + gx0, 8u)) {
                st_vec<VX>(xout_base + o, out);
                if constexpr (XD) st_vec<VX>(dout_base + o, inc);
                if constexpr (FOURIER) {
                    // the next step's extrapolated point, input of its forward transform
                    if (P.ybuf) {
                        float yv[VX];
#pragma unroll
                        for (int i = 0; i < VX; i++) yv[i] = fmaf(beta_next, inc[i], out[i]);
                        st_vec<VX>(P.ybuf + o, yv);
                    }
                }
            }
        }
#pragma unroll
        for (int i = 0; i < VX; i++) {
            xz[i] = xc[i];
            dz[i] = dc[i];
            pp[0][i] = pc[0][i];
            pp[1][i] = pc[1][i];
            pp[2][i] = pc[2][i];
        }
        o += plane_elems;
        slot_prev = slot;
        slot = slot == 2 ? 0 : slot + 1;
    }

    if (!aborted && (REC || DOT)) {
        // reduction of the item's sums over the row warps (the halo warp has
        // none and goes on), fixed order, in float-float or, where that could
        // overflow, in double (spg_ff.cuh)
        const ff::FF d = kdl.value_x();
        const ff::FF v[4] = {{0.5f * d.hi, 0.5f * d.lo}, kdl.value_y(), kt.value(), kr.value()};
        const bool big = ff::too_big(v[0]) || ff::too_big(v[1]) || ff::too_big(v[2]) || ff::too_big(v[3]);
        const bool wide = __syncthreads_or(big ? 1 : 0) != 0;
        if (main_warp) {
            if (!wide) {
                ff::FF *const red = reinterpret_cast<ff::FF *>(sh.red);
                const ff::FF s = ff::warp_sum4(v, lane);
                if ((lane & 7) == 0) red[warp * 4 + (lane >> 3)] = s;
                row_warps_sync<TY>();
                if (warp == 0) {
                    const ff::FF t = ff::cross_warp_sum4(red, TY, lane, ff::FF{0.f, 0.f});
                    if (lane < 4) part[lane] = ff::to_double(t);
                }
            } else {
                const double w[4] = {ff::to_double(v[0]), ff::to_double(v[1]), ff::to_double(v[2]),
                                     ff::to_double(v[3])};
                const double s = ff::warp_sum4(w, lane);
                if ((lane & 7) == 0) sh.red[warp * 4 + (lane >> 3)] = s;
                row_warps_sync<TY>();
                if (warp == 0) {
                    const double t = ff::cross_warp_sum4(sh.red, TY, lane, 0.0);
                    if (lane < 4) part[lane] = t;
                }
            }
        }
        if constexpr (DOT) __syncthreads();  // the next iteration's extrapolation depends on the sums
    } else {
        __syncthreads();
    }
    if (!aborted) pp_.gstep = g0 + nsteps;
    return aborted;
}

// Barrier over the CTAs of the grid (all resident: cooperative launch), the
// producer lane's half: the CTA's stores of the iteration precede it (a CTA
// barrier), are made visible, and the other CTAs' are visible to this CTA's
// copies when it returns true. False when it gave up (bounded, or another
// CTA did).
__device__ __forceinline__ bool grid_barrier(DevState *st, unsigned target, long long limit_ns)
{
    // the next copies (async proxy) read what the grid's threads wrote with
    // ordinary stores
    asm volatile("fence.proxy.async;" ::: "memory");
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&st->bar) : "memory");
    const long long t0 = global_ns();
    for (;;) {
        for (int i = 0; i < 64; i++) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&st->bar) : "memory");
            if (v >= target) {
                asm volatile("fence.proxy.async;" ::: "memory");
                return true;
            }
        }
        if (*(volatile int *)&st->err == (int)SPG_ETIMEOUT || global_ns() - t0 > limit_ns) return false;
    }
}

// Iterations of this launch before iteration i that record the objective
// (rec0 < every; the distances fit an unsigned for every `every` an int holds).
__host__ __device__ __forceinline__ int recorded_before(int rec0, int every, int i)
{
    if (every <= 0) return 0;
    const unsigned first = rec0 > 0 ? (unsigned)every - (unsigned)rec0 : 0u;  // the first that records
    return (unsigned)i <= first ? 0 : (int)(((unsigned)i - first - 1u) / (unsigned)every) + 1;
}

// Sums of volume V's item partials (one warp, fixed order): every lane gets
// all four.
__device__ __forceinline__ void volume_sums(const VolDesc &V, const double *part, int lane, double (&a)[4])
{
    a[0] = a[1] = a[2] = a[3] = 0.0;
#pragma unroll 4
    for (int q = V.item_begin + lane; q < V.item_end; q += 32) {
        const double2 *p = reinterpret_cast<const double2 *>(part + (long long)q * 4);
        const double2 u = __ldcg(p), w = __ldcg(p + 1);
        a[0] += u.x;
        a[1] += u.y;
        a[2] += w.x;
        a[3] += w.y;
    }
    const double s = ff::warp_sum4(a, lane);
#pragma unroll
    for (int c = 0; c < 4; c++) a[c] = __shfl_sync(FULL, s, 8 * c);
}

// The restart product of volume V alone.
__device__ __forceinline__ double volume_dot(const VolDesc &V, const double *part, int lane)
{
    double a = 0.0;
#pragma unroll 4
    for (int q = V.item_begin + lane; q < V.item_end; q += 32) a += __ldcg(part + (long long)q * 4 + 3);
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) a += __shfl_xor_sync(FULL, a, m);
    return a;
}

// History entry number `entry` of volume v: F(x_k) from its sums (one thread).
__device__ __forceinline__ void history_entry(const StepParams &P, const VolDesc &V, int v, long long entry,
                                              long long k, const double (&a)[4])
{
    if (!SPG_GUARD(P.st, entry >= 0 && v >= 0 && v < P.nvol, 11u)) return;
    double *h = P.hist + ((entry % P.hist_cap) * P.nvol + v) * 5;
    const double l1 = (double)V.lambda_l1 * a[1], tv = (double)V.lambda_tv * a[2];
    const double tot = a[0] + l1 + tv;
    h[0] = (double)k;
    h[1] = a[0];
    h[2] = l1;
    h[3] = tv;
    h[4] = tot;
    if (!isfinite(tot)) atomicCAS(&P.st->err, 0, (int)SPG_ENONFINITE);
}

// Objective history of the launch: warp w of `nw` takes the (iteration,
// volume) pairs w, w + nw, ... of those that record. Of more than hist_cap
// entries only the newest are written (the ring keeps no others).
__device__ __forceinline__ void write_history(const StepParams &P, const StateSnap &S, int w, int nw, int lane)
{
    const int total = recorded_before(S.rec0, P.hist_every, P.niter);
    for (long long e = w; e < (long long)P.niter * P.nvol; e += nw) {
        const int i = (int)(e / P.nvol), v = (int)(e % P.nvol);
        if (P.hist_every <= 0 || ((unsigned)S.rec0 + (unsigned)i) % (unsigned)P.hist_every != 0) continue;
        const int rank = recorded_before(S.rec0, P.hist_every, i);
        if (total - rank > P.hist_cap) continue;
        const VolDesc V = P.vols[v];
        double a[4];
        volume_sums(V, P.partials + (long long)i * P.nitems * 4, lane, a);
        if (lane == 0) history_entry(P, V, v, (long long)S.hist_count + rank, S.k_total + i, a);
    }
}

template <int VX, int TY, int S, bool BF16, bool XD, int MINB>
__global__ void __launch_bounds__(32 * (TY + 1), MINB)
    spg_step_kernel(const StepParams P)
{
    using C = Cfg<VX, TY, S, BF16>;
    extern __shared__ unsigned char smem_raw[];
    Smem sh;
    // 128-byte aligned start, kept as an offset into the shared array so the
    // compiler addresses every tile as shared memory
    sh.sm = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    sh.bars = reinterpret_cast<uint64_t *>(sh.sm + C::OFF_BAR);
    sh.py_ring = reinterpret_cast<float *>(sh.sm + C::OFF_PY);
    sh.hx_ring = reinterpret_cast<float *>(sh.sm + C::OFF_HX);
    sh.red = reinterpret_cast<double *>(sh.sm + C::OFF_RED);
    sh.snap = reinterpret_cast<StateSnap *>(sh.sm + C::OFF_ST);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    sh.next = reinterpret_cast<WorkItem *>(sh.sm + C::OFF_ST + 64);
    sh.items = reinterpret_cast<WorkItem *>(sh.sm + C::OFF_IT);
    sh.kmom = reinterpret_cast<int *>(sh.sm + C::OFF_KM);
    const bool producer = (warp == TY) && (lane == 0);

    if (tid == 0) {
        volatile DevState *st = P.st;
        StateSnap s;
        s.cur = st->cur;
        s.k_round = st->k_round;
        s.k_total = st->k_total;
        s.hist_count = st->hist_count;
        s.rec0 = P.hist_every > 0 ? (int)(s.k_total % P.hist_every) : 0;
        s.last = 0;
        s.pad = 0;
        *sh.snap = s;
        for (int i = 0; i < S; i++) mbar_init(&sh.bars[i], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int p0 = P.sched[blockIdx.x], p_end = P.sched[blockIdx.x + 1];
    // the plan against the room it was made for: items, partial sums and planned
    // steps per iteration, and (restart) extrapolation indices in shared memory
    const bool plan_ok =
        SPG_GUARD(P.st, p0 >= 0 && p0 <= p_end && p_end <= P.nitems && P.niter >= 1 && P.niter <= P.iter_cap &&
                            (!P.restart || P.niter == 1 || p_end - p0 <= kMaxCtaItems), 9u);
    const int p1 = plan_ok ? p_end : p0;
    // the CTA's items (P.items is in schedule order; pad0: the item's number among
    // its volume's partial sums), with the volume's extrapolation index at the
    // start of the launch (pad1): the barrier between iterations
    // drops L1, and the chain schedule, item, descriptor from L2 would delay the
    // next iteration's first copies
    auto load_item = [&](int p) {
        WorkItem W = P.items[p];
        if (!SPG_GUARD(P.st, W.vol >= 0 && W.vol < P.nvol && W.pad0 >= 0 && W.pad0 < P.nitems, 10u)) W.vol = W.pad0 = 0;
        return W;
    };
    auto item_at = [&](int p) {
        if (p - p0 < kItemCache) return sh.items[p - p0];
        WorkItem W = load_item(p);
        W.pad1 = P.vols[W.vol].kmom;
        return W;
    };
    if (tid < kItemCache && p0 + tid < p1) {
        const WorkItem W = load_item(p0 + tid);
        sh.items[tid] = W;
        // not waited for by the copies below: stored once it arrives
        sh.items[tid].pad1 = P.vols[W.vol].kmom;
    }
    __syncthreads();
    // select without indexing the parameter array (keeps the parameters out of local memory)
    auto pick = [&](int i) { return i == 0 ? P.xbuf[0] : (i == 1 ? P.xbuf[1] : (i == 2 ? P.xbuf[2] : P.xbuf[3])); };
    const bool many = P.niter > 1;

    Pipe pipe{0, 0, 0, 0};
    bool aborted = !plan_ok;
    // copies of the first S plane steps of an iteration (of its first item, or
    // of the first two where that has only 3 steps)
    auto first_steps = [&](auto f) {
        const WorkItem W = sh.items[0];
        const int n = (W.z1 - W.z0) + 2;
#pragma unroll
        for (int d = 0; d < S; d++) {
            if (d < n) f(W, pipe.gstep, d);
            else if (p0 + 1 < p1) f(item_at(p0 + 1), pipe.gstep + (unsigned)n, d - n);
        }
    };
    auto first_fixed = [&](const TmapSet *tm) {
        first_steps([&](const WorkItem &W, unsigned g, int j) {
            if (!BF16 && XD && P.fourier)
                issue_fixed<C, S, false>(sh.sm, sh.bars, tm + W.vol, W, g, j);
            else
                issue_fixed<C, S, true>(sh.sm, sh.bars, tm + W.vol, W, g, j);
            pipe.issued++;
        });
    };
    auto first_iterate = [&](const TmapSet *tm, int ia, int ib) {
        first_steps([&](const WorkItem &W, unsigned g, int j) {
            issue_iterate<C, S>(sh.sm, sh.bars, tm + W.vol, W, ia, ib, g, j);
        });
    };
    int cur = sh.snap->cur;
    int rec_in = sh.snap->rec0;  // iterations since the last recorded one (0: this one records)
    for (int itn = 0; itn < P.niter && !aborted; itn++) {
        // buffers: XD keeps x in 0/1 and d in 2/3; otherwise x_{k-1}, x_k, x_{k+1} rotate over 0..2
        const int nxt = XD ? (cur ^ 1) : (cur + 1) % 3;
        const int ia = cur, ib = XD ? 2 + cur : (cur + 2) % 3;
        const bool rec = P.hist_every > 0 && rec_in == 0;
        float *const xout_base = P.xouts ? P.xouts[itn] : pick(nxt);
        float *const dout_base = XD ? pick(2 + nxt) : nullptr;
        const TmapSet *const tm = P.tmaps + (long long)itn * P.tm_step;
        pipe.iter_first = pipe.gstep;
        if (producer && itn == 0 && p0 < p1) {
            const TmapSet *t = tm + sh.items[0].vol;
            prefetch_tmap(&t->x[ia]);
            prefetch_tmap(&t->x[ib]);
            prefetch_tmap(&t->omtv);
            prefetch_tmap(&t->b);
            prefetch_tmap(&t->w);
            prefetch_tmap(&t->om1);
            first_fixed(tm);
            first_iterate(tm, ia, ib);
        }
        for (int p = p0; p < p1 && !aborted; p++) {
            const WorkItem W = item_at(p);
            const int it = W.pad0;
            const bool has_next = p + 1 < p1;
            if (producer && has_next) *sh.next = item_at(p + 1);
            const int kmom = (P.restart && many && itn > 0) ? sh.kmom[p - p0] : W.pad1 + itn;
            double *const part = P.partials + ((long long)itn * P.nitems + it) * 4;
            bool done = false;
            if constexpr (!BF16 && XD) {
                // Fourier-domain data term (float32 storage, increment storage only)
                if (P.fourier) {
                    aborted = rec ? run_item<VX, TY, S, BF16, XD, true, false, true>(P, sh, pipe, W, has_next, part, kmom, tm, ia, ib, xout_base, dout_base)
                                  : run_item<VX, TY, S, BF16, XD, false, false, true>(P, sh, pipe, W, has_next, part, kmom, tm, ia, ib, xout_base, dout_base);
                    done = true;
                }
            }
            if (!done) {
                if (P.restart)
                    aborted = rec ? run_item<VX, TY, S, BF16, XD, true, true, false>(P, sh, pipe, W, has_next, part, kmom, tm, ia, ib, xout_base, dout_base)
                                  : run_item<VX, TY, S, BF16, XD, false, true, false>(P, sh, pipe, W, has_next, part, kmom, tm, ia, ib, xout_base, dout_base);
                else
                    aborted = rec ? run_item<VX, TY, S, BF16, XD, true, false, false>(P, sh, pipe, W, has_next, part, kmom, tm, ia, ib, xout_base, dout_base)
                                  : run_item<VX, TY, S, BF16, XD, false, false, false>(P, sh, pipe, W, has_next, part, kmom, tm, ia, ib, xout_base, dout_base);
            }
        }
        if (aborted) break;
        if (many) {
            bool ok = true;
            // The last iteration's sums are read by other CTAs behind the grid
            // barrier, and the producer's warp does not wait for the row warps
            // that store them (run_item): a barrier over the CTA before the
            // producer arrives. The earlier iterations' are ordered by the
            // barriers of the plane steps that follow them.
            if (itn + 1 == P.niter) __syncthreads();
            if (producer) {
                // the next iteration's first copies: what no iteration writes before
                // the barrier, the iterate behind it (also after a failure, so that
                // the stages complete and can be drained)
                const bool more = itn + 1 < P.niter && p0 < p1;
                const TmapSet *const tn = tm + P.tm_step;
                const int ja = nxt, jb = XD ? 2 + nxt : (nxt + 2) % 3;
                if (more) {
                    if (P.tm_step) {
                        prefetch_tmap(&tn[sh.items[0].vol].x[ja]);
                        prefetch_tmap(&tn[sh.items[0].vol].x[jb]);
                    }
                    first_fixed(tn);
                }
                ok = grid_barrier(P.st, (unsigned)(itn + 1) * gridDim.x, P.timeout_ns);
                if (more) first_iterate(tn, ja, jb);
            }
            if (__syncthreads_or(ok ? 0 : 1)) {
                aborted = true;
                pipe.drain_from = pipe.gstep;
            } else if (P.restart && itn + 1 < P.niter) {
                // the extrapolation index of the next iteration, per item
                const double *const parts = P.partials + (long long)itn * P.nitems * 4;
                for (int p = p0 + warp; p < p1; p += TY + 1) {
                    const VolDesc V = P.vols[item_at(p).vol];
                    const int km = itn > 0 ? sh.kmom[p - p0] : V.kmom;
                    const bool again = volume_dot(V, parts, lane) > 0.0;
                    if (lane == 0) sh.kmom[p - p0] = again ? 0 : km + 1;
                }
                __syncthreads();
            }
        }
        cur = nxt;
        rec_in = rec_in >= P.hist_every - 1 ? 0 : rec_in + 1;
    }

    if (aborted && producer) {
        // record the timeout, then wait (bounded) for copies still in flight
        atomicCAS(&P.st->err, 0, (int)SPG_ETIMEOUT);
        for (unsigned q = pipe.drain_from; q < pipe.issued; q++) {
            const int s = (int)(q % S);
            (void)mbar_wait(&sh.bars[s], (uint32_t)((q / S) & 1), P.timeout_ns);
        }
    }

    // ---- objective history, extrapolation indices, device state ----
    VolDesc *const vols_rw = const_cast<VolDesc *>(P.vols);
    const StateSnap snap = *sh.snap;
    if (many && !aborted) {
        // every CTA's partials were stored before it arrived at the last grid barrier
        write_history(P, snap, blockIdx.x * (TY + 1) + warp, gridDim.x * (TY + 1), lane);
        const double *const parts = P.partials + (long long)(P.niter - 1) * P.nitems * 4;
        for (int p = p0 + warp; p < p1; p += TY + 1) {
            // a volume's descriptor is advanced by the CTA that runs its first item
            const WorkItem W = item_at(p);
            const int v = W.vol;
            const VolDesc V = P.vols[v];
            if (W.pad0 != V.item_begin) continue;
            const int km = P.restart ? sh.kmom[p - p0] : V.kmom + P.niter - 1;  // index of the last iteration
            const bool again = P.restart && volume_dot(V, parts, lane) > 0.0;
            if (lane == 0) {
                vols_rw[v].beta_last = P.beta[km];
                vols_rw[v].kmom = again ? 0 : km + 1;
            }
        }
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        const unsigned t = atomicAdd(&P.st->ticket, 1u);
        sh.snap->last = (t == gridDim.x - 1) ? 1 : 0;
    }
    __syncthreads();
    if (!sh.snap->last) return;
    __threadfence();
    if (!many) {
        // one iteration: the last CTA sums the objective and advances every
        // volume, a warp per volume
        const bool rec = P.hist_every > 0 && snap.rec0 == 0;
        for (int v = warp; v < P.nvol; v += TY + 1) {
            const VolDesc V = P.vols[v];
            const float beta_used = P.beta[V.kmom];
            double a[4] = {0.0, 0.0, 0.0, 0.0};
            if (rec || P.restart) volume_sums(V, P.partials, lane, a);
            if (lane == 0) {
                if (rec) history_entry(P, V, v, snap.hist_count, snap.k_total, a);
                vols_rw[v].beta_last = beta_used;
                vols_rw[v].kmom = (P.restart && a[3] > 0.0) ? 0 : V.kmom + 1;
            }
        }
    }
    __syncthreads();
    if (tid == 0) {
        DevState *st = P.st;
        st->hist_count = snap.hist_count + recorded_before(snap.rec0, P.hist_every, P.niter);
        st->cur = XD ? (snap.cur + P.niter) & 1 : (snap.cur + P.niter) % 3;
        st->k_round = snap.k_round + P.niter;
        st->k_total = snap.k_total + P.niter;
        st->ticket = 0;
        st->bar = 0;
        __threadfence();
    }
}

template <int VX, int TY, int S, bool BF16, bool XD, int MINB>
struct Launcher {
    using C = Cfg<VX, TY, S, BF16>;
    static cudaError_t configure(int *ctas_per_sm)
    {
        auto k = spg_step_kernel<VX, TY, S, BF16, XD, MINB>;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, C::TOTAL);
        if (e != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, k, C::THREADS, C::TOTAL);
    }
    static cudaError_t launch(int grid, const StepParams &p, cudaStream_t s)
    {
        auto k = spg_step_kernel<VX, TY, S, BF16, XD, MINB>;
        if (p.niter == 1) {
            k<<<grid, C::THREADS, C::TOTAL, s>>>(p);
            return cudaGetLastError();
        }
        // the iterations of one launch wait on one another: all CTAs resident
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(grid);
        cfg.blockDim = dim3(C::THREADS);
        cfg.dynamicSmemBytes = C::TOTAL;
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeCooperative;
        at[0].val.cooperative = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, k, p);
    }
};

// Every compiled variant: (vx, ty, stages, minimum resident CTAs per SM).
#define SPG_VARIANTS(X) \
    X(4, 8, 3, 2)       \
    X(4, 7, 3, 2)       \
    X(4, 7, 4, 2)       \
    X(4, 15, 2, 1)      \
    X(4, 4, 4, 3)       \
    X(2, 8, 4, 2)       \
    X(2, 7, 4, 2)       \
    X(2, 4, 4, 3)

}  // namespace

// Dispatch over the compiled variants for one data dtype (BF16_).
#define SPG_DEFINE_DISPATCH(BF16_, SUFFIX)                                                          \
    size_t step_smem_bytes_##SUFFIX(const StepVariant &v)                                           \
    {                                                                                               \
        SPG_VARIANTS(SPG_SM_CASE)                                                                   \
        return 0;                                                                                   \
    }                                                                                               \
    cudaError_t step_configure_##SUFFIX(const StepVariant &v, int *occ)                             \
    {                                                                                               \
        SPG_VARIANTS(SPG_CF_CASE)                                                                   \
        return cudaErrorInvalidValue;                                                               \
    }                                                                                               \
    cudaError_t step_launch_##SUFFIX(const StepVariant &v, int grid, const StepParams &p, cudaStream_t s) \
    {                                                                                               \
        SPG_VARIANTS(SPG_LN_CASE)                                                                   \
        return cudaErrorInvalidValue;                                                               \
    }
#define SPG_SM_CASE(VX_, TY_, S_, MB_) \
    if (v.vx == VX_ && v.ty == TY_ && v.stages == S_) return Cfg<VX_, TY_, S_, SPG_BF16_FLAG>::TOTAL;
#define SPG_CF_CASE(VX_, TY_, S_, MB_)                                                             \
    if (v.vx == VX_ && v.ty == TY_ && v.stages == S_)                                              \
        return v.xd ? Launcher<VX_, TY_, S_, SPG_BF16_FLAG, true, MB_>::configure(occ)              \
                    : Launcher<VX_, TY_, S_, SPG_BF16_FLAG, false, MB_>::configure(occ);
#define SPG_LN_CASE(VX_, TY_, S_, MB_)                                                             \
    if (v.vx == VX_ && v.ty == TY_ && v.stages == S_)                                              \
        return v.xd ? Launcher<VX_, TY_, S_, SPG_BF16_FLAG, true, MB_>::launch(grid, p, s)          \
                    : Launcher<VX_, TY_, S_, SPG_BF16_FLAG, false, MB_>::launch(grid, p, s);

}  // namespace spg
