// Kernel-regression back-projection (Sec. 2.2, Eq. 24-28) on the GPU.
//
// Image i's coefficient X at 2-D frequency index (kx, ky) lands at the 3-D
// position p = R_i (kx, ky, 0) (Eq. 24). Every grid point n of the kernel's
// support around p receives
//     num(n) += P K CTF X,    N(n) += P K CTF^2        (Eq. 26-28)
// with P the posterior weight of the image-pose pair (1 for known poses) and
// K = exp(-|p - n|^2 / h) on the 27 points round(p) + {-1,0,1}^3 (the
// Gaussian kernel of Sec. 2.2) or the trilinear weights on the 8 corners of
// p's cell (the interpolation kernel the paper attributes to Relion).
//
// Images are real, so X(-k) = conj X(k), and CTFs are centro-symmetric: the
// coefficient -k lands at -p with the conjugate contribution. Only the half
// ky > 0 (and kx >= 0 on ky = 0) is read, and each contribution is added at n
// or, mirrored, at -n, whichever lies in the stored half spectrum
// [n][n][n/2+1] (both on the planes kx = 0 and kx = n/2). This halves both
// the atomics and the accumulator against a full-spectrum scatter and gives
// the same sums. A warp takes an 8 x 4 tile of one image's coefficients,
// sums their FP32 deposits in a shared-memory box of its own and adds each
// touched point once, with FP64 atomics, into an interleaved accumulator
// (Re num, Im num, N, unused: one 32-byte sector per grid point). A finishing
// pass writes the Eq. 31 data term: N' = V N and
// y = (-1)^(kx+ky+kz) num / sqrt(N), the sign moving the
// transform's origin from the box centre (image convention) to voxel 0 (the
// solver's convention; n even).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <string>

#include "spg.h"
#include "spg_ff.cuh"
#include "spg_trace.h"

namespace {

thread_local std::string g_grid_err = "no error";

constexpr int kThreads = 256;
constexpr int kMaxBlocks = 152 * 16;

__device__ __forceinline__ int wrap(int i, int n) { return ((i % n) + n) % n; }

// Add (re, im, w) at full-spectrum point (x, y, z) (any integers), and, unless
// the sample is its own mate (k = 0), the mate's (re, -im, w) at (-x, -y, -z):
// each where it falls in the stored half.
__device__ __forceinline__ void deposit(double *acc, int n, int x, int y, int z, double re, double im, double w,
                                        bool self_mate)
{
    const int nh = n / 2 + 1;
    const int xw = wrap(x, n);
    if (xw < nh) {
        double *a = acc + 4 * (((long long)wrap(z, n) * n + wrap(y, n)) * nh + xw);
        atomicAdd(a + 0, re);
        atomicAdd(a + 1, im);
        atomicAdd(a + 2, w);
    }
    if (self_mate) return;
    const int mx = wrap(-x, n);
    if (mx < nh) {
        double *a = acc + 4 * (((long long)wrap(-z, n) * n + wrap(-y, n)) * nh + mx);
        atomicAdd(a + 0, re);
        atomicAdd(a + 1, -im);
        atomicAdd(a + 2, w);
    }
}

// One image coefficient's contribution: the first grid point of its support
// on each axis, its position relative to that support, and the values it
// spreads.
struct Sample {
    int bx, by, bz;
    float fx, fy, fz;  // position minus the support's centre (kernel 0) or first point (kernel 1)
    float vre, vim, vcc;
};

// p = r0 kx + r1 ky on one axis: the nearest point (half to even, kernel 0) or
// floor (kernel 1) b and the remainder f.
struct AxisPos {
    int b;
    float f;
};

// In double, for positions beyond split_axis's range (matrices that are no
// rotations). b saturates; a Gaussian weight so far from b is zero.
__device__ __noinline__ AxisPos split_axis_wide(float r0, float r1, int kx, int ky, int kernel)
{
    const double p = __dadd_rn(__dmul_rn(r0, kx), __dmul_rn(r1, ky));
    AxisPos a;
    if (kernel == 0) {
        a.b = __double2int_rn(p);
        a.f = (float)(p - a.b);
    } else {
        const double c = floor(p);
        a.b = __double2int_rn(c);
        a.f = (float)(p - c);
    }
    return a;
}

// As exact arithmetic on the float32 entries gives them, where |p| < 2^22. The
// products are exact pairs (fused multiply-add), their
// leading parts are added exactly and the sum is normalised (the tails can
// exceed an ulp of the sum where the products cancel), so p = s + lo with |lo|
// at most half an ulp of s (an eighth) and an error far below any half-way case of
// float32 rotations; doubles gave the same decisions at 9 FP64 operations a coefficient and
// half a dozen conversions, more than a millisecond of GB300's FP64 pipe for
// 2048 images of 256^2. False beyond 2^22, where lo grows past the point s decides
// on: the caller then takes them (no rotation of n <= 1290 comes near).
__device__ __forceinline__ bool split_axis(float r0, float r1, int kx, int ky, int kernel, int &b, float &f)
{
    const float x = (float)kx, y = (float)ky;
    const float p = __fmul_rn(r0, x), q = __fmul_rn(r1, y);
    const spg::ff::FF u = spg::ff::two_sum(p, q);
    const spg::ff::FF v =
        spg::ff::two_sum(u.hi, __fadd_rn(u.lo, __fadd_rn(__fmaf_rn(r0, x, -p), __fmaf_rn(r1, y, -q))));
    const float s = v.hi, lo = v.lo;
    if (kernel == 0) {
        float c = rintf(s);
        const float r = __fsub_rn(s, c);
        // the rounding of s decides unless lo carries p across the half-way point
        if (__fadd_rn(__fsub_rn(r, 0.5f), lo) > 0.f) c += 1.f;
        else if (__fadd_rn(__fadd_rn(r, 0.5f), lo) < 0.f) c -= 1.f;
        b = (int)c;
        f = __fadd_rn(__fsub_rn(s, c), lo);
    } else {
        float c = floorf(s);
        if (__fsub_rn(s, c) == 0.f && lo < 0.f) c -= 1.f;
        b = (int)c;
        f = __fadd_rn(__fsub_rn(s, c), lo);
    }
    return fabsf(s) < 4194304.f;  // false for NaN too
}

__device__ __forceinline__ void make_sample(int n, const float *__restrict__ R, const float2 *__restrict__ X,
                                            const float *__restrict__ ctf, float pw, int kernel, int kx, int ky,
                                            Sample &S)
{
    const int src = ky * n + (kx < 0 ? kx + n : kx);
    const float2 x = __ldcs(X + src);
    const float c = __ldcs(ctf + src);
    const float pc = pw * c;
    S.vre = pc * x.x;
    S.vim = pc * x.y;
    S.vcc = pc * c;
    // row-major 3x3; columns 0 and 1 span the image plane
    const bool nx = split_axis(R[0], R[1], kx, ky, kernel, S.bx, S.fx);
    const bool ny = split_axis(R[3], R[4], kx, ky, kernel, S.by, S.fy);
    const bool nz = split_axis(R[6], R[7], kx, ky, kernel, S.bz, S.fz);
    if (!(nx && ny && nz)) {
        const AxisPos ax = split_axis_wide(R[0], R[1], kx, ky, kernel);
        const AxisPos ay = split_axis_wide(R[3], R[4], kx, ky, kernel);
        const AxisPos az = split_axis_wide(R[6], R[7], kx, ky, kernel);
        S.bx = ax.b;
        S.by = ay.b;
        S.bz = az.b;
        S.fx = ax.f;
        S.fy = ay.f;
        S.fz = az.f;
    }
    if (kernel == 0) {
        S.bx -= 1;
        S.by -= 1;
        S.bz -= 1;
    }
}

// Kernel weights of one axis: the kernel factorises over the axes, a product
// of 1-D Gaussians exp(-e^2/h) (3 points) or of 1-D hat functions (2 points).
__device__ __forceinline__ void axis_weights(int kernel, float ih, float f, float (&w)[3])
{
    if (kernel == 0) {
#pragma unroll
        for (int d = 0; d < 3; d++) {
            const float e = f - (d - 1);
            w[d] = expf(-e * e * ih);
        }
    } else {
        w[0] = 1.f - f;
        w[1] = f;
        w[2] = 0.f;
    }
}

// All deposits of one sample straight into the FP64 accumulator (rare: kept
// out of line).
__device__ __noinline__ void deposit_sample(double *acc, int n, int kernel, float ih, Sample S, bool self_mate)
{
    const int span = kernel == 0 ? 3 : 2;
    float wx[3], wy[3], wz[3];
    axis_weights(kernel, ih, S.fx, wx);
    axis_weights(kernel, ih, S.fy, wy);
    axis_weights(kernel, ih, S.fz, wz);
    for (int dz = 0; dz < span; dz++)
        for (int dy = 0; dy < span; dy++) {
            const float kyz = wy[dy] * wz[dz];
            for (int dx = 0; dx < span; dx++) {
                const float K = wx[dx] * kyz;
                deposit(acc, n, S.bx + dx, S.by + dy, S.bz + dz, (double)(K * S.vre), (double)(K * S.vim),
                        (double)(K * S.vcc), self_mate);
            }
        }
}

// The double that equals v, by integer operations for ordinary values (the
// conversion runs on the FP64 pipe, 16 cycles a warp).
__device__ __forceinline__ double widen(float v)
{
    const float a = fabsf(v);
    if (!(a >= 1.17549435e-38f && a <= 3.4028235e38f)) return (double)v;  // zero, denormal, infinite, NaN
    const int u = __float_as_int(v);
    return __hiloint2double(((u >> 3) & (int)0x8fffffff) + 0x38000000, u << 29);
}

// Bound: a coefficient's 27 deposits are a read-modify-write of 27 points in
// shared memory (float4: re, im, N, unused) and its share of the tile's points
// goes to L2 as FP64 atomics; reading the images takes 0.1 of 12 ms at 2048
// images of 256^2 into 256^3.
//
// One warp per tile of 8 x 4 coefficients, in its own box: the lanes are the
// support points of one sample at a time (27 or 8), so no two lanes meet and
// the box needs no atomics (float32 atomics in shared memory are
// compare-and-swap loops; they were what a form with a thread per sample waited
// for). The samples' weights and values pass through shared memory, one row of
// 32 samples each, so a lane fetches those of 4 samples at a time. The box's row
// and plane strides are padded where that still fits (rows to 3 .. 5 modulo 8
// points, planes to 1): the rows of a support then fall on different bank
// groups. A tile whose box
// exceeds the capacity is done in halves; what still does not fit (matrices
// that are no rotations), and the coefficient k = 0 (its own mate), deposits
// directly. In the flush the lanes are 10 points of a row by 3 values, so an
// atomic instruction covers a run of whole 32-byte sectors. Tiles go out tile
// by tile over all images, not image by image: the tiles of one |k| touch a
// spherical shell of the accumulator (32 MB at the rim of 256^3), which stays
// in L2.
//
// Measured, add and finish, against the thread-per-sample form (8 x 8 tiles,
// float32 atomics in the box): 2048 images of 256^2 12.4 -> 7.3 ms (trilinear
// 7.8 -> 5.6), 128 images 1.08 -> 0.73, 2048 of 128^2 3.20 -> 1.95, 4096 of 64^2
// 1.64 -> 1.10, 512 of 288^2 4.24 -> 2.63; with one wrapping addition per index of
// the boxes that cross the box's faces, instead of two integer divisions for
// each of six indices of a point, 7.0 (5.35), 0.72, 1.78, 0.99 and 2.54; 7.1 for the
// first with the test of a position's range (make_sample). What bounds it now, at 256^2: shared
// memory (800 wavefronts a tile, 64 % of its rate) and issue (2900 instructions
// a tile, 53 %) with the 16 warps an SM's shared memory holds.
constexpr int kTileX = 8, kTileY = 4;
constexpr int kBoxCap = 768;   // box points per warp (12 KB)
constexpr int kWarps = 8;      // per CTA; two CTAs per SM
constexpr int kStageRow = 36;  // floats; rows 4 banks apart
constexpr int kWarpSmem = kBoxCap * 16 + 13 * kStageRow * 4;

__global__ void __launch_bounds__(kWarps * 32, 2)
    scatter_tile_kernel(int n, int m, const float *__restrict__ rot, const float2 *__restrict__ X,
                        const float *__restrict__ ctf, const float *__restrict__ pw, int kernel, float h, double *acc)
{
    extern __shared__ __align__(16) unsigned char gsm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float4 *const box = reinterpret_cast<float4 *>(gsm + (size_t)warp * kWarpSmem);
    // rows of 32 samples: wx[3], wy[3], wz[3], re, im, N, box offset
    float *const stage = reinterpret_cast<float *>(box + kBoxCap);
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int q = lane; q < kBoxCap; q += 32) box[q] = zero4;
    const int span = kernel == 0 ? 3 : 2;
    const float ih = 1.0f / h;
    const int dx = lane % span, dy = (lane / span) % span, dz = lane / (span * span);
    const bool point = lane < span * span * span;
    const int nh = n / 2 + 1;
    const int ntx = (n + kTileX - 1) / kTileX, nty = (n / 2 + kTileY - 1) / kTileY;
    const float rmax2 = (n * 0.5f - 2.0f) * (n * 0.5f - 2.0f);
    const int fpx = lane / 3, fcomp = lane - 3 * fpx;  // flush: point of the row and value
    const unsigned conj = fcomp == 1 ? 0x80000000u : 0u;
    const long long ys = 4LL * nh, zs = ys * n;        // accumulator strides, doubles
    // work item (tile, image), the image counting faster, advanced by the number
    // of warps without a division per item
    const long long t0 = (long long)blockIdx.x * kWarps + warp, nwarps = (long long)gridDim.x * kWarps;
    const int dtile = (int)(nwarps / m), dimg = (int)(nwarps % m);
    int tile = (int)(t0 / m), img = (int)(t0 % m);
    const int ntiles = nty * ntx;
    auto next = [&]() {
        tile += dtile;
        img += dimg;
        if (img >= m) {
            img -= m;
            tile++;
        }
    };
    for (; tile < ntiles; next()) {
        const int kx0 = -n / 2 + (tile % ntx) * kTileX, ky0 = (tile / ntx) * kTileY;
        {
            // the tile's nearest coefficient to the origin lies outside the disc
            const int nx = kx0 > 0 ? kx0 : (kx0 + kTileX - 1 < 0 ? kx0 + kTileX - 1 : 0);
            if ((float)(nx * nx + ky0 * ky0) > rmax2) continue;
        }
        const long long img2 = (long long)img * n * n;
        const int kx = kx0 + lane % kTileX, ky = ky0 + lane / kTileX;
        const bool ok = kx < n / 2 && ky < n / 2 && (ky > 0 || kx >= 0) && (float)(kx * kx + ky * ky) <= rmax2;
        Sample S;
        if (ok)
            make_sample(n, rot + (long long)img * 9, X + img2, ctf + img2, pw ? pw[img] : 1.f, kernel, kx, ky, S);
        const bool self = kx == 0 && ky == 0;
        if (ok && self) deposit_sample(acc, n, kernel, ih, S, true);
        unsigned todo = __ballot_sync(0xffffffffu, ok && !self);
        unsigned now = todo;  // samples of this pass: all that are left, or a half of the tile
        while (todo) {
            const bool mine = (now >> lane & 1u) != 0;
            const int lx = __reduce_min_sync(0xffffffffu, mine ? S.bx : INT_MAX);
            const int ly = __reduce_min_sync(0xffffffffu, mine ? S.by : INT_MAX);
            const int lz = __reduce_min_sync(0xffffffffu, mine ? S.bz : INT_MAX);
            const int ux = __reduce_max_sync(0xffffffffu, mine ? S.bx : INT_MIN);
            const int uy = __reduce_max_sync(0xffffffffu, mine ? S.by : INT_MIN);
            const int uz = __reduce_max_sync(0xffffffffu, mine ? S.bz : INT_MIN);
            const long long ex = (long long)ux - lx + span, ey = (long long)uy - ly + span, ez = (long long)uz - lz + span;
            // compared one factor at a time: the extents of non-rotations are unbounded
            const bool fits = ex <= kBoxCap && ey <= kBoxCap && ez <= kBoxCap && ex * ey * ez <= kBoxCap;
            if (!fits) {
                const unsigned half = now & 0xffffu;
                if (half && half != now) {
                    now = half;
                    continue;
                }
                if (mine) deposit_sample(acc, n, kernel, ih, S, false);
                todo &= ~now;
                now = todo;
                continue;
            }
            const int EX = (int)ex, EY = (int)ey, EZ = (int)ez;
            const int r8 = EX & 7;
            int DX = EX + (r8 < 3 ? 3 - r8 : (r8 > 5 ? 11 - r8 : 0));
            if (DX * EY * EZ > kBoxCap) DX = EX;
            int DXY = DX * EY + ((1 - DX * EY) & 7);
            if (DXY * EZ > kBoxCap) DXY = DX * EY;
            const int vol = DXY * EZ;
            {
                // a lane without a sample in this pass stages a deposit of nothing (at a
                // position off every point: on one, 1/h = infinity would weigh it NaN)
                float wx[3], wy[3], wz[3];
                axis_weights(kernel, ih, mine ? S.fx : 0.25f, wx);
                axis_weights(kernel, ih, mine ? S.fy : 0.25f, wy);
                axis_weights(kernel, ih, mine ? S.fz : 0.25f, wz);
                const int off = mine ? (S.bz - lz) * DXY + (S.by - ly) * DX + (S.bx - lx) : 0;
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    stage[d * kStageRow + lane] = wx[d];
                    stage[(3 + d) * kStageRow + lane] = wy[d];
                    stage[(6 + d) * kStageRow + lane] = wz[d];
                }
                stage[9 * kStageRow + lane] = mine ? S.vre : 0.f;
                stage[10 * kStageRow + lane] = mine ? S.vim : 0.f;
                stage[11 * kStageRow + lane] = mine ? S.vcc : 0.f;
                stage[12 * kStageRow + lane] = __int_as_float(off);
            }
            __syncwarp();
            // deposits: one sample at a time, a lane per support point
            float4 *const mybox = box + (point ? dz * DXY + dy * DX + dx : 0);
            const float *const swx = stage + (point ? dx : 0) * kStageRow;
            const float *const swy = stage + (3 + dy) * kStageRow;
            const float *const swz = stage + (6 + (point ? dz : 0)) * kStageRow;
#pragma unroll 1
            for (int j = 0; j < 32; j += 4) {
                if (!(now >> j & 15u)) continue;
                auto row4 = [&](const float *r) { return *reinterpret_cast<const float4 *>(r + j); };
                const float4 ax = row4(swx), ay = row4(swy), az = row4(swz), of = row4(stage + 12 * kStageRow);
                const float4 re = row4(stage + 9 * kStageRow), im = row4(stage + 10 * kStageRow);
                const float4 cc = row4(stage + 11 * kStageRow);
                auto add = [&](float x, float y, float z, float o, float r, float i, float c) {
                    const float K = x * (y * z);
                    if (point) {
                        float4 *const p = mybox + __float_as_int(o);
                        float4 v = *p;
                        v.x += K * r;
                        v.y += K * i;
                        v.z += K * c;
                        *p = v;
                    }
                    __syncwarp();
                };
                add(ax.x, ay.x, az.x, of.x, re.x, im.x, cc.x);
                add(ax.y, ay.y, az.y, of.y, re.y, im.y, cc.y);
                add(ax.z, ay.z, az.z, of.z, re.z, im.z, cc.z);
                add(ax.w, ay.w, az.w, of.w, re.w, im.w, cc.w);
            }
            // flush: row by row, 10 points by 3 values. Point x goes to the
            // stored half where x (modulo n) <= n/2, its mirror -x, conjugated,
            // where that does; on the planes 0 and n/2 both do.
            const int wx0 = wrap(lx, n), wy0 = wrap(ly, n), wz0 = wrap(lz, n);
            // boxes that cross no plane where an index wraps or changes sides
            // (four of five): one direction, rows and planes at fixed strides
            const bool fwd = wx0 > 0 && wx0 + EX <= nh - 1, back = wx0 >= nh && wx0 + EX <= n;
            if ((fwd || back) && wy0 > 0 && wy0 + EY <= n && wz0 > 0 && wz0 + EZ <= n) {
                const long long sy = fwd ? ys : -ys, sz = (fwd ? zs : -zs) - (long long)EY * sy;
                const unsigned flip = fwd ? 0u : conj;
                for (int x0 = 0; x0 < EX; x0 += 10) {
                    const int px = x0 + fpx;
                    const bool on = lane < 30 && px < EX;
                    double *to = acc + (fwd ? 4LL * (wx0 + px) + fcomp + zs * wz0 + ys * wy0
                                            : 4LL * (n - wx0 - px) + fcomp + zs * (n - wz0) + ys * (n - wy0));
                    const float *src = reinterpret_cast<const float *>(box + (on ? px : 0)) + fcomp;
                    for (int z = 0; z < EZ; z++, to += sz, src += 4 * (DXY - EY * DX)) {
                        int y = 0;
                        for (; y + 4 <= EY; y += 4, src += 16 * DX) {
                            float v[4];
#pragma unroll
                            for (int c = 0; c < 4; c++) v[c] = on ? src[4 * c * DX] : 0.f;
#pragma unroll
                            for (int c = 0; c < 4; c++, to += sy)
                                if (v[c] != 0.f) atomicAdd(to, widen(__uint_as_float(__float_as_uint(v[c]) ^ flip)));
                        }
                        for (; y < EY; y++, src += 4 * DX, to += sy) {
                            const float v = on ? *src : 0.f;
                            if (v != 0.f) atomicAdd(to, widen(__uint_as_float(__float_as_uint(v) ^ flip)));
                        }
                    }
                }
            } else {
                // a lane per box point, every index wrapped on its own (by one
                // addition: the box starts in [0, n) after wrapping its corner,
                // and is no longer than n on any axis for rotations)
                const bool near = EX <= n && EY <= n && EZ <= n;
                const int EXY = EX * EY;
                const int q0 = lane < EXY * EZ ? lane : 0;
                int z = q0 / EXY, y = (q0 - z * EXY) / EX, x = q0 - z * EXY - y * EX;
                // 32 points on
                const int sz = 32 / EXY, sy = (32 - sz * EXY) / EX, sx = 32 - sz * EXY - sy * EX;
                for (int q = lane; q < EXY * EZ; q += 32) {
                    const float4 v = box[z * DXY + y * DX + x];
                    if (v.x != 0.f || v.y != 0.f || v.z != 0.f) {
                        const double re = widen(v.x), im = widen(v.y), nn = widen(v.z);
                        if (near) {
                            const int ax = wx0 + x < n ? wx0 + x : wx0 + x - n;
                            const int ay = wy0 + y < n ? wy0 + y : wy0 + y - n;
                            const int az = wz0 + z < n ? wz0 + z : wz0 + z - n;
                            if (ax < nh) {
                                double *p = acc + (4LL * ax + zs * az + ys * ay);
                                atomicAdd(p, re);
                                atomicAdd(p + 1, im);
                                atomicAdd(p + 2, nn);
                            }
                            const int mx = ax == 0 ? 0 : n - ax;
                            if (mx < nh) {
                                double *p = acc + (4LL * mx + zs * (az == 0 ? 0 : n - az) + ys * (ay == 0 ? 0 : n - ay));
                                atomicAdd(p, re);
                                atomicAdd(p + 1, -im);
                                atomicAdd(p + 2, nn);
                            }
                        } else {
                            deposit(acc, n, lx + x, ly + y, lz + z, re, im, nn, false);
                        }
                    }
                    x += sx;
                    y += sy;
                    z += sz;
                    if (x >= EX) {
                        x -= EX;
                        y++;
                    }
                    if (y >= EY) {
                        y -= EY;
                        z++;
                    }
                }
            }
            __syncwarp();
            for (int q = lane; q < vol; q += 32) box[q] = zero4;
            __syncwarp();  // the box and the stage are reused
            todo &= ~now;
            now = todo;
        }
    }
}

__global__ void finish_kernel(int n, const double *__restrict__ acc, float2 *y_half, float *N_half)
{
    const int nh = n / 2 + 1;
    const long long total = (long long)n * n * nh;
    const double V = (double)n * n * n;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
         q += (long long)gridDim.x * blockDim.x) {
        const int kx = (int)(q % nh);
        const int ky = (int)((q / nh) % n);
        const int kz = (int)(q / ((long long)nh * n));
        const double *a = acc + 4 * q;
        const double w = a[2];
        const double sgn = ((kx + ky + kz) & 1) ? -1.0 : 1.0;
        float2 y = make_float2(0.f, 0.f);
        if (w > 0) {
            // 1/sqrt(w) to 44 bits: a float32 estimate and one Newton step in
            // double (the results are float32; double sqrt and division kept
            // the narrow FP64 pipe busy for 30 operations a point)
            const float wf = (float)w;
            double s;
            if (wf > 1e-37f && wf < 1e38f) {
                const double r = (double)rsqrtf(wf);
                s = sgn * fma(0.5 * r, fma(-w * r, r, 1.0), r);
            } else {
                s = sgn / sqrt(w);
            }
            y = make_float2((float)(a[0] * s), (float)(a[1] * s));
        }
        y_half[q] = y;
        N_half[q] = (float)(V * w);
    }
}

int blocks_for(long long work)
{
    const long long b = (work + kThreads - 1) / kThreads;
    return (int)(b < kMaxBlocks ? (b > 0 ? b : 1) : kMaxBlocks);
}

bool on_device(const void *p)
{
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace

struct spg_grid {
    int n = 0, kernel = 0;
    float h = 2.f;
    cudaStream_t stream = nullptr;
    double *acc = nullptr;  // [n][n][n/2+1][4]
    void *stage = nullptr;  // device copies of host inputs / outputs
    size_t stage_bytes = 0;
    long long images = 0;
    std::string err = "no error";
    size_t half() const { return (size_t)n * n * (n / 2 + 1); }
};

namespace {

spg_status gfail(spg_grid *g, spg_status s, const std::string &m)
{
    (g ? g->err : g_grid_err) = m;
    return s;
}

spg_status cuda_fail(spg_grid *g, cudaError_t e, const char *what)
{
    cudaGetLastError();
    return gfail(g, e == cudaErrorMemoryAllocation ? SPG_ENOMEM : SPG_ECUDA,
                 std::string(what) + ": " + cudaGetErrorString(e));
}

// Make sure the staging buffer holds `bytes`; waits for the stream before
// replacing a buffer that queued work may still read.
cudaError_t ensure_stage(spg_grid *g, size_t bytes)
{
    if (bytes <= g->stage_bytes) return cudaSuccess;
    cudaError_t e = cudaStreamSynchronize(g->stream);
    if (e != cudaSuccess) return e;
    if (g->stage) cudaFree(g->stage);
    g->stage = nullptr;
    g->stage_bytes = 0;
    e = cudaMalloc(&g->stage, bytes);
    if (e == cudaSuccess) g->stage_bytes = bytes;
    return e;
}

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

}  // namespace

extern "C" spg_status spg_grid_create(int n, int kernel, float h, void *stream, spg_grid **out)
{
    SPG_TRACE();
    if (!out) return gfail(nullptr, SPG_EINVAL, "spg_grid_create: null output");
    *out = nullptr;
    if (n < 4 || n % 2 || (kernel != 0 && kernel != 1) || !(h > 0.f))
        return gfail(nullptr, SPG_EINVAL, "spg_grid_create: bad arguments (even n >= 4, kernel 0 or 1, h > 0)");
    if ((long long)n * n * n > (1LL << 31)) return gfail(nullptr, SPG_EINVAL, "spg_grid_create: volume too large");
    spg_grid *g = new spg_grid;
    g->n = n;
    g->kernel = kernel;
    g->h = h;
    g->stream = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMalloc(&g->acc, g->half() * 4 * sizeof(double));
    if (e == cudaSuccess) e = cudaMemsetAsync(g->acc, 0, g->half() * 4 * sizeof(double), g->stream);
    if (e != cudaSuccess) {
        spg_status s = cuda_fail(nullptr, e, "spg_grid_create");
        if (g->acc) cudaFree(g->acc);
        delete g;
        return s;
    }
    *out = g;
    return SPG_OK;
}

extern "C" spg_status spg_grid_add(spg_grid *g, int m, const float *rot, const void *X, const float *ctf,
                                   const float *pw)
{
    SPG_TRACE();
    if (!g) return gfail(nullptr, SPG_EINVAL, "spg_grid_add: null accumulator");
    if (m < 1 || !rot || !X || !ctf) return gfail(g, SPG_EINVAL, "spg_grid_add: m >= 1 and non-null arrays");
    const int n = g->n;
    const size_t img = (size_t)m * n * n;
    struct In {
        const void *src;
        size_t bytes;
        const void *dev;
        bool host;
    } in[4] = {{rot, (size_t)m * 9 * sizeof(float), nullptr, false},
               {X, img * sizeof(float2), nullptr, false},
               {ctf, img * sizeof(float), nullptr, false},
               {pw, pw ? (size_t)m * sizeof(float) : 0, nullptr, false}};
    size_t need = 0;
    for (auto &a : in) {
        a.host = a.src && !on_device(a.src);
        if (a.host) need += align256(a.bytes);
    }
    cudaError_t e = ensure_stage(g, need);
    if (e != cudaSuccess) return cuda_fail(g, e, "spg_grid_add: staging buffer");
    size_t off = 0;
    for (auto &a : in) {
        if (!a.host) {
            a.dev = a.src;
            continue;
        }
        void *dst = static_cast<char *>(g->stage) + off;
        e = cudaMemcpyAsync(dst, a.src, a.bytes, cudaMemcpyHostToDevice, g->stream);
        if (e != cudaSuccess) return cuda_fail(g, e, "spg_grid_add: copy");
        a.dev = dst;
        off += align256(a.bytes);
    }
    // the warps' boxes exceed the default 48 KB (set per call: per device)
    constexpr int smem = kWarps * kWarpSmem;
    e = cudaFuncSetAttribute(scatter_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return cuda_fail(g, e, "spg_grid_add: configure");
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long long tiles =
        (long long)m * ((n / 2 + kTileY - 1) / kTileY) * ((n + kTileX - 1) / kTileX);
    const int grid = (int)std::min<long long>((tiles + kWarps - 1) / kWarps, (long long)std::max(nsm, 1) * 2);
    scatter_tile_kernel<<<grid, kWarps * 32, smem, g->stream>>>(
        n, m, static_cast<const float *>(in[0].dev), static_cast<const float2 *>(in[1].dev),
        static_cast<const float *>(in[2].dev), static_cast<const float *>(in[3].dev), g->kernel, g->h, g->acc);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(g, e, "spg_grid_add: launch");
    g->images += m;
    return SPG_OK;
}

extern "C" spg_status spg_grid_finish(spg_grid *g, void *y_half, float *N_half)
{
    SPG_TRACE();
    if (!g) return gfail(nullptr, SPG_EINVAL, "spg_grid_finish: null accumulator");
    if (!y_half || !N_half) return gfail(g, SPG_EINVAL, "spg_grid_finish: null output");
    const size_t half = g->half();
    const bool dy = on_device(y_half), dn = on_device(N_half);
    const size_t ybytes = dy ? 0 : align256(half * sizeof(float2));
    const size_t need = ybytes + (dn ? 0 : align256(half * sizeof(float)));
    cudaError_t e = ensure_stage(g, need);
    if (e != cudaSuccess) return cuda_fail(g, e, "spg_grid_finish: staging buffer");
    float2 *yo = dy ? static_cast<float2 *>(y_half) : static_cast<float2 *>(g->stage);
    float *no = dn ? N_half : reinterpret_cast<float *>(static_cast<char *>(g->stage) + ybytes);
    finish_kernel<<<blocks_for((long long)half), kThreads, 0, g->stream>>>(g->n, g->acc, yo, no);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(g, e, "spg_grid_finish: launch");
    if (!dy) {
        e = cudaMemcpyAsync(y_half, yo, half * sizeof(float2), cudaMemcpyDeviceToHost, g->stream);
        if (e != cudaSuccess) return cuda_fail(g, e, "spg_grid_finish: copy");
    }
    if (!dn) {
        e = cudaMemcpyAsync(N_half, no, half * sizeof(float), cudaMemcpyDeviceToHost, g->stream);
        if (e != cudaSuccess) return cuda_fail(g, e, "spg_grid_finish: copy");
    }
    e = cudaStreamSynchronize(g->stream);
    if (e != cudaSuccess) return cuda_fail(g, e, "spg_grid_finish: synchronise");
    return SPG_OK;
}

extern "C" spg_status spg_grid_reset(spg_grid *g)
{
    SPG_TRACE();
    if (!g) return gfail(nullptr, SPG_EINVAL, "spg_grid_reset: null accumulator");
    cudaError_t e = cudaMemsetAsync(g->acc, 0, g->half() * 4 * sizeof(double), g->stream);
    if (e != cudaSuccess) return cuda_fail(g, e, "spg_grid_reset");
    g->images = 0;
    return SPG_OK;
}

extern "C" long long spg_grid_count(const spg_grid *g) { return g ? g->images : 0; }

extern "C" const char *spg_grid_last_error(const spg_grid *g) { return g ? g->err.c_str() : g_grid_err.c_str(); }

extern "C" void spg_grid_destroy(spg_grid *g)
{
    SPG_TRACE();
    if (!g) return;
    cudaStreamSynchronize(g->stream);
    if (g->acc) cudaFree(g->acc);
    if (g->stage) cudaFree(g->stage);
    delete g;
}

extern "C" const char *spg_backproject_last_error(void) { return g_grid_err.c_str(); }

extern "C" spg_status spg_backproject(int n, int m, const float *rot, const void *X, const float *ctf,
                                      const float *pw, int kernel, float h, void *y_half, float *N_half, void *stream)
{
    SPG_TRACE();
    spg_grid *g = nullptr;
    spg_status s = spg_grid_create(n, kernel, h, stream, &g);
    if (s != SPG_OK) return s;  // message already in g_grid_err
    s = spg_grid_add(g, m, rot, X, ctf, pw);
    if (s == SPG_OK) s = spg_grid_finish(g, y_half, N_half);
    if (s != SPG_OK) g_grid_err = g->err;
    spg_grid_destroy(g);
    return s;
}
