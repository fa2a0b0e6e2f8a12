// Auxiliary kernels of the GB300 SPG solver: input validation and dtype
// conversion, the re-weighting pass (Eq. 11), the objective (Eq. 14 / 31),
// the strong-convexity certificate, the passes of the adjoint of one step,
// and the plain step used under alternative readings of the paper.
//
// All use plain global loads.
// The adopted reading's re-weighting and objective, the validation and the
// anchor march over z: a CTA takes 8 rows (a warp each) of a 128-voxel chunk over
// a run of planes (AuxParams::items), each lane 4 voxels by 16-byte loads, the
// plane below kept in registers and the loads of several planes issued
// together; the certificate marches as the adjoint passes do. The kernels of the
// alternative readings and the parameter scales run AUX_SEG CTAs per z-plane
// (one per row segment).
// Every reduction keeps one partial per CTA, and the last CTA to finish sums
// the partials of each volume in a fixed order, so the results are
// deterministic; the adjoint passes keep one scalar partial per CTA, summed per
// step by adjoint_scalars_kernel (the host adds the steps' results). No kernel
// here waits on another CTA of its grid; the adjoint passes, launched ahead of
// the end of the pass before them, wait for that grid (griddepcontrol.wait).
//
// Sums across a CTA run in float-float (spg_ff.cuh): with double shuffles
// GB300's narrow FP64 pipe took most of these passes' time on small volumes.
// Measured (whole calls, host work included), a CTA per row segment with double
// sums -> march with float-float sums: re-weighting 64^3 23.0 -> 12.1 us,
// 101 x 147 x 183 42.9 -> 25.2, 256^3 114 -> 62, 512^3 520 -> 349 (12 bytes a
// voxel at the copy rate: 237); objective 50.1 -> 38.2, 61.3 -> 50.3, 124 -> 100,
// 495 -> 436 (20 bytes: 396); spg_set_data with its validation 45.2 -> 33.3,
// 84.4 -> 71.9, 146 -> 98, 717 -> 518 (host arrays and reversed contexts still go
// this way; device arrays are taken in by one pass, ingest_kernel).
#include <cuda_bf16.h>

#include <algorithm>

#include "spg_ff.cuh"
#include "spg_internal.h"

namespace spg {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int AUX_THREADS = 256;

// Each z-plane is split into AUX_SEG row segments, one CTA each; partial sums
// are kept per segment (index plane * AUX_SEG + segment).
__device__ __forceinline__ void seg_rows(int ny, int seg, int &r0, int &r1)
{
    r0 = (int)((long long)ny * seg / AUX_SEG);
    r1 = (int)((long long)ny * (seg + 1) / AUX_SEG);
}

struct KSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float v)
    {
        float y = v - c;
        float t = s + y;
        c = (t - s) - y;
        s = t;
    }
    __device__ __forceinline__ double value() const { return (double)s - (double)c; }
    __device__ __forceinline__ ff::FF pair() const { return {s, -c}; }
};

__device__ __forceinline__ float ld_data(const void *p, bool bf16, long long i)
{
    if (bf16) return __uint_as_float(((uint32_t) reinterpret_cast<const uint16_t *>(p)[i]) << 16);
    return reinterpret_cast<const float *>(p)[i];
}

// Block-wide sum of up to 4 doubles in a fixed order; result valid in thread 0.
template <int N>
__device__ void block_sum(double (&v)[N], double *scratch /* 32*N */)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < N; q++) v[q] += __shfl_down_sync(FULL, v[q], o);
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < N; q++) scratch[warp * N + q] = v[q];
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = blockDim.x / 32;
        for (int q = 0; q < N; q++) {
            double a = 0;
            for (int k = 0; k < nw; k++) a += scratch[k * N + q];
            v[q] = a;
        }
    }
    __syncthreads();
}

__device__ __forceinline__ double block_max(double v, double *scratch)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(FULL, v, o));
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = blockDim.x / 32;
        for (int k = 0; k < nw; k++) v = fmax(v, scratch[k]);
    }
    __syncthreads();
    return v;
}

// CTA sums of 4 float-float values (double where those could overflow), fixed
// order; lane q < 4 of warp 0 returns quantity q. red: 4 doubles per warp.
__device__ __forceinline__ double block_sum4(const ff::FF (&v)[4], double *red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const bool big = ff::too_big(v[0]) || ff::too_big(v[1]) || ff::too_big(v[2]) || ff::too_big(v[3]);
    double r = 0.0;
    if (!__syncthreads_or(big ? 1 : 0)) {
        ff::FF *const rf = reinterpret_cast<ff::FF *>(red);
        const ff::FF s = ff::warp_sum4(v, lane);
        if ((lane & 7) == 0) rf[warp * 4 + (lane >> 3)] = s;
        __syncthreads();
        if (warp == 0) r = ff::to_double(ff::cross_warp_sum4(rf, nw, lane, ff::FF{0.f, 0.f}));
    } else {
        const double w[4] = {ff::to_double(v[0]), ff::to_double(v[1]), ff::to_double(v[2]), ff::to_double(v[3])};
        const double s = ff::warp_sum4(w, lane);
        if ((lane & 7) == 0) red[warp * 4 + (lane >> 3)] = s;
        __syncthreads();
        if (warp == 0) r = ff::cross_warp_sum4(red, nw, lane, 0.0);
    }
    __syncthreads();
    return r;
}

// CTA maximum of floats (exact); valid in thread 0. red: one float per warp.
__device__ __forceinline__ float block_fmax(float v, float *red)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < (int)(blockDim.x >> 5) ? red[lane] : v;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
    }
    __syncthreads();
    return v;
}

// A CTA's partial of a march: three sums and, as a float in the first slot, a
// maximum (or a fourth sum).
__device__ __forceinline__ float *part_max(double *pp) { return reinterpret_cast<float *>(pp); }

// Last CTA: sums (slots 1 .. 3, or 0 .. 3 without a maximum) and the maximum of
// the partials [b, e) of one volume, by `nw` warps of which this is warp w, in
// a fixed order: every lane gets all values. With nw > 1 the warps' results
// meet in `red` (4 doubles a warp) behind CTA barriers.
__device__ __forceinline__ void part_total(double *part, int b, int e, int w, int nw, bool has_max, double *red,
                                           double (&a)[4], float &mx)
{
    const int lane = threadIdx.x & 31;
    a[0] = a[1] = a[2] = a[3] = 0.0;
    mx = 0.f;
    for (int q = b + w * 32 + lane; q < e; q += 32 * nw) {
        double *pp = part + (long long)q * 4;
        if (has_max) mx = fmaxf(mx, __ldcg(part_max(pp)));
        else a[0] += __ldcg(pp);
        a[1] += __ldcg(pp + 1);
        a[2] += __ldcg(pp + 2);
        a[3] += __ldcg(pp + 3);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, o));
    double s = ff::warp_sum4(a, lane);
    if (nw > 1) {
        float *const rm = reinterpret_cast<float *>(red + 32 * 4);
        if ((lane & 7) == 0) red[w * 4 + (lane >> 3)] = s;
        if (lane == 0) rm[w] = mx;
        __syncthreads();
        s = ff::cross_warp_sum4(red, nw, lane, 0.0);
        s = __shfl_sync(FULL, s, lane >> 3);
        for (int k = 0; k < nw; k++) mx = fmaxf(mx, rm[k]);
        __syncthreads();
    }
#pragma unroll
    for (int c = 0; c < 4; c++) a[c] = __shfl_sync(FULL, s, 8 * c);
}

// Last-CTA election on a counter; returns true in every thread of the last CTA.
__device__ bool last_block(unsigned int *ticket, int *flag_smem)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned t = atomicAdd(ticket, 1u);
        *flag_smem = (t == gridDim.x - 1) ? 1 : 0;
    }
    __syncthreads();
    const bool last = *flag_smem != 0;
    if (last) __threadfence();
    return last;
}

// Sec. 2.5 scales: sum (w b)^2, sum w, max w, min w of one volume.
__global__ void scales_kernel(AuxParams a, int vol, const void *b, const void *w, bool bf16)
{
    __shared__ double scratch[32 * 4];
    __shared__ int flag;
    const VolDesc V = a.vols[vol];
    const int z = blockIdx.x / AUX_SEG;
    int r0, r1;
    seg_rows(V.ny, blockIdx.x % AUX_SEG, r0, r1);
    KSum s2, sw;
    double mx = 0.0, mn = INFINITY;
    for (int t = threadIdx.x; t < (r1 - r0) * V.nx; t += blockDim.x) {
        const int x = t % V.nx, y = r0 + t / V.nx;
        const long long i = V.off + ((long long)z * V.ny + y) * V.pitch + x;
        const float wv = ld_data(w, bf16, i), bv = ld_data(b, bf16, i);
        const float n = wv * bv;
        s2.add(n * n);
        sw.add(wv);
        mx = fmax(mx, (double)wv);
        mn = fmin(mn, (double)wv);
    }
    mx = block_max(mx, scratch);
    const double nmn = block_max(-mn, scratch);
    double v[2] = {s2.value(), sw.value()};
    block_sum<2>(v, scratch);
    if (threadIdx.x == 0) {
        double *pp = a.plane_part + (long long)blockIdx.x * 4;
        pp[0] = v[0];
        pp[1] = v[1];
        pp[2] = mx;
        pp[3] = -nmn;
    }
    if (!last_block(&a.st->ticket_aux, &flag)) return;
    double c2[2] = {0, 0}, m = 0, n = INFINITY;
    for (int q = threadIdx.x; q < V.nz * AUX_SEG; q += blockDim.x) {
        const double *pp = a.plane_part + (long long)q * 4;
        c2[0] += __ldcg(pp + 0);
        c2[1] += __ldcg(pp + 1);
        m = fmax(m, __ldcg(pp + 2));
        n = fmin(n, __ldcg(pp + 3));
    }
    block_sum<2>(c2, scratch);
    m = block_max(m, scratch);
    n = -block_max(-n, scratch);
    if (threadIdx.x == 0) {
        const double q2 = c2[0], qw = c2[1];
        const double cnt = (double)V.nx * V.ny * V.nz;
        double *o = a.vol_out + (long long)vol * 8;
        o[0] = sqrt(q2 / cnt);
        o[1] = qw / cnt;
        o[2] = m;
        o[3] = n;
        a.st->ticket_aux = 0;
        __threadfence();
    }
}

__global__ void to_bf16_kernel(const float *src, uint16_t *dst, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        __nv_bfloat16 h = __float2bfloat16_rn(src[i]);
        dst[i] = *reinterpret_cast<uint16_t *>(&h);
    }
}

__global__ void to_f32_kernel(const uint16_t *src, float *dst, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = __uint_as_float(((uint32_t)src[i]) << 16);
}

// ---------------- stencil helpers (plain global loads) ----------------

// Value of u = x_k + beta (x_k - x_{k-1}) is never formed; differences are
// taken of x_k and of d = x_k - x_{k-1} separately (one rounding each).
struct Field {
    const float *xk, *xkm1;   // xkm1 may be null (then d = 0, unless dk is given)
    float beta;
    const float *dk = nullptr;  // stored increment x_k - x_{k-1}, if any
    __device__ __forceinline__ float x(long long i) const { return xk[i]; }
    __device__ __forceinline__ float d(long long i) const
    {
        return dk ? dk[i] : (xkm1 ? xk[i] - xkm1[i] : 0.f);
    }
};

// D u at (x, y, z) under the SPG_READ_* flags of the volume (forward
// differences and/or a periodic boundary); kept out of line so the adopted
// reading's code below stays small.
__device__ __noinline__ void grad_at_readings(const VolDesc &V, const Field &F, int x, int y, int z, float g[3])
{
    const long long i = V.off + ((long long)z * V.ny + y) * V.pitch + x;
    const float xc = F.x(i), dc = F.d(i);
    const bool fwd = (V.readings & SPG_READ_FORWARD) != 0, per = (V.readings & SPG_READ_PERIODIC) != 0;
    const int co[3] = {x, y, z}, ext[3] = {V.nx, V.ny, V.nz};
    const long long stp[3] = {1, V.pitch, (long long)V.pitch * V.ny};
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int c = co[a], n = ext[a];
        long long j;
        if (!fwd) {
            if (c >= 1) j = i - stp[a];
            else if (per && n > 1) j = i + (long long)(n - 1) * stp[a];
            else { g[a] = 0.f; continue; }
            g[a] = (xc - F.x(j)) + F.beta * (dc - F.d(j));
        } else {
            if (c + 1 <= n - 1) j = i + stp[a];
            else if (per && n > 1) j = i - (long long)(n - 1) * stp[a];
            else { g[a] = 0.f; continue; }
            g[a] = (F.x(j) - xc) + F.beta * (F.d(j) - dc);
        }
    }
}

// D u at (x, y, z) in volume V. Adopted reading: backward differences that
// vanish on the first plane of each axis (Eq. 12).
__device__ __forceinline__ void grad_at(const VolDesc &V, const Field &F, int x, int y, int z, float g[3])
{
    if (V.readings != 0) {
        grad_at_readings(V, F, x, y, z, g);
        return;
    }
    const long long i = V.off + ((long long)z * V.ny + y) * V.pitch + x;
    const float xc = F.x(i), dc = F.d(i);
    g[0] = x >= 1 ? (xc - F.x(i - 1)) + F.beta * (dc - F.d(i - 1)) : 0.f;
    g[1] = y >= 1 ? (xc - F.x(i - V.pitch)) + F.beta * (dc - F.d(i - V.pitch)) : 0.f;
    const long long ps = (long long)V.pitch * V.ny;
    g[2] = z >= 1 ? (xc - F.x(i - ps)) + F.beta * (dc - F.d(i - ps)) : 0.f;
}

// p = omtv * D u / max(mu, |D u|) at (x, y, z) (without omtv under
// SPG_READ_POST_DIV); zero outside the volume.
__device__ __forceinline__ void p_at(const VolDesc &V, const Field &F, const float *omtv, int x, int y, int z,
                                     float p[3])
{
    if (x < 0 || y < 0 || z < 0 || x >= V.nx || y >= V.ny || z >= V.nz) {
        p[0] = p[1] = p[2] = 0.f;
        return;
    }
    float g[3];
    grad_at(V, F, x, y, z, g);
    const long long i = V.off + ((long long)z * V.ny + y) * V.pitch + x;
    const float s2 = g[0] * g[0] + g[1] * g[1] + g[2] * g[2];
    const float om = (V.readings & SPG_READ_POST_DIV) ? 1.0f : omtv[i];
    const float sc = om * fminf(1.0f / V.mu, rsqrtf(s2));
    p[0] = g[0] * sc;
    p[1] = g[1] * sc;
    p[2] = g[2] * sc;
}

// (D^T p)(x, y, z) with p evaluated on the fly (Eq. 17 for the adopted
// reading; the adjoint of the selected D otherwise, times omtv under
// SPG_READ_POST_DIV).
__device__ __forceinline__ float div_at(const VolDesc &V, const Field &F, const float *omtv, int x, int y, int z)
{
    float pc[3], px[3], pyv[3], pz[3];
    p_at(V, F, omtv, x, y, z, pc);
    if (V.readings == 0) {
        p_at(V, F, omtv, x + 1, y, z, px);
        p_at(V, F, omtv, x, y + 1, z, pyv);
        p_at(V, F, omtv, x, y, z + 1, pz);
        return (pc[0] - px[0]) + (pc[1] - pyv[1]) + (pc[2] - pz[2]);
    }
    const bool fwd = (V.readings & SPG_READ_FORWARD) != 0, per = (V.readings & SPG_READ_PERIODIC) != 0;
    // neighbour along each axis: successor (backward D) or predecessor (forward D),
    // wrapped under the periodic boundary, else possibly outside (p = 0 there)
    auto nb = [&](int c, int n) {
        const int d = fwd ? c - 1 : c + 1;
        return per ? (d + n) % n : d;
    };
    p_at(V, F, omtv, nb(x, V.nx), y, z, px);
    p_at(V, F, omtv, x, nb(y, V.ny), z, pyv);
    p_at(V, F, omtv, x, y, nb(z, V.nz), pz);
    float r = fwd ? (px[0] - pc[0]) + (pyv[1] - pc[1]) + (pz[2] - pc[2])
                  : (pc[0] - px[0]) + (pc[1] - pyv[1]) + (pc[2] - pz[2]);
    if (V.readings & SPG_READ_POST_DIV) r *= omtv[V.off + ((long long)z * V.ny + y) * V.pitch + x];
    return r;
}

// ---------------- row-vector walks for the adopted reading ----------------
// The re-weighting and the objective read every voxel once plus three
// neighbours; with one voxel per thread they wait on memory latency. The
// adopted reading's kernels instead walk a row segment in 128-voxel chunks:
// each warp takes a chunk of a row, each lane 4 consecutive voxels (16-byte
// loads: rows start 32-byte aligned, the pitch being a multiple of 8 and
// volume offsets of 64 elements). The x-neighbour of a lane's first voxel
// comes from the lane before it (the first lane of a chunk loads it).
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

__device__ __forceinline__ float4 ld4_data(const void *p, bool bf16, long long i)
{
    if (!bf16) return ld4(reinterpret_cast<const float *>(p) + i);
    const uint2 u = *reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(p) + i);
    return make_float4(__uint_as_float((u.x & 0xffffu) << 16), __uint_as_float(u.x & 0xffff0000u),
                       __uint_as_float((u.y & 0xffffu) << 16), __uint_as_float(u.y & 0xffff0000u));
}

__device__ __forceinline__ void unpack4(const float4 v, float (&o)[4])
{
    o[0] = v.x;
    o[1] = v.y;
    o[2] = v.z;
    o[3] = v.w;
}

// Where a thread of a march works: its row, first voxel and planes.
struct March {
    int x0, y, z0, z1, lane;
    bool act;      // row and first voxel inside the volume
    long long i;   // element index of voxel x0 of the row on plane z0
    long long PS;  // plane stride
};

__device__ __forceinline__ March march_place(const VolDesc &V, const WorkItem &W)
{
    March M;
    M.lane = threadIdx.x & 31;
    M.x0 = W.x0 + 4 * M.lane;
    M.y = W.y0 + (threadIdx.x >> 5);
    M.z0 = W.z0;
    M.z1 = W.z1;
    M.act = M.y < V.ny && M.x0 < V.nx;
    M.PS = (long long)V.pitch * V.ny;
    M.i = V.off + ((long long)W.z0 * V.ny + (M.y < V.ny ? M.y : 0)) * V.pitch + (M.x0 < V.nx ? M.x0 : 0);
    return M;
}

// ---------------- validation ----------------
__device__ __forceinline__ void st_data(void *p, bool bf16, long long i, float v)
{
    if (bf16) {
        __nv_bfloat16 h = __float2bfloat16_rn(v);
        reinterpret_cast<uint16_t *>(p)[i] = *reinterpret_cast<uint16_t *>(&h);
    } else {
        reinterpret_cast<float *>(p)[i] = v;
    }
}

// 4 values in one store (rows start 32-byte aligned; a value widened from
// bfloat16 goes back unchanged).
template <bool BF16>
__device__ __forceinline__ void st4_data(void *p, long long i, const float (&v)[4])
{
    if constexpr (BF16) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(v[0], v[1]), hi = __floats2bfloat162_rn(v[2], v[3]);
        uint2 u;
        u.x = *reinterpret_cast<const uint32_t *>(&lo);
        u.y = *reinterpret_cast<const uint32_t *>(&hi);
        *reinterpret_cast<uint2 *>(reinterpret_cast<uint16_t *>(p) + i) = u;
    } else {
        *reinterpret_cast<float4 *>(reinterpret_cast<float *>(p) + i) = make_float4(v[0], v[1], v[2], v[3]);
    }
}

// What validation collects: max and min w (finite ones), values of w that are
// not finite and positive, values of b that are not finite.
struct DataCheck {
    float mx = 0.f, nmn = -INFINITY;
    int bad_w = 0, bad_b = 0;
    __device__ __forceinline__ void add(float bv, float wv)
    {
        const bool wfin = isfinite(wv);
        bad_w += (!(wv > 0.f) || !wfin) ? 1 : 0;
        bad_b += isfinite(bv) ? 0 : 1;
        if (wfin) {
            mx = fmaxf(mx, wv);
            nmn = fmaxf(nmn, -wv);
        }
    }
};

// The CTA's check into its partial; the last CTA's totals into vol_out and max w.
__device__ void check_finish(const AuxParams &a, int vol, const VolDesc &V, DataCheck c, double *maxw_out)
{
    __shared__ float red[32];
    __shared__ int cnt[2], flag;
    if (threadIdx.x < 2) cnt[threadIdx.x] = 0;
    const float mx = block_fmax(c.mx, red), nm = block_fmax(c.nmn, red);
    c.bad_w = __reduce_add_sync(FULL, c.bad_w);
    c.bad_b = __reduce_add_sync(FULL, c.bad_b);
    if ((threadIdx.x & 31) == 0 && (c.bad_w | c.bad_b)) {
        atomicAdd(&cnt[0], c.bad_w);
        atomicAdd(&cnt[1], c.bad_b);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float *pp = part_max(a.plane_part + (long long)blockIdx.x * 4);
        pp[0] = mx;
        pp[1] = nm;
        pp[2] = __int_as_float(cnt[0]);
        pp[3] = __int_as_float(cnt[1]);
    }
    if (!last_block(&a.st->ticket_aux, &flag)) return;
    float m = 0.f, n = -INFINITY;
    int bw = 0, bb = 0;
    for (int q = threadIdx.x; q < V.aux_end - V.aux_begin; q += blockDim.x) {
        const float4 p = __ldcg(reinterpret_cast<const float4 *>(a.plane_part + (long long)q * 4));
        m = fmaxf(m, p.x);
        n = fmaxf(n, p.y);
        bw |= __float_as_int(p.z);
        bb |= __float_as_int(p.w);
    }
    m = block_fmax(m, red);
    n = block_fmax(n, red);
    const bool any_w = __syncthreads_or(bw) != 0, any_b = __syncthreads_or(bb) != 0;
    if (threadIdx.x != 0) return;
    double *o = a.vol_out + (long long)vol * 8;
    o[0] = m;
    o[1] = -n;
    o[2] = any_w ? 1.0 : 0.0;  // whether there are any; the counts are not used
    o[3] = any_b ? 1.0 : 0.0;
    maxw_out[vol] = m;
    a.st->ticket_aux = 0;
    __threadfence();
}

// The stored b and w of volume `vol`, over its march items.
__global__ void __launch_bounds__(AUX_THREADS)
    validate_kernel(AuxParams a, int vol, const void *b, const void *w, bool bf16, double *maxw_out)
{
    const VolDesc V = a.vols[vol];
    const WorkItem W = a.items[V.aux_begin + blockIdx.x];
    const March M = march_place(V, W);
    DataCheck C;
    constexpr int U = 4;
    for (int z = M.z0; z < M.z1; z += U) {
        float4 bv[U], wv[U];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (M.act && z + u < M.z1) {
                const long long i = M.i + (long long)(z + u - M.z0) * M.PS;
                bv[u] = ld4_data(b, bf16, i);
                wv[u] = ld4_data(w, bf16, i);
            }
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (!(M.act && z + u < M.z1)) continue;
            float bb[4], ww[4];
            unpack4(bv[u], bb);
            unpack4(wv[u], ww);
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (M.x0 + q < V.nx) C.add(bb[q], ww[q]);
        }
    }
    check_finish(a, vol, V, C, maxw_out);
}

// Device-resident b and w: copied (or converted) into the context's layout and
// validated in one pass, 16 bytes a voxel, instead of a copy of each and a pass
// over the copies, 24 (and 4 more with a staged conversion). VEC: rows of the
// caller's arrays start on 4-element boundaries and a lane takes 4 neighbouring
// voxels; otherwise a lane takes voxels 32 apart, so that any row start gives
// coalesced accesses (and rows narrower than their pitch need no 2-D copy).
// Checked are the values as stored. Whole call, before -> after:
// 101 x 147 x 183 72 -> 33 us, 256^3 98 -> 69, 512^3 518 -> 343 (at the copy rate 317).
template <bool SRC16, bool DST16, bool VEC>
__global__ void __launch_bounds__(AUX_THREADS)
    ingest_kernel(AuxParams a, int vol, const void *__restrict__ sb, const void *__restrict__ sw, void *b, void *w,
                  double *maxw_out)
{
    const VolDesc V = a.vols[vol];
    const WorkItem W = a.items[V.aux_begin + blockIdx.x];
    const int lane = threadIdx.x & 31, y = W.y0 + (threadIdx.x >> 5);
    DataCheck C;
    auto stored = [](float v) {
        return DST16 && !SRC16 ? __uint_as_float((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(v)) << 16) : v;
    };
    if (y < V.ny) {
        constexpr int U = VEC ? 4 : 2;
        const long long sps = (long long)V.nx * V.ny, dps = (long long)V.pitch * V.ny;
        const long long si = (long long)W.z0 * sps + (long long)y * V.nx + W.x0;
        const long long di = V.off + (long long)W.z0 * dps + (long long)y * V.pitch + W.x0;
        for (int z = W.z0; z < W.z1; z += U) {
            float bv[U][4], wv[U][4];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const long long i = si + (long long)(z + u - W.z0) * sps;
                if constexpr (VEC) {
                    if (z + u < W.z1 && W.x0 + 4 * lane < V.nx) {
                        unpack4(ld4_data(sb, SRC16, i + 4 * lane), bv[u]);
                        unpack4(ld4_data(sw, SRC16, i + 4 * lane), wv[u]);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 4; q++)
                        if (z + u < W.z1 && W.x0 + lane + 32 * q < V.nx) {
                            bv[u][q] = ld_data(sb, SRC16, i + lane + 32 * q);
                            wv[u][q] = ld_data(sw, SRC16, i + lane + 32 * q);
                        }
                }
            }
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (z + u >= W.z1) break;
                const long long i = di + (long long)(z + u - W.z0) * dps;
                if constexpr (VEC) {
                    if (W.x0 + 4 * lane < V.nx) {
#pragma unroll
                        for (int q = 0; q < 4; q++) C.add(stored(bv[u][q]), stored(wv[u][q]));
                        st4_data<DST16>(b, i + 4 * lane, bv[u]);
                        st4_data<DST16>(w, i + 4 * lane, wv[u]);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 4; q++)
                        if (W.x0 + lane + 32 * q < V.nx) {
                            C.add(stored(bv[u][q]), stored(wv[u][q]));
                            st_data(b, DST16, i + lane + 32 * q, bv[u][q]);
                            st_data(w, DST16, i + lane + 32 * q, wv[u][q]);
                        }
                }
            }
        }
    }
    check_finish(a, vol, V, C, maxw_out);
}

// ---------------- implicit-gradient anchor (Eq. 22 / Eq. 31) ----------------
// w' = w + 2 gamma, b' = (w b + 2 gamma a) / w'; then max w' of the volume.
__global__ void __launch_bounds__(AUX_THREADS)
    anchor_kernel(AuxParams a, int vol, void *b, void *w, bool bf16, const float *anchor, float gamma, double *maxw_out)
{
    __shared__ float red[32];
    __shared__ int flag;
    const VolDesc V = a.vols[vol];
    const WorkItem W = a.items[V.aux_begin + blockIdx.x];
    const March M = march_place(V, W);
    float mx = 0.f;
    constexpr int U = 2;
    for (int z = M.z0; z < M.z1; z += U) {
        float4 bv[U], wv[U], av[U];
#pragma unroll
        for (int u = 0; u < U; u++)
            if (M.act && z + u < M.z1) {
                const long long i = M.i + (long long)(z + u - M.z0) * M.PS;
                bv[u] = ld4_data(b, bf16, i);
                wv[u] = ld4_data(w, bf16, i);
                av[u] = ld4(anchor + i);
            }
#pragma unroll
        for (int u = 0; u < U; u++) {
            if (!(M.act && z + u < M.z1)) continue;
            const long long i = M.i + (long long)(z + u - M.z0) * M.PS;
            float bb[4], ww[4], an[4];
            unpack4(bv[u], bb);
            unpack4(wv[u], ww);
            unpack4(av[u], an);
#pragma unroll
            for (int q = 0; q < 4; q++) {
                if (M.x0 + q >= V.nx) continue;  // the padding stays as it is
                const float w2 = ww[q] + 2.0f * gamma;
                const float b2 = (ww[q] * bb[q] + 2.0f * gamma * an[q]) / w2;
                st_data(w, bf16, i + q, w2);
                st_data(b, bf16, i + q, b2);
                mx = fmaxf(mx, bf16 ? __uint_as_float((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(w2)) << 16) : w2);
            }
        }
    }
    mx = block_fmax(mx, red);
    if (threadIdx.x == 0) *part_max(a.plane_part + (long long)blockIdx.x * 4) = mx;
    if (!last_block(&a.st->ticket_aux, &flag)) return;
    float m = 0.f;
    for (int q = threadIdx.x; q < V.aux_end - V.aux_begin; q += blockDim.x)
        m = fmaxf(m, __ldcg(part_max(a.plane_part + (long long)q * 4)));
    m = block_fmax(m, red);
    if (threadIdx.x == 0) {
        maxw_out[vol] = m;
        a.st->ticket_aux = 0;
        __threadfence();
    }
}

// D x (Eq. 12) at 4 voxels: c on their row, xl at x0-1, u on the row above
// (y-1), w on the plane below; a missing neighbour is the voxel itself.
__device__ __forceinline__ void grad4(const float (&c)[4], float xl, const float (&u)[4], const float (&w)[4],
                                      float (&gx)[4], float (&gy)[4], float (&gz)[4])
{
#pragma unroll
    for (int q = 0; q < 4; q++) {
        gx[q] = c[q] - (q ? c[q - 1] : xl);
        gy[q] = c[q] - u[q];
        gz[q] = c[q] - w[q];
    }
}

// x on U planes from plane z on, and what their differences need: the row
// above and, for a chunk's first lane, the voxel to the left. Planes from z1 on
// are not read.
template <int U>
struct XRows {
    float4 c[U], u[U];
    float l[U];
    __device__ __forceinline__ void load(const VolDesc &V, const March &M, const float *x, int z)
    {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int k = 0; k < U; k++) {
            const bool ok = M.act && z + k < M.z1;
            const long long i = M.i + (long long)(z + k - M.z0) * M.PS;
            c[k] = ok ? ld4(x + i) : zero;
            u[k] = (ok && M.y >= 1) ? ld4(x + i - V.pitch) : c[k];
            l[k] = (ok && M.lane == 0 && M.x0 >= 1) ? x[i - 1] : 0.f;
        }
    }
    // neighbours of plane k: xl from the lane before (every lane calls it)
    __device__ __forceinline__ void take(const March &M, int k, float (&cc)[4], float &xl, float (&uu)[4]) const
    {
        unpack4(c[k], cc);
        unpack4(u[k], uu);
        xl = __shfl_up_sync(FULL, cc[3], 1);
        if (M.lane == 0) xl = l[k];
        if (M.x0 == 0) xl = cc[0];
    }
};

// One volume's re-weighting statistics and step tau = 1/L (FP64).
__device__ __forceinline__ void set_round(const AuxParams &a, int v, const VolDesc &W, double m, double n, double s1,
                                          double s2, const double *maxw, double *rstats, VolDesc *vols_rw)
{
    const double L = maxw[v] + 12.0 * (double)W.lambda_tv * m / (double)W.mu;
    const double tau = 1.0 / L;
    double *o = rstats + (long long)v * 6;
    o[0] = m;
    o[1] = n;
    o[2] = s1;
    o[3] = s2;
    o[4] = L;
    o[5] = tau;
    vols_rw[v].tau = (float)tau;
    vols_rw[v].kmom = 0;  // extrapolation restarts with the round
    vols_rw[v].beta_last = 0.f;
}

__device__ __forceinline__ void set_objective(const AuxParams &a, int v, const VolDesc &W, double d, double l, double t)
{
    double *o = a.vol_out + (long long)v * 8;
    o[0] = d;
    o[1] = (double)W.lambda_l1 * l;
    o[2] = (double)W.lambda_tv * t;
    o[3] = o[0] + o[1] + o[2];
}

// Last CTA of a march over all volumes: f(volume, descriptor, sums, maximum)
// once per volume, by one thread: a warp per volume, or all warps together
// where there are fewer volumes than warps.
template <class F>
__device__ __forceinline__ void per_volume(const AuxParams &a, bool has_max, double *red, F f)
{
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    const bool together = a.nvol < nw;
    for (int v = together ? 0 : warp; v < a.nvol; v += together ? 1 : nw) {
        const VolDesc W = a.vols[v];
        double s[4];
        float mx;
        part_total(a.plane_part, W.aux_begin, W.aux_end, together ? warp : 0, together ? nw : 1, has_max, red, s, mx);
        if (lane == 0 && (!together || warp == 0)) f(v, W, s, mx);
    }
    __syncthreads();
}

// Last CTA of a re-weighting launch over row segments: per-volume max omtv,
// nnz, sums, and tau = 1/L, then the round restarts.
__device__ void reweight_finish(const AuxParams &a, const double *maxw, double *rstats, VolDesc *vols_rw,
                                double *scratch)
{
    for (int v = 0; v < a.nvol; v++) {
        const VolDesc W = a.vols[v];
        double m = 0, c3[3] = {0, 0, 0};
        for (int q = (W.plane_begin + W.halo_lo) * AUX_SEG + threadIdx.x; q < (W.plane_begin + W.nz - W.halo_hi) * AUX_SEG; q += blockDim.x) {
            const double *pp = a.plane_part + (long long)q * 4;
            m = fmax(m, __ldcg(pp + 0));
            c3[0] += __ldcg(pp + 1);
            c3[1] += __ldcg(pp + 2);
            c3[2] += __ldcg(pp + 3);
        }
        m = block_max(m, scratch);
        block_sum<3>(c3, scratch);
        const double n = c3[0], s1 = c3[1], s2 = c3[2];
        if (threadIdx.x == 0) set_round(a, v, W, m, n, s1, s2, maxw, rstats, vols_rw);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a.st->k_round = 0;
        a.st->ticket_aux = 0;
        __threadfence();
    }
}

// Last CTA of an objective launch over row segments.
__device__ void objective_finish(const AuxParams &a, double *scratch)
{
    for (int v = 0; v < a.nvol; v++) {
        const VolDesc W = a.vols[v];
        double c3[3] = {0, 0, 0};
        for (int q = (W.plane_begin + W.halo_lo) * AUX_SEG + threadIdx.x; q < (W.plane_begin + W.nz - W.halo_hi) * AUX_SEG; q += blockDim.x) {
            const double *pp = a.plane_part + (long long)q * 4;
            c3[0] += __ldcg(pp + 0);
            c3[1] += __ldcg(pp + 1);
            c3[2] += __ldcg(pp + 2);
        }
        block_sum<3>(c3, scratch);
        if (threadIdx.x != 0) continue;
        set_objective(a, v, W, c3[0], c3[1], c3[2]);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a.st->ticket_aux = 0;
        __threadfence();
    }
}

// ---------------- re-weighting (Eq. 11, eps scaling of Sec. 2.5) ----------------
__global__ void reweight_kernel(AuxParams a, const float *xcur, float *om1, float *omtv, const double *maxw,
                                double *rstats, VolDesc *vols_rw)
{
    __shared__ double scratch[32 * 4];
    __shared__ int flag;
    const int plane = blockIdx.x / AUX_SEG;
    const int vol = a.plane_vol[plane];
    const VolDesc V = a.vols[vol];
    const int z = plane - V.plane_begin;
    int r0, r1;
    seg_rows(V.ny, blockIdx.x % AUX_SEG, r0, r1);
    const Field F{xcur, nullptr, 0.f};
    float fmx = 0.f;
    KSum c1, c2;
    float nnz = 0.f;
    for (int t = threadIdx.x; t < (r1 - r0) * V.nx; t += blockDim.x) {
        const int x = t % V.nx, y = r0 + t / V.nx;
        const long long i = V.off + ((long long)z * V.ny + y) * V.pitch + x;
        float g[3];
        grad_at(V, F, x, y, z, g);
        const float gn = sqrtf(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]);
        const float xv = xcur[i];
        const float o1 = V.eps / (fabsf(xv) + V.eps);
        const float ot = V.eps_tv / (gn + V.eps_tv);
        om1[i] = o1;
        omtv[i] = ot;
        fmx = fmaxf(fmx, ot);
        nnz += xv != 0.f ? 1.f : 0.f;
        c1.add(o1);
        c2.add(ot);
    }
    const double mx = block_max((double)fmx, scratch);
    double s[3] = {(double)nnz, c1.value(), c2.value()};
    block_sum<3>(s, scratch);
    if (threadIdx.x == 0) {
        double *pp = a.plane_part + (long long)blockIdx.x * 4;
        pp[0] = mx;
        pp[1] = s[0];
        pp[2] = s[1];
        pp[3] = s[2];
    }
    if (!last_block(&a.st->ticket_aux, &flag)) return;
    reweight_finish(a, maxw, rstats, vols_rw, scratch);
}

// ---------------- objective F(x) at the current iterate ----------------
__global__ void objective_kernel(AuxParams a, const float *xcur, const void *b, const void *w, bool bf16,
                                 const float *om1, const float *omtv)
{
    __shared__ double scratch[32 * 4];
    __shared__ int flag;
    const int plane = blockIdx.x / AUX_SEG;
    const int vol = a.plane_vol[plane];
    const VolDesc V = a.vols[vol];
    const int z = plane - V.plane_begin;
    int r0, r1;
    seg_rows(V.ny, blockIdx.x % AUX_SEG, r0, r1);
    const Field F{xcur, nullptr, 0.f};
    KSum kd, kl, kt;
    const float mu = V.mu;
    for (int t = threadIdx.x; t < (r1 - r0) * V.nx; t += blockDim.x) {
        const int x = t % V.nx, y = r0 + t / V.nx;
        const long long i = V.off + ((long long)z * V.ny + y) * V.pitch + x;
        float g[3];
        grad_at(V, F, x, y, z, g);
        const float q = g[0] * g[0] + g[1] * g[1] + g[2] * g[2];
        const float h = q <= mu * mu ? q * (0.5f / mu) : q * rsqrtf(q) - 0.5f * mu;
        const float xv = xcur[i];
        if (w) {  // no real-space data term when the Fourier-domain term is in use
            const float r = xv - ld_data(b, bf16, i);
            kd.add(0.5f * ld_data(w, bf16, i) * r * r);
        }
        kl.add(om1[i] * fabsf(xv));
        kt.add(omtv[i] * h);
    }
    double s[3] = {kd.value(), kl.value(), kt.value()};
    block_sum<3>(s, scratch);
    if (threadIdx.x == 0) {
        double *pp = a.plane_part + (long long)blockIdx.x * 4;
        pp[0] = s[0];
        pp[1] = s[1];
        pp[2] = s[2];
        pp[3] = 0;
    }
    if (!last_block(&a.st->ticket_aux, &flag)) return;
    objective_finish(a, scratch);
}

// Re-weighting of the adopted reading, march (same results as
// reweight_kernel; padding columns of the pitch get zero weights). Bound: x
// read once, two volumes written, 12 bytes a voxel.
__global__ void __launch_bounds__(AUX_THREADS, 4)
    reweight_march_kernel(AuxParams a, const float *xcur, float *om1, float *omtv, const double *maxw, double *rstats,
                          VolDesc *vols_rw)
{
    __shared__ double red[32 * 4 + 16];
    __shared__ int flag;
    const WorkItem W = a.items[blockIdx.x];
    const VolDesc V = a.vols[W.vol];
    const March M = march_place(V, W);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float pw[4];  // the plane below
    unpack4((M.act && M.z0 >= 1) ? ld4(xcur + M.i - M.PS) : zero, pw);
    float fmx = 0.f;
    int nnz = 0;
    KSum c1, c2;
    constexpr int U = 4;  // planes whose loads are in flight together
    for (int z = M.z0; z < M.z1; z += U) {
        XRows<U> X;
        X.load(V, M, xcur, z);
#pragma unroll
        for (int k = 0; k < U; k++) {
            if (z + k >= M.z1) break;
            float xc[4], uu[4], xl, gx[4], gy[4], gz[4], o1[4], ot[4];
            X.take(M, k, xc, xl, uu);
            if (z + k == 0)
#pragma unroll
                for (int q = 0; q < 4; q++) pw[q] = xc[q];
            grad4(xc, xl, uu, pw, gx, gy, gz);
            const bool own = z + k >= V.halo_lo && z + k < V.nz - V.halo_hi;  // not a neighbour's plane
            float s1 = 0.f, s2 = 0.f;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const bool valid = M.act && M.x0 + q < V.nx;
                const float gn = sqrtf(gx[q] * gx[q] + gy[q] * gy[q] + gz[q] * gz[q]);
                o1[q] = valid ? V.eps / (fabsf(xc[q]) + V.eps) : 0.f;
                ot[q] = valid ? V.eps_tv / (gn + V.eps_tv) : 0.f;
                if (own) {
                    fmx = fmaxf(fmx, ot[q]);
                    nnz += (valid && xc[q] != 0.f) ? 1 : 0;
                    s1 += o1[q];
                    s2 += ot[q];
                }
                pw[q] = xc[q];
            }
            if (M.act) {
                const long long i = M.i + (long long)(z + k - M.z0) * M.PS;
                *reinterpret_cast<float4 *>(om1 + i) = make_float4(o1[0], o1[1], o1[2], o1[3]);
                *reinterpret_cast<float4 *>(omtv + i) = make_float4(ot[0], ot[1], ot[2], ot[3]);
            }
            c1.add(s1);
            c2.add(s2);
        }
    }
    fmx = block_fmax(fmx, reinterpret_cast<float *>(red));
    const ff::FF v[4] = {{0.f, 0.f}, {(float)nnz, 0.f}, c1.pair(), c2.pair()};
    const double s = block_sum4(v, red);
    double *pp = a.plane_part + (long long)blockIdx.x * 4;
    if (threadIdx.x == 0) *part_max(pp) = fmx;
    else if (threadIdx.x < 4) pp[threadIdx.x] = s;
    if (!last_block(&a.st->ticket_aux, &flag)) return;
    per_volume(a, true, red, [&](int vol, const VolDesc &D, const double (&t)[4], float mx) {
        set_round(a, vol, D, (double)mx, t[1], t[2], t[3], maxw, rstats, vols_rw);
    });
    if (threadIdx.x == 0) {
        a.st->k_round = 0;
        a.st->ticket_aux = 0;
        __threadfence();
    }
}

// Objective of the adopted reading, march (same sums as objective_kernel;
// padding columns contribute nothing). Bound: 20 bytes a voxel.
__global__ void __launch_bounds__(AUX_THREADS, 4)
    objective_march_kernel(AuxParams a, const float *xcur, const void *b, const void *w, bool bf16, const float *om1,
                           const float *omtv)
{
    __shared__ double red[32 * 4 + 16];
    __shared__ int flag;
    const WorkItem W = a.items[blockIdx.x];
    const VolDesc V = a.vols[W.vol];
    const March M = march_place(V, W);
    const float mu = V.mu;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float pw[4];
    unpack4((M.act && M.z0 >= 1) ? ld4(xcur + M.i - M.PS) : zero, pw);
    KSum kd, kl, kt;
    constexpr int U = 1;  // more warps per SM beat more planes per warp here (2 planes at 2 CTAs: 522 us)
    for (int z = M.z0; z < M.z1; z += U) {
        XRows<U> X;
        X.load(V, M, xcur, z);
        float4 f1[U], ft[U], fb[U], fw[U];
#pragma unroll
        for (int k = 0; k < U; k++) {
            const bool ok = M.act && z + k < M.z1;
            const long long i = M.i + (long long)(z + k - M.z0) * M.PS;
            f1[k] = ok ? ld4(om1 + i) : zero;
            ft[k] = ok ? ld4(omtv + i) : zero;
            fb[k] = (ok && w) ? ld4_data(b, bf16, i) : zero;
            fw[k] = (ok && w) ? ld4_data(w, bf16, i) : zero;
        }
#pragma unroll
        for (int k = 0; k < U; k++) {
            if (z + k >= M.z1) break;
            float xc[4], uu[4], xl, gx[4], gy[4], gz[4], o1[4], ot[4], bv[4], wv[4];
            X.take(M, k, xc, xl, uu);
            if (z + k == 0)
#pragma unroll
                for (int q = 0; q < 4; q++) pw[q] = xc[q];
            grad4(xc, xl, uu, pw, gx, gy, gz);
            unpack4(f1[k], o1);
            unpack4(ft[k], ot);
            unpack4(fb[k], bv);
            unpack4(fw[k], wv);
            const bool own = z + k >= V.halo_lo && z + k < V.nz - V.halo_hi;
            float sd = 0.f, sl = 0.f, st = 0.f;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const float x = xc[q];
                pw[q] = x;
                if (!(own && M.act && M.x0 + q < V.nx)) continue;
                const float qq = gx[q] * gx[q] + gy[q] * gy[q] + gz[q] * gz[q];
                const float h = qq <= mu * mu ? qq * (0.5f / mu) : qq * rsqrtf(qq) - 0.5f * mu;
                const float r = x - bv[q];
                sd += 0.5f * wv[q] * r * r;
                sl += o1[q] * fabsf(x);
                st += ot[q] * h;
            }
            kd.add(sd);
            kl.add(sl);
            kt.add(st);
        }
    }
    const ff::FF v[4] = {kd.pair(), kl.pair(), kt.pair(), {0.f, 0.f}};
    const double s = block_sum4(v, red);
    if (threadIdx.x < 4) a.plane_part[(long long)blockIdx.x * 4 + threadIdx.x] = s;
    if (!last_block(&a.st->ticket_aux, &flag)) return;
    per_volume(a, false, red, [&](int vol, const VolDesc &D, const double (&t)[4], float) {
        set_objective(a, vol, D, t[0], t[1], t[2]);
    });
    if (threadIdx.x == 0) {
        a.st->ticket_aux = 0;
        __threadfence();
    }
}

// ---------------- one iteration under alternative readings ----------------
// The fused step's arithmetic for volumes with SPG_READ_* flags, written
// plainly: one CTA per row segment of a z-plane; D^T(p) re-evaluates p at the
// voxel and its three neighbours; the objective at x_k is summed when the
// step records history. The last CTA writes the history entries, advances
// each volume's extrapolation index and the device state, as the fused
// kernel does, so the two paths are interchangeable between launches.
__global__ void generic_step_kernel(GenericParams g)
{
    __shared__ double scratch[32 * 4];
    __shared__ int flag, s_cur, s_rec, s_kr;
    __shared__ long long s_kt;
    if (threadIdx.x == 0) {
        volatile DevState *st = g.st;
        s_cur = st->cur;
        s_kr = st->k_round;
        s_kt = st->k_total;
        s_rec = (g.hist_every > 0 && (s_kt % g.hist_every) == 0) ? 1 : 0;
    }
    __syncthreads();
    const int cur = s_cur;
    const bool rec = s_rec != 0;
    const int nxt = g.xd ? (cur ^ 1) : (cur + 1) % 3;
    auto pick = [&](int i) { return i == 0 ? g.xbuf[0] : (i == 1 ? g.xbuf[1] : (i == 2 ? g.xbuf[2] : g.xbuf[3])); };
    const float *xk = pick(cur);
    const float *aux = pick(g.xd ? 2 + cur : (cur + 2) % 3);
    float *xout = pick(nxt);
    float *dout = g.xd ? pick(2 + nxt) : nullptr;

    const int plane = blockIdx.x / AUX_SEG;
    const int vol = g.plane_vol[plane];
    const VolDesc V = g.vols[vol];
    const int z = plane - V.plane_begin;
    int r0, r1;
    seg_rows(V.ny, blockIdx.x % AUX_SEG, r0, r1);
    const float beta = g.beta[V.kmom];
    const Field F{xk, g.xd ? nullptr : aux, beta, g.xd ? aux : nullptr};
    const Field X0{xk, nullptr, 0.f};
    const float tau = V.tau, tl1 = V.tau * V.lambda_l1, mu = V.mu;
    KSum kd, kl, kt;
    for (int t = threadIdx.x; t < (r1 - r0) * V.nx; t += blockDim.x) {
        const int x = t % V.nx, y = r0 + t / V.nx;
        const long long i = V.off + ((long long)z * V.ny + y) * V.pitch + x;
        const float xc = xk[i], dc = F.d(i), wv = g.w[i], o1 = g.om1[i];
        const float res = xc - g.b[i];
        const float gtot = fmaf(V.lambda_tv, div_at(V, F, g.omtv, x, y, z), wv * fmaf(beta, dc, res));
        const float delta = fmaf(beta, dc, -tau * gtot);
        const float zz = xc + delta;
        const float th = tl1 * o1;
        const float inc = fabsf(zz) < th ? -xc : delta - copysignf(th, zz);
        xout[i] = xc + inc;
        if (dout) dout[i] = inc;
        if (rec) {
            float gq[3];
            grad_at(V, X0, x, y, z, gq);
            const float q = gq[0] * gq[0] + gq[1] * gq[1] + gq[2] * gq[2];
            const float h = q <= mu * mu ? q * (0.5f / mu) : q * rsqrtf(q) - 0.5f * mu;
            kd.add(0.5f * wv * res * res);
            kl.add(o1 * fabsf(xc));
            kt.add(g.omtv[i] * h);
        }
    }
    if (rec) {
        double sm[3] = {kd.value(), kl.value(), kt.value()};
        block_sum<3>(sm, scratch);
        if (threadIdx.x == 0) {
            double *pp = g.plane_part + (long long)blockIdx.x * 4;
            pp[0] = sm[0];
            pp[1] = sm[1];
            pp[2] = sm[2];
        }
    }
    if (!last_block(&g.st->ticket, &flag)) return;
    const int hslot = g.st->hist_count % g.hist_cap;
    for (int v = 0; v < g.nvol; v++) {
        const VolDesc W = g.vols[v];
        if (rec) {
            double c3[3] = {0, 0, 0};
            for (int q = (W.plane_begin + W.halo_lo) * AUX_SEG + threadIdx.x; q < (W.plane_begin + W.nz - W.halo_hi) * AUX_SEG;
                 q += blockDim.x) {
                const double *pp = g.plane_part + (long long)q * 4;
                c3[0] += __ldcg(pp + 0);
                c3[1] += __ldcg(pp + 1);
                c3[2] += __ldcg(pp + 2);
            }
            block_sum<3>(c3, scratch);
            if (threadIdx.x == 0) {
                double *h = g.hist + ((long long)hslot * g.nvol + v) * 5;
                const double l1 = (double)W.lambda_l1 * c3[1], tv = (double)W.lambda_tv * c3[2];
                const double tot = c3[0] + l1 + tv;
                h[0] = (double)s_kt;
                h[1] = c3[0];
                h[2] = l1;
                h[3] = tv;
                h[4] = tot;
                if (!isfinite(tot)) atomicCAS(&g.st->err, 0, (int)SPG_ENONFINITE);
            }
        }
        if (threadIdx.x == 0) {
            g.vols[v].beta_last = g.beta[W.kmom];
            g.vols[v].kmom = W.kmom + 1;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        DevState *st = g.st;
        if (rec) st->hist_count = st->hist_count + 1;
        st->cur = nxt;
        st->k_round = s_kr + 1;
        st->k_total = s_kt + 1;
        st->ticket = 0;
        __threadfence();
    }
}

// ---------------- adjoint of one step ----------------
// Two passes, each a march over z (a CTA owns TY rows of a 128-voxel chunk
// of x over ZC planes, warp r row y0 + r, one more warp the row below the
// tile), 4 voxels per lane with 16-byte loads and x-neighbours by shuffle:
//   1. mask: p = omtv grad h_mu(D y) (Eq. 12, 16), tvg = D^T p (Eq. 17),
//      the step's z, the soft-threshold mask m = gnext [pass] (Eq. 21), the
//      l1 / TV scalar partials, gb += tau w m, gw += -tau (y - b) m;
//   2. apply: hq = omtv H_mu(D y) D m, H_mu = I/mu inside the smoothing ball
//      and (I - e e^T)/|D y| outside (the Hessian of Eq. 14);
//      ybar = m - tau (w m + lambda_tv D^T hq); gcur += (1+beta) ybar,
//      gprev += -beta ybar (gprev is written, not accumulated, when it has
//      no earlier contribution).
// Each step of the march evaluates p (hq) on the next plane once per voxel
// and keeps it in registers, where it is the forward z-neighbour now and the
// voxel's own value one step later; the y-component of the row below comes
// from the warp that owns that row through a 3-plane shared ring; the
// x-neighbour from the next lane (a chunk's last lane evaluates it). Only m
// is stored between the passes.
struct Lane4 {
    int x0, y, z, lane;
    bool act;
    long long i;  // element index of voxel x0 of the row
};

__device__ __forceinline__ float4 ldz4(const float *p, bool ok)
{
    return ok ? *reinterpret_cast<const float4 *>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
}

__device__ __forceinline__ void st4(float *p, const float (&v)[4])
{
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

namespace adj {
constexpr int TY = 7;                  // output rows per CTA
constexpr int THREADS = 32 * (TY + 1); // warp TY: the row below the tile
constexpr int ZC = 8;                  // planes per CTA
}  // namespace adj

// (D y)_a at the lane's 4 voxels (Eq. 12 on y = x_k + beta (x_k - x_{k-1})),
// differences of x_k and of d = x_k - x_{k-1} taken separately: xc, mc on
// the voxels' row (xl, ml at x0-1), xu, mu_ on the row below in y, xw, mw on
// the plane below.
__device__ __forceinline__ void dy4(const float (&xc)[4], const float (&mc)[4], float xl, float ml,
                                    const float (&xu)[4], const float (&mu_)[4], const float (&xw)[4],
                                    const float (&mw)[4], float beta, float (&g)[3][4])
{
#pragma unroll
    for (int q = 0; q < 4; q++) {
        const float dc = xc[q] - mc[q];
        const float lx = q ? xc[q - 1] : xl, lm = q ? mc[q - 1] : ml;
        g[0][q] = (xc[q] - lx) + beta * (dc - (lx - lm));
        g[1][q] = (xc[q] - xu[q]) + beta * (dc - (xu[q] - mu_[q]));
        g[2][q] = (xc[q] - xw[q]) + beta * (dc - (xw[q] - mw[q]));
    }
}

// The same at one voxel: (xa, ma) there, (xl, ml) at x-1, (xu, mu_) at y-1,
// (xw, mw) at z-1.
__device__ __forceinline__ void dy1(float xa, float ma, float xl, float ml, float xu, float mu_, float xw, float mw,
                                    float beta, float (&g)[3])
{
    const float dc = xa - ma;
    g[0] = (xa - xl) + beta * (dc - (xl - ml));
    g[1] = (xa - xu) + beta * (dc - (xu - mu_));
    g[2] = (xa - xw) + beta * (dc - (xw - mw));
}

// omtv / max(mu, |g|): the factor by which omtv grad h_mu(g) (Eq. 16) scales g.
__device__ __forceinline__ float p_scale(float g0, float g1, float g2, float ot, float mu)
{
    const float s2 = g0 * g0 + g1 * g1 + g2 * g2;
    return ot * fminf(1.0f / mu, rsqrtf(s2));
}

// omtv H_mu(g) q at one voxel, H_mu the Hessian of the smoothed norm (Eq. 14):
// I/mu inside the ball |g| <= mu, (I - e e^T)/|g| with e = g/|g| outside.
__device__ __forceinline__ void hq1(float g0, float g1, float g2, float q0, float q1, float q2, float ot, float mu,
                                    float (&h)[3])
{
    const float s = sqrtf(g0 * g0 + g1 * g1 + g2 * g2);
    if (s <= mu) {
        const float c = ot / mu;
        h[0] = q0 * c;
        h[1] = q1 * c;
        h[2] = q2 * c;
    } else {
        const float inv = 1.0f / s;
        const float e0 = g0 * inv, e1 = g1 * inv, e2 = g2 * inv;
        const float eq = e0 * q0 + e1 * q1 + e2 * q2;
        const float c = ot * inv;
        h[0] = (q0 - e0 * eq) * c;
        h[1] = (q1 - e1 * eq) * c;
        h[2] = (q2 - e2 * eq) * c;
    }
}

// Where a thread of the two passes works: chunk of x, tile of rows, planes.
struct AdjPlace {
    Lane4 L;
    int r, z0, z1;
    bool row_in;   // the warp's row is inside the volume
    long long PS;  // plane stride
};

__device__ __forceinline__ AdjPlace adj_place(const VolDesc &V, int zc = adj::ZC)
{
    AdjPlace P;
    const int nchunk = (V.nx + 127) / 128, ntile = (V.ny + adj::TY - 1) / adj::TY;
    int b = blockIdx.x;
    const int cx = b % nchunk;
    b /= nchunk;
    const int by = b % ntile, bz = b / ntile;
    P.r = threadIdx.x >> 5;
    P.L.lane = threadIdx.x & 31;
    P.L.x0 = cx * 128 + 4 * P.L.lane;
    P.L.y = by * adj::TY + P.r;
    P.row_in = P.L.y < V.ny;
    P.L.act = P.row_in && P.L.x0 < V.nx;
    P.z0 = bz * zc;
    P.z1 = min(V.nz, P.z0 + zc);
    P.PS = (long long)V.pitch * V.ny;
    return P;
}

// element index of voxel x0 of row (y, z); only formed for rows in the volume
__device__ __forceinline__ long long adj_row(const VolDesc &V, int x0, int y, int z)
{
    return V.off + ((long long)z * V.ny + y) * V.pitch + x0;
}

// One field's loads for a plane of the march, issued an iteration before their
// use: the warp's row, the row above and, for a chunk's first lane, the voxel
// to the left.
struct RowLoads {
    float4 c, u;
    float l;
    __device__ __forceinline__ void load(const VolDesc &V, const Lane4 &L, const float *f, long long i, bool ok)
    {
        c = ldz4(f + i, ok);
        u = ldz4(f + i - V.pitch, ok && L.y >= 1);
        l = (L.lane == 0 && ok && L.x0 >= 1) ? f[i - 1] : 0.f;
    }
    // the values, with the voxel itself for a missing neighbour (every lane calls it)
    __device__ __forceinline__ void take(const Lane4 &L, float (&cc)[4], float &cl, float (&uu)[4]) const
    {
        unpack4(c, cc);
        cl = __shfl_up_sync(FULL, cc[3], 1);
        if (L.lane == 0) cl = l;
        if (L.x0 == 0) cl = cc[0];
        if (L.y >= 1) {
            unpack4(u, uu);
        } else {
#pragma unroll
            for (int q = 0; q < 4; q++) uu[q] = cc[q];
        }
    }
};

// Both passes may be launched before the pass ahead of them has ended
// (programmatic stream serialisation, see launch_adjoint): what that pass
// writes is read after pdl_wait, what neither of the passes writes (the
// iterates, the weights, b and w) before it. A backward call of 50 steps at
// 128^3 (100 passes of about 19 us): 3.40 -> 3.20 ms.
__device__ __forceinline__ void pdl_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Bound (both passes, 128^3): the latency of their loads with the 16 warps an
// SM holds; 36 + 12 and 24 + 8 bytes a voxel, mostly from L2. The loads of a
// plane are therefore issued one iteration ahead: the next plane's rows before
// this plane's barrier, the rest once this plane's are consumed (24.2 -> 19.0 us
// and 23.5 -> 19.7 us a pass, 125 registers).
__global__ void __launch_bounds__(adj::THREADS, 2) adjoint_mask_kernel(AdjParams a)
{
    __shared__ __align__(16) float ring[3][adj::TY + 1][128];  // p_y of the tile's rows and the row below it
    __shared__ double scratch[32 * 4 + 16];
    pdl_start();
    const VolDesc V = a.vols[0];
    AdjPlace P = adj_place(V);
    Lane4 &L = P.L;
    const float beta = a.beta, mu = V.mu;
    const bool writes = P.r < adj::TY && P.row_in;
    KSum k1, k2;
    // x_k, x_{k-1} on the warp's row of the current plane, and p there
    float xc[4], mc[4], pc[3][4];
    RowLoads rx, rm;
    float4 rot, fb, fw, f1, fg, fgb, fgw;  // omtv of the next plane; b, w, om1, gnext, gb, gw of this one
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load_rows = [&](long long i, bool ok) {
        rx.load(V, L, a.xk, i, ok);
        rm.load(V, L, a.xkm1, i, ok);
        rot = ldz4(a.omtv + i, ok);
    };
    auto load_given = [&](long long i, bool ok) {
        fb = ok ? ld4_data(a.b, a.bf16, i) : zero;
        fw = ok ? ld4_data(a.w, a.bf16, i) : zero;
        f1 = ldz4(a.om1 + i, ok);
    };
    auto load_made = [&](long long i, bool ok) {  // by earlier passes
        fg = ldz4(a.gnext + i, ok);
        fgb = ldz4(a.gb + i, ok);
        fgw = ldz4(a.gw + i, ok);
    };
    // p at the loaded rows' plane z, the plane below in (xw, mw); into the ring
    auto p_rows = [&](const float (&xw)[4], const float (&mw)[4], bool have, bool ok, int z, float (&xn)[4],
                      float (&mn)[4], float (&pn)[3][4]) {
        float xu[4], mu_[4], ot[4], g[3][4], xl, ml;
        rx.take(L, xn, xl, xu);
        rm.take(L, mn, ml, mu_);
        unpack4(rot, ot);
        if (have)
            dy4(xn, mn, xl, ml, xu, mu_, xw, mw, beta, g);
        else
            dy4(xn, mn, xl, ml, xu, mu_, xn, mn, beta, g);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const bool valid = ok && L.x0 + q < V.nx;
            const float sc = p_scale(g[0][q], g[1][q], g[2][q], ot[q], mu);
#pragma unroll
            for (int c = 0; c < 3; c++) pn[c][q] = valid ? g[c][q] * sc : 0.f;
        }
        *reinterpret_cast<float4 *>(&ring[z % 3][P.r][4 * L.lane]) = make_float4(pn[1][0], pn[1][1], pn[1][2], pn[1][3]);
    };
    L.i = P.row_in ? adj_row(V, L.x0, L.y, P.z0) : 0;
    {
        float xw[4], mw[4];
        load_rows(L.i, L.act);
        unpack4(ldz4(a.xk + L.i - P.PS, L.act && P.z0 >= 1), xw);
        unpack4(ldz4(a.xkm1 + L.i - P.PS, L.act && P.z0 >= 1), mw);
        load_given(L.i, L.act && writes);
        pdl_wait();
        load_made(L.i, L.act && writes);
        p_rows(xw, mw, P.z0 >= 1, L.act, P.z0, xc, mc, pc);
        load_rows(L.i + P.PS, L.act && P.z0 + 1 < V.nz);
    }
    for (int z = P.z0; z < P.z1; z++) {
        // p on the next plane (zero beyond the volume)
        const long long in_ = L.i + P.PS;
        float xn[4], mn[4], pn[3][4];
        p_rows(xc, mc, true, L.act && z + 1 < V.nz, z + 1, xn, mn, pn);
        load_rows(in_ + P.PS, L.act && z + 1 < P.z1 && z + 2 < V.nz);
        __syncthreads();  // p_y of plane z of every row of the tile is in the ring
        // p_x at x+1: the next lane's first voxel; a chunk's last lane evaluates it
        float pxn = __shfl_down_sync(FULL, pc[0][0], 1);
        if (L.lane == 31) {
            pxn = 0.f;
            if (L.act && L.x0 + 4 < V.nx) {
                const long long j = L.i + 4;
                const float xa = a.xk[j], ma = a.xkm1[j];
                const float xau = L.y >= 1 ? a.xk[j - V.pitch] : xa, mau = L.y >= 1 ? a.xkm1[j - V.pitch] : ma;
                const float xaw = z >= 1 ? a.xk[j - P.PS] : xa, maw = z >= 1 ? a.xkm1[j - P.PS] : ma;
                float ga[3];
                dy1(xa, ma, xc[3], mc[3], xau, mau, xaw, maw, beta, ga);
                pxn = ga[0] * p_scale(ga[0], ga[1], ga[2], a.omtv[j], mu);
            }
        }
        if (writes) {
            float px[4] = {pc[0][1], pc[0][2], pc[0][3], pxn};
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (L.x0 + q + 1 >= V.nx) px[q] = 0.f;
            const float4 pyv = *reinterpret_cast<const float4 *>(&ring[z % 3][P.r + 1][4 * L.lane]);
            const float py[4] = {pyv.x, pyv.y, pyv.z, pyv.w};  // zero when row y + 1 is outside
            float bv[4], wv[4], o1[4], gn[4], gb[4], gw[4], m[4];
            unpack4(fb, bv);
            unpack4(fw, wv);
            unpack4(f1, o1);
            unpack4(fg, gn);
            unpack4(fgb, gb);
            unpack4(fgw, gw);
            load_given(in_, L.act && z + 1 < P.z1);
            load_made(in_, L.act && z + 1 < P.z1);
            float s1 = 0.f, s2 = 0.f;
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const bool valid = L.act && L.x0 + q < V.nx;
                const float d = xc[q] - mc[q];
                const float tvg = (pc[0][q] - px[q]) + (pc[1][q] - py[q]) + (pc[2][q] - pn[2][q]);
                const float g = wv[q] * ((xc[q] - bv[q]) + beta * d) + V.lambda_tv * tvg;
                const float delta = beta * d - V.tau * g;
                const float zz = xc[q] + delta;
                const float th = V.tau * V.lambda_l1 * o1[q];
                const bool pass = fabsf(zz) > th || th <= 0.f;
                m[q] = (valid && pass) ? gn[q] : 0.f;
                const float sg = zz > 0.f ? 1.f : (zz < 0.f ? -1.f : 0.f);
                s1 += -V.tau * o1[q] * sg * m[q];
                s2 += -V.tau * tvg * m[q];
                gb[q] += V.tau * wv[q] * m[q];
                gw[q] += -V.tau * ((xc[q] - bv[q]) + beta * d) * m[q];
            }
            if (L.act) {
                st4(a.m + L.i, m);
                st4(a.gb + L.i, gb);
                st4(a.gw + L.i, gw);
            }
            k1.add(s1);
            k2.add(s2);
        }
        // the next plane becomes the current one
#pragma unroll
        for (int q = 0; q < 4; q++) {
            xc[q] = xn[q];
            mc[q] = mn[q];
#pragma unroll
            for (int c = 0; c < 3; c++) pc[c][q] = pn[c][q];
        }
        L.i = in_;
    }
    const ff::FF fv[4] = {k1.pair(), k2.pair(), {0.f, 0.f}, {0.f, 0.f}};
    const double sm = block_sum4(fv, scratch);
    if (threadIdx.x < 2) a.plane_part[(long long)blockIdx.x * 4 + threadIdx.x] = sm;
}

// hq at the lane's 4 voxels from D y and D m there (zero where !ok or beyond nx)
__device__ __forceinline__ void hq4(const float (&g)[3][4], const float (&qc)[4], float ql, const float (&qu)[4],
                                    const float (&qw)[4], const float (&ot)[4], float mu, bool ok, int x0, int nx,
                                    float (&h)[3][4])
{
#pragma unroll
    for (int q = 0; q < 4; q++) {
        float t[3];
        hq1(g[0][q], g[1][q], g[2][q], qc[q] - (q ? qc[q - 1] : ql), qc[q] - qu[q], qc[q] - qw[q], ot[q], mu, t);
        const bool valid = ok && x0 + q < nx;
#pragma unroll
        for (int c = 0; c < 3; c++) h[c][q] = valid ? t[c] : 0.f;
    }
}

__global__ void __launch_bounds__(adj::THREADS, 2) adjoint_apply_kernel(AdjParams a)
{
    __shared__ __align__(16) float ring[3][adj::TY + 1][128];  // hq_y of the tile's rows and the row below it
    pdl_start();
    const VolDesc V = a.vols[0];
    AdjPlace P = adj_place(V);
    Lane4 &L = P.L;
    const float beta = a.beta, mu = V.mu;
    const bool writes = P.r < adj::TY && P.row_in;
    const bool alias = a.gprev == a.gcur;  // k = 0: x_{-1} = x_0
    // x_k, x_{k-1} and m on the warp's row of the current plane, and hq there
    float xc[4], mc[4], qc[4], hc[3][4];
    RowLoads rx, rm, rq;
    float4 rot, fw, fgc, fgp;  // omtv of the next plane; w, gcur, gprev of this one
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load_rows = [&](long long i, bool ok) {
        rx.load(V, L, a.xk, i, ok);
        rm.load(V, L, a.xkm1, i, ok);
        rq.load(V, L, a.m, i, ok);
        rot = ldz4(a.omtv + i, ok);
    };
    auto load_rest = [&](long long i, bool ok) {
        fw = ok ? ld4_data(a.w, a.bf16, i) : zero;
        fgc = ldz4(a.gcur + i, ok);
        fgp = ldz4(a.gprev + i, ok && !alias && !a.prev_fresh);
    };
    auto h_rows = [&](const float (&xw)[4], const float (&mw)[4], const float (&qw)[4], bool have, bool ok, int z,
                      float (&xn)[4], float (&mn)[4], float (&qn)[4], float (&hn)[3][4]) {
        float xu[4], mu_[4], qu[4], ot[4], g[3][4], xl, ml, ql;
        rx.take(L, xn, xl, xu);
        rm.take(L, mn, ml, mu_);
        rq.take(L, qn, ql, qu);
        unpack4(rot, ot);
        if (have) {
            dy4(xn, mn, xl, ml, xu, mu_, xw, mw, beta, g);
            hq4(g, qn, ql, qu, qw, ot, mu, ok, L.x0, V.nx, hn);
        } else {
            dy4(xn, mn, xl, ml, xu, mu_, xn, mn, beta, g);
            hq4(g, qn, ql, qu, qn, ot, mu, ok, L.x0, V.nx, hn);
        }
        *reinterpret_cast<float4 *>(&ring[z % 3][P.r][4 * L.lane]) = make_float4(hn[1][0], hn[1][1], hn[1][2], hn[1][3]);
    };
    L.i = P.row_in ? adj_row(V, L.x0, L.y, P.z0) : 0;
    {
        float xw[4], mw[4], qw[4];
        const bool below = L.act && P.z0 >= 1;
        rx.load(V, L, a.xk, L.i, L.act);
        rm.load(V, L, a.xkm1, L.i, L.act);
        rot = ldz4(a.omtv + L.i, L.act);
        unpack4(ldz4(a.xk + L.i - P.PS, below), xw);
        unpack4(ldz4(a.xkm1 + L.i - P.PS, below), mw);
        pdl_wait();
        rq.load(V, L, a.m, L.i, L.act);
        unpack4(ldz4(a.m + L.i - P.PS, below), qw);
        load_rest(L.i, L.act && writes);
        h_rows(xw, mw, qw, P.z0 >= 1, L.act, P.z0, xc, mc, qc, hc);
        load_rows(L.i + P.PS, L.act && P.z0 + 1 < V.nz);
    }
    for (int z = P.z0; z < P.z1; z++) {
        const long long in_ = L.i + P.PS;
        float xn[4], mn[4], qn[4], hn[3][4];
        h_rows(xc, mc, qc, true, L.act && z + 1 < V.nz, z + 1, xn, mn, qn, hn);
        load_rows(in_ + P.PS, L.act && z + 1 < P.z1 && z + 2 < V.nz);
        __syncthreads();  // hq_y of plane z of every row of the tile is in the ring
        // hq_x at x+1: the next lane's first voxel; a chunk's last lane evaluates it
        float hxn = __shfl_down_sync(FULL, hc[0][0], 1);
        if (L.lane == 31) {
            hxn = 0.f;
            if (L.act && L.x0 + 4 < V.nx) {
                const long long j = L.i + 4;
                const float xa = a.xk[j], ma = a.xkm1[j], qa = a.m[j];
                const bool u = L.y >= 1, w = z >= 1;
                const float xau = u ? a.xk[j - V.pitch] : xa, mau = u ? a.xkm1[j - V.pitch] : ma;
                const float qau = u ? a.m[j - V.pitch] : qa;
                const float xaw = w ? a.xk[j - P.PS] : xa, maw = w ? a.xkm1[j - P.PS] : ma;
                const float qaw = w ? a.m[j - P.PS] : qa;
                float ga[3], h[3];
                dy1(xa, ma, xc[3], mc[3], xau, mau, xaw, maw, beta, ga);
                hq1(ga[0], ga[1], ga[2], qa - qc[3], qa - qau, qa - qaw, a.omtv[j], mu, h);
                hxn = h[0];
            }
        }
        if (writes) {
            float hx[4] = {hc[0][1], hc[0][2], hc[0][3], hxn};
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (L.x0 + q + 1 >= V.nx) hx[q] = 0.f;
            const float4 hyv = *reinterpret_cast<const float4 *>(&ring[z % 3][P.r + 1][4 * L.lane]);
            const float hy[4] = {hyv.x, hyv.y, hyv.z, hyv.w};
            float wv[4], gc[4], gp[4];
            unpack4(fw, wv);
            unpack4(fgc, gc);
            unpack4(fgp, gp);
            load_rest(in_, L.act && z + 1 < P.z1);
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const bool valid = L.act && L.x0 + q < V.nx;
                const float dtv = (hc[0][q] - hx[q]) + (hc[1][q] - hy[q]) + (hc[2][q] - hn[2][q]);
                const float ybar = valid ? qc[q] - V.tau * (wv[q] * qc[q] + V.lambda_tv * dtv) : 0.f;
                gc[q] += (1.f + beta) * ybar;
                if (alias) gc[q] += -beta * ybar;
                else if (a.prev_fresh) gp[q] = -beta * ybar;
                else gp[q] += -beta * ybar;
            }
            if (L.act) {
                st4(a.gcur + L.i, gc);
                if (!alias) st4(a.gprev + L.i, gp);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; q++) {
            xc[q] = xn[q];
            mc[q] = mn[q];
            qc[q] = qn[q];
#pragma unroll
            for (int c = 0; c < 3; c++) hc[c][q] = hn[c][q];
        }
        L.i = in_;
    }
}

// One CTA per step: its CTAs' scalar partials, summed in a fixed order (the
// host read and summed all of them: 0.5 MB at 128^3 and 50 steps).
__global__ void adjoint_scalars_kernel(const double *part, int nblk, double *out)
{
    __shared__ double scratch[32 * 2];
    const double *p = part + (long long)blockIdx.x * nblk * 4;
    double v[2] = {0.0, 0.0};
    for (int q = threadIdx.x; q < nblk; q += blockDim.x) {
        v[0] += p[(long long)q * 4 + 0];
        v[1] += p[(long long)q * 4 + 1];
    }
    block_sum<2>(v, scratch);
    if (threadIdx.x == 0) {
        out[blockIdx.x * 2 + 0] = v[0];
        out[blockIdx.x * 2 + 1] = v[1];
    }
}

// ---------------- certificate ----------------
// Q = P(x+) - P(y) with P = omtv grad h_mu(D .), then
// r = (y - x+)(1/tau - w) + lambda_tv D^T Q and the sum of r^2 (D^T is
// linear: D^T P(x+) - D^T P(y) = D^T Q). One march like the adjoint passes'
// (a CTA owns TY rows of a 128-voxel chunk over zc planes, one more warp the
// row below the tile): Q is evaluated once per voxel on the next plane and kept
// in registers, its y-component passing through a 3-plane shared ring; nothing
// is stored. Bound: x+, x_k, the pair, omtv and w, 20 bytes a voxel; as in the
// adjoint passes the loads of a plane are issued an iteration before their use
// (issued where they were used, this march took 1649 us at 512^3, more than the
// 1307 of two passes that stored Q as three fields). Whole call, the two passes ->
// this: 128^3 56 -> 43 us, 256^3 224 -> 159, 512^3 1307 -> 1024 (at the copy rate
// 396): with 16 warps per SM still the latency of their loads.
// x+, x_k and aux (d_k with xd, else x_{k-1}) are iterate buffers.
struct CertRow {
    float xp[4], xk[4], d[4];  // x+, x_k, d_k
};

// Q at one voxel from the differences of x+ and of y.
__device__ __forceinline__ void cert_q1(const float (&gp)[3], const float (&gy)[3], float ot, float mu, float (&q)[3])
{
    const float sp = ot * fminf(1.0f / mu, rsqrtf(gp[0] * gp[0] + gp[1] * gp[1] + gp[2] * gp[2]));
    const float sy = ot * fminf(1.0f / mu, rsqrtf(gy[0] * gy[0] + gy[1] * gy[1] + gy[2] * gy[2]));
#pragma unroll
    for (int c = 0; c < 3; c++) q[c] = gp[c] * sp - gy[c] * sy;
}

__global__ void __launch_bounds__(adj::THREADS, 2)
    certificate_kernel(AuxParams a, int vol, int zc, const float *xplus, const float *xk, const float *aux, int xd_,
                       const void *w, bool bf16, const float *omtv)
{
    __shared__ __align__(16) float ring[3][adj::TY + 1][128];
    __shared__ double red[32 * 4 + 16];
    __shared__ int flag;
    const VolDesc V = a.vols[vol];
    const bool xd = xd_ != 0;
    AdjPlace P = adj_place(V, zc);
    Lane4 &L = P.L;
    const float beta = V.beta_last;  // extrapolation weight of the step that produced x+
    const float mu = V.mu, inv_tau = 1.0f / V.tau;
    const bool writes = P.r < adj::TY && P.row_in;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    RowLoads rp, rk, ra;
    float4 rot, fw;  // omtv of the next plane, w of this one
    auto load_rows = [&](long long i, bool ok) {
        rp.load(V, L, xplus, i, ok);
        rk.load(V, L, xk, i, ok);
        ra.load(V, L, aux, i, ok);
        rot = ldz4(omtv + i, ok);
    };
    auto load_w = [&](long long i, bool ok) { fw = ok ? ld4_data(w, bf16, i) : zero; };
    // Q at the loaded rows' plane z, the plane below in b (have: there is one);
    // also into the ring
    auto q_rows = [&](const CertRow &b, bool have, bool ok, int z, CertRow &c, float (&Q)[3][4]) {
        float up[4], uk[4], ua[4], ac[4], ot[4], pl, kl, al;
        rp.take(L, c.xp, pl, up);
        rk.take(L, c.xk, kl, uk);
        ra.take(L, ac, al, ua);
        unpack4(rot, ot);
#pragma unroll
        for (int q = 0; q < 4; q++) c.d[q] = xd ? ac[q] : c.xk[q] - ac[q];
        const float dl = xd ? al : kl - al;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float ud = xd ? ua[q] : uk[q] - ua[q];
            const float wp = have ? b.xp[q] : c.xp[q], wk = have ? b.xk[q] : c.xk[q], wd = have ? b.d[q] : c.d[q];
            const float lp = q ? c.xp[q - 1] : pl, lk = q ? c.xk[q - 1] : kl, ld = q ? c.d[q - 1] : dl;
            const float gp[3] = {c.xp[q] - lp, c.xp[q] - up[q], c.xp[q] - wp};
            const float gy[3] = {(c.xk[q] - lk) + beta * (c.d[q] - ld), (c.xk[q] - uk[q]) + beta * (c.d[q] - ud),
                                 (c.xk[q] - wk) + beta * (c.d[q] - wd)};
            float t[3];
            cert_q1(gp, gy, ot[q], mu, t);
            const bool valid = ok && L.x0 + q < V.nx;
#pragma unroll
            for (int k = 0; k < 3; k++) Q[k][q] = valid ? t[k] : 0.f;
        }
        *reinterpret_cast<float4 *>(&ring[z % 3][P.r][4 * L.lane]) = make_float4(Q[1][0], Q[1][1], Q[1][2], Q[1][3]);
    };
    KSum ks;
    CertRow c;
    float Qc[3][4];
    L.i = P.row_in ? adj_row(V, L.x0, L.y, P.z0) : 0;
    {
        CertRow b;
        float ab[4];
        const bool below = L.act && P.z0 >= 1;
        load_rows(L.i, L.act);
        unpack4(ldz4(xplus + L.i - P.PS, below), b.xp);
        unpack4(ldz4(xk + L.i - P.PS, below), b.xk);
        unpack4(ldz4(aux + L.i - P.PS, below), ab);
#pragma unroll
        for (int q = 0; q < 4; q++) b.d[q] = xd ? ab[q] : b.xk[q] - ab[q];
        load_w(L.i, L.act && writes);
        q_rows(b, P.z0 >= 1, L.act, P.z0, c, Qc);
        load_rows(L.i + P.PS, L.act && P.z0 + 1 < V.nz);
    }
    for (int z = P.z0; z < P.z1; z++) {
        const long long in_ = L.i + P.PS;
        CertRow n;
        float Qn[3][4];
        q_rows(c, true, L.act && z + 1 < V.nz, z + 1, n, Qn);
        load_rows(in_ + P.PS, L.act && z + 1 < P.z1 && z + 2 < V.nz);
        __syncthreads();  // Q_y of plane z of every row of the tile is in the ring
        // Q_x at x+1: the next lane's first voxel; a chunk's last lane evaluates it
        float qxn = __shfl_down_sync(FULL, Qc[0][0], 1);
        if (L.lane == 31) {
            qxn = 0.f;
            if (L.act && L.x0 + 4 < V.nx) {
                const long long j = L.i + 4;
                auto d_at = [&](long long e) { return xd ? aux[e] : xk[e] - aux[e]; };
                const bool u = L.y >= 1, b = z >= 1;
                const float p0 = xplus[j], k0 = xk[j], d0 = d_at(j);
                const long long ju = j - V.pitch, jb = j - P.PS;
                const float pu = u ? xplus[ju] : p0, ku = u ? xk[ju] : k0, du = u ? d_at(ju) : d0;
                const float pb = b ? xplus[jb] : p0, kb = b ? xk[jb] : k0, db = b ? d_at(jb) : d0;
                const float gp[3] = {p0 - c.xp[3], p0 - pu, p0 - pb};
                const float gy[3] = {(k0 - c.xk[3]) + beta * (d0 - c.d[3]), (k0 - ku) + beta * (d0 - du),
                                     (k0 - kb) + beta * (d0 - db)};
                float t[3];
                cert_q1(gp, gy, omtv[j], mu, t);
                qxn = t[0];
            }
        }
        if (writes) {
            const float4 qyv = *reinterpret_cast<const float4 *>(&ring[z % 3][P.r + 1][4 * L.lane]);
            const float qy[4] = {qyv.x, qyv.y, qyv.z, qyv.w};  // zero when row y + 1 is outside
            float wv[4];
            unpack4(fw, wv);
            load_w(in_, L.act && z + 1 < P.z1);
            float acc = 0.f;
            if (z >= V.halo_lo && z < V.nz - V.halo_hi) {
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    if (!(L.act && L.x0 + q < V.nx)) continue;
                    const float qx = L.x0 + q + 1 >= V.nx ? 0.f : (q < 3 ? Qc[0][q + 1] : qxn);
                    const float dy = (c.xk[q] - c.xp[q]) + beta * c.d[q];
                    const float dv = (Qc[0][q] - qx) + (Qc[1][q] - qy[q]) + (Qc[2][q] - Qn[2][q]);
                    const float r = dy * (inv_tau - wv[q]) + V.lambda_tv * dv;
                    acc += r * r;
                }
            }
            ks.add(acc);
        }
        c = n;
#pragma unroll
        for (int k = 0; k < 3; k++)
#pragma unroll
            for (int q = 0; q < 4; q++) Qc[k][q] = Qn[k][q];
        L.i = in_;
    }
    const ff::FF v[4] = {ks.pair(), {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    const double s = block_sum4(v, red);
    if (threadIdx.x < 4) a.plane_part[(long long)blockIdx.x * 4 + threadIdx.x] = s;
    if (!last_block(&a.st->ticket_aux, &flag)) return;
    double t[4];
    float mx;
    part_total(a.plane_part, 0, (int)gridDim.x, (int)(threadIdx.x >> 5), (int)(blockDim.x >> 5), false, red, t, mx);
    if (threadIdx.x == 0) {
        a.vol_out[(long long)vol * 8 + 4] = t[0];
        a.st->ticket_aux = 0;
        __threadfence();
    }
}

}  // namespace

cudaError_t launch_validate(const AuxParams &a, int vol, int nitems, const void *b, const void *w, bool bf16,
                            double *maxw_out, cudaStream_t s)
{
    validate_kernel<<<nitems, AUX_THREADS, 0, s>>>(a, vol, b, w, bf16, maxw_out);
    return cudaGetLastError();
}

cudaError_t launch_ingest(const AuxParams &a, int vol, int nitems, int nx, const void *sb, const void *sw, bool src16,
                          void *b, void *w, bool dst16, double *maxw_out, cudaStream_t s)
{
    const uintptr_t align = src16 ? 8 : 16;
    const bool vec = nx % 4 == 0 && ((reinterpret_cast<uintptr_t>(sb) | reinterpret_cast<uintptr_t>(sw)) % align) == 0;
    auto go = [&](auto k) { k<<<nitems, AUX_THREADS, 0, s>>>(a, vol, sb, sw, b, w, maxw_out); };
    if (src16 && dst16)
        vec ? go(ingest_kernel<true, true, true>) : go(ingest_kernel<true, true, false>);
    else if (src16)
        vec ? go(ingest_kernel<true, false, true>) : go(ingest_kernel<true, false, false>);
    else if (dst16)
        vec ? go(ingest_kernel<false, true, true>) : go(ingest_kernel<false, true, false>);
    else
        vec ? go(ingest_kernel<false, false, true>) : go(ingest_kernel<false, false, false>);
    return cudaGetLastError();
}

cudaError_t launch_anchor(const AuxParams &a, int vol, int nitems, void *b, void *w, bool bf16, const float *anchor,
                          float gamma, double *maxw_out, cudaStream_t s)
{
    anchor_kernel<<<nitems, AUX_THREADS, 0, s>>>(a, vol, b, w, bf16, anchor, gamma, maxw_out);
    return cudaGetLastError();
}

cudaError_t launch_scales(const AuxParams &a, int vol, int nz, const void *b, const void *w, bool bf16,
                          cudaStream_t s)
{
    scales_kernel<<<nz * AUX_SEG, AUX_THREADS, 0, s>>>(a, vol, b, w, bf16);
    return cudaGetLastError();
}

// In-place reversal of every axis of one pitched volume: element (z, y, x)
// trades places with (nz-1-z, ny-1-y, nx-1-x). Element i of the unpadded
// order pairs with element nvox-1-i, so the first half of the order visits
// every pair once (the middle element of an odd volume stays); padding is
// not touched.
template <typename T>
__global__ void __launch_bounds__(256) reverse_axes_kernel(T *v, int nx, int ny, int pitch, long long nvox)
{
    const long long half = nvox / 2;
    const long long nxy = (long long)nx * ny;
    auto at = [&](long long i) {
        const long long z = i / nxy;
        const long long r = i - z * nxy;
        const long long y = r / nx;
        return (z * ny + y) * pitch + (r - y * nx);
    };
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < half;
         i += (long long)gridDim.x * blockDim.x) {
        const long long a = at(i), b = at(nvox - 1 - i);
        const T t = v[a];
        v[a] = v[b];
        v[b] = t;
    }
}

cudaError_t launch_reverse_axes(void *v, size_t es, int nx, int ny, int nz, int pitch, cudaStream_t s)
{
    const long long nvox = (long long)nx * ny * nz;
    const long long half = nvox / 2;
    if (half == 0) return cudaSuccess;
    const int grid = (int)std::min<long long>((half + 255) / 256, 4096);
    if (es == 4)
        reverse_axes_kernel<uint32_t><<<grid, 256, 0, s>>>(static_cast<uint32_t *>(v), nx, ny, pitch, nvox);
    else if (es == 2)
        reverse_axes_kernel<uint16_t><<<grid, 256, 0, s>>>(static_cast<uint16_t *>(v), nx, ny, pitch, nvox);
    else
        return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_convert_to_bf16(const float *src, uint16_t *dst, long long n, cudaStream_t s)
{
    to_bf16_kernel<<<1024, 256, 0, s>>>(src, dst, n);
    return cudaGetLastError();
}

cudaError_t launch_convert_to_f32(const uint16_t *src, float *dst, long long n, cudaStream_t s)
{
    to_f32_kernel<<<1024, 256, 0, s>>>(src, dst, n);
    return cudaGetLastError();
}

cudaError_t launch_reweight(const AuxParams &a, const float *const *xbuf, float *om1, float *omtv,
                            const double *maxw, double *rstats, VolDesc *vols_rw, cudaStream_t s)
{
    if (a.readings == 0)
        reweight_march_kernel<<<a.nitems, AUX_THREADS, 0, s>>>(a, xbuf[0], om1, omtv, maxw, rstats, vols_rw);
    else
        reweight_kernel<<<a.nplanes * AUX_SEG, AUX_THREADS, 0, s>>>(a, xbuf[0], om1, omtv, maxw, rstats, vols_rw);
    return cudaGetLastError();
}

cudaError_t launch_objective(const AuxParams &a, const float *const *xbuf, const void *b, const void *w,
                             bool bf16, const float *om1, const float *omtv, cudaStream_t s)
{
    if (a.readings == 0)
        objective_march_kernel<<<a.nitems, AUX_THREADS, 0, s>>>(a, xbuf[0], b, w, bf16, om1, omtv);
    else
        objective_kernel<<<a.nplanes * AUX_SEG, AUX_THREADS, 0, s>>>(a, xbuf[0], b, w, bf16, om1, omtv);
    return cudaGetLastError();
}

// Planes per CTA of the certificate: about 4 waves of 2 CTAs per SM, at most 32.
static int certificate_chunk(int nx, int ny, int nz)
{
    const long long tiles = (long long)((nx + 127) / 128) * ((ny + adj::TY - 1) / adj::TY) * nz;
    return (int)std::max<long long>(2, std::min<long long>(32, tiles / 1216));
}

int certificate_blocks(int nx, int ny, int nz)
{
    const int zc = certificate_chunk(nx, ny, nz);
    return ((nx + 127) / 128) * ((ny + adj::TY - 1) / adj::TY) * ((nz + zc - 1) / zc);
}

cudaError_t launch_certificate(const AuxParams &a, int vol, int nx, int ny, int nz, const float *const *xbuf,
                               const void *w, bool bf16, const float *omtv, cudaStream_t s)
{
    const bool xd = xbuf[3] != nullptr;
    certificate_kernel<<<certificate_blocks(nx, ny, nz), adj::THREADS, 0, s>>>(
        a, vol, certificate_chunk(nx, ny, nz), xbuf[0], xbuf[1], xd ? xbuf[3] : xbuf[2], xd ? 1 : 0, w, bf16, omtv);
    return cudaGetLastError();
}

std::vector<WorkItem> aux_items(const std::vector<VolDesc> &vols, std::vector<std::pair<int, int>> *ranges)
{
    long long tiles = 0;
    for (const auto &d : vols) tiles += (long long)((d.nx + 127) / 128) * ((d.ny + 7) / 8) * d.nz;
    // planes per item: about two waves of 4 CTAs per SM, 2 .. 32 planes (an
    // item reads the plane below its first one again)
    const int zc = (int)std::max<long long>(2, std::min<long long>(32, tiles / 1216));
    std::vector<WorkItem> items;
    ranges->clear();
    for (size_t j = 0; j < vols.size(); j++) {
        const auto &d = vols[j];
        const int begin = (int)items.size();
        for (int z = 0; z < d.nz; z += zc)
            for (int y = 0; y < d.ny; y += 8)
                for (int x = 0; x < d.nx; x += 128)
                    items.push_back(WorkItem{(int)j, x, y, z, std::min(d.nz, z + zc), 0, 0, 0});
        ranges->push_back({begin, (int)items.size()});
    }
    return items;
}

cudaError_t launch_generic_step(const GenericParams &g, cudaStream_t s)
{
    generic_step_kernel<<<g.nplanes * AUX_SEG, AUX_THREADS, 0, s>>>(g);
    return cudaGetLastError();
}

// `early`: the launch ahead on the stream is the other pass (then its CTAs may
// still be running, and the CTAs of this one start as they end and load what
// that pass does not write); false behind anything else.
static cudaError_t launch_adjoint(void (*kernel)(AdjParams), const AdjParams &a, bool early, cudaStream_t s)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)a.nblocks);
    cfg.blockDim = dim3(adj::THREADS);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, a);
}

cudaError_t launch_adjoint_mask(const AdjParams &a, bool early, cudaStream_t s)
{
    return launch_adjoint(adjoint_mask_kernel, a, early, s);
}

cudaError_t launch_adjoint_scalars(const double *part, int nblk, int K, double *out, cudaStream_t s)
{
    adjoint_scalars_kernel<<<K, 128, 0, s>>>(part, nblk, out);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_apply(const AdjParams &a, cudaStream_t s)
{
    return launch_adjoint(adjoint_apply_kernel, a, true, s);  // always behind its mask pass
}

int adjoint_blocks(int nx, int ny, int nz)
{
    return ((nx + 127) / 128) * ((ny + adj::TY - 1) / adj::TY) * ((nz + adj::ZC - 1) / adj::ZC);
}

}  // namespace spg
