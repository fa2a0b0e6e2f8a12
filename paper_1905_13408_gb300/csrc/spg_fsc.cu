// Fourier shell correlation of two maps (Sec. 2.3, Eq. 30) on the GPU:
// cuFFT real-to-complex transforms of both maps, then one pass that bins
// every coefficient of the half spectrum into its shell and accumulates
// Re(F G*), |F|^2, |G|^2 and the coefficient count. Coefficients with
// 0 < h < n/2 stand for themselves and their conjugates (weight 2).
#include <cuda_runtime.h>
#include <cufft.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>
#include <vector>

#include <stdint.h>

#include "spg.h"
#include "spg_trace.h"
#include "spg_cufft.h"
#include "spg_ff.cuh"
#include "spg_range.h"

namespace {

using spg::ff::FF;

constexpr int kThreads = 256;
constexpr int kBlocks = 1216;  // 8 per SM on 152 SMs

thread_local std::string g_fsc_err = "no error";

// Nearest integer to sqrt(r2) for an integer r2 (no tie: (s + 1/2)^2 is never an integer).
__device__ __forceinline__ int shell_of(long long r2)
{
    long long s = (long long)sqrt((double)r2);
    while (s * s > r2) s--;
    while ((s + 1) * (s + 1) <= r2) s++;
    return (int)(r2 > s * s + s ? s + 1 : s);
}

__device__ __forceinline__ int freq(int i, int n) { return i <= (n - 1) / 2 ? i : i - n; }

// ---- shell sums, float-float ----
// Bound: reading the two half spectra inside the sphere of radius n/2 (half of
// all coefficients: 70 MB of 135 at 256^3, 10 us). A pass with one FP64
// shared-memory atomic per coefficient and sum took 538 us there (atomics on
// doubles loop, and neighbouring lanes hit the same shell; the FP64 pipe
// alone would need 140 us), and the counts, with global atomics on n/2 + 1
// addresses, another 600. The whole call on two 256^3 device maps went from 2.68
// to 0.30 ms with this pass, the kept plans and the caller's workspace.
//
// A lane takes one h and the up to 8 coefficients (h, +-k, +-l), (h, +-l, +-k),
// which lie on one shell: their products are exact pairs (Dekker's
// two-product by fused multiply-add) summed in float-float registers. The
// shell index does not fall with h, so the lanes of a warp (32 consecutive h)
// that share a shell are neighbours: a segmented scan over the lanes leaves
// each segment's sum in its last lane, which adds it to the warp's own table in
// shared memory without atomics. The sums' order is fixed.
//
// Range: the pairs need |component| < 1e14 (sums of squares below 1e38) and,
// for the rounding terms, a largest component above 1e-8 (or 0) of each map in
// each lane (the squares of one map do not see the other's scale); otherwise
// `flag` is set and the caller runs the double kernel below.
__device__ __forceinline__ FF two_prod_add(FF acc, float a, float b)
{
    const float p = __fmul_rn(a, b);
    return spg::ff::add(acc, FF{p, fmaf(a, b, -p)});
}

__device__ __forceinline__ FF ff_shfl_up(FF a, int d)
{
    return {__shfl_up_sync(0xffffffffu, a.hi, d), __shfl_up_sync(0xffffffffu, a.lo, d)};
}

__global__ void __launch_bounds__(256) fsc_shell_ff_kernel(const float2 *__restrict__ F, const float2 *__restrict__ G,
                                                           int n, int nshell, double *__restrict__ partials, int *flag)
{
    extern __shared__ FF tab[];  // [warps][nshell][3], then counts [warps][nshell]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    FF *const mine = tab + (size_t)warp * nshell * 3;
    unsigned *const counts = reinterpret_cast<unsigned *>(tab + (size_t)warps * nshell * 3);
    unsigned *const mycount = counts + (size_t)warp * nshell;
    for (int i = lane; i < nshell * 3; i += 32) mine[i] = FF{0.f, 0.f};
    for (int i = lane; i < nshell; i += 32) mycount[i] = 0;
    __syncwarp();
    const int nh = n / 2 + 1, Q = n / 2 + 1;  // |k|, |l| = 0 .. n/2
    const int R = nshell - 1;                 // last shell; s <= R <=> r^2 <= R^2 + R
    const int r2max = R * R + R;
    bool bad = false;
    for (int it = blockIdx.x * warps + warp; it < Q * Q; it += gridDim.x * warps) {
        const int l = it / Q, k = it % Q;
        const int kl2 = k * k + l * l;
        if (k > l || kl2 > r2max) continue;
        // index lists of |k| and |l| (the Nyquist index of an even n and 0 have one)
        const int nk = (k == 0 || 2 * k == n) ? 1 : 2, nl = (l == 0 || 2 * l == n) ? 1 : 2;
        const int swaps = k == l ? 1 : 2;
        for (int h0 = 0; h0 < nh && kl2 + h0 * h0 <= r2max; h0 += 32) {
            const int h = h0 + lane;
            const int r2 = kl2 + h * h;
            const bool in = h < nh && r2 <= r2max;
            FF re{0.f, 0.f}, fa{0.f, 0.f}, gb{0.f, 0.f};
            int key = nshell;  // lanes outside: a segment of their own, dropped
            unsigned cnt = 0;
            if (in) {
                int s = (int)sqrtf((float)r2);
                while (s * s > r2) s--;
                while ((s + 1) * (s + 1) <= r2) s++;
                key = r2 > s * s + s ? s + 1 : s;
                float2 a[8], b[8];
                float ma = 0.f, mb = 0.f;
#pragma unroll
                for (int c = 0; c < 8; c++) {
                    const int sw = c >> 2, ik = (c >> 1) & 1, il = c & 1;
                    a[c] = b[c] = make_float2(0.f, 0.f);
                    if (sw < swaps && ik < nk && il < nl) {
                        const int kk = ik ? n - k : k, ll = il ? n - l : l;
                        const long long row = sw ? (long long)kk * n + ll : (long long)ll * n + kk;
                        a[c] = __ldcs(F + row * nh + h);
                        b[c] = __ldcs(G + row * nh + h);
                    }
                }
#pragma unroll
                for (int c = 0; c < 8; c++) {
                    const float4 v = make_float4(fabsf(a[c].x), fabsf(a[c].y), fabsf(b[c].x), fabsf(b[c].y));
                    // written so that a NaN fails the test
                    if (!(v.x < 1e14f && v.y < 1e14f && v.z < 1e14f && v.w < 1e14f)) bad = true;
                    ma = fmaxf(ma, fmaxf(v.x, v.y));
                    mb = fmaxf(mb, fmaxf(v.z, v.w));
                    re = two_prod_add(two_prod_add(re, a[c].x, b[c].x), a[c].y, b[c].y);
                    fa = two_prod_add(two_prod_add(fa, a[c].x, a[c].x), a[c].y, a[c].y);
                    gb = two_prod_add(two_prod_add(gb, b[c].x, b[c].x), b[c].y, b[c].y);
                }
                if ((ma > 0.f && ma < 1e-8f) || (mb > 0.f && mb < 1e-8f)) bad = true;
                cnt = nk * nl * swaps;
                if (h > 0 && 2 * h != n) {  // the conjugates (exact doubling)
                    re = {2.f * re.hi, 2.f * re.lo};
                    fa = {2.f * fa.hi, 2.f * fa.lo};
                    gb = {2.f * gb.hi, 2.f * gb.lo};
                    cnt *= 2;
                }
            }
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int ku = __shfl_up_sync(0xffffffffu, key, d);
                const FF ur = ff_shfl_up(re, d), uf = ff_shfl_up(fa, d), ug = ff_shfl_up(gb, d);
                const unsigned uc = __shfl_up_sync(0xffffffffu, cnt, d);
                if (lane >= d && ku == key) {
                    re = spg::ff::add(ur, re);
                    fa = spg::ff::add(uf, fa);
                    gb = spg::ff::add(ug, gb);
                    cnt += uc;
                }
            }
            const int kn = __shfl_down_sync(0xffffffffu, key, 1);
            if (key < nshell && (lane == 31 || kn != key)) {
                FF *const t = mine + 3 * key;
                t[0] = spg::ff::add(t[0], re);
                t[1] = spg::ff::add(t[1], fa);
                t[2] = spg::ff::add(t[2], gb);
                mycount[key] += cnt;
            }
            __syncwarp();
        }
    }
    if (__syncthreads_or(bad ? 1 : 0) && threadIdx.x == 0) *flag = 1;
    // the block's sums: warps in order; partials[quantity][shell][block]
    for (int i = threadIdx.x; i < nshell * 4; i += blockDim.x) {
        const int s = i >> 2, q = i & 3;
        double v = 0.0;
        if (q < 3) {
            FF t = tab[3 * s + q];
            for (int w = 1; w < warps; w++) t = spg::ff::add(t, tab[((size_t)w * nshell + s) * 3 + q]);
            v = spg::ff::to_double(t);
        } else {
            unsigned long long c = 0;
            for (int w = 0; w < warps; w++) c += counts[(size_t)w * nshell + s];
            v = (double)c;
        }
        partials[((size_t)q * nshell + s) * gridDim.x + blockIdx.x] = v;
    }
}

// One warp per (quantity, shell): its block partials, summed in a fixed order.
__global__ void fsc_sum_kernel(const double *__restrict__ partials, int nblocks, int nout, double *out)
{
    const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= nout) return;
    double s = 0.0;
    for (int b = lane; b < nblocks; b += 32) s += partials[(size_t)i * nblocks + b];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) out[i] = s;
}

// ---- shell sums in double, for values outside the float-float range ----
// Per-block shell sums in shared memory, written to partials[block][shell][3].
__global__ void fsc_shell_kernel(const cufftComplex *__restrict__ F, const cufftComplex *__restrict__ G, int n,
                                 int nshell, double *partials)
{
    extern __shared__ double acc[];  // [nshell][3]
    for (int i = threadIdx.x; i < nshell * 3; i += blockDim.x) acc[i] = 0.0;
    __syncthreads();
    const int nh = n / 2 + 1;
    const long long total = (long long)n * n * nh;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < total;
         q += (long long)gridDim.x * blockDim.x) {
        const int h = (int)(q % nh);
        const int k = (int)((q / nh) % n);
        const int l = (int)(q / ((long long)nh * n));
        const long long fk = freq(k, n), fl = freq(l, n);
        const int s = shell_of((long long)h * h + fk * fk + fl * fl);
        if (s >= nshell) continue;
        const double wgt = (h == 0 || (n % 2 == 0 && h == n / 2)) ? 1.0 : 2.0;
        const cufftComplex a = F[q], b = G[q];
        const double re = (double)a.x * b.x + (double)a.y * b.y;
        const double fa = (double)a.x * a.x + (double)a.y * a.y;
        const double gb = (double)b.x * b.x + (double)b.y * b.y;
        atomicAdd(&acc[s * 3 + 0], wgt * re);
        atomicAdd(&acc[s * 3 + 1], wgt * fa);
        atomicAdd(&acc[s * 3 + 2], wgt * gb);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nshell * 3; i += blockDim.x) partials[(long long)blockIdx.x * nshell * 3 + i] = acc[i];
}

// Sum the block partials of every shell in block order; out[shell][3].
__global__ void fsc_reduce_kernel(const double *partials, int nblocks, int nshell, double *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nshell * 3) return;
    double s = 0.0;
    for (int b = 0; b < nblocks; b++) s += partials[(long long)b * nshell * 3 + i];
    out[i] = s;
}

// Plans kept between calls: making one costs more than the two transforms.
// A plan holds no work area (each call passes its own) and is in one call's
// hands at a time, so calls from several threads and streams use plans of
// their own; a call returns its plan after it has waited for its stream. At
// most kMaxIdle plans are idle; the one idle longest is destroyed.
struct PlanPool {
    static constexpr size_t kMaxIdle = 4;
    struct Entry {
        int dev, n;
        cufftHandle h;
        size_t work;
    };
    std::mutex mu;
    std::vector<Entry> idle;

    bool take(int dev, int n, Entry *e)
    {
        std::lock_guard<std::mutex> lk(mu);
        for (size_t i = idle.size(); i-- > 0;)
            if (idle[i].dev == dev && idle[i].n == n) {
                *e = idle[i];
                idle.erase(idle.begin() + i);
                return true;
            }
        return false;
    }
    void give(const Entry &e)
    {
        Entry old{};
        bool drop = false;
        {
            std::lock_guard<std::mutex> lk(mu);
            idle.push_back(e);
            if (idle.size() > kMaxIdle) {
                old = idle.front();
                idle.erase(idle.begin());
                drop = true;
            }
        }
        if (drop) spg::cufft_api().destroy(old.h);
    }
};

PlanPool &plan_pool()
{
    static PlanPool *p = new PlanPool;  // never destroyed: cuFFT may be gone by process exit
    return *p;
}

// The plan of one call: from the pool or new, back to the pool in the end
// (destroyed instead after a failure).
struct CallPlan {
    PlanPool::Entry e{};
    bool have = false, good = false;
    bool get(int dev, int n)
    {
        if (plan_pool().take(dev, n, &e)) return have = true;
        const spg::CufftApi &cf = spg::cufft_api();
        e.dev = dev;
        e.n = n;
        if (cf.create(&e.h) != CUFFT_SUCCESS) return false;
        if (cf.set_auto_allocation(e.h, 0) != CUFFT_SUCCESS ||
            cf.make_plan3d(e.h, n, n, n, CUFFT_R2C, &e.work) != CUFFT_SUCCESS) {
            cf.destroy(e.h);
            return false;
        }
        return have = true;
    }
    ~CallPlan()
    {
        if (!have) return;
        if (good)
            plan_pool().give(e);
        else
            spg::cufft_api().destroy(e.h);
    }
};

struct Buf {
    void *p = nullptr;
    ~Buf()
    {
        if (p) cudaFree(p);
    }
};

// Launch shape of the shell pass: warps per block (each with a table of the
// shells, 28 bytes a shell) and blocks.
struct ShellShape {
    int warps, blocks;
    size_t smem;
};

ShellShape shell_shape(int n)
{
    const int nshell = n / 2 + 1;
    const size_t per_warp = (size_t)nshell * (3 * sizeof(FF) + sizeof(unsigned));
    ShellShape s;
    s.warps = (int)std::max<size_t>(1, std::min<size_t>(8, (96 * 1024) / per_warp));
    s.smem = per_warp * s.warps;
    const long long items = (long long)nshell * nshell;
    s.blocks = (int)std::min<long long>(456, (items + s.warps - 1) / s.warps);  // 3 per SM
    return s;
}

// Byte offsets of a call's device buffers in its workspace.
struct Layout {
    size_t fa, fb, work, part, sums, flag, ra, rb, total;
};

size_t up256(size_t b) { return (b + 255) & ~size_t(255); }

Layout layout(int n, size_t work, bool copy_a, bool copy_b)
{
    const int nshell = n / 2 + 1;
    const size_t vox = (size_t)n * n * n * sizeof(float);
    const size_t spec = (size_t)n * n * (n / 2 + 1) * sizeof(float2);
    Layout L{};
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off += up256(bytes);
        return at;
    };
    L.fa = take(spec);
    L.fb = take(spec);
    L.work = take(work);
    L.part = take((size_t)shell_shape(n).blocks * nshell * 4 * sizeof(double));
    L.sums = take((size_t)(nshell * 4 + 1) * sizeof(double));  // sums, counts, then the range flag
    L.flag = L.sums + (size_t)nshell * 4 * sizeof(double);
    L.ra = copy_a ? take(vox) : 0;
    L.rb = copy_b ? take(vox) : 0;
    L.total = off;
    return L;
}

spg_status fsc_fail(spg_status s, const std::string &m)
{
    g_fsc_err = m;
    return s;
}

}  // namespace

extern "C" const char *spg_fsc_last_error(void) { return g_fsc_err.c_str(); }

namespace {

#define FSC_CK(call)                                                                                \
    do {                                                                                            \
        cudaError_t e_ = (call);                                                                    \
        if (e_ != cudaSuccess) {                                                                    \
            cudaGetLastError();                                                                     \
            return fsc_fail(e_ == cudaErrorMemoryAllocation ? SPG_ENOMEM : SPG_ECUDA,               \
                            std::string("spg_fsc: ") + cudaGetErrorString(e_));                     \
        }                                                                                           \
    } while (0)

// The double kernels: shell sums, then the counts stay those of the first pass.
spg_status sums_in_double(const float2 *fa, const float2 *fb, int n, int nshell, double *sums_d, double *hs,
                          cudaStream_t s)
{
    Buf part;
    FSC_CK(cudaMalloc(&part.p, (size_t)kBlocks * nshell * 3 * sizeof(double)));
    fsc_shell_kernel<<<kBlocks, kThreads, (size_t)nshell * 3 * sizeof(double), s>>>(fa, fb, n, nshell,
                                                                                     static_cast<double *>(part.p));
    fsc_reduce_kernel<<<(nshell * 3 + 255) / 256, 256, 0, s>>>(static_cast<double *>(part.p), kBlocks, nshell, sums_d);
    FSC_CK(cudaGetLastError());
    std::vector<double> h3((size_t)nshell * 3);
    FSC_CK(cudaMemcpyAsync(h3.data(), sums_d, h3.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
    FSC_CK(cudaStreamSynchronize(s));
    for (int k = 0; k < nshell; k++)
        for (int q = 0; q < 3; q++) hs[q * nshell + k] = h3[(size_t)k * 3 + q];
    return SPG_OK;
}

spg_status fsc_run(int n, const float *a, const float *b, double *fsc, double *counts, void *ws, size_t ws_bytes,
                   void *stream, size_t *need_out)
{
    const int nshell = n / 2 + 1;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int dev = 0;
    FSC_CK(cudaGetDevice(&dev));
    if ((size_t)nshell * 3 * sizeof(double) > 48 * 1024)
        return fsc_fail(SPG_EINVAL, "spg_fsc: too many shells (n <= 2046)");
    const spg::CufftApi &cf = spg::cufft_api();
    if (!cf.ok) return fsc_fail(SPG_ECUDA, "spg_fsc: cuFFT library could not be loaded");
    const size_t vox = (size_t)n * n * n * sizeof(float);
    const spg::Extent ea = spg::device_extent(a, vox), eb = spg::device_extent(b, vox);
    if (ea == spg::Extent::too_short || eb == spg::Extent::too_short)
        return fsc_fail(SPG_EINVAL, "spg_fsc: a device map is shorter than n^3 values");
    CallPlan plan;
    if (!plan.get(dev, n)) return fsc_fail(SPG_ECUDA, "spg_fsc: cufft plan");
    // a transform reads a map in place when it lies on this device, aligned as
    // an allocation of its own would be; otherwise it is copied first
    const bool ca = ea != spg::Extent::holds || (reinterpret_cast<uintptr_t>(a) & 255) != 0;
    const bool cb = eb != spg::Extent::holds || (reinterpret_cast<uintptr_t>(b) & 255) != 0;
    const Layout L = layout(n, plan.e.work, ca, cb);
    if (need_out) {  // workspace query
        *need_out = L.total;
        plan.good = true;
        return SPG_OK;
    }
    Buf own;
    if (!ws || ws_bytes < L.total) {
        FSC_CK(cudaMalloc(&own.p, L.total));
        ws = own.p;
    }
    char *const base = static_cast<char *>(ws);
    if (ca) FSC_CK(cudaMemcpyAsync(base + L.ra, a, vox, cudaMemcpyDefault, s));
    if (cb) FSC_CK(cudaMemcpyAsync(base + L.rb, b, vox, cudaMemcpyDefault, s));
    float2 *const fa = reinterpret_cast<float2 *>(base + L.fa), *const fb = reinterpret_cast<float2 *>(base + L.fb);
    double *const part = reinterpret_cast<double *>(base + L.part), *const sums = reinterpret_cast<double *>(base + L.sums);
    int *const flag = reinterpret_cast<int *>(base + L.flag);
    float *const ra = ca ? reinterpret_cast<float *>(base + L.ra) : const_cast<float *>(a);
    float *const rb = cb ? reinterpret_cast<float *>(base + L.rb) : const_cast<float *>(b);
    const bool ok = cf.set_stream(plan.e.h, s) == CUFFT_SUCCESS &&
                    cf.set_work_area(plan.e.h, base + L.work) == CUFFT_SUCCESS &&
                    cf.exec_r2c(plan.e.h, ra, fa) == CUFFT_SUCCESS && cf.exec_r2c(plan.e.h, rb, fb) == CUFFT_SUCCESS;
    if (!ok) {
        cudaStreamSynchronize(s);
        return fsc_fail(SPG_ECUDA, "spg_fsc: cufft execution");
    }
    FSC_CK(cudaMemsetAsync(flag, 0, sizeof(double), s));
    const ShellShape sh = shell_shape(n);
    if (sh.smem > 48 * 1024)
        FSC_CK(cudaFuncSetAttribute(fsc_shell_ff_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh.smem));
    fsc_shell_ff_kernel<<<sh.blocks, sh.warps * 32, sh.smem, s>>>(fa, fb, n, nshell, part, flag);
    fsc_sum_kernel<<<(nshell * 4 + 7) / 8, 256, 0, s>>>(part, sh.blocks, nshell * 4, sums);
    FSC_CK(cudaGetLastError());
    std::vector<double> hs((size_t)nshell * 4 + 1);
    FSC_CK(cudaMemcpyAsync(hs.data(), sums, hs.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
    FSC_CK(cudaStreamSynchronize(s));
    if (*reinterpret_cast<const int *>(&hs[(size_t)nshell * 4]) != 0) {
        const spg_status st = sums_in_double(fa, fb, n, nshell, sums, hs.data(), s);
        if (st != SPG_OK) return st;
    }
    plan.good = true;
    for (int k = 0; k < nshell; k++) {
        const double d = std::sqrt(hs[nshell + k] * hs[2 * nshell + k]);
        fsc[k] = d > 0 ? hs[k] / d : NAN;
        if (counts) counts[k] = hs[3 * nshell + k];
    }
    return SPG_OK;
}
#undef FSC_CK

spg_status check_args(int n, const float *a, const float *b, bool rest_ok)
{
    if (n < 2 || !a || !b || !rest_ok)
        return fsc_fail(SPG_EINVAL, "spg_fsc: bad arguments (n >= 2, max_shells >= n/2 + 1)");
    if ((long long)n * n * n > (1LL << 31)) return fsc_fail(SPG_EINVAL, "spg_fsc: volume too large");
    return SPG_OK;
}

}  // namespace

extern "C" spg_status spg_fsc(int n, const float *a, const float *b, int max_shells, double *fsc, double *counts,
                              void *stream)
{
    return spg_fsc_ws(n, a, b, max_shells, fsc, counts, nullptr, 0, stream);
}

extern "C" spg_status spg_fsc_ws(int n, const float *a, const float *b, int max_shells, double *fsc, double *counts,
                                 void *workspace, size_t workspace_bytes, void *stream)
{
    SPG_TRACE();
    const spg_status st = check_args(n, a, b, fsc && max_shells >= n / 2 + 1);
    if (st != SPG_OK) return st;
    if (workspace && (reinterpret_cast<uintptr_t>(workspace) & 255) != 0)
        return fsc_fail(SPG_EINVAL, "spg_fsc: the workspace must be 256-byte aligned");
    return fsc_run(n, a, b, fsc, counts, workspace, workspace_bytes, stream, nullptr);
}

extern "C" spg_status spg_fsc_workspace(int n, const float *a, const float *b, size_t *bytes)
{
    SPG_TRACE();
    const spg_status st = check_args(n, a, b, bytes != nullptr);
    if (st != SPG_OK) return st;
    return fsc_run(n, a, b, nullptr, nullptr, nullptr, 0, nullptr, bytes);
}
