// Passes of the Fourier-domain data term (Sec. 2.5, Eq. 31) for boxes that the
// power-of-two row pass (spg_xpass.cu) does not take, of nx and nz 16 .. 512
// with prime factors of at most 13. As there, an iteration is rows of
// y_k = x_k + beta d_k to spectra held kx-major, [nz][nx/2+1][ny], the library's
// transform along y over contiguous lines, one pass along z (here for nz no
// power of two) with the residual N F / V - C between the forward and the
// inverse transform, y back, and rows back into the b slot.
//
// What it replaces: the library's 3-D transforms around a spectrum pass, which
// moved the spectrum nine times and read a y_k that the fused step wrote for
// them: at 180^3 (where all of it stays in L2) 27 us for the rows of either
// direction, 14.8 for each of four passes along y and z, 12.3 for the spectrum
// pass. What bounds it: latency, its loads' and its barriers' (issue slots 48 %
// taken, 42 % of an SM's warps resident), at about 29 instructions per element
// and radix stage: rows 24 and 22 us, z pass 30 (cold caches, under a profiler).
// An iteration, library -> here: 180^3 170 -> 144 us, 220 x 208 x 176 194 -> 182,
// 224^3 316 -> 260, 300 x 200 x 240 350 -> 308, 384^3 1328 -> 1061, 400^3 2074 ->
// 1420, 448^3 2556 -> 1974, 256 x 256 x 64 90.3 -> 85.7, 112 x 512 x 90 130 -> 122.
// Smaller boxes, where a launch's fixed cost counts, are mixed (128 x 256 x 64
// 56.2 -> 51.2, 140 x 130 x 120 65.9 -> 61.9, 160^3 109.9 -> 108.4, 128 x 176 x 100
// 55.2 -> 56.9) or lose (100^3 41.2 -> 42.4, 64^3 24.7 -> 27.9), and setting the
// data takes two transposes more (20 us), so the line lies at 2^21 coefficients
// (kMixMinHalf), above the last of these.
//
// Tried and slower at 180^3: own passes along y too, on the standard half
// layout (148 us: 18 us a pass), two lines per thread (160: fewer
// instructions, but fewer warps to wait with), 8 columns per CTA in the z pass
// (39 us under the profiler against 30).
//
// Each line goes through a Stockham auto-sort transform (Govindaraju et al.,
// SC 2008; as in spg_zfft.cu) of mixed radices 2 .. 13: for a stage of radix R
// over sub-transforms of span Ns, butterfly j takes the inputs j + r n/R,
// multiplies input r by w^(r k n/(Ns R)) (k = j mod Ns), transforms them with
// an R-point DFT and writes output q to (j - k) R + k + q Ns. A CTA holds 16
// columns, or 8 pairs of rows; consecutive threads take the same butterfly of
// its lines, so that shared memory is free of bank conflicts but for the first
// exchange of even radices (columns: [position][16]; rows: [line][2 modulo
// 16]), the z pass reads and writes runs of 128 bytes and the row passes runs
// of 16 rows, and a stage's index arithmetic is that of one line. The stages go
// from one buffer to the other; the first stage of the z pass reads global
// memory and its last one writes it.
//
// The inverse transform is the forward one with real and imaginary parts
// exchanged before and after. With the radices in reversed order its first
// stage takes exactly the values that a thread holds after the forward
// transform's last stage, so the residual is formed in registers.
//
// Rows are transformed two at a time: u = row_a + i row_b, and
//   A[k] = (U[k] + conj U[n-k]) / 2,  B[k] = -i (U[k] - conj U[n-k]) / 2,
// which takes odd nx as well; back, Z[k] = A[k] + i B[k] and
// Z[n-k] = conj A[k] + i conj B[k], of A[0], A[n/2] only the real parts.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "spg_fft.cuh"
#include "spg_internal.h"

namespace spg {
namespace {

using namespace fft;

constexpr int kRowLines = 8;   // row pairs of a CTA
constexpr int kColLines = 16;  // columns of a CTA

// cos and sin of 2 pi a / b at compile time (Taylor series on [-pi, pi]).
constexpr double series(double x, bool sine)
{
    double term = sine ? x : 1.0, sum = term;
    for (int i = sine ? 3 : 2; i < 40; i += 2) {
        term *= -x * x / ((double)i * (i - 1));
        sum += term;
    }
    return sum;
}
constexpr double angle(int a, int b)
{
    const int m = a % b;
    return 2.0 * 3.14159265358979323846 * (2 * m > b ? m - b : m) / b;
}
template <int A, int B>
struct Root {  // w_B^A = c - i s
    static constexpr float c = (float)series(angle(A, B), false), s = (float)series(angle(A, B), true);
};

template <int I, int N>
struct Static {
    template <class F>
    __device__ static __forceinline__ void run(F &&f)
    {
        if constexpr (I < N) {
            f(std::integral_constant<int, I>{});
            Static<I + 1, N>::run(f);
        }
    }
};

// Forward R-point DFT in place.
template <int R>
__device__ __forceinline__ void dft(float2 (&v)[R])
{
    if constexpr (R == 2) {
        const float2 a = v[0];
        v[0] = cadd(a, v[1]);
        v[1] = csub(a, v[1]);
    } else if constexpr (R == 4) {
        dft4<-1>(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 8) {
        dft8<-1>(v);
    } else if constexpr (R == 6 || R == 9 || R == 10) {
        // R = A B: A-point transforms of the inputs B apart, w_R^(i k), B-point ones
        constexpr int A = R == 9 ? 3 : 2, B = R / A;
        float2 t[A][B];
        Static<0, B>::run([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            float2 u[A];
#pragma unroll
            for (int q = 0; q < A; q++) u[q] = v[B * q + i];
            dft<A>(u);
            Static<0, A>::run([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                using W = Root<i * k, R>;
                t[k][i] = i * k == 0 ? u[k] : cmul(u[k], make_float2(W::c, -W::s));
            });
        });
#pragma unroll
        for (int k = 0; k < A; k++) {
            dft<B>(t[k]);
#pragma unroll
            for (int q = 0; q < B; q++) v[k + A * q] = t[k][q];
        }
    } else {
        // odd: sums and differences of the inputs j and R - j meet the cosines and the sines
        static_assert(R % 2 == 1, "odd radix");
        constexpr int H = (R - 1) / 2;
        const float2 x0 = v[0];
        float2 p[H], m[H];
#pragma unroll
        for (int j = 0; j < H; j++) {
            p[j] = cadd(v[1 + j], v[R - 1 - j]);
            m[j] = csub(v[1 + j], v[R - 1 - j]);
        }
#pragma unroll
        for (int j = 0; j < H; j++) v[0] = cadd(v[0], p[j]);
        Static<1, H + 1>::run([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            float2 a = x0, b = make_float2(0.f, 0.f);
            Static<0, H>::run([&](auto jc) {
                constexpr int j = decltype(jc)::value;
                using W = Root<k *(j + 1), R>;
                a = make_float2(fmaf(p[j].x, W::c, a.x), fmaf(p[j].y, W::c, a.y));
                b = make_float2(fmaf(m[j].x, W::s, b.x), fmaf(m[j].y, W::s, b.y));
            });
            v[k] = make_float2(a.x + b.y, a.y - b.x);  // a - i b
            v[R - k] = make_float2(a.x - b.y, a.y + b.x);
        });
    }
}

extern __shared__ __align__(16) unsigned char msm[];

// Shared memory by byte offset: 32-bit address arithmetic, whichever of the
// two buffers an offset lies in.
__device__ __forceinline__ float2 &at(int byte) { return *reinterpret_cast<float2 *>(msm + byte); }

// A line in shared memory, its positions BYTES apart; in and out are called
// with a position, a step, and a multiple of it known at compile time.
template <int BYTES>
struct Line {
    int base;
    __device__ __forceinline__ float2 operator()(int first, int step, int r) const
    {
        return at(base + first * BYTES + r * (step * BYTES));
    }
    __device__ __forceinline__ void operator()(int first, int step, int r, float2 v) const
    {
        at(base + first * BYTES + r * (step * BYTES)) = v;
    }
};

// One stage of the CTA's lines; the thread's line is threadIdx.x % LINES. tw:
// byte offset of the table.
template <int R, int LINES, class In, class Out>
__device__ __forceinline__ void stage(int tw, int n, int Ns, unsigned inv, const In &in, const Out &out)
{
    const int m = n / R, step = m / Ns;
    for (int j = threadIdx.x / LINES; j < m; j += blockDim.x / LINES) {
        const int k = j - Ns * (int)(((unsigned)j * inv) >> 20);  // j mod Ns
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; r++) v[r] = in(j, m, r);
        if (Ns > 1) {
            const int w = k * step * 8;
#pragma unroll
            for (int r = 1; r < R; r++) v[r] = cmul(v[r], at(tw + r * w));
        }
        dft<R>(v);
        const int to = (j - k) * R + k;
#pragma unroll
        for (int q = 0; q < R; q++) out(to, Ns, q, v[q]);
    }
}

// Last forward stage, `mid` on each value, first inverse stage (real and
// imaginary parts exchanged): outputs at j R + q.
template <int R, int LINES, class In, class Mid, class Out>
__device__ __forceinline__ void turn(int tw, int n, const In &in, const Mid &mid, const Out &out)
{
    const int m = n / R;
    for (int j = threadIdx.x / LINES; j < m; j += blockDim.x / LINES) {
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; r++) v[r] = in(j, m, r);
#pragma unroll
        for (int r = 1; r < R; r++) v[r] = cmul(v[r], at(tw + r * (j * 8)));
        dft<R>(v);
        mid(j, m, v);
        dft<R>(v);
#pragma unroll
        for (int q = 0; q < R; q++) out(j * R, 1, q, v[q]);
    }
}

template <class F>
__device__ __forceinline__ void with_radix(int R, F &&f)
{
    switch (R) {  // the same for every thread
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    case 6: f(std::integral_constant<int, 6>{}); break;
    case 7: f(std::integral_constant<int, 7>{}); break;
    case 8: f(std::integral_constant<int, 8>{}); break;
    case 9: f(std::integral_constant<int, 9>{}); break;
    case 10: f(std::integral_constant<int, 10>{}); break;
    case 11: f(std::integral_constant<int, 11>{}); break;
    case 13: f(std::integral_constant<int, 13>{}); break;
    }
}

struct ColArgs {
    float2 *F;        // [n][inner]
    const float *N;   // as F
    const float2 *C;
    long long inner;
    float scale;
    const float2 *tw;
    MixAxis ax;
};

__global__ void __launch_bounds__(kMixMaxThreads, 4) mix_residual_kernel(const __grid_constant__ ColArgs a)
{
    const int n = a.ax.n, S = a.ax.nst;
    const int c = threadIdx.x % kColLines;
    using Col = Line<kColLines * 8>;
    const int tw = 2 * n * kColLines * 8;
    Col get{c * 8}, put{n * kColLines * 8 + c * 8};
    const long long col = (long long)blockIdx.x * kColLines + c;
    const bool valid = col < a.inner;
    float2 *const F = a.F + col;
    const float *const N = a.N + col;
    const float2 *const C = a.C + col;
    const int inner = (int)a.inner;  // a plane of the half spectrum; the host checks
    for (int i = threadIdx.x; i < n; i += blockDim.x) at(tw + i * 8) = a.tw[i];
    auto load = [&](int first, int step, int r) {
        return valid ? F[(long long)first * inner + r * ((long long)step * inner)] : make_float2(0.f, 0.f);
    };
    auto store = [&](int first, int step, int q, float2 v) {
        if (valid) F[(long long)first * inner + q * ((long long)step * inner)] = make_float2(v.y, v.x);
    };
    auto residual = [&](int first, int step, auto &v) {
        constexpr int R = sizeof(v) / sizeof(float2);
        const long long g = (long long)first * inner, d = (long long)step * inner;
#pragma unroll
        for (int q = 0; q < R; q++) {
            const float m = valid ? N[g + q * d] * a.scale : 0.f;
            const float2 cd = valid ? C[g + q * d] : make_float2(0.f, 0.f);
            v[q] = make_float2(fmaf(v[q].y, m, -cd.y), fmaf(v[q].x, m, -cd.x));
        }
    };
    auto next = [&] {
        __syncthreads();
        const Col t = get;
        get = put;
        put = t;
    };
    with_radix(a.ax.radix[0],
               [&](auto R) { stage<decltype(R)::value, kColLines>(tw, n, 1, 1u << 20, load, put); });
    int Ns = a.ax.radix[0];
    next();
    for (int s = 1; s < S - 1; s++) {
        with_radix(a.ax.radix[s],
                   [&](auto R) { stage<decltype(R)::value, kColLines>(tw, n, Ns, a.ax.inv[s], get, put); });
        Ns *= a.ax.radix[s];
        next();
    }
    with_radix(a.ax.radix[S - 1],
               [&](auto R) { turn<decltype(R)::value, kColLines>(tw, n, get, residual, put); });
    Ns = a.ax.radix[S - 1];
    next();
    for (int s = S - 2; s > 0; s--) {
        with_radix(a.ax.radix[s],
                   [&](auto R) { stage<decltype(R)::value, kColLines>(tw, n, Ns, a.ax.rinv[s], get, put); });
        Ns *= a.ax.radix[s];
        next();
    }
    with_radix(a.ax.radix[0],
               [&](auto R) { stage<decltype(R)::value, kColLines>(tw, n, Ns, a.ax.rinv[0], get, store); });
}

struct RowArgs {
    const float *xs[2], *ds[2];  // forward: the increment-storage pairs
    const DevState *st;
    const VolDesc *vols;
    const float *beta;
    float *out;   // back: [rows][pitch]
    float2 *F;    // [nz][n/2+1][ny]
    long long rows;
    int ny, pitch;
    const float2 *tw;
    MixAxis ax;
};

// Distance of a line's values from the next line's: 2 modulo 16, so that 8
// lines at two neighbouring positions fall on 16 different bank pairs.
__host__ __device__ constexpr int row_stride(int n) { return (n + 13) / 16 * 16 + 2; }

// The lines' transform, from the first of two buffers on; returns the byte
// offset of the result's.
__device__ __forceinline__ int row_stages(const MixAxis &ax, int tw)
{
    const int bytes = row_stride(ax.n) * 8, c = threadIdx.x % kRowLines * bytes;
    int from = 0, to = bytes * kRowLines, Ns = 1;
    for (int s = 0; s < ax.nst; s++) {
        __syncthreads();
        const Line<8> in{from + c}, out{to + c};
        with_radix(ax.radix[s],
                   [&](auto R) { stage<decltype(R)::value, kRowLines>(tw, ax.n, Ns, ax.inv[s], in, out); });
        Ns *= ax.radix[s];
        const int t = from;
        from = to;
        to = t;
    }
    __syncthreads();
    return from;
}

// Where the spectra of rows `row` and `row + 1` start, [nz][n/2+1][ny].
struct RowPair {
    bool in0, in1;
    long long f0, f1;
    __device__ __forceinline__ RowPair(const RowArgs &a, long long row, int nxh)
        : in0(row < a.rows), in1(row + 1 < a.rows)
    {
        const long long z = (unsigned)row / (unsigned)a.ny;  // rows < 2^31
        const int y = (int)(row - z * a.ny);
        f0 = z * nxh * a.ny + y;
        f1 = y + 1 < a.ny ? f0 + 1 : (z + 1) * nxh * a.ny;
    }
};

__global__ void __launch_bounds__(kMixMaxThreads, 4) mix_r2c_kernel(const __grid_constant__ RowArgs a)
{
    const int n = a.ax.n, stride = row_stride(n), nxh = n / 2 + 1;
    float2 *const buf = &at(0);
    const int tw = 2 * stride * kRowLines * 8;
    for (int i = threadIdx.x; i < n; i += blockDim.x) at(tw + i * 8) = a.tw[i];
    // the solver's current pair and extrapolation weight, as the device state holds them when this launch runs
    const int cur = a.st->cur;
    const float *const X = cur == 0 ? a.xs[0] : a.xs[1], *const D = cur == 0 ? a.ds[0] : a.ds[1];
    const float beta = a.beta[a.vols[0].kmom];
    const int lane = threadIdx.x % 32, nwarp = blockDim.x / 32;
    for (int c = threadIdx.x / 32; c < kRowLines; c += nwarp) {
        const long long row = 2 * ((long long)blockIdx.x * kRowLines + c);
        const bool in0 = row < a.rows, in1 = row + 1 < a.rows;
        const float *const x0 = X + row * a.pitch, *const d0 = D + row * a.pitch;
        const float *const x1 = x0 + a.pitch, *const d1 = d0 + a.pitch;
        // two voxels at a time: rows start on 32-byte boundaries and are padded to multiples of 8
#pragma unroll 2
        for (int i = 2 * lane; i < n; i += 64) {
            float2 v0 = make_float2(0.f, 0.f), v1 = v0;
            if (in0) {
                const float2 x = __ldg(reinterpret_cast<const float2 *>(x0 + i));
                const float2 d = __ldg(reinterpret_cast<const float2 *>(d0 + i));
                v0 = make_float2(fmaf(beta, d.x, x.x), fmaf(beta, d.y, x.y));
            }
            if (in1) {
                const float2 x = __ldg(reinterpret_cast<const float2 *>(x1 + i));
                const float2 d = __ldg(reinterpret_cast<const float2 *>(d1 + i));
                v1 = make_float2(fmaf(beta, d.x, x.x), fmaf(beta, d.y, x.y));
            }
            // (an odd row's last pair spills into the line's padding)
            *reinterpret_cast<float4 *>(buf + c * stride + i) = make_float4(v0.x, v1.x, v0.y, v1.y);
        }
    }
    const int c = threadIdx.x % kRowLines;
    const int u = row_stages(a.ax, tw) + c * stride * 8;
    const RowPair rp(a, 2 * ((long long)blockIdx.x * kRowLines + c), nxh);
    const bool wide = a.ny % 2 == 0;  // both rows in one plane, on a 16-byte boundary
    for (int k = threadIdx.x / kRowLines; k < nxh; k += blockDim.x / kRowLines) {
        const float2 p = at(u + k * 8), q = at(u + (k == 0 ? 0 : n - k) * 8);
        const float4 f = make_float4(0.5f * (p.x + q.x), 0.5f * (p.y - q.y), 0.5f * (p.y + q.y), 0.5f * (q.x - p.x));
        float2 *const to = a.F + (long long)k * a.ny;
        if (wide) {
            if (rp.in0) *reinterpret_cast<float4 *>(to + rp.f0) = f;
        } else {
            if (rp.in0) to[rp.f0] = make_float2(f.x, f.y);
            if (rp.in1) to[rp.f1] = make_float2(f.z, f.w);
        }
    }
}

__global__ void __launch_bounds__(kMixMaxThreads, 4) mix_c2r_kernel(const __grid_constant__ RowArgs a)
{
    const int n = a.ax.n, stride = row_stride(n), nxh = n / 2 + 1;
    float2 *const buf = &at(0);
    const int tw = 2 * stride * kRowLines * 8;
    for (int i = threadIdx.x; i < n; i += blockDim.x) at(tw + i * 8) = a.tw[i];
    {
        const int c = threadIdx.x % kRowLines;
        const RowPair rp(a, 2 * ((long long)blockIdx.x * kRowLines + c), nxh);
        const bool wide = a.ny % 2 == 0;
        float2 *const z = buf + c * stride;
#pragma unroll 4
        for (int k = threadIdx.x / kRowLines; k < nxh; k += blockDim.x / kRowLines) {
            const float2 *const from = a.F + (long long)k * a.ny;
            float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
            if (wide) {
                if (rp.in0) f = *reinterpret_cast<const float4 *>(from + rp.f0);
            } else {
                if (rp.in0) {
                    const float2 g = from[rp.f0];
                    f.x = g.x;
                    f.y = g.y;
                }
                if (rp.in1) {
                    const float2 g = from[rp.f1];
                    f.z = g.x;
                    f.w = g.y;
                }
            }
            const bool self = k == 0 || 2 * k == n;
            if (self) f.y = f.w = 0.f;
            // Z[k] and Z[n-k], real and imaginary parts exchanged
            z[k] = make_float2(f.y + f.z, f.x - f.w);
            if (!self) z[n - k] = make_float2(f.z - f.y, f.x + f.w);
        }
    }
    const int u = row_stages(a.ax, tw);
    const int lane = threadIdx.x % 32, nwarp = blockDim.x / 32;
    for (int c = threadIdx.x / 32; c < kRowLines; c += nwarp) {
        const long long row = 2 * ((long long)blockIdx.x * kRowLines + c);
        const bool in0 = row < a.rows, in1 = row + 1 < a.rows;
        float *const y0 = a.out + row * a.pitch, *const y1 = y0 + a.pitch;
        for (int i = lane; i < n; i += 32) {
            const float2 v = at(u + (c * stride + i) * 8);
            if (in0) y0[i] = v.y;
            if (in1) y1[i] = v.x;
        }
    }
}

size_t col_smem(int n) { return (size_t)(n + 2 * n * kColLines) * sizeof(float2); }
size_t row_smem(int n) { return (size_t)(n + 2 * row_stride(n) * kRowLines) * sizeof(float2); }

// Threads of a CTA of `lines` lines: the count that leaves the fewest of them
// without a butterfly in the stages' last rounds, among those that keep an SM
// at 960 threads or more (registers allow 1024, shared memory 227 KB).
int pick_threads(const MixAxis &q, int lines, size_t smem)
{
    double best = 0;
    int threads = 128;
    for (int T = 64; T <= kMixMaxThreads; T += 32) {
        int used = 0, slots = 0;
        for (int s = 0; s < q.nst; s++) {
            const int m = q.n / q.radix[s], per = T / lines;
            used += m * q.radix[s];
            slots += (m + per - 1) / per * per * q.radix[s];
        }
        const int ctas = std::min((int)(227 * 1024 / (smem + 1024)), 1024 / T);
        const double score = (double)used / slots * std::min(1.0, ctas * T / 960.0);
        if (score > best) {
            best = score;
            threads = T;
        }
    }
    return threads;
}

// n as `depth` radices of those above, each from smallest to largest.
bool split(int n, int depth, int largest, int smallest, int *out)
{
    if (depth == 1) {
        if (n > largest || n < smallest || n == 12) return false;
        out[0] = n;
        return true;
    }
    for (int r = largest; r >= smallest; r--)
        if (r != 12 && n % r == 0 && split(n / r, depth - 1, r, smallest, out + 1)) {
            out[0] = r;
            return true;
        }
    return false;
}

cudaError_t set_limits()
{
    const struct {
        const void *kernel;
        size_t smem;
    } ks[] = {{(const void *)mix_residual_kernel, col_smem(kMixMaxN)},
              {(const void *)mix_r2c_kernel, row_smem(kMixMaxN)},
              {(const void *)mix_c2r_kernel, row_smem(kMixMaxN)}};
    for (const auto &k : ks) {
        const cudaError_t e =
            cudaFuncSetAttribute(k.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

bool mix_plan(int n, MixAxis *ax, std::vector<float2> *table)
{
    if (n < kMixMinN || n > kMixMaxN) return false;
    MixAxis q{};
    q.n = n;
    // fewest stages, and of those splits the one whose smallest radix is the
    // largest (a stage of radix 2 has its exchange but little else to do)
    for (int depth = 2; depth <= kMixStages && !q.nst; depth++)
        for (int smallest = 13; smallest >= 2 && !q.nst; smallest--)
            if (split(n, depth, 13, smallest, q.radix)) q.nst = depth;
    if (!q.nst) return false;
    // ceil(2^20 / Ns) divides j < 512 by Ns < 512 exactly: its excess over
    // 2^20 / Ns is below 1, and j * 1 < 2^20 / Ns
    for (int s = 0, Ns = 1; s < q.nst; Ns *= q.radix[s++]) q.inv[s] = ((1u << 20) + Ns - 1) / Ns;
    for (int s = q.nst - 1, Ns = 1; s >= 0; Ns *= q.radix[s--]) q.rinv[s] = ((1u << 20) + Ns - 1) / Ns;
    q.row_threads = pick_threads(q, kRowLines, row_smem(n));
    q.col_threads = pick_threads(q, kColLines, col_smem(n));
    if (set_limits() != cudaSuccess) return false;  // of the current device
    const double pi = 3.14159265358979323846;
    for (int j = 0; j < n; j++) {
        const double w = -2.0 * pi * (double)j / (double)n;
        table->push_back(make_float2((float)std::cos(w), (float)std::sin(w)));
    }
    *ax = q;
    return true;
}

cudaError_t launch_mix_residual(float2 *F, const float *N, const float2 *C, float scale, const MixAxis &ax,
                                const float2 *tw, long long inner, cudaStream_t s)
{
    ColArgs a{};
    a.F = F;
    a.N = N;
    a.C = C;
    a.inner = inner;
    a.scale = scale;
    a.tw = tw;
    a.ax = ax;
    mix_residual_kernel<<<(unsigned)((inner + kColLines - 1) / kColLines), ax.col_threads, col_smem(ax.n), s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_mix_r2c(const MixAxis &ax, const float2 *tw, const DevState *st, const VolDesc *vols,
                           const float *beta, float *const *xbuf, int pitch, int ny, int nz, float2 *F, cudaStream_t s)
{
    RowArgs a{};
    a.xs[0] = xbuf[0];
    a.xs[1] = xbuf[1];
    a.ds[0] = xbuf[2];
    a.ds[1] = xbuf[3];
    a.st = st;
    a.vols = vols;
    a.beta = beta;
    a.F = F;
    a.rows = (long long)nz * ny;
    a.ny = ny;
    a.pitch = pitch;
    a.tw = tw;
    a.ax = ax;
    const unsigned grid = (unsigned)((a.rows + 2 * kRowLines - 1) / (2 * kRowLines));
    mix_r2c_kernel<<<grid, ax.row_threads, row_smem(ax.n), s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_mix_c2r(const MixAxis &ax, const float2 *tw, float2 *F, int ny, int nz, float *out, int pitch,
                           cudaStream_t s)
{
    RowArgs a{};
    a.out = out;
    a.F = F;
    a.rows = (long long)nz * ny;
    a.ny = ny;
    a.pitch = pitch;
    a.tw = tw;
    a.ax = ax;
    const unsigned grid = (unsigned)((a.rows + 2 * kRowLines - 1) / (2 * kRowLines));
    mix_c2r_kernel<<<grid, ax.row_threads, row_smem(ax.n), s>>>(a);
    return cudaGetLastError();
}

}  // namespace spg
