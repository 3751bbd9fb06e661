// Front end (Table 2's first row: flat-field and dark-field preprocessing).
//
// k_gain: the detector's normalised gain g = (flat - dark) / mean(flat - dark),
// the mean over the pixels where flat > dark (g = 0 elsewhere).  Computed
// once per flat field, by one CTA: each thread sums its pixels in order in
// FP64, a fixed tree combines the threads, then the same CTA writes the map.
// k_calibrate: every frame sample (raw - dark) / g, 0 where g = 0; an
// elementwise pass bound by HBM (2 or 4 bytes read, 4 written per sample).
// A thread keeps the dark and gain of four neighbouring pixels and walks the
// frames (the pixel index is never divided out of the sample index); frames
// whose pixel count or pointers do not keep every frame's row of four aligned
// go one pixel a thread.  100 uint16 frames of 2560 x 2160 (3.3 GB): 2.02 ->
// 0.58 ms, 5.7 TB/s.
#include <algorithm>
#include <type_traits>

#include "sm_internal.h"

namespace {

using smi::PlanDev;

constexpr int GAIN_THREADS = 1024;
constexpr int CAL_THREADS = 256;

__global__ void __launch_bounds__(GAIN_THREADS)
k_gain(int npx, const float* __restrict__ flat, const float* __restrict__ dark, float* __restrict__ gain) {
    __shared__ double ssum[GAIN_THREADS];
    __shared__ long long scnt[GAIN_THREADS];
    double s = 0.0;
    long long c = 0;
    for (int i = threadIdx.x; i < npx; i += GAIN_THREADS) {
        const double d = (double)flat[i] - (double)dark[i];
        if (d > 0.0) { s += d; ++c; }
    }
    ssum[threadIdx.x] = s;
    scnt[threadIdx.x] = c;
    __syncthreads();
    for (int h = GAIN_THREADS / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            ssum[threadIdx.x] += ssum[threadIdx.x + h];
            scnt[threadIdx.x] += scnt[threadIdx.x + h];
        }
        __syncthreads();
    }
    const double mean = scnt[0] > 0 ? ssum[0] / (double)scnt[0] : 0.0;
    for (int i = threadIdx.x; i < npx; i += GAIN_THREADS) {
        const double d = (double)flat[i] - (double)dark[i];
        gain[i] = (d > 0.0 && mean > 0.0) ? (float)(d / mean) : 0.f;
    }
}

__device__ __forceinline__ float calibrated(float raw, float dark, float g) { return g > 0.f ? (raw - dark) / g : 0.f; }

// V pixels a thread (4: vector loads and stores, 1: any size and alignment).
template <typename In, int V>
__global__ void __launch_bounds__(CAL_THREADS)
k_calibrate(int npx, int F, const In* __restrict__ raw, const float* __restrict__ dark, const float* __restrict__ gain,
            float* __restrict__ out) {
    const int px = (blockIdx.x * CAL_THREADS + threadIdx.x) * V;
    if (px >= npx) return;
    float d[V], g[V];
#pragma unroll
    for (int i = 0; i < V; ++i) {
        d[i] = __ldg(dark + px + i);
        g[i] = __ldg(gain + px + i);
    }
#pragma unroll 4
    for (int f = blockIdx.y; f < F; f += gridDim.y) {
        const size_t at = (size_t)f * npx + px;
        if constexpr (V == 4) {
            float r[4];
            if constexpr (std::is_same<In, float>::value) {
                const float4 t = __ldcs(reinterpret_cast<const float4*>(raw + at));
                r[0] = t.x; r[1] = t.y; r[2] = t.z; r[3] = t.w;
            } else {
                const ushort4 t = __ldcs(reinterpret_cast<const ushort4*>(raw + at));
                r[0] = t.x; r[1] = t.y; r[2] = t.z; r[3] = t.w;
            }
            *reinterpret_cast<float4*>(out + at) = make_float4(calibrated(r[0], d[0], g[0]), calibrated(r[1], d[1], g[1]),
                                                               calibrated(r[2], d[2], g[2]), calibrated(r[3], d[3], g[3]));
        } else {
            out[at] = calibrated((float)raw[at], d[0], g[0]);
        }
    }
}

// Blocks along the frames, so that small images fill the GPU too.
template <typename In>
cudaError_t calibrate(int npx, int F, const In* raw, const float* dark, const float* gain, float* out, cudaStream_t st) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool vec = npx % 4 == 0 && reinterpret_cast<uintptr_t>(raw) % (4 * sizeof(In)) == 0 &&
                     reinterpret_cast<uintptr_t>(out) % 16 == 0;
    const int bx = ((vec ? npx / 4 : npx) + CAL_THREADS - 1) / CAL_THREADS;
    const int by = std::max(1, std::min(std::min(F, 65535), 16 * sms / bx));
    if (vec) k_calibrate<In, 4><<<dim3(bx, by), CAL_THREADS, 0, st>>>(npx, F, raw, dark, gain, out);
    else k_calibrate<In, 1><<<dim3(bx, by), CAL_THREADS, 0, st>>>(npx, F, raw, dark, gain, out);
    return cudaGetLastError();
}

}  // namespace

namespace smk {

cudaError_t launch_gain(const smi::PlanDev& p, const float* flat, const float* dark, float* gain, cudaStream_t st) {
    k_gain<<<1, GAIN_THREADS, 0, st>>>(p.W * p.H, flat, dark, gain);
    return cudaGetLastError();
}

cudaError_t launch_calibrate(const smi::PlanDev& p, const void* raw, int frame_type, int F, const float* dark,
                             const float* gain, float* out, cudaStream_t st) {
    if (frame_type == SM_U16) return calibrate(p.W * p.H, F, static_cast<const uint16_t*>(raw), dark, gain, out, st);
    return calibrate(p.W * p.H, F, static_cast<const float*>(raw), dark, gain, out, st);
}

}  // namespace smk

// Correlation tracking (Table 2's correlation-tracking row): per frame the
// integer shift s = (sx, sy), |sx|, |sy| <= S, maximising
// C(s) = sum over the central G x G window of a(x + s) (r(x) - mean r),
// r the reference frame, the first maximum in row-major (sy, sx) order;
// then the frames shifted by s with edge pixels replicated.
//
// k_track_ref: the reference window minus its mean (FP64 sum over a cluster of
// CTAs).  k_track_cc: a cluster per frame, its CTAs sharing the window's rows;
// a thread owns 12 neighbouring shifts sx of one sy and slides a register
// window along the row, so 4 samples cost two 16-byte shared loads and 48
// FMAs (bound by FP32 FMA issue: 100 frames, G = 256, S = 16 in 0.52 ms, with
// the pick; one thread per shift and row by row staging took 3.3 + 0.53 ms).
// Products are summed in FP32 over 32-sample chunks; the chunks are summed as
// float-float pairs (48 bits, on the FP32 pipe: adding each chunk in
// FP64 would alone take 0.4 ms for 100 frames of a 256^2 window and S = 16 on
// GB300's FP64 units), or in FP64 where a pair's sum is not finite, and threads
// and CTAs in FP64.  The cluster's first CTA
// writes the surface and picks the first maximum.  k_shift: a warp per row
// (100 float frames of 2560 x 2160, 4.4 GB: 1.78 -> 0.67 ms, 6.7 TB/s).
namespace {

constexpr int TRACK_MAX_S = 31;        // 2S + 1 <= 63 shifts per axis
constexpr int TRACK_CLUSTER = 8;       // CTAs per frame (and for the reference window)
constexpr int TRACK_THREADS = 448;     // two CTAs per SM at 72 registers a thread
constexpr int SG = 12;                 // shifts along x per thread
constexpr int XT = 256;                // window columns per staged tile
constexpr int RB = 16;                 // window rows per staged tile

template <typename In>
__device__ __forceinline__ float sample(const In* f, size_t i) { return (float)f[i]; }

__device__ __forceinline__ unsigned cta_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// *at (own shared memory) of CTA `rank` of the cluster
__device__ __forceinline__ double load_cluster(const double* at, unsigned rank) {
    unsigned a = (unsigned)__cvta_generic_to_shared(at), r;
    double v;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(r) : "memory");
    return v;
}

template <typename In>
__global__ void __launch_bounds__(TRACK_THREADS)
k_track_ref(const In* __restrict__ frames, int W, int H, int ref, int x0, int y0, int G, float* __restrict__ rw) {
    __shared__ double red[TRACK_THREADS / 32], mine;
    const In* r = frames + (size_t)ref * W * H + (size_t)y0 * W + x0;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w0 = (int)cta_rank() * (TRACK_THREADS / 32) + warp, nw = TRACK_CLUSTER * (TRACK_THREADS / 32);
    double s = 0.0;
    for (int y = w0; y < G; y += nw)
        for (int x = lane; x < G; x += 32) s += (double)sample(r, (size_t)y * W + x);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < TRACK_THREADS / 32; ++i) t += red[i];
        mine = t;
    }
    cluster_sync();
    double tot = 0.0;
    for (unsigned c = 0; c < TRACK_CLUSTER; ++c) tot += load_cluster(&mine, c);
    const float mean = (float)(tot / ((double)G * G));
    for (int y = w0; y < G; y += nw)
        for (int x = lane; x < G; x += 32) rw[y * G + x] = sample(r, (size_t)y * W + x) - mean;
    cluster_sync();                                       // every CTA has read every sum
}

// Launch shape of k_track_cc for n = 2S + 1 shifts per axis.
struct TrackShape {
    int ng, slots, rs, pitch;          // thread groups along sx, threads per row share, row shares, tile row pitch
    int threads;
    size_t smem;
};
__host__ inline TrackShape track_shape(int S) {
    TrackShape t;
    const int n = 2 * S + 1;
    t.ng = (n + SG - 1) / SG;
    t.slots = n * t.ng;
    t.rs = 8;
    while (t.rs * t.slots > TRACK_THREADS) t.rs /= 2;
    t.threads = (t.rs * t.slots + 31) / 32 * 32;
    // 16-byte rows whose slot count is odd: neighbouring sy read different banks
    const int q = (XT + SG * t.ng + 4 + 3) / 4;
    t.pitch = 4 * (q | 1);
    const size_t tile = ((size_t)(RB + 2 * S) * t.pitch + (size_t)RB * XT) * sizeof(float);
    const size_t red = ((size_t)t.rs * t.slots * SG + (size_t)n * n) * sizeof(double);
    t.smem = std::max(tile, red);
    return t;
}

// (hi, lo) += p, exactly up to the rounding of lo (Knuth's two-sum).
__device__ __forceinline__ void pair_add(float& hi, float& lo, float p) {
    const float s = __fadd_rn(hi, p), v = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, v)), __fsub_rn(p, v)));
    hi = s;
}

// A thread's SG shifts over its share of the window rows [ya, yb) -- of every RB
// rows those share, share + rs, ... -- from column x0 on of the rows at a, the
// products as the kernel below forms them, the chunks summed in FP64; some
// shifts at a time, so that the registers of the kernel's own loop suffice, and
// no further once all of them are NaN.  Columns past the frame, which only
// shifts past the last one (count) have, are held at its edge.
template <typename In>
__device__ __forceinline__ void row_share_fp64(const In* a, int W, int x0, int G, int ya, int yb, int share, int rs,
                                               const float* rw, int count, double* out) {
    constexpr int N = 6;
    static_assert(SG % N == 0, "whole groups of shifts");
#pragma unroll 1
    for (int k0 = 0; k0 < count; k0 += N) {
        bool live = true;
        double t[N];
#pragma unroll
        for (int k = 0; k < N; ++k) t[k] = 0.0;
#pragma unroll 1
        for (int yt = ya; yt < yb && live; yt += RB)
#pragma unroll 1
            for (int y = yt + share; y < min(yt + RB, yb) && live; y += rs) {
                const In* const row = a + (size_t)y * W;
                float w[N], part[N];
#pragma unroll
                for (int k = 1; k < N; ++k) w[k] = sample(row, min(x0 + k0 + k - 1, W - 1));
#pragma unroll 1
                for (int c = 0; c < G && live; c += 32) {
#pragma unroll
                    for (int k = 0; k < N; ++k) part[k] = 0.f;
#pragma unroll 4
                    for (int x = c; x < min(c + 32, G); ++x) {
#pragma unroll
                        for (int k = 0; k < N - 1; ++k) w[k] = w[k + 1];
                        w[N - 1] = sample(row, min(x0 + k0 + x + N - 1, W - 1));
                        const float r = rw[y * G + x];
#pragma unroll
                        for (int k = 0; k < N; ++k) part[k] = fmaf(w[k], r, part[k]);
                    }
#pragma unroll
                    for (int k = 0; k < N; ++k) t[k] += (double)part[k];
                    live = false;
#pragma unroll
                    for (int k = 0; k < N; ++k) live = live || (k0 + k < count && !isnan(t[k]));
                }
            }
#pragma unroll
        for (int k = 0; k < N; ++k) out[k0 + k] = t[k];
    }
}

template <typename In>
__global__ void __launch_bounds__(TRACK_THREADS, 2)
k_track_cc(const In* __restrict__ frames, int W, int H, int x0, int y0, int G, int S, TrackShape sh,
           const float* __restrict__ rw, double* __restrict__ cc, int* __restrict__ shifts) {
    extern __shared__ __align__(16) unsigned char smem[];
    float* const tile = reinterpret_cast<float*>(smem);                  // [RB + 2S][pitch]
    const int n = 2 * S + 1, P = sh.pitch;
    float* const rtile = tile + (RB + 2 * S) * P;                        // [RB][XT]
    const int f = blockIdx.x / TRACK_CLUSTER, rank = (int)cta_rank();
    const In* a = frames + (size_t)f * W * H;
    const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31, nw = nt >> 5;
    const int share = tid / sh.slots, slot = tid - share * sh.slots;
    const int syi = slot % n, s0 = slot / n * SG;                        // sy fastest: a phase's lanes read 8 rows
    const bool work = share < sh.rs;
    float hi[SG], lo[SG];
#pragma unroll
    for (int k = 0; k < SG; ++k) hi[k] = lo[k] = 0.f;
    const int per = (G + TRACK_CLUSTER - 1) / TRACK_CLUSTER;
    const int ya = min(rank * per, G), yb = min(ya + per, G);
    for (int yt = ya; yt < yb; yt += RB) {
        const int rows = min(RB, yb - yt);
        for (int xt = 0; xt < G; xt += XT) {
            const int cols = min(XT, G - xt);
            __syncthreads();
            for (int y = warp; y < rows + 2 * S; y += nw) {
                const size_t row = (size_t)(y0 + yt + y - S) * W + (x0 - S + xt);
                for (int x = lane; x < cols + 2 * S; x += 32) tile[y * P + x] = sample(a, row + x);
            }
            for (int y = warp; y < rows; y += nw)
                for (int x = lane; x < cols; x += 32) rtile[y * XT + x] = rw[(yt + y) * G + xt + x];
            __syncthreads();
            if (!work) continue;
            for (int y = share; y < rows; y += sh.rs) {
                const float* const tr = tile + (y + syi) * P + s0;
                const float* const rr = rtile + y * XT;
                for (int c = 0; c < cols; c += 32) {
                    float part[SG], w[SG + 4];
#pragma unroll
                    for (int k = 0; k < SG; ++k) part[k] = 0.f;
                    const int e = min(c + 32, cols);
                    int x = c;
                    if (e - c == 32) {
#pragma unroll
                        for (int k = 0; k < SG; k += 4)
                            *reinterpret_cast<float4*>(w + k) = *reinterpret_cast<const float4*>(tr + c + k);
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            *reinterpret_cast<float4*>(w + SG) = *reinterpret_cast<const float4*>(tr + c + 4 * q + SG);
                            const float4 r = *reinterpret_cast<const float4*>(rr + c + 4 * q);
#pragma unroll
                            for (int k = 0; k < SG; ++k) part[k] = fmaf(w[k], r.x, part[k]);
#pragma unroll
                            for (int k = 0; k < SG; ++k) part[k] = fmaf(w[k + 1], r.y, part[k]);
#pragma unroll
                            for (int k = 0; k < SG; ++k) part[k] = fmaf(w[k + 2], r.z, part[k]);
#pragma unroll
                            for (int k = 0; k < SG; ++k) part[k] = fmaf(w[k + 3], r.w, part[k]);
#pragma unroll
                            for (int k = 0; k < SG; ++k) w[k] = w[k + 4];
                        }
                        x = e;
                    }
                    for (; x < e; ++x)
#pragma unroll
                        for (int k = 0; k < SG; ++k) part[k] = fmaf(tr[x + k], rr[x], part[k]);
#pragma unroll
                    for (int k = 0; k < SG; ++k) pair_add(hi[k], lo[k], part[k]);
                }
            }
        }
    }
    __syncthreads();
    // row shares in order, then the cluster's CTAs in order
    double* const red = reinterpret_cast<double*>(smem);                 // [rs][n][ng * SG]
    double* const mine = red + (size_t)sh.rs * sh.slots * SG;            // [n][n]
    const int cw = sh.ng * SG;
    bool finite = true;
    if (work) {
        double* const own = red + ((size_t)share * n + syi) * cw + s0;
#pragma unroll
        for (int k = 0; k < SG; ++k) {
            own[k] = (double)hi[k] + (double)lo[k];
            finite = finite && (s0 + k >= n || isfinite(hi[k]));
        }
    }
    // chunks that are not finite, or sums past the range of a float: such a
    // thread's chunks once more, summed in FP64
    if (__syncthreads_or(std::is_same<In, float>::value && !finite)) {
        if (!finite)
            row_share_fp64(a + (size_t)(y0 + syi - S) * W, W, x0 + s0 - S, G, ya, yb, share, sh.rs, rw,
                           min(SG, n - s0), red + ((size_t)share * n + syi) * cw + s0);
        __syncthreads();
    }
    for (int k = tid; k < n * n; k += nt) {
        const int j = k / n, i = k - j * n;
        double t = 0.0;
        for (int r = 0; r < sh.rs; ++r) t += red[((size_t)r * n + j) * cw + i];
        mine[k] = t;
    }
    cluster_sync();
    if (rank == 0) {
        // the surface, and its first maximum in row-major order: a value not
        // above any other (a NaN) is only picked when it comes first
        __shared__ double bv[TRACK_THREADS / 32];
        __shared__ int bk[TRACK_THREADS / 32];
        double best = -INFINITY;
        int at = n * n;
        for (int k = tid; k < n * n; k += nt) {
            double t = 0.0;
            for (unsigned c = 0; c < TRACK_CLUSTER; ++c) t += load_cluster(mine + k, c);
            cc[(size_t)f * n * n + k] = t;
            if (k == 0 && isnan(t)) t = INFINITY, at = -1, best = t;
            else if (t > best) best = t, at = k;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double v = __shfl_xor_sync(0xffffffffu, best, o);
            const int k = __shfl_xor_sync(0xffffffffu, at, o);
            if (v > best || (v == best && k < at)) best = v, at = k;
        }
        if (lane == 0) bv[warp] = best, bk[warp] = at;
        __syncthreads();
        if (tid == 0) {
            for (int i = 1; i < nw; ++i)
                if (bv[i] > best || (bv[i] == best && bk[i] < at)) best = bv[i], at = bk[i];
            if (at < 0 || at >= n * n) at = 0;
            shifts[2 * f] = at % n - S;
            shifts[2 * f + 1] = at / n - S;
        }
    }
    cluster_sync();                                       // the other CTAs' sums have been read
}

// Frames moved by their shifts, edges replicated: a warp per row, four
// coalesced samples a lane in flight (bound by HBM: 2 or 4 bytes read and 4
// written per sample).
constexpr int SHIFT_THREADS = 256;
template <typename In>
__global__ void __launch_bounds__(SHIFT_THREADS)
k_shift(int F, int W, int H, const In* __restrict__ frames, const int* __restrict__ shifts, float* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const long long nrow = (long long)F * H, step = (long long)gridDim.x * (SHIFT_THREADS / 32);
    for (long long r = (long long)blockIdx.x * (SHIFT_THREADS / 32) + (threadIdx.x >> 5); r < nrow; r += step) {
        const int f = (int)(r / H), y = (int)(r - (long long)f * H);
        const int sx = __ldg(shifts + 2 * f), sy = __ldg(shifts + 2 * f + 1);
        const In* const src = frames + ((size_t)f * H + min(max(y + sy, 0), H - 1)) * W;
        float* const dst = out + (size_t)r * W;
        int x = lane;
        for (; x + 96 < W; x += 128) {
            float v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = (float)__ldcs(src + min(max(x + 32 * i + sx, 0), W - 1));
#pragma unroll
            for (int i = 0; i < 4; ++i) __stcs(dst + x + 32 * i, v[i]);
        }
        for (; x < W; x += 32) dst[x] = sample(src, min(max(x + sx, 0), W - 1));
    }
}

template <typename Kernel, typename... Args>
cudaError_t launch_cluster(Kernel kern, int blocks, int threads, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = TRACK_CLUSTER;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <typename In>
cudaError_t track(const smi::PlanDev& p, const In* frames, int F, int ref, int G, int S, float* rw, double* cc,
                  int* shifts, cudaStream_t st) {
    const int x0 = (p.W - G) / 2, y0 = (p.H - G) / 2;
    cudaError_t e = launch_cluster(k_track_ref<In>, TRACK_CLUSTER, TRACK_THREADS, 0, st, frames, p.W, p.H, ref, x0, y0,
                                   G, rw);
    if (e != cudaSuccess) return e;
    const TrackShape sh = track_shape(S);
    e = cudaFuncSetAttribute(k_track_cc<In>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    return launch_cluster(k_track_cc<In>, F * TRACK_CLUSTER, sh.threads, sh.smem, st, frames, p.W, p.H, x0, y0, G, S, sh,
                          static_cast<const float*>(rw), cc, shifts);
}

}  // namespace

namespace smk {

int track_max_search() { return TRACK_MAX_S; }

cudaError_t launch_track(const smi::PlanDev& p, const void* frames, int frame_type, int F, int ref, int G, int S,
                         float* rw, double* cc, int* shifts, cudaStream_t st) {
    if (frame_type == SM_U16)
        return track(p, static_cast<const uint16_t*>(frames), F, ref, G, S, rw, cc, shifts, st);
    return track(p, static_cast<const float*>(frames), F, ref, G, S, rw, cc, shifts, st);
}

cudaError_t launch_shift(const smi::PlanDev& p, const void* frames, int frame_type, int F, const int* shifts,
                         float* out, cudaStream_t st) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long rows = (long long)F * p.H;
    const int blocks = (int)std::min<long long>((long long)sms * 8, (rows + SHIFT_THREADS / 32 - 1) / (SHIFT_THREADS / 32));
    if (frame_type == SM_U16)
        k_shift<uint16_t><<<blocks, SHIFT_THREADS, 0, st>>>(F, p.W, p.H, static_cast<const uint16_t*>(frames), shifts, out);
    else
        k_shift<float><<<blocks, SHIFT_THREADS, 0, st>>>(F, p.W, p.H, static_cast<const float*>(frames), shifts, out);
    return cudaGetLastError();
}

}  // namespace smk
