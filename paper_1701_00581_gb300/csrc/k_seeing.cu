// Seeing estimate (Sect. 3.1: spectral ratio technique, von der Luehe 1984).
//
// The burst is cut into non-overlapping N x N cubes; each cube's spectral
// ratio |<I>|^2 / <|I|^2>, averaged over annuli of unit width, is fitted by
// the model ratio |T_LE|^2 / STF of a seeing D/r0 (Fried's long-exposure OTF
// T0 exp(-3.44 (rho D/r0)^(5/3)) squared over the model STF
// T0^2 exp(-6.88 (rho D/r0)^(5/3)) + ck (r0/D)^2 T0, both 1 at k = 0), and the
// cubes' r0 are averaged.  The cubes are subfields of the reconstruction
// grid, so their P, M and noise floor come from the stats stage.
//
// GB300's FP64 units do two FMAs per clock and SM, so the FP64 work is kept
// small.  k_seeing: one CTA per subfield of the chunk (non-cubes return at
// once).  Warps sum the annuli from the plan's index lists in FP64 (a fixed
// shuffle tree, so the result does not depend on scheduling).  The
// least-squares cost of the 256 log-spaced D/r0 candidates is first evaluated
// in FP32 with a bound on its error; the candidates that the bound leaves in
// question (a handful) and their neighbours are evaluated in FP64, the first
// minimum is taken and refined by a parabola in log D/r0.  The model's factors
// (T0 and rho^(5/3) of an annulus, x^(5/3) and ck / x^2 of a candidate) come
// from the plan, so an FP64 evaluation is one exponential and one division.
// k_seeing_stf: the mean r0 and the model STF table at it, on the centred
// N x N grid, from the plan's T0 and rho^(5/3).
// 80 cubes of 256^2: 439 -> 91 us; 64 of 128^2: 289 -> 49 us (all candidates
// in FP64 with pow, acos and sqrt each time); the STF table 39 -> 12 us.
#include <algorithm>

#include "sm_internal.h"

namespace {

using smi::PlanDev;

constexpr int SE_THREADS = 256;
constexpr int SE_GRID = smi::SEEING_GRID;     // D/r0 candidates, log-spaced
constexpr double SE_LO = smi::SEEING_LO, SE_HI = smi::SEEING_HI;
constexpr double SE_STOP = 0.05;              // fit annuli until the observed ratio drops below this
constexpr int SE_MAXB = 136;                  // annuli held in shared memory (K + 2 for fc N < 134)
static_assert(SE_GRID == SE_THREADS, "one candidate per thread");
static_assert(SE_MAXB <= SE_THREADS, "one annulus per thread");

// |T_LE|^2 / STF of an annulus (T0, rho^(5/3)) at a candidate x
// (x^(5/3), a = ck / x^2), both normalised at k = 0:
// T0^2 e (1 + a) / (T0^2 e + a T0), e = exp(-6.88 (rho x)^(5/3)).
__device__ __forceinline__ double ratio_model(double2 m, double2 c) {
    const double e = m.x * exp(-6.88 * m.y * c.x);
    return e * (1.0 + c.y) / (e + c.y);
}

__device__ __forceinline__ double log_candidate(double llo, double lhi, int i) {
    return llo + (lhi - llo) * ((double)i / (double)(SE_GRID - 1));
}

__global__ void __launch_bounds__(SE_THREADS)
k_seeing(PlanDev p, int F, int sub0, const float* __restrict__ P, const float2* __restrict__ M,
         const float* __restrict__ noise, double* __restrict__ seeing) {
    const int sl = blockIdx.x;
    const int cube = p.cube_of_sub[sub0 + sl];
    if (cube < 0) return;
    __shared__ double num[SE_MAXB], den[SE_MAXB], eps[SE_MAXB], J[SE_GRID];
    __shared__ double2 model[SE_MAXB];
    __shared__ float feps[SE_MAXB];
    __shared__ float2 fmodel[SE_MAXB];
    __shared__ float fred[SE_THREADS / 32];
    __shared__ unsigned keep[SE_GRID / 32];
    __shared__ int fail[SE_THREADS / 32], bi[SE_THREADS / 32];
    const size_t hb = (size_t)p.hb_rows * p.box_pitch;
    const float* Ps = P + sl * hb;
    const float2* Ms = M + sl * hb;
    const double nz = noise[sl], fF = (double)F;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // annulus sums: num_b = sum (F |M|^2 - P) / (F - 1), den_b = sum (P - noise)
    for (int b = warp; b < p.n_bins; b += SE_THREADS / 32) {
        double m2 = 0.0, pv = 0.0;
        const int i0 = p.ann_start[b], i1 = p.ann_start[b + 1];
        for (int i = i0 + lane; i < i1; i += 32) {
            const int e = p.ann_idx[i];
            const float2 m = Ms[e];
            pv += (double)Ps[e];
            m2 = fma((double)m.x, (double)m.x, fma((double)m.y, (double)m.y, m2));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            m2 += __shfl_xor_sync(0xffffffffu, m2, o);
            pv += __shfl_xor_sync(0xffffffffu, pv, o);
        }
        if (lane == 0) {
            num[b] = (fF * m2 - pv) / (fF - 1.0);
            den[b] = pv - (double)(i1 - i0) * nz;
        }
    }
    __syncthreads();
    // fitted annuli: b = 1, 2, ... inside the cutoff while den_b > 0 and the
    // observed ratio stays at or above SE_STOP
    {
        const int b = tid + 1;
        bool bad = true;
        if (b < p.n_bins) {
            const double r = num[b] / den[b];
            bad = !((double)b < p.rcut) || !(den[b] > 0.0) || r < SE_STOP;
            const double2 m = p.ann_model[b];
            eps[tid] = r;
            model[tid] = m;
            feps[tid] = (float)r;
            fmodel[tid] = make_float2((float)m.x, (float)m.y);
        }
        const unsigned v = __ballot_sync(0xffffffffu, bad);
        if (lane == 0) fail[warp] = v ? warp * 32 + __ffs(v) - 1 : SE_THREADS;
    }
    __syncthreads();
    int n = fail[0];
#pragma unroll
    for (int w = 1; w < SE_THREADS / 32; ++w) n = min(n, fail[w]);
    if (n == 0) {                                  // no usable annulus: nothing to fit (n is the same in every thread)
        if (tid == 0) seeing[cube] = SE_HI;
        return;
    }
    // FP32 cost of candidate tid and a bound on its error: the exponent's
    // rounding (|6.88 (rho x)^(5/3)| < 104 where e > 0, three roundings) moves
    // the model by less than 2.2e-5 of its value <= 1, taken as 4e-5.  Where e
    // is denormal the model is below 2e-8 itself, unless a is as small: such a
    // candidate (a constant ck that hardly differs from 0) goes to FP64 unscreened
    const double2 c = p.cand[tid];
    float j32 = 0.f, ad = 0.f;
    {
        const float x53 = (float)c.x, a = (float)c.y;
        for (int k = 0; k < n; ++k) {
            const float2 m = fmodel[k];
            const float e = m.x * expf(-6.88f * (m.y * x53));
            const float d = feps[k] - e * (1.f + a) / (e + a);
            j32 = fmaf(d, d, j32);
            ad += fabsf(d);
        }
    }
    if (c.y > 0.0 && c.y < 1e-30) j32 = NAN;
    const float err = 8e-5f * ad + 2e-9f * n + 1e-5f * j32;
    float up = j32 + err;                          // a NaN drops out of the minimum
    if (!(up == up)) up = INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) up = fminf(up, __shfl_xor_sync(0xffffffffu, up, o));
    if (lane == 0) fred[warp] = up;
    J[tid] = INFINITY;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < SE_THREADS / 32; ++w) up = fminf(up, fred[w]);
    const unsigned in = __ballot_sync(0xffffffffu, !(j32 - err > up));     // and keeps its candidate
    if (lane == 0) keep[warp] = in;
    __syncthreads();
    // FP64 cost of the kept candidates and of their neighbours: a warp per
    // candidate, the lanes over the annuli
    for (int i = warp; i < SE_GRID; i += SE_THREADS / 32) {
        bool want = false;
#pragma unroll
        for (int o = -1; o <= 1; ++o) {
            const int q = i + o;
            if (q >= 0 && q < SE_GRID) want |= (keep[q >> 5] >> (q & 31)) & 1u;
        }
        if (!want) continue;
        const double2 ci = p.cand[i];
        double s = 0.0;
        for (int k = lane; k < n; k += 32) {
            const double d = eps[k] - ratio_model(model[k], ci);
            s += d * d;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) J[i] = s;
    }
    __syncthreads();
    // first minimum (a NaN is only taken at candidate 0)
    double best = J[tid];
    int im = tid;
    if (!(best == best)) best = tid == 0 ? -INFINITY : INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double v = __shfl_xor_sync(0xffffffffu, best, o);
        const int k = __shfl_xor_sync(0xffffffffu, im, o);
        if (v < best || (v == best && k < im)) best = v, im = k;
    }
    if (lane == 0) {
        num[warp] = best;                          // the sums are done with
        bi[warp] = im;
    }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < SE_THREADS / 32; ++w)
            if (num[w] < best || (num[w] == best && bi[w] < im)) best = num[w], im = bi[w];
        const double llo = log(SE_LO), lhi = log(SE_HI);
        double t = log_candidate(llo, lhi, im);
        if (im > 0 && im < SE_GRID - 1) {
            const double curv = J[im - 1] - 2.0 * J[im] + J[im + 1];
            if (curv > 0.0) {
                const double h = log_candidate(llo, lhi, 1) - log_candidate(llo, lhi, 0);
                t += 0.5 * h * (J[im - 1] - J[im + 1]) / curv;
            }
        }
        seeing[cube] = exp(t);
    }
}

__global__ void __launch_bounds__(SE_THREADS)
k_seeing_stf(PlanDev p, double* __restrict__ seeing, double* __restrict__ stf) {
    __shared__ double xs, xe;
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        double s = 0.0;
        for (int c = lane; c < p.n_cubes; c += 32) s += 1.0 / seeing[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) {
            xs = 1.0 / (s / (double)p.n_cubes);     // D over the mean r0
            xe = -6.88 * pow(xs, 5.0 / 3.0);
            if (blockIdx.x == 0) seeing[p.n_cubes] = xs;
        }
    }
    __syncthreads();
    const double x = xs, a = p.ck / (x * x);
    const int N = p.N, K = p.K;
    const double norm = 1.0 / (1.0 + a);             // over the model at k = 0
    const double x53 = xe;
    // a pair of conjugate frequencies per thread: k and -k have one value
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < N * N; e += gridDim.x * blockDim.x) {
        const int ky = e / N - N / 2, kx = e % N - N / 2;
        const bool in = kx * kx + ky * ky <= p.r2i;
        const bool upper = ky > 0 || (ky == 0 && kx >= 0);
        if (in && !upper) continue;                  // written with its mirror
        double v = 0.0;
        if (in) {
            const size_t o = (size_t)ky * p.box_pitch + kx + K;
            const double T0 = p.t0[o];
            v = (T0 * T0 * exp(x53 * p.r53[o]) + a * T0) * norm;
            stf[(size_t)(N / 2 - ky) * N + N / 2 - kx] = v;
        }
        stf[e] = v;
    }
}

}  // namespace

namespace smk {

cudaError_t launch_seeing(const smi::PlanDev& p, int F, int sub0, int nsub, const float* P, const float2* M,
                          const float* noise, double* seeing, cudaStream_t st) {
    k_seeing<<<nsub, SE_THREADS, 0, st>>>(p, F, sub0, P, M, noise, seeing);
    return cudaGetLastError();
}

cudaError_t launch_seeing_stf(const smi::PlanDev& p, double* seeing, double* stf, cudaStream_t st) {
    const int blocks = std::min(256, (p.N * p.N + SE_THREADS - 1) / SE_THREADS);
    k_seeing_stf<<<blocks, SE_THREADS, 0, st>>>(p, seeing, stf);
    return cudaGetLastError();
}

int seeing_max_bins() { return SE_MAXB; }

}  // namespace smk
