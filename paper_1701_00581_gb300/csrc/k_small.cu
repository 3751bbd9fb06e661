// Per-subfield statistics (Eq. 1 numerator and the noise floor), the
// Labeyrie modulus (Eq. 1) and the mosaic merge (Sect. 3.2).
#include <algorithm>

#include "sm_internal.h"

namespace {

using smi::PlanDev;

constexpr int STAT_THREADS = 256;
constexpr int STAT_CTAS = 8;           // CTAs (one cluster) per subfield at most
constexpr int STAT_LOADS = 10;         // frames whose loads are in flight together

// Two neighbouring spectrum values as stored, and as floats.
template <int PREC> struct Pair { using T = float4; };
template <> struct Pair<SM_FP16> { using T = uint2; };
template <> struct Pair<SM_BF16> { using T = uint2; };
template <int PREC> __device__ __forceinline__ float4 pair_values(float4 v) { return v; }
template <int PREC> __device__ __forceinline__ float4 pair_values(uint2 v) {
    float2 a, b;
    if (PREC == SM_FP16) {
        a = __half22float2(*reinterpret_cast<const __half2*>(&v.x));
        b = __half22float2(*reinterpret_cast<const __half2*>(&v.y));
        a.x *= smi::FP16_INV_SCALE; a.y *= smi::FP16_INV_SCALE;
        b.x *= smi::FP16_INV_SCALE; b.y *= smi::FP16_INV_SCALE;
    } else {
        a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.x));
        b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&v.y));
    }
    return make_float4(a.x, a.y, b.x, b.y);
}

// P = <|I_i|^2>, M = <I_i> over the F frames on the half box ky = 0..K;
// noise = mean of P over {ky >= 1, |k|^2 > r^2} (the half-box corners).
// HBM bound: a cluster of up to 8 CTAs per subfield streams its F spectra once,
// each thread summing two neighbouring values over the frames in order
// (16-byte loads of FP32 spectra, ten frames in flight: a single subfield is
// bound by the latency of its chain of loads).  The corners' sum runs over a
// fixed tree of threads and CTAs.  304 subfields of 256^2, 100 frames: 0.47 ->
// 0.40 ms; 225 of 64^2 68 -> 33 us; one of 64^2 16.7 -> 12.5 us, against one CTA of
// 1024 threads with four frames in flight.
template <int PREC>
__global__ void __launch_bounds__(STAT_THREADS)
k_stats(PlanDev p, int ctas, const void* __restrict__ spec, int F, float* __restrict__ P,
        float2* __restrict__ M, float* __restrict__ noise) {
    using PT = typename Pair<PREC>::T;
    __shared__ double red_s[STAT_THREADS / 32], part_s;
    __shared__ int red_n[STAT_THREADS / 32], part_n;
    const int sl = blockIdx.x / ctas, part = blockIdx.x - sl * ctas, tid = threadIdx.x;
    const size_t box2 = (size_t)p.box_rows * p.box_pitch / 2;
    const size_t hb = (size_t)p.hb_rows * p.box_pitch;
    // the pitch is a multiple of 4; the last value of a row pairs with the
    // row's padding, which is read but not stored
    const int hp = p.box_pitch / 2, ne2 = p.hb_rows * hp;
    const PT* s2 = reinterpret_cast<const PT*>(spec) + (size_t)sl * F * box2 + (size_t)p.R * hp;
    const float invF = 1.0f / (float)F;
    double cs = 0.0;
    int cn = 0;
    for (int e = part * STAT_THREADS + tid; e < ne2; e += ctas * STAT_THREADS) {
        const int ky = e / hp, col = 2 * (e - ky * hp);
        float ps0 = 0.f, ps1 = 0.f;
        float2 m0 = make_float2(0.f, 0.f), m1 = make_float2(0.f, 0.f);
        auto add = [&](PT t) {
            const float4 v = pair_values<PREC>(t);
            ps0 = fmaf(v.x, v.x, fmaf(v.y, v.y, ps0));
            ps1 = fmaf(v.z, v.z, fmaf(v.w, v.w, ps1));
            m0.x += v.x; m0.y += v.y;
            m1.x += v.z; m1.y += v.w;
        };
        int f = 0;
        for (; f + STAT_LOADS <= F; f += STAT_LOADS) {
            PT t[STAT_LOADS];
#pragma unroll
            for (int i = 0; i < STAT_LOADS; ++i) t[i] = __ldg(s2 + (size_t)(f + i) * box2 + e);
#pragma unroll
            for (int i = 0; i < STAT_LOADS; ++i) add(t[i]);
        }
        for (; f < F; ++f) add(__ldg(s2 + (size_t)f * box2 + e));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int cc = col + h, kx = cc - p.K;
            if (cc >= p.box_cols) break;
            const float pm = (h ? ps1 : ps0) * invF;
            const float2 ms = h ? m1 : m0;
            const size_t o = (size_t)sl * hb + (size_t)ky * p.box_pitch + cc;
            P[o] = pm;
            M[o] = make_float2(ms.x * invF, ms.y * invF);
            if (ky >= 1 && kx * kx + ky * ky > p.r2i) {
                cs += pm;
                ++cn;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cs += __shfl_xor_sync(0xffffffffu, cs, o);
        cn += __shfl_xor_sync(0xffffffffu, cn, o);
    }
    if ((tid & 31) == 0) {
        red_s[tid >> 5] = cs;
        red_n[tid >> 5] = cn;
    }
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        int n = 0;
        for (int i = 0; i < STAT_THREADS / 32; ++i) {
            s += red_s[i];
            n += red_n[i];
        }
        part_s = s;
        part_n = n;
    }
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (part == 0 && tid == 0) {
        double s = 0.0;
        int n = 0;
        for (int c = 0; c < ctas; ++c) {
            unsigned as = (unsigned)__cvta_generic_to_shared(&part_s), an = (unsigned)__cvta_generic_to_shared(&part_n);
            double ps;
            int pn;
            asm("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(as) : "r"(c));
            asm("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(an) : "r"(c));
            asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(ps) : "r"(as) : "memory");
            asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(pn) : "r"(an) : "memory");
            s += ps;
            n += pn;
        }
        noise[sl] = n > 0 ? (float)(s / n) : 0.f;
    }
    // the parts have been read
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// A = sqrt(max(P - noise, 0) / max(STF, 1e-4)) * T0 on U, A(0) = 1, 0 outside,
// rounded once from about 46 bits.  A thread owns one frequency and walks the
// subfields: the factor T0 / sqrt(max(STF, 1e-4)) is formed once in FP64 and
// split in two floats, and per subfield the difference, the root and the
// product run on pairs of floats (GB300's FP64 unit would take 0.2 ms for the
// 3.3 M values of a TiO burst; this takes 35 us).  Values whose pairs would run
// out of a float's range take the formula in FP64.
__global__ void __launch_bounds__(256)
k_amplitude(PlanDev p, int nsub, const double* __restrict__ stf, const float* __restrict__ P,
            const float* __restrict__ noise, float* __restrict__ A) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const int ne = p.hb_rows * p.box_cols;
    if (e >= ne) return;
    const int ky = e / p.box_cols, col = e - ky * p.box_cols, kx = col - p.K;
    const size_t hb = (size_t)p.hb_rows * p.box_pitch;
    const size_t o = (size_t)ky * p.box_pitch + col;
    const double t0 = p.t0[o];
    const bool dc = kx == 0 && ky == 0, in = t0 > 0.0;
    float gh = 0.f, gl = 0.f;
    double s = 1.0;
    if (in) {
        s = fmax(stf[(size_t)(ky + p.N / 2) * p.N + kx + p.N / 2], 1e-4);
        const double g = t0 / sqrt(s);
        gh = (float)g;
        gl = (float)(g - (double)gh);
    }
    for (int sl = blockIdx.y; sl < nsub; sl += gridDim.y) {
        float a = 0.f;
        if (dc) {
            a = 1.f;
        } else if (in) {
            // P - noise exactly, as hi + lo
            const float x = P[(size_t)sl * hb + o], y = -noise[sl];
            const float hi = __fadd_rn(x, y), bb = __fsub_rn(hi, x);
            const float lo = __fadd_rn(__fsub_rn(x, __fsub_rn(hi, bb)), __fsub_rn(y, bb));
            if (hi > 0.f) {                          // a NaN counts as no power, as the maximum has it
                const float r = sqrtf(hi), q = __fmul_rn(r, gh);
                if (hi >= 1e-30f && hi < INFINITY && fminf(q, gh) >= 1e-30f) {
                    // the rest c of the root, then (r + c)(gh + gl): every term
                    // dropped or rounded is below 2^-44 q, and a float holds it
                    const float c = __fdiv_rn(__fadd_rn(__fmaf_rn(-r, r, hi), lo), 2.f * r);
                    a = __fadd_rn(q, __fmaf_rn(c, gh, __fmaf_rn(r, gl, __fmaf_rn(r, gh, -q))));
                } else {
                    a = (float)(sqrt(fmax((double)x + (double)y, 0.0) / s) * t0);
                }
            }
        }
        A[(size_t)sl * hb + o] = a;
    }
}

// out(x) = sum_s rec_s(x - o_s) / sum_s window_s(x - o_s); a gather over the
// (at most ceil(N/stride)^2) subfields covering the pixel, no atomics.
__global__ void k_mosaic(PlanDev p, const float* __restrict__ rec, float* __restrict__ out,
                         uint8_t* __restrict__ valid) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= p.W || y >= p.H) return;
    if (p.mosaic_mode == SM_MOSAIC_CENTRAL) {
        // the one subfield whose central stride x stride block holds (x, y)
        const int h0 = (p.N - p.stride) / 2;
        const int i = x >= h0 ? (x - h0) / p.stride : -1, j = y >= h0 ? (y - h0) / p.stride : -1;
        const bool ok = i >= 0 && i < p.nsx && j >= 0 && j < p.nsy;
        float v = 0.f;
        if (ok) {
            const int s = j * p.nsx + i;
            const int4 sb = p.subs[s];
            const int lx = x - sb.x, ly = y - sb.y;       // in [h0, h0 + stride)
            v = rec[((size_t)s * p.N + ly) * p.N + lx] /
                (p.winx[(size_t)s * p.N + lx] * p.winy[(size_t)s * p.N + ly]);
        }
        out[(size_t)y * p.W + x] = v;
        if (valid) valid[(size_t)y * p.W + x] = ok ? 1 : 0;
        return;
    }
    const int ilo = x - p.N + 1 > 0 ? (x - p.N + p.stride) / p.stride : 0;
    const int ihi = min(p.nsx - 1, x / p.stride);
    const int jlo = y - p.N + 1 > 0 ? (y - p.N + p.stride) / p.stride : 0;
    const int jhi = min(p.nsy - 1, y / p.stride);
    float num = 0.f, den = 0.f;
    for (int j = jlo; j <= jhi; ++j) {
        for (int i = ilo; i <= ihi; ++i) {
            const int s = j * p.nsx + i;
            const int4 sb = p.subs[s];
            const int lx = x - sb.x, ly = y - sb.y;
            if (lx < 0 || ly < 0 || lx >= sb.z || ly >= sb.w) continue;
            num += rec[((size_t)s * p.N + ly) * p.N + lx];
            den += p.winx[(size_t)s * p.N + lx] * p.winy[(size_t)s * p.N + ly];
        }
    }
    const bool ok = den >= 0.25f;
    out[(size_t)y * p.W + x] = ok ? num / den : 0.f;
    if (valid) valid[(size_t)y * p.W + x] = ok ? 1 : 0;
}

// Photon-noise bias of the mean bispectrum (Wirnitzer 1985), removed in
// place at every used pair of every tile: B -= (P(u) + P(v) + P(w)) <1/N>
// - 2 <1/N^2> (real), u = w - v, P(-k) = P(k) from the half box, N_f the
// photon count of frame f's windowed tile.  A CTA walks tiles of one subfield,
// laid out as the bispectrum kernel's, so the means over the frames are formed
// once per CTA and not per tile (63 subfields of 128^2, R = 16, 80 frames:
// 2.9 -> 0.44 ms; 0.95 GB of tiles).
__global__ void __launch_bounds__(smi::BISPEC_THREADS)
k_unbias(PlanDev p, int F, const float* __restrict__ flux, const float* __restrict__ P, float2* __restrict__ B) {
    __shared__ float a12[2];
    const int sl = blockIdx.y;
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31, wyl = lane >> 2, gx = lane & 3;
    const float* Ps = P + (size_t)sl * p.hb_rows * p.box_pitch;
    if (threadIdx.x < 32) {             // <1/N_f>, <1/N_f^2>, N_f = photon_gain * flux_f
        double a1 = 0.0, a2 = 0.0;
        for (int f = lane; f < F; f += 32) {
            const double nf = p.photon_gain * (double)flux[(size_t)sl * F + f];
            if (nf > 0.0) {
                const double r = 1.0 / nf;
                a1 += r;
                a2 += r * r;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a1 += __shfl_xor_sync(0xffffffffu, a1, o);
            a2 += __shfl_xor_sync(0xffffffffu, a2, o);
        }
        if (lane == 0) {
            a12[0] = (float)(a1 / F);
            a12[1] = (float)(a2 / F);
        }
    }
    __syncthreads();
    const float a1 = a12[0], a2 = a12[1];
    // P of any frequency at signed index ky * pitch + kx (P(-k) = P(k); the
    // pitch exceeds 2 K + 1, and row 0 holds both signs with equal values)
    const int pitch = p.box_pitch;
    auto pget = [&](int kx, int ky) -> float { return __ldg(Ps + abs(ky * pitch + kx) + p.K); };
    for (int tile = blockIdx.x; tile < p.n_tiles; tile += gridDim.x) {
        const int4 T = p.tiles[tile];
        if (((__ldg(p.tile_masks + tile) >> (8 * q)) & 0xffu) == 0) continue;      // no used pair in this row
        float2* Bt = B + (size_t)(sl * p.n_tiles + tile) * smi::TILE_PAIRS;
        const int wy = T.y + wyl, vy = T.w + q;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int wx = T.x + 4 * gx + j, w2 = wx * wx + wy * wy;
            const bool okw = (wy > 0 || (wy == 0 && wx > 0)) && w2 >= 2 && w2 <= p.r2i;
            if (!okw) continue;
            const float pw = pget(wx, wy);
            float2* const row = Bt + (wyl * smi::WBX + 4 * gx + j) * smi::TILE_V + q * smi::VBX;
            float2 b[smi::VBX];
            bool ok[smi::VBX];
#pragma unroll
            for (int kk = 0; kk < smi::VBX; ++kk) {
                const int vx = T.z + kk, v2 = vx * vx + vy * vy, ux = wx - vx, uy = wy - vy;
                ok[kk] = v2 > 0 && v2 <= p.R * p.R && v2 < w2 && ux * ux + uy * uy < w2;
                if (ok[kk]) b[kk] = row[kk];
            }
#pragma unroll
            for (int kk = 0; kk < smi::VBX; ++kk)
                if (ok[kk]) {
                    const int vx = T.z + kk;
                    b[kk].x -= (pget(wx - vx, wy - vy) + pget(vx, vy) + pw) * a1 - 2.f * a2;
                    row[kk] = b[kk];
                }
        }
    }
}

}  // namespace

namespace smk {

namespace {

template <int PREC>
cudaError_t stats_go(const smi::PlanDev& p, const void* spec, int F, int nsub, float* P, float2* M, float* noise,
                     cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    // as many CTAs as hold a value each per thread; more would only wait for the
    // others at the cluster's barriers (225 subfields of 64^2: 70 us with 8)
    const int ctas = std::min(STAT_CTAS, (p.hb_rows * p.box_pitch / 2 + STAT_THREADS - 1) / STAT_THREADS);
    cfg.gridDim = dim3(nsub * ctas);
    cfg.blockDim = dim3(STAT_THREADS);
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_stats<PREC>, p, ctas, spec, F, P, M, noise);
}

int sm_count() {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

}  // namespace

cudaError_t launch_stats(const smi::PlanDev& p, const void* spec, int F, int nsub, float* P,
                         float2* M, float* noise, cudaStream_t st) {
    if (p.prec == SM_FP32) return stats_go<SM_FP32>(p, spec, F, nsub, P, M, noise, st);
    if (p.prec == SM_FP16) return stats_go<SM_FP16>(p, spec, F, nsub, P, M, noise, st);
    return stats_go<SM_BF16>(p, spec, F, nsub, P, M, noise, st);
}

// Blocks along the subfields: about two per SM in all, so that the FP64
// factors are formed a few times, not once per subfield.
cudaError_t launch_amplitude(const smi::PlanDev& p, int nsub, const double* stf, const float* P,
                             const float* noise, float* A, cudaStream_t st) {
    const int bx = (p.hb_rows * p.box_cols + 255) / 256;
    const int by = std::max(1, std::min(nsub, 2 * sm_count() / bx));
    k_amplitude<<<dim3(bx, by), 256, 0, st>>>(p, nsub, stf, P, noise, A);
    return cudaGetLastError();
}

cudaError_t launch_unbias(const smi::PlanDev& p, int F, int nsub, const float* flux, const float* P, float2* B,
                          cudaStream_t st) {
    const int bx = std::max(1, std::min(p.n_tiles, 32 * sm_count() / nsub));
    k_unbias<<<dim3(bx, nsub), smi::BISPEC_THREADS, 0, st>>>(p, F, flux, P, B);
    return cudaGetLastError();
}

cudaError_t launch_mosaic(const smi::PlanDev& p, const float* rec, float* out, uint8_t* valid,
                          cudaStream_t st) {
    dim3 grid((p.W + 255) / 256, p.H);
    k_mosaic<<<grid, 256, 0, st>>>(p, rec, out, valid);
    return cudaGetLastError();
}

}  // namespace smk
