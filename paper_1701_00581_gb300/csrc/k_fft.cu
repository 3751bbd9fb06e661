// Subfield spectra (Sect. 2: Fourier transform of every subimage) and the
// inverse transform of modulus and phase (Sect. 2, Sect. 3.2).
//
// One CTA per (frame, subfield): the tile is cut from the frame, apodised by
// the separable window, its windowed mean is removed, and the 2-D DFT is
// taken as real row FFTs (two rows packed per complex FFT) followed by
// column FFTs of only the K+1 non-negative columns inside the cutoff box.
// The transforms are four-step FFTs (N = P x Q) computed in registers by
// groups of 16 threads with one shared-memory exchange.
#include "sm_fft_dev.cuh"

namespace {

using smi::PlanDev;
using smf::four_step;
using smf::load_sample;
using smf::Split;
using smf::store_spec;

// Thread groups of the four-step transform: G threads per transform, each
// forming U groups of P outputs.  TB: the exchange tile's elements (it holds a
// row for the inverse; groups of 8 threads start half the banks apart).
template <int N, int THREADS, int OUT, int RESIDENT> struct Grp {
    static constexpr int P = Split<N>::P, Q = Split<N>::Q;
    static constexpr int T = THREADS, U = OUT, G = Q / OUT, CTAS = RESIDENT;
    static constexpr int NG = T / G;
    static constexpr int TB0 = Q * (P + 1) > N ? Q * (P + 1) : N;
    static constexpr int TB = G == 8 ? (TB0 + 7) / 16 * 16 + 8 : TB0;
    static_assert(G >= P && (N / 2) % NG == 0, "a thread per first-stage input, whole rounds of row pairs");
};

// Spectra.  N = 256: 32 groups of 16 threads; one CTA per SM fits in shared
// memory, so latency is hidden by the warps within it.  N = 128: groups of 8
// threads with two output sets each, so that no lane idles in the first stage.
// Smaller transforms run several CTAs to an SM, which hide each other's
// barriers and chains.
template <int N> struct SpecGrp;
template <> struct SpecGrp<64> : Grp<64, 128, 1, 6> {};
template <> struct SpecGrp<128> : Grp<128, 128, 2, 3> {};
template <> struct SpecGrp<256> : Grp<256, 512, 1, 1> {};
// N = 64 with few tiles: twice the threads per tile.  100 tiles: 5.3 us against
// 6.6 with 128 threads; 400 (a wave of three per SM): 7.4 against 8.7; 500:
// 11.4 against 9.7; 36100: 471 against 376.
struct SpecGrpFew : Grp<64, 256, 1, 3> {};

// Inverse: one CTA per subfield, as many threads as the rows keep busy.
template <int N> struct InvGrp : Grp<N, N >= 128 ? 512 : 256, 1, 1> {};

template <typename GP>
__host__ __device__ constexpr size_t fft_smem(int N, int K) {
    return (size_t)(K + 1) * (N + 1) * sizeof(float2)        // column buffer
           + (size_t)GP::NG * GP::TB * sizeof(float2)        // the groups' exchange tiles
           + (size_t)N * sizeof(float2)                      // twiddles
           + (size_t)(K + 1) * sizeof(float2)                // window transform
           + (size_t)2 * N * sizeof(float)                   // windows
           + (size_t)18 * sizeof(double);                    // reductions and scalars
}

// Spectra of one (frame, subfield): the tile times the window is transformed
// row by row (two real rows per complex transform), the windowed mean mu is
// read off the row transforms' DC terms, mu * window is removed through the
// window's own transform, and the K+1 non-negative columns are transformed.
// Bound by issue and shared-memory wavefronts, not by HBM (a quarter of the
// copy rate at most): rotations by sixteenth roots are constants of the code,
// the four-step roots are read in lane order, the row pairs are taken apart by
// shuffles and the mean goes in the columns' load.  100 frames of uint16:
// 304 subfields of 256^2 5.36 -> 4.47 ms, 225 of 128^2 2.56 -> 0.97 ms, 361 of
// 64^2 0.45 -> 0.38 ms, one of 64^2 6.2 -> 5.7 us.
template <typename GP, int N, typename TIn, int PREC>
__global__ void __launch_bounds__(GP::T, GP::CTAS)
k_spectra(PlanDev p, const TIn* __restrict__ frames, int F, int sub0, void* __restrict__ spec,
          float* __restrict__ flux, float* __restrict__ mu) {
    constexpr int P = GP::P, Q = GP::Q, G = GP::G, NG = GP::NG, TB = GP::TB, U = GP::U;
    constexpr int TS = GP::T, WS = TS / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int K1 = p.K + 1, CP = N + 1;
    float2* C = reinterpret_cast<float2*>(smem);
    float2* scratch = C + (size_t)K1 * CP;
    float2* stw = scratch + NG * TB;
    float2* swf = stw + N;
    float* swx = reinterpret_cast<float*>(swf + K1);
    float* swy = swx + N;
    double* red = reinterpret_cast<double*>(swy + N);

    // frame-major grid: consecutive CTAs cut neighbouring subfields of one
    // frame, whose tiles overlap, so most tile reads hit L2
    const int sl = blockIdx.x, f = blockIdx.y, s = sub0 + sl;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int grp = tid / G, g = tid - grp * G;
    float2* T = scratch + grp * TB;
    const int4 sb = p.subs[s];
    const int x0 = sb.x, y0 = sb.y, w = sb.z, h = sb.w;
    {
        // the whole tile towards L2 now, so the row rounds after the first
        // do not wait on DRAM: one prefetch per 128-byte line of each row
        const char* fb = reinterpret_cast<const char*>(frames + (size_t)f * p.H * p.W + (size_t)y0 * p.W);
        const size_t b0 = (size_t)x0 * sizeof(TIn), b1 = (size_t)(x0 + w) * sizeof(TIn);
        const int l0 = (int)(b0 >> 7), nl = (int)(((b1 - 1) >> 7) - (b0 >> 7)) + 1;
        for (int e = tid; e < h * nl; e += TS) {
            const int y = e / nl, l = e - y * nl;
            const size_t off = (size_t)y * p.W * sizeof(TIn) + ((size_t)(l0 + l) << 7);
            const size_t lo = (size_t)y * p.W * sizeof(TIn) + b0;   // stay inside the tile's row
            asm volatile("prefetch.global.L2 [%0];" :: "l"(fb + (off > lo ? off : lo)));
        }
    }
    const TIn* fr = frames + (size_t)f * p.H * p.W + (size_t)y0 * p.W + x0;
    // row transforms: group grp of round r handles rows 2(r NG + grp), +1; a
    // round's samples are on their way while the round before is taken apart
    float raw[2][Q];
    auto fetch = [&](int pr) {
        const int y1 = 2 * pr, y2 = y1 + 1;
#pragma unroll
        for (int n2 = 0; n2 < Q; ++n2) {
            const int x = g + P * n2;
            const bool inx = (G == P || g < P) && x < w;
            raw[0][n2] = inx && y1 < h ? load_sample(fr + (size_t)y1 * p.W + x) : 0.f;
            raw[1][n2] = inx && y2 < h ? load_sample(fr + (size_t)y2 * p.W + x) : 0.f;
        }
    };
    fetch(grp);
    for (int i = tid; i < N; i += TS) {
        stw[i] = p.tw[smf::step_root<N>(i)];
        swx[i] = p.winx[(size_t)s * N + i];
        swy[i] = p.winy[(size_t)s * N + i];
    }
    for (int i = tid; i < K1; i += TS) swf[i] = p.winft[(size_t)s * K1 + i];
    __syncthreads();

    const double wsum = tid == 0 ? p.winsum[s] : 0.0;
#pragma unroll 1
    for (int pr0 = 0; pr0 < N / 2; pr0 += NG) {
        const int pr = pr0 + grp, y1 = 2 * pr, y2 = y1 + 1;
        float2 v[Q], X[U * P];
#pragma unroll
        for (int n2 = 0; n2 < Q; ++n2) {
            const float wx = swx[(g + P * n2) & (N - 1)];
            v[n2] = make_float2(wx * swy[y1] * raw[0][n2], wx * swy[y2] * raw[1][n2]);
        }
        four_step<N, false, U>(v, X, T, stw, g);
        if (pr0 + NG < N / 2) fetch(pr + NG);
        // the two rows' transforms from X(kx) and X(N - kx), which is the
        // value [U - 1 - u][P - 1 - k1] of lane G - g (lane 0: its own, one
        // place on); kx <= K < N / 2
        const int partner = (lane & ~(G - 1)) | ((G - g) & (G - 1));
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int k1 = 0; k1 < P / 2; ++k1) {
                if (G * u + Q * k1 >= K1) break;
                const float2 za = X[u * P + k1], m = X[(U - 1 - u) * P + P - 1 - k1];
                float2 zb = make_float2(__shfl_sync(0xffffffffu, m.x, partner), __shfl_sync(0xffffffffu, m.y, partner));
                if (g == 0) zb = u > 0 ? X[(U - u) % U * P + P - 1 - k1] : X[(P - k1) % P];
                const int kx = g + G * u + Q * k1;
                if (kx < K1) {
                    C[kx * CP + y1] = make_float2(0.5f * (za.x + zb.x), 0.5f * (za.y - zb.y));
                    C[kx * CP + y2] = make_float2(0.5f * (za.y + zb.y), -0.5f * (za.x - zb.x));
                }
            }
    }
    __syncthreads();

    // windowed mean from the DC terms of the row transforms: the warps
    // holding DC terms reduce them, thread 0 forms the scalars once
    if (tid < N) {
        double dacc = 0.0;
        for (int y = tid; y < N; y += TS) dacc += (double)C[y].x;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dacc += __shfl_xor_sync(0xffffffffu, dacc, o);
        if (lane == 0) red[warp] = dacc;
    }
    __syncthreads();
    if (tid == 0) {
        double tot = 0.0;
#pragma unroll
        for (int i = 0; i < (N < TS ? N : TS) / 32; ++i) tot += red[i];
        const float m = (float)(tot / wsum);
        reinterpret_cast<float*>(red + WS + 1)[1] = m;
    }
    __syncthreads();
    const float mean = reinterpret_cast<const float*>(red + WS + 1)[1];
    if (tid == 0) {
        const double fl = (double)mean * wsum;
        red[WS] = fl;                                  // flux, then its reciprocal
        reinterpret_cast<float*>(red + WS + 1)[0] = (float)(1.0 / fl);
    }

    // column transforms of kx = 0..K (groups past K transform column K and
    // drop it), with mean * window removed on the way in: the row transform of
    // w_x(x) w_y(y) mu is mu w_y(y) Wx(kx)
    for (int c0 = 0; c0 < K1; c0 += NG) {
        const int kx = c0 + grp;
        const int kc = kx < K1 ? kx : K1 - 1;
        const float2 wf = swf[kc];
        float2 v[Q], X[U * P];
#pragma unroll
        for (int n2 = 0; n2 < Q; ++n2) {
            const int y = g + P * n2;
            float2 c = make_float2(0.f, 0.f);
            if (G == P || g < P) {
                c = C[kc * CP + y];
                if (y < h) {
                    const float a = mean * swy[y];
                    c.x -= a * wf.x;
                    c.y -= a * wf.y;
                }
            }
            v[n2] = c;
        }
        four_step<N, false, U>(v, X, T, stw, g);
        if (kx < K1) {
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int k1 = 0; k1 < P; ++k1) C[kx * CP + g + G * u + Q * k1] = X[u * P + k1];
        }
        __syncwarp();
    }
    __syncthreads();

    // normalise by the windowed flux and store the box ky = -R..K (a warp
    // per box row, coalesced along it)
    const double fl = red[WS];
    const float inv = reinterpret_cast<const float*>(red + WS + 1)[0];
    const size_t base = ((size_t)sl * F + f) * p.box_rows * p.box_pitch;
    for (int row = warp; row < p.box_rows; row += WS)
    for (int col = lane; col < p.box_cols; col += 32) {
        const int ky = row - p.R, kx = col - p.K;
        float2 v;
        if (kx >= 0) {
            v = C[kx * CP + (ky & (N - 1))];
        } else {
            v = C[(-kx) * CP + ((-ky) & (N - 1))];
            v.y = -v.y;
        }
        v.x *= inv;
        v.y *= inv;
        if (kx == 0 && ky == 0) v = make_float2(1.f, 0.f);
        store_spec<PREC>(spec, base + (size_t)row * p.box_pitch + col, v);
    }
    if (tid == 0) {
        flux[(size_t)sl * F + f] = (float)fl;
        mu[(size_t)sl * F + f] = mean;
    }
}

// a * v rounded to FP32.  The FP32 recursion's phasors are FP64 copies of
// floats: their bits are repacked on the integer pipe and multiplied in FP32,
// which rounds the same exact product; anything else takes the FP64 product
// (GB300's FP64 unit converts and multiplies two values per clock and SM).
__device__ __forceinline__ float scaled(float a, double v) {
    const int hi = __double2hiint(v), lo = __double2loint(v);
    const int e = (hi >> 20) & 0x7ff;
    if (e < 897 || e > 1150 || (lo & 0x1fffffff)) return (float)(a * v);
    return a * __int_as_float((hi & 0x80000000) | ((e - 896) << 23) | ((hi & 0xfffff) << 3) | ((unsigned)lo >> 29));
}

// Inverse: O = A z on the disk (Hermitian), DC removed; columns first, then
// pairs of Hermitian rows packed into one complex inverse FFT, by the forward
// transform's four-step groups.  304 subfields of
// 256^2: 237 -> 85 us; 225 of 128^2: 66 -> 38 us; one of 64^2: 25 -> 12 us
// (warp-wide radix-2 passes in shared memory, FP64 products and a serial sum
// over the frames before).
template <int N>
__global__ void __launch_bounds__(InvGrp<N>::T, InvGrp<N>::CTAS)
k_inverse(PlanDev p, int F, int sub0, const float* __restrict__ A, const double2* __restrict__ z,
          const float* __restrict__ flux, const float* __restrict__ mu, float* __restrict__ rec) {
    using GP = InvGrp<N>;
    constexpr int P = GP::P, Q = GP::Q, G = GP::G, NG = GP::NG, TB = GP::TB;
    constexpr int TS = GP::T, WS = TS / 32;
    static_assert(GP::U == 1, "one output set per thread");
    extern __shared__ __align__(16) unsigned char smem[];
    const int K = p.K, K1 = K + 1, CP = N + 1;
    float2* C = reinterpret_cast<float2*>(smem);
    float2* scratch = C + (size_t)K1 * CP;
    float2* stw = scratch + NG * TB;
    float* swx = reinterpret_cast<float*>(stw + N + K1);
    float* swy = swx + N;
    double* red = reinterpret_cast<double*>(swy + N);

    const int sl = blockIdx.x, s = sub0 + sl;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int grp = tid / G, g = tid - grp * G;
    float2* T = scratch + grp * TB;
    for (int i = tid; i < N; i += TS) {
        stw[i] = p.tw[smf::step_root<N>(i)];
        swx[i] = p.winx[(size_t)s * N + i];
        swy[i] = p.winy[(size_t)s * N + i];
    }
    if (warp == 0) {
        double fs = 0.0, ms = 0.0;
        for (int f = lane; f < F; f += 32) {
            fs += flux[(size_t)sl * F + f];
            ms += mu[(size_t)sl * F + f];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            fs += __shfl_xor_sync(0xffffffffu, fs, o);
            ms += __shfl_xor_sync(0xffffffffu, ms, o);
        }
        if (lane == 0) {
            red[0] = fs / F;
            red[1] = ms / F;
        }
    }
    for (int e = tid; e < K1 * CP; e += TS) C[e] = make_float2(0.f, 0.f);
    __syncthreads();
    // the half box row by row: (kx, ky) into column kx, its mirror (-kx, -ky)
    // conjugated into column -kx
    const size_t hb = (size_t)p.hb_rows * p.box_pitch;
    const float* As = A + (size_t)sl * hb;
    const double2* zs = z + (size_t)sl * hb;
    for (int ky = warp; ky <= K; ky += WS)
        for (int col = lane; col < p.box_cols; col += 32) {
            const int kx = col - K;
            if (kx * kx + ky * ky > p.r2i || (ky == 0 && kx <= 0)) continue;
            const size_t o = (size_t)ky * p.box_pitch + col;
            const double2 zz = zs[o];
            const float a = As[o];
            const float2 v = make_float2(scaled(a, zz.x), scaled(a, zz.y));
            if (kx >= 0) C[kx * CP + ky] = v;
            if (kx <= 0) C[-kx * CP + N - ky] = make_float2(v.x, -v.y);
        }
    __syncthreads();
    const float mmean = (float)red[1];
    const float scale = (float)(red[0] / ((double)N * N));

    for (int c0 = 0; c0 < K1; c0 += NG) {
        const int kx = c0 + grp;
        const int kc = kx < K1 ? kx : K1 - 1;
        float2 v[Q], X[P];
#pragma unroll
        for (int n2 = 0; n2 < Q; ++n2) v[n2] = g < P ? C[kc * CP + g + P * n2] : make_float2(0.f, 0.f);
        four_step<N, true>(v, X, T, stw, g);
        if (kx < K1 && g < Q) {
#pragma unroll
            for (int k1 = 0; k1 < P; ++k1) C[kx * CP + g + Q * k1] = X[k1];
        }
        __syncwarp();
    }
    __syncthreads();

    float* out = rec + (size_t)s * N * N;
    for (int pr0 = 0; pr0 < N / 2; pr0 += NG) {
        const int y1 = 2 * (pr0 + grp), y2 = y1 + 1;
        for (int kx = g; kx < N; kx += G) T[kx] = make_float2(0.f, 0.f);
        __syncwarp();
        for (int kx = g; kx < K1; kx += G) {
            const float2 a = C[kx * CP + y1], b = C[kx * CP + y2];
            T[kx] = make_float2(a.x - b.y, a.y + b.x);
            if (kx > 0) T[N - kx] = make_float2(a.x + b.y, -a.y + b.x);
        }
        __syncwarp();
        float2 v[Q], X[P];
#pragma unroll
        for (int n2 = 0; n2 < Q; ++n2) v[n2] = g < P ? T[g + P * n2] : make_float2(0.f, 0.f);
        __syncwarp();
        four_step<N, true>(v, X, T, stw, g);
        if (g < Q) {
#pragma unroll
            for (int k1 = 0; k1 < P; ++k1) {
                const int x = g + Q * k1;
                out[(size_t)y1 * N + x] = X[k1].x * scale + mmean * swx[x] * swy[y1];
                out[(size_t)y2 * N + x] = X[k1].y * scale + mmean * swx[x] * swy[y2];
            }
        }
        __syncwarp();
    }
}

template <typename GP, int N>
cudaError_t spectra_n(const PlanDev& p, const void* frames, int frame_type, int F, int sub0,
                      int nsub, void* spec, float* flux, float* mu, cudaStream_t st) {
    const size_t sm = fft_smem<GP>(N, p.K);
    dim3 grid(nsub, F);
    cudaError_t e = cudaSuccess;
#define SM_LAUNCH(TIN, PREC)                                                                    \
    do {                                                                                        \
        e = cudaFuncSetAttribute(k_spectra<GP, N, TIN, PREC>,                                       \
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);         \
        if (e != cudaSuccess) return e;                                                         \
        k_spectra<GP, N, TIN, PREC><<<grid, GP::T, sm, st>>>(                                         \
            p, reinterpret_cast<const TIN*>(frames), F, sub0, spec, flux, mu);                  \
    } while (0)
    if (frame_type == SM_U16) {
        if (p.prec == SM_FP32) SM_LAUNCH(uint16_t, SM_FP32);
        else if (p.prec == SM_FP16) SM_LAUNCH(uint16_t, SM_FP16);
        else SM_LAUNCH(uint16_t, SM_BF16);
    } else {
        if (p.prec == SM_FP32) SM_LAUNCH(float, SM_FP32);
        else if (p.prec == SM_FP16) SM_LAUNCH(float, SM_FP16);
        else SM_LAUNCH(float, SM_BF16);
    }
#undef SM_LAUNCH
    return cudaGetLastError();
}

template <int N>
cudaError_t inverse_n(const PlanDev& p, int F, int sub0, int nsub, const float* A, const double2* z,
                      const float* flux, const float* mu, float* rec, cudaStream_t st) {
    const size_t sm = fft_smem<InvGrp<N>>(N, p.K);
    cudaError_t e = cudaFuncSetAttribute(k_inverse<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sm);
    if (e != cudaSuccess) return e;
    k_inverse<N><<<nsub, InvGrp<N>::T, sm, st>>>(p, F, sub0, A, z, flux, mu, rec);
    return cudaGetLastError();
}

// Tiles up to which a 64 x 64 tile gets 256 threads instead of 128: one wave
// of them.
long long few_tiles() {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (long long)SpecGrpFew::CTAS * sms;
}

}  // namespace

namespace smk {

size_t spectra_smem_bytes(int N, int K) {
    return N == 64    ? fft_smem<InvGrp<64>>(N, K)
           : N == 128 ? fft_smem<InvGrp<128>>(N, K)
                      : fft_smem<InvGrp<256>>(N, K);
}

cudaError_t launch_spectra(const smi::PlanDev& p, const void* frames, int frame_type, int F,
                           int sub0, int nsub, void* spec, float* flux, float* mu,
                           cudaStream_t st) {
    switch (p.N) {
        case 64:
            if ((long long)nsub * F <= few_tiles())
                return spectra_n<SpecGrpFew, 64>(p, frames, frame_type, F, sub0, nsub, spec, flux, mu, st);
            return spectra_n<SpecGrp<64>, 64>(p, frames, frame_type, F, sub0, nsub, spec, flux, mu, st);
        case 128: return spectra_n<SpecGrp<128>, 128>(p, frames, frame_type, F, sub0, nsub, spec, flux, mu, st);
        case 256: return spectra_n<SpecGrp<256>, 256>(p, frames, frame_type, F, sub0, nsub, spec, flux, mu, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_inverse(const smi::PlanDev& p, int F, int sub0, int nsub, const float* A,
                           const double2* z, const float* flux, const float* mu, float* rec,
                           cudaStream_t st) {
    switch (p.N) {
        case 64: return inverse_n<64>(p, F, sub0, nsub, A, z, flux, mu, rec, st);
        case 128: return inverse_n<128>(p, F, sub0, nsub, A, z, flux, mu, rec, st);
        case 256: return inverse_n<256>(p, F, sub0, nsub, A, z, flux, mu, rec, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace smk
