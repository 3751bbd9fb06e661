// Device helpers of the subfield transforms (Sect. 2: Fourier transform of
// every subimage), shared by the per-stage kernels (k_fft.cu) and the batched
// persistent launch (k_batch.cu): an in-register radix-2 FFT and the
// four-step split of an N-point transform over a group of threads.
#pragma once
#include "sm_internal.h"

namespace smf {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// In-register radix-2 FFT of length 8 or 16 (decimation in time, bit-reversed
// input order resolved at compile time).  INV conjugates.
__host__ __device__ constexpr int bitrev(int i, int bits) {
    int r = 0;
    for (int b = 0; b < bits; ++b) r |= ((i >> b) & 1) << (bits - 1 - b);
    return r;
}
__host__ __device__ constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n / 2); }

// b W_16^E (E < 8), the conjugate for INV: the factors are constants of the
// code, so the eighth roots cost two products and the quarter root none.
template <int E, bool INV>
__device__ __forceinline__ float2 rotate16(float2 b) {
    constexpr float h = 0.70710678118654752440f;     // cos(pi/4)
    constexpr float c = 0.92387953251128675613f;     // cos(pi/8)
    constexpr float s = 0.38268343236508977173f;     // sin(pi/8)
    if constexpr (E == 0) return b;
    else if constexpr (E == 4) return INV ? make_float2(-b.y, b.x) : make_float2(b.y, -b.x);
    else if constexpr (E == 2)
        return INV ? make_float2(h * (b.x - b.y), h * (b.x + b.y)) : make_float2(h * (b.x + b.y), h * (b.y - b.x));
    else if constexpr (E == 6)
        return INV ? make_float2(-h * (b.x + b.y), h * (b.x - b.y)) : make_float2(h * (b.y - b.x), -h * (b.x + b.y));
    else {
        constexpr float wx = E == 1 ? c : E == 3 ? s : E == 5 ? -s : -c;
        constexpr float wy = (E == 1 ? -s : E == 3 ? -c : E == 5 ? -c : -s) * (INV ? -1.f : 1.f);
        return cmul(b, make_float2(wx, wy));
    }
}

// One butterfly level of the FFT below: blocks of LEN, factor W_LEN^J.
template <int L, int LEN, int J, bool INV>
__device__ __forceinline__ void fft_level(float2 (&v)[L]) {
    if constexpr (J < LEN / 2) {
#pragma unroll
        for (int i = 0; i < L; i += LEN) {
            const float2 a = v[i + J];
            const float2 t = rotate16<J * (16 / LEN), INV>(v[i + J + LEN / 2]);
            v[i + J] = make_float2(a.x + t.x, a.y + t.y);
            v[i + J + LEN / 2] = make_float2(a.x - t.x, a.y - t.y);
        }
        fft_level<L, LEN, J + 1, INV>(v);
    }
}

template <int L, bool INV>
__device__ __forceinline__ void reg_fft(float2 (&v)[L]) {
    constexpr int LB = ilog2(L);
    static_assert(L == 8 || L == 16, "rotations are sixteenth roots");
#pragma unroll
    for (int i = 0; i < L; ++i) {
        const int j = bitrev(i, LB);
        if (j > i) {
            const float2 t = v[i];
            v[i] = v[j];
            v[j] = t;
        }
    }
    fft_level<L, 2, 0, INV>(v);
    fft_level<L, 4, 0, INV>(v);
    fft_level<L, 8, 0, INV>(v);
    if constexpr (L == 16) fft_level<L, 16, 0, INV>(v);
}

// Four-step split of an N-point transform: N = P * Q, thread n1 < P of a
// group holds x[n1 + P n2] (n2 < Q) on entry; on exit thread k2 < Q holds
// X[k2 + Q k1] (k1 < P) in out[].  T is the group's [Q][P+1] exchange tile.
template <int N> struct Split;
template <> struct Split<64> { static constexpr int P = 8, Q = 8; };
template <> struct Split<128> { static constexpr int P = 8, Q = 16; };
template <> struct Split<256> { static constexpr int P = 16, Q = 16; };

// Entry i = k2 P + g of the four-step table: exp(-2 pi i g k2 / N), so that a
// group's lanes read neighbouring words (in the plan's order W_N^j the reads
// of stage k2 would share gcd(k2, 16) banks and cost as much as the exchange).
template <int N>
__device__ __forceinline__ int step_root(int i) { return (i % Split<N>::P) * (i / Split<N>::P); }

// U: outputs of the second stage per thread, of G = Q / U threads: output
// k = g + G u + Q k1 is out[u P + k1].
template <int N, bool INV, int U = 1>
__device__ __forceinline__ void four_step(float2 (&v)[Split<N>::Q], float2 (&out)[U * Split<N>::P],
                                          float2* T, const float2* tw, int g) {
    constexpr int P = Split<N>::P, Q = Split<N>::Q, G = Q / U;
    if (G == P || g < P) {
        reg_fft<Q, INV>(v);
#pragma unroll
        for (int k2 = 0; k2 < Q; ++k2) {
            float2 w = tw[k2 * P + g];
            if (INV) w.y = -w.y;
            T[k2 * (P + 1) + g] = k2 == 0 ? v[k2] : cmul(v[k2], w);
        }
    }
    __syncwarp();
    if (g < G) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float2 o[P];
#pragma unroll
            for (int n1 = 0; n1 < P; ++n1) o[n1] = T[(g + G * u) * (P + 1) + n1];
            reg_fft<P, INV>(o);
#pragma unroll
            for (int k1 = 0; k1 < P; ++k1) out[u * P + k1] = o[k1];
        }
    }
    __syncwarp();
}

__device__ __forceinline__ float load_sample(const uint16_t* p) { return (float)__ldg(p); }
__device__ __forceinline__ float load_sample(const float* p) { return __ldg(p); }

template <int PREC>
__device__ __forceinline__ void store_spec(void* spec, size_t idx, float2 v) {
    if (PREC == SM_FP32) {
        reinterpret_cast<float2*>(spec)[idx] = v;
    } else if (PREC == SM_FP16) {
        reinterpret_cast<__half2*>(spec)[idx] =
            __floats2half2_rn(v.x * smi::FP16_SCALE, v.y * smi::FP16_SCALE);
    } else {
        reinterpret_cast<__nv_bfloat162*>(spec)[idx] = __floats2bfloat162_rn(v.x, v.y);
    }
}


}  // namespace smf
