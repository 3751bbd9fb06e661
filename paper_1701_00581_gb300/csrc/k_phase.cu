// Recursive Fourier phase from the mean bispectrum (Sect. 3.2: speckle
// masking phase, Lohmann, Weigelt & Wirnitzer 1983).
//
// Since arg B(w - v, v) = phi(w - v) + phi(v) - phi(w), each split of a
// target w into two already known frequencies gives a phasor estimate of
// exp(i phi(w)).  One CTA per subfield walks the rings of equal |w|^2 in
// ascending order (points of one ring never depend on each other).
//
// A ring by itself is a few points of ~750 terms each, and what bounds a
// ring-by-ring walk is the latency of its chain (load, products, reduction,
// barrier), not its work.  So the plan groups the rings into batches of
// about PHASE_BATCH points and splits each point's terms in two:
//
//   early  both u = w - v and v lie on rings before the batch (about 97 % of
//          the terms): summed for all points of the batch at once, in units
//          of 32 tile rows of a point, one warp per unit, no barrier in
//          between -- this part streams B;
//   late   u or v is on an earlier ring of the batch itself: their B values
//          are gathered into shared memory beside the early sums, and the
//          rings are walked with nothing but shared-memory reads in the
//          chain, one warp per point: z(w) = S / |S|.
//
// When there are too few subfields to fill the GPU, a cluster of CTAs shares
// one: each takes its part of the early units and writes the sums into every
// CTA's shared memory; all of them walk the rings, each on its own copy of
// the phasors.
//
// What bounds it: with the GPU full (304 subfields of 256^2, R = 24, two CTAs
// per SM) the early part, by instruction issue and load latency -- 5.3 ms, of
// which 2.3 ms is the time of the 15.7 GB of B at HBM rate (a ring-by-ring
// walk took 10.6 ms); with few subfields the rings, about 0.3 us each.
// 15 subfields: 8.2 -> 1.4 ms (3.4 ms without clusters); float-float
// 14.2 -> 2.5 ms; 225 subfields of 128^2, R = 16: 1.5 -> 0.69 ms; one subfield
// of 64^2, R = 8: 218 -> 75 us; SNR weights, 225 subfields of 128^2 2.5 -> 1.4 ms.
//
// Every sum runs in a fixed order (per lane over a unit's rows, a butterfly
// over the lanes; a point's units and late terms over the lanes, a
// butterfly), so the result does not depend on scheduling or on the cluster.
// Arithmetic is FP32 by default (GB300's FP64 unit is shared by the SM's warps
// and a small fraction of its FP32 rate), or FP64 or float-float when the
// channel asks for it; the known phasors live in shared memory in that type
// and the result is stored as FP64.
#include <type_traits>

#include "sm_internal.h"

namespace {

using smi::PlanDev;
using smi::TILE_PAIRS;

constexpr int PH_WARPS = 16, TH = 32 * PH_WARPS;   // warps and threads of a CTA
constexpr int PH_STEPS = 8;            // steps of 4 tile rows whose B loads are in flight together
constexpr int PH_SNR_STEPS = 4;        // the same with SNR weights, whose P loads are in flight as well
constexpr int PH_LATE_WARPS = 8;       // warps that walk the rings (a ring has 4 to 6 points on average)

// Complex values of the recursion's arithmetic type T.
template <typename T> struct Cx;
template <> struct Cx<float> {
    using T2 = float2;
    __device__ static float2 make(float x, float y) { return make_float2(x, y); }
    __device__ static float rnorm(float n2) { return rsqrtf(n2); }
};
template <> struct Cx<double> {
    using T2 = double2;
    __device__ static double2 make(double x, double y) { return make_double2(x, y); }
    __device__ static double rnorm(double n2) { return 1.0 / sqrt(n2); }
};

// Float-float ("double-single") numbers: an unevaluated sum hi + lo of two
// floats, |lo| <= ulp(hi) / 2, with about 48 significant bits, computed on
// the FP32 pipe -- GB300's FP64 unit runs at a small fraction of its FP32
// rate.  The error-free transformations are Knuth's two-sum, Dekker's
// fast-two-sum and the FMA-based two-product (the product's exact low part
// is fma(a, b, -a b)); addition and multiplication are the classical
// double-single ones, division and the reciprocal square root one Newton
// correction of the float estimate.  The type and its functions live in a
// namespace of their own: argument-dependent lookup adds them to the
// overloads of sqrt and __shfl_xor_sync without hiding the built-in ones.
namespace ffa {
struct ff {
    float hi, lo;
    __device__ ff() : hi(0.f), lo(0.f) {}
    __device__ ff(int v) : hi((float)v), lo(0.f) {}
    __device__ ff(float v) : hi(v), lo(0.f) {}
    __device__ ff(float h, float l) : hi(h), lo(l) {}
    __device__ explicit ff(double v) : hi((float)v), lo((float)(v - (double)(float)v)) {}
    __device__ explicit operator double() const { return (double)hi + (double)lo; }
};
__device__ __forceinline__ ff fast_two_sum(float a, float b) {       // |a| >= |b|
    const float s = __fadd_rn(a, b);
    return ff(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ ff two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float v = __fsub_rn(s, a);
    return ff(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v)));
}
__device__ __forceinline__ ff operator+(ff a, ff b) {
    ff s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ ff operator-(ff a) { return ff(-a.hi, -a.lo); }
__device__ __forceinline__ ff operator-(ff a, ff b) { return a + (-b); }
__device__ __forceinline__ ff operator*(ff a, ff b) {
    const float p = __fmul_rn(a.hi, b.hi);
    const float e = __fmaf_rn(a.hi, b.hi, -p);
    return fast_two_sum(p, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e)));
}
__device__ __forceinline__ ff operator/(ff a, ff b) {
    const float q1 = __fdiv_rn(a.hi, b.hi);
    const ff r = a - b * ff(q1);
    return fast_two_sum(q1, __fdiv_rn(r.hi, b.hi));
}
__device__ __forceinline__ ff& operator+=(ff& a, ff b) { return a = a + b; }
__device__ __forceinline__ bool operator>(ff a, ff b) { return a.hi > b.hi || (a.hi == b.hi && a.lo > b.lo); }
__device__ __forceinline__ ff sqrt(ff a) {
    if (!(a.hi > 0.f)) return ff(0.f);
    const float s = sqrtf(a.hi);
    const ff r = a - ff(s) * ff(s);                  // exact residual of s^2
    return fast_two_sum(s, __fdiv_rn(r.hi, 2.f * s));
}
__device__ __forceinline__ ff __shfl_xor_sync(unsigned mask, ff v, int o) {
    return ff(::__shfl_xor_sync(mask, v.hi, o), ::__shfl_xor_sync(mask, v.lo, o));
}
}  // namespace ffa
using ffa::ff;
struct ff2 { ff x, y; };
template <> struct Cx<ff> {
    using T2 = ff2;
    __device__ static ff2 make(ff x, ff y) { return ff2{x, y}; }
    // 1 / sqrt(n2): the float estimate r, then r (3 - n2 r^2) / 2 in float-float
    __device__ static ff rnorm(ff n2) {
        const ff r(rsqrtf(n2.hi));
        return r * (ff(3.f) - n2 * r * r) * ff(0.5f);
    }
};

// Shared memory: the phasor table (complex values of e2 bytes); the sums of a
// batch's early units, twice (another CTA of the cluster may write the next
// batch's before this one has read its own); of a batch the point records,
// the late terms (B values, offset indices) and the first point of every
// ring; 32 tile rows per warp.
struct PhaseLayout {
    size_t ep, rec, lb, liv, rs, ent, bytes;
};
__host__ __device__ inline PhaseLayout phase_layout(int hb_rows, int zpitch, int max_points, int max_units, int max_late,
                                                    size_t e2) {
    PhaseLayout l;
    l.ep = ((size_t)hb_rows * zpitch * e2 + 15) & ~(size_t)15;
    l.rec = l.ep + ((2 * (size_t)max_units * e2 + 15) & ~(size_t)15);
    l.lb = l.rec + (size_t)(max_points + 1) * sizeof(int4);
    l.liv = l.lb + (size_t)max_late * sizeof(float2);
    l.rs = l.liv + (size_t)max_late * sizeof(int);
    l.ent = (l.rs + (size_t)(max_points + 1) * sizeof(int) + 15) & ~(size_t)15;
    l.bytes = l.ent + (size_t)TH * sizeof(int2);
    return l;
}

// The phasor table holds z on the upper half plane: frequency (kx, ky) has
// the signed index i = ky * zpitch + kx (zpitch > 2 K + 1), z(k) is entry |i|,
// conjugated when i < 0.  Indices add like frequencies: i(w - v) = i(w) - i(v).
// They are kept as byte offsets into the table.
__device__ __forceinline__ float2 zget(const float2* zs, int i) {
    float2 t = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(zs) + abs(i));
    t.y = __int_as_float(__float_as_int(t.y) ^ (i & 0x80000000));
    return t;
}
template <typename T2> __device__ __forceinline__ T2 zget(const T2* zs, int i) {
    T2 t = *reinterpret_cast<const T2*>(reinterpret_cast<const char*>(zs) + abs(i));
    if (i < 0) t.y = -t.y;
    return t;
}

// A warp-uniform value, known so to the compiler (a warp reduction), which
// keeps the loops over it free of divergence handling.
__device__ __forceinline__ int uniform(int v) { return (int)__reduce_or_sync(0xffffffffu, (unsigned)v); }

// Sum over the 32 lanes along a butterfly, in every lane.
template <typename T> __device__ __forceinline__ void reduce_warp(T& x, T& y) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
    }
}

__device__ __forceinline__ unsigned cluster_size() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Stores v at the place of `at` (own shared memory) in the shared memory of
// CTA `rank` of the cluster.
template <typename T2> __device__ __forceinline__ void store_cluster(T2* at, unsigned rank, const T2& v) {
    const unsigned long long* u = reinterpret_cast<const unsigned long long*>(&v);
    unsigned a = (unsigned)__cvta_generic_to_shared(at), r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    if constexpr (sizeof(T2) == 8)
        asm volatile("st.shared::cluster.u64 [%0], %1;" :: "r"(r), "l"(u[0]) : "memory");
    else
        asm volatile("st.shared::cluster.v2.u64 [%0], {%1, %2};" :: "r"(r), "l"(u[0]), "l"(u[1]) : "memory");
}

// WEIGHT: the term weighting (SM_W_*).
template <typename T, int WEIGHT>
__global__ void __launch_bounds__(TH, sizeof(T) == 4 ? 2 : 1)
k_phase(PlanDev p, const float2* __restrict__ B, const float2* __restrict__ M, const float* __restrict__ P,
        double2* __restrict__ z) {
    using T2 = typename Cx<T>::T2;
    extern __shared__ __align__(16) unsigned char smem[];
    const int K = p.K, zp = p.zpitch;
    const size_t hb = (size_t)p.hb_rows * p.box_pitch;
    const PhaseLayout lay = phase_layout(p.hb_rows, zp, p.max_batch_points, p.max_batch_units, p.max_batch_late,
                                         sizeof(T2));
    T2* const zs = reinterpret_cast<T2*>(smem);
    T2* const ep = reinterpret_cast<T2*>(smem + lay.ep);
    int4* const srec = reinterpret_cast<int4*>(smem + lay.rec);
    float2* const lb = reinterpret_cast<float2*>(smem + lay.lb);
    int* const liv = reinterpret_cast<int*>(smem + lay.liv);
    int* const rs = reinterpret_cast<int*>(smem + lay.rs);
    const unsigned cl = cluster_size(), rank = cluster_rank();
    const int sl = blockIdx.x / cl, tid = threadIdx.x, lane = tid & 31;
    const int warp = uniform(tid >> 5);
    constexpr int ZB = sizeof(T2);
    int2* const ent = reinterpret_cast<int2*>(smem + lay.ent) + warp * 32;
    double2* const zo = z + (size_t)sl * hb;
    for (int e = tid; e < p.hb_rows * zp; e += TH) zs[e] = Cx<T>::make(0, 0);
    __syncthreads();
    // anchors: z(0) = 1, z(e_x) = M(e_x)/|M(e_x)|, z(e_y) = M(e_y)/|M(e_y)|
    if (tid == 0) {
        zs[0] = Cx<T>::make(1, 0);
        zo[K] = make_double2(1.0, 0.0);
    } else if (tid == 32 || tid == 64) {
        const bool ex = tid == 32;
        const float2 m = M[(size_t)sl * hb + (ex ? K + 1 : p.box_pitch + K)];
        const double n2 = (double)m.x * m.x + (double)m.y * m.y, r = rsqrt(n2);
        const double2 a = n2 > 0 ? make_double2(m.x * r, m.y * r) : make_double2(1.0, 0.0);
        zs[ex ? 1 : zp] = Cx<T>::make((T)a.x, (T)a.y);
        if (ex) {
            zo[K + 1] = a;
            zo[K - 1] = make_double2(a.x, -a.y);
        } else {
            zo[p.box_pitch + K] = a;
        }
    }

    const float* const Ps = P + (size_t)sl * hb;   // power spectrum, for the SNR weighting
    auto pget = [&](int i) { return __ldg(Ps + abs(i) / ZB + K); };    // P at signed index i (box pitch); P(-k) = P(k)
    const float2* const Bs = B + (size_t)sl * p.n_tiles * TILE_PAIRS;
    // s += z(u) z(v) conj b, weighted, for the split of w (index iw) by v (iv);
    // SNR weights: p2 = P(u), P(v)
    auto add_term = [&](T& sx, T& sy, float2 b, int iw, int iv, float2 p2) {
        const T bx = (T)b.x, by = (T)b.y;
        const T2 zu = zget(zs, iw - iv);
        const T2 zv = zget(zs, iv);
        const T2 c = Cx<T>::make(zu.x * zv.x - zu.y * zv.y, zu.x * zv.y + zu.y * zv.x);
        if constexpr (WEIGHT == SM_W_BISPEC) {
            if constexpr (std::is_same<T, float>::value) {
                sx = fmaf(c.x, bx, fmaf(c.y, by, sx));
                sy = fmaf(c.y, bx, fmaf(-c.x, by, sy));
            } else {
                sx += c.x * bx + c.y * by;
                sy += c.y * bx - c.x * by;
            }
        } else {
            // the divisor of the term: |B|, or the speckle-noise variance of B
            T den;
            if constexpr (WEIGHT == SM_W_UNIT) den = sqrt(bx * bx + by * by);
            else den = (T)p2.x * (T)p2.y * (T)pget(iw);
            if (den > (T)0) {
                sx += (c.x * bx + c.y * by) / den;
                sy += (c.y * bx - c.x * by) / den;
            }
        }
    };
    // Early sums of a batch's units [u0, u1): a warp per unit, eight lanes per
    // tile row of 8 offsets, four rows at a time from the unit's up to 32
    // rows (an entry: the row's place in B, and the index of its first offset
    // << 8 | mask of its early offsets).  A row keeps 70 % of its lanes busy
    // where a whole tile kept 53 %.  The lanes load the entries, one unit
    // ahead, and read them back from shared memory; a unit's record comes two
    // units ahead, those of the batch's first units during the batch before.
    const int l8 = lane & 7, stride = (int)cl * PH_WARPS, first = (int)rank * PH_WARPS + warp;
    int2 unit0 = make_int2(0, 0), unit1 = make_int2(0, 0), mine = make_int2(0, 0);
    auto load_unit = [&](int u, int u1) { return u < u1 ? __ldg(p.units + u) : make_int2(0, 0); };
    auto load_entries = [&](int2 unit) {                   // a unit: first entry, entries | point << 6
        return lane < (unit.y & 63) ? __ldg(p.items + unit.x + lane) : make_int2(0, 0);
    };
    auto early = [&](int u0, int u1, T2* sums) {
        const int2* const my_ent = ent + (lane >> 3);
        for (int u = u0 + first; u < u1; u += stride) {
            const int4 rec = srec[unit0.y >> 6];
            const int n = uniform(unit0.y & 63);
            __syncwarp();
            ent[lane] = mine;
            __syncwarp();
            unit0 = unit1;
            mine = load_entries(unit0);
            unit1 = load_unit(u + 2 * stride, u1);
            const float2* const Bw = Bs + rec.w * smi::TILE_V + l8;
            T sx = 0, sy = 0;
            auto rows = [&](auto steps, int g) {           // 4 rows a step
                constexpr int ST = decltype(steps)::value;
                float2 b[ST], p2[ST];
                int iv[ST];
#pragma unroll
                for (int i = 0; i < ST; ++i) {
                    const int2 e = my_ent[g + 4 * i];      // past n: mask 0
                    const bool ok = (e.y >> l8) & 1;
                    b[i] = make_float2(0.f, 0.f);
                    if (ok) b[i] = __ldcs(Bw + (size_t)e.x * smi::VBX);
                    iv[i] = ok ? (e.y >> 8) + l8 * ZB : 0;        // otherwise adds z(w) conj 0
                    p2[i] = make_float2(0.f, 0.f);
                    if (WEIGHT == SM_W_SNR && ok) p2[i] = make_float2(pget(rec.x - iv[i]), pget(iv[i]));
                }
#pragma unroll
                for (int i = 0; i < ST; ++i) add_term(sx, sy, b[i], rec.x, iv[i], p2[i]);
            };
            if constexpr (WEIGHT == SM_W_SNR) {
#pragma unroll 1
                for (int g = 0; g < n; g += 4 * PH_SNR_STEPS) rows(std::integral_constant<int, PH_SNR_STEPS>{}, g);
            } else {
                if (n > 16) rows(std::integral_constant<int, PH_STEPS>{}, 0);
                else rows(std::integral_constant<int, PH_STEPS / 2>{}, 0);
            }
            reduce_warp(sx, sy);
            const T2 s = Cx<T>::make(sx, sy);
            if (cl == 1) {
                if (lane == 0) sums[u - u0] = s;
            } else if (lane < (int)cl) {
                store_cluster(sums + (u - u0), lane, s);
            }
        }
    };

    // What a batch needs in shared memory before its sums: records, ring
    // starts and late terms.  The warps that do not walk the rings load the
    // next batch's into registers while the others do.
    constexpr int PF_THREADS = (PH_WARPS - PH_LATE_WARPS) * 32;
    constexpr int PF = smi::PHASE_LATE / 256;               // late terms per loading thread
    static_assert(PF_THREADS >= 256 && 2 * smi::PHASE_BATCH_MAX <= PF_THREADS, "one record, PF late terms per thread");
    struct Ahead {
        int4 rec;
        int ring;
        int2 t[PF];
        float2 b[PF];
    };
    const int pt = tid - (TH - PF_THREADS);                 // index among the loading threads
    auto load_ahead = [&](Ahead& h, int bt) {
        if (pt < 0 || bt >= p.n_batches) return;
        const int r0 = p.batch_ring[bt], r1 = p.batch_ring[bt + 1];
        const int q0 = p.ring_start[r0], q1 = p.ring_start[r1];
        const int l0 = p.point_rec[q0].z, l1 = p.point_rec[q1].z;
        if (pt <= q1 - q0) h.rec = p.point_rec[q0 + pt];
        if (pt <= r1 - r0) h.ring = p.ring_start[r0 + pt];
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            h.t[i].x = -1;
            if (l0 + pt + i * PF_THREADS < l1) h.t[i] = __ldg(p.late + l0 + pt + i * PF_THREADS);
        }
#pragma unroll
        for (int i = 0; i < PF; ++i)
            if (h.t[i].x >= 0) h.b[i] = __ldg(Bs + h.t[i].x);
    };
    auto store_ahead = [&](const Ahead& h) {
        if (pt < 0) return;
        if (pt < p.max_batch_points + 1) {
            srec[pt] = h.rec;
            rs[pt] = h.ring;
        }
#pragma unroll
        for (int i = 0; i < PF; ++i)
            if (h.t[i].x >= 0) {
                lb[pt + i * PF_THREADS] = h.b[i];
                liv[pt + i * PF_THREADS] = h.t[i].y;
            }
    };
    // the first units of batch bt: their records, then their first entries
    auto first_units = [&](int bt) {
        if (bt >= p.n_batches) return;
        const int u0 = p.batch_unit[bt] + first, u1 = p.batch_unit[bt + 1];
        unit0 = load_unit(u0, u1);
        unit1 = load_unit(u0 + stride, u1);
    };
    Ahead ahead;
    load_ahead(ahead, 0);
    first_units(0);
    mine = load_entries(unit0);
    if (cl > 1) cluster_sync();                   // every CTA of the cluster has started
    for (int bt = 0; bt < p.n_batches; ++bt) {
        store_ahead(ahead);
        const int nr = uniform(p.batch_ring[bt + 1] - p.batch_ring[bt]);
        const int u0 = uniform(p.batch_unit[bt]), u1 = uniform(p.batch_unit[bt + 1]);
        T2* const sums = ep + (bt & 1) * p.max_batch_units;
        __syncthreads();                          // the batch's tables visible, phasors of earlier batches too
        const int q0 = uniform(rs[0]), l0 = uniform(srec[0].z);
        early(u0, u1, sums);
        first_units(bt + 1);
        // early sums complete.  In a cluster every CTA has also walked the
        // batch before, so the other half of the sums may be written again.
        if (cl > 1) cluster_sync();
        else __syncthreads();
        mine = load_entries(unit0);
        if (warp >= PH_LATE_WARPS) {
            load_ahead(ahead, bt + 1);
        } else {
            // Points go round the walking warps in order, so that the few
            // warps with a point in one ring are mostly not those of the
            // next: a warp reads its next point's record, early sums and
            // first late term while others finish theirs.
            struct Point {
                int iw, a, end, iv;               // late terms a, a + 32, ... < end of this lane
                float2 b;
                T2 s;
            };
            auto fetch = [&](int q) {
                Point t;
                const int4 rec = srec[q - q0], nxt = srec[q - q0 + 1];
                t.iw = rec.x;
                t.a = rec.z - l0 + lane;
                t.end = nxt.z - l0;
                t.s = Cx<T>::make(0, 0);
                for (int u = rec.y + lane; u < nxt.y; u += 32) {
                    const T2 s = sums[u - u0];
                    t.s.x += s.x;
                    t.s.y += s.y;
                }
                t.iv = 0;
                t.b = make_float2(0.f, 0.f);
                if (t.a < t.end) {
                    t.iv = liv[t.a];
                    t.b = lb[t.a];
                }
                return t;
            };
            auto finish = [&](const Point& t) {
                T sx = t.s.x, sy = t.s.y;
                auto late_term = [&](float2 b, int iv) {
                    float2 p2 = make_float2(0.f, 0.f);
                    if (WEIGHT == SM_W_SNR) p2 = make_float2(pget(t.iw - iv), pget(iv));
                    add_term(sx, sy, b, t.iw, iv, p2);
                };
                if (t.a < t.end) late_term(t.b, t.iv);
                for (int a = t.a + 32; a < t.end; a += 32) late_term(lb[a], liv[a]);
                reduce_warp(sx, sy);
                const T n2 = sx * sx + sy * sy;
                T2 zz = Cx<T>::make(1, 0);
                if (n2 > (T)0) {
                    const T inv = Cx<T>::rnorm(n2);
                    zz = Cx<T>::make(sx * inv, sy * inv);
                }
                if (lane == 0) *reinterpret_cast<T2*>(smem + t.iw) = zz;
            };
            int q = q0 + warp;                    // the warp's next point
            const int q1 = rs[nr];
            Point cur;
            if (q < q1) cur = fetch(q);
            for (int r = 0; r < nr; ++r) {
                const int qb = rs[r + 1];         // end of the ring's points
                const bool had = q < qb;
                while (q < qb) {
                    finish(cur);
                    q += PH_LATE_WARPS;
                    if (q < qb) cur = fetch(q);
                }
                // the ring's phasors become visible to the walking warps
                asm volatile("bar.sync 1, %0;" :: "n"(PH_LATE_WARPS * 32) : "memory");
                if (had && q < q1) cur = fetch(q);
            }
        }
        __syncthreads();                          // the batch's phasors are visible to all
    }
    // the result, from the table (FP64 conversions in the chain above would
    // queue at the SM's slow FP64 unit); zero outside the cutoff
    for (int e = (int)rank * TH + tid; e < (int)hb; e += (int)cl * TH) {
        const int ky = e / p.box_pitch, kx = e - ky * p.box_pitch - K, q = kx * kx + ky * ky;
        if (q < 2) continue;
        double2 v = make_double2(0.0, 0.0);
        if (q <= p.r2i) {
            const T2 t = zget(zs, (ky * zp + kx) * ZB);
            v = make_double2((double)t.x, (double)t.y);
        }
        zo[e] = v;
    }
}

}  // namespace

namespace smk {

size_t phase_smem_bytes(int hb_rows, int zpitch, int max_points, int max_units, int max_late, int phase_prec) {
    return phase_layout(hb_rows, zpitch, max_points, max_units, max_late,
                        phase_prec == SM_PHASE_FP32 ? sizeof(float2) : 16).bytes;
}

namespace {

// CTAs per subfield: as many as keep the whole grid resident (two CTAs per SM
// when their shared memory allows it) and a unit of the largest batch for
// every warp, up to a portable cluster of 8.
template <typename T, int WEIGHT>
cudaError_t phase_go(const smi::PlanDev& p, int nsub, const float2* B, const float2* M, const float* P, double2* z,
                     size_t sm, cudaStream_t st) {
    auto* const kern = k_phase<T, WEIGHT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    int dev = 0, sms = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int slots = sms * (sizeof(T) == 4 && sm <= 113 * 1024 ? 2 : 1);
    int cl = 1;
    while (cl < 8 && nsub * 2 * cl <= slots && 2 * cl * PH_WARPS <= p.max_batch_units) cl *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nsub * cl);
    cfg.blockDim = dim3(TH);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = cl;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, p, B, M, P, z);
}

template <typename T>
cudaError_t phase_weighted(const smi::PlanDev& p, int nsub, const float2* B, const float2* M, const float* P, double2* z,
                           size_t sm, cudaStream_t st) {
    if (p.weight == SM_W_UNIT) return phase_go<T, SM_W_UNIT>(p, nsub, B, M, P, z, sm, st);
    if (p.weight == SM_W_SNR) return phase_go<T, SM_W_SNR>(p, nsub, B, M, P, z, sm, st);
    return phase_go<T, SM_W_BISPEC>(p, nsub, B, M, P, z, sm, st);
}

}  // namespace

cudaError_t launch_phase(const smi::PlanDev& p, int nsub, const float2* B, const float2* M, const float* P,
                         double2* z, cudaStream_t st) {
    const size_t sm = phase_smem_bytes(p.hb_rows, p.zpitch, p.max_batch_points, p.max_batch_units, p.max_batch_late,
                                       p.phase_prec);
    if (p.phase_prec == SM_PHASE_FP64) return phase_weighted<double>(p, nsub, B, M, P, z, sm, st);
    if (p.phase_prec == SM_PHASE_FF) return phase_weighted<ff>(p, nsub, B, M, P, z, sm, st);
    return phase_weighted<float>(p, nsub, B, M, P, z, sm, st);
}

}  // namespace smk
