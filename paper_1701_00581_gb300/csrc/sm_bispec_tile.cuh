// Bispectrum task body (Sect. 2 and Sect. 3.2: speckle masking, Weigelt 1977),
// shared by the per-stage kernel (k_bispec.cu) and the batched persistent
// launch (k_batch.cu).
#pragma once
#include <type_traits>

#include "sm_internal.h"

namespace smb {

using smi::PlanDev;
using smi::TILE_PAIRS;
using smi::TILE_V;

// A task is up to 32 quads (4 neighbouring targets of a 16-wide strip) per
// offset row, packed from at most BIS_ROWS rows of targets.
constexpr int ROWS = smi::BIS_ROWS;     // 14
constexpr int PW = 18;                  // row pitch of W in smem (float2)
constexpr int PU = 26;                  // row pitch of U in smem (float2)
constexpr int PV = 10;                  // row pitch of V in smem (float2)
constexpr int UC = smi::WBX + smi::VBX - 1;     // 23 cols of U
constexpr int OFF_W = 0;
constexpr int OFF_V = ROWS * PW;
constexpr int OFF_U = OFF_V + smi::VBY * PV;
constexpr int BUF = OFF_U + (ROWS + smi::VBY - 1) * PU;   // 734 float2 per frame buffer
constexpr int THREADS = smi::BISPEC_THREADS;
static_assert(OFF_V % 2 == 0 && OFF_U % 2 == 0 && BUF % 2 == 0 && PW % 2 == 0 && PU % 2 == 0 && PV % 2 == 0,
              "16-byte shared accesses need even float2 offsets");

// Staging in chunks of two values (16 bytes of FP32 spectra): W as rows x 8
// chunks, V as 4 rows x 4 chunks (VCH: its first column is even) or x 5 (one
// value earlier, read one value in), U as (rows + 3) x 12 chunks (24 columns;
// the 24th is read by no used pair); chunk c of W|V|U goes to copy slot
// c / 128 of thread c % 128.
constexpr int UCH = (UC + 1) / 2;                         // 12 chunks per U row
constexpr int WCH = smi::WBX / 2;                         // 8 chunks per W row
constexpr int SLOTS = (ROWS * WCH + smi::VBY * 5 + (ROWS + smi::VBY - 1) * UCH + THREADS - 1) / THREADS;   // 3
static_assert(smi::WBX % 2 == 0, "targets start at even box columns");
static_assert(smi::VBX == 8, "a lane's differences lie in at most three blocks of offsets");

// Bank check (16-byte loads, 8-lane phases): lanes 0..7 of a packed row list
// hold mostly two neighbouring rows and gx = 0..3.  Targets: 16-byte slot
// 9 row + 2 gx (+ j/2) -> {0,2,4,6} + {0,1} mod 8, distinct.  Differences:
// slot 13 row + 2 gx + q, rows differ by 1 -> {0,2,4,6} + {0,5} mod 8,
// distinct.  Offsets: broadcast.

// Asynchronous copies global -> shared of 8 or 16 bytes; the first `bytes`
// bytes come from global memory, the rest of the copy is zero-filled.
__device__ __forceinline__ void cp_async8(unsigned smem_addr, const void* gmem, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" :: "r"(smem_addr), "l"(gmem), "r"(bytes));
}
__device__ __forceinline__ void cp_async16(unsigned smem_addr, const void* gmem, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" :: "r"(smem_addr), "l"(gmem), "r"(bytes));
}
// Chunk copies of two E-byte spectrum values.
template <int E> __device__ __forceinline__ void cp_pair(unsigned s, const void* g, int bytes) {
    if (E == 8) cp_async16(s, g, bytes); else cp_async8(s, g, bytes);
}

// acc += t with Kahan compensation (c carries the rounding error of the sum);
// explicit round-to-nearest intrinsics keep the compiler from fusing or
// reassociating the correction away.
__device__ __forceinline__ void kahan_add(float& acc, float& c, float t) {
    const float y = __fsub_rn(t, c);
    const float s = __fadd_rn(acc, y);
    c = __fsub_rn(__fsub_rn(s, acc), y);
    acc = s;
}

// One frame of the thread's 4 targets x NC neighbouring offset columns from
// the staged rectangles, added into acc.  w: the lane's first target; u: the
// first of the NC + 3 differences of its window (an even column); v: the
// first offset (16-byte aligned with VCH).
template <int NC, bool VCH>
__device__ __forceinline__ void accumulate_frame(const float2* __restrict__ w, const float2* __restrict__ u,
                                                 const float2* __restrict__ v, float2 (&acc)[4][NC]) {
    const float4* w4 = reinterpret_cast<const float4*>(w);
    const float4 w01 = w4[0], w23 = w4[1];
    const float2 a[4] = {make_float2(w01.x, -w01.y), make_float2(w01.z, -w01.w),   // conj I(w)
                         make_float2(w23.x, -w23.y), make_float2(w23.z, -w23.w)};
    const float4* u4 = reinterpret_cast<const float4*>(u);
    float2 c[NC + 4];                                // I(w - v), m = j - k + NC - 1
#pragma unroll
    for (int q = 0; q < NC / 2 + 2; ++q) {
        const float4 t = u4[q];
        c[2 * q] = make_float2(t.x, t.y);
        c[2 * q + 1] = make_float2(t.z, t.w);
    }
#pragma unroll
    for (int k2 = 0; k2 < NC / 2; ++k2) {
        float2 b2[2];                                           // I(v) for two columns (broadcast)
        if (VCH) {
            const float4 t = *reinterpret_cast<const float4*>(v + 2 * k2);
            b2[0] = make_float2(t.x, t.y);
            b2[1] = make_float2(t.z, t.w);
        } else {
            b2[0] = v[2 * k2];
            b2[1] = v[2 * k2 + 1];
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int k = 2 * k2 + e;
            const float2 b = b2[e];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 t = c[j - k + NC - 1];
                const float px = fmaf(t.x, b.x, -t.y * b.y);
                const float py = fmaf(t.x, b.y, t.y * b.x);
                acc[j][k].x = fmaf(px, a[j].x, fmaf(-py, a[j].y, acc[j][k].x));
                acc[j][k].y = fmaf(px, a[j].y, fmaf(py, a[j].x, acc[j][k].y));
            }
        }
    }
}

// Staging: spectra go from global to shared memory by cp.async (zero-filled
// outside the box), FB frames per stage in a two-stage ring, so one barrier
// serves FB frames.  FP32 values (E = 8 bytes) are multiplied out from the
// ring itself.  Half-precision values (E = 4: half2 or bfloat162) are
// copied raw, at half the bytes, and converted to FP32 once per stage into
// one of two compute buffers, a stage ahead of the products, so the inner
// loop and the barrier count are those of FP32.  Shared memory per CTA:
// 2 FB BUF float2 (FP32 ring), or a 2 FB BUF raw ring and 2 FB BUF float2
// of compute buffers (half precision).
// Half precision takes three frames per stage, so that four CTAs' buffers fit
// an SM (its compensated sums, three CTAs, four).
template <int PREC, bool KAHAN> struct Staging {
    static constexpr int E = PREC == SM_FP32 ? 8 : 4;
    static constexpr int FB = E == 4 && !KAHAN ? 3 : 4;
};

template <int PREC>
__device__ __forceinline__ float2 raw_to_float2(unsigned w) {
    if (PREC == SM_FP16) {
        return __half22float2(*reinterpret_cast<const __half2*>(&w));      // still scaled
    } else {
        return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
    }
}

// Box index of spectrum value (kx, ky), or -1 outside the stored box.
__device__ __forceinline__ int box_index(const PlanDev& p, int kx, int ky) {
    const bool in = ky >= -p.R && ky <= p.K && kx >= -p.K && kx <= p.K;
    return in ? (ky + p.R) * p.box_pitch + (kx + p.K) : -1;
}

// Source, destination and size (in 8-byte values) of chunk c of a task's
// W|V|U: two spectrum values from an even box column, both, the first or
// neither inside the box (the box's last column 2K is even, so a chunk never
// starts outside it and ends inside); dst < 0 past the last chunk.
template <bool VCH>
__device__ __forceinline__ void chunk_copy(const PlanDev& p, int c, int rows, int wx0, int wy0, int vx0, int vy0,
                                           int& src, int& dst, int& bytes) {
    constexpr int VC = VCH ? 4 : 5;
    int kx = 0, ky = 0;
    src = 0; dst = -1; bytes = 0;
    if (c < rows * WCH) {
        const int r = c / WCH, h = c % WCH;
        kx = wx0 + 2 * h; ky = wy0 + r; dst = OFF_W + r * PW + 2 * h;
    } else if (c < rows * WCH + smi::VBY * VC) {
        const int c2 = c - rows * WCH, r = c2 / VC, h = c2 - r * VC;
        kx = vx0 - (VCH ? 0 : 1) + 2 * h; ky = vy0 + r; dst = OFF_V + r * PV + 2 * h;
    } else {
        const int c2 = c - rows * WCH - smi::VBY * VC, r = c2 / UCH, h = c2 - r * UCH;
        if (r >= rows + smi::VBY - 1) return;
        kx = wx0 - vx0 - (smi::VBX - 1) + 2 * h; ky = wy0 - vy0 - (smi::VBY - 1) + r;
        dst = OFF_U + r * PU + 2 * h;
    }
    const int i0 = box_index(p, kx, ky), i1 = box_index(p, kx + 1, ky);
    src = i0 >= 0 ? i0 : 0;
    bytes = i0 < 0 ? 0 : (i1 >= 0 ? 16 : 8);
}

// One task (blockIdx-free) of subfield slot `sl`: B of spec[sl] at the task's
// pairs into B[sl]; S is the CTA's staging area, staging_float2<PREC, KAHAN>() float2
// of 16-byte aligned shared memory (2 FB BUF for FP32 spectra, 3 FB BUF for
// half precision).  Runs on 128 threads and synchronises them (barriers 0 and
// 1), so the whole CTA must call it.  VCH: V starts at an even box column.  KAHAN: blocked
// compensated sums -- each block of two stages (2 FB frames) is summed plainly
// into a partial, which is then added to the running sum with Kahan
// compensation; partial, sum and correction fill the registers of 4 columns
// three times over, so the frames stream twice, 4 columns per pass.
template <int PREC, bool VCH, bool KAHAN>
__device__ __forceinline__ void bispec_tile(const PlanDev& p, const void* __restrict__ spec, int F,
                                            float2* __restrict__ B, int task, int sl, float2* __restrict__ S) {
    constexpr int FB = Staging<PREC, KAHAN>::FB, E = Staging<PREC, KAHAN>::E;
    constexpr bool RAW = E == 4;                  // half precision: raw ring + FP32 compute buffer
    const int4 T = __ldg(p.bis_tasks + 2 * task), T2 = __ldg(p.bis_tasks + 2 * task + 1);
    const int wx0 = T.x, wy0 = T.y, vx0 = T.z, vy0 = T.w, rows = T2.x;
    const int tid = threadIdx.x, warp = tid >> 5;
    // the lane's quad: row and place in the strip (an idle lane shares quad 0)
    const int quad = __ldg(p.bis_lanes + (size_t)task * THREADS + tid);
    const int wyl = (quad >> 2) & 15, gx = quad & 3;

    // First offset column and number of columns that this warp computes: the
    // pairs of columns from the first to the last that some lane needs (a
    // warp's needed columns are neighbours but for the one of v = 0), through
    // a warp reduction so that the compiler knows them to be uniform.
    const unsigned range = __reduce_or_sync(0xffffffffu, (unsigned)T2.y >> (8 * warp) & 0xffu);
    const int wfirst = range & 15, wcount = range >> 4;

    constexpr int NP = KAHAN ? 2 : 1;                // passes over the frames
    constexpr int NCP = smi::VBX / NP;               // offset columns per pass
    const size_t box = (size_t)p.box_rows * p.box_pitch;
    const size_t sbase = (size_t)sl * F * box;
    float2* const Bs = B + (size_t)sl * p.n_tiles * TILE_PAIRS;
    // 1 / F, with the FP16 storage scale of the three factors taken out again
    const float sc = 1.0f / (float)F * (PREC == SM_FP16 ? smi::FP16_INV_SCALE * smi::FP16_INV_SCALE *
                                                              smi::FP16_INV_SCALE : 1.0f);
    // spectrum values as E-byte words: float2, or half2 / bfloat162
    using Word = typename std::conditional<E == 8, float2, unsigned>::type;
    const Word* sp = reinterpret_cast<const Word*>(spec) + sbase;
    const int nst = (F + FB - 1) / FB;
    // The ring: E-byte slots, 2 stages x FB frames x BUF; the half-
    // precision compute buffers (2 x FB x BUF float2) follow it.
    Word* ring = reinterpret_cast<Word*>(S);
    float2* cbuf = S + FB * BUF;
    // Copy slots, fixed for the CTA: global source at frame 0, shared
    // destination in buffer 0 and size (chunk_copy counts 8-byte values).
    const Word* g[SLOTS];
    int dst[SLOTS], nb[SLOTS];                       // dst < 0: no copy
    const unsigned s0 = (unsigned)__cvta_generic_to_shared(ring);
#pragma unroll
    for (int i = 0; i < SLOTS; ++i) {
        int src;
        chunk_copy<VCH>(p, tid + i * THREADS, rows, wx0, wy0, vx0, vy0, src, dst[i], nb[i]);
        nb[i] = nb[i] * E / 8;
        g[i] = sp + src;
    }
    auto copy = [&](unsigned soff, size_t goff) {
#pragma unroll
        for (int i = 0; i < SLOTS; ++i)
            if (dst[i] >= 0) cp_pair<E>(s0 + dst[i] * E + soff, g[i] + goff, nb[i]);
    };
    // Stage st holds frames FB st .. FB st + FB - 1, the last one those up to F.
    auto issue = [&](int st) {
        if (st < nst) {
            const unsigned sb = (unsigned)((st & 1) * FB * BUF * E);
            if (st * FB + FB <= F) {
#pragma unroll
                for (int ff = 0; ff < FB; ++ff)
                    copy(sb + ff * BUF * E, (size_t)(st * FB + ff) * box);
            } else {
#pragma unroll 1
                for (int ff = 0; ff < F - st * FB; ++ff) copy(sb + ff * BUF * E, (size_t)(st * FB + ff) * box);
            }
        }
        asm volatile("cp.async.commit_group;");
    };
    // Half precision converts stage st + 1 while stage st is multiplied out,
    // so one barrier per stage serves both: at the barrier of iteration st the
    // raw stage st + 1 has landed, the conversion of stage st (into compute
    // buffer st & 1) is complete and the products of stage st - 1 are done
    // with compute buffer (st + 1) & 1.  A thread converts the chunks that it
    // copied itself; the raw ring slot st & 1 is refilled with stage st + 2
    // after that.
    auto convert = [&](int st) {
        const unsigned* rs = reinterpret_cast<const unsigned*>(ring) + (st & 1) * FB * BUF;
        float2* cb = cbuf + (st & 1) * FB * BUF;
#pragma unroll
        for (int i = 0; i < SLOTS; ++i)
            if (dst[i] >= 0) {
#pragma unroll
                for (int ff = 0; ff < FB; ++ff) {
                    const uint2 t = *reinterpret_cast<const uint2*>(rs + ff * BUF + dst[i]);
                    const float2 a = raw_to_float2<PREC>(t.x), b = raw_to_float2<PREC>(t.y);
                    *reinterpret_cast<float4*>(cb + ff * BUF + dst[i]) = make_float4(a.x, a.y, b.x, b.y);
                }
            }
    };
    // Stage st ready in shared memory, the next on its way; the frames' buffers.
    // A CTA's warps come here from different code, each from the loop made for
    // its columns, which __syncthreads() does not allow; a barrier named by its
    // number, on which every warp arrives for its 32 threads, does.  Every
    // branch below calls this nst times.
    auto next_stage = [&](int st) -> const float2* {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        // stage st visible to all; stage st-1 fully consumed
        asm volatile("bar.sync 1, %0;" :: "n"(THREADS) : "memory");
        if constexpr (RAW) {
            issue(st + 2);
            if (st + 1 < nst) convert(st + 1);
            return cbuf + (st & 1) * FB * BUF;
        } else {
            issue(st + 1);
            return reinterpret_cast<const float2*>(ring) + (st & 1) * FB * BUF;
        }
    };
    // The warp's frames over NC columns from col0 (even) on: every warp runs
    // a loop made for the number of columns it needs, without column tests.
    auto run = [&](auto columns, int col0) {
        constexpr int NC = decltype(columns)::value;
        float2 acc[4][NC];                         // the sums (KAHAN: the running sums)
        float2 part[4][KAHAN ? NC : 1];            // KAHAN: this block's plain partial sums
        float2 comp[4][KAHAN ? NC : 1];            // KAHAN: the running sums' corrections
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int k = 0; k < NC; ++k) acc[j][k] = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < (KAHAN ? NC : 1); ++k) {
                comp[j][k] = make_float2(0.f, 0.f);
                part[j][k] = make_float2(0.f, 0.f);
            }
        }
        const int ow = OFF_W + wyl * PW + 4 * gx, ov = OFF_V + warp * PV + (VCH ? 0 : 1) + col0;
        const int ou = OFF_U + (wyl - warp + smi::VBY - 1) * PU + 4 * gx + smi::VBX - col0 - NC;
        for (int st = 0; st < nst; ++st) {
            const float2* Sst = next_stage(st);
            const int nf = min(FB, F - st * FB);
#pragma unroll 1
            for (int ff = 0; ff < nf; ++ff) {
                const float2* const Sf = Sst + ff * BUF;
                if constexpr (KAHAN) accumulate_frame<NC, VCH>(Sf + ow, Sf + ou, Sf + ov, part);
                else accumulate_frame<NC, VCH>(Sf + ow, Sf + ou, Sf + ov, acc);
            }
            // KAHAN: every second stage (8 frames) and after the last one,
            // the partial sums go into the running sums
            if constexpr (KAHAN) if ((st & 1) == 1 || st + 1 == nst) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int k = 0; k < NC; ++k) {
                        kahan_add(acc[j][k].x, comp[j][k].x, part[j][k].x);
                        kahan_add(acc[j][k].y, comp[j][k].y, part[j][k].y);
                        part[j][k] = make_float2(0.f, 0.f);
                    }
            }
        }
        // Store.  A pair whose two offsets v and u = w - v both lie within R
        // is stored at both (B(u, v) = B(v, u)) and computed at one of them,
        // the one that pair_at_lower keeps; tasks without such pairs store
        // their columns whole (a slot of an unused pair may hold anything).
        if (quad < 0) return;
        const int wy = wy0 + wyl, vy = vy0 + warp;
        const int wb = (wy / smi::WBY) * p.n_wbx + (wx0 + p.K) / smi::WBX;
        const int slot = (wy % smi::WBY) * smi::WBX + 4 * gx;
        const int* const tiles = p.tile_of + (size_t)wb * p.n_vbx * p.n_vby;
        float2* const out = Bs + (size_t)__ldg(tiles + T2.z) * TILE_PAIRS + slot * TILE_V + warp * smi::VBX + col0;
        const bool whole = T2.w == 0;
        // The tiles of the other order: u lies in one row of offset blocks and, over
        // the lane's pairs, in at most three neighbouring ones.  Loaded together, up
        // front: one by one in the loop, each would wait for the one before (one
        // subfield of 64^2, 10 frames: 14.5 us, now 10.6).
        const int cx0 = wx0 + 4 * gx - (vx0 + col0 + NC - 1) - p.v_org, cy = wy - vy + p.R;
        int other[3] = {0, 0, 0};
        if (!whole) {
            const int* const row = tiles + min(max(cy, 0), 2 * p.R) / smi::VBY * p.n_vbx;
#pragma unroll
            for (int i = 0; i < 3; ++i) other[i] = __ldg(row + min(max((cx0 >> 3) + i, 0), p.n_vbx - 1));
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (whole) {
                float4* o = reinterpret_cast<float4*>(out + j * TILE_V);
#pragma unroll
                for (int q = 0; q < NC / 2; ++q)
                    o[q] = make_float4(acc[j][2 * q].x * sc, acc[j][2 * q].y * sc,
                                       acc[j][2 * q + 1].x * sc, acc[j][2 * q + 1].y * sc);
                continue;
            }
            const int wx = wx0 + 4 * gx + j, w2 = wx * wx + wy * wy;
            const bool okw = (wy > 0 || (wy == 0 && wx > 0)) && w2 >= 2 && w2 <= p.r2i;
#pragma unroll
            for (int k = 0; k < NC; ++k) {
                const int vx = vx0 + col0 + k, ux = wx - vx, uy = wy - vy;
                const int v2 = vx * vx + vy * vy, u2 = ux * ux + uy * uy;
                if (!(okw && v2 > 0 && v2 <= p.R * p.R && v2 < w2 && u2 < w2)) continue;
                const bool both = u2 <= p.R * p.R;
                if (both && !smi::pair_at_lower(vx, vy, ux, uy)) continue;
                const float2 val = make_float2(acc[j][k].x * sc, acc[j][k].y * sc);
                out[j * TILE_V + k] = val;
                if (both) {
                    const int cx = (cx0 & 7) + j - k + NC - 1;          // from the first block on
                    const int t = cx < 8 ? other[0] : cx < 16 ? other[1] : other[2];
                    Bs[(size_t)t * TILE_PAIRS + (slot + j) * TILE_V + (cy % smi::VBY) * smi::VBX + cx % smi::VBX] = val;
                }
            }
        }
    };
#pragma unroll
    for (int pass = 0; pass < NP; ++pass) {
        if constexpr (KAHAN) {                     // a pass that no warp has a column in (the same for all warps)
            const unsigned ranges = __reduce_or_sync(0xffffffffu, (unsigned)T2.y);
            bool any = false;
#pragma unroll
            for (int q = 0; q < smi::VBY; ++q) {
                const int f = ranges >> (8 * q) & 15, c = ranges >> (8 * q + 4) & 15;
                any |= c > 0 && f < (pass + 1) * NCP && f + c > pass * NCP;
            }
            if (!any) continue;
        }
        __syncwarp();                              // a warp's idle lanes leave run() before the others
        if (pass > 0) __syncthreads();             // the previous pass is done with the ring
        issue(0);
        if constexpr (RAW) {
            issue(1);
            asm volatile("cp.async.wait_group 1;");
            __syncthreads();                      // raw stage 0 visible
            convert(0);
        }
        // the warp's columns of this pass (first and count are even)
        const int col0 = max(wfirst, pass * NCP), n = max(0, min(wfirst + wcount, (pass + 1) * NCP) - col0);
        if (n == 0) {
            for (int st = 0; st < nst; ++st) next_stage(st);
        } else if (n == 2) {
            run(std::integral_constant<int, 2>{}, col0);
        } else if (NCP == 4 || n == 4) {
            run(std::integral_constant<int, 4>{}, col0);
        } else if (n == 6) {
            if constexpr (NCP == 8) run(std::integral_constant<int, 6>{}, col0);
        } else {
            if constexpr (NCP == 8) run(std::integral_constant<int, 8>{}, col0);
        }
        asm volatile("cp.async.wait_group 0;");
    }
}


// float2 elements of the staging area bispec_tile<PREC, VCH, KAHAN> takes
template <int PREC, bool KAHAN> __host__ __device__ constexpr int staging_float2() {
    return (Staging<PREC, KAHAN>::E == 8 ? 2 : 3) * Staging<PREC, KAHAN>::FB * BUF;
}
template <bool KAHAN> __host__ __device__ constexpr size_t staging_bytes(int prec) {
    return (size_t)(prec == SM_FP32 ? staging_float2<SM_FP32, KAHAN>() : staging_float2<SM_FP16, KAHAN>()) * 8;
}

}  // namespace smb
