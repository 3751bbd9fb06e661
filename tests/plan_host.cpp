// Checks a plan's host-built tables without a GPU: the CUDA allocation calls below keep them in host memory.
// usage: plan_host N R fc phase_prec
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "sm_plan.h"

extern "C" {
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = calloc(n, 1); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
}

using namespace smi;

static int bad = 0;
static void check(bool ok, const char* what) {
    if (!ok && bad++ < 10) printf("wrong: %s\n", what);
}

template <typename F> static double best_ms(F f) {
    double best = 1e30;
    for (int i = 0; i < 5; ++i) {
        const auto t0 = std::chrono::steady_clock::now();
        f();
        best = std::min(best, std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count());
    }
    return best;
}

int main(int argc, char** argv) {
    sm_channel ch;
    memset(&ch, 0, sizeof(ch));
    ch.N = ch.W = ch.H = atoi(argv[1]); ch.R = atoi(argv[2]); ch.fc = atof(argv[3]); ch.phase_prec = atoi(argv[4]);
    ch.stride = ch.N / 2; ch.max_frames = 10; ch.ck = 0.435;
    sm_plan* pl = nullptr;
    if (sm_plan_create(&ch, 0, &pl) != SM_OK) { printf("refused: %s\n", sm_last_error()); return 1; }
    const PlanDev& d = pl->dev;
    const int K = d.K, R = d.R, nvb = pl->n_vbx * pl->n_vby;
    auto used = [&](int wx, int wy, int vx, int vy) { return pair_used_host(wx, wy, vx, vy, d.r2i, R * R); };

    // the slots of every tile, one by one (timed: what the plan's own construction is compared with)
    long long n_pairs = 0;
    int n_tiles = 0;
    auto slots = [&](bool look) {
        n_pairs = n_tiles = 0;
        for (int wb = 0; wb < d.n_wbx * d.n_wby; ++wb)
            for (int vb = 0; vb < nvb; ++vb) {
                const int wx0 = -K + WBX * (wb % d.n_wbx), wy0 = WBY * (wb / d.n_wbx);
                const int vx0 = d.v_org + VBX * (vb % pl->n_vbx), vy0 = -R + VBY * (vb / pl->n_vbx);
                unsigned mask = 0;
                for (int a = 0; a < WBY; ++a)
                    for (int b = 0; b < WBX; ++b)
                        for (int l = 0; l < TILE_V; ++l)
                            if (used(wx0 + b, wy0 + a, vx0 + l % VBX, vy0 + l / VBX)) { ++n_pairs; mask |= 1u << l; }
                const int t = pl->tile_of[(size_t)wb * nvb + vb];
                if (look) check(mask ? t == n_tiles && pl->tile_masks[t] == mask && pl->tiles[t].x == wx0 &&
                                           pl->tiles[t].y == wy0 && pl->tiles[t].z == vx0 && pl->tiles[t].w == vy0
                                     : t < 0, "tile list");
                n_tiles += mask != 0;
            }
    };
    slots(true);
    check(n_tiles == d.n_tiles && n_pairs == pl->n_pairs, "pairs or tiles counted");

    // the bispectrum's tasks, stored as the kernel does: every used pair once, no slot twice
    std::vector<unsigned char> stores((size_t)d.n_tiles * TILE_PAIRS, 0);
    for (int k = 0; k < d.n_bis_tasks; ++k) {
        const int4 a = pl->bis_tasks[2 * k], b = pl->bis_tasks[2 * k + 1];
        check(b.x >= 1 && b.x <= BIS_ROWS, "rows of a task");
        for (int i = 0; i < BISPEC_THREADS; ++i) {
            const int lane = pl->bis_lanes[(size_t)k * BISPEC_THREADS + i], q = i / 32;
            if (lane < 0) continue;
            check((lane >> 2) < b.x, "row of a lane");
            const int wy = a.y + (lane >> 2), vy = a.w + q, first = b.y >> (8 * q) & 15, count = (unsigned)b.y >> (8 * q + 4) & 15;
            const int wb = wy / WBY * d.n_wbx + (a.x + K) / WBX;
            for (int j = 0; j < 4; ++j)
                for (int e = first; e < first + count; ++e) {
                    const int wx = a.x + 4 * (lane & 3) + j, vx = a.z + e, ux = wx - vx, uy = wy - vy;
                    auto store = [&](int x, int y) {
                        const int t = pl->tile_of[(size_t)wb * nvb + (y + R) / VBY * pl->n_vbx + (x - d.v_org) / VBX];
                        check(t >= 0, "stored outside the tiles");
                        ++stores[(size_t)t * TILE_PAIRS + (wy % WBY * WBX + 4 * (lane & 3) + j) * TILE_V +
                                 (y + R) % VBY * VBX + (x - d.v_org) % VBX];
                    };
                    const bool both = ux * ux + uy * uy <= R * R;
                    if (b.w == 0) store(vx, vy);
                    else if (used(wx, wy, vx, vy) && !(both && !pair_at_lower(vx, vy, ux, uy))) {
                        store(vx, vy);
                        if (both && (ux != vx || uy != vy)) store(ux, uy);       // u = v: one slot
                    }
                }
        }
    }
    for (int t = 0; t < d.n_tiles; ++t)
        for (int s = 0; s < TILE_PAIRS; ++s) {
            const int4 T = pl->tiles[t];
            const int n = stores[(size_t)t * TILE_PAIRS + s], wl = s / TILE_V, vl = s % TILE_V;
            check(used(T.x + wl % WBX, T.y + wl / WBX, T.z + vl % VBX, T.w + vl / VBX) ? n == 1 : n <= 1, "stores of a pair");
        }

    // the recursion: every used pair of a point early or late; early terms read rings before the batch, late ones
    // earlier rings of it
    const int zb = d.phase_prec == SM_PHASE_FP32 ? 8 : 16;
    std::vector<int> ring_of((size_t)(K + 1) * (2 * K + 1), -1);          // anchors: -1
    for (int r = 0; r < d.n_rings; ++r)
        for (int p = pl->ring_start[r]; p < pl->ring_start[r + 1]; ++p)
            ring_of[(size_t)pl->points[p].y * (2 * K + 1) + pl->points[p].x + K] = r;
    auto ring = [&](int x, int y) {
        if (y < 0 || (y == 0 && x < 0)) { x = -x; y = -y; }
        return ring_of[(size_t)y * (2 * K + 1) + x + K];
    };
    std::vector<int> seen((size_t)(2 * R + 1) * (2 * R + 1));
    for (int b = 0; b + 1 < (int)pl->batch_ring.size(); ++b) {
        const int r0 = pl->batch_ring[b], p0 = pl->ring_start[r0];
        for (int r = r0; r < pl->batch_ring[b + 1]; ++r)
            for (int p = pl->ring_start[r]; p < pl->ring_start[r + 1]; ++p) {
                const int wx = pl->points[p].x, wy = pl->points[p].y;
                const int4 rec = pl->point_rec[p], nxt = pl->point_rec[p + 1];
                std::fill(seen.begin(), seen.end(), 0);
                auto term = [&](int t, int slot, int l, int iv, bool late) {
                    const int4 T = pl->tiles[t];
                    const int vx = T.z + l % VBX, vy = T.w + l / VBX, last = std::max(ring(vx, vy), ring(wx - vx, wy - vy));
                    check(slot == rec.w && T.x + slot % WBX == wx && T.y + slot / WBX == wy, "target of a term");
                    check(used(wx, wy, vx, vy) && iv == (vy * d.zpitch + vx) * zb, "offset of a term");
                    check(late ? last >= r0 && last < r : last < r0, late ? "late term" : "early term");
                    ++seen[(size_t)(vy + R) * (2 * R + 1) + vx + R];
                };
                check(rec.x == (wy * d.zpitch + wx) * zb, "index of a point");
                for (int u = rec.y; u < nxt.y; ++u) {
                    const int2 unit = pl->units[u];
                    check((unit.y >> 6) == p - p0 && u >= pl->batch_unit[b] && u < pl->batch_unit[b + 1], "unit of a point");
                    for (int i = 0; i < (unit.y & 63); ++i) {
                        const int2 it = pl->items[unit.x + i];
                        for (int e = 0; e < VBX; ++e)
                            if (it.y >> e & 1)
                                term(it.x / (TILE_W * VBY), rec.w, it.x % (TILE_W * VBY) * VBX + e, (it.y >> 8) + e * zb, false);
                    }
                }
                for (int a = rec.z; a < nxt.z; ++a) {
                    const int2 t = pl->late[a];
                    term(t.x / TILE_PAIRS, t.x % TILE_PAIRS / TILE_V, t.x % TILE_V, t.y, true);
                }
                for (int vy = -R; vy <= R; ++vy)
                    for (int vx = -R; vx <= R; ++vx)
                        check(seen[(size_t)(vy + R) * (2 * R + 1) + vx + R] == (used(wx, wy, vx, vy) ? 1 : 0), "terms of a point");
            }
    }
    const double slots_ms = best_ms([&] { slots(false); });
    sm_plan_destroy(pl);
    const double plan_ms = best_ms([&] { sm_plan* q; sm_plan_create(&ch, 0, &q); sm_plan_destroy(q); });
    printf("%d wrong, %lld pairs, plan %.3f ms, slots %.3f ms\n", bad, n_pairs, plan_ms, slots_ms);
    return bad != 0;
}
