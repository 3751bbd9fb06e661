// Checks a batch's device queue without a GPU: the CUDA calls below keep it in host memory.
// usage: batch_host launch tile_order lookahead
#include <array>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>

#include "sm_batch.cpp"

extern "C" {
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 227 * 1024;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) { memset(a, 0, sizeof(*a)); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 4;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { *p = calloc(n, 1); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = calloc(n, 1); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
}

int main(int, char** argv) {
    // two channels, one with a ragged grid; the first twice
    sm_plan* plans[3];
    int F[3] = {5, 3, 7}, ft[3] = {SM_U16, SM_F32, SM_U16};
    for (int i = 0; i < 2; ++i) {
        sm_channel ch;
        memset(&ch, 0, sizeof(ch));
        ch.N = i ? 128 : 64; ch.R = i ? 9 : 8; ch.W = i ? 200 : 150; ch.H = i ? 128 : 110;
        ch.fc = 0.2885; ch.stride = ch.N / 2; ch.max_frames = 10; ch.ck = 0.435;
        if (sm_plan_create(&ch, 0, &plans[i]) != SM_OK) { printf("refused: %s\n", sm_last_error()); return 1; }
    }
    plans[2] = plans[0];
    sm_batch_opts o = {};
    o.launch = atoi(argv[1]); o.tile_order = atoi(argv[2]); o.lookahead = atoi(argv[3]); o.ctas_per_sm = 4;
    sm_batch* bt = nullptr;
    if (sm_batch_create(3, plans, F, ft, &o, &bt) != SM_OK) { printf("refused: %s\n", sm_last_error()); return 1; }
    const bool fused = o.launch == SM_BATCH_FUSED;
    std::map<std::array<int, 4>, int> at;                  // item -> its place in the queue
    int bad = 0, covered = 0;
    for (int i = 0; i < bt->n_items; ++i) {
        const int4 it = bt->d_items[i];
        bad += !at.insert({{it.x, it.y, it.z, it.w}, i}).second;                       // twice
    }
    for (int b = 0; b < 3; ++b) {
        const PlanDev& d = plans[b]->dev;
        for (int s = 0; s < d.n_sub; ++s) {
            int last = -1;                                 // the subfield's last transform: before its first task
            for (int f = 0; fused && f < F[b]; ++f) {
                auto p = at.find({0, b, s, f});
                if (p == at.end()) { ++bad; continue; }
                last = std::max(last, p->second);
                at.erase(p);
                ++covered;
            }
            for (int t = 0; t < d.n_bis_tasks; ++t) {
                auto p = at.find({1, b, s, t});
                if (p == at.end() || p->second < last) { ++bad; continue; }
                at.erase(p);
            }
            covered += d.n_tiles;
        }
    }
    bad += (int)at.size();                                 // anything else
    int n_items = 0, grid = 0;
    size_t bytes = 0;
    sm_batch_info(bt, &n_items, &grid, &bytes);
    bad += n_items != covered || bytes < (size_t)bt->n_items * sizeof(int4);
    int least = 1 << 30;                                   // items of the smallest subfield
    for (int b = 0; b < 3; ++b) least = std::min(least, F[b] + plans[b]->dev.n_bis_tasks);
    printf("%d wrong, %d items, lookahead %d, in flight %d of %d a subfield\n", bad, bt->n_items, bt->opts.lookahead, grid,
           least);
    sm_batch_destroy(bt);
    sm_plan_destroy(plans[0]);
    sm_plan_destroy(plans[1]);
    return bad != 0;
}
