// Mean bispectrum accumulation (Sect. 2 and Sect. 3.2: speckle masking,
// Weigelt 1977): for every pair (w, v) that the phase recursion reads,
//
//     B(w - v, v) = (1/F) sum_i I_i(w - v) I_i(v) conj I_i(w),
//
// with w in the upper half plane, 0 < |v| <= R, |v| < |w| and |w - v| < |w|.
//
// Work decomposition: a CTA owns a task of one subfield: 8 x 4 offsets v and
// up to 128 quads of four neighbouring targets, 32 per offset row.  Warp q
// owns offset row vy0 + q; each lane owns one quad and the warp's offset
// columns: up to 32 complex accumulators in registers for the whole burst.
// Per frame the CTA stages three rectangles of the frame spectrum in shared
// memory: the targets W (up to 14 rows of a 16-wide strip), the offsets V
// (4 x 8) and U = W - V (3 rows more, 24 wide).  For its 32 pairs a thread
// reads 4 values of W, 8 broadcast values of V and an 11-wide sliding window
// of U (12 shared loads of 16 bytes for 32 pairs), so each triple product
// costs 8 FP32 FMA-pipe instructions.
//
// What bounds it is FP32 issue: FMAs of three register operands issue at 0.77
// of the pipe's peak (the register file's ports; a loop of nothing else
// measures the same, and packed f32x2 FMAs do worse, 0.70), so what can be
// saved is products and instructions beside them.  The plan packs the quads
// that hold a pair to compute, offset row by offset row (fixed 16 x 8 blocks
// of targets computed 37 % more pairs than are used at N = 256, R = 24 and
// 78 % at N = 128, R = 16; the packed tasks 22 % and 42 %), and of the two
// orders of a pair with both offsets inside |v| <= R one is computed and
// stored twice.  Every warp runs a loop made for the number of column pairs
// it needs, one frame to an iteration: four such loops unrolled over the
// frames of a stage overflow the instruction cache (7.1 against 4.8 ms for 15
// subfields of 256^2).
//
// Spectra are staged by cp.async, four frames per barrier, while the
// previous four frames are multiplied out (half-precision spectra at half
// the bytes, three frames per barrier, converted to FP32 once per stage in
// shared memory).  W and U start at even box
// columns (the plan places the offset grid so that they do), so they move in
// 16-byte copies of two spectrum values, and so does V, from one value
// earlier when its own start is odd.  A last, partial stage holds its own
// frames only.  Accumulators are written once per burst.
//
// 304 subfields of 256^2, R = 24, 100 frames: 102.0 -> 89.4 ms; 225 of 128^2,
// R = 16: 11.5 -> 8.7 ms; one of 64^2, R = 8: 47 -> 36 us; 25 of 256^2, 30 frames:
// FP32 3.07 -> 2.70 ms, FP16 3.66 -> 3.22, with compensated sums too 5.37 -> 5.03.
#include "sm_bispec_tile.cuh"

namespace {

using smi::PlanDev;
using smb::THREADS;

// Four CTAs per SM (128 registers a thread); the compensated sums keep a
// partial, a running sum and a correction per pair and take three (168).
template <int PREC, bool VCH, bool KAHAN>
__global__ void __launch_bounds__(THREADS, KAHAN ? 3 : 4)
k_bispectrum(PlanDev p, const void* __restrict__ spec, int F, float2* __restrict__ B) {
    extern __shared__ __align__(16) float2 S[];
    smb::bispec_tile<PREC, VCH, KAHAN>(p, spec, F, B, blockIdx.x, blockIdx.y, S);
}

template <int PREC, bool VCH, bool KAHAN>
cudaError_t bispec_go(const PlanDev& p, const void* spec, int F, int nsub, float2* B, cudaStream_t st) {
    constexpr size_t sm = smb::staging_bytes<KAHAN>(PREC);
    const cudaError_t e = cudaFuncSetAttribute(k_bispectrum<PREC, VCH, KAHAN>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k_bispectrum<PREC, VCH, KAHAN><<<dim3(p.n_bis_tasks, nsub), THREADS, sm, st>>>(p, spec, F, B);
    return cudaGetLastError();
}

template <int PREC, bool KAHAN>
cudaError_t bispec_v(const PlanDev& p, const void* spec, int F, int nsub, float2* B, cudaStream_t st) {
    const bool vch = ((p.v_org + p.K) & 1) == 0;     // every task's V starts at an even column
    return vch ? bispec_go<PREC, true, KAHAN>(p, spec, F, nsub, B, st)
               : bispec_go<PREC, false, KAHAN>(p, spec, F, nsub, B, st);
}

}  // namespace

namespace smk {

cudaError_t launch_bispectrum(const smi::PlanDev& p, const void* spec, int F, int nsub, float2* B,
                              cudaStream_t st) {
    if (p.acc_mode == SM_ACC_KAHAN) {
        if (p.prec == SM_FP32) return bispec_v<SM_FP32, true>(p, spec, F, nsub, B, st);
        if (p.prec == SM_FP16) return bispec_v<SM_FP16, true>(p, spec, F, nsub, B, st);
        return bispec_v<SM_BF16, true>(p, spec, F, nsub, B, st);
    }
    if (p.prec == SM_FP32) return bispec_v<SM_FP32, false>(p, spec, F, nsub, B, st);
    if (p.prec == SM_FP16) return bispec_v<SM_FP16, false>(p, spec, F, nsub, B, st);
    return bispec_v<SM_BF16, false>(p, spec, F, nsub, B, st);
}

}  // namespace smk
