// lbm_reduce.cu -- FP64 reduction of the observable partials (arXiv
// 2403.16122: the global volume, solid, enthalpy and mass sums and the
// mass-source integral of Sections 4.1-4.3, plus the front and velocity
// records). The step kernels leave one partial per tile or strip item and
// observable; this kernel turns them into one record per lattice.
//
// FP64 arithmetic runs at two additions a cycle and SM on this GPU, and the
// kernel is otherwise a chain of load latencies (700-800 cycles each), cold
// instruction fetches and barriers: a lattice's partials are spread over CTAs of
// kPer, eight threads an observable load their values at once, straight into
// registers, and add them in a tree, and a lattice that fits one CTA needs no
// second pass. With more CTAs the last one to finish (an atomic count) combines
// the CTA sums in the same way. Every sum is taken in an order fixed by the
// partial indices alone, so the result does not depend on scheduling. A call of
// one step and a read of its observables, in us: 256 x 256 sites 30.6 with the
// values staged through shared memory, 23.4 so (18 without a reduction at all);
// 1024 x 1024 78.5 in CTAs of 256 summed in two levels of 16, 70.2 in CTAs of 64,
// 66 so (59). One copy of the summing code for both passes was 1 us slower.
#include "lbm_reduce.h"

#include "lbm_load.cuh"

namespace lbmk {
namespace {

constexpr int kPer = 64;              // partials per CTA
constexpr int kThreads = 128;
constexpr int kSums = kObs + 1;       // the observables, then the mdot running sums
constexpr int kLanes = 8;             // threads that sum one observable
constexpr int kSumThreads = kSums * kLanes;
static_assert(kSumThreads == 96 && kPer == 8 * kLanes, "three warps sum, one has the profile");

__device__ __forceinline__ double combine(int j, double a, double b) {
    return j == 9 ? fmax(a, b) : a + b;  // slot 9: max |u|; 0 is neutral for it too
}

// Sum over n <= kPer values at p + q * stride for observable j, by its kLanes
// threads: thread c takes values c, c + 8, .. c + 56, all loaded at once, and
// adds them pairwise; then the threads pairwise. Valid in every thread.
__device__ __forceinline__ double sum_values(const double* p, long long stride, int n, int j, int c) {
    double a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = c + 8 * k < n ? ld_live(p + (c + 8 * k) * stride) : 0.0;
#pragma unroll
    for (int w = 4; w > 0; w >>= 1)
#pragma unroll
        for (int k = 0; k < w; ++k) a[k] = combine(j, a[k], a[k + w]);
    double s = a[0];
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) s = combine(j, s, __shfl_xor_sync(0xffffffffu, s, o));
    return s;
}

// CTA (k, b) sums the partials begin + b * kPer .. of lattice k. The last CTA
// of the lattice writes the observable record and the freezing record and
// re-arms the count. The column profile that the observable step accumulated is
// published (copied to prof_out, the accumulator zeroed for the next
// observable step) by all of the lattice's CTAs, a share each.
__global__ void __launch_bounds__(kThreads)
reduce_obs_split(const Inst* __restrict__ insts, const double* __restrict__ partials,
                 double* __restrict__ out, double* __restrict__ out_host,
                 double* __restrict__ frz, double* __restrict__ scratch,
                 unsigned* __restrict__ counts, long long step) {
    __shared__ double tot[kSums];
    __shared__ bool last;
    // Programmatic dependent launch: this grid is scheduled while the
    // observable step drains and reads nothing that step writes before it has
    // completed; the next step's grid may be scheduled as soon as every CTA
    // here has started (it waits for this grid in turn). No-ops without the
    // attribute.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int k = blockIdx.x, b = blockIdx.y, t = threadIdx.x;
    const Inst& I = insts[k];
    const int begin = I.part_begin, n = I.part_end - I.part_begin;
    const int n_cta = n > 0 ? (n + kPer - 1) / kPer : 1;
    if (b >= n_cta) return;  // whole CTA, before any barrier or count
    const int j = t / kLanes, c = t % kLanes;
    const int at = begin + b * kPer, here = n - b * kPer < kPer ? n - b * kPer : kPer;
    const double* const row = j < kObs ? partials + (long long)j * I.part_stride + at
                                       : (I.macc ? I.macc + at : nullptr);
    double* const prof = I.prof;
    double* const prof_out = I.prof_out;
    const int nx = I.nx;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    double s = 0.0;
    if (t < kSumThreads) {
        s = sum_values(row, 1, row ? here : 0, j, c);
    } else if (prof && prof_out) {  // the last warp: a share of the column profile
        for (int x = b * 32 + (t & 31); x < nx; x += n_cta * 32) {
            prof_out[x] = ld_live(prof + x);
            prof[x] = 0.0;
        }
    }
    if (n_cta > 1) {
        // the scratch slots of lattice k: floor(begin / kPer) + k onwards (disjoint
        // across lattices, fewer than max_parts / kPer + n_inst + 1 in all)
        double* const mine = scratch + (long long)(begin / kPer + k) * kSums;
        if (t < kSumThreads && c == 0) {
            mine[(long long)b * kSums + j] = s;
            __threadfence();
        }
        __syncthreads();
        if (t == 0) last = atomicAdd(counts + k, 1u) == (unsigned)(n_cta - 1);
        __syncthreads();
        if (!last) return;
        __threadfence();
        if (t < kSumThreads) {
            s = 0.0;
            for (int c0 = 0; c0 < n_cta; c0 += kPer)
                s = combine(j, s, sum_values(mine + (long long)c0 * kSums + j, kSums,
                                             n_cta - c0 < kPer ? n_cta - c0 : kPer, j, c));
        }
    }
    if (t < kSumThreads && c == 0) {
        tot[j] = s;
        if (j < kObs) {
            out[(long long)k * kObs + j] = s;
            if (out_host) out_host[(long long)k * kObs + j] = s;
        }
    }
    __syncthreads();
    if (t == 0) {
        if (n_cta > 1) counts[k] = 0u;  // the next reduction is stream-ordered after this one
        if (frz) {
            double* r = frz + (long long)k * kFrz;
            const double vol = tot[LBM_OBS_VOLUME], sol = tot[LBM_OBS_SOLID];
            const double X = vol > 0.0 ? sol / vol : 0.0;
            r[LBM_FRZ_STEP] = (double)step;
            r[LBM_FRZ_MDOT_INTEGRAL] = tot[kObs];
            if (X >= kFreezeFraction && r[LBM_FRZ_FREEZE_STEP] < 0.0) r[LBM_FRZ_FREEZE_STEP] = (double)step;
            r[LBM_FRZ_SOLID_FRACTION] = X;
        }
    }
}

}  // namespace

int reduce_slots(int max_parts, int n_inst) { return max_parts / kPer + n_inst + 1; }

cudaError_t launch_reduce_obs(const Inst* d_inst, int n_inst, int max_lattice_parts,
                              const double* d_partials, double* d_obs, double* d_obs_host,
                              double* d_frz, double* d_scratch, unsigned* d_counts,
                              long long step, cudaStream_t s) {
    if (n_inst <= 0) return cudaSuccess;
    const int per = (max_lattice_parts + kPer - 1) / kPer;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_inst, (unsigned)(per > 0 ? per : 1));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, reduce_obs_split, d_inst, d_partials, d_obs, d_obs_host, d_frz,
                              d_scratch, d_counts, step);
}

}  // namespace lbmk
