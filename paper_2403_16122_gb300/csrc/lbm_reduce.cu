// lbm_reduce.cu -- FP64 reduction of the observable partials (arXiv
// 2403.16122: the global volume, solid, enthalpy and mass sums and the
// mass-source integral of Sections 4.1-4.3, plus the front and velocity
// records). The step kernels leave one partial per tile or strip item and
// observable; this kernel turns them into one record per lattice.
//
// FP64 arithmetic runs at two additions a cycle and SM on this GPU, and the
// kernel is otherwise a chain of load latencies and barriers: a lattice's
// partials are spread over CTAs of kPer, a CTA sums only the values it has, by
// eight threads an observable and three shuffles, and a lattice that fits one
// CTA needs no second pass. With more CTAs the last one to finish (an atomic
// count) combines the CTA sums in the same way. Every sum is taken in an order
// fixed by the partial indices alone, so the result does not depend on
// scheduling. Against CTAs of 256 summed in two levels of 16 with a barrier
// between them, a call of one step takes 60.4 us instead of 69.5 on 1024 x 1024
// sites, 28.3 instead of 32.8 on 512 x 512, 9.5 instead of 13.1 on 256 x 8.
#include "lbm_reduce.h"

namespace lbmk {
namespace {

constexpr int kPer = 64;              // partials per CTA
constexpr int kThreads = 128;
constexpr int kSums = kObs + 1;       // the observables, then the mdot running sums
constexpr int kLanes = 8;             // threads that sum one observable
static_assert(kSums * kLanes <= kThreads && kPer % kLanes == 0, "reduction shape");

__device__ __forceinline__ double combine(int j, double a, double b) {
    return j == 9 ? fmax(a, b) : a + b;  // slot 9: max |u|; 0 is neutral for it too
}

// Sum of the n <= kPer values staged in v[j], by thread t = j * kLanes + c: the
// values c, c + kLanes, ... in order, then the lanes of the observable pairwise.
// Whole warps take part; the result is valid where t < kSums * kLanes.
__device__ __forceinline__ double sum_staged(const double (*v)[kPer + 1], int n, int t) {
    const int j = t / kLanes < kSums ? t / kLanes : 0, c = t % kLanes;
    double s = 0.0;
    for (int q = c; q < n; q += kLanes) s = combine(j, s, v[j][q]);
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
    __shared__ double v[kSums][kPer + 1];
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
    const int begin = I.part_begin, n = I.part_end - I.part_begin, stride = I.part_stride;
    const int nx = I.nx;
    double* const macc = I.macc;
    double* const prof = I.prof;
    double* const prof_out = I.prof_out;
    const int n_cta = n > 0 ? (n + kPer - 1) / kPer : 1;
    if (b >= n_cta) return;  // whole CTA, before any barrier or count
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int here = n - b * kPer < kPer ? n - b * kPer : kPer;
    for (int q = t; q < kSums * kPer; q += kThreads) {
        const int j = q / kPer, p = q % kPer;
        if (p < here) {
            const int at = begin + b * kPer + p;
            v[j][p] = j < kObs ? partials[(long long)j * stride + at] : (macc ? macc[at] : 0.0);
        }
    }
    if (prof && prof_out)
        for (int x = b * kThreads + t; x < nx; x += n_cta * kThreads) {
            prof_out[x] = __ldcg(prof + x);
            prof[x] = 0.0;
        }
    __syncthreads();
    double s = sum_staged(v, here, t);
    if (n_cta > 1) {
        // the scratch slots of lattice k: floor(begin / kPer) + k onwards (disjoint
        // across lattices, fewer than max_parts / kPer + n_inst + 1 in all)
        double* const mine = scratch + (long long)(begin / kPer + k) * kSums;
        if (t < kSums * kLanes && t % kLanes == 0) {
            mine[(long long)b * kSums + t / kLanes] = s;
            __threadfence();
        }
        __syncthreads();
        if (t == 0) last = atomicAdd(counts + k, 1u) == (unsigned)(n_cta - 1);
        __syncthreads();
        if (!last) return;
        __threadfence();
        s = 0.0;
        for (int c0 = 0; c0 < n_cta; c0 += kPer) {
            const int nc = n_cta - c0 < kPer ? n_cta - c0 : kPer;
            for (int q = t; q < nc * kSums; q += kThreads)
                v[q % kSums][q / kSums] = __ldcg(mine + (long long)c0 * kSums + q);
            __syncthreads();
            s = combine(t / kLanes, s, sum_staged(v, nc, t));
            __syncthreads();
        }
    }
    if (t < kSums * kLanes && t % kLanes == 0) {
        const int j = t / kLanes;
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
            if (r[LBM_FRZ_FREEZE_STEP] < 0.0 && X >= kFreezeFraction) r[LBM_FRZ_FREEZE_STEP] = (double)step;
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
