// lbm_noalloc.cu -- lbm_step_noalloc: one time step of one lattice without a
// handle and without any device allocation. The observable partials of the
// step live in a fixed array that is part of the library's device image.
#include <mutex>

#include "lbm.h"
#include "lbm_internal.h"

namespace {

constexpr int kMaxDevices = 64;

// Per-tile observable partials of lbm_step_noalloc (720 KiB per device).
static __device__ __align__(256) double g_noalloc_partials[LBM_NOALLOC_MAX_TILES * lbmk::kObs];

std::mutex g_mu;
double* g_scratch[kMaxDevices] = {};
int g_warps[kMaxDevices] = {};  // resident strip warps (0: strips not available)
int g_wave[kMaxDevices] = {};   // resident 32 x 4 tile CTAs

// Device address of the scratch array on the current device, and what of the
// step kernels it holds resident at once. In host code the array's name only
// stands for the symbol, so the address is looked up once per device (with that
// device current) and cached, and so are the other two.
int device_facts(double** out, int* warps, int* wave) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return LBM_ECUDA;
    if (dev < 0 || dev >= kMaxDevices) return LBM_EINVAL;
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_scratch[dev]) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_noalloc_partials) != cudaSuccess || !ptr)
            return LBM_ECUDA;
        g_warps[dev] = lbmk::noalloc_strip_warps();
        g_wave[dev] = lbmk::tile_resident_ctas(LBM_STORE_FP32);
        g_scratch[dev] = static_cast<double*>(ptr);
    }
    *out = g_scratch[dev];
    *warps = g_warps[dev];
    *wave = g_wave[dev];
    return LBM_OK;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// [a, a + na) and [b, b + nb) (bytes) share at least one byte.
bool overlap(const void* a, size_t na, const void* b, size_t nb) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + nb && y < x + na;
}

}  // namespace

extern "C" int lbm_step_noalloc(const lbm_params* p, const float* pops_in, const float* aux_in,
                                float* pops_out, float* aux_out, int32_t pitch, double* d_obs,
                                void* cuda_stream) {
    if (!p || !pops_in || !aux_in || !pops_out || !aux_out || !d_obs) return LBM_EINVAL;
    if (!lbmk::params_valid(*p) || pitch < p->nx || pitch % 32 != 0) return LBM_EINVAL;
    if (!aligned16(pops_in) || !aligned16(aux_in) || !aligned16(pops_out) || !aligned16(aux_out))
        return LBM_EINVAL;
    if ((long long)pitch * p->ny * 27 >= (1LL << 31)) return LBM_EINVAL;
    const int tiles_x = (p->nx + 31) / 32;
    const long long n_tiles = (long long)tiles_x * ((p->ny + 7) / 8);
    if (n_tiles > LBM_NOALLOC_MAX_TILES) return LBM_ETOOLARGE;
    // the step reads neighbouring sites of the input while other CTAs write
    // the output: an output buffer may share no byte with any other buffer
    const size_t plane = (size_t)pitch * (size_t)p->ny;
    const size_t pop_b = plane * lbmk::kPopElems * sizeof(float);
    const size_t aux_b = plane * (lbmk::kAuxBlock / 32) * sizeof(float);
    if (overlap(pops_out, pop_b, pops_in, pop_b) || overlap(pops_out, pop_b, aux_in, aux_b) ||
        overlap(pops_out, pop_b, aux_out, aux_b) || overlap(aux_out, aux_b, pops_in, pop_b) ||
        overlap(aux_out, aux_b, aux_in, aux_b))
        return LBM_EINVAL;
    double* scratch = nullptr;
    int warps = 0, wave = 0;
    int rc = device_facts(&scratch, &warps, &wave);
    if (rc != LBM_OK) return rc;
    lbmk::Inst I;
    double L = 0.0;
    lbmk::inst_from_params(*p, &I, &L);
    I.pitch = pitch;
    I.plane = (long long)pitch * p->ny;
    I.pop[0] = const_cast<float*>(pops_in);
    I.pop[1] = pops_out;
    I.aux[0] = const_cast<float*>(aux_in);
    I.aux[1] = aux_out;
    // Layout as lbm_create chooses it: 32 x 4 tiles while they are two waves or
    // less (four steps: 67 us on 256 x 256 sites, 136 us in the 32 x 8 tiles of
    // before), else strips in one wave where the lattice is periodic in x (512 x
    // 512: 91 us against 172 in tiles), else tiles, 32 x 8 where the shorter ones
    // are more than the LBM_NOALLOC_MAX_TILES slots (closed 512 x 512: 146 us in
    // 32 x 8, 363 before).
    const long long small_tiles = (long long)tiles_x * ((p->ny + 3) / 4);
    const int strips = (p->nx + lbmk::kStripW - 1) / lbmk::kStripW;
    int ty = small_tiles <= LBM_NOALLOC_MAX_TILES ? 4 : 8;
    int parts = (int)(ty == 4 ? small_tiles : n_tiles), rows = 0;
    if (small_tiles > 2 * wave && p->periodic_x && warps > 0) {
        int lo = 2, hi = p->ny;  // fewest rows of one wave (or all, if none is)
        while (lo < hi) {
            const int mid = (lo + hi) / 2;
            if ((long long)strips * ((p->ny + mid - 1) / mid) <= warps) hi = mid; else lo = mid + 1;
        }
        const long long items = (long long)strips * ((p->ny + lo - 1) / lo);
        if (items <= LBM_NOALLOC_MAX_TILES) {
            rows = lo;
            parts = (int)items;
        }
    }
    I.part_begin = 0;
    I.part_end = parts;
    I.part_stride = parts;
    const cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    cudaError_t e = rows ? lbmk::launch_step_noalloc_strip(I, rows, parts, scratch, s)
                         : lbmk::launch_step_noalloc(I, ty, tiles_x, parts, scratch, s);
    if (e == cudaSuccess) e = lbmk::launch_reduce_noalloc(parts, scratch, d_obs, s);
    return e == cudaSuccess ? LBM_OK : LBM_ECUDA;
}
