// lbm_api.cu -- host side of the C-ABI declared in include/lbm.h: parameter
// checks, the workspace layout, tile tables, launches and state transfer.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <functional>
#include <new>
#include <queue>
#include <string>
#include <vector>

#include <cuda_fp16.h>

#include "lbm.h"
#include "lbm_internal.h"
#include "lbm_reduce.h"

using lbmk::Inst;
using lbmk::Item;
using lbmk::Tile;

namespace {

constexpr uint64_t kAlign = 256;
constexpr unsigned long long kBarrierLimitNs = 2000000000ull;  // device-wide barrier wait
constexpr int kMaxChunk = 1 << 16;

// Device-side synchronisation words of a handle (in the workspace).
struct SyncBlock {
    unsigned bar;        // barrier counter of the persistent kernel
    int err;             // raised by a barrier wait that ran out
    unsigned probe_bar;  // the barrier self-test's own pair
    int probe_err;
};

uint64_t align_up(uint64_t v) { return (v + kAlign - 1) / kAlign * kAlign; }
int pitch_of(int nx) { return lbmk::pitch_for(nx); }

bool valid_params(const lbm_params& p) {
    if (p.nx < 3 || p.ny < 3) return false;
    if ((p.periodic_x != 0 && p.periodic_x != 1) || (p.periodic_y != 0 && p.periodic_y != 1)) return false;
    if ((long long)pitch_of(p.nx) * p.ny * 27 >= (1LL << 31)) return false;  // 32-bit plane offsets
    if (!(p.W > 0) || !(p.sigma >= 0) || !(p.mobility > 0)) return false;
    if (!(p.tau_f_liquid > 0.5) || !(p.tau_h > 0.5)) return false;
    if (!(p.rho_l > 0) || !(p.rho_ratio_lg > 0) || !(p.rho_ratio_sl > 0)) return false;
    if (!(p.mu_ratio_lg > 0) || !(p.Ste > 0) || !(p.Cp > 0) || !(p.Cp_ref > 0)) return false;
    if (!(p.T_w < p.T_m)) return false;
    if (!(p.theta_deg > 0 && p.theta_deg < 180)) return false;
    if (!(p.pc_ramp > 0)) return false;
    if (!(p.normal_eps > 0) || !isfinite(p.normal_eps)) return false;
    if (!isfinite(p.T_m) || !isfinite(p.T_w) || !isfinite(p.sigma)) return false;
    if (!isfinite(p.gx) || !isfinite(p.gy) || !isfinite(p.beta_T) || !isfinite(p.T_ref) ||
        !isfinite(p.rho_0))
        return false;
    if (!(p.Cp_ratio_sl > 0) || !(p.Cp_ratio_gl > 0) || !(p.k_ratio_sl > 0) ||
        !(p.k_ratio_gl > 0) || !isfinite(p.Cp_ratio_sl) || !isfinite(p.Cp_ratio_gl) ||
        !isfinite(p.k_ratio_sl) || !isfinite(p.k_ratio_gl))
        return false;
    return true;
}

int elem_size(int storage) { return storage == LBM_STORE_FP32 ? 4 : 2; }
using lbmk::aux_at;
using lbmk::own0_at;
using lbmk::pop_at;
// own-site region, floats per site: (g_0, h_0, f_0, f_l), ((phi u)_x,
// (phi u)_y, p, S) and (phi_ref, T_ref), the last used by 16-bit storage only
// (every storage keeps the same block size, lbmk::kAuxBlock)
int aux_planes(int /*storage*/) { return lbmk::kAuxBlock / 32; }

// D2Q9 directions and weights of the host-side state conversion (Eqs. 22-23)
const int kCx[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1};
const int kCy[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
const float kWf[9] = {0x1.c71c72p-2f, 0x1.c71c72p-4f, 0x1.c71c72p-4f, 0x1.c71c72p-4f,
                      0x1.c71c72p-4f, 0x1.c71c70p-6f, 0x1.c71c70p-6f, 0x1.c71c70p-6f,
                      0x1.c71c70p-6f};

// Site a population of (x, y) streams into along c_i (the site itself when
// the link ends behind a wall).
size_t dest_site(const lbm_params& p, int x, int y, int i) {
    int xd = x + kCx[i], yd = y + kCy[i];
    bool wall = false;
    if (xd < 0 || xd >= p.nx) { if (p.periodic_x) xd = (xd + p.nx) % p.nx; else wall = true; }
    if (yd < 0 || yd >= p.ny) { if (p.periodic_y) yd = (yd + p.ny) % p.ny; else wall = true; }
    return wall ? (size_t)y * p.nx + x : (size_t)yd * p.nx + xd;
}

struct Layout {
    uint64_t inst_off, tile_off, item_off, part_off, obs_off, stage_off, sync_off;
    uint64_t macc_off, frz_off, prof_off, prof_out_off, prof_bytes, red_off, cnt_off, cnt_end;
    std::vector<uint64_t> prof_at;  // doubles from prof_off (prof_out_off) to each lattice's profile
    std::vector<uint64_t> pop_off[2], aux_off[2];
    uint64_t total;
    int max_tiles, max_items, max_parts, max_sites;
};

int max_tiles_of(const lbm_params& p) {
    // tiles of the smallest supported shape (32 x 4)
    return ((p.nx + 31) / 32) * ((p.ny + 3) / 4);
}

// Default tile. Against 32 x 8 the shorter block spreads a small lattice over
// twice the SMs: 2.7 us against 3.2 us a step on 256 x 8 sites, 3.6 against 4.1
// on 203 x 151, 13.8 against 14.7 on 500 x 500.
constexpr int kTileX = 32, kTileY = 4;
constexpr int kMinRows = 2;  // shortest strip segment
int max_items_of(const lbm_params& p) {
    return ((p.nx + lbmk::kStripW - 1) / lbmk::kStripW) * ((p.ny + kMinRows - 1) / kMinRows);
}

Layout make_layout(const lbm_params* p, int n, int storage) {
    Layout L;
    uint64_t off = 0;
    L.max_tiles = 0;
    L.max_items = 0;
    L.max_sites = 0;
    for (int k = 0; k < n; ++k) {
        L.max_tiles += max_tiles_of(p[k]);
        if (p[k].periodic_x) L.max_items += max_items_of(p[k]);
        L.max_sites = std::max(L.max_sites, p[k].nx * p[k].ny);
    }
    L.max_parts = std::max(L.max_tiles, L.max_items);
    L.inst_off = off; off = align_up(off + sizeof(Inst) * (uint64_t)n);
    L.tile_off = off; off = align_up(off + sizeof(Tile) * (uint64_t)L.max_tiles);
    L.item_off = off; off = align_up(off + sizeof(Item) * (uint64_t)std::max(L.max_items, 1));
    L.part_off = off; off = align_up(off + sizeof(double) * lbmk::kObs * (uint64_t)L.max_parts);
    L.obs_off = off;  off = align_up(off + sizeof(double) * lbmk::kObs * (uint64_t)n);
    L.stage_off = off; off = align_up(off + sizeof(double) * 2 * (uint64_t)L.max_sites);
    L.sync_off = off; off = align_up(off + sizeof(SyncBlock));
    // running mdot sums (one per partial slot), freezing records, column profiles
    L.macc_off = off; off = align_up(off + sizeof(double) * (uint64_t)L.max_parts);
    L.frz_off = off;  off = align_up(off + sizeof(double) * lbmk::kFrz * (uint64_t)n);
    L.prof_at.resize(n);
    uint64_t prof_n = 0;
    for (int k = 0; k < n; ++k) { L.prof_at[k] = prof_n; prof_n += (uint64_t)p[k].nx; }
    L.prof_bytes = sizeof(double) * prof_n;
    L.prof_off = off; off = align_up(off + L.prof_bytes);
    L.prof_out_off = off; off = align_up(off + L.prof_bytes);
    // the observable reduction's per-CTA sums and per-lattice arrival counts
    L.red_off = off;
    off = align_up(off + sizeof(double) * (lbmk::kObs + 1) *
                             (uint64_t)lbmk::reduce_slots(L.max_parts, n));
    L.cnt_off = off; L.cnt_end = off + sizeof(unsigned) * (uint64_t)n; off = align_up(L.cnt_end);
    for (int b = 0; b < 2; ++b) {
        L.pop_off[b].resize(n);
        L.aux_off[b].resize(n);
    }
    for (int k = 0; k < n; ++k) {
        const uint64_t plane = (uint64_t)pitch_of(p[k].nx) * p[k].ny;
        for (int b = 0; b < 2; ++b) {
            L.pop_off[b][k] = off; off = align_up(off + plane * lbmk::kPopElems * elem_size(storage));
            L.aux_off[b][k] = off; off = align_up(off + plane * aux_planes(storage) * sizeof(float));
        }
    }
    L.total = off;
    return L;
}

}  // namespace

struct lbm_handle {
    std::vector<lbm_params> params;
    int n_inst = 0;
    int storage = 0;
    int kind = LBM_KERNEL_TILE;
    int tx = kTileX, ty = kTileY;        // tile shape
    bool chosen = true;                  // the layout is still the one lbm_create chose
    bool small = false;                  // all lattices together: two waves of tiles at most
    bool tables_ok = false;              // host and device tables are those of the layout
    int warps = 4, rows = 16, regs = 168; // strip layouts (rows: effective)
    int rows_req = 16;                    // requested rows per item, 0 = one wave
    std::vector<Item> items;
    Item* d_items = nullptr;
    cudaStream_t stream = nullptr;
    char* ws = nullptr;
    Layout layout;
    std::vector<Inst> inst;
    std::vector<Tile> tiles;
    Inst* d_inst = nullptr;
    Tile* d_tiles = nullptr;
    double* d_part = nullptr;
    double* d_obs = nullptr;
    double* h_obs = nullptr;   // pinned host mirror of d_obs (null: copy to the caller directly)
    double* d_obs_map = nullptr;  // h_obs as the device sees it when mapped: the reduction
                                  // writes the records there too (no copy per read)
    double* d_stage = nullptr;
    double* d_macc = nullptr;  // running mdot sum per partial slot
    double* d_frz = nullptr;   // freezing records (kFrz doubles per lattice)
    double* d_prof = nullptr;  // column profiles of f_s being summed (nx doubles per lattice)
    double* d_prof_out = nullptr;  // the profiles of the last observable step
    double* d_red = nullptr;   // per-CTA sums of the observable reduction
    unsigned* d_cnt = nullptr; // its per-lattice arrival counts
    int max_lattice_parts = 0; // most observable partials of one lattice
    double* h_frz = nullptr;   // pinned mirror of d_frz
    std::vector<double> mdot_base;  // mdot summed out of retired slot tables, per lattice
    std::vector<double> frz_base;   // mdot_base as of the last observable step
    std::vector<int64_t> step0;     // clock when each lattice was (re)started
    int64_t clock = 0;              // steps taken by the handle, never reset
    int parity = 0;
    int64_t steps = 0;
    int64_t launches = 0;
    bool initialised = false;
    bool have_obs = false;
    std::vector<double> init_L;  // double L per instance (state conversion)
    // execution form of lbm_step
    int exec = LBM_EXEC_LAUNCH;
    int chunk = 64;
    int persist_grid = 0;              // CTAs of one persistent launch
    SyncBlock* d_sync = nullptr;
    bool persist_pending = false;      // a persistent launch ran since the last check
    bool failed = false;               // a barrier wait ran out: state is not usable
    cudaStream_t cap_stream = nullptr; // private stream for graph capture
    cudaGraphExec_t graph[2] = {nullptr, nullptr};  // `chunk` steps from parity 0 / 1
    ~lbm_handle() {
        if (h_obs) cudaFreeHost(h_obs);
        if (h_frz) cudaFreeHost(h_frz);
    }
};

namespace {

// Code of a failed call. The error is reported here: cleared, so that the check
// after a later launch does not find it.
int cuda_fail(cudaError_t e) {
    (void)e;
    cudaGetLastError();
    return LBM_ECUDA;
}

void fill_inst(lbm_handle* h, int k) {
    const lbm_params& p = h->params[k];
    Inst I;
    double L = 0.0;
    lbmk::inst_from_params(p, &I, &L);
    I.part_stride = h->layout.max_parts;
    I.macc = h->d_macc;
    I.prof = h->d_prof + h->layout.prof_at[k];
    I.prof_out = h->d_prof_out + h->layout.prof_at[k];
    for (int b = 0; b < 2; ++b) {
        I.pop[b] = h->ws + h->layout.pop_off[b][k];
        I.aux[b] = reinterpret_cast<float*>(h->ws + h->layout.aux_off[b][k]);
    }
    h->inst[k] = I;
    h->init_L[k] = L;
}

void build_tiles(lbm_handle* h) {
    h->tiles.clear();
    for (int k = 0; k < h->n_inst; ++k) {
        const lbm_params& p = h->params[k];
        h->inst[k].part_begin = (int)h->tiles.size();
        for (int y0 = 0; y0 < p.ny; y0 += h->ty)
            for (int x0 = 0; x0 < p.nx; x0 += h->tx) {
                Tile t;
                t.inst = k;
                t.x0 = x0;
                t.y0 = y0;
                t.tw = std::min(h->tx, p.nx - x0);
                t.th = std::min(h->ty, p.ny - y0);
                t.part = (int)h->tiles.size();
                h->tiles.push_back(t);
            }
        h->inst[k].part_end = (int)h->tiles.size();
    }
}

// Strip items ordered by (lattice, row segment, strip) so that warps that run
// together touch neighbouring columns of the same rows.
bool is_strip(int kind) {
    return kind == LBM_KERNEL_STRIP || kind == LBM_KERNEL_STAGED || kind == LBM_KERNEL_BLOCK;
}
// Whether the steps of a handle run in tiles: the tile layout, or the layout
// lbm_create chose for lattices that are at most two waves of tile CTAs (one
// thread per site; 155,648 sites on 152 SMs). There a step is one chain of
// latencies, and a strip item's is some rows longer than a tile's. A plain step
// in tiles and in strips, us: 2.7 and 7.7 on 128 x 128 sites, 4.1 and 7.9 on
// 256 x 256, 6.8 and 8.7 on 320 x 320, 8.1 and 10.3 on 384 x 384; in 16-bit
// storage 2.9 and 10.0, 4.2 and 10.0, 7.4 and 10.9, 8.7 and 15.5. A call of one
// step with its observables: 13.1 and 16.0 on 256 x 256, 16.9 and 16.5 on 320 x
// 320, 20.4 and 18.9 on 384 x 384 (16-bit 13.5 and 17.7, 18.5 and 18.4, 19.8
// and 22.1). Beyond, the strips are level: 9.6 and 11.5 a plain step on 400 x
// 400 but 26.4 and 24.3 with the observables read, 13.4 and 14.6 on 512 x 512,
// 23.3 and 18.1 on 620 x 620. The persistent form stays with the strips.
bool tiled(const lbm_handle* h) {
    return h->kind == LBM_KERNEL_TILE ||
           (h->chosen && h->small && h->exec != LBM_EXEC_PERSISTENT);
}

// Output columns of one item of a strip-like layout.
int item_width(int kind) { return kind == LBM_KERNEL_BLOCK ? lbmk::kBlockW : lbmk::kStripW; }

// Number of strip items of every lattice at `rows` rows an item.
int items_at(const lbm_handle* h, int rows) {
    const int wd = item_width(h->kind);
    int n = 0;
    for (const auto& p : h->params)
        n += ((p.nx + wd - 1) / wd) * ((p.ny + rows - 1) / rows);
    return n;
}

// Estimated time of a step at `rows` rows an item, in rows of a fully occupied
// device: the CTAs (h->warps items each, in table order) go to the first free
// of `slots` places; a CTA takes its longest item's rows and kItemCost rows for
// the two rows beyond it and its start, and while only a fraction f of the
// places is taken each CTA runs at 1 / (kTailA + kTailB f) of the full
// device's pace at most. Fitted to measured steps of 15 sets of lattices (one of
// 300 x 300 to 2501 x 2501, 8 to 256 of mixed sizes) at 4 to 12 row counts
// each: the choice below is within 1 % of the fastest but for 500 x 500 in FP16
// storage (11 %).
constexpr double kItemCost = 1.0, kTailA = 0.4, kTailB = 0.6;
double step_estimate(const lbm_handle* h, int rows, int slots) {
    const int wd = item_width(h->kind);
    // ends of running CTAs, equal ones together (with one entry a CTA
    // lbm_create of 48 unequal lattices took 0.95 ms, this way 0.70)
    struct Group { double end; int n; };
    auto later = [](const Group& a, const Group& b) { return a.end > b.end; };
    std::priority_queue<Group, std::vector<Group>, decltype(later)> ends(later);
    double start = 0.0;
    int taken = 0, run = 0, run_rows = 0;
    auto place = [&]() {  // `run` CTAs of run_rows rows
        while (run > 0) {
            Group g{0.0, slots - taken};
            if (g.n == 0) {
                g = ends.top();
                ends.pop();
                start = g.end;
            }
            const int k = std::min(run, g.n);
            if (taken == slots && g.n > k) ends.push({g.end, g.n - k});
            if (taken < slots) taken += k;
            ends.push({g.end + run_rows + kItemCost, k});
            run -= k;
        }
    };
    int in_cta = 0, longest = 0;
    auto flush = [&]() {
        if (longest != run_rows) {
            place();
            run_rows = longest;
        }
        ++run;
        in_cta = longest = 0;
    };
    for (const auto& p : h->params) {
        const int strips = (p.nx + wd - 1) / wd;
        for (int y0 = 0; y0 < p.ny; y0 += rows) {
            const int height = std::min(rows, p.ny - y0);
            for (int left = strips; left > 0;) {
                const int k = std::min(left, h->warps - in_cta);
                longest = std::max(longest, height);
                in_cta += k;
                left -= k;
                if (in_cta == h->warps) flush();
            }
        }
    }
    if (in_cta) flush();
    place();
    double t = start, at = start;  // full until the last CTA starts
    for (; !ends.empty(); ends.pop()) {
        const double f = (double)taken / slots;
        t += (ends.top().end - at) * std::min(1.0, kTailA + kTailB * f);
        at = ends.top().end;
        taken -= ends.top().n;
    }
    return t;
}

// Rows per strip item: as requested, or (0) the count with the shortest
// estimated step among those that fill 1, 2, 3, 4, 6 or 8 waves of resident
// warps (for one wave also one and two rows more or less). A single large
// lattice is fastest in one wave; many lattices are not, as their last segments
// are short (48 drops on 128 .. 512 squared: 341 us a step in one wave, 213 us
// at 32 rows; 256 drops in FP16 storage on 64 .. 256: 449 us and 298 us at 20
// rows; 64 drops: 118 us and 87 us at 18), nor is one whose rounding leaves a
// few items for a second wave (2501 x 2501: 267 us at 116 rows, 254 us at 118).
int item_rows(const lbm_handle* h) {
    if (h->rows_req > 0) return h->rows_req;
    int max_ny = kMinRows;
    for (const auto& p : h->params) max_ny = std::max(max_ny, p.ny);
    const int warps = h->kind == LBM_KERNEL_BLOCK
                          ? lbmk::block_resident_warps(h->warps, h->regs, h->storage)
                          : lbmk::strip_resident_warps(h->kind == LBM_KERNEL_STAGED, h->warps,
                                                       h->regs, h->storage);
    if (warps <= 0) return 16;
    const int slots = std::max(1, warps / h->warps);
    int best = 0, last = 0;
    double best_t = 0.0;
    for (const int waves : {1, 2, 3, 4, 6, 8}) {
        int lo = kMinRows, hi = max_ny;  // fewest rows with at most `waves` waves of items
        while (lo < hi) {
            const int mid = (lo + hi) / 2;
            if (items_at(h, mid) <= waves * warps) hi = mid; else lo = mid + 1;
        }
        // (just below one wave, the few items too many may be short ones)
        const bool one = waves == 1;
        for (int r = one ? std::max(kMinRows, lo - 2) : lo; r <= (one ? std::min(lo + 2, max_ny) : lo); ++r) {
            if (!one && r >= last) break;  // tried with fewer waves
            const double t = step_estimate(h, r, slots);
            if (best == 0 || t < best_t) { best = r; best_t = t; }
        }
        last = last ? std::min(last, lo) : lo;
        // one lattice: always the first (and lbm_create stays short)
        if (lo == kMinRows || h->n_inst == 1) break;
    }
    return best;
}

void build_items(lbm_handle* h) {
    h->items.clear();
    for (int k = 0; k < h->n_inst; ++k) {
        const lbm_params& p = h->params[k];
        h->inst[k].part_begin = (int)h->items.size();
        for (int y0 = 0; y0 < p.ny; y0 += h->rows)
            for (int x0 = 0; x0 < p.nx; x0 += item_width(h->kind)) {
                Item it;
                memset(&it, 0, sizeof(it));
                it.inst = k;
                it.x0 = x0;
                it.y0 = y0;
                it.y1 = std::min(y0 + h->rows, p.ny);
                it.part = (int)h->items.size();
                h->items.push_back(it);
            }
        h->inst[k].part_end = (int)h->items.size();
    }
}

void drop_graphs(lbm_handle* h) {
    for (auto& g : h->graph) {
        if (g) cudaGraphExecDestroy(g);
        g = nullptr;
    }
}

// The running mdot sums live in the slots of the current tile or item table;
// before the table is rebuilt they are summed per lattice (in slot order, in
// FP64) into mdot_base and the slots are cleared.
int fold_mdot(lbm_handle* h) {
    if (!h->initialised) return LBM_OK;
    int n_parts = 0;
    for (int k = 0; k < h->n_inst; ++k) n_parts = std::max(n_parts, h->inst[k].part_end);
    if (n_parts <= 0) return LBM_OK;
    std::vector<double> v((size_t)n_parts);
    cudaError_t e = cudaMemcpyAsync(v.data(), h->d_macc, v.size() * sizeof(double),
                                    cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->d_macc, 0, v.size() * sizeof(double), h->stream);
    if (e != cudaSuccess) return cuda_fail(e);
    for (int k = 0; k < h->n_inst; ++k) {
        double sum = 0.0;
        for (int q = h->inst[k].part_begin; q < h->inst[k].part_end; ++q) sum += v[(size_t)q];
        h->mdot_base[k] += sum;
    }
    return LBM_OK;
}

// A lattice starts a new run (lbm_init_fields, lbm_set_state): its running
// mdot sums, profile and freezing record restart.
int restart_records(lbm_handle* h, int k) {
    const Inst& I = h->inst[k];
    cudaError_t e = cudaSuccess;
    if (I.part_end > I.part_begin)
        e = cudaMemsetAsync(h->d_macc + I.part_begin, 0,
                            sizeof(double) * (size_t)(I.part_end - I.part_begin), h->stream);
    if (e == cudaSuccess)  // an accumulator left by a failed call starts clean
        e = cudaMemsetAsync(h->d_prof + h->layout.prof_at[k], 0,
                            sizeof(double) * (size_t)h->params[k].nx, h->stream);
    const double rec[lbmk::kFrz] = {0.0, 0.0, -1.0, 0.0};
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(h->d_frz + (size_t)k * lbmk::kFrz, rec, sizeof(rec),
                            cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);  // rec is on this stack
    if (e != cudaSuccess) return cuda_fail(e);
    h->mdot_base[k] = 0.0;
    h->frz_base[k] = 0.0;
    h->step0[k] = h->clock;
    return LBM_OK;
}

// (a failure leaves tables_ok down, and the next step rebuilds them first)
int upload_tables(lbm_handle* h) {
    h->tables_ok = false;
    drop_graphs(h);  // captured launches carry the old item counts
    {
        const int rc = fold_mdot(h);
        if (rc != LBM_OK) return rc;
    }
    if (h->kind == LBM_KERNEL_STAGED) {
        cudaError_t e = lbmk::prepare_staged(h->warps, h->regs, h->storage);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    if (h->kind == LBM_KERNEL_BLOCK) {
        cudaError_t e = lbmk::prepare_block(h->warps, h->regs, h->storage);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    if (is_strip(h->kind)) h->rows = item_rows(h);
    if (tiled(h)) build_tiles(h); else build_items(h);
    h->max_lattice_parts = 0;
    for (int k = 0; k < h->n_inst; ++k)
        h->max_lattice_parts =
            std::max(h->max_lattice_parts, h->inst[k].part_end - h->inst[k].part_begin);
    cudaError_t e = cudaMemcpyAsync(h->d_inst, h->inst.data(), sizeof(Inst) * h->n_inst,
                                    cudaMemcpyHostToDevice, h->stream);
    if (e != cudaSuccess) return cuda_fail(e);
    if (!tiled(h))
        e = cudaMemcpyAsync(h->d_items, h->items.data(), sizeof(Item) * h->items.size(),
                            cudaMemcpyHostToDevice, h->stream);
    else
        e = cudaMemcpyAsync(h->d_tiles, h->tiles.data(), sizeof(Tile) * h->tiles.size(),
                            cudaMemcpyHostToDevice, h->stream);
    if (e != cudaSuccess) return cuda_fail(e);
    e = cudaStreamSynchronize(h->stream);  // host tables may change after return
    if (e != cudaSuccess) return cuda_fail(e);
    h->persist_grid = h->kind == LBM_KERNEL_BLOCK
                          ? lbmk::block_persistent_grid(h->warps, h->regs, h->storage,
                                                        items_at(h, h->rows))
                          : (is_strip(h->kind)
                                 ? lbmk::persistent_grid(h->kind == LBM_KERNEL_STAGED, h->warps,
                                                         h->regs, h->storage, items_at(h, h->rows))
                                 : 0);
    h->tables_ok = true;
    return LBM_OK;
}

// One time step through the ordinary kernels (obs != 0: with observable partials).
cudaError_t enqueue_step(lbm_handle* h, int parity, int obs, cudaStream_t s) {
    if (tiled(h))
        return lbmk::launch_step(h->tx, h->ty, h->storage, h->d_inst, h->d_tiles,
                                 (int)h->tiles.size(), parity, obs, h->d_part, s);
    if (h->kind == LBM_KERNEL_BLOCK)
        return lbmk::launch_step_block(h->warps, h->regs, h->storage, h->d_inst, h->d_items,
                                       (int)h->items.size(), parity, obs, h->d_part,
                                       &h->d_sync->err, s);
    if (h->kind == LBM_KERNEL_STAGED)
        return lbmk::launch_step_staged(h->warps, h->regs, h->storage, h->d_inst, h->d_items,
                                        (int)h->items.size(), parity, obs, h->d_part, s);
    return lbmk::launch_step_strip(h->warps, h->regs, h->storage, h->d_inst, h->d_items,
                                   (int)h->items.size(), parity, obs, h->d_part, s);
}

// n steps without observables from `parity` as one persistent launch.
cudaError_t enqueue_persistent(lbm_handle* h, int parity, int n, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(&h->d_sync->bar, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    if (h->kind == LBM_KERNEL_BLOCK)
        return lbmk::launch_step_block_persistent(h->warps, h->regs, h->storage, h->persist_grid,
                                                  h->d_inst, h->d_items, (int)h->items.size(),
                                                  parity, n, &h->d_sync->bar, &h->d_sync->err,
                                                  kBarrierLimitNs, s);
    return lbmk::launch_step_strip_persistent(h->kind == LBM_KERNEL_STAGED, h->warps, h->regs,
                                              h->storage, h->persist_grid,
                                              h->d_inst, h->d_items, (int)h->items.size(),
                                              parity, n, &h->d_sync->bar, &h->d_sync->err,
                                              kBarrierLimitNs, s);
}

// Capture `chunk` steps from `parity` (one launch per step, or one persistent
// launch) into an executable graph on the handle's private stream.
int capture_chunk(lbm_handle* h, int parity, cudaGraphExec_t* out) {
    if (!h->cap_stream) {
        cudaError_t e = cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) { h->cap_stream = nullptr; return cuda_fail(e); }
    }
    cudaError_t e = cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_fail(e);
    cudaError_t ee = cudaSuccess;
    if (h->exec == LBM_EXEC_PERSISTENT) {
        ee = enqueue_persistent(h, parity, h->chunk, h->cap_stream);
    } else {
        for (int k = 0; k < h->chunk && ee == cudaSuccess; ++k)
            ee = enqueue_step(h, parity ^ (k & 1), 0, h->cap_stream);
    }
    cudaGraph_t g = nullptr;
    e = cudaStreamEndCapture(h->cap_stream, &g);  // always ends the capture
    if (ee == cudaSuccess) ee = e;
    if (ee == cudaSuccess) ee = cudaGraphInstantiate(out, g, 0);
    if (g) cudaGraphDestroy(g);
    return ee == cudaSuccess ? LBM_OK : cuda_fail(ee);
}

// Launches of our kernels that one enqueued unit of n steps amounts to.
int64_t kernels_per(const lbm_handle* h, int64_t n) {
    return h->exec == LBM_EXEC_PERSISTENT ? 1 : n;
}

bool inst_ok(const lbm_handle* h, int32_t inst) { return h && inst >= 0 && inst < h->n_inst; }

// Synchronise the handle's stream; after persistent launches also read the
// barrier error word (h->failed is raised when a wait ran out).
cudaError_t sync_checked(lbm_handle* h) {
    static thread_local int err_host = 0;
    cudaError_t e = cudaSuccess;
    const bool check = h->persist_pending;
    if (check) e = cudaMemcpyAsync(&err_host, &h->d_sync->err, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return e;
    if (check) {
        h->persist_pending = false;
        if (err_host != 0) h->failed = true;
    }
    return cudaSuccess;
}

// A record reports an unstable step: a non-finite field, or a speed above
// 0.5 (NaN compares false, so a NaN maximum is caught by the count).
constexpr double kMaxSpeed = 0.5;
bool unstable(const double* rec) {
    return rec[LBM_OBS_NONFINITE] > 0 || rec[LBM_OBS_UMAX] > kMaxSpeed;
}

// n doubles of the observable records from offset off to the caller's out:
// when the mirror is mapped, the reduction has written it and a synchronising
// check suffices; otherwise a copy into the pinned mirror (a copy straight
// into pageable memory would be staged by the CUDA runtime with an extra
// synchronisation), then the check.
cudaError_t read_obs(lbm_handle* h, size_t off, size_t n, double* out) {
    if (h->d_obs_map) {  // the reduction wrote the records into host memory itself
        cudaError_t e = sync_checked(h);
        if (e == cudaSuccess) memcpy(out, h->h_obs + off, n * sizeof(double));
        return e;
    }
    double* dst = h->h_obs ? h->h_obs + off : out;
    cudaError_t e = cudaMemcpyAsync(dst, h->d_obs + off, n * sizeof(double), cudaMemcpyDeviceToHost,
                                    h->stream);
    if (e == cudaSuccess) e = sync_checked(h);
    if (e == cudaSuccess && h->h_obs) memcpy(out, dst, n * sizeof(double));
    return e;
}

}  // namespace

extern "C" {

int lbm_workspace_size(const lbm_params* p, int32_t n_inst, int32_t storage, uint64_t* bytes) {
    if (!p || !bytes || n_inst < 1) return LBM_EINVAL;
    if (storage != LBM_STORE_FP32 && storage != LBM_STORE_FP16 && storage != LBM_STORE_BF16)
        return LBM_EINVAL;
    for (int k = 0; k < n_inst; ++k) {
        if (!valid_params(p[k])) return LBM_EINVAL;
        // 16-bit storage runs in the strip layout, which needs periodic x
        if (storage != LBM_STORE_FP32 && !p[k].periodic_x) return LBM_EINVAL;
    }
    *bytes = make_layout(p, n_inst, storage).total;
    return LBM_OK;
}

int lbm_create(const lbm_params* p, int32_t n_inst, int32_t storage, void* d_workspace,
               uint64_t workspace_bytes, void* cuda_stream, lbm_handle** out) {
    if (!out) return LBM_EINVAL;
    *out = nullptr;
    uint64_t need = 0;
    int rc = lbm_workspace_size(p, n_inst, storage, &need);
    if (rc != LBM_OK) return rc;
    if (!d_workspace || ((uintptr_t)d_workspace % kAlign) != 0) return LBM_EINVAL;
    if (workspace_bytes < need) return LBM_ENOMEM;
    lbm_handle* h = new (std::nothrow) lbm_handle();
    if (!h) return LBM_ENOMEM;
    h->params.assign(p, p + n_inst);
    h->n_inst = n_inst;
    h->storage = storage;
    h->stream = static_cast<cudaStream_t>(cuda_stream);
    h->ws = static_cast<char*>(d_workspace);
    h->layout = make_layout(p, n_inst, storage);
    h->inst.resize(n_inst);
    h->init_L.resize(n_inst);
    h->d_inst = reinterpret_cast<Inst*>(h->ws + h->layout.inst_off);
    h->d_tiles = reinterpret_cast<Tile*>(h->ws + h->layout.tile_off);
    h->d_items = reinterpret_cast<Item*>(h->ws + h->layout.item_off);
    h->d_part = reinterpret_cast<double*>(h->ws + h->layout.part_off);
    h->d_obs = reinterpret_cast<double*>(h->ws + h->layout.obs_off);
    h->d_stage = reinterpret_cast<double*>(h->ws + h->layout.stage_off);
    h->d_sync = reinterpret_cast<SyncBlock*>(h->ws + h->layout.sync_off);
    h->d_macc = reinterpret_cast<double*>(h->ws + h->layout.macc_off);
    h->d_frz = reinterpret_cast<double*>(h->ws + h->layout.frz_off);
    h->d_prof = reinterpret_cast<double*>(h->ws + h->layout.prof_off);
    h->d_prof_out = reinterpret_cast<double*>(h->ws + h->layout.prof_out_off);
    h->d_red = reinterpret_cast<double*>(h->ws + h->layout.red_off);
    h->d_cnt = reinterpret_cast<unsigned*>(h->ws + h->layout.cnt_off);
    h->mdot_base.assign(n_inst, 0.0);
    h->frz_base.assign(n_inst, 0.0);
    h->step0.assign(n_inst, 0);
    if (cudaMallocHost(&h->h_frz, sizeof(double) * lbmk::kFrz * n_inst) != cudaSuccess) {
        h->h_frz = nullptr;  // the records are then copied to the caller's memory directly
        cudaGetLastError();
    }
    if (cudaHostAlloc(&h->h_obs, sizeof(double) * lbmk::kObs * n_inst, cudaHostAllocMapped) ==
        cudaSuccess) {
        if (cudaHostGetDevicePointer(reinterpret_cast<void**>(&h->d_obs_map), h->h_obs, 0) !=
            cudaSuccess) {
            h->d_obs_map = nullptr;  // copied per read instead
            cudaGetLastError();
        }
    } else if (cudaMallocHost(&h->h_obs, sizeof(double) * lbmk::kObs * n_inst) != cudaSuccess) {
        h->h_obs = nullptr;  // the observables are then copied to the caller's memory directly
        cudaGetLastError();
    }
    if (cudaMemsetAsync(h->d_sync, 0, sizeof(SyncBlock), h->stream) != cudaSuccess ||
        cudaMemsetAsync(h->d_macc, 0, h->layout.cnt_end - h->layout.macc_off, h->stream) != cudaSuccess) {
        delete h;
        return LBM_ECUDA;
    }
    for (int k = 0; k < n_inst; ++k) fill_inst(h, k);
    bool all_px = true;
    for (int k = 0; k < n_inst; ++k) all_px = all_px && p[k].periodic_x;
    // row-staged strips, one wave of items; small lattices run in tiles
    h->kind = all_px ? LBM_KERNEL_STAGED : LBM_KERNEL_TILE;
    h->rows_req = 0;
    long long n_tiles = 0;
    for (int k = 0; k < n_inst; ++k)
        n_tiles += (long long)((p[k].nx + kTileX - 1) / kTileX) * ((p[k].ny + kTileY - 1) / kTileY);
    h->small = n_tiles <= 2 * lbmk::tile_resident_ctas(storage);
    rc = upload_tables(h);
    if (rc != LBM_OK) {
        delete h;
        return rc;
    }
    *out = h;
    return LBM_OK;
}

int lbm_init_fields(lbm_handle* h, int32_t inst, const double* phi0, const double* T0) {
    if (!inst_ok(h, inst) || !phi0 || !T0) return LBM_EINVAL;
    const lbm_params& p = h->params[inst];
    const size_t n = (size_t)p.nx * p.ny;
    cudaError_t e = cudaMemcpyAsync(h->d_stage, phi0, n * sizeof(double), cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(h->d_stage + h->layout.max_sites, T0, n * sizeof(double),
                            cudaMemcpyHostToDevice, h->stream);
    if (e != cudaSuccess) return cuda_fail(e);
    lbmk::InitConst c;
    c.L = h->init_L[inst];
    c.Hs = p.Cp * p.T_m;
    c.Hl = p.Cp * p.T_m + c.L;
    c.Tm = p.T_m;
    c.Cp = p.Cp;
    c.Cpref = p.Cp_ref;
    c.inv_ramp = 1.0 / p.pc_ramp;
    c.Cp_s = p.Cp * p.Cp_ratio_sl;
    c.Cp_g = p.Cp * p.Cp_ratio_gl;
    e = lbmk::launch_init(h->d_inst, inst, (int)n, h->storage, c, h->d_stage,
                          h->d_stage + h->layout.max_sites, h->parity, h->stream);
    h->launches++;
    if (e != cudaSuccess) return cuda_fail(e);
    // the staging area is reused by the next call: finish the copies first
    e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return cuda_fail(e);
    h->initialised = true;
    h->have_obs = false;
    if (inst == 0) h->steps = 0;
    {
        const int rc = restart_records(h, inst);
        if (rc != LBM_OK) return rc;
    }
    if (h->failed) {  // a fresh state clears an expired barrier wait
        e = cudaMemsetAsync(&h->d_sync->err, 0, sizeof(int), h->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
        if (e != cudaSuccess) return cuda_fail(e);
        h->failed = false;
    }
    return LBM_OK;
}

int lbm_step(lbm_handle* h, int64_t n) {
    if (!h || n < 0) return LBM_EINVAL;
    if (!h->initialised) return LBM_ESTATE;
    if (h->failed) return LBM_ETIMEOUT;
    if (!h->tables_ok) {
        const int rc = upload_tables(h);
        if (rc != LBM_OK) return rc;
    }
    h->clock += n;
    if (h->kind == LBM_KERNEL_BLOCK && n > 0) h->persist_pending = true;  // its error word too
    // every step but the last runs without observables, in the handle's form
    int64_t body = n > 0 ? n - 1 : 0;
    if (h->exec != LBM_EXEC_LAUNCH) {
        while (body >= h->chunk) {
            cudaGraphExec_t& g = h->graph[h->parity];
            if (!g) {
                const int rc = capture_chunk(h, h->parity, &g);
                if (rc != LBM_OK) return rc;
            }
            cudaError_t e = cudaGraphLaunch(g, h->stream);
            if (e != cudaSuccess) return cuda_fail(e);
            h->launches += kernels_per(h, h->chunk);
            h->persist_pending |= h->exec == LBM_EXEC_PERSISTENT;
            h->parity ^= h->chunk & 1;
            h->steps += h->chunk;
            body -= h->chunk;
        }
        if (body > 0 && h->exec == LBM_EXEC_PERSISTENT) {
            cudaError_t e = enqueue_persistent(h, h->parity, (int)body, h->stream);
            if (e != cudaSuccess) return cuda_fail(e);
            h->launches += 1;
            h->persist_pending = true;
            h->parity ^= (int)(body & 1);
            h->steps += body;
            body = 0;
        }
    }
    for (int64_t k = 0; k < body + (n > 0 ? 1 : 0); ++k) {
        // the observable step adds each column's f_s to the profile accumulator,
        // which the reduction below publishes and zeroes again
        const int obs = (k == body);
        cudaError_t e = enqueue_step(h, h->parity, obs, h->stream);
        h->launches++;
        if (e != cudaSuccess) return cuda_fail(e);
        h->parity ^= 1;
        h->steps++;
    }
    if (n > 0) {
        cudaError_t e = lbmk::launch_reduce_obs(h->d_inst, h->n_inst, h->max_lattice_parts,
                                                h->d_part, h->d_obs, h->d_obs_map, h->d_frz,
                                                h->d_red, h->d_cnt, h->clock, h->stream);
        h->launches++;
        if (e != cudaSuccess) return cuda_fail(e);
        h->have_obs = true;
        h->frz_base = h->mdot_base;
    }
    return LBM_OK;
}

int lbm_observables_all(lbm_handle* h, double* out) {
    if (!h || !out) return LBM_EINVAL;
    if (!h->have_obs) return LBM_ESTATE;
    cudaError_t e = read_obs(h, 0, (size_t)lbmk::kObs * h->n_inst, out);
    if (e != cudaSuccess) return cuda_fail(e);
    if (h->failed) return LBM_ETIMEOUT;
    for (int k = 0; k < h->n_inst; ++k)
        if (unstable(out + (size_t)k * lbmk::kObs)) return LBM_EUNSTABLE;
    return LBM_OK;
}

int lbm_freezing(lbm_handle* h, int32_t inst, double* out) {
    if (!inst_ok(h, inst) || !out) return LBM_EINVAL;
    if (!h->have_obs) return LBM_ESTATE;
    double* dst = h->h_frz ? h->h_frz + (size_t)inst * lbmk::kFrz : out;
    cudaError_t e = cudaMemcpyAsync(dst, h->d_frz + (size_t)inst * lbmk::kFrz,
                                    sizeof(double) * lbmk::kFrz, cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = sync_checked(h);
    if (e != cudaSuccess) return cuda_fail(e);
    if (h->h_frz) memcpy(out, dst, sizeof(double) * lbmk::kFrz);
    // steps count from this lattice's own start; slot sums retired by a table
    // rebuild before the record was taken are added back
    const double s0 = (double)h->step0[inst];
    out[LBM_FRZ_STEP] -= s0;
    if (out[LBM_FRZ_FREEZE_STEP] >= 0.0) out[LBM_FRZ_FREEZE_STEP] -= s0;
    out[LBM_FRZ_MDOT_INTEGRAL] += h->frz_base[inst];
    return h->failed ? LBM_ETIMEOUT : LBM_OK;
}

int lbm_solid_profile(lbm_handle* h, int32_t inst, double* out) {
    if (!inst_ok(h, inst) || !out) return LBM_EINVAL;
    if (!h->have_obs) return LBM_ESTATE;
    cudaError_t e = cudaMemcpyAsync(out, h->d_prof_out + h->layout.prof_at[inst],
                                    sizeof(double) * (size_t)h->params[inst].nx,
                                    cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = sync_checked(h);
    if (e != cudaSuccess) return cuda_fail(e);
    return h->failed ? LBM_ETIMEOUT : LBM_OK;
}

int lbm_observables(lbm_handle* h, int32_t inst, double* out) {
    if (!inst_ok(h, inst) || !out) return LBM_EINVAL;
    if (!h->have_obs) return LBM_ESTATE;
    cudaError_t e = read_obs(h, (size_t)inst * lbmk::kObs, lbmk::kObs, out);
    if (e != cudaSuccess) return cuda_fail(e);
    if (h->failed) return LBM_ETIMEOUT;
    return unstable(out) ? LBM_EUNSTABLE : LBM_OK;
}

namespace {

extern "C++" {
// Planar host staging of one lattice's stored state in 16-bit storage,
// nx-compact: tp holds 27 planes of the storage type (set s, direction i in
// plane 9 s + i; the rest planes 0, 9, 18 are unused), ta the 10 FP32 planes in
// the order of lbmk::aux_at (the carried fields f_l .. S, phi_ref, T_ref and the
// rest populations g_0, h_0, f_0).
template <typename T>
int download_planar(lbm_handle* h, int32_t inst, std::vector<T>& tp, std::vector<float>& ta) {
    const lbm_params& p = h->params[inst];
    const Inst& I = h->inst[inst];
    const int plane = (int)I.plane;
    std::vector<T> rp((size_t)lbmk::kPopElems * plane);
    std::vector<float> ra((size_t)aux_planes(h->storage) * plane);
    cudaError_t e = cudaMemcpyAsync(rp.data(), I.pop[h->parity], rp.size() * sizeof(T),
                                    cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(ra.data(), I.aux[h->parity], ra.size() * sizeof(float),
                            cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return cuda_fail(e);
    const size_t n = (size_t)p.nx * p.ny;
    const int na = 10;
    tp.assign((size_t)27 * n, T());
    ta.assign((size_t)na * n, 0.f);
    for (int y = 0; y < p.ny; ++y)
        for (int x = 0; x < p.nx; ++x) {
            const size_t k = (size_t)y * p.nx + x;
            const int site = y * I.pitch + x;
            for (int set = 0; set < 3; ++set)
                for (int i = 1; i < 9; ++i) tp[(9 * set + i) * n + k] = rp[pop_at(set, i, site)];
            for (int a = 0; a < na; ++a) ta[a * n + k] = ra[aux_at(a, site)];
        }
    return LBM_OK;
}

template <typename T>
int upload_planar(lbm_handle* h, int32_t inst, const std::vector<T>& tp, const std::vector<float>& ta) {
    const lbm_params& p = h->params[inst];
    const Inst& I = h->inst[inst];
    const int plane = (int)I.plane;
    std::vector<T> rp((size_t)lbmk::kPopElems * plane, T());
    std::vector<float> ra((size_t)aux_planes(h->storage) * plane, 0.f);
    const size_t n = (size_t)p.nx * p.ny;
    const int na = 10;
    for (int y = 0; y < p.ny; ++y)
        for (int x = 0; x < p.nx; ++x) {
            const size_t k = (size_t)y * p.nx + x;
            const int site = y * I.pitch + x;
            for (int set = 0; set < 3; ++set)
                for (int i = 1; i < 9; ++i) rp[pop_at(set, i, site)] = tp[(9 * set + i) * n + k];
            for (int a = 0; a < na; ++a) ra[aux_at(a, site)] = ta[a * n + k];
        }
    cudaError_t e = cudaMemcpyAsync(I.pop[h->parity], rp.data(), rp.size() * sizeof(T),
                                    cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(I.aux[h->parity], ra.data(), ra.size() * sizeof(float),
                            cudaMemcpyHostToDevice, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);  // host arrays die on return
    return e == cudaSuccess ? LBM_OK : cuda_fail(e);
}

// 16-bit storage (FP16 or BF16): download, then decode every population with
// the references of the site it streams into (the kernels' decode).
template <typename ST>
int get_state_16(lbm_handle* h, int32_t inst, double* pops, double* aux) {
    using C16 = lbmk::Bits16<ST>;
    const lbm_params& p = h->params[inst];
    const Inst& I = h->inst[inst];
    const size_t n = (size_t)p.nx * p.ny;
    std::vector<ST> tp;
    std::vector<float> ta;
    const int rc = download_planar(h, inst, tp, ta);
    if (rc != LBM_OK) return rc;
    const double L = h->init_L[inst];
    const float* phr = ta.data() + 5 * n;
    const float* Tr = ta.data() + 6 * n;
    if (pops) {
        for (int y = 0; y < p.ny; ++y)
            for (int x = 0; x < p.nx; ++x) {
                const size_t k = (size_t)y * p.nx + x;
                pops[k] = ta[7 * n + k];                                   // g_0
                pops[9 * n + k] = (double)ta[8 * n + k] + L * (double)ta[k]; // h_0 + L f_l
                pops[18 * n + k] = ta[9 * n + k];                           // f_0
                for (int i = 1; i < 9; ++i) {
                    const size_t kd = dest_site(p, x, y, i);
                    const float rg = C16::to_f(tp[i * n + k]);
                    const float rh = C16::to_f(tp[(9 + i) * n + k]);
                    const float rf = C16::to_f(tp[(18 + i) * n + k]);
                    pops[i * n + k] = rg + kWf[i] * phr[kd];
                    pops[(9 + i) * n + k] = rh + kWf[i] * I.Cpref * Tr[kd];
                    pops[(18 + i) * n + k] = rf * (1.f / 4096.f) + kWf[i] * 3.f * ta[3 * n + k];
                }
            }
    }
    if (aux)
        for (size_t k = 0; k < (size_t)5 * n; ++k) aux[k] = ta[k];
    return LBM_OK;
}

// 16-bit storage: choose the references of every site from the given state
// (phi_ref = sum g, T_ref from Eq. 9 on sum h), then encode.
template <typename ST>
int set_state_16(lbm_handle* h, int32_t inst, const double* pops, const double* aux) {
    using C16 = lbmk::Bits16<ST>;
    const lbm_params& p = h->params[inst];
    const Inst& I = h->inst[inst];
    const size_t n = (size_t)p.nx * p.ny;
    const double L = h->init_L[inst];
    std::vector<float> ta((size_t)10 * n);
    for (size_t k = 0; k < (size_t)5 * n; ++k) ta[k] = (float)aux[k];
    float* phr = ta.data() + 5 * n;
    float* Tr = ta.data() + 6 * n;
    const double Hs = p.Cp * p.T_m;
    for (size_t k = 0; k < n; ++k) {
        double phi = 0.0, H = 0.0;
        for (int i = 0; i < 9; ++i) { phi += pops[i * n + k]; H += pops[(9 + i) * n + k]; }
        double fl = (H - Hs) / L;
        fl = fl < 0 ? 0 : (fl > 1 ? 1 : fl);
        phr[k] = (float)phi;
        // Eq. 9b with the local heat capacity (Eq. 1; uniform: Cp)
        const double ph = phi < 0 ? 0 : (phi > 1 ? 1 : phi);
        double chi = (phi - 0.5) / p.pc_ramp + 0.5;
        chi = chi < 0 ? 0 : (chi > 1 ? 1 : chi);
        const double fs = chi * (1.0 - fl);
        const double cp = fs * p.Cp * p.Cp_ratio_sl +
                          (1.0 - fs) * (ph * p.Cp + (1.0 - ph) * p.Cp * p.Cp_ratio_gl);
        Tr[k] = (float)(p.T_m + (H - Hs - L * fl) / cp);
    }
    std::vector<ST> tp((size_t)27 * n, C16::from_f(0.f));
    for (int y = 0; y < p.ny; ++y)
        for (int x = 0; x < p.nx; ++x) {
            const size_t k = (size_t)y * p.nx + x;
            ta[7 * n + k] = (float)pops[k];
            ta[8 * n + k] = (float)(pops[9 * n + k] - L * (double)ta[k]);
            ta[9 * n + k] = (float)pops[18 * n + k];
            for (int i = 1; i < 9; ++i) {
                const size_t kd = dest_site(p, x, y, i);
                tp[i * n + k] = C16::from_d(pops[i * n + k] - (double)(kWf[i] * phr[kd]));
                tp[(9 + i) * n + k] =
                    C16::from_d(pops[(9 + i) * n + k] - (double)(kWf[i] * I.Cpref * Tr[kd]));
                const double fr = (double)(kWf[i] * 3.f * ta[3 * n + k]);
                tp[(18 + i) * n + k] = C16::from_d((pops[(18 + i) * n + k] - fr) * 4096.0);
            }
        }
    const int rc = upload_planar(h, inst, tp, ta);
    if (rc != LBM_OK) return rc;
    h->initialised = true;
    h->have_obs = false;
    return LBM_OK;
}
}  // extern "C++"

// FP32 storage: the planes are converted on the device, two at a time through
// the staging area of lbm_init_fields, and copied to or from the caller's
// arrays. (Converted on the host, from the raw buffers through two vectors, a
// round trip of 384 x 300 sites took 8.6 ms against 1.0 ms.)
int get_state_fp32(lbm_handle* h, int32_t inst, double* pops, double* aux) {
    const size_t n = (size_t)h->params[inst].nx * h->params[inst].ny;
    auto planes = [&](int q0, int q1, double* out) {
        cudaError_t e = cudaSuccess;
        for (int q = q0; q < q1 && e == cudaSuccess; q += 2) {
            const int m = std::min(2, q1 - q);
            e = lbmk::launch_planes_from_state(h->d_inst, inst, (int)n, h->parity, h->init_L[inst], q, m,
                                               h->d_stage, h->stream);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(out + (size_t)(q - q0) * n, h->d_stage, n * m * sizeof(double),
                                    cudaMemcpyDeviceToHost, h->stream);
        }
        return e;
    };
    cudaError_t e = pops ? planes(0, 27, pops) : cudaSuccess;
    if (e == cudaSuccess && aux) e = planes(27, 32, aux);
    // also after a failure: no copy to the caller's arrays outlives the call
    const cudaError_t done = cudaStreamSynchronize(h->stream);
    if (e == cudaSuccess) e = done;
    return e == cudaSuccess ? LBM_OK : cuda_fail(e);
}

int set_state_fp32(lbm_handle* h, int32_t inst, const double* pops, const double* aux) {
    const size_t n = (size_t)h->params[inst].nx * h->params[inst].ny;
    auto plane = [&](int q) { return q < 27 ? pops + (size_t)q * n : aux + (size_t)(q - 27) * n; };
    // every plane once: h_0 with f_l, which its shift needs, the others in pairs
    int order[32] = {9, 27}, n_order = 2;
    for (int q = 0; q < 32; ++q)
        if (q != 9 && q != 27) order[n_order++] = q;
    cudaError_t e = cudaSuccess;
    for (int a = 0; a < 32 && e == cudaSuccess; a += 2) {
        for (int b = 0; b < 2 && e == cudaSuccess; ++b)
            e = cudaMemcpyAsync(h->d_stage + b * n, plane(order[a + b]), n * sizeof(double),
                                cudaMemcpyHostToDevice, h->stream);
        if (e == cudaSuccess)
            e = lbmk::launch_state_from_planes(h->d_inst, inst, (int)n, h->parity, h->init_L[inst],
                                               order[a], order[a + 1], h->d_stage, h->stream);
    }
    // also after a failure: no copy from the caller's arrays outlives the call
    const cudaError_t done = cudaStreamSynchronize(h->stream);
    if (e == cudaSuccess) e = done;
    if (e != cudaSuccess) return cuda_fail(e);
    h->initialised = true;
    h->have_obs = false;
    return LBM_OK;
}

}  // namespace

int lbm_get_state(lbm_handle* h, int32_t inst, double* pops, double* aux) {
    if (!inst_ok(h, inst)) return LBM_EINVAL;
    if (!h->initialised) return LBM_ESTATE;
    if (h->storage == LBM_STORE_FP16) return get_state_16<__half>(h, inst, pops, aux);
    if (h->storage == LBM_STORE_BF16) return get_state_16<__nv_bfloat16>(h, inst, pops, aux);
    return get_state_fp32(h, inst, pops, aux);
}

int lbm_set_state(lbm_handle* h, int32_t inst, const double* pops, const double* aux) {
    if (!inst_ok(h, inst) || !pops || !aux) return LBM_EINVAL;
    int rc;
    if (h->storage == LBM_STORE_FP16) rc = set_state_16<__half>(h, inst, pops, aux);
    else if (h->storage == LBM_STORE_BF16) rc = set_state_16<__nv_bfloat16>(h, inst, pops, aux);
    else rc = set_state_fp32(h, inst, pops, aux);
    if (rc != LBM_OK) return rc;
    return restart_records(h, inst);  // a new run: the freezing record restarts
}

int lbm_set_thermal_walls(lbm_handle* h, int32_t inst, int32_t x_lo, int32_t x_hi,
                          int32_t y_lo, int32_t y_hi) {
    if (!inst_ok(h, inst)) return LBM_EINVAL;
    const int32_t v[4] = {x_lo, x_hi, y_lo, y_hi};
    for (int32_t f : v)
        if (f != 0 && f != 1) return LBM_EINVAL;
    lbm_params& p = h->params[inst];
    if ((p.periodic_x && (x_lo || x_hi)) || (p.periodic_y && (y_lo || y_hi))) return LBM_EINVAL;
    p.dirichlet_x_lo = x_lo;
    p.dirichlet_x_hi = x_hi;
    p.dirichlet_y_lo = y_lo;
    p.dirichlet_y_hi = y_hi;
    const int keep = lbmk::kDirXlo | lbmk::kDirXhi | lbmk::kDirYlo | lbmk::kDirYhi;
    h->inst[inst].flags = (h->inst[inst].flags & ~keep) | (x_lo ? lbmk::kDirXlo : 0) |
                          (x_hi ? lbmk::kDirXhi : 0) | (y_lo ? lbmk::kDirYlo : 0) |
                          (y_hi ? lbmk::kDirYhi : 0);
    return upload_tables(h);  // instance table, item tables; drops graphs; synchronises
}

int lbm_set_kernel(lbm_handle* h, int32_t kind, int32_t a, int32_t b, int32_t c) {
    if (!h) return LBM_EINVAL;
    if (kind == LBM_KERNEL_TILE) {
        if (!lbmk::tile_supported(a, b, h->storage)) return LBM_EINVAL;
        if (h->exec == LBM_EXEC_PERSISTENT) return LBM_EINVAL;  // persistent form is strip-only
        h->kind = kind; h->tx = a; h->ty = b;
    } else if (kind == LBM_KERNEL_BLOCK) {
        for (int k = 0; k < h->n_inst; ++k)
            if (!h->params[k].periodic_x) return LBM_EINVAL;
        if (!lbmk::block_supported(a, c) || (b != 0 && b < kMinRows)) return LBM_EINVAL;
        h->kind = kind; h->warps = a; h->rows_req = b; h->regs = c;
    } else if (kind == LBM_KERNEL_STRIP || kind == LBM_KERNEL_STAGED) {
        for (int k = 0; k < h->n_inst; ++k)
            if (!h->params[k].periodic_x) return LBM_EINVAL;
        if (b != 0 && b < kMinRows) return LBM_EINVAL;
        if (kind == LBM_KERNEL_STAGED ? !lbmk::staged_supported(a, c, h->storage)
                                      : !lbmk::strip_supported(a, c))
            return LBM_EINVAL;
        if (kind == LBM_KERNEL_STRIP && h->storage == LBM_STORE_BF16) return LBM_EINVAL;  // staged only
        h->kind = kind; h->warps = a; h->rows_req = b; h->regs = c;
    } else {
        return LBM_EINVAL;
    }
    h->chosen = false;
    h->have_obs = false;  // partial slots are renumbered
    return upload_tables(h);
}

int lbm_set_exec(lbm_handle* h, int32_t mode, int32_t chunk) {
    if (!h || chunk < 1 || chunk > kMaxChunk) return LBM_EINVAL;
    if (mode != LBM_EXEC_LAUNCH && mode != LBM_EXEC_GRAPH && mode != LBM_EXEC_PERSISTENT)
        return LBM_EINVAL;
    if (mode == LBM_EXEC_PERSISTENT && (!is_strip(h->kind) || h->persist_grid <= 0))
        return LBM_EINVAL;
    drop_graphs(h);
    const bool was_tiled = tiled(h);
    const int old_mode = h->exec, old_chunk = h->chunk;
    h->exec = mode;
    h->chunk = chunk;
    if (tiled(h) == was_tiled) return LBM_OK;
    const int rc = upload_tables(h);
    if (rc != LBM_OK) {  // as it was (the tables are rebuilt before the next step)
        h->exec = old_mode;
        h->chunk = old_chunk;
    }
    return rc;
}

int lbm_get_exec(const lbm_handle* h, int32_t* out) {
    if (!h || !out) return LBM_EINVAL;
    out[0] = h->exec;
    out[1] = h->chunk;
    out[2] = h->persist_grid;
    return LBM_OK;
}

int lbm_barrier_selftest(lbm_handle* h, uint64_t limit_ns, int32_t* err_flag) {
    if (!h || !err_flag || limit_ns == 0 || limit_ns > kBarrierLimitNs) return LBM_EINVAL;
    static thread_local int v = 0;
    cudaError_t e = cudaMemsetAsync(&h->d_sync->probe_bar, 0, 2 * sizeof(int), h->stream);
    if (e == cudaSuccess)
        e = lbmk::launch_barrier_timeout_probe(&h->d_sync->probe_bar, &h->d_sync->probe_err,
                                               limit_ns, h->stream);
    h->launches++;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&v, &h->d_sync->probe_err, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return cuda_fail(e);
    *err_flag = v;
    return LBM_OK;
}

int lbm_get_kernel(const lbm_handle* h, int32_t* out) {
    if (!h || !out) return LBM_EINVAL;
    out[0] = h->kind;
    if (is_strip(h->kind)) { out[1] = h->warps; out[2] = h->rows; out[3] = h->regs; }
    else { out[1] = h->tx; out[2] = h->ty; out[3] = 0; }
    return LBM_OK;
}

int lbm_get_step_kernel(const lbm_handle* h, int32_t* out) {
    if (!h || !out) return LBM_EINVAL;
    if (!tiled(h)) return lbm_get_kernel(h, out);
    out[0] = LBM_KERNEL_TILE;
    out[1] = h->tx;
    out[2] = h->ty;
    out[3] = 0;
    return LBM_OK;
}

int lbm_autotune(lbm_handle* h, int32_t steps, double* times_ms, int32_t cap, int32_t* n_tried) {
    if (!h || steps < 1) return LBM_EINVAL;
    if (!h->initialised) return LBM_ESTATE;
    struct Cand { int kind, a, b, c; };
    std::vector<Cand> cands;
    bool all_px = true;
    for (int k = 0; k < h->n_inst; ++k) all_px = all_px && h->params[k].periodic_x;
    if (all_px) {
        const int rows[] = {0, 8, 16, 32};
        const int var[][2] = {{4, 168}, {4, 128}, {8, 128}, {4, 255}};
        for (int r : rows)
            for (auto& v : var) cands.push_back({LBM_KERNEL_STRIP, v[0], r, v[1]});
        for (int r : rows)
            for (auto& v : var) cands.push_back({LBM_KERNEL_STAGED, v[0], r, v[1]});
        const int bvar[][2] = {{4, 128}, {4, 168}, {8, 128}};
        for (int r : rows)
            for (auto& v : bvar) cands.push_back({LBM_KERNEL_BLOCK, v[0], r, v[1]});
    }
    if (h->exec != LBM_EXEC_PERSISTENT) {  // the persistent form is strip-only
        cands.push_back({LBM_KERNEL_TILE, 32, 4, 0});
        cands.push_back({LBM_KERNEL_TILE, 32, 8, 0});
        cands.push_back({LBM_KERNEL_TILE, 64, 4, 0});
        cands.push_back({LBM_KERNEL_TILE, 32, 16, 0});
    }
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return LBM_ECUDA;
    if (cudaEventCreate(&e1) != cudaSuccess) { cudaEventDestroy(e0); return LBM_ECUDA; }
    int best = -1, tried = 0;
    float best_ms = 0.f;
    int rc = LBM_OK;
    for (size_t j = 0; j < cands.size() && rc == LBM_OK; ++j) {
        const Cand& cd = cands[j];
        if (lbm_set_kernel(h, cd.kind, cd.a, cd.b, cd.c) != LBM_OK) continue;
        rc = lbm_step(h, 1);
        if (rc != LBM_OK) break;
        float ms = 0.f;
        for (int rep = 0; rep < 2 && rc == LBM_OK; ++rep) {  // the shorter of two timings
            cudaEventRecord(e0, h->stream);
            rc = lbm_step(h, steps);
            cudaEventRecord(e1, h->stream);
            if (rc != LBM_OK) break;
            if (cudaEventSynchronize(e1) != cudaSuccess) { rc = LBM_ECUDA; break; }
            float t = 0.f;
            cudaEventElapsedTime(&t, e0, e1);
            t /= (float)steps;
            ms = rep == 0 ? t : std::min(ms, t);
        }
        if (rc != LBM_OK) break;
        if (times_ms && tried < cap) times_ms[tried] = ms;
        ++tried;
        if (best < 0 || ms < best_ms) { best = (int)j; best_ms = ms; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (n_tried) *n_tried = tried;
    if (rc != LBM_OK) return rc;
    if (best < 0) return LBM_EINVAL;
    return lbm_set_kernel(h, cands[best].kind, cands[best].a, cands[best].b, cands[best].c);
}

int64_t lbm_step_count(const lbm_handle* h) { return h ? h->steps : -1; }

int64_t lbm_launch_count(const lbm_handle* h) { return h ? h->launches : -1; }

void lbm_destroy(lbm_handle* h) {
    if (!h) return;
    cudaStreamSynchronize(h->stream);
    drop_graphs(h);
    if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
    delete h;
}

const char* lbm_error_string(int code) {
    switch (code) {
        case LBM_OK: return "ok";
        case LBM_EINVAL: return "invalid argument or parameter set";
        case LBM_ENOMEM: return "workspace smaller than lbm_workspace_size";
        case LBM_ECUDA: return "CUDA call failed";
        case LBM_ETIMEOUT: return "device-side wait timed out";
        case LBM_EUNSTABLE: return "non-finite fields";
        case LBM_ESTATE: return "call out of order";
        case LBM_ETOOLARGE: return "lattice exceeds the fixed scratch of lbm_step_noalloc";
        default: return "unknown error";
    }
}

}  // extern "C"

namespace lbmk {

void inst_from_params(const lbm_params& p, Inst* out, double* Lout) {
    const double cs2 = 1.0 / 3.0;
    Inst I;
    memset(&I, 0, sizeof(I));
    I.nx = p.nx; I.ny = p.ny; I.pitch = pitch_for(p.nx);
    I.flags = (p.periodic_x ? kPeriodicX : 0) | (p.periodic_y ? kPeriodicY : 0) |
              (p.dirichlet_x_lo ? kDirXlo : 0) | (p.dirichlet_x_hi ? kDirXhi : 0) |
              (p.dirichlet_y_lo ? kDirYlo : 0) | (p.dirichlet_y_hi ? kDirYhi : 0) |
              (p.st_mask_liquid ? kStMask : 0);
    I.plane = (long long)I.pitch * p.ny;
    const double L = p.Cp * (p.T_m - p.T_w) / p.Ste;  // Eq. 42
    const double tau_g = p.mobility / cs2 + 0.5;
    const double rho_g = p.rho_l / p.rho_ratio_lg, rho_s = p.rho_l * p.rho_ratio_sl;
    const double mu_l = p.rho_l * cs2 * (p.tau_f_liquid - 0.5);
    const double pi = acos(-1.0);
    I.L = (float)L;
    I.Hs = (float)(p.Cp * p.T_m);
    I.Tm = (float)p.T_m;
    I.Cp = (float)p.Cp;
    I.Cpref = (float)p.Cp_ref;
    I.Tw = (float)p.T_w;
    I.omega_g = (float)(1.0 / tau_g);
    I.omega_h = (float)(1.0 / p.tau_h);
    I.kappa = (float)(1.5 * p.sigma * p.W);
    I.beta = (float)(12.0 * p.sigma / p.W);
    I.lam_coef = (float)(4.0 / p.W);
    I.rho_s = (float)rho_s;
    I.rho_l = (float)p.rho_l;
    I.rho_g = (float)rho_g;
    I.mu_s = (float)(mu_l * p.rho_ratio_sl);
    I.mu_l = (float)mu_l;
    I.mu_g = (float)(mu_l / p.mu_ratio_lg);
    I.mdot_coef = (float)(1.0 - rho_s / p.rho_l);
    I.tan_w = (float)tan(pi / 2.0 - p.theta_deg * pi / 180.0);
    I.inv_ramp = (float)(1.0 / p.pc_ramp);
    I.normal_eps2 = (float)(p.normal_eps * p.normal_eps);
    I.inv_L = (float)(1.0 / L);
    I.inv_Cp = (float)(1.0 / p.Cp);
    I.buoy_x = (float)(-p.rho_0 * p.beta_T * p.gx);  // Section 4.3, Boussinesq
    I.buoy_y = (float)(-p.rho_0 * p.beta_T * p.gy);
    I.T_ref = (float)p.T_ref;
    if (I.buoy_x != 0.f || I.buoy_y != 0.f) I.flags |= kBuoy;
    // per-phase thermal properties (Eq. 1 for C_p and k; tau_h - 1/2 ~ k)
    I.Cp_s = (float)(p.Cp * p.Cp_ratio_sl);
    I.Cp_g = (float)(p.Cp * p.Cp_ratio_gl);
    I.k_s = (float)p.k_ratio_sl;
    I.k_g = (float)p.k_ratio_gl;
    I.dtau_h = (float)(p.tau_h - 0.5);
    if (p.Cp_ratio_sl != 1.0 || p.Cp_ratio_gl != 1.0 || p.k_ratio_sl != 1.0 || p.k_ratio_gl != 1.0)
        I.flags |= kPhaseProps;
    *out = I;
    *Lout = L;
}

bool params_valid(const lbm_params& p) { return valid_params(p); }

}  // namespace lbmk
