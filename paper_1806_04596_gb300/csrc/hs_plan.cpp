// Plan construction: everything the operators derive from the uv coverage.
//
//  * grid coordinates t = u K / (2 pi) per axis, split into the cell floor(t)
//    (mod K) and the fraction; FP32 plans store both in one 32-bit fixed-point
//    word per axis (fraction resolution 2^-23 .. 2^-20 cells, computed in FP64
//    so the FP32 kernels never form t themselves), FP64 plans store the exact
//    FP64 fraction;
//  * a per-channel sort of the visibilities by the 32 x 32 grid tile holding
//    the start of their 8 x 8 window, then by cell, so that consecutive
//    visibilities touch neighbouring grid cells;
//  * the gridding lists, consumed without atomics: for grids of at least
//    64 x 64 cells, per (channel, 32-column strip, row range) the windows that
//    reach it, grouped by start row into disjoint column ranges (sweep
//    kernel); otherwise, and for the compensated kernel, per (channel, 32 x 32
//    tile) the windows that overlap it (a window straddles at most 2 x 2 tiles);
//  * the Kaiser-Bessel polynomial pieces, the Z scaling, the FFT twiddles;
//  * all scratch buffers, so that no compute call allocates.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <exception>
#include <functional>
#include <map>
#include <memory>
#include <mutex>
#include <thread>
#include <tuple>
#include <vector>

#include "hs_internal.h"

namespace hs {

hs_status dwt_init();
hs_status fft_init();
hs_status nufft_init();
hs_status prox_init();
hs_status eig_init();
int64_t gram_part_doubles(int L);

// Device memory held by the library's plans and PD states (process-wide), and
// the optional cap on it (hs_set_device_limit; 0: none).
static std::atomic<int64_t> g_lib_bytes{0};
static std::atomic<int64_t> g_lib_limit{0};

void set_device_limit(int64_t bytes) { g_lib_limit.store(bytes < 0 ? 0 : bytes); }
int64_t device_bytes_held() { return g_lib_bytes.load(); }
int64_t device_limit() { return g_lib_limit.load(); }

hs_status lib_alloc(void** ptr, size_t bytes) {
    *ptr = nullptr;
    const int64_t lim = g_lib_limit.load();
    const int64_t now = g_lib_bytes.fetch_add((int64_t)bytes) + (int64_t)bytes;
    if (lim > 0 && now > lim) {
        g_lib_bytes.fetch_sub((int64_t)bytes);
        return fail(HS_ERR_NOMEM, "allocation of %zu bytes would pass the library's device limit (%lld of %lld held)",
                    bytes, (long long)(now - (int64_t)bytes), (long long)lim);
    }
    cudaError_t e = cudaMalloc(ptr, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *ptr = nullptr;
        g_lib_bytes.fetch_sub((int64_t)bytes);
        return fail(HS_ERR_NOMEM, "cudaMalloc(%zu bytes) failed: %s", bytes, cudaGetErrorString(e));
    }
    return HS_OK;
}

void lib_free(void* ptr, size_t bytes) {
    if (ptr) {
        cudaFree(ptr);
        g_lib_bytes.fetch_sub((int64_t)bytes);
    }
}

hs_status plan_alloc(Plan* p, void** ptr, size_t bytes) {
    *ptr = nullptr;
    if (bytes == 0) return HS_OK;
    HS_TRY(lib_alloc(ptr, bytes));
    p->allocs.push_back(*ptr);
    p->alloc_bytes.push_back(bytes);
    p->device_bytes += (int64_t)bytes;
    return HS_OK;
}

// Free one allocation of the plan (lists rebuilt at creation).
static void plan_release(Plan* p, void* ptr) {
    for (size_t k = 0; k < p->allocs.size(); ++k)
        if (p->allocs[k] == ptr) {
            lib_free(ptr, p->alloc_bytes[k]);
            p->device_bytes -= (int64_t)p->alloc_bytes[k];
            p->allocs.erase(p->allocs.begin() + k);
            p->alloc_bytes.erase(p->alloc_bytes.begin() + k);
            return;
        }
}

void plan_free(Plan* p) {
    if (p->fft_ev_col) cudaEventDestroy(p->fft_ev_col);
    if (p->fft_ev_join) cudaEventDestroy(p->fft_ev_join);
    if (p->fft_side) cudaStreamDestroy(p->fft_side);
    p->fft_ev_col = p->fft_ev_join = nullptr;
    p->fft_side = nullptr;
    for (size_t k = 0; k < p->allocs.size(); ++k) lib_free(p->allocs[k], p->alloc_bytes[k]);
    p->allocs.clear();
    p->alloc_bytes.clear();
}

static bool pow2(int v) { return v > 0 && (v & (v - 1)) == 0; }
// x mod K for any x (grids need not be powers of two).
static inline int modk(int64_t x, int K) { return (int)(((x % K) + K) % K); }
// Image sides the kernels support: r 2^a with r in {1, 3, 5} (FFT lines of
// 2 r 2^a), at least 16, and multiples of 16 unless powers of two (gridding
// tiles and strips of 32 cells).
static bool side_ok(int n) {
    if (n < 16 || n > 2048) return false;
    if (pow2(n)) return true;
    int m = n;
    if (m % 5 == 0) m /= 5;
    else if (m % 3 == 0) m /= 3;
    return pow2(m) && n % 16 == 0;
}
static int ilog2(int v) {
    int r = 0;
    while ((1 << r) < v) ++r;
    return r;
}

template <typename T> static hs_status upload(Plan* p, void** dst, const std::vector<T>& h) {
    HS_TRY(plan_alloc(p, dst, h.size() * sizeof(T)));
    if (!h.empty()) HS_CHECK_CUDA(cudaMemcpy(*dst, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice));
    return HS_OK;
}

template <typename R>
static hs_status upload_real(Plan* p, void** dst, const std::vector<double>& h) {
    std::vector<R> v(h.size());
    for (size_t i = 0; i < h.size(); ++i) v[i] = (R)h[i];
    return upload(p, dst, v);
}

static hs_status download_real(const Plan* p, const void* src, int64_t n, std::vector<double>& out,
                               cudaStream_t s) {
    out.assign((size_t)n, 0.0);
    if (n == 0) return HS_OK;
    if (p->prec == HS_F32) {
        std::vector<float> tmp((size_t)n);
        HS_CHECK_CUDA(cudaMemcpyAsync(tmp.data(), src, n * sizeof(float), cudaMemcpyDeviceToHost, s));
        HS_CHECK_CUDA(cudaStreamSynchronize(s));
        for (int64_t i = 0; i < n; ++i) out[i] = tmp[i];
    } else {
        HS_CHECK_CUDA(cudaMemcpyAsync(out.data(), src, n * sizeof(double), cudaMemcpyDeviceToHost, s));
        HS_CHECK_CUDA(cudaStreamSynchronize(s));
    }
    return HS_OK;
}

// fn(k) for k = 0 .. n - 1 on the host's cores (channels and blocks are
// independent; results are placed by k, so they do not depend on the threads).
// items: visibilities in all; one more thread per 32 768 (below that, starting
// threads costs more than it gains: 60 channels of 16 took 5.7 instead of 2.5 ms).
// An exception of any call is thrown again here.
static void parallel_for(int n, int64_t items, const std::function<void(int)>& fn) {
    const int64_t most = std::min<int64_t>(std::max(1u, std::thread::hardware_concurrency()), 1 + items / 32768);
    const int nt = (int)std::min<int64_t>(n, std::min<int64_t>(16, most));
    std::atomic<int> next{0};
    std::exception_ptr err;
    std::mutex mu;
    auto work = [&]() {
        for (int k; (k = next.fetch_add(1)) < n;) {
            try {
                fn(k);
            } catch (...) {
                std::lock_guard<std::mutex> lock(mu);
                if (!err) err = std::current_exception();
            }
        }
    };
    std::vector<std::thread> ts;
    try {
        ts.reserve(nt);
        for (int t = 1; t < nt; ++t) ts.emplace_back(work);
    } catch (const std::exception&) {   // no more threads, or no memory for one: the ones there are do the work
    }
    work();
    for (auto& t : ts) t.join();
    if (err) std::rethrow_exception(err);
}

// f(), with host allocation failures as a status (no exception passes the C boundary).
template <typename F> static hs_status no_throw(F f) {
    try {
        return f();
    } catch (const std::exception& e) {
        return fail(HS_ERR_NOMEM, "host allocation failed while building a plan: %s", e.what());
    }
}

// Gridding lists of the sweep kernel (grids of at least 64 x 64 cells). A work
// item is one channel, one 32-column strip and its output rows [row0, row1);
// its list holds every window that overlaps the strip and starts in rows
// row0 - 7 .. row1 - 1 (circularly), as groups of 4 slots (-1 pads) whose
// windows cover disjoint columns of the strip (slots in increasing start
// column) and start in the same 4-row band (relative start row y, band
// floor(y / 4)), so that they all lie in that band and the next two. Windows are
// placed in increasing start row, first fit over the band's groups; groups are
// stored by band. Rows are cut after hmax rows, or earlier once the list
// would pass cap windows (at least one row per item). Items are stored
// heaviest first.
// Host part: window start cells k0x[r], k0y[r] in the order the kernel indexes
// them (list entries are these positions r), channel ranges off[0..L].
hs_status sweep_lists(int Kx, int Ky, int L, const int64_t* off, const int* k0xs, const int* k0ys, int hmax_req,
                      int cap, std::vector<SweepItem>& items, std::vector<int>& ent) {
    const int nstrip = Kx / GRID_TILE;
    const int hmax = std::min(hmax_req, Ky - 8);
    struct Win {
        int y, x, r;   // start row (absolute, then relative to row0), start column relative to the strip
    };
    struct Grp {
        int y, m;        // band, windows held
        uint32_t mask;   // strip columns covered
        int e[4], x[4];  // sorted visibility indices and start columns, by start column
    };
    // channels in parallel, their lists joined in channel order
    std::vector<std::vector<SweepItem>> ch_items(L);
    std::vector<std::vector<int>> ch_ent(L);
    parallel_for(L, off[L], [&](int l) {
        std::vector<std::vector<Win>> strips(nstrip);
        std::vector<int64_t> rowcnt(Ky);
        std::vector<Win> seg;
        std::vector<Grp> open;
        std::vector<SweepItem>& items = ch_items[l];
        std::vector<int>& ent = ch_ent[l];
        for (int64_t r = off[l]; r < off[l + 1]; ++r) {
            const int k0x = k0xs[r], k0y = k0ys[r];
            const int s0 = k0x / GRID_TILE, s1 = modk(k0x + 7, Kx) / GRID_TILE;
            strips[s0].push_back({k0y, k0x - s0 * GRID_TILE, (int)r});
            if (s1 != s0) strips[s1].push_back({k0y, modk(k0x - s1 * GRID_TILE + 7, Kx) - 7, (int)r});
        }
        for (int st = 0; st < nstrip; ++st) {
            std::vector<Win>& ws = strips[st];
            // by start row (then column, index): a row range is a contiguous run
            std::sort(ws.begin(), ws.end(), [](const Win& a, const Win& b) {
                return a.y != b.y ? a.y < b.y : (a.x != b.x ? a.x < b.x : a.r < b.r);
            });
            auto row_at = [&](int y) {   // first window starting in row >= y
                return std::lower_bound(ws.begin(), ws.end(), y, [](const Win& w, int v) { return w.y < v; });
            };
            std::fill(rowcnt.begin(), rowcnt.end(), 0);
            for (const Win& w : ws) ++rowcnt[w.y];
            for (int row0 = 0; row0 < Ky;) {
                int64_t cnt = 0;
                for (int d = 1; d <= 7; ++d) cnt += rowcnt[modk(row0 - d, Ky)];
                int row1 = row0;
                while (row1 < Ky && row1 - row0 < hmax && (row1 == row0 || cnt + rowcnt[row1] <= cap))
                    cnt += rowcnt[row1++];
                // windows starting in rows row0 - 7 .. row1 - 1 (circularly), in order of
                // their start row relative to row0 (the wrapped rows come first)
                seg.clear();
                auto take = [&](int ya, int yb) {
                    for (auto it = row_at(ya); it != ws.end() && it->y < yb; ++it)
                        seg.push_back({modk(it->y - row0 + 7, Ky) - 7, it->x, it->r});
                };
                if (row0 >= 7) {
                    take(row0 - 7, row1);
                } else {
                    take(Ky + row0 - 7, Ky);
                    take(0, row1);
                }
                const int e0 = (int)ent.size();
                open.clear();
                size_t first = 0;
                for (const Win& w : seg) {
                    const int b = std::max(w.x, 0), e = std::min(w.x + 8, GRID_TILE);
                    const uint32_t mask = (uint32_t)(((uint64_t)1 << e) - ((uint64_t)1 << b));
                    const int band = (w.y + 8) / 4 - 2;   // floor(y / 4), y >= -7
                    while (first < open.size() && open[first].y < band) ++first;
                    size_t gi = first;
                    while (gi < open.size() && (open[gi].m == 4 || (open[gi].mask & mask))) ++gi;
                    if (gi == open.size()) open.push_back({band, 0, 0u, {-1, -1, -1, -1}, {0, 0, 0, 0}});
                    Grp& gr = open[gi];
                    int k = gr.m++;   // keep the slots in increasing start column
                    for (; k > 0 && gr.x[k - 1] > w.x; --k) {
                        gr.e[k] = gr.e[k - 1];
                        gr.x[k] = gr.x[k - 1];
                    }
                    gr.e[k] = w.r;
                    gr.x[k] = w.x;
                    gr.mask |= mask;
                }
                for (const Grp& gr : open) ent.insert(ent.end(), gr.e, gr.e + 4);
                items.push_back({l, st, row0, row1, e0, (int)ent.size()});
                row0 = row1;
            }
        }
    });
    items.clear();
    ent.clear();
    size_t n_items = 0, n_ent = 0;
    for (int l = 0; l < L; ++l) {
        n_items += ch_items[l].size();
        n_ent += ch_ent[l].size();
    }
    if (n_ent >= ((size_t)1 << 31)) return fail(HS_ERR_ARG, "too many gridding list entries");
    items.reserve(n_items);
    ent.reserve(n_ent);
    for (int l = 0; l < L; ++l) {
        const int e = (int)ent.size();
        for (SweepItem it : ch_items[l]) {
            it.e0 += e;
            it.e1 += e;
            items.push_back(it);
        }
        ent.insert(ent.end(), ch_ent[l].begin(), ch_ent[l].end());
    }
    std::stable_sort(items.begin(), items.end(), [](const SweepItem& a, const SweepItem& b) {
        return (a.e1 - a.e0) + 4 * (a.row1 - a.row0) > (b.e1 - b.e0) + 4 * (b.row1 - b.row0);
    });
    return HS_OK;
}

// Grids whose strips no window reaches twice take the sweep kernel.
static bool sweep_grid(const Plan* p) { return p->g.Kx >= 2 * GRID_TILE && p->g.Ky >= 2 * GRID_TILE; }

static hs_status build_sweep(Plan* p) {
    const int Kx = p->g.Kw, Ky = p->g.Ky;   // half plane: no window reaches the pitch, so none wraps
    std::vector<SweepItem> items;
    std::vector<int> ent;
    HS_TRY(sweep_lists(Kx, Ky, p->g.L, p->off_h.data(), p->k0x_h.data(), p->k0y_h.data(), p->sw_rows,
                       p->sw_cap, items, ent));
    if (p->half) {   // cells that no window of the channel reaches are never read
        auto unread = [&](const SweepItem& it) {
            const int4 r = p->rng_h[it.l];
            const int c0 = it.strip * GRID_TILE;
            return (c0 >= r.x && c0 + GRID_TILE <= r.y) || (it.row0 >= r.z && it.row1 <= r.w);
        };
        items.erase(std::remove_if(items.begin(), items.end(), unread), items.end());
    }
    if (p->sw_items) {   // rebuilt by the autotuner: replace the previous lists
        plan_release(p, p->sw_items);
        plan_release(p, p->sw_ent);
        p->sw_items = nullptr;
        p->sw_ent = nullptr;
    }
    p->n_sw_items = (int64_t)items.size();
    p->n_sw_ent = (int64_t)ent.size();
    HS_TRY(upload(p, &p->sw_items, items));
    HS_TRY(upload(p, (void**)&p->sw_ent, ent));
    return HS_OK;
}

// ---------------------------------------------------------------- autotuner
// Plan-time choice of the parameters that depend on the problem's size and
// sampling density, by timing the candidates on this plan with CUDA events
// (inputs: zeroed plan scratch; the values do not change the work):
//   * sweep gridding row cut and list cap, (32, 512), (64, 1024), (128, 2048):
//     short items balance dense coverage, tall items cut the halo rows; on the half plane also
//     4 or 8 warps to an item (64, 32 or 16 rows), for plans with few items;
//   * FP32 Gram matrix of the nuclear prox on the tensor cores or the CUDA
//     cores (the tensor-core form streams 64-pixel chunks per SM and wins on
//     large cubes; the CUDA-core form wins when N L is small);
//   * F^H in one column-pass / row-pass pair over all channels, or in channel
//     chunks sized to keep the intermediate in L2.
// Choices are cached per process by (grid, L, visibilities, precision, flags),
// so plans of the same shape skip the timing.
namespace {
struct TuneKey {
    int Kx, Ky, L, prec;
    unsigned flags;
    int64_t M;
    bool operator<(const TuneKey& o) const {
        return std::tie(Kx, Ky, L, prec, flags, M) < std::tie(o.Kx, o.Ky, o.L, o.prec, o.flags, o.M);
    }
};
struct TuneVal {
    int gram_tc, hmax, cap, rows, rcap, coop, fft_chunk;
    double grid_ms[3], gram_ms[2], fft_ms[2];
};
std::mutex g_tune_mu;
std::map<TuneKey, TuneVal> g_tune_cache;
}  // namespace

static hs_status time_ms(cudaStream_t s, int reps, const std::function<hs_status()>& fn, double* out) {
    HS_TRY(fn());   // warm-up
    cudaEvent_t e0, e1;
    HS_CHECK_CUDA(cudaEventCreate(&e0));
    HS_CHECK_CUDA(cudaEventCreate(&e1));
    hs_status st = HS_OK;
    HS_CHECK_CUDA(cudaEventRecord(e0, s));
    for (int r = 0; r < reps && st == HS_OK; ++r) st = fn();
    HS_CHECK_CUDA(cudaEventRecord(e1, s));
    HS_CHECK_CUDA(cudaEventSynchronize(e1));
    float ms = 0.f;
    HS_CHECK_CUDA(cudaEventElapsedTime(&ms, e0, e1));
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    *out = ms / reps;
    return st;
}

static TuneKey tune_key(const Plan* p) {
    return {p->g.Kx, p->g.Ky, p->g.L, (int)p->prec, p->flags | (p->half ? 0u : 0x80000000u), p->M_total};
}

// Choices of an earlier plan of the same shape, before the lists are built (they are
// then built once).
static void take_tuned(Plan* p) {
    if (p->flags & HS_PLAN_NO_TUNE) return;
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto it = g_tune_cache.find(tune_key(p));
    if (it == g_tune_cache.end()) return;
    const TuneVal& v = it->second;
    p->gram_tc = v.gram_tc;
    p->fft_adj_chunk = v.fft_chunk;
    p->sweep_hmax = v.hmax;
    p->sweep_cap = v.cap;
    p->sw_rows = v.rows;
    p->sw_cap = v.rcap;
    p->sw_coop = v.coop;
    std::copy(v.grid_ms, v.grid_ms + 3, p->tune_grid_ms);
    std::copy(v.gram_ms, v.gram_ms + 2, p->tune_gram_ms);
    std::copy(v.fft_ms, v.fft_ms + 2, p->tune_fft_ms);
    p->tuned = 2;
}

static hs_status autotune(Plan* p, cudaStream_t s) {
    const auto t0 = std::chrono::steady_clock::now();
    const bool sweep = sweep_grid(p);
    if (p->tuned == 2) return HS_OK;   // taken from the cache
    const int L = p->g.L;
    const int64_t N = p->N();
    const int reps = 3;
    if (sweep && !(p->flags & HS_PLAN_COMPENSATED) && p->M_total > 0) {
        static const int cand[3][2] = {{32, 512}, {64, 1024}, {128, 2048}};
        HS_CHECK_CUDA(cudaMemsetAsync(p->vis, 0, (size_t)p->M_total * p->csize(), s));
        int best = -1;
        auto time_lists = [&](int rows, int cap, int coop, double* ms) -> hs_status {
            p->sw_rows = rows;
            p->sw_cap = cap;
            p->sw_coop = coop;
            HS_TRY(build_sweep(p));
            GridArgs a{};
            a.mode = GIN_SORTED;
            a.in = p->vis;
            return time_ms(s, reps, [&]() { return grid(p, a, s); }, ms);
        };
        for (int c = 0; c < 3; ++c) {
            HS_TRY(time_lists(cand[c][0], cand[c][1], 0, &p->tune_grid_ms[c]));
            if (best < 0 || p->tune_grid_ms[c] < p->tune_grid_ms[best]) best = c;
        }
        p->sweep_hmax = cand[best][0];
        p->sweep_cap = cand[best][1];
        int form[3] = {p->sweep_hmax, p->sweep_cap, 0};
        if (p->half) {   // several warps to an item: kept when it gains more than 3 %
            static const int shared[4][2] = {{64, 4}, {32, 4}, {32, 8}, {16, 8}};   // rows, warps
            double t = 0.97 * p->tune_grid_ms[best];
            for (const auto& q : shared) {
                double ms = 0.0;
                HS_TRY(time_lists(q[0], SWEEP_CAP * q[1], q[1], &ms));
                if (ms < t) {
                    t = ms;
                    form[0] = q[0];
                    form[1] = SWEEP_CAP * q[1];
                    form[2] = q[1];
                }
            }
        }
        p->sw_coop = form[2];
        if (p->sw_rows != form[0] || p->sw_cap != form[1]) {
            p->sw_rows = form[0];
            p->sw_cap = form[1];
            HS_TRY(build_sweep(p));
        }
    }
    if (p->half && p->prec == HS_F32 && !(p->flags & HS_PLAN_GRAM_FMA) && L <= MAX_L_NUC) {
        HS_CHECK_CUDA(cudaMemsetAsync(p->xbuf, 0, (size_t)L * N * p->rsize(), s));
        HS_CHECK_CUDA(cudaMemsetAsync(p->xbuf2, 0, (size_t)L * N * p->rsize(), s));
        for (int c = 0; c < 2; ++c) {
            p->gram_tc = c == 0;
            HS_TRY(time_ms(s, reps, [&]() { return gram_matrix(p, p->xbuf, p->xbuf2, s); }, &p->tune_gram_ms[c]));
        }
        p->gram_tc = p->tune_gram_ms[0] <= p->tune_gram_ms[1];
    }
    if (!(p->flags & HS_PLAN_FFT_CHUNKED)) {   // F^H: all channels in one pass pair, or L2-sized channel chunks
        const int C = fft_adjoint_chunk(p);
        if (C < L) {
            p->fft_adj_chunk = 0;
            HS_TRY(time_ms(s, reps, [&]() { return fft_adjoint(p, p->xbuf, s); }, &p->tune_fft_ms[0]));
            p->fft_adj_chunk = C;
            HS_TRY(time_ms(s, reps, [&]() { return fft_adjoint(p, p->xbuf, s); }, &p->tune_fft_ms[1]));
            if (p->tune_fft_ms[1] >= p->tune_fft_ms[0]) p->fft_adj_chunk = 0;
        }
    }
    HS_CHECK_CUDA(cudaStreamSynchronize(s));
    {
        std::lock_guard<std::mutex> lock(g_tune_mu);
        TuneVal v{p->gram_tc, p->sweep_hmax, p->sweep_cap, p->sw_rows, p->sw_cap, p->sw_coop, p->fft_adj_chunk, {}, {}, {}};
        std::copy(p->tune_grid_ms, p->tune_grid_ms + 3, v.grid_ms);
        std::copy(p->tune_gram_ms, p->tune_gram_ms + 2, v.gram_ms);
        std::copy(p->tune_fft_ms, p->tune_fft_ms + 2, v.fft_ms);
        g_tune_cache[tune_key(p)] = v;
    }
    p->tuned = 1;
    p->tune_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    return HS_OK;
}

// Tables that depend on the grid alone: kernel pieces, Z scale, twiddles, channel offsets.
static hs_status build_tables(Plan* p) {
    const Geo& g = p->g;
    const int Kx = g.Kx, Ky = g.Ky;
    HS_TRY(upload(p, (void**)&p->off_d, p->off_h));
    std::vector<double> kbc;
    p->kb_terms = p->prec == HS_F32 ? KB_TERMS_F32 : KB_TERMS_F64;
    p->kb_fit_err = kb_poly_fit(p->J, p->beta, p->kb_terms, &kbc);
    p->kbc_h = kbc;
    std::vector<double> cx(g.nx), cy(g.ny);
    for (int i = 0; i < g.nx; ++i) cx[i] = 1.0 / kb_phihat((double)(i - g.nx / 2) / Kx, p->J, p->beta);
    for (int i = 0; i < g.ny; ++i) cy[i] = 1.0 / kb_phihat((double)(i - g.ny / 2) / Ky, p->J, p->beta);
    std::vector<double> twx(2 * (size_t)Kx), twy(2 * (size_t)Ky);
    for (int m = 0; m < Kx; ++m) {
        twx[2 * m] = std::cos(2.0 * M_PI * m / Kx);
        twx[2 * m + 1] = -std::sin(2.0 * M_PI * m / Kx);
    }
    for (int m = 0; m < Ky; ++m) {
        twy[2 * m] = std::cos(2.0 * M_PI * m / Ky);
        twy[2 * m + 1] = -std::sin(2.0 * M_PI * m / Ky);
    }
    if (p->prec == HS_F32) {
        HS_TRY(upload_real<float>(p, &p->kbc, kbc));
        HS_TRY(upload_real<float>(p, &p->cxs, cx));
        HS_TRY(upload_real<float>(p, &p->cys, cy));
        HS_TRY(upload_real<float>(p, &p->twx, twx));
        HS_TRY(upload_real<float>(p, &p->twy, twy));
    } else {
        HS_TRY(upload_real<double>(p, &p->kbc, kbc));
        HS_TRY(upload_real<double>(p, &p->cxs, cx));
        HS_TRY(upload_real<double>(p, &p->cys, cy));
        HS_TRY(upload_real<double>(p, &p->twx, twx));
        HS_TRY(upload_real<double>(p, &p->twy, twy));
    }
    return HS_OK;
}

// Everything of a plan that depends on the coverage and on the plane kept (half
// or whole): sorted order, coordinates, work lists, tables, grid scratch.
// uvh, wh, uh: caller order (wh, uh empty for 1).
static hs_status build_layout(Plan* p, const std::vector<double>& uvh, const std::vector<double>& wh,
                              const std::vector<double>& uh, cudaStream_t s) {
    Geo& g = p->g;
    const int L = g.L;
    const int64_t M = p->M_total;
    g.Kc = p->half ? g.nx + 8 : g.Kx;
    g.Kw = p->half ? (g.Kc + GRID_TILE - 1) / GRID_TILE * GRID_TILE : g.Kx;
    g.kwm = pow2(g.Kw) ? g.Kw - 1 : -1;
    g.tx = std::min(GRID_TILE, g.Kw);
    g.ty = std::min(GRID_TILE, g.Ky);
    g.ntx = g.Kw / g.tx;
    g.nty = g.Ky / g.ty;
    const int Kx = g.Kx, Ky = g.Ky, TX = g.tx, TY = g.ty;
    // per-visibility cells and fractions (FP64, same expression as t = u K / (2 pi)).
    // Half plane: samples with u < 0 are mirrored to (-u, -v): the window of -t is the mirror image of
    // the window of t, cells floor(t) - 3 .. floor(t) + 4 reversed, also on a cell
    // (t an integer), where the fraction of the mirrored sample is 1. cellx is the window's
    // start column in memory (kx = floor(t) - 3: column floor(t) of the half plane, kx mod Kx
    // of the whole one), celly the cell floor(t) mod Ky.
    std::vector<int> cellx(M), celly(M);
    std::vector<double> fx(M), fy(M);
    std::vector<uint8_t> mirrored(M);
    parallel_for(p->nblk, M, [&](int kb) {
        for (int64_t i = p->blk_off_h[kb]; i < p->blk_off_h[kb + 1]; ++i) {
            double tu = uvh[2 * i] * Kx / (2.0 * M_PI);
            double tv = uvh[2 * i + 1] * Ky / (2.0 * M_PI);
            const bool mir = p->half && tu < 0.0;
            if (mir) {
                tu = -tu;
                tv = -tv;
            }
            double flu = std::floor(tu), flv = std::floor(tv);
            fx[i] = tu - flu;
            fy[i] = tv - flv;
            if (mir && fx[i] == 0.0) {
                flu -= 1.0;
                fx[i] = 1.0;
            }
            if (mir && fy[i] == 0.0) {
                flv -= 1.0;
                fy[i] = 1.0;
            }
            mirrored[i] = mir;
            cellx[i] = p->half ? (int)flu : modk((int64_t)flu - 3, Kx);
            celly[i] = modk((int64_t)flv, Ky);
        }
    });
    // sort each block (each channel without blocks) by (tile of the window start, cell)
    std::vector<int> perm(M);
    parallel_for(p->nblk, M, [&](int kb) {
        std::vector<uint64_t> keys;
        const int64_t a = p->blk_off_h[kb], b = p->blk_off_h[kb + 1];
        keys.resize(b - a);
        for (int64_t i = a; i < b; ++i) {
            const int k0x = cellx[i], k0y = modk(celly[i] - 3, Ky);
            const uint64_t tile = (uint64_t)(k0y / TY) * g.ntx + (uint64_t)(k0x / TX);
            const uint64_t key = (tile * TY + (uint64_t)(k0y % TY)) * TX + (uint64_t)(k0x % TX);
            keys[i - a] = (key << 32) | (uint64_t)(i - a);
        }
        std::sort(keys.begin(), keys.end());
        for (int64_t r = 0; r < b - a; ++r) perm[a + r] = (int)(a + (int64_t)(keys[r] & 0xffffffffu));
    });
    {
        std::vector<uint32_t> pm(M);
        for (int64_t r = 0; r < M; ++r) pm[r] = (uint32_t)perm[r] | (mirrored[perm[r]] ? PERM_MIRROR : 0u);
        HS_TRY(upload(p, (void**)&p->perm, pm));
    }
    if (p->nblk != L) {   // block of every sorted visibility (gridding scale lookup)
        std::vector<int> bid(M);
        for (int kb = 0; kb < p->nblk; ++kb)
            for (int64_t r = p->blk_off_h[kb]; r < p->blk_off_h[kb + 1]; ++r) bid[r] = kb;
        HS_TRY(upload(p, (void**)&p->blk_id, bid));
    }
    // de-gridding work items: runs of one window-start tile in each block's
    // sorted range (cells before the fixed-point carry, as in the sort key), split
    // into chunks of at most DEGRID_CHUNK visibilities; slot = block * items_max + k
    {
        std::vector<int> items;
        const int nb = p->nblk;
        std::vector<std::vector<int>> b_items(nb);
        const int64_t ntl = (int64_t)g.ntx * g.nty;
        parallel_for(nb, M, [&](int kb) {
            const int l = p->blk_ch[kb];
            const int64_t a = p->blk_off_h[kb], b = p->blk_off_h[kb + 1];
            int64_t r = a;
            while (r < b) {
                auto tile_of = [&](int64_t rr) {
                    const int64_t i = perm[rr];
                    const int k0x = cellx[i], k0y = modk(celly[i] - 3, Ky);
                    return (int64_t)(k0y / TY) * g.ntx + k0x / TX;
                };
                const int64_t t = tile_of(r);
                int64_t e = r + 1;
                while (e < b && tile_of(e) == t) ++e;
                for (int64_t c0 = r; c0 < e; c0 += DEGRID_CHUNK) {
                    const int64_t c1 = std::min<int64_t>(e, c0 + DEGRID_CHUNK);
                    b_items[kb].insert(b_items[kb].end(), {(int)(l * ntl + t), (int)c0, (int)c1, kb});
                }
                r = e;
            }
        });
        int mx = 1;
        for (int kb = 0; kb < nb; ++kb) {
            mx = std::max(mx, (int)(b_items[kb].size() / 4));
            items.insert(items.end(), b_items[kb].begin(), b_items[kb].end());
        }
        std::vector<int> seen(nb, 0);
        for (size_t k = 0; k < items.size(); k += 4) {   // slot = block * items_max + rank in block
            const int kb = items[k + 3];
            items[k + 3] = kb * mx + seen[kb]++;
        }
        p->dg_items_max = mx;
        p->n_dg_items = (int64_t)items.size() / 4;
        HS_TRY(upload(p, &p->dg_items, items));
    }

    if (p->prec == HS_F32) {
        std::vector<uint32_t> c((size_t)2 * M);
        parallel_for(p->nblk, M, [&](int kb) {
        for     (int64_t r = p->blk_off_h[kb]; r < p->blk_off_h[kb + 1]; ++r) {
                const int64_t i = perm[r];
                int cxv = cellx[i], cyv = celly[i];
                uint64_t qx = (uint64_t)std::llround(std::ldexp(fx[i], g.fbx));
                uint64_t qy = (uint64_t)std::llround(std::ldexp(fy[i], g.fby));
                if (qx >= (1ull << g.fbx)) {
                    qx = 0;
                    cxv = p->half ? cxv + 1 : modk(cxv + 1, Kx);   // half plane: at most Kx / 2
                }
                if (qy >= (1ull << g.fby)) {
                    qy = 0;
                    cyv = modk(cyv + 1, Ky);
                }
                c[2 * r] = ((uint32_t)cxv << g.fbx) | (uint32_t)qx;
                c[2 * r + 1] = ((uint32_t)cyv << g.fby) | (uint32_t)qy;
                cellx[i] = cxv;   // tile membership below uses the stored cell
                celly[i] = cyv;
            }
        });
        HS_TRY(upload(p, &p->coords, c));
    } else {
        std::vector<Coord64> c(M);
        for (int64_t r = 0; r < M; ++r) {
            const int64_t i = perm[r];
            c[r].fx = fx[i];
            c[r].fy = fy[i];
            c[r].cx = cellx[i];
            c[r].cy = celly[i];
        }
        HS_TRY(upload(p, &p->coords, c));
    }
    // cells that each channel's windows reach, from the stored start cells
    p->rng_h.resize(L);
    parallel_for(L, M, [&](int l) {
        int xmax = 0, xmin = 0, ymax = 0, ymin = 0;   // [xmin, xmax) around frequency 0
        for (int64_t i = p->off_h[l]; i < p->off_h[l + 1]; ++i) {
            const int x = cellx[i], y = modk(celly[i] - 3, Ky);
            const int sx = (!p->half && x >= Kx / 2) ? x - Kx : x, sy = y >= Ky / 2 ? y - Ky : y;
            xmax = std::max(xmax, sx + 8);
            xmin = std::min(xmin, sx);
            ymax = std::max(ymax, sy + 8);
            ymin = std::min(ymin, sy);
        }
        const int ncol = p->half ? g.Kw : Kx;
        p->rng_h[l] = {std::min((xmax + 7) / 8 * 8, ncol), xmin < 0 ? (ncol + xmin) / 8 * 8 : ncol,
                       std::min(ymax, Ky), Ky + ymin};
    });
    HS_TRY(upload(p, (void**)&p->rng, p->rng_h));
    if (!wh.empty()) {
        std::vector<double> ws(M);
        for (int64_t r = 0; r < M; ++r) ws[r] = wh[perm[r]];
        HS_TRY(p->prec == HS_F32 ? upload_real<float>(p, &p->w_sorted, ws)
                                 : upload_real<double>(p, &p->w_sorted, ws));
    }
    if (!uh.empty()) {
        std::vector<double> us(M);
        for (int64_t r = 0; r < M; ++r) us[r] = uh[perm[r]];
        HS_TRY(p->prec == HS_F32 ? upload_real<float>(p, &p->u_sorted, us)
                                 : upload_real<double>(p, &p->u_sorted, us));
    }

    // gridding lists: the sweep kernel's for grids of at least 64 x 64 cells;
    // per-tile lists for smaller grids and the compensated kernel
    take_tuned(p);
    const bool sweep = sweep_grid(p);
    if (sweep) {
        p->k0x_h.resize(M);
        p->k0y_h.resize(M);
        for (int64_t r = 0; r < M; ++r) {
            p->k0x_h[r] = cellx[perm[r]];
            p->k0y_h[r] = modk(celly[perm[r]] - 3, Ky);
        }
        HS_TRY(build_sweep(p));
    }
    if (!sweep || (p->flags & HS_PLAN_COMPENSATED)) {
        // gridding lists: every (channel, tile) overlapped by a window
        const int64_t nt = p->ntiles();
        std::vector<int64_t> toff((size_t)L * nt + 1, 0);
        auto tiles_of = [&](int64_t r, int* txs, int* tys, int& ntx_, int& nty_) {
            const int64_t i = perm[r];
            const int k0x = cellx[i], k0y = modk(celly[i] - 3, Ky);
            txs[0] = k0x / TX;
            txs[1] = modk(k0x + 7, g.Kw) / TX;
            tys[0] = k0y / TY;
            tys[1] = modk(k0y + 7, Ky) / TY;
            ntx_ = txs[1] != txs[0] ? 2 : 1;
            nty_ = tys[1] != tys[0] ? 2 : 1;
        };
        for (int l = 0; l < L; ++l)
            for (int64_t r = p->off_h[l]; r < p->off_h[l + 1]; ++r) {
                int txs[2], tys[2], a, b;
                tiles_of(r, txs, tys, a, b);
                for (int yy = 0; yy < b; ++yy)
                    for (int xx = 0; xx < a; ++xx) ++toff[1 + (size_t)l * nt + tys[yy] * g.ntx + txs[xx]];
            }
        for (size_t k = 1; k < toff.size(); ++k) toff[k] += toff[k - 1];
        if (toff.back() >= ((int64_t)1 << 30)) return fail(HS_ERR_ARG, "too many gridding list entries");
        std::vector<int> ent((size_t)toff.back());
        {
            std::vector<int64_t> fill(toff.begin(), toff.end() - 1);
            for (int l = 0; l < L; ++l)
                for (int64_t r = p->off_h[l]; r < p->off_h[l + 1]; ++r) {
                    int txs[2], tys[2], a, b;
                    tiles_of(r, txs, tys, a, b);
                    for (int yy = 0; yy < b; ++yy)
                        for (int xx = 0; xx < a; ++xx)
                            ent[fill[(size_t)l * nt + tys[yy] * g.ntx + txs[xx]]++] = (int)r;
                }
        }
        // Regroup every list into groups of 4 entries whose windows do not overlap
        // (circular distance >= 8 cells in x or y), padding with -1, so that the
        // gridding kernel can add the 4 windows of a group at once without atomics.
        // Greedy, in list order: an entry joins the first open group it fits; at
        // most GROUP_OPEN groups are open, the oldest is closed (padded) to make room.
        std::vector<int64_t> goff((size_t)L * nt + 1, 0);
        std::vector<int> gent;
        gent.reserve((size_t)(toff.back() + toff.back() / 4 + 64));
        {
            constexpr int GROUP_OPEN = 64;
            struct Group {
                int m;
                int e[4], x[4], y[4];
            };
            auto circ = [](int d, int K) {
                d &= K - 1;
                return d < K - d ? d : K - d;
            };
            auto circx = [&](int d) { return p->half ? std::abs(d) : circ(d, Kx); };
            std::vector<Group> open;
            auto emit = [&](const Group& g) {
                for (int k = 0; k < 4; ++k) gent.push_back(k < g.m ? g.e[k] : -1);
            };
            for (int64_t tix = 0; tix < (int64_t)L * nt; ++tix) {
                open.clear();
                for (int64_t q = toff[tix]; q < toff[tix + 1]; ++q) {
                    const int r = ent[q];
                    const int64_t i = perm[r];
                    const int x = cellx[i], y = modk(celly[i] - 3, Ky);
                    bool placed = false;
                    for (size_t gi = 0; gi < open.size() && !placed; ++gi) {
                        Group& g = open[gi];
                        bool fits = true;
                        for (int k = 0; k < g.m && fits; ++k)
                            fits = circx(x - g.x[k]) >= 8 || circ(y - g.y[k], Ky) >= 8;
                        if (!fits) continue;
                        g.e[g.m] = r;
                        g.x[g.m] = x;
                        g.y[g.m] = y;
                        if (++g.m == 4) {
                            emit(g);
                            open.erase(open.begin() + gi);
                        }
                        placed = true;
                    }
                    if (placed) continue;
                    if ((int)open.size() == GROUP_OPEN) {
                        emit(open.front());
                        open.erase(open.begin());
                    }
                    Group g{};
                    g.m = 1;
                    g.e[0] = r;
                    g.x[0] = x;
                    g.y[0] = y;
                    open.push_back(g);
                }
                for (const Group& g : open) emit(g);
                goff[tix + 1] = (int64_t)gent.size();
            }
        }
        p->n_ent = goff.back();
        if (p->n_ent >= ((int64_t)1 << 31)) return fail(HS_ERR_ARG, "too many gridding list entries");
        HS_TRY(upload(p, (void**)&p->tile_off, goff));
        HS_TRY(upload(p, (void**)&p->tile_ent, gent));
        // work items: lists longer than GRID_CAP entries are split at group
        // boundaries; split tiles are merged
        {
            std::vector<int> items, merges;
            int slots = 0;
            for (int64_t tix = 0; tix < (int64_t)L * nt; ++tix) {
                const int64_t a = goff[tix], b = goff[tix + 1];
                const int64_t ng = (b - a) / 4;
                const int parts = ng * 4 <= GRID_CAP ? 1 : (int)((ng * 4 + GRID_CAP - 1) / GRID_CAP);
                if (parts == 1) {
                    items.insert(items.end(), {(int)tix, (int)a, (int)b, -1});
                } else {
                    merges.insert(merges.end(), {(int)tix, slots, parts});
                    for (int k = 0; k < parts; ++k) {
                        const int64_t e0 = a + 4 * (ng * k / parts), e1 = a + 4 * (ng * (k + 1) / parts);
                        items.insert(items.end(), {(int)tix, (int)e0, (int)e1, slots + k});
                    }
                    slots += parts;
                }
            }
            p->n_items = (int64_t)items.size() / 4;
            p->n_merges = (int64_t)merges.size() / 3;
            HS_TRY(upload(p, &p->grid_items, items));
            HS_TRY(upload(p, &p->grid_merges, merges));
            HS_TRY(plan_alloc(p, &p->grid_partial, (size_t)std::max(slots, 1) * g.tx * g.ty * p->csize()));
        }
    }
    if (sweep && !(p->flags & HS_PLAN_COMPENSATED)) p->n_ent = p->n_sw_ent;
    if (p->half) {   // the whole-plane layout of the same plan uses these tables and this scratch (plane_plan)
        HS_TRY(build_tables(p));
        const bool wide = p->prec == HS_F32 && L <= MAX_L_NUC;
        HS_TRY(plan_alloc(p, &p->grid, (size_t)L * Ky * (wide ? Kx : g.Kw) * p->csize()));
        HS_TRY(plan_alloc(p, &p->tmp, (size_t)L * g.ny * (wide ? Kx : g.Kc) * p->csize()));
        HS_TRY(plan_alloc(p, &p->vis, (size_t)std::max<int64_t>(M, 1) * p->csize()));
    }
    HS_CHECK_CUDA(cudaStreamCreateWithFlags(&p->fft_side, cudaStreamNonBlocking));
    HS_CHECK_CUDA(cudaEventCreateWithFlags(&p->fft_ev_col, cudaEventDisableTiming));
    HS_CHECK_CUDA(cudaEventCreateWithFlags(&p->fft_ev_join, cudaEventDisableTiming));
    HS_TRY(fft_prepare(p));
    if ((p->flags & HS_PLAN_FFT_CHUNKED) && p->tuned != 2) p->fft_adj_chunk = fft_adjoint_chunk(p);
    return HS_OK;
}

// Room for the tap tables of an FP64 plan (128 bytes per visibility, up to TAPS_MAX). They are
// taken from memory nobody asked for: under a device limit only where the half plane saves as
// much of the grid scratch, so that a plan never takes the room of the states and plans that
// fit beside one with the whole plane and no tables; without a limit while half of the device's memory
// stays free.
static bool taps_fit(const Plan* p) {
    const Geo& g = p->g;
    const int64_t need = 16 * 8 * p->M_total;
    if (need > TAPS_MAX) return false;
    const int64_t saved = (int64_t)g.L * ((int64_t)g.Ky * (g.Kx - g.Kw) + (int64_t)g.ny * (g.Kx - g.Kc)) * (int64_t)p->csize() -
                          (int64_t)(g.L * sizeof(int4));
    if (need <= saved) return true;
    size_t avail = 0, total = 0;
    return device_limit() == 0 && cudaMemGetInfo(&avail, &total) == cudaSuccess && avail >= total / 2 + (size_t)need;
}

static hs_status build(Plan* p, const int64_t* vis_offsets, int nblocks, const int64_t* block_offsets,
                       const void* uv, const void* weights, const void* precond, cudaStream_t s) {
    Geo& g = p->g;
    const int L = g.L;
    p->off_h.assign(vis_offsets, vis_offsets + L + 1);
    if (p->off_h[0] != 0) return fail(HS_ERR_ARG, "vis_offsets[0] must be 0");
    int64_t Mmax = 0;
    for (int l = 0; l < L; ++l) {
        const int64_t m = p->off_h[l + 1] - p->off_h[l];
        if (m < 0) return fail(HS_ERR_ARG, "vis_offsets must be nondecreasing (channel %d)", l);
        Mmax = std::max(Mmax, m);
    }
    const int64_t M = p->off_h[L];
    if (M >= ((int64_t)1 << 31)) return fail(HS_ERR_ARG, "total visibilities must be < 2^31");
    if (M > 0 && uv == nullptr) return fail(HS_ERR_ARG, "uv is null");
    p->M_total = M;
    p->Mmax = (int)Mmax;
    // data blocks (Sec. 2.1, M_l^b): contiguous caller ranges inside channels
    if (block_offsets == nullptr) {
        p->blk_off_h = p->off_h;
    } else {
        if (nblocks < L) return fail(HS_ERR_ARG, "nblocks (%d) must be >= L (%d)", nblocks, L);
        p->blk_off_h.assign(block_offsets, block_offsets + nblocks + 1);
        if (p->blk_off_h[0] != 0 || p->blk_off_h[nblocks] != M)
            return fail(HS_ERR_ARG, "block_offsets must run from 0 to the total visibility count");
        for (int k = 0; k < nblocks; ++k)
            if (p->blk_off_h[k + 1] < p->blk_off_h[k]) return fail(HS_ERR_ARG, "block_offsets must be nondecreasing");
        for (int l = 1; l < L; ++l)   // every channel boundary must be a block boundary
            if (!std::binary_search(p->blk_off_h.begin(), p->blk_off_h.end(), p->off_h[l]))
                return fail(HS_ERR_ARG, "block_offsets must contain every channel boundary (channel %d)", l);
    }
    p->nblk = (int)p->blk_off_h.size() - 1;
    p->blk_ch.assign(p->nblk, 0);
    for (int k = 0; k < p->nblk; ++k) {   // channel of a block: the last channel starting at or before it
        const int64_t x = p->blk_off_h[k];
        const int l = (int)(std::upper_bound(p->off_h.begin(), p->off_h.end() - 1, x) - p->off_h.begin()) - 1;
        p->blk_ch[k] = std::max(0, std::min(L - 1, l));
    }

    std::vector<double> uvh, wh, uh;
    HS_TRY(download_real(p, uv, 2 * M, uvh, s));
    if (weights) HS_TRY(download_real(p, weights, M, wh, s));
    if (precond) HS_TRY(download_real(p, precond, M, uh, s));
    for (int64_t i = 0; i < 2 * M; ++i) {
        const double v = uvh[i];
        if (!std::isfinite(v) || v < -M_PI || v >= M_PI)
            return fail(HS_ERR_ARG, "uv[%lld] = %g outside [-pi, pi)", (long long)(i / 2), v);
    }
    for (int64_t i = 0; i < (int64_t)uh.size(); ++i)
        if (!(uh[i] > 0.0) || !std::isfinite(uh[i]))
            return fail(HS_ERR_ARG, "precond[%lld] must be finite and > 0", (long long)i);

    HS_TRY(build_layout(p, uvh, wh, uh, s));
    if (p->prec == HS_F32 && L <= MAX_L_NUC) p->uv_h.assign(uvh.begin(), uvh.end());   // exact: FP32 inputs

    // scratch
    const size_t rs = p->rsize(), cs = p->csize();
    const int64_t N = p->N();
    // lowpass blocks between wavelet levels: the finest a level reads or writes is N / 4
    HS_TRY(plan_alloc(p, &p->dwt_a, (size_t)NW * L * (N / 4) * rs));
    HS_TRY(plan_alloc(p, &p->dwt_b, (size_t)NW * L * (N / 4) * rs));
    HS_TRY(plan_alloc(p, &p->xbuf, (size_t)L * N * rs));
    HS_TRY(plan_alloc(p, &p->xbuf2, (size_t)L * N * rs));
    const int64_t nbx = (Mmax + DEGRID_CHUNK - 1) / DEGRID_CHUNK;
    p->part_n = std::max<int64_t>({(int64_t)L * std::max<int64_t>(nbx, 1),
                                   gram_part_doubles(std::min(L, MAX_L_NUC)), 8192});
    HS_TRY(plan_alloc(p, (void**)&p->part, (size_t)p->part_n * sizeof(double)));
    HS_TRY(plan_alloc(p, (void**)&p->gram, sizeof(double) * MAX_L_NUC * MAX_L_NUC));
    HS_TRY(plan_alloc(p, (void**)&p->eigf, sizeof(double) * LR_TOTAL_DOUBLES));
    HS_TRY(plan_alloc(p, (void**)&p->sv, sizeof(double) * MAX_L_NUC));
    HS_TRY(plan_alloc(p, (void**)&p->dscal, sizeof(double) * 6 * std::max(L, 1)));
    HS_TRY(plan_alloc(p, (void**)&p->err_d, sizeof(int)));
    HS_CHECK_CUDA(cudaMemsetAsync(p->err_d, 0, sizeof(int), s));
    if (p->prec == HS_F64 && M > 0 && taps_fit(p)) {   // optional: else the taps are evaluated
        if (plan_alloc(p, &p->taps, (size_t)M * 16 * sizeof(double)) == HS_OK) HS_TRY(nufft_taps(p, s));
        else clear_error();
    }
    if (p->flags & HS_PLAN_GRAM_FMA) p->gram_tc = 0;
    if (!(p->flags & HS_PLAN_NO_TUNE)) HS_TRY(autotune(p, s));
    p->k0x_h.clear();
    p->k0y_h.clear();
    p->k0x_h.shrink_to_fit();
    p->k0y_h.shrink_to_fit();
    HS_CHECK_CUDA(cudaStreamSynchronize(s));
    return HS_OK;
}

hs_status plan_create(Plan** out, int nx, int ny, int L, const int64_t* vis_offsets, int nblocks,
                      const int64_t* block_offsets, const void* uv, const void* weights, const void* precond,
                      int oversample, int J, double kb_beta, int levels, hs_prec prec, unsigned flags,
                      cudaStream_t s) {
    if (out == nullptr) return fail(HS_ERR_ARG, "out is null");
    *out = nullptr;
    if (vis_offsets == nullptr) return fail(HS_ERR_ARG, "vis_offsets is null");
    if (!side_ok(nx) || !side_ok(ny))
        return fail(HS_ERR_ARG, "nx, ny must be in [16, 2048] and powers of two, or 3 or 5 times a power of two "
                                "and multiples of 16 (got %d x %d)", nx, ny);
    if (L < 1 || L > 1024) return fail(HS_ERR_ARG, "L must be in [1, 1024] (got %d)", L);
    if (oversample != 2) return fail(HS_ERR_ARG, "oversample must be 2 (got %d)", oversample);
    if (J != 8) return fail(HS_ERR_ARG, "J must be 8 (got %d)", J);
    if (levels < 1 || levels > 8 || (nx >> levels) < 1 || (ny >> levels) < 1 ||
        nx % (1 << levels) || ny % (1 << levels))
        return fail(HS_ERR_ARG, "wavelet_levels %d incompatible with %d x %d", levels, nx, ny);
    for (int lev = 0; lev < levels; ++lev) {   // DWT tiles: 16 coefficients per subband side, or one tile
        const int hy = ny >> (lev + 1), hx = nx >> (lev + 1);
        if ((hy >= 16 && hy % 16) || (hx >= 16 && hx % 16))
            return fail(HS_ERR_ARG, "wavelet_levels %d: level %d subbands of %d x %d are not multiples of 16",
                        levels, lev, hy, hx);
    }
    if (prec != HS_F32 && prec != HS_F64) return fail(HS_ERR_ARG, "bad precision %d", (int)prec);
    if (flags & ~(unsigned)(HS_PLAN_COMPENSATED | HS_PLAN_GRAM_FMA | HS_PLAN_NO_TUNE | HS_PLAN_FFT_CHUNKED))
        return fail(HS_ERR_ARG, "unknown plan flags 0x%x", flags);
    HS_TRY(dwt_init());
    HS_TRY(fft_init());
    HS_TRY(nufft_init());
    HS_TRY(prox_init());
    HS_TRY(eig_init());
    std::unique_ptr<Plan> p(new Plan());
    p->prec = prec;
    p->flags = flags;
    p->levels = levels;
    p->J = J;
    p->o = oversample;
    p->beta = kb_beta > 0 ? kb_beta
                          : M_PI * std::sqrt((double)(J * J) / (oversample * oversample) *
                                                 (oversample - 0.5) * (oversample - 0.5) - 0.8);
    Geo& g = p->g;
    g.nx = nx;
    g.ny = ny;
    g.L = L;
    g.Kx = oversample * nx;
    g.Ky = oversample * ny;
    g.fbx = std::min(23, 32 - ilog2(g.Kx));
    g.fby = std::min(23, 32 - ilog2(g.Ky));
    g.kym = pow2(g.Ky) ? g.Ky - 1 : -1;
    const hs_status st =
        no_throw([&]() { return build(p.get(), vis_offsets, nblocks, block_offsets, uv, weights, precond, s); });
    if (st != HS_OK) {
        plan_free(p.get());
        return st;
    }
    *out = p.release();
    return HS_OK;
}

// The whole-plane companion of an FP32 plan: same coverage, blocks, weights and
// flags, lists and coordinates of its own, the plan's tables and grid scratch (as the plan's own
// calls and every state on it use that, in stream order); p stays unchanged but for the
// shared reference. The plan keeps it for its next states (building it again took 38 ms per
// state at 256 x 256, L = 60, where the state itself takes 0.7), but under a device limit
// it goes with the last state that uses it.
static hs_status make_plane(Plan* p, std::shared_ptr<Plan>* out, cudaStream_t s);
hs_status plane_plan(Plan* p, std::shared_ptr<Plan>* out, cudaStream_t s) {
    return no_throw([&]() { return make_plane(p, out, s); });
}

void drop_plane(Plan* p) {
    std::lock_guard<std::mutex> lock(p->plane_mu);
    p->plane_keep.reset();
}

int64_t plane_bytes(Plan* p) {
    std::lock_guard<std::mutex> lock(p->plane_mu);
    const std::shared_ptr<Plan> c = p->plane.lock();
    return c ? c->device_bytes : 0;
}

// Under a device limit the layout only takes what the wavelet scratch between levels leaves
// of the two coefficient cubes it could be (48 bytes per pixel and channel, about 1.7 to 2
// visibilities), so that as many states and plans fit as beside one layout. Without the rule the
// first state of a denser plan took the room of the second.
static hs_status plane_room(const Plan* p, int64_t bytes) {
    const int64_t room = 2 * NW * p->g.L * (p->N() - p->N() / 4) * (int64_t)p->rsize();
    if (device_limit() == 0 || bytes <= room) return HS_OK;
    return fail(HS_ERR_NOMEM, "whole-plane layout: %lld bytes, %lld left for it under the device limit", (long long)bytes,
                (long long)room);
}

static hs_status make_plane(Plan* p, std::shared_ptr<Plan>* out, cudaStream_t s) {
    std::lock_guard<std::mutex> lock(p->plane_mu);
    *out = p->plane.lock();
    if (*out) return HS_OK;
    if (p->prec != HS_F32 || (int64_t)p->uv_h.size() != 2 * p->M_total)
        return fail(HS_ERR_STATE, "whole-plane layout: the plan keeps no coverage");
    HS_TRY(plane_room(p, 16 * p->M_total));   // coordinates, permutation and list entries: at least
    std::shared_ptr<Plan> c(new Plan(), [](Plan* q) {
        plan_free(q);
        delete q;
    });
    c->half = false;
    c->g = p->g;
    c->levels = p->levels;
    c->J = p->J;
    c->o = p->o;
    c->prec = p->prec;
    c->flags = p->flags;
    c->beta = p->beta;
    c->M_total = p->M_total;
    c->Mmax = p->Mmax;
    c->off_h = p->off_h;
    c->blk_off_h = p->blk_off_h;
    c->blk_ch = p->blk_ch;
    c->nblk = p->nblk;
    c->off_d = p->off_d;   // tables of the plan (a state never outlives it)
    c->kb_terms = p->kb_terms;
    c->kb_fit_err = p->kb_fit_err;
    c->kbc_h = p->kbc_h;
    c->kbc = p->kbc;
    c->cxs = p->cxs;
    c->cys = p->cys;
    c->twx = p->twx;
    c->twy = p->twy;
    const int64_t M = p->M_total;
    std::vector<double> uvh(p->uv_h.begin(), p->uv_h.end()), wh, uh;
    if (p->w_sorted || p->u_sorted) {   // back to caller order
        std::vector<uint32_t> pm(M);
        HS_CHECK_CUDA(cudaMemcpy(pm.data(), p->perm, M * sizeof(uint32_t), cudaMemcpyDeviceToHost));
        auto unsorted = [&](const void* d, std::vector<double>& h) -> hs_status {
            if (d == nullptr) return HS_OK;
            std::vector<float> v(M);
            HS_CHECK_CUDA(cudaMemcpy(v.data(), d, M * sizeof(float), cudaMemcpyDeviceToHost));
            h.resize(M);
            for (int64_t r = 0; r < M; ++r) h[pm[r] & ~PERM_MIRROR] = v[r];
            return HS_OK;
        };
        HS_TRY(unsorted(p->w_sorted, wh));
        HS_TRY(unsorted(p->u_sorted, uh));
    }
    HS_TRY(build_layout(c.get(), uvh, wh, uh, s));
    if (!(c->flags & HS_PLAN_NO_TUNE) && c->tuned == 0) {
        // the candidates run on scratch of their own: another state may be iterating on the plan's.
        // Without room for it the layout keeps the default choices.
        const size_t bytes[4] = {(size_t)c->g.L * c->g.Ky * c->g.Kw * c->csize(),
                                 (size_t)c->g.L * c->g.ny * c->g.Kc * c->csize(),
                                 (size_t)std::max<int64_t>(M, 1) * c->csize(), (size_t)c->g.L * c->N() * c->rsize()};
        void** const buf[4] = {&c->grid, &c->tmp, &c->vis, &c->xbuf};
        int got = 0;
        while (got < 4 && lib_alloc(buf[got], bytes[got]) == HS_OK) ++got;
        hs_status e = HS_OK;
        cudaError_t ce = cudaSuccess;
        if (got == 4) {
            e = no_throw([&]() { return autotune(c.get(), s); });
            ce = cudaStreamSynchronize(s);
        } else {
            clear_error();
        }
        for (int k = 0; k < got; ++k) lib_free(*buf[k], bytes[k]);
        c->xbuf = nullptr;
        HS_TRY(e);
        HS_CHECK_CUDA(ce);
    }
    HS_TRY(plane_room(p, c->device_bytes));
    c->grid = p->grid;
    c->tmp = p->tmp;
    c->vis = p->vis;
    c->k0x_h.clear();
    c->k0y_h.clear();
    c->k0x_h.shrink_to_fit();
    c->k0y_h.shrink_to_fit();
    HS_CHECK_CUDA(cudaStreamSynchronize(s));
    p->plane = c;
    if (!device_limit()) p->plane_keep = c;
    *out = c;
    return HS_OK;
}

}  // namespace hs
