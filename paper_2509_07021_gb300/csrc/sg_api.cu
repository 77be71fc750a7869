// C ABI of the SG-splatting rasterizer: argument checks, workspace layout and
// the launch sequence of the forward and backward passes.
#include "sg_internal.cuh"

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <memory>
#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

using namespace sgk;

namespace {
std::atomic<int64_t> &launch_counter();
}

void sgk::count_launches(int n) { launch_counter() += n; }

namespace {

thread_local char g_err[512] = "";

int fail(int code, const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}

int cuda_fail(cudaError_t e, const char *where) {
    return fail(SG_ERR_CUDA, "%s: %s (%s)", where, cudaGetErrorName(e), cudaGetErrorString(e));
}

#define SG_CUDA(call, where)                                 \
    do {                                                     \
        cudaError_t e_ = (call);                             \
        if (e_ != cudaSuccess) return cuda_fail(e_, where);  \
    } while (0)

// ---------------------------------------------------------------------------
// stage profiler: CUDA events recorded on the caller's stream
// ---------------------------------------------------------------------------
enum Stage {
    ST_SETUP = 0, ST_PRE, ST_DEPTH_SORT, ST_OFFSETS, ST_READ_PAIRS, ST_DUPLICATE, ST_TILE_SORT,
    ST_RANGES, ST_BLEND_FWD, ST_BWD_CLEAR, ST_BLEND_BWD, ST_PRE_BWD, ST_N
};
static_assert(ST_N == SG_PROFILE_STAGES, "stage count");
const char *const kStageNames[ST_N] = {"setup", "preprocess", "depth_sort", "pair_offsets",
                                       "read_pairs", "duplicate", "tile_sort", "tile_ranges",
                                       "blend_fwd", "bwd_clear", "blend_bwd", "preprocess_bwd"};

struct Profiler {
    std::mutex mu;
    int flags = 0;
    uint32_t stage_mask = 0xFFFFFFFFu;
    std::vector<cudaEvent_t> pool;
    struct Pending { int stage; cudaEvent_t a, b; };
    std::vector<Pending> pending;
    double ms[ST_N] = {};
    int64_t launches[ST_N] = {};
    int64_t evals[2] = {};
    cudaEvent_t get() {
        if (!pool.empty()) { cudaEvent_t e = pool.back(); pool.pop_back(); return e; }
        cudaEvent_t e = nullptr;
        cudaEventCreate(&e);
        return e;
    }
};
Profiler &prof() { static Profiler p; return p; }

std::atomic<int64_t> &launch_counter() {
    static std::atomic<int64_t> c{0};
    return c;
}

// Brackets one stage with events when profiling is on.
struct StageTimer {
    int stage;
    cudaStream_t s;
    cudaEvent_t a = nullptr;
    StageTimer(int st, cudaStream_t stream) : stage(st), s(stream) {
        Profiler &p = prof();
        if (!(p.flags & SG_PROFILE_EVENTS) || !((p.stage_mask >> st) & 1u)) return;
        std::lock_guard<std::mutex> g(p.mu);
        a = p.get();
        if (a) cudaEventRecord(a, s);
    }
    ~StageTimer() {
        if (!a) return;
        Profiler &p = prof();
        std::lock_guard<std::mutex> g(p.mu);
        cudaEvent_t b = p.get();
        if (!b) return;
        cudaEventRecord(b, s);
        p.pending.push_back({stage, a, b});
    }
};

// Process-wide kernel shape choices (sg_set_tuning); defaults from measurement
// (1M Gaussians at 1920x1080: both blends persistent, 4 and 8 pixels per thread;
// with fewer tiles auto_shapes lets the tile count choose, auto_pixels).
constexpr sg_tuning kDefaultTuning = {4, 8, 1, 1, 0, 0, 0, 3};
constexpr int kDefaultBatch = 64;
sg_tuning &tuning() {
    static sg_tuning t = kDefaultTuning;
    return t;
}

bool ppt_ok(int p) { return p == 1 || p == 2 || p == 4 || p == 8; }

constexpr size_t ALIGN = 256;
size_t al(size_t x) { return (x + ALIGN - 1) / ALIGN * ALIGN; }

bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

bool dtype_ok(int dg, int dl, int ds) {
    return (dg == SG_F32 && dl == SG_F32 && ds == SG_F32) ||
           (dg == SG_F16 && dl == SG_F16 && (ds == SG_F16 || ds == SG_BF16));
}

int tile_bits_for(uint64_t n_tiles) {
    if (n_tiles <= 1) return 0;
    int b = 0;
    while ((1ull << b) < n_tiles) ++b;
    return b;
}

// Fills the batch table from host structs. Pointers of the scenes are
// validated only when check_ptrs is set (the query does not need them).
int build_batch(const sg_scene *scenes, int n_scenes, const sg_camera *cams, const int32_t *view_scene,
                int n_views, bool check_ptrs, Batch &b) {
    if (!scenes || !cams) return fail(SG_ERR_INVALID_ARG, "scene and cameras must not be NULL");
    if (n_views < 1 || n_views > SG_MAX_VIEWS)
        return fail(SG_ERR_INVALID_ARG, "n_views = %d outside [1, %d]", n_views, SG_MAX_VIEWS);
    if (n_scenes < 1 || n_scenes > SG_MAX_SCENES)
        return fail(SG_ERR_INVALID_ARG, "n_scenes = %d outside [1, %d]", n_scenes, SG_MAX_SCENES);
    std::memset(&b, 0, sizeof(Batch));
    b.n_views = n_views;
    b.n_scenes = n_scenes;
    uint64_t bwd_blk = 0, runs = 0;
    for (int s = 0; s < n_scenes; ++s) {
        const sg_scene &sc = scenes[s];
        if (sc.n < 0 || sc.n > (int64_t)INT32_MAX - PRE_THREADS)
            return fail(SG_ERR_INVALID_ARG, "scene %d: n = %lld out of range", s, (long long)sc.n);
        if (sc.n_lobes < 0 || sc.n_lobes > (int64_t)INT32_MAX)
            return fail(SG_ERR_INVALID_ARG, "scene %d: n_lobes = %lld out of range", s, (long long)sc.n_lobes);
        if (!dtype_ok(sc.dtype_geom, sc.dtype_lobe, sc.dtype_sharp))
            return fail(SG_ERR_INVALID_ARG, "scene %d: unsupported dtype combination (%d, %d, %d)", s,
                        sc.dtype_geom, sc.dtype_lobe, sc.dtype_sharp);
        if (s > 0 && (sc.dtype_geom != scenes[0].dtype_geom || sc.dtype_lobe != scenes[0].dtype_lobe ||
                      sc.dtype_sharp != scenes[0].dtype_sharp || sc.color_model != scenes[0].color_model))
            return fail(SG_ERR_INVALID_ARG, "scene %d: all scenes of a call must share storage types and colour model",
                        s);
        const bool sh3 = sc.color_model == SG_COLOR_SH3;
        if (sc.color_model != SG_COLOR_SG && !sh3)
            return fail(SG_ERR_INVALID_ARG, "scene %d: unknown colour model %d", s, sc.color_model);
        if (sh3 && (sc.n_lobes != 0 || sc.dtype_geom != SG_F32))
            return fail(SG_ERR_INVALID_ARG, "scene %d: the SH3 colour model takes binary32 geometry and no lobes", s);
        if (check_ptrs && sc.n > 0) {
            const void *req_sg[] = {sc.means, sc.scales, sc.quats, sc.opac, sc.gmask, sc.c0, sc.lobe_off};
            const void *req_sh[] = {sc.means, sc.scales, sc.quats, sc.opac, sc.gmask, sc.sh, sc.sh};
            for (const void *p : (sh3 ? req_sh : req_sg))
                if (!p || !aligned(p, 16))
                    return fail(SG_ERR_INVALID_ARG, "scene %d: a Gaussian array is NULL or not 16-byte aligned", s);
        }
        if (check_ptrs && sc.n_lobes > 0) {
            const void *req[] = {sc.axis, sc.sharp, sc.amp, sc.lmask};
            for (const void *p : req)
                if (!p || !aligned(p, 16))
                    return fail(SG_ERR_INVALID_ARG, "scene %d: a lobe array is NULL or not 16-byte aligned", s);
        }
        SceneDesc &d = b.scene[s];
        d.means = sc.means; d.scales = sc.scales; d.quats = sc.quats; d.opac = sc.opac;
        d.gmask = sc.gmask; d.c0 = sc.c0; d.lobe_off = sc.lobe_off;
        d.axis = sc.axis; d.sharp = sc.sharp; d.amp = sc.amp; d.lmask = sc.lmask;
        d.sh = sc.sh;
        d.color_model = sc.color_model;
        d.n = sc.n; d.n_lobes = sc.n_lobes;
        d.dtype_geom = sc.dtype_geom; d.dtype_lobe = sc.dtype_lobe; d.dtype_sharp = sc.dtype_sharp;
        d.blk_off = (uint32_t)bwd_blk;
        bwd_blk += div_up((uint64_t)sc.n, PRE_THREADS);
        d.run_off = (uint32_t)runs;
        runs += div_up((uint64_t)sc.n, PRE_RUN);
    }
    uint64_t tiles = 0, groups = 0, pix = 0, ent = 0;
    for (int v = 0; v < n_views; ++v) {
        const sg_camera &c = cams[v];
        const int s = view_scene ? view_scene[v] : 0;
        if (s < 0 || s >= n_scenes) return fail(SG_ERR_INVALID_ARG, "view %d: scene index %d", v, s);
        if (c.width < 1 || c.height < 1 || c.width > 16 * 65535 || c.height > 16 * 65535)
            return fail(SG_ERR_INVALID_ARG, "view %d: bad image size %dx%d", v, c.width, c.height);
        if (!(c.fx > 0.f) || !(c.fy > 0.f) || !std::isfinite(c.fx) || !std::isfinite(c.fy) ||
            !std::isfinite(c.cx) || !std::isfinite(c.cy) || !(c.near_plane >= 0.f))
            return fail(SG_ERR_INVALID_ARG, "view %d: bad intrinsics", v);
        for (int i = 0; i < 12; ++i)
            if (!std::isfinite(c.viewmat[i])) return fail(SG_ERR_INVALID_ARG, "view %d: non-finite viewmat", v);
        ViewDesc &d = b.view[v];
        d.fx = c.fx; d.fy = c.fy; d.cx = c.cx; d.cy = c.cy;
        std::memcpy(d.V, c.viewmat, sizeof(d.V));
        // camera centre -R^T t (FP64 on the host)
        for (int i = 0; i < 3; ++i) {
            double acc = 0.0;
            for (int k = 0; k < 3; ++k) acc -= (double)c.viewmat[4 * k + i] * (double)c.viewmat[4 * k + 3];
            d.campos[i] = (float)acc;
        }
        d.near_plane = c.near_plane;
        d.bg[0] = c.bg[0]; d.bg[1] = c.bg[1]; d.bg[2] = c.bg[2];
        d.W = c.width; d.H = c.height;
        // one rounded operation per step, as the decision recipe states them
        const float tanx = (0.5f * (float)c.width) / c.fx, tany = (0.5f * (float)c.height) / c.fy;
        d.limx = 1.3f * tanx;
        d.limy = 1.3f * tany;
        d.tiles_x = (c.width + TILE - 1) / TILE;
        d.tiles_y = (c.height + TILE - 1) / TILE;
        d.scene = s;
        d.tile_off = (uint32_t)tiles;
        d.grp_off = (uint32_t)groups;
        groups += div_up((uint64_t)d.tiles_x * d.tiles_y, 32);
        d.pix_off = pix;
        d.ent_off = ent;
        tiles += (uint64_t)d.tiles_x * d.tiles_y;
        pix += (uint64_t)c.width * c.height;
        ent += (uint64_t)scenes[s].n;
    }
    if (tiles >= (1ull << 31)) return fail(SG_ERR_INVALID_ARG, "too many tiles (%llu)", (unsigned long long)tiles);
    if (ent >= (1ull << 32) - 1)
        return fail(SG_ERR_INVALID_ARG, "too many (view, Gaussian) entries (%llu)", (unsigned long long)ent);
    if (bwd_blk >= (1ull << 31)) return fail(SG_ERR_INVALID_ARG, "too many blocks");
    b.n_tiles = (uint32_t)tiles;
    b.n_groups = (uint32_t)groups;
    b.n_entries = ent;
    b.scene_blocks = (uint32_t)bwd_blk;
    b.scene_runs = (uint32_t)runs;
    uint32_t per_scene[SG_MAX_SCENES] = {};
    b.max_views_per_scene = 0;
    for (int v = 0; v < n_views; ++v) {
        const uint32_t c = ++per_scene[b.view[v].scene];
        b.max_views_per_scene = c > b.max_views_per_scene ? c : b.max_views_per_scene;
    }
    return SG_OK;
}

uint64_t n_pixels_of(const Batch &b) {
    const ViewDesc &last = b.view[b.n_views - 1];
    return last.pix_off + (uint64_t)last.W * last.H;
}

// Calls whose views have at most this many tiles in all keep no sorted tile ids.
constexpr uint64_t kNoKeyTiles = 12288;
// Pairs per row of the binning's count matrix that the per-pair size reports.
constexpr uint64_t kMatrixShare = 8192;

// The workspace holds what the forward leaves for the backward and the pairs. What only the
// sorts need, the depth sort's look-back flags and the binning's count matrix, lives in the
// image, which the blend writes after the placement has read the last count (12 bytes per
// pixel hold 760 rows of a counter per tile, fewer where the frame's edge cuts many tiles).
// Regions that follow cap hold a rounding unit at least: fixed + per pair x pairs bounds
// the total.
WsLayout make_layout(const Batch &b, uint64_t cap) {
    WsLayout L{};
    const uint64_t M = b.n_entries, T = b.n_tiles;
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t r = o; o += al(bytes); return r; };
    uint64_t row = 0;
    for (int v = 0; v < b.n_views; ++v)
        row = std::max<uint64_t>(row, (uint64_t)b.view[v].tiles_x * b.view[v].tiles_y);
    row = div_up(row, 4) * 4;
    // chunks where one chunk's counters of the largest view fit shared memory, and enough
    // chunks at once for the pairs
    L.chunked = row <= BIN_MAX_ROW && cap <= bin_max_pairs((uint32_t)row);
    L.bin_row = (uint32_t)row;
    // the chunks are cut view by view; the radix passes' digits hold the view
    L.by_view = L.chunked && b.n_views > 1;
    const uint64_t img_rows = 3 * n_pixels_of(b) / row, own_rows = (uint64_t)b.n_views + 1;
    L.matrix_in_img = img_rows >= own_rows;
    if (L.chunked)
        L.bin_chunks = (uint32_t)std::min<uint64_t>(bin_chunks(cap, L.bin_row, b.n_views),
                                                    L.matrix_in_img ? img_rows : own_rows);
    L.batch = take(sizeof(Batch));
    L.counters = take(CNT_N * sizeof(uint64_t));
    L.rec = take(M * sizeof(Rec));
    L.tiles_touched = take(M * 4);
    L.rect = take(M * 8);
    L.clamp = take(M);
    L.dup_flags = take(div_up(M, 256) * 8 + 8);   // look-back words of the chunk cutter / the duplicate
    L.ranges = take(T * 8);
    L.order = take(T * 4);   // tile order of the persistent blends (by list length)
    // the forward's tile order: its counts and cursors; the backward's: its counts
    L.order_scratch = take((TILE_ORDER_WORDS + TB_BUCKETS) * 4);
    L.bin = take(sizeof(BinTab));
    const uint64_t cuts = std::min<uint64_t>(BIN_MAX_CHUNKS, b.n_views + std::max<uint64_t>(cap / BIN_MIN_CHUNK, 1)) + 1;
    L.bin_start = take(8 * cuts + ALIGN);   // chunks' first entries, then first pairs
    L.scan_words = take(8 * (1 + (uint64_t)b.n_groups));
    L.tile_bits = tile_bits_for(T);
    L.tile_passes = L.chunked ? 0 : radix_passes(L.tile_bits);
    const bool keys = T > kNoKeyTiles;   // the layout keeps the sorted tile ids
    // Pairs: region A receives the depth-ordered (tile, entry) pairs, region B the
    // placed ones (radix passes alternate between the two). The depth sort's
    // four buffers live in B: B is first written by the placement, after
    // the pairs' kernel has read the depth order. The backward reads only the final
    // entries (chunked: B; radix: A after an even number of passes, B after an odd one)
    // and, chunked, the tiles' places by walk length, which take A after the placement.
    const size_t pairs4 = al(cap * 4), m4 = al(M * 4), unit = 2 * ALIGN;
    const size_t a_bytes = std::max(keys ? 2 * pairs4 : al(cap * 2) + pairs4, unit);
    const size_t B = take(std::max({(keys ? 2 : 1) * pairs4, 4 * m4, unit}));
    const size_t A = take(a_bytes);
    L.walk = L.chunked && walk_ordered(T) && 4 * T <= a_bytes;
    L.walk_place = A;
    L.dkey0 = B;
    L.dval0 = B + m4;
    L.dkey1 = B + 2 * m4;
    L.dval1 = B + 3 * m4;
    if (L.chunked) {
        L.pkey_final = keys ? B : NO_OFFSET;
        L.pval_final = keys ? B + pairs4 : B;
        L.pkey_tmp = A;
        L.pval_tmp = A + al(cap * 2);
    } else {
        const size_t fin = L.tile_passes % 2 == 1 ? B : A, tmp = fin == A ? B : A;
        L.pkey_final = fin;
        L.pval_final = fin + pairs4;
        L.pkey_tmp = tmp;
        L.pval_tmp = tmp + pairs4;
    }
    // look-back flags of the depth sort's passes (one more by view), where the
    // image cannot hold them, then those of the tile sort's radix passes (chunked: the
    // count matrix of a frame that cannot hold it)
    const uint64_t depth_words = depth_flag_words(M, b.n_views > 1 ? 5 : 4);
    L.depth_in_img = depth_words <= 3 * n_pixels_of(b);
    const uint64_t tile_words = !L.chunked ? sort_flag_words(std::max<uint64_t>(cap, 1), L.tile_passes)
                                           : L.matrix_in_img ? 0 : own_rows * row;
    L.hist = take(std::max<uint64_t>(L.depth_in_img ? 0 : depth_words, tile_words) * 4);
    L.aux_depth = take(sizeof(SortAux));
    L.aux_tile = take(L.chunked ? 0 : sizeof(SortAux));
    L.total = o;
    L.M = M;
    L.n_tiles = T;
    L.cap = cap;
    return L;
}

uint64_t capacity_for(const Batch &b, size_t ws_bytes) {
    if (make_layout(b, 0).total > ws_bytes) return UINT64_MAX;   // not even the fixed part
    uint64_t lo = 0, hi = (1ull << 32) - 1;
    while (lo < hi) {
        const uint64_t mid = lo + (hi - lo + 1) / 2;
        if (make_layout(b, mid).total <= ws_bytes) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Backward scratch: batch table, counters, the [M][9] 2D gradients and, last, the
// persistent backward's own tile order (where walk_ordered). A scratch without room for
// the order is enough: the backward then walks the tiles in the forward's order.
struct BwdLayout {
    size_t batch, counters, dg, needed, order, total;
};

BwdLayout bwd_layout(const Batch &b) {
    BwdLayout L{};
    size_t o = 0;
    auto take = [&](size_t bytes) { size_t r = o; o += al(bytes); return r; };
    L.batch = take(sizeof(Batch));
    L.counters = take(CNT_N * sizeof(uint64_t));
    L.dg = take(9 * b.n_entries * sizeof(float));
    L.needed = o;
    L.order = take(walk_ordered(b.n_tiles) ? 4 * (size_t)b.n_tiles : 0);
    L.total = o;
    return L;
}

// Pixels per thread under auto_shapes: with few tiles a warp's walk of its list is the
// critical path, so a tile is given to more warps; with many, fewer warps per tile issue less
// in all. Measured (us, forward / backward, 1, 2, 4, 8 pixels per thread; clustered scenes):
//   tiles  pairs a tile     1         2         4         8
//     494       57       22/46     28/63     37/78     60/121
//     475     1336      172/395   217/536   323/619   630/951
//    1200      130       51/143    67/181   100/217   157/319
//    1200     1719      149/404   191/431   276/505   472/799
//    2500       47       30/78     37/92     56/108    84/177
//    2500      531      145/496   162/395   224/382   349/608
//    2500     1936      223/731   250/638   298/618   479/801
//    2880      317      119/381   137/357   194/358   308/553
//    2880     1704      174/576   178/454   197/409   297/468
//    3600       62       47/143    48/114    72/128   106/192
//    3600      281      130/435   142/342   180/320   254/475
//    3600      875      188/640   194/508   214/439   300/526
//    5400       58       64/202    60/154    76/131   101/197
//    5400      381      238/857   234/637   232/529   296/510
//    5700      369      249/887   241/658   235/544   313/495
//    7728      157      218/795   208/582   198/482   260/409
//    8160      329      326/1177  316/860   302/715   387/589
// The lines lie between these points. The count does not see the lists' length: where
// they are long in few tiles the backward's choice is up to 1.3 times the best (2500 tiles),
// and near the lines to more pixels a choice is 3 or 4 % above its neighbour (5400, 5700).
int auto_pixels(bool backward, uint64_t n_tiles) {
    if (backward) return n_tiles <= 2560 ? 1 : n_tiles <= 3072 ? 2 : n_tiles <= 5632 ? 4 : 8;
    return n_tiles <= 3600 ? 1 : n_tiles <= 7680 ? 2 : 4;
}

// Blend shape of this call: pixels per thread from the tuning (from the tile
// count under auto_shapes), and for the persistent form the resident
// grid, the work counter and the tile order.
int blend_shape(bool backward, uint64_t n_tiles, const uint32_t *order, uint32_t *queue, BlendShape &sh) {
    const sg_tuning &t = tuning();
    sh.pixels_per_thread = backward ? t.bwd_pixels_per_thread : t.fwd_pixels_per_thread;
    sh.persistent = (backward ? t.bwd_persistent : t.fwd_persistent) != 0;
    const int nb = backward ? t.bwd_batch : t.fwd_batch;
    const sg_tuning &d = kDefaultTuning;
    if (((t.auto_shapes >> (backward ? 1 : 0)) & 1) && nb == 0 && sh.persistent &&
        sh.pixels_per_thread == (backward ? d.bwd_pixels_per_thread : d.fwd_pixels_per_thread))
        sh.pixels_per_thread = auto_pixels(backward, n_tiles);
    sh.tile_order = sh.persistent ? order : nullptr;
    sh.queue = queue;
    sh.batch = nb ? nb : kDefaultBatch;
    sh.grid = sh.persistent ? blend_persistent_grid(backward, sh.pixels_per_thread, sh.batch) : 0;
    if (sh.persistent && sh.grid <= 0)
        return fail(SG_ERR_CUDA, "persistent blend: occupancy query failed");
    return SG_OK;
}

void fill_sizes(const Batch &b, const WsLayout &L, uint64_t n_pairs, sg_sizes *out) {
    if (!out) return;
    out->n_entries = b.n_entries;
    out->n_tiles = b.n_tiles;
    out->n_pixels = n_pixels_of(b);
    out->n_pairs = n_pairs;
    out->pair_capacity = L.cap;
    out->ws_fixed_bytes = make_layout(b, 0).total;
    // at most: pair buffers (16-bit tile ids and entries, then the placed entries: 10; with
    // sorted tile ids kept, 32-bit ids and entries twice: 16), with room for a share of the
    // count matrix, or for the radix passes' look-back words (a third of a byte a pass)
    out->ws_per_pair_bytes = b.n_tiles > kNoKeyTiles ? 17 + (L.tile_passes > 3 ? 1 : 0)
                                                     : 10 + div_up(4 * (uint64_t)L.bin_row, kMatrixShare);
    out->ws_bytes = L.total;
    out->bwd_ws_bytes = bwd_layout(b).total;
}

// Per-thread pinned host words, mapped into the device, and an event for the
// plain form's read of the pair count: the kernel that knows the total (chunk cutter or
// duplicate) stores it there, the tile sort's last one the status, and the host waits on
// the event after them.
struct CountReadback {
    uint64_t *host = nullptr;     // [0] pairs, [1] status
    uint64_t *dev_ptr = nullptr;  // the same words as the current device sees them
    cudaEvent_t ev = nullptr;
    int device = -1;
};

static cudaError_t count_readback(CountReadback *&out) {
    thread_local CountReadback rb;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (!rb.host) {
        void *p = nullptr;
        e = cudaHostAlloc(&p, 64, cudaHostAllocPortable | cudaHostAllocMapped);
        if (e != cudaSuccess) return e;
        rb.host = static_cast<uint64_t *>(p);
    }
    if (!rb.ev || rb.device != dev) {
        if (rb.ev) cudaEventDestroy(rb.ev);
        rb.ev = nullptr;
        e = cudaEventCreateWithFlags(&rb.ev, cudaEventDisableTiming);
        if (e != cudaSuccess) return e;
        void *dp = nullptr;
        e = cudaHostGetDevicePointer(&dp, rb.host, 0);
        if (e != cudaSuccess) return e;
        rb.dev_ptr = static_cast<uint64_t *>(dp);
        rb.device = dev;
    }
    out = &rb;
    return cudaSuccess;
}

// Both forms queue the whole forward at once with grids sized by the pair
// capacity; the pair count stays on the device, which handles an overflow
// (no pairs are written, every tile list is empty). sync = true: the plain
// form also copies the count to the host behind an event and waits for that
// copy alone after queueing everything, to return SG_ERR_CAPACITY (or the
// depth sort's SG_ERR_TIMEOUT) and the count. sync = false: the batched form
// (overflow recorded in the device status, graph capturable).
int forward_impl(const sg_scene *scenes, int n_scenes, const sg_camera *cams, const int32_t *view_scene,
                 int n_views, void *ws, size_t ws_bytes, float *img, float *T_final, int32_t *last,
                 float *const *importance, sg_sizes *out, cudaStream_t stream, bool sync) {
    std::unique_ptr<Batch> hb(new Batch);
    int st = build_batch(scenes, n_scenes, cams, view_scene, n_views, true, *hb);
    if (st != SG_OK) return st;
    Batch &b = *hb;
    bool want_importance = false;
    if (importance) {
        for (int s = 0; s < n_scenes; ++s) {
            if (scenes[s].n > 0 && (!importance[s] || !aligned(importance[s], 4)))
                return fail(SG_ERR_INVALID_ARG, "importance[%d] is NULL or misaligned", s);
            b.scene[s].importance = importance[s];
            want_importance = want_importance || scenes[s].n > 0;
        }
    }
    if (!img || !T_final || !last) return fail(SG_ERR_INVALID_ARG, "output pointers must not be NULL");
    if (!aligned(img, 16) || !aligned(T_final, 16) || !aligned(last, 16))
        return fail(SG_ERR_INVALID_ARG, "outputs must be 16-byte aligned");
    if (!ws || !aligned(ws, ALIGN)) return fail(SG_ERR_INVALID_ARG, "workspace NULL or not 256-byte aligned");
    const uint64_t cap = capacity_for(b, ws_bytes);
    if (cap == UINT64_MAX) {
        WsLayout L0 = make_layout(b, 0);
        fill_sizes(b, L0, 0, out);
        return fail(SG_ERR_WORKSPACE, "workspace of %zu bytes is below the fixed part (%zu bytes)", ws_bytes,
                    L0.total);
    }
    const WsLayout L = make_layout(b, cap);
    char *w = static_cast<char *>(ws);
    Batch *db = reinterpret_cast<Batch *>(w + L.batch);
    uint64_t *counters = reinterpret_cast<uint64_t *>(w + L.counters);
    Rec *rec = reinterpret_cast<Rec *>(w + L.rec);
    uint32_t *tt = reinterpret_cast<uint32_t *>(w + L.tiles_touched);
    uint2 *rect = reinterpret_cast<uint2 *>(w + L.rect);
    uint32_t *dkey0 = reinterpret_cast<uint32_t *>(w + L.dkey0);
    uint32_t *dval0 = reinterpret_cast<uint32_t *>(w + L.dval0);
    uint32_t *dkey1 = reinterpret_cast<uint32_t *>(w + L.dkey1);
    uint32_t *dval1 = reinterpret_cast<uint32_t *>(w + L.dval1);
    uint64_t *dup_flags = reinterpret_cast<uint64_t *>(w + L.dup_flags);
    uint2 *ranges = reinterpret_cast<uint2 *>(w + L.ranges);
    uint32_t *hist = reinterpret_cast<uint32_t *>(w + L.hist);
    SortAux *aux_depth = reinterpret_cast<SortAux *>(w + L.aux_depth), *aux_tile = reinterpret_cast<SortAux *>(w + L.aux_tile);
    BinTab *tab = reinterpret_cast<BinTab *>(w + L.bin);
    const uint64_t M = L.M;

    const bool counting = (prof().flags & SG_PROFILE_COUNT) != 0;
    {
        // the setup kernel also clears the sorts' scratch, the binning's totals
        // and look-back words (chunked) or marks every tile range empty (radix)
        ZeroRegions z;
        int r = 0;
        auto zero = [&](void *ptr, uint64_t words, uint32_t even = 0u) {
            z.ptr[r] = static_cast<uint32_t *>(ptr);
            z.words[r] = words;
            z.even[r++] = even;
        };
        zero(aux_depth, sizeof(SortAux) / 4);
        zero(dup_flags, 2 * div_up(M, 256));
        zero(w + L.order_scratch, TILE_ORDER_WORDS + TB_BUCKETS);
        zero(tab, sizeof(tab->view_pairs) / 4);
        if (L.chunked) {
            zero(w + L.scan_words, 2 * (1 + (uint64_t)b.n_groups));
        } else {
            zero(aux_tile, sizeof(SortAux) / 4);
            zero(ranges, 2 * L.n_tiles, RANGE_EMPTY);
        }
        StageTimer t(ST_SETUP, stream);
        SG_CUDA(launch_setup(b, db, counters, stream, z), "setup");
    }
    {
        StageTimer t(ST_PRE, stream);
        SG_CUDA(launch_preprocess(b, db, rec, tt, rect, dkey0, reinterpret_cast<uint8_t *>(w + L.clamp),
                                  tab->view_pairs, aux_depth->hist[VIEW_PASS], stream),
                "preprocessSG");
    }
    {
        // once per entry; entries that reach no tile are left out of the order
        StageTimer t(ST_DEPTH_SORT, stream);
        SG_CUDA(launch_depth_sort(db, L.by_view, dkey0, dval0, dkey1, dval1, counters + CNT_ENTRIES, M,
                                  L.depth_in_img ? reinterpret_cast<uint32_t *>(img) : hist, aux_depth, stream),
                "depth sort");
    }
    const uint32_t *order = L.by_view ? dval1 : dval0;   // entries by ((view,) depth)
    CountReadback *rb = nullptr;   // plain form: where the duplicate leaves the pair count for the host
    if (sync) SG_CUDA(count_readback(rb), "pair count readback");
    // grids sized by the capacity (at most SORT_MAX_KEYS pairs); counts read on the device
    const uint64_t cap_dev = std::min<uint64_t>(cap, SORT_MAX_KEYS);
    uint32_t *pk_final = L.pkey_final == NO_OFFSET ? nullptr : reinterpret_cast<uint32_t *>(w + L.pkey_final);
    uint32_t *pv_final = reinterpret_cast<uint32_t *>(w + L.pval_final);
    uint32_t *pk_tmp = reinterpret_cast<uint32_t *>(w + L.pkey_tmp);
    uint32_t *pv_tmp = reinterpret_cast<uint32_t *>(w + L.pval_tmp);
    uint64_t *mirror = rb ? rb->dev_ptr : nullptr;   // plain form: pair count and status for the host
    uint32_t *order_counts = reinterpret_cast<uint32_t *>(w + L.order_scratch);
    if (L.chunked) {
        BinArgs a{};
        a.db = db;
        a.n_views = n_views;
        a.M = M;
        a.cap = cap_dev;
        a.max_chunks = L.bin_chunks;
        a.row = L.bin_row;
        a.n_groups = b.n_groups;
        a.n_tiles = b.n_tiles;
        a.sorted_ent = order;
        a.aux = aux_depth;
        a.tiles_touched = tt;
        a.rect = rect;
        a.rec = rec;
        a.counters = counters;
        a.tab = tab;
        a.start = reinterpret_cast<uint32_t *>(w + L.bin_start);
        a.pair = a.start + L.bin_chunks + 1;
        a.poff = dkey1;   // the depth keys are no longer needed
        a.flags = dup_flags;
        a.pkey = reinterpret_cast<uint16_t *>(pk_tmp);
        a.pval = pv_tmp;
        a.matrix = L.matrix_in_img ? reinterpret_cast<uint32_t *>(img) : hist;
        a.words = reinterpret_cast<uint64_t *>(w + L.scan_words);
        a.ranges = ranges;
        a.order_counts = order_counts;
        a.ovals = pv_final;
        a.okeys = pk_final;
        a.mirror = mirror;
        {
            StageTimer t(ST_DUPLICATE, stream);
            SG_CUDA(launch_bin_pairs(a, stream), "duplicateWithKeys");
        }
        StageTimer t(ST_TILE_SORT, stream);
        SG_CUDA(launch_bin_place(a, stream), "tile sort");
    } else {
        // duplicate into the buffer from which the radix passes end in *_final
        const bool dup_final = L.tile_passes % 2 == 0;
        uint32_t *k0 = dup_final ? pk_final : pk_tmp, *v0 = dup_final ? pv_final : pv_tmp;
        uint32_t *k1 = dup_final ? pk_tmp : pk_final, *v1 = dup_final ? pv_tmp : pv_final;
        {
            StageTimer t(ST_DUPLICATE, stream);
            SG_CUDA(launch_duplicate(db, M, order, aux_depth, tt, rect, rec, counters, cap_dev, k0, v0, dup_flags,
                                     mirror, stream, L.tile_passes, aux_tile, hist,
                                     sort_flag_words(cap_dev, L.tile_passes)),
                    "duplicateWithKeys");
        }
        StageTimer t(ST_TILE_SORT, stream);
        SG_CUDA(launch_tile_radix_sort(k0, v0, k1, v1, counters, cap_dev, L.tile_bits, hist, aux_tile, ranges,
                                       L.n_tiles, order_counts, mirror ? mirror + 1 : nullptr, stream),
                "tile sort");
    }
    if (sync) SG_CUDA(cudaEventRecord(rb->ev, stream), "read pairs");
    unsigned long long *evals =
        counting ? reinterpret_cast<unsigned long long *>(counters + CNT_EVALS) : nullptr;
    if (counting) SG_CUDA(cudaMemsetAsync(evals, 0, 8, stream), "clear counter");
    BlendShape shape{};
    st = blend_shape(false, b.n_tiles, reinterpret_cast<uint32_t *>(w + L.order),
                     reinterpret_cast<uint32_t *>(counters + CNT_QUEUE), shape);
    if (st != SG_OK) return st;
    shape.status = counters + CNT_STATUS;
    if (L.walk) {
        shape.walk_counts = order_counts + TILE_ORDER_WORDS;
        shape.walk_place = reinterpret_cast<uint32_t *>(w + L.walk_place);
    }
    shape.importance = want_importance && !counting;
    if (shape.importance)
        for (int s = 0; s < n_scenes; ++s)
            if (scenes[s].n > 0)
                SG_CUDA(cudaMemsetAsync(importance[s], 0, (size_t)scenes[s].n * sizeof(float), stream),
                        "clear importance");
    {
        // built for every forward: the persistent backward walks tiles in this order too
        StageTimer t(ST_RANGES, stream);
        SG_CUDA(launch_tile_order(ranges, b.n_tiles, reinterpret_cast<uint32_t *>(w + L.order), order_counts, stream),
                "tile order");
    }
    {
        StageTimer t(ST_BLEND_FWD, stream);
        SG_CUDA(launch_blend_forward(db, b.n_tiles, ranges, pv_final, rec, img, T_final, last, shape, evals,
                                     stream),
                "blend forward");
    }
    if (counting) {
        uint64_t ne = 0;
        SG_CUDA(cudaMemcpyAsync(&ne, evals, 8, cudaMemcpyDeviceToHost, stream), "read counter");
        SG_CUDA(cudaStreamSynchronize(stream), "read counter");
        std::lock_guard<std::mutex> g(prof().mu);
        prof().evals[0] += (int64_t)ne;
    }
    if (sync) {
        SG_CUDA(cudaEventSynchronize(rb->ev), "read pairs");
        const volatile uint64_t *mirror = rb->host;
        const uint64_t n_pairs = mirror[0];
        if (mirror[1] == SG_ERR_TIMEOUT)
            return fail(SG_ERR_TIMEOUT, "a sort's bounded device wait expired (outputs unspecified)");
        if (n_pairs > cap_dev) {
            const WsLayout need = make_layout(b, n_pairs);
            fill_sizes(b, need, n_pairs, out);
            if (n_pairs > SORT_MAX_KEYS)
                return fail(SG_ERR_CAPACITY, "%llu pairs exceed the %llu one call can sort",
                            (unsigned long long)n_pairs, (unsigned long long)SORT_MAX_KEYS);
            return fail(SG_ERR_CAPACITY, "%llu pairs exceed the workspace capacity %llu (need %zu bytes)",
                        (unsigned long long)n_pairs, (unsigned long long)cap, need.total);
        }
        fill_sizes(b, L, n_pairs, out);
        return SG_OK;
    }
    fill_sizes(b, L, cap_dev, out);
    return SG_OK;
}

int backward_impl(const sg_scene *scenes, int n_scenes, const sg_camera *cams, const int32_t *view_scene,
                  int n_views, const void *ws, size_t ws_bytes, const float *T_final, const int32_t *last,
                  const float *d_img, void *bwd_ws, size_t bwd_ws_bytes, const sg_grads *grads,
                  cudaStream_t stream) {
    std::unique_ptr<Batch> hb(new Batch);
    int st = build_batch(scenes, n_scenes, cams, view_scene, n_views, true, *hb);
    if (st != SG_OK) return st;
    Batch &b = *hb;
    if (!grads) return fail(SG_ERR_INVALID_ARG, "grads must not be NULL");
    for (int s = 0; s < n_scenes; ++s) b.scene[s].grads = grads[s];
    if (!T_final || !last || !d_img) return fail(SG_ERR_INVALID_ARG, "T_final, last and d_img must not be NULL");
    if (!ws || !aligned(ws, ALIGN)) return fail(SG_ERR_INVALID_ARG, "workspace NULL or not 256-byte aligned");
    if (!bwd_ws || !aligned(bwd_ws, ALIGN))
        return fail(SG_ERR_INVALID_ARG, "backward scratch NULL or not 256-byte aligned");
    const BwdLayout BL = bwd_layout(b);
    if (bwd_ws_bytes < BL.needed)
        return fail(SG_ERR_WORKSPACE, "backward scratch of %zu bytes, %zu needed", bwd_ws_bytes, BL.needed);
    const uint64_t cap = capacity_for(b, ws_bytes);
    if (cap == UINT64_MAX) return fail(SG_ERR_WORKSPACE, "workspace smaller than its fixed part");
    const WsLayout L = make_layout(b, cap);
    const char *w = static_cast<const char *>(ws);
    const Rec *rec = reinterpret_cast<const Rec *>(w + L.rec);
    const uint32_t *tt = reinterpret_cast<const uint32_t *>(w + L.tiles_touched);
    const uint2 *ranges = reinterpret_cast<const uint2 *>(w + L.ranges);
    const uint32_t *pv_final = reinterpret_cast<const uint32_t *>(w + L.pval_final);
    char *bw = static_cast<char *>(bwd_ws);
    Batch *db = reinterpret_cast<Batch *>(bw + BL.batch);
    uint64_t *counters = reinterpret_cast<uint64_t *>(bw + BL.counters);
    float *dg = reinterpret_cast<float *>(bw + BL.dg);
    const uint64_t M = L.M;

    const bool counting = (prof().flags & SG_PROFILE_COUNT) != 0;
    unsigned long long *evals =
        counting ? reinterpret_cast<unsigned long long *>(counters + CNT_EVALS) : nullptr;
    BlendShape shape{};
    // Tiles by the forward's largest last position: the walk's length, where the list's
    // is only its bound (a list's tail lies behind stopped pixels). With two or three
    // tiles per resident warp the last ones to start decide when the kernel ends.
    TileOrder walk;
    if (L.walk && bwd_ws_bytes >= BL.total) {
        walk.counts = reinterpret_cast<const uint32_t *>(w + L.order_scratch) + TILE_ORDER_WORDS;
        walk.place = reinterpret_cast<const uint32_t *>(w + L.walk_place);
        walk.fallback = reinterpret_cast<const uint32_t *>(w + L.order);
        walk.order = reinterpret_cast<uint32_t *>(bw + BL.order);
        walk.n = b.n_tiles;
    }
    st = blend_shape(true, b.n_tiles, walk.n ? walk.order : reinterpret_cast<const uint32_t *>(w + L.order),
                     reinterpret_cast<uint32_t *>(counters + CNT_QUEUE), shape);
    if (!shape.persistent) walk = TileOrder();
    if (st != SG_OK) return st;
    shape.status = reinterpret_cast<const uint64_t *>(w + L.counters) + CNT_STATUS;   // the forward's
    {
        // the setup kernel also clears the 2D-gradient accumulators
        StageTimer t(ST_BWD_CLEAR, stream);
        ZeroRegions z;
        z.ptr[0] = reinterpret_cast<uint32_t *>(dg);
        z.words[0] = 9 * M;
        SG_CUDA(launch_setup(b, db, counters, stream, z, walk), "setup");
    }
    {
        StageTimer t(ST_BLEND_BWD, stream);
        SG_CUDA(launch_blend_backward(db, b.n_tiles, ranges, pv_final, rec, T_final, last, d_img, dg, shape,
                                      evals, stream),
                "blend backward");
    }
    {
        StageTimer t(ST_PRE_BWD, stream);
        SG_CUDA(launch_preprocess_backward(b, db, tt, reinterpret_cast<const uint8_t *>(w + L.clamp), dg, M, stream), "preprocess backward");
    }
    if (counting) {
        uint64_t ne = 0;
        SG_CUDA(cudaMemcpyAsync(&ne, evals, 8, cudaMemcpyDeviceToHost, stream), "read counter");
        SG_CUDA(cudaStreamSynchronize(stream), "read counter");
        std::lock_guard<std::mutex> g(prof().mu);
        prof().evals[1] += (int64_t)ne;
    }
    return SG_OK;
}

}  // namespace

extern "C" {

int sg_profile_enable(int flags) {
    Profiler &p = prof();
    std::lock_guard<std::mutex> g(p.mu);
    p.flags = flags & (SG_PROFILE_EVENTS | SG_PROFILE_COUNT);
    return SG_OK;
}

int sg_profile_set_stages(uint32_t stage_mask) {
    Profiler &p = prof();
    std::lock_guard<std::mutex> g(p.mu);
    p.stage_mask = stage_mask;
    return SG_OK;
}

int sg_profile_read(double *ms, int64_t *launches, int64_t *pair_evals, int reset) {
    Profiler &p = prof();
    std::lock_guard<std::mutex> g(p.mu);
    int rc = SG_OK;
    for (auto &q : p.pending) {
        cudaError_t e = cudaEventSynchronize(q.b);
        float t = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&t, q.a, q.b);
        if (e != cudaSuccess) rc = cuda_fail(e, "profile read");
        p.ms[q.stage] += t;
        p.launches[q.stage] += 1;
        p.pool.push_back(q.a);
        p.pool.push_back(q.b);
    }
    p.pending.clear();
    for (int i = 0; i < ST_N; ++i) {
        if (ms) ms[i] = p.ms[i];
        if (launches) launches[i] = p.launches[i];
    }
    if (pair_evals) { pair_evals[0] = p.evals[0]; pair_evals[1] = p.evals[1]; }
    if (reset) {
        for (int i = 0; i < ST_N; ++i) { p.ms[i] = 0.0; p.launches[i] = 0; }
        p.evals[0] = p.evals[1] = 0;
    }
    return rc;
}

int64_t sg_kernel_launches(void) { return launch_counter().load(); }

int sg_set_tuning(const sg_tuning *t) {
    if (!t) {
        tuning() = kDefaultTuning;
        set_sort_wait_polls(0);
        return SG_OK;
    }
    if (!ppt_ok(t->fwd_pixels_per_thread) || !ppt_ok(t->bwd_pixels_per_thread))
        return fail(SG_ERR_INVALID_ARG, "pixels per thread must be 1, 2, 4 or 8 (got %d, %d)",
                    t->fwd_pixels_per_thread, t->bwd_pixels_per_thread);
    if (t->sort_wait_polls < 0) return fail(SG_ERR_INVALID_ARG, "sort_wait_polls = %d < 0", t->sort_wait_polls);
    if (!(t->fwd_batch == 0 || t->fwd_batch == 32 || t->fwd_batch == 64 || t->fwd_batch == 128))
        return fail(SG_ERR_INVALID_ARG, "fwd_batch must be 0, 32, 64 or 128 (got %d)", t->fwd_batch);
    if (!(t->bwd_batch == 0 || t->bwd_batch == 32 || t->bwd_batch == 64))
        return fail(SG_ERR_INVALID_ARG, "bwd_batch must be 0, 32 or 64 (got %d)", t->bwd_batch);
    tuning() = *t;
    tuning().auto_shapes &= 3;
    set_sort_wait_polls((uint32_t)t->sort_wait_polls);
    return SG_OK;
}

int sg_get_tuning(sg_tuning *t) {
    if (!t) return fail(SG_ERR_INVALID_ARG, "t must not be NULL");
    *t = tuning();
    return SG_OK;
}

const char *sg_profile_stage_name(int i) { return (i >= 0 && i < ST_N) ? kStageNames[i] : nullptr; }

int sg_version(void) { return SG_ABI_VERSION; }

const char *sg_last_error(void) { return g_err; }

int sg_workspace_query(const sg_scene *scene, const sg_camera *cams, int n_views, uint64_t pair_capacity,
                       sg_sizes *out) {
    if (!out) return fail(SG_ERR_INVALID_ARG, "out must not be NULL");
    std::unique_ptr<Batch> hb(new Batch);
    int st = build_batch(scene, 1, cams, nullptr, n_views, false, *hb);
    if (st != SG_OK) return st;
    if (pair_capacity >= (1ull << 32) - 1) return fail(SG_ERR_INVALID_ARG, "pair capacity too large");
    const WsLayout L = make_layout(*hb, pair_capacity);
    fill_sizes(*hb, L, 0, out);
    return SG_OK;
}

static int layout_of(const sg_scene *scenes, int n_scenes, const sg_camera *cams, const int32_t *view_scene,
                     int n_views, size_t ws_bytes, sg_ws_layout *out) {
    if (!out) return fail(SG_ERR_INVALID_ARG, "out must not be NULL");
    std::unique_ptr<Batch> hb(new Batch);
    int st = build_batch(scenes, n_scenes, cams, view_scene, n_views, false, *hb);
    if (st != SG_OK) return st;
    const uint64_t cap = capacity_for(*hb, ws_bytes);
    if (cap == UINT64_MAX) return fail(SG_ERR_WORKSPACE, "workspace smaller than its fixed part");
    const WsLayout L = make_layout(*hb, cap);
    out->rec = L.rec;
    out->tiles_touched = L.tiles_touched;
    out->rect = L.rect;
    out->depth_order = L.by_view ? L.dval1 : L.dval0;
    out->ranges = L.ranges;
    out->pair_tile = L.pkey_final;
    out->pair_entry = L.pval_final;
    out->total_bytes = L.total;
    return SG_OK;
}

int sg_workspace_layout(const sg_scene *scene, const sg_camera *cams, int n_views, size_t ws_bytes,
                        sg_ws_layout *out) {
    return layout_of(scene, 1, cams, nullptr, n_views, ws_bytes, out);
}

int sg_batched_workspace_layout(const sg_scene *scenes, int n_scenes, const sg_camera *cams,
                                const int32_t *view_scene, int n_views, size_t ws_bytes, sg_ws_layout *out) {
    if (!view_scene) return fail(SG_ERR_INVALID_ARG, "view_scene must not be NULL");
    return layout_of(scenes, n_scenes, cams, view_scene, n_views, ws_bytes, out);
}

int sg_render_forward(const sg_scene *scene, const sg_camera *cams, int n_views, void *ws, size_t ws_bytes,
                      float *img, float *T_final, int32_t *last, sg_sizes *out, void *stream) {
    g_err[0] = '\0';
    return forward_impl(scene, 1, cams, nullptr, n_views, ws, ws_bytes, img, T_final, last, nullptr, out,
                        static_cast<cudaStream_t>(stream), true);
}

int sg_render_forward_importance(const sg_scene *scene, const sg_camera *cams, int n_views, void *ws,
                                 size_t ws_bytes, float *img, float *T_final, int32_t *last, float *importance,
                                 sg_sizes *out, void *stream) {
    g_err[0] = '\0';
    float *const imp[1] = {importance};
    return forward_impl(scene, 1, cams, nullptr, n_views, ws, ws_bytes, img, T_final, last, imp, out,
                        static_cast<cudaStream_t>(stream), true);
}

int sg_render_backward(const sg_scene *scene, const sg_camera *cams, int n_views, const void *ws,
                       size_t ws_bytes, const float *T_final, const int32_t *last, const float *d_img,
                       void *bwd_ws, size_t bwd_ws_bytes, const sg_grads *grads, void *stream) {
    g_err[0] = '\0';
    return backward_impl(scene, 1, cams, nullptr, n_views, ws, ws_bytes, T_final, last, d_img, bwd_ws,
                         bwd_ws_bytes, grads, static_cast<cudaStream_t>(stream));
}

// Times every blend shape (pixels per thread 1, 2, 4, 8; one block per tile or
// persistent) on the caller's workload: each candidate runs `reps` forward and
// backward calls after one untimed pair; the forward and the backward pick
// their fastest shape independently (only the blend kernels differ between
// candidates, so whole-call times rank them). The choice is installed with
// sg_set_tuning and written to *chosen; times_ms (nullable) receives [2][8]
// mean milliseconds, forward then backward, candidate c = 2 * log2(P) + persistent.
int sg_autotune(const sg_scene *scene, const sg_camera *cams, int n_views, void *ws, size_t ws_bytes,
                float *img, float *T_final, int32_t *last, const float *d_img, void *bwd_ws,
                size_t bwd_ws_bytes, const sg_grads *grads, int reps, sg_tuning *chosen, float *times_ms,
                void *stream) {
    g_err[0] = '\0';
    if (!chosen) return fail(SG_ERR_INVALID_ARG, "chosen must not be NULL");
    if (reps < 1 || reps > 100) return fail(SG_ERR_INVALID_ARG, "reps = %d out of [1, 100]", reps);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const sg_tuning saved = tuning();
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
    for (auto &e : ev)
        if (cudaEventCreate(&e) != cudaSuccess) {
            for (auto &x : ev) if (x) cudaEventDestroy(x);
            return cuda_fail(cudaGetLastError(), "autotune events");
        }
    float best_f = 1e30f, best_b = 1e30f;
    int bf = 0, bb = 0;
    int st = SG_OK;
    for (int c = 0; c < 8 && st == SG_OK; ++c) {
        sg_tuning t = saved;
        t.fwd_pixels_per_thread = t.bwd_pixels_per_thread = 1 << (c >> 1);
        t.fwd_persistent = t.bwd_persistent = c & 1;
        t.fwd_batch = t.bwd_batch = kDefaultBatch;
        t.auto_shapes = 0;   // the candidate itself, not the tile count's choice
        tuning() = t;
        float tf = 0.f, tb = 0.f;
        for (int r = 0; r <= reps && st == SG_OK; ++r) {
            sg_sizes sz{};
            cudaEventRecord(ev[0], s);
            st = forward_impl(scene, 1, cams, nullptr, n_views, ws, ws_bytes, img, T_final, last, nullptr, &sz, s,
                              true);
            if (st != SG_OK) break;
            cudaEventRecord(ev[1], s);
            st = backward_impl(scene, 1, cams, nullptr, n_views, ws, ws_bytes, T_final, last, d_img, bwd_ws,
                               bwd_ws_bytes, grads, s);
            if (st != SG_OK) break;
            cudaEventRecord(ev[2], s);
            const cudaError_t e = cudaEventSynchronize(ev[2]);
            if (e != cudaSuccess) { st = cuda_fail(e, "autotune"); break; }
            float a = 0.f, b = 0.f;
            cudaEventElapsedTime(&a, ev[0], ev[1]);
            cudaEventElapsedTime(&b, ev[1], ev[2]);
            if (r > 0) { tf += a; tb += b; }   // the first pair is untimed
        }
        if (st != SG_OK) break;
        tf /= (float)reps;
        tb /= (float)reps;
        if (times_ms) { times_ms[c] = tf; times_ms[8 + c] = tb; }
        if (tf < best_f) { best_f = tf; bf = c; }
        if (tb < best_b) { best_b = tb; bb = c; }
    }
    // then the batch sizes for the chosen shapes (forward 32 / 64 / 128, backward 32 / 64)
    sg_tuning t = saved;
    t.fwd_pixels_per_thread = 1 << (bf >> 1);
    t.fwd_persistent = bf & 1;
    t.bwd_pixels_per_thread = 1 << (bb >> 1);
    t.bwd_persistent = bb & 1;
    t.auto_shapes = 0;
    int best_fb = 64, best_bb = 64;
    best_f = best_b = 1e30f;
    for (int c = 0; c < 3 && st == SG_OK; ++c) {
        sg_tuning u = t;
        u.fwd_batch = 32 << c;
        u.bwd_batch = c < 2 ? 32 << c : 64;
        tuning() = u;
        float tf = 0.f, tb = 0.f;
        for (int r = 0; r <= reps && st == SG_OK; ++r) {
            sg_sizes sz{};
            cudaEventRecord(ev[0], s);
            st = forward_impl(scene, 1, cams, nullptr, n_views, ws, ws_bytes, img, T_final, last, nullptr, &sz, s,
                              true);
            if (st != SG_OK) break;
            cudaEventRecord(ev[1], s);
            st = backward_impl(scene, 1, cams, nullptr, n_views, ws, ws_bytes, T_final, last, d_img, bwd_ws,
                               bwd_ws_bytes, grads, s);
            if (st != SG_OK) break;
            cudaEventRecord(ev[2], s);
            const cudaError_t e = cudaEventSynchronize(ev[2]);
            if (e != cudaSuccess) { st = cuda_fail(e, "autotune"); break; }
            float a = 0.f, b = 0.f;
            cudaEventElapsedTime(&a, ev[0], ev[1]);
            cudaEventElapsedTime(&b, ev[1], ev[2]);
            if (r > 0) { tf += a; tb += b; }
        }
        if (st != SG_OK) break;
        if (tf < best_f) { best_f = tf; best_fb = u.fwd_batch; }
        if (c < 2 && tb < best_b) { best_b = tb; best_bb = u.bwd_batch; }
    }
    for (auto &e : ev) cudaEventDestroy(e);
    if (st != SG_OK) {
        tuning() = saved;
        return st;
    }
    t.fwd_batch = best_fb;
    t.bwd_batch = best_bb;
    tuning() = t;
    *chosen = t;
    return SG_OK;
}

int sg_batched_workspace_query(const sg_scene *scenes, int n_scenes, const sg_camera *cams,
                               const int32_t *view_scene, int n_views, uint64_t pair_capacity, sg_sizes *out) {
    if (!out) return fail(SG_ERR_INVALID_ARG, "out must not be NULL");
    if (!view_scene) return fail(SG_ERR_INVALID_ARG, "view_scene must not be NULL");
    std::unique_ptr<Batch> hb(new Batch);
    int st = build_batch(scenes, n_scenes, cams, view_scene, n_views, false, *hb);
    if (st != SG_OK) return st;
    if (pair_capacity >= (1ull << 32) - 1) return fail(SG_ERR_INVALID_ARG, "pair capacity too large");
    fill_sizes(*hb, make_layout(*hb, pair_capacity), 0, out);
    return SG_OK;
}

int sg_render_batched_forward(const sg_scene *scenes, int n_scenes, const sg_camera *cams,
                              const int32_t *view_scene, int n_views, void *ws, size_t ws_bytes, float *img,
                              float *T_final, int32_t *last, float *const *importance, void *stream) {
    g_err[0] = '\0';
    if (!view_scene) return fail(SG_ERR_INVALID_ARG, "view_scene must not be NULL");
    return forward_impl(scenes, n_scenes, cams, view_scene, n_views, ws, ws_bytes, img, T_final, last,
                        importance, nullptr, static_cast<cudaStream_t>(stream), false);
}

int sg_render_batched_backward(const sg_scene *scenes, int n_scenes, const sg_camera *cams,
                               const int32_t *view_scene, int n_views, const void *ws, size_t ws_bytes,
                               const float *T_final, const int32_t *last, const float *d_img, void *bwd_ws,
                               size_t bwd_ws_bytes, const sg_grads *grads, void *stream) {
    g_err[0] = '\0';
    if (!view_scene) return fail(SG_ERR_INVALID_ARG, "view_scene must not be NULL");
    return backward_impl(scenes, n_scenes, cams, view_scene, n_views, ws, ws_bytes, T_final, last, d_img, bwd_ws,
                         bwd_ws_bytes, grads, static_cast<cudaStream_t>(stream));
}

size_t sg_admm_workspace_bytes(int64_t n) { return admm_workspace_bytes(n); }

static int admm_check(int64_t n, const void *ws, size_t ws_bytes) {
    if (n < 0 || n >= (int64_t)UINT32_MAX) return fail(SG_ERR_INVALID_ARG, "n = %lld out of range", (long long)n);
    if (n > 0 && (!ws || !aligned(ws, ALIGN)))
        return fail(SG_ERR_INVALID_ARG, "workspace NULL or not 256-byte aligned");
    if (ws_bytes < admm_workspace_bytes(n))
        return fail(SG_ERR_WORKSPACE, "workspace of %zu bytes, %zu needed", ws_bytes, admm_workspace_bytes(n));
    return SG_OK;
}

int sg_admm_opacity_step(int64_t n, const float *opac, const float *importance, int64_t kappa, float *lambda,
                         float *opac_tilde, void *ws, size_t ws_bytes, void *stream) {
    g_err[0] = '\0';
    int st = admm_check(n, ws, ws_bytes);
    if (st != SG_OK) return st;
    if (n > 0 && (!opac || !lambda || !opac_tilde))
        return fail(SG_ERR_INVALID_ARG, "opac, lambda and opac_tilde must not be NULL");
    SG_CUDA(launch_admm_step(0, n, opac, importance, nullptr, kappa, lambda, opac_tilde, ws,
                             static_cast<cudaStream_t>(stream)),
            "ADMM opacity step");
    return SG_OK;
}

int sg_admm_sharpness_step(int64_t n_lobes, const float *sharp, const float *amp, int64_t kappa, float *lambda,
                           float *sharp_tilde, void *ws, size_t ws_bytes, void *stream) {
    g_err[0] = '\0';
    int st = admm_check(n_lobes, ws, ws_bytes);
    if (st != SG_OK) return st;
    if (n_lobes > 0 && (!sharp || !amp || !lambda || !sharp_tilde))
        return fail(SG_ERR_INVALID_ARG, "sharp, amp, lambda and sharp_tilde must not be NULL");
    SG_CUDA(launch_admm_step(1, n_lobes, sharp, nullptr, amp, kappa, lambda, sharp_tilde, ws,
                             static_cast<cudaStream_t>(stream)),
            "ADMM sharpness step");
    return SG_OK;
}

int sg_admm_penalty_grad(int64_t n, const float *x, const float *x_tilde, const float *lambda, float delta,
                         float *grad, void *stream) {
    g_err[0] = '\0';
    if (n < 0) return fail(SG_ERR_INVALID_ARG, "n < 0");
    if (n > 0 && (!x || !x_tilde || !lambda || !grad))
        return fail(SG_ERR_INVALID_ARG, "x, x_tilde, lambda and grad must not be NULL");
    SG_CUDA(launch_penalty_grad(n, x, x_tilde, lambda, delta, grad, static_cast<cudaStream_t>(stream)),
            "ADMM penalty gradient");
    return SG_OK;
}

size_t sg_postprocess_workspace_bytes(int64_t n) { return post_workspace_bytes(n); }

static int post_check(const sg_scene *in, const void *ws, size_t ws_bytes) {
    if (!in) return fail(SG_ERR_INVALID_ARG, "scene must not be NULL");
    if (in->n < 0 || in->n >= (int64_t)INT32_MAX || in->n_lobes < 0 || in->n_lobes >= (int64_t)INT32_MAX)
        return fail(SG_ERR_INVALID_ARG, "sizes out of range");
    if (in->dtype_geom != SG_F32 || in->dtype_lobe != SG_F32 || in->dtype_sharp != SG_F32)
        return fail(SG_ERR_INVALID_ARG, "post-processing reads binary32 scenes only");
    if (in->n > 0) {
        const void *req[] = {in->means, in->scales, in->quats, in->opac, in->gmask, in->c0, in->lobe_off};
        for (const void *p : req)
            if (!p) return fail(SG_ERR_INVALID_ARG, "a Gaussian array is NULL");
    }
    if (in->n_lobes > 0 && (!in->axis || !in->sharp || !in->amp || !in->lmask))
        return fail(SG_ERR_INVALID_ARG, "a lobe array is NULL");
    if (!ws || !aligned(ws, ALIGN)) return fail(SG_ERR_INVALID_ARG, "workspace NULL or not 256-byte aligned");
    if (ws_bytes < post_workspace_bytes(in->n))
        return fail(SG_ERR_WORKSPACE, "workspace of %zu bytes, %zu needed", ws_bytes, post_workspace_bytes(in->n));
    return SG_OK;
}

int sg_postprocess_plan(const sg_scene *in, float tau_opacity, float tau_sharpness, void *ws, size_t ws_bytes,
                        int64_t *n_out, int64_t *l_out, void *stream) {
    g_err[0] = '\0';
    int st = post_check(in, ws, ws_bytes);
    if (st != SG_OK) return st;
    uint64_t totals[3] = {0, 0, 0};   // Gaussians, lobes, device status
    SG_CUDA(launch_post_plan(*in, tau_opacity, tau_sharpness, ws, totals, static_cast<cudaStream_t>(stream)),
            "post-processing plan");
    if (totals[2] != (uint64_t)SG_OK)
        return fail(SG_ERR_TIMEOUT, "the plan's bounded device wait expired (workspace unspecified)");
    if (n_out) *n_out = (int64_t)totals[0];
    if (l_out) *l_out = (int64_t)totals[1];
    return SG_OK;
}

int sg_postprocess_apply(const sg_scene *in, float tau_opacity, float tau_sharpness, const void *ws,
                         size_t ws_bytes, const sg_scene *out, void *stream) {
    g_err[0] = '\0';
    int st = post_check(in, ws, ws_bytes);
    if (st != SG_OK) return st;
    if (!out || !out->lobe_off) return fail(SG_ERR_INVALID_ARG, "out and out->lobe_off must not be NULL");
    if (out->n > 0) {
        const void *req[] = {out->means, out->scales, out->quats, out->opac, out->gmask, out->c0};
        for (const void *p : req)
            if (!p) return fail(SG_ERR_INVALID_ARG, "an output Gaussian array is NULL");
    }
    if (out->n_lobes > 0 && (!out->axis || !out->sharp || !out->amp || !out->lmask))
        return fail(SG_ERR_INVALID_ARG, "an output lobe array is NULL");
    SG_CUDA(launch_post_apply(*in, tau_sharpness, ws, *out, out->n, out->n_lobes,
                              static_cast<cudaStream_t>(stream)),
            "post-processing apply");
    return SG_OK;
}

int sg_forward_status(const void *ws, uint64_t *n_pairs, int32_t *status, void *stream) {
    if (!ws || !aligned(ws, ALIGN)) return fail(SG_ERR_INVALID_ARG, "workspace NULL or not 256-byte aligned");
    // the counters sit right after the batch table, whatever the sizes
    const uint64_t *counters = reinterpret_cast<const uint64_t *>(static_cast<const char *>(ws) + al(sizeof(Batch)));
    uint64_t host[CNT_N] = {};
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    SG_CUDA(cudaMemcpyAsync(host, counters, sizeof(host), cudaMemcpyDeviceToHost, s), "read status");
    SG_CUDA(cudaStreamSynchronize(s), "read status");
    if (n_pairs) *n_pairs = host[CNT_PAIRS];
    if (status) *status = (int32_t)host[CNT_STATUS];
    return SG_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Backward with library-owned scratch, for callers that cannot allocate
// device memory while rendering
// ---------------------------------------------------------------------------
namespace {

// Scratch of sg_render_backward_noalloc: batch table, counters and the
// [M][9] per-entry 2D-gradient accumulators. Every device that loads the
// library holds it until the process exits.
__device__ __align__(256) unsigned char g_noalloc_scratch[SG_NOALLOC_SCRATCH_BYTES];

constexpr int kNoallocMaxDevices = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_addr[kNoallocMaxDevices] = {};

// Device address of g_noalloc_scratch on the current device. In host code the
// array's name stands for the symbol, not for device memory, so the address is
// looked up once per device (with that device current) and cached.
int noalloc_scratch(void **out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "no-alloc backward: cudaGetDevice");
    if (dev < 0 || dev >= kNoallocMaxDevices)
        return fail(SG_ERR_INVALID_ARG, "no-alloc backward: device %d out of range", dev);
    std::lock_guard<std::mutex> g(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "no-alloc backward: cudaGetSymbolAddress");
        g_noalloc_addr[dev] = p;
    }
    *out = g_noalloc_addr[dev];
    return SG_OK;
}

}  // namespace

extern "C" int sg_render_backward_noalloc(const sg_scene *scene, const sg_camera *cams, int n_views,
                                          const void *ws, size_t ws_bytes, const float *T_final,
                                          const int32_t *last, const float *d_img, const sg_grads *grads,
                                          void *stream_) {
    g_err[0] = '\0';
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    Batch b;   // host table on the stack: no heap allocation either
    int st = build_batch(scene, 1, cams, nullptr, n_views, true, b);
    if (st != SG_OK) return st;
    if (!grads) return fail(SG_ERR_INVALID_ARG, "grads must not be NULL");
    b.scene[0].grads = grads[0];
    if (!T_final || !last || !d_img) return fail(SG_ERR_INVALID_ARG, "T_final, last and d_img must not be NULL");
    if (!ws || !aligned(ws, ALIGN)) return fail(SG_ERR_INVALID_ARG, "workspace NULL or not 256-byte aligned");
    const size_t need = bwd_layout(b).needed;   // one block per tile: no tile order
    if (need > (size_t)SG_NOALLOC_SCRATCH_BYTES)
        return fail(SG_ERR_WORKSPACE,
                    "no-alloc backward needs %zu bytes of scratch for %llu entries; the static scratch holds "
                    "%zu bytes; use sg_render_backward with caller scratch",
                    need, (unsigned long long)b.n_entries, (size_t)SG_NOALLOC_SCRATCH_BYTES);
    const uint64_t cap = capacity_for(b, ws_bytes);
    if (cap == UINT64_MAX) return fail(SG_ERR_WORKSPACE, "workspace smaller than its fixed part");
    void *scratch = nullptr;
    st = noalloc_scratch(&scratch);
    if (st != SG_OK) return st;
    const WsLayout L = make_layout(b, cap);
    const char *w = static_cast<const char *>(ws);
    const Rec *rec = reinterpret_cast<const Rec *>(w + L.rec);
    const uint32_t *tt = reinterpret_cast<const uint32_t *>(w + L.tiles_touched);
    const uint2 *ranges = reinterpret_cast<const uint2 *>(w + L.ranges);
    const uint32_t *pv_final = reinterpret_cast<const uint32_t *>(w + L.pval_final);
    char *bw = static_cast<char *>(scratch);
    const BwdLayout BL = bwd_layout(b);
    Batch *db = reinterpret_cast<Batch *>(bw + BL.batch);
    uint64_t *counters = reinterpret_cast<uint64_t *>(bw + BL.counters);
    float *dg = reinterpret_cast<float *>(bw + BL.dg);
    const uint64_t M = L.M;
    BlendShape shape{};   // one block per tile: no tile order or work counter needed
    shape.pixels_per_thread = tuning().bwd_pixels_per_thread;
    shape.batch = tuning().bwd_batch ? tuning().bwd_batch : kDefaultBatch;
    shape.status = reinterpret_cast<const uint64_t *>(w + L.counters) + CNT_STATUS;   // the forward's
    // the setup kernel rewrites the table and counters and clears the accumulators
    ZeroRegions z;
    z.ptr[0] = reinterpret_cast<uint32_t *>(dg);
    z.words[0] = 9 * M;
    SG_CUDA(launch_setup(b, db, counters, stream, z), "setup");
    SG_CUDA(launch_blend_backward(db, b.n_tiles, ranges, pv_final, rec, T_final, last, d_img, dg, shape,
                                  nullptr, stream),
            "blend backward");
    SG_CUDA(launch_preprocess_backward(b, db, tt, reinterpret_cast<const uint8_t *>(w + L.clamp), dg, M, stream), "preprocess backward");
    return SG_OK;
}
