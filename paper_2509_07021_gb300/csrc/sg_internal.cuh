// Internal declarations shared by the kernel translation units of the
// SG-splatting rasterizer (sm_103a). Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <cstddef>
#include <cstdint>

#include "../../include/sgsplat.h"

namespace sgk {

constexpr int TILE = SG_TILE;             // 16x16 pixel tiles
constexpr int BLEND_THREADS = TILE * TILE;
constexpr int PRE_THREADS = 256;
constexpr int PRE_RUN = 512;    // scene Gaussians per block of the several-view preprocess kernels

// Per-view camera and packing offsets. Built on the host, copied into the
// workspace by k_setup so that kernels take a single pointer.
struct ViewDesc {
    float fx, fy, cx, cy;
    float V[12];          // world->camera [R|t], row-major
    float campos[3];      // camera centre in world space (-R^T t)
    float near_plane;
    float bg[3];
    int32_t W, H, tiles_x, tiles_y;
    int32_t scene;        // index into Batch::scene
    uint32_t tile_off;    // first global tile id of the view
    uint32_t grp_off;     // first group of 32 tiles of the view (the binning's scan)
    float limx, limy;     // guard band: 1.3 tan(fov / 2) per axis
    uint64_t pix_off;     // first pixel of the view in T_final / last (img: x3)
    uint64_t ent_off;     // first (view, Gaussian) entry of the view
};

struct SceneDesc {
    const void *means, *scales, *quats, *opac;
    const float *gmask, *c0;
    const int32_t *lobe_off;
    const void *axis, *sharp, *amp;
    const float *lmask;
    const float *sh;      // SH3 coefficients [3][16][N] (color_model SH3)
    float *importance;    // forward output: sum of alpha T per Gaussian (null: not wanted)
    sg_grads grads;
    int64_t n, n_lobes;
    int32_t dtype_geom, dtype_lobe, dtype_sharp, color_model;
    uint32_t blk_off;     // first block of the scene in the per-Gaussian grids (PRE_THREADS a block)
    uint32_t run_off;     // and in the several-view grids (PRE_RUN a block)
};

struct Batch {
    int32_t n_views, n_scenes;
    uint32_t n_tiles;
    uint32_t scene_blocks;   // blocks of 256 scene Gaussians over all scenes
    uint32_t max_views_per_scene;
    uint32_t n_groups;       // groups of 32 tiles over all views
    uint32_t scene_runs;     // blocks of PRE_RUN scene Gaussians over all scenes
    uint32_t pad0;
    uint64_t n_entries;
    ViewDesc view[SG_MAX_VIEWS];
    SceneDesc scene[SG_MAX_SCENES];
};

// One projected Gaussian: 48 bytes. The tile binning reads the first 24 bytes
// (one 32-byte sector), the blend the first 40.
struct __align__(16) Rec {
    float4 a;   // x, y, conic A, conic B
    float4 b;   // conic C, tile-binning bound t (tile_reach_threshold), o' = m_g * o, r
    float4 c;   // g, b, radius, depth
};

// Device counters kept in the workspace.
enum : int {
    CNT_ENTRIES = 0,   // (view, Gaussian) entries
    CNT_PAIRS = 1,     // (tile, Gaussian) pairs of the forward
    CNT_STATUS = 2,    // sg_status of the last batched forward
    CNT_EVALS = 3,     // pair evaluations (counting kernels)
    CNT_TILES = 4,     // tiles
    CNT_QUEUE = 5,     // persistent-blend work counter
    CNT_DUP_BLOCK = 6, // chunk cutter / duplicate kernel: next logical block
    CNT_WRITTEN = 7,   // pairs written (min(pairs, capacity)): the tile sort's count
    CNT_N = 8
};

// Radix sort / scan geometry.
constexpr int RS_THREADS = 256;
#ifndef SG_RS_ITEMS
#define SG_RS_ITEMS 12
#endif
constexpr int RS_ITEMS = SG_RS_ITEMS;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;   // 3072 keys per block
constexpr int RS_RADIX = 256;

// Byte offsets of every workspace buffer (host computed, identical for the
// forward and the backward of one call).
struct WsLayout {
    size_t batch, counters, rec, tiles_touched, rect, clamp, dkey0, dval0, dkey1, dval1,
        dup_flags, ranges, order, order_scratch, walk_place, bin, bin_start, scan_words, hist, aux_depth, aux_tile;
    size_t pval_final, pkey_final, pval_tmp, pkey_tmp, total;
    uint64_t M, n_tiles, cap;
    int tile_bits, tile_passes;
    bool chunked;         // tile sort by chunks (launch_bin_pairs) instead of radix passes
    bool by_view;         // the depth sort orders the entries by view first
    bool matrix_in_img;   // the count matrix takes the image's memory (else hist's)
    bool depth_in_img;    // so do, before it, the depth sort's look-back flags
    bool walk;            // the forward files walk lengths for the backward's tile order
    uint32_t bin_chunks;  // most chunks: rows of the matrix
    uint32_t bin_row;     // words per row of the matrix: the largest view's tiles, padded to 4
};

__host__ __device__ inline uint64_t div_up(uint64_t a, uint64_t b) { return (a + b - 1) / b; }

// A workspace buffer the layout does not hold.
constexpr size_t NO_OFFSET = ~(size_t)0;

// ---------------------------------------------------------------------------
// Tight tile binning. A pair (tile, Gaussian) can only blend where
// alpha = o' exp(-q / 2) >= 1/255, q = A dx^2 + 2 B dx dy + C dy^2 (the conic),
// i.e. inside the ellipse q <= 2 ln(255 o'). Of the tiles of the 3-sigma
// rectangle, only those whose box of pixel centres meets that ellipse get a
// pair; the others would be skipped at every pixel, so leaving them out changes
// no image and no gradient. The ellipse is enlarged (1 % + 0.01 in q, 0.02 px)
// so that binary32 rounding here or in the blend can only keep extra tiles.
// Preprocess counts the tiles and duplicate enumerates them with this same
// code (explicitly rounded operations), so the two agree exactly.
// ---------------------------------------------------------------------------
struct TileReach {
    float x, y, B, det, At, ymax, m, invA;
    int mode;   // 0: reaches nothing, 1: ellipse, 2: whole rectangle (degenerate conic)
};

// The tile binning is a decision recipe like cull and rectangle: every step is
// one binary32 operation with round-to-nearest (no contraction), so that a
// restatement in numpy float32 states exactly which tiles are kept. Its
// constants are exact binary32 values (hexadecimal literals).
constexpr float TR_C7 = 0x1.24924ap-3f;      // 1/7
constexpr float TR_C5 = 0x1.99999ap-3f;      // 1/5
constexpr float TR_C3 = 0x1.555556p-2f;      // 1/3
constexpr float TR_INV_LN2 = 0x1.715476p+0f; // 1/ln 2
constexpr float TR_LN2X2 = 0x1.62e430p+0f;   // 2 ln 2
constexpr float TR_GROW = 0x1.028f5cp+0f;    // 1.01
constexpr float TR_ADD = 0x1.47ae14p-7f;     // 0.01
constexpr float TR_PAD = 0x1.47ae14p-6f;     // 0.02 px

// log2 of a positive normal x: exponent plus ln(m) / ln 2 for the mantissa
// m in [1, 2), ln m = 2 atanh(s) with s = (m - 1) / (m + 1) <= 1/3, summed to
// s^7 (relative error below 1e-5, far inside the 1 % enlargement below).
__device__ __forceinline__ float log2_recipe(float x) {
    const uint32_t u = __float_as_uint(x);
    const float e = (float)((int)((u >> 23) & 255u) - 127);
    const float m = __uint_as_float((u & 0x007FFFFFu) | 0x3F800000u);
    const float s = __fdiv_rn(__fsub_rn(m, 1.0f), __fadd_rn(m, 1.0f));
    const float s2 = __fmul_rn(s, s);
    float P = __fadd_rn(__fmul_rn(s2, TR_C7), TR_C5);
    P = __fadd_rn(__fmul_rn(P, s2), TR_C3);
    P = __fadd_rn(__fmul_rn(P, s2), 1.0f);
    const float lnm = __fmul_rn(__fmul_rn(2.0f, s), P);
    return __fadd_rn(e, __fmul_rn(lnm, TR_INV_LN2));
}

// Enlarged bound on q where alpha can reach 1/255: 2 ln(255 o') (1 + 1 %) + 0.01;
// negative when o' < 1/255 (alpha <= o' < 1/255 everywhere). Computed once per
// entry by preprocess and kept in its record.
__device__ __forceinline__ float tile_reach_threshold(float op) {
    if (!(op >= 1.0f / 255.0f)) return -1.0f;
    const float t0 = __fmul_rn(TR_LN2X2, log2_recipe(__fmul_rn(255.0f, op)));
    return __fadd_rn(__fmul_rn(t0, TR_GROW), TR_ADD);
}

__device__ __forceinline__ void tile_reach_init(float x, float y, float A, float B, float C, float t,
                                                TileReach &R) {
    R.x = x; R.y = y; R.B = B;
    R.det = R.At = R.ymax = R.m = R.invA = 0.f;
    if (!(t >= 0.f)) { R.mode = 0; return; }
    R.det = __fsub_rn(__fmul_rn(A, C), __fmul_rn(B, B));
    if (!(A > 0.f) || !(C > 0.f) || !(R.det > 0.f) || !isfinite(t) || !isfinite(R.det)) {
        R.mode = 2;
        return;
    }
    R.At = __fmul_rn(A, t);
    R.ymax = __fsqrt_rn(__fdiv_rn(R.At, R.det));
    const float xmax = __fsqrt_rn(__fdiv_rn(__fmul_rn(C, t), R.det));
    R.m = __fdiv_rn(__fmul_rn(B, xmax), C);   // dy of the right-most point is -m, of the left-most +m
    R.invA = __frcp_rn(A);
    R.mode = isfinite(R.ymax) && isfinite(R.m) && isfinite(R.At) && isfinite(R.invA) ? 1 : 2;
}

// Columns [c0, c1) of tile row ty (within [x0, x1)) that the enlarged ellipse
// reaches. Over the row's band of dy, the ellipse's right edge
// x_r(dy) = (-B dy + sqrt(A t - det dy^2)) / A is concave with its maximum at
// dy = -m (m = B xmax / C), the left edge convex with its minimum at dy = +m:
// both extremes are taken at those points clamped into the band.
__device__ __forceinline__ void tile_reach_row(const TileReach &R, int ty, int x0, int x1, int &c0, int &c1) {
    c0 = c1 = x0;
    if (R.mode == 0) return;
    if (R.mode == 2) { c1 = x1; return; }
    const float pad = TR_PAD;
    float lo = __fsub_rn(__fsub_rn((float)(ty * SG_TILE), R.y), pad);
    float hi = __fadd_rn(__fsub_rn((float)(ty * SG_TILE + SG_TILE - 1), R.y), pad);
    lo = fmaxf(lo, -R.ymax);
    hi = fminf(hi, R.ymax);
    if (!(lo <= hi)) return;
    const float dr = fminf(fmaxf(-R.m, lo), hi), dl = fminf(fmaxf(R.m, lo), hi);
    const float sr = __fsqrt_rn(fmaxf(0.f, __fsub_rn(R.At, __fmul_rn(R.det, __fmul_rn(dr, dr)))));
    const float sl = __fsqrt_rn(fmaxf(0.f, __fsub_rn(R.At, __fmul_rn(R.det, __fmul_rn(dl, dl)))));
    const float xr = __fadd_rn(__fadd_rn(R.x, __fmul_rn(__fsub_rn(sr, __fmul_rn(R.B, dr)), R.invA)), pad);
    const float xl = __fsub_rn(__fsub_rn(R.x, __fmul_rn(__fadd_rn(sl, __fmul_rn(R.B, dl)), R.invA)), pad);
    // tile tx is reached iff 16 tx <= xr and 16 tx + 15 >= xl (clamped to the rectangle first;
    // scaling by 1/16 is exact)
    const float fx0 = (float)(x0 * SG_TILE - SG_TILE), fx1 = (float)(x1 * SG_TILE);
    const float a = ceilf(__fmul_rn(__fsub_rn(fminf(fmaxf(xl, fx0), fx1), (float)(SG_TILE - 1)), 1.0f / SG_TILE));
    const float b = floorf(__fmul_rn(fminf(fmaxf(xr, fx0), fx1), 1.0f / SG_TILE));
    c0 = max(x0, (int)a);
    c1 = max(c0, min(x1, (int)b + 1));
}

// ---------------------------------------------------------------------------
// block-wide exclusive scan helpers
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T warp_inclusive(T x) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) >= (unsigned)o) x += y;
    }
    return x;
}

// exclusive scan over blockDim.x (multiple of 32, <= 1024) values; returns the
// exclusive prefix and writes the block total.
template <typename T>
__device__ __forceinline__ T block_exclusive(T x, T &total, T *sh /* >= 32 */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const T inc = warp_inclusive(x);
    if (lane == 31) sh[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nw ? sh[lane] : T(0);
        const T wi = warp_inclusive(w);
        sh[lane] = wi - w;
        if (lane == 31) sh[32] = wi;
    }
    __syncthreads();
    const T r = sh[warp] + inc - x;
    total = sh[32];
    __syncthreads();
    return r;
}

// Decoupled look-back words of 64 bits (the duplicate blocks, the ADMM
// selection): 2 status bits (aggregate, inclusive prefix) and a 62-bit count.
constexpr uint64_t DL_AGG = 1ull << 62, DL_INC = 2ull << 62, DL_VAL = (1ull << 62) - 1ull;

__device__ __forceinline__ uint64_t ld_relaxed64(const uint64_t *p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed64(uint64_t *p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" : : "l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ uint64_t warp_sum64(uint64_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Exclusive prefix of the counts of logical blocks [0, blk) (warp 0 of the
// block; all its lanes return it). The block has published its own count
// (DL_AGG) before it calls this, so successors never wait on a block that waits. Predecessors are read 32 at a time;
// a run of ready words ending in an inclusive prefix completes the sum. Unready
// words are polled at most spin_limit times; past that the status word gets
// SG_ERR_TIMEOUT and the (smaller) partial prefix is returned.
__device__ __forceinline__ uint64_t block_lookback64(uint64_t *__restrict__ dflags, uint64_t blk, uint64_t count,
                                                 uint32_t spin_limit, uint64_t *status) {
    const int lane = threadIdx.x & 31;
    uint64_t excl = 0;
    int64_t p = (int64_t)blk - 1;
    uint32_t spins = 0;
    while (p >= 0) {
        const int64_t q = p - lane;
        const uint64_t f = q >= 0 ? ld_relaxed64(dflags + q) : DL_INC;   // before block 0: prefix 0
        const uint32_t unready = __ballot_sync(0xffffffffu, (f & ~DL_VAL) == 0ull);
        const uint32_t inc = __ballot_sync(0xffffffffu, (f & DL_INC) != 0ull);
        const int first_unready = unready ? __ffs(unready) - 1 : 32;
        const int first_inc = inc ? __ffs(inc) - 1 : 32;
        if (first_inc < first_unready) {
            excl += warp_sum64(lane <= first_inc ? (f & DL_VAL) : 0ull);
            break;
        }
        excl += warp_sum64(lane < first_unready ? (f & DL_VAL) : 0ull);
        p -= first_unready;
        if (first_unready < 32) {
            if (++spins >= spin_limit) {
                if (lane == 0) atomicExch(reinterpret_cast<unsigned long long *>(status),
                                          (unsigned long long)SG_ERR_TIMEOUT);
                break;
            }
            __nanosleep(32);
        }
    }
    if (lane == 0) st_relaxed64(dflags + blk, DL_INC | ((excl + count) & DL_VAL));
    return excl;
}

// ---------------------------------------------------------------------------
// Programmatic dependent launch along the render chain. Each kernel of the
// chain is launched with programmatic stream serialisation, so the GPU may
// schedule its blocks while the kernel before it drains; its first statement
// waits until that kernel has completed and its writes are visible, so the
// chain keeps plain stream order. Right after the wait it lets the next kernel
// be scheduled in turn (the binning kernels do not, see chain_wait, and k_duplicate is
// launched in plain order). Both instructions are no-ops for a kernel launched
// without the attribute.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void chain_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// For a kernel whose successor needs most of an SM's shared memory: without the
// early trigger the successor's blocks are only placed once this kernel has
// drained, evenly over the SMs, instead of wherever it leaves room (measured
// on the placement after the scan: 328 -> 175 us at 11.8M pairs).
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_chain_smem(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                     cudaStream_t s, Args &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Args &&>(args)...);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_chain(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t s,
                                Args &&...args) {
    return launch_chain_smem(kernel, grid, block, 0, s, static_cast<Args &&>(args)...);
}

// Process-wide count of kernels this library has launched (sg_kernel_launches).
void count_launches(int n);

// ---- launchers (host side, defined in the .cu files) ----
// Buckets by list length on a log scale with 8 buckets per octave (exponent and
// the 3 bits below the leading one), longest bucket first; inside a bucket the
// order is whatever the atomics give (it only steers scheduling).
constexpr int TB_BUCKETS = 256;
__device__ __forceinline__ uint32_t len_bucket(uint32_t len) {
    len |= 1u;
    const uint32_t e = 31u - (uint32_t)__clz(len);              // 0..31
    const uint32_t m = e >= 3u ? (len >> (e - 3u)) & 7u : (len << (3u - e)) & 7u;
    return e * 8u + m;                                           // 0..255
}

// Tiles by descending walk length (a tile's largest last position): written by the
// setup kernel's last blocks while the others zero their regions (n = 0: none).
struct TileOrder {
    const uint32_t *counts = nullptr;   // [TB_BUCKETS] tiles per walk-length bucket
    const uint32_t *place = nullptr;    // [n] bucket << 24 | rank inside it
    const uint32_t *fallback = nullptr; // [n] the order where the counts do not add up to n (an
                                        // importance forward files no walk lengths)
    uint32_t *order = nullptr;          // [n]
    uint32_t n = 0;
};
// Up to N device regions of 32-bit words that the setup kernel zeroes.
// Regions the setup kernel fills: word i of region r gets even[r] if i is
// even, else 0 (even[r] = 0: plain zeroing).
struct ZeroRegions {
    static constexpr int N = 6;
    uint32_t *ptr[N] = {};
    uint64_t words[N] = {};
    uint32_t even[N] = {};
};
cudaError_t launch_setup(const Batch &b, Batch *dst, uint64_t *counters, cudaStream_t s,
                         const ZeroRegions &z = ZeroRegions(), const TileOrder &o = TileOrder());
// clamp [M]: bit ch set where colour channel ch was clamped by max(c, 0).
// view_pairs, view_visible (zeroed): receive each view's pairs and its entries
// with at least one pair.
cudaError_t launch_preprocess(const Batch &hb, const Batch *db, Rec *rec, uint32_t *tiles_touched,
                              uint2 *rect, uint32_t *dkey, uint8_t *clamp,
                              unsigned long long *view_pairs, uint32_t *view_visible, cudaStream_t s);
cudaError_t launch_preprocess_backward(const Batch &hb, const Batch *db,
                                       const uint32_t *tiles_touched, const uint8_t *clamp, const float *dg,
                                       uint64_t M, cudaStream_t s);

// Most keys one sort takes (its look-back words carry 30-bit counts).
constexpr uint64_t SORT_MAX_KEYS = (1ull << 30) - 1;
constexpr uint32_t SORT_DROP_KEY = 0xFFFFFFFFu;
int radix_passes(int bits);
// Bound on a sort block's polls of an unpublished predecessor before it gives
// up and records SG_ERR_TIMEOUT (0: the default, 2^20).
void set_sort_wait_polls(uint32_t polls);
uint32_t sort_wait_polls();
// Look-back flag words of `passes` passes over up to max_n keys (of the depth sort: with
// the group words of its grouped look-back).
uint64_t sort_flag_words(uint64_t max_n, int passes);
uint64_t depth_flag_words(uint64_t max_n, int passes);

// Stable sort of the entries by depth bits or (by_view) by (view, depth bits), entries whose
// key in k0 is SORT_DROP_KEY left out (k0: one key per entry; the values, entry indices, are
// made by the first pass): the four depth digits, then, by_view, one pass whose
// digit is the entry's view (its counts, aux hist row VIEW_PASS, are
// preprocess's). The order ends in (k0, v0), by_view in (k1, v1); aux (zeroed by the caller) then holds the kept count and the status.
constexpr int VIEW_PASS = 4;
struct SortAux {
    uint32_t hist[5][RS_RADIX];   // global digit counts per pass
    uint32_t tile_ctr[5];         // tile counter per pass
    uint32_t status;              // 0 or SG_ERR_TIMEOUT
    uint64_t kept;                // keys other than SORT_DROP_KEY (drop mode)
};
cudaError_t launch_depth_sort(const Batch *db, bool by_view, uint32_t *k0, uint32_t *v0, uint32_t *k1, uint32_t *v1,
                              const uint64_t *n_dev, uint64_t max_n, uint32_t *hist, SortAux *aux, cudaStream_t s);

// ---------------------------------------------------------------------------
// Binning by chunks: (tile, entry) pairs in (tile, depth, entry) order without
// a sort of the pairs by key digits, for views of up to BIN_MAX_ROW tiles (one
// chunk's tile counters fit shared memory) and up to bin_max_pairs. The depth-ordered entries of each
// view are cut into chunks of about equal cost; each chunk counts its
// pairs per tile while it writes them out, one scan of the count matrix gives
// every (chunk, tile) its first output position and every tile its range, and
// each chunk places its pairs in order. Larger views take launch_duplicate and
// radix passes over the tile digits.
// ---------------------------------------------------------------------------
constexpr uint32_t BIN_MAX_ROW = 56 * 1024;
// Fewest pairs a chunk is cut for: one placing warp walks 32 pairs a round.
constexpr uint32_t BIN_MIN_CHUNK = 256;
// An entry's share of a chunk's cost besides its pairs (one each).
constexpr uint32_t BIN_ENTRY_COST = 1;
constexpr uint32_t BIN_MAX_CHUNKS = 5 * 152;
// Per-call tables of the binning (workspace; view_pairs zeroed by the setup kernel).
struct BinTab {
    unsigned long long view_pairs[SG_MAX_VIEWS];   // pairs of each view (preprocess)
    uint32_t n_chunks;                             // chunks in use
    uint32_t first_chunk[SG_MAX_VIEWS + 1];        // first chunk of each view
};
// Room for more pairs than this takes the radix passes: a view of more tiles leaves fewer
// chunks a place on the chip (one per SM past 28.8k tiles, two past 18.9k), whose serial
// rounds then take longer than two passes over the pairs. Measured (us, chunks / radix, from
// the ordered entries to the placed pairs): 32400 tiles 7.8M pairs 372 / 413, 15.3M 687 / 661,
// 21.5M 945 / 689, 56M 2618 / 2049; 49152 tiles 10.8M 496 / 499, 44M 2025 / 1291; 27600 tiles 13M
// 420 / 635, 49M 1897 / 1786; 22600 tiles 42M 1565 / 1504; 16000 tiles 32.5M 1030 / 1129. The
// line at two per SM lies between its points.
inline uint64_t bin_max_pairs(uint32_t row) {
    const uint32_t per_sm = (227u * 1024u) / (row * 4u + 1024u);
    return per_sm <= 1u ? 12ull << 20 : per_sm == 2u ? 32ull << 20 : ~0ull;
}
uint32_t bin_chunks(uint64_t cap, uint32_t row, int n_views);   // most chunks of a call with room for cap pairs
struct BinArgs {
    const Batch *db;
    int n_views;
    uint64_t M, cap;                 // entries; pairs the buffers hold (below 2^30)
    uint32_t max_chunks, row, n_groups, n_tiles;
    const uint32_t *sorted_ent;      // the depth sort's order
    const SortAux *aux;              // its kept count and status
    const uint32_t *tiles_touched;
    const uint2 *rect;
    const Rec *rec;
    uint64_t *counters;
    BinTab *tab;
    uint32_t *start, *pair;          // max_chunks + 1 each: first entry (depth order) and first pair of a chunk
    uint32_t *poff;                  // scratch, M words: first pair of each entry of the order
    uint64_t *flags;                 // zeroed, a word per 256 entries (at most that many used): look-back
    uint16_t *pkey;                  // depth-ordered pairs: tile inside the view
    uint32_t *pval;                  //   and entry
    uint32_t *matrix;                // max_chunks x row words, 16-byte aligned
    uint64_t *words;                 // zeroed, 1 + n_groups: ticket and look-back of the scan
    uint2 *ranges;                   // every tile's [first, last + 1) ((0, 0): none)
    uint32_t *order_counts;          // zeroed tile-order bucket counts
    uint32_t *ovals;                 // the placed entries
    uint32_t *okeys;                 // nullable: their global tile ids
    uint64_t *mirror;                // nullable host words: [0] pairs, [1] status
};
constexpr int BIN_CUT_THREADS = 1024, BIN_ITEMS = 8;   // the chunk cutter's most threads, entries per thread
cudaError_t launch_bin_pairs(const BinArgs &a, cudaStream_t s);   // chunks and their pairs
cudaError_t launch_bin_place(const BinArgs &a, cudaStream_t s);   // scan and placement

// duplicateWithKeys over the depth-sorted entries, for the radix tile sort.
// Every block of 256 entries finds the offset of its pairs by a decoupled
// look-back over its predecessors' pair counts (dup_flags: div_up(M, 256) zeroed
// 64-bit words, and counters[CNT_DUP_BLOCK] zeroed), so no separate scan runs.
// The entry count and the depth sort's status come from aux. The last block
// writes the pair total to counters[CNT_PAIRS] (and to mirror[0], host memory
// mapped into the device, when given), min(total, cap) to counters[CNT_WRITTEN],
// and SG_ERR_CAPACITY to counters[CNT_STATUS] when the pairs exceed cap; pairs
// at positions >= cap are not written. It also clears the tile sort's look-back
// flags and builds its digit histograms.
cudaError_t launch_duplicate(const Batch *db, uint64_t M, const uint32_t *sorted_ent, const SortAux *depth_aux,
                             const uint32_t *tiles_touched, const uint2 *rect, const Rec *rec,
                             uint64_t *counters, uint64_t cap, uint32_t *pkey, uint32_t *pval,
                             uint64_t *dup_flags, uint64_t *mirror, cudaStream_t s, int hist_passes,
                             SortAux *sort_aux, uint32_t *flags, uint64_t flag_words);
// Stable LSD radix sort by tile id of launch_duplicate's (key, val) pairs on
// bits [0, bits); counters[CNT_WRITTEN] of them, at most max_n (below 2^30).
// Ping-pongs between (k0,v0) and (k1,v1); the result ends in (k0,v0) when the
// pass count is even, else in (k1,v1). hist: the sort_flag_words(max_n, passes)
// look-back words, aux: the digit histograms, both prepared by
// launch_duplicate. Nothing is sorted when counters[CNT_STATUS] is not SG_OK on
// entry (a bounded wait gave up: the input may hold stale words; or the pairs
// overflowed the capacity); a look-back that gives up sets it to
// SG_ERR_TIMEOUT. ranges: every tile's [first, last + 1) positions, (0, 0) for
// a tile with no pair; on entry every range must hold (RANGE_EMPTY, 0).
// order_counts: the tile order's zeroed bucket counts, incremented here.
// status_mirror (nullable, host memory mapped into the device): receives the
// status after the sort.
constexpr uint32_t RANGE_EMPTY = 0xFFFFFFFFu;
cudaError_t launch_tile_radix_sort(uint32_t *k0, uint32_t *v0, uint32_t *k1, uint32_t *v1, uint64_t *counters,
                                   uint64_t max_n, int bits, uint32_t *hist, SortAux *aux, uint2 *ranges,
                                   uint64_t n_ranges, uint32_t *order_counts, uint64_t *status_mirror,
                                   cudaStream_t s);
// Tiles by descending list length (256 length buckets) into order[n_tiles].
// scratch: TILE_ORDER_WORDS zeroed words whose first 256 already hold the
// bucket counts (filled by the tile sort).
constexpr int TILE_ORDER_WORDS = 512;
// Tile counts whose backward gets an order of its own: its 8-pixel form starts at
// 5632 tiles, and with two or three tiles per resident warp the longest of the last
// decide when the kernel ends (8160 tiles, 5.4M pairs: 646 -> 613 us; 2.7M: 597 -> 588;
// 6700, 3.4M: 632 -> 618; 16000, 9.1M: 1035 -> 1016).
// With fewer tiles several warps share each (3600: 305 us with either order, and the
// forward pays 1 us for the ranks); with more, a warp takes several tiles and the
// forward's order ends as evenly (six scenes in four views each: the same with either).
constexpr uint32_t WALK_ORDER_MIN = 5632, WALK_ORDER_MAX = 16384;
inline bool walk_ordered(uint64_t n_tiles) { return n_tiles > WALK_ORDER_MIN && n_tiles <= WALK_ORDER_MAX; }
cudaError_t launch_tile_order(const uint2 *ranges, uint32_t n_tiles, uint32_t *order, uint32_t *scratch,
                              cudaStream_t s);

// Blend launch shape.
struct BlendShape {
    int pixels_per_thread;
    bool persistent;              // resident blocks pull tiles from *queue
    const uint32_t *tile_order;   // persistent: tiles in this order (null: natural order)
    uint32_t *queue;              // persistent: zeroed work counter
    int grid;                     // persistent: resident blocks
    bool importance;              // forward: accumulate SceneDesc::importance
    const uint64_t *status;       // the forward's status word: SG_ERR_TIMEOUT = lists unusable
    uint32_t *walk_counts;        // forward: TileOrder::counts (zeroed) and ::place, for the backward's
    uint32_t *walk_place;         // tile order (null: none wanted)
    int batch;                    // Gaussians staged per shared-memory batch
};

cudaError_t launch_blend_forward(const Batch *db, uint32_t n_tiles, const uint2 *ranges,
                                 const uint32_t *pval, const Rec *rec, float *img,
                                 float *T_final, int32_t *last, const BlendShape &shape,
                                 unsigned long long *evals, cudaStream_t s);
cudaError_t launch_blend_backward(const Batch *db, uint32_t n_tiles, const uint2 *ranges,
                                  const uint32_t *pval, const Rec *rec, const float *T_final,
                                  const int32_t *last, const float *d_img, float *dg,
                                  const BlendShape &shape, unsigned long long *evals, cudaStream_t s);
// ADMM proximal + dual step (kind 0: opacity, 1: sharpness) and the penalty
// gradient term; workspace bytes for n items.
size_t admm_workspace_bytes(int64_t n);
cudaError_t launch_admm_step(int kind, int64_t n, const float *x, const float *score, const float *amp,
                             int64_t kappa, float *lam, float *x_tilde, void *ws, cudaStream_t s);
cudaError_t launch_penalty_grad(int64_t n, const float *x, const float *x_tilde, const float *lam, float delta,
                                float *grad, cudaStream_t s);

// Post-processing (Sec. 3.3.3): plan (positions; totals and the device status
// read back into totals_host[3]) and apply.
size_t post_workspace_bytes(int64_t n);
cudaError_t launch_post_plan(const sg_scene &sc, float tau_o, float tau_s, void *ws, uint64_t *totals_host,
                             cudaStream_t s);
cudaError_t launch_post_apply(const sg_scene &sc, float tau_s, const void *ws, const sg_scene &out,
                              int64_t n_out, int64_t l_out, cudaStream_t s);

// Resident blocks per SM x SMs for the persistent blend of this shape.
int blend_persistent_grid(bool backward, int pixels_per_thread, int batch);

}  // namespace sgk
