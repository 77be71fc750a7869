// Binning: stable LSD radix sort of u32 (key, value) pairs, duplicateWithKeys,
// the chunked binning and per-tile ranges.
//
// The (tile, depth) ordering of the paper's tile-depth-Gaussian key table
// (Sec. 1, rendering VRAM; the 3DGS binning it inherits) is the order of an
// LSD radix sort of 64-bit keys tile << 32 | depth_bits, equal keys by
// Gaussian id. The depth digits of every pair of one Gaussian are equal, so
// the depth passes are run once per (view, Gaussian) entry, before the
// entries are duplicated into pairs, and the pairs are then binned by tile
// (chunks; radix passes over the tile digits for a view of more tiles than a
// chunk's counters hold, and for large views with many pairs). Duplication walks the entries in depth order and
// both binnings are stable, so the result is identical to the 64-bit sort.
#include "sg_internal.cuh"

#include <algorithm>
#include <atomic>

namespace sgk {

__device__ __forceinline__ uint32_t lanemask_lt() {
    return (1u << (threadIdx.x & 31)) - 1u;
}


// ---------------------------------------------------------------------------
// stable LSD radix sort, 8-bit digits, RS_TILE keys per block, one sweep per pass
// ---------------------------------------------------------------------------
// One kernel histograms every digit position at once and clears the look-back
// flags of every pass (for the radix tile sort the duplicate does both). Each
// pass is then a single kernel: blocks take key
// tiles in order from an atomic counter, rank their keys stably (warp
// match_any + per-warp digit counters), scan the pass's digit histogram for
// the digit bases, publish their digit counts, and get their offsets among
// the tiles before them by looking back (decoupled look-back). A look-back
// spin is bounded: past the bound the block records SG_ERR_TIMEOUT in the
// status word and carries on with a smaller offset (wrong order, still inside
// the array) instead of waiting forever.

__device__ __forceinline__ int find_entry_view(const Batch &b, uint64_t e) {
    int lo = 0, hi = b.n_views - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (b.view[mid].ent_off <= e) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// packed look-back word: 2 status bits, 30 count bits
constexpr uint32_t LB_AGG = 1u << 30, LB_INC = 2u << 30, LB_VAL = (1u << 30) - 1u;
static_assert(LB_VAL == SORT_MAX_KEYS, "look-back count width");
constexpr uint32_t LB_SPIN_LIMIT = 1u << 20;   // default bound on unanswered look-back polls
constexpr int LB_WINDOW = 16;

// Process-wide bound on the polls a block makes of an unpublished predecessor
// before it gives up (sg_tuning.sort_wait_polls; 0 = LB_SPIN_LIMIT).
static std::atomic<uint32_t> g_spin_limit{0};
void set_sort_wait_polls(uint32_t polls) { g_spin_limit.store(polls); }
uint32_t sort_wait_polls() {
    const uint32_t v = g_spin_limit.load();
    return v ? v : LB_SPIN_LIMIT;
}

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed(uint32_t *p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" : : "l"(p), "r"(v) : "memory");
}

// Per-warp private shared histograms keep the shared-memory atomics of keys
// with few distinct digits (the high tile bits) from serialising.
__global__ void __launch_bounds__(RS_THREADS) k_os_hist(const uint32_t *__restrict__ keys,
                                                        const uint64_t *__restrict__ n_dev, uint64_t max_n,
                                                        SortAux *aux, uint32_t *__restrict__ flags,
                                                        uint64_t flag_words) {
    chain_enter();
    constexpr int NW = RS_THREADS / 32;
    __shared__ uint32_t h[NW][4][RS_RADIX];
    constexpr int passes = 4;
    // the look-back flags of every pass start at zero (the passes run after this kernel)
    for (uint64_t i = (uint64_t)blockIdx.x * RS_THREADS + threadIdx.x; i < flag_words;
         i += (uint64_t)gridDim.x * RS_THREADS)
        flags[i] = 0u;
    const int warp = threadIdx.x >> 5;
    for (int w = 0; w < NW; ++w)
        for (int p = 0; p < 4; ++p) h[w][p][threadIdx.x] = 0u;
    __syncthreads();
    const uint64_t n = min(*n_dev, max_n);
    const uint64_t stride = (uint64_t)gridDim.x * RS_THREADS;
    uint32_t kept = 0u;
    auto count = [&](uint32_t k) {
        if (k == SORT_DROP_KEY) return;
        ++kept;
#pragma unroll
        for (int p = 0; p < passes; ++p) atomicAdd(&h[warp][p][(k >> (8 * p)) & 255u], 1u);
    };
    // four keys per 16-byte load (the key arrays are 256-byte aligned), then the tail
    const uint64_t n4 = n / 4;
    const uint4 *k4 = reinterpret_cast<const uint4 *>(keys);
    for (uint64_t j = (uint64_t)blockIdx.x * RS_THREADS + threadIdx.x; j < n4; j += stride) {
        const uint4 q = k4[j];
        count(q.x);
        count(q.y);
        count(q.z);
        count(q.w);
    }
    for (uint64_t j = 4 * n4 + (uint64_t)blockIdx.x * RS_THREADS + threadIdx.x; j < n; j += stride)
        count(keys[j]);
    const uint32_t wk = __reduce_add_sync(0xffffffffu, kept);
    if ((threadIdx.x & 31) == 0 && wk)
        atomicAdd(reinterpret_cast<unsigned long long *>(&aux->kept), (unsigned long long)wk);
    __syncthreads();
    for (int p = 0; p < passes; ++p) {
        uint32_t c = 0u;
        for (int w = 0; w < NW; ++w) c += h[w][p][threadIdx.x];
        if (c) atomicAdd(&aux->hist[p][threadIdx.x], c);
    }
}

// three resident blocks per SM (80 registers a thread); GROUPED: see the look-back;
// VIEW: the digit is the view of the entry `value` (else bits of the key)
template <bool GROUPED, bool VIEW>
__global__ void __launch_bounds__(RS_THREADS, 3) k_os_pass(
    const uint32_t *__restrict__ kin, const uint32_t *__restrict__ vin, uint32_t *__restrict__ kout,
    uint32_t *__restrict__ vout, const uint64_t *__restrict__ n_dev, uint64_t max_n, int pass, int shift,
    uint32_t mask, bool drop, uint32_t *__restrict__ flags, SortAux *aux, uint2 *__restrict__ ranges,
    uint64_t n_ranges, uint32_t spin_limit, const uint64_t *__restrict__ skip_status,
    const Batch *__restrict__ view_of, uint32_t *__restrict__ groups) {
    chain_enter();
    constexpr int NW = RS_THREADS / 32;
    __shared__ uint32_t s_ent[VIEW ? SG_MAX_VIEWS : 1];   // the views' first entries
    auto digit = [&](uint32_t key, uint32_t val) -> uint32_t {
        if (!VIEW) return (key >> shift) & mask;
        int lo = 0, hi = view_of->n_views - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_ent[mid] <= val) lo = mid; else hi = mid - 1;
        }
        return (uint32_t)lo;
    };
    constexpr int PER_WARP = RS_TILE / NW;   // 512 consecutive keys per warp
    __shared__ uint32_t cnt[NW][RS_RADIX];
    __shared__ uint32_t dstart[RS_RADIX];
    __shared__ uint32_t gstart[RS_RADIX];
    __shared__ uint32_t sk[RS_TILE];
    __shared__ uint32_t sv[RS_TILE];
    __shared__ uint32_t shs[33];
    __shared__ uint32_t s_tile;

    // an earlier bounded wait gave up (stale words) or the pairs overflowed (uniform)
    if (skip_status && *skip_status != 0ull) return;
    if (threadIdx.x == 0) s_tile = atomicAdd(&aux->tile_ctr[pass], 1u);
    __syncthreads();
    const uint32_t t = s_tile;
    const uint64_t n = min(*n_dev, max_n);
    const uint64_t base = (uint64_t)t * RS_TILE;
    if (base >= n) return;   // uniform across the block; later tiles exit too
    if (VIEW && (int)threadIdx.x < view_of->n_views) s_ent[threadIdx.x] = (uint32_t)view_of->view[threadIdx.x].ent_off;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int i = 0; i < NW; ++i) cnt[i][threadIdx.x] = 0u;
    __syncthreads();

    uint32_t k[RS_ITEMS], v[RS_ITEMS], r[RS_ITEMS];
    const uint64_t wbase = base + (uint64_t)warp * PER_WARP;
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        const uint64_t j = wbase + (uint64_t)i * 32 + lane;
        const bool ok = j < n;
        k[i] = ok ? kin[j] : 0u;
        v[i] = !ok ? 0u : vin ? vin[j] : (uint32_t)j;   // no values yet: the key's index
    }
    // Warp-local stable ranks. Per item, the lowest lane of each group of equal
    // digits adds the group's size to the warp's counter; shared-memory atomics
    // of one warp take effect in issue order, so the returned bases follow the
    // key order. All atomics are issued before any base is broadcast.
    const uint32_t lt = lanemask_lt();
    uint32_t meta[RS_ITEMS];   // leader lane | (rank inside the group << 5)
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        const uint64_t j = wbase + (uint64_t)i * 32 + lane;
        const bool ok = j < n && !(drop && k[i] == SORT_DROP_KEY);
        const uint32_t d = ok ? digit(k[i], v[i]) : 0x100u;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t below = peers & lt;
        r[i] = (ok && below == 0u) ? atomicAdd(&cnt[warp][d], (uint32_t)__popc(peers)) : 0u;
        meta[i] = (uint32_t)(__ffs(peers) - 1) | ((uint32_t)__popc(below) << 5) | d << 16;
    }
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i)
        r[i] = __shfl_sync(0xffffffffu, r[i], (int)(meta[i] & 31u)) + ((meta[i] >> 5) & 63u);
    __syncthreads();
    // per digit: exclusive offsets over warps, block total, block-local start
    uint32_t run = 0u;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        const uint32_t c = cnt[w][threadIdx.x];
        cnt[w][threadIdx.x] = run;
        run += c;
    }
    const uint32_t d = threadIdx.x;
    // publish this tile's count, then look back for the exclusive prefix
    uint32_t *my = flags + (uint64_t)t * RS_RADIX + d;
    st_relaxed(my, LB_AGG | run);
    uint32_t excl = 0u;
    uint32_t spins = 0;
    if (GROUPED) {
        // A short sort: its tiles all start together, so none finds an inclusive
        // prefix near by and each would add up every count before its own, 16 a step.
        // Instead each group of 16 tiles adds its counts up in one word per digit
        // (5 bits of tiles, 27 of keys), and a tile adds the words of the groups before
        // its own and the counts of its group: two steps up to 256 tiles (549k of
        // 1M keys: 17 -> 12 us a pass).
        const uint32_t g = t / LB_WINDOW;
        atomicAdd(groups + (uint64_t)g * RS_RADIX + d, (1u << 27) + run);
        for (uint32_t q0 = 0; q0 <= g; q0 += LB_WINDOW) {   // windows of groups; the last step: the tile's own group
            const bool own = q0 + LB_WINDOW > g;
            for (int part = 0; part < (own ? 2 : 1); ++part) {
                const uint32_t first = part ? g * LB_WINDOW : q0, last = part ? t : min(g, q0 + LB_WINDOW);
                const uint32_t *src = part ? flags : groups;
                for (;;) {
                    uint32_t fv[LB_WINDOW], sum = 0u;
#pragma unroll
                    for (uint32_t i = 0; i < LB_WINDOW; ++i)
                        fv[i] = first + i < last ? ld_relaxed(src + (uint64_t)(first + i) * RS_RADIX + d) : 0u;
                    bool ready = true;
#pragma unroll
                    for (uint32_t i = 0; i < LB_WINDOW; ++i) {
                        if (first + i >= last) continue;
                        ready = ready && (part ? (fv[i] & ~LB_VAL) != 0u : (fv[i] >> 27) == (uint32_t)LB_WINDOW);
                        sum += part ? fv[i] & LB_VAL : fv[i] & ((1u << 27) - 1u);
                    }
                    if (!ready && ++spins < spin_limit) {
                        __nanosleep(32);
                        continue;
                    }
                    if (!ready) atomicExch(&aux->status, (uint32_t)SG_ERR_TIMEOUT);
                    excl += sum;
                    break;
                }
            }
        }
    } else {
        for (int64_t p = (int64_t)t - 1; p >= 0;) {
            uint32_t fv[LB_WINDOW];
#pragma unroll
            for (int i = 0; i < LB_WINDOW; ++i)
                fv[i] = (p - i >= 0) ? ld_relaxed(flags + (uint64_t)(p - i) * RS_RADIX + d) : LB_INC;
            int used = 0;
            bool found = false, stalled = false;
#pragma unroll
            for (int i = 0; i < LB_WINDOW; ++i) {
                if (found || stalled) continue;
                if ((fv[i] & ~LB_VAL) == 0u) { stalled = true; continue; }
                excl += fv[i] & LB_VAL;
                ++used;
                if (fv[i] & LB_INC) found = true;
            }
            if (found) break;
            p -= used;
            if (stalled) {
                if (++spins >= spin_limit) {
                    atomicExch(&aux->status, (uint32_t)SG_ERR_TIMEOUT);
                    break;
                }
                __nanosleep(32);
            }
        }
        st_relaxed(my, LB_INC | ((excl + run) & LB_VAL));
    }
    uint32_t tot, all;
    const uint32_t ds = block_exclusive<uint32_t>(run, tot, shs);
    // global start of digit d in this pass: keys of smaller digits (all tiles) + earlier tiles
    const uint32_t dbase = block_exclusive<uint32_t>(aux->hist[pass][d], all, shs);
    dstart[d] = ds;
    gstart[d] = dbase + excl;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RS_ITEMS; ++i) {
        const uint64_t j = wbase + (uint64_t)i * 32 + lane;
        if (j < n && !(drop && k[i] == SORT_DROP_KEY)) {
            const uint32_t dd = meta[i] >> 16;
            const uint32_t pos = dstart[dd] + cnt[warp][dd] + r[i];
            sk[pos] = k[i];
            sv[pos] = v[i];
        }
    }
    __syncthreads();
    const int items = (int)tot;   // the block's kept keys
    // Last pass with ranges: the block's keys are now in full key order (its
    // input is sorted by the lower digits, its local sort by this one is
    // stable), so each run of one key is contiguous in the output; its ends
    // bound that key's range. Skipped when the count exceeded the capacity.
    const bool want_ranges = ranges != nullptr && *n_dev <= max_n;
    for (int p = threadIdx.x; p < items; p += RS_THREADS) {
        const uint32_t key = sk[p];
        const uint32_t dd = digit(key, sv[p]);
        const uint32_t o = gstart[dd] + (uint32_t)p - dstart[dd];
        // after a pass that gave up a wait, stale keys can disagree with the
        // histogram: their positions are cut at the buffers' end
        if (o >= max_n) continue;
        kout[o] = key;
        vout[o] = sv[p];
        if (want_ranges && key < n_ranges) {
            if (p == 0 || sk[p - 1] != key) atomicMin(&ranges[key].x, o);
            if (p == items - 1 || sk[p + 1] != key) atomicMax(&ranges[key].y, o + 1u);
        }
    }
}

int radix_passes(int bits) { return bits <= 0 ? 0 : (bits + 7) / 8; }

uint64_t sort_flag_words(uint64_t max_n, int passes) {
    return div_up(max_n, RS_TILE) * RS_RADIX * (uint64_t)passes;   // a word per tile and digit
}

uint64_t depth_flag_words(uint64_t max_n, int passes) {
    const uint64_t tiles = div_up(max_n, RS_TILE);   // and a word per group of tiles and digit
    return (tiles + div_up(tiles, LB_WINDOW)) * RS_RADIX * (uint64_t)passes;
}

__device__ __forceinline__ uint32_t len_bucket(const uint2 r) { return len_bucket(r.y - r.x); }

// After the radix tile sort: tiles that got no pair get the range (0, 0), every
// tile joins its list-length bucket (len_bucket), and the sort's status is
// merged into the call's (and written to the host word).
__global__ void __launch_bounds__(256) k_os_finish(const SortAux *aux, uint64_t *counters, uint2 *ranges,
                                                   uint64_t n_ranges, uint64_t *status_mirror,
                                                   uint32_t *bucket_counts) {
    chain_enter();
    __shared__ uint32_t h[TB_BUCKETS];
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        if (aux->status) counters[CNT_STATUS] = aux->status;
        if (status_mirror) *status_mirror = counters[CNT_STATUS];
    }
    uint2 rg = make_uint2(0u, 0u);
    if (i < n_ranges) {
        rg = ranges[i];
        if (rg.x == RANGE_EMPTY) {
            rg = make_uint2(0u, 0u);
            ranges[i] = rg;
        }
    }
    h[threadIdx.x] = 0u;
    __syncthreads();
    if (i < n_ranges) atomicAdd(&h[len_bucket(rg)], 1u);
    __syncthreads();
    if (h[threadIdx.x]) atomicAdd(&bucket_counts[threadIdx.x], h[threadIdx.x]);
}

// Opts a kernel into dynamic shared memory where this call's `bytes` need it (beside a few
// KB of static; 48 KB in all need no opting in). The limit belongs to the function on its
// device, not to the call: it is set to the most any call may ask for, never to this
// call's size, so that no host thread lowers it between another's set and launch.
template <typename K>
static cudaError_t allow_smem(K kernel, size_t bytes, size_t most) {
    if (bytes <= 32 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

// A launch that was refused: the runtime's record of it is taken back as well.
static cudaError_t refused(cudaError_t e) {
    (void)cudaGetLastError();
    return e;
}

// The whole depth sort of at most 1024 ITEMS keys in one block: the same stable
// digit passes with the keys in registers between them and shared memory for the
// scatter, no look-back and one launch instead of five or six, which is what bounds the
// short sorts (1000 keys: 38 -> 14 us). Warp w holds the positions
// [32 ITEMS w, 32 ITEMS (w + 1)).
constexpr uint32_t DS_MAX = 8192;
template <int ITEMS>
__global__ void __launch_bounds__(1024) k_depth_small(const uint32_t *__restrict__ keys, uint32_t M,
                                                      uint32_t *__restrict__ vout, SortAux *aux,
                                                      const Batch *__restrict__ b, int passes) {
    chain_enter();
    extern __shared__ uint32_t ds_smem[];
    uint32_t *sk = ds_smem, *sv = sk + 1024 * ITEMS, *cnt = sv + 1024 * ITEMS;   // cnt[32][RS_RADIX]
    __shared__ uint32_t dstart[RS_RADIX], shs[33], s_ent[SG_MAX_VIEWS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t p0 = (uint32_t)(warp * 32 * ITEMS + lane);
    if (passes > VIEW_PASS && (int)threadIdx.x < b->n_views) s_ent[threadIdx.x] = (uint32_t)b->view[threadIdx.x].ent_off;
    uint32_t k[ITEMS], v[ITEMS], r[ITEMS], meta[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        v[i] = p0 + 32u * i;
        k[i] = v[i] < M ? keys[v[i]] : SORT_DROP_KEY;
    }
    uint32_t n = M;
    for (int p = 0; p < passes; ++p) {   // uniform
        for (int i = threadIdx.x; i < 32 * RS_RADIX; i += 1024) cnt[i] = 0u;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const bool ok = p0 + 32u * i < n && (p > 0 || k[i] != SORT_DROP_KEY);   // pass 0 drops
            uint32_t d = 0x100u;
            if (ok && p < VIEW_PASS) d = (k[i] >> (8 * p)) & 255u;
            if (ok && p == VIEW_PASS) {
                int lo = 0, hi = b->n_views - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (s_ent[mid] <= v[i]) lo = mid; else hi = mid - 1;
                }
                d = (uint32_t)lo;
            }
            const uint32_t peers = __match_any_sync(0xffffffffu, d);
            const uint32_t below = peers & lanemask_lt();
            r[i] = (ok && below == 0u) ? atomicAdd(&cnt[warp * RS_RADIX + d], (uint32_t)__popc(peers)) : 0u;
            meta[i] = (uint32_t)(__ffs(peers) - 1) | (uint32_t)__popc(below) << 5 | d << 16;
            __syncwarp();
        }
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            r[i] = __shfl_sync(0xffffffffu, r[i], (int)(meta[i] & 31u)) + ((meta[i] >> 5) & 63u);
        __syncthreads();
        uint32_t run = 0u;
        if (threadIdx.x < RS_RADIX) {
#pragma unroll 8
            for (int w = 0; w < 32; ++w) {
                const uint32_t c = cnt[w * RS_RADIX + threadIdx.x];
                cnt[w * RS_RADIX + threadIdx.x] = run;
                run += c;
            }
        }
        uint32_t kept;
        const uint32_t ds = block_exclusive<uint32_t>(run, kept, shs);
        if (threadIdx.x < RS_RADIX) dstart[threadIdx.x] = ds;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const uint32_t d = meta[i] >> 16;
            if (d < RS_RADIX) {
                const uint32_t pos = dstart[d] + cnt[warp * RS_RADIX + d] + r[i];
                sk[pos] = k[i];
                sv[pos] = v[i];
            }
        }
        __syncthreads();
        n = kept;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
            if (p0 + 32u * i < n) {
                k[i] = sk[p0 + 32u * i];
                v[i] = sv[p0 + 32u * i];
            }
    }
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
        if (p0 + 32u * i < n) vout[p0 + 32u * i] = v[i];
    if (threadIdx.x == 0) aux->kept = n;
}

template <int ITEMS>
static cudaError_t depth_small(const Batch *db, const uint32_t *keys, uint32_t M, uint32_t *vout, SortAux *aux,
                               int passes, cudaStream_t s) {
    constexpr size_t smem = (size_t)(2 * 1024 * ITEMS + 32 * RS_RADIX) * 4;
    const cudaError_t e = allow_smem(k_depth_small<ITEMS>, smem, smem);
    if (e != cudaSuccess) return e;
    (void)launch_chain_smem(k_depth_small<ITEMS>, dim3(1), dim3(1024), smem, s, keys, M, vout, aux, db, passes);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_depth_sort(const Batch *db, bool by_view, uint32_t *k0, uint32_t *v0, uint32_t *k1, uint32_t *v1,
                              const uint64_t *n_dev, uint64_t max_n, uint32_t *hist, SortAux *aux, cudaStream_t s) {
    const uint32_t nblocks = (uint32_t)div_up(max_n, RS_TILE);
    if (nblocks == 0) return cudaSuccess;
    if (max_n > SORT_MAX_KEYS) return cudaErrorInvalidValue;   // counts must fit the look-back word
    const int passes = by_view ? 5 : 4;
    if (max_n <= DS_MAX) {
        uint32_t *out = by_view ? v1 : v0;
        const uint32_t M = (uint32_t)max_n;
        return M <= 2048 ? depth_small<2>(db, k0, M, out, aux, passes, s)
                         : M <= 4096 ? depth_small<4>(db, k0, M, out, aux, passes, s)
                                     : depth_small<8>(db, k0, M, out, aux, passes, s);
    }
    // Grouped look-back where the kept keys' tiles may all be resident at once
    // (three per SM) or not far more; beyond, inclusive prefixes are found near by.
    const bool grouped = nblocks <= 8u * 3u * 152u;
    const uint64_t pass_words = depth_flag_words(max_n, 1);
    const unsigned hgrid = nblocks < 4u * 152u ? nblocks : 4u * 152u;
    cudaError_t e = launch_chain(k_os_hist, dim3(hgrid), dim3(RS_THREADS), s, (const uint32_t *)k0, n_dev, max_n, aux,
                                 hist, pass_words * passes);
    uint32_t *ki = k0, *vi = v0, *ko = k1, *vo = v1;
    for (int p = 0; p < passes && e == cudaSuccess; ++p) {
        // pass 0 leaves SORT_DROP_KEY out and later passes see only the kept keys
        const bool view = p == VIEW_PASS;
        e = launch_chain(grouped ? view ? k_os_pass<true, true> : k_os_pass<true, false>
                                 : view ? k_os_pass<false, true> : k_os_pass<false, false>,
                         dim3(nblocks), dim3(RS_THREADS), s,
                         (const uint32_t *)ki, p > 0 ? (const uint32_t *)vi : (const uint32_t *)nullptr, ko, vo,
                         p > 0 ? (const uint64_t *)&aux->kept : n_dev, max_n, p, 8 * p, 255u, p == 0,
                         hist + pass_words * p, aux, (uint2 *)nullptr, (uint64_t)0, sort_wait_polls(),
                         (const uint64_t *)nullptr, view ? db : (const Batch *)nullptr,
                         hist + pass_words * p + (uint64_t)nblocks * RS_RADIX);
        std::swap(ki, ko);
        std::swap(vi, vo);
    }
    if (e != cudaSuccess) return refused(e);
    count_launches(1 + passes);
    return cudaGetLastError();
}

cudaError_t launch_tile_radix_sort(uint32_t *k0, uint32_t *v0, uint32_t *k1, uint32_t *v1, uint64_t *counters,
                                   uint64_t max_n, int bits, uint32_t *hist, SortAux *aux, uint2 *ranges,
                                   uint64_t n_ranges, uint32_t *order_counts, uint64_t *status_mirror,
                                   cudaStream_t s) {
    const uint32_t nblocks = (uint32_t)div_up(max_n, RS_TILE);
    const int passes = nblocks ? radix_passes(bits) : 0;
    if (max_n > SORT_MAX_KEYS) return cudaErrorInvalidValue;
    const uint64_t pass_words = sort_flag_words(max_n, 1);
    uint32_t *ki = k0, *vi = v0, *ko = k1, *vo = v1;
    cudaError_t e = cudaSuccess;
    for (int p = 0; p < passes && e == cudaSuccess; ++p) {
        const int shift = 8 * p;
        const uint32_t mask = (1u << std::min(8, bits - shift)) - 1u;
        e = launch_chain(k_os_pass<false, false>, dim3(nblocks), dim3(RS_THREADS), s, (const uint32_t *)ki,
                         (const uint32_t *)vi, ko, vo, (const uint64_t *)(counters + CNT_WRITTEN), max_n, p, shift,
                         mask, false, hist + pass_words * p, aux, p == passes - 1 ? ranges : (uint2 *)nullptr,
                         n_ranges, sort_wait_polls(), (const uint64_t *)(counters + CNT_STATUS),
                         (const Batch *)nullptr, (uint32_t *)nullptr);
        std::swap(ki, ko);
        std::swap(vi, vo);
    }
    if (e != cudaSuccess) return refused(e);
    (void)launch_chain(k_os_finish, dim3((unsigned)std::max<uint64_t>(div_up(n_ranges, 256), 1)), dim3(256), s,
                       (const SortAux *)aux, counters, ranges, n_ranges, status_mirror, order_counts);
    count_launches(passes + 1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// binning by chunks
// ---------------------------------------------------------------------------
// k_bin_cut    finds every entry's first pair (decoupled look-back) and cuts each
//              view's entries into chunks of about equal pair counts
// k_bin_emit   a block per chunk: enumerates its entries' tiles, writes the
//              (tile, entry) pairs in depth order and counts them per tile in
//              shared memory: row c of the [chunks][row] matrix
// k_bin_scan   scans the matrix in (tile, chunk) order: row c becomes the first
//              output position of chunk c's pairs of every tile; every range
// k_bin_place  a warp per chunk walks its pairs in order and puts each at its
//              tile's next position
// Inside a tile the pairs follow the chunks in order and, inside a chunk, their
// depth order: the result is the stable sort by tile of the depth-ordered pairs.
// Measured (pairs and their placement, against a duplicate with its own
// look-back followed by chunks of 8192 pairs or, past 12288 tiles, three radix
// passes): 32k pairs 82 -> 31 us, 116k 91 -> 41, 3.9M 162 -> 122, 5.4M 195 -> 151,
// 11.8M over four views 450 -> 328, 252M over 16 views 10.5 -> 6.4 ms. The
// placement is bound by its warps' serial rounds (~400 cycles each, five warps
// per SM) up to some 20M pairs, beyond by its scattered 4-byte stores.
uint32_t bin_chunks(uint64_t cap, uint32_t row, int n_views) {
    // Resident placing blocks, each holding one row of cursors in shared memory:
    // five one-warp blocks per SM, four below 1M pairs (a smaller matrix). More
    // place no faster and cost the matrix's scan (4 / 5 / 6 per SM: emission, scan and
    // placement 155 / 151 / 164 us at 5.4M pairs, 125 / 122 / 129 at 3.9M).
    // Past 16M pairs the chunks' open output sectors (chunks x tiles x 32 bytes,
    // over every view) no longer fit L2: four per SM place faster (252M pairs:
    // eight 5.0 ms, four 3.8).
    const uint32_t want = cap > (1u << 20) && cap <= (16u << 20) ? 5u : 4u;
    const uint64_t fit = 152u * std::max(std::min(want, (227u * 1024u) / (row * 4u + 1024u)), 1u);
    // one chunk a view, and another for every BIN_MIN_CHUNK pairs: no more are cut
    return (uint32_t)std::min<uint64_t>(fit, (uint64_t)n_views + std::max<uint64_t>(cap / BIN_MIN_CHUNK, 1));
}

__device__ __forceinline__ uint32_t bin_view_of_chunk(const BinTab &tab, int n_views, uint32_t c) {
    int lo = 0, hi = n_views - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tab.first_chunk[mid] <= c) lo = mid; else hi = mid - 1;
    }
    return (uint32_t)lo;
}

// Blocks take BIN_ITEMS entries per thread of the depth order at a time, in order, from a
// ticket. An entry costs its pairs plus BIN_ENTRY_COST (the emitting and the
// placing warp spend time on both), so entry j's cost starts at
// X = its first pair + BIN_ENTRY_COST j. A chunk of view v starts at the first
// entry whose cost starts at or past B_v + q len_v (q = 0, 1, ..; B_v: the cost of the
// views before it): entry j marks the chunks whose threshold lies in
// (X, X + its cost] with the start j + 1. Every block recomputes the views' tables
// from preprocess's totals; block 0 publishes them.
__global__ void __launch_bounds__(BIN_CUT_THREADS) k_bin_cut(BinArgs a, uint32_t spin_limit) {
    chain_wait();
    __shared__ unsigned long long s_out0;
    __shared__ uint64_t shs64[33];
    __shared__ uint32_t shs[33];
    __shared__ uint32_t s_blk;
    __shared__ uint32_t s_base[SG_MAX_VIEWS + 1], s_len[SG_MAX_VIEWS], s_first[SG_MAX_VIEWS + 1], s_ent[SG_MAX_VIEWS];
    if (a.aux->status) {   // the depth sort gave up a bounded wait: its order may hold stale words (uniform)
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            a.counters[CNT_STATUS] = a.aux->status;
            if (a.mirror) a.mirror[0] = 0;
        }
        return;
    }
    const int tid = threadIdx.x;
    const uint64_t V = min(a.M, a.aux->kept);
    uint64_t p = tid < a.n_views ? a.tab->view_pairs[tid] : 0ull;
    uint64_t K, cost;
    (void)block_exclusive<uint64_t>(p, K, shs64);
    const bool fits = K <= a.cap;
    if (blockIdx.x == 0 && tid == 0) {
        a.counters[CNT_PAIRS] = K;
        a.counters[CNT_WRITTEN] = min(K, a.cap);
        if (a.mirror) a.mirror[0] = K;
        if (!fits) a.counters[CNT_STATUS] = (uint64_t)SG_ERR_CAPACITY;
    }
    if (!fits) return;   // uniform
    // chunks of each view: one, and a share of the others by its cost (below
    // 2^32: no more entries than pairs, BIN_ENTRY_COST + 1 times 2^30)
    if (tid < a.n_views) p += (uint64_t)BIN_ENTRY_COST * a.aux->hist[VIEW_PASS][tid];
    const uint64_t base = block_exclusive<uint64_t>(p, cost, shs64);
    const uint64_t spare = min((uint64_t)(a.max_chunks - (uint32_t)a.n_views), K / BIN_MIN_CHUNK);
    const uint32_t nc = tid < a.n_views ? 1u + (uint32_t)(spare * p / max(cost, (uint64_t)1)) : 0u;
    uint32_t total_chunks;
    const uint32_t fc = block_exclusive<uint32_t>(nc, total_chunks, shs);
    if (tid < a.n_views) {
        s_base[tid] = (uint32_t)base;
        s_len[tid] = (uint32_t)max(div_up(p, nc), (uint64_t)1);
        s_first[tid] = fc;
        s_ent[tid] = (uint32_t)a.db->view[tid].ent_off;
    }
    if (tid == 0) {
        s_base[a.n_views] = (uint32_t)cost;
        s_first[a.n_views] = total_chunks;
    }
    __syncthreads();
    if (blockIdx.x == 0) {
        BinTab &t = *a.tab;
        if (tid < a.n_views) t.first_chunk[tid] = fc;
        if (tid == 0) {
            t.n_chunks = total_chunks;
            t.first_chunk[a.n_views] = total_chunks;
            a.start[total_chunks] = (uint32_t)V;
            a.pair[total_chunks] = (uint32_t)K;
            // chunks whose threshold is 0: the first view's first chunk, and
            // every chunk of the views before the first entry
            for (int v = 0; v < a.n_views && s_base[v] == 0u; ++v) {
                const uint32_t last = s_base[v + 1] == 0u ? s_first[v + 1] : s_first[v] + 1u;
                for (uint32_t c = s_first[v]; c < last; ++c) a.start[c] = a.pair[c] = 0u;
            }
        }
    }
    for (;;) {
        __syncthreads();   // every thread is past the previous block's shared words
        if (tid == 0)
            s_blk = (uint32_t)atomicAdd(reinterpret_cast<unsigned long long *>(a.counters + CNT_DUP_BLOCK), 1ull);
        __syncthreads();
        const uint32_t blk = s_blk;
        const uint64_t e0 = (uint64_t)blk * blockDim.x * BIN_ITEMS;   // the block's first entry
        if (e0 >= V) return;   // uniform
        // BIN_ITEMS consecutive entries per thread
        const uint64_t j0 = e0 + (uint64_t)(BIN_ITEMS * tid);
        uint32_t e[BIN_ITEMS], n[BIN_ITEMS], sum = 0;
#pragma unroll
        for (int i = 0; i < BIN_ITEMS; i += 4) {   // the order's array is 256-byte aligned
            if (j0 + i + 3 < V) {
                const uint4 q = *reinterpret_cast<const uint4 *>(a.sorted_ent + j0 + i);
                e[i] = q.x; e[i + 1] = q.y; e[i + 2] = q.z; e[i + 3] = q.w;
            } else {
#pragma unroll
                for (int k = i; k < i + 4; ++k) e[k] = j0 + k < V ? a.sorted_ent[j0 + k] : 0xFFFFFFFFu;
            }
        }
#pragma unroll
        for (int i = 0; i < BIN_ITEMS; ++i) {
            n[i] = e[i] < a.M ? a.tiles_touched[e[i]] : 0u;
            sum += n[i];
        }
        uint32_t total;
        uint32_t at = block_exclusive<uint32_t>(sum, total, shs);
        if (tid < 32) {
            if (tid == 0) st_relaxed64(a.flags + blk, DL_AGG | (uint64_t)total);
            const uint64_t excl = block_lookback64(a.flags, blk, total, spin_limit, a.counters + CNT_STATUS);
            if (tid == 0) s_out0 = excl;
        }
        __syncthreads();
        at += (uint32_t)s_out0;
        int v = 0;
#pragma unroll
        for (int i = 0; i < BIN_ITEMS; ++i) {
            if (j0 + i >= V) break;
            a.poff[j0 + i] = at;
            const uint32_t end = at + n[i];   // pairs; x0, x1: cost
            const uint32_t x0 = at + BIN_ENTRY_COST * (uint32_t)(j0 + i), x1 = end + BIN_ENTRY_COST * (uint32_t)(j0 + i + 1);
            // the entry's view (entries are numbered view after view, the order has views in turn)
            if (v + 1 < a.n_views && e[i] >= s_ent[v + 1]) {
                int lo = v + 1, hi = a.n_views - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (s_ent[mid] <= e[i]) lo = mid; else hi = mid - 1;
                }
                v = lo;
            }
            const uint32_t vb = s_base[v], len = s_len[v], vc = s_first[v + 1] - s_first[v];
            // chunks q of the view with q len in (x0 - vb, x1 - vb]
            uint32_t q0 = (x0 - vb) / len + 1u, q1 = min((x1 - vb) / len, vc - 1u);
            const bool last = x1 == s_base[v + 1];
            if (last) q1 = vc - 1u;   // thresholds past the view's cost: empty chunks at its end
            for (uint32_t q = q0; q <= q1; ++q) {
                a.start[s_first[v] + q] = (uint32_t)(j0 + i + 1);
                a.pair[s_first[v] + q] = end;
            }
            if (last) {   // the first chunk of the next view with entries, and all of the empty views before it
                for (int u = v + 1; u < a.n_views && s_base[u] == x1; ++u) {
                    const uint32_t stop = s_base[u + 1] == x1 ? s_first[u + 1] : s_first[u] + 1u;
                    for (uint32_t c = s_first[u]; c < stop; ++c) {
                        a.start[c] = (uint32_t)(j0 + i + 1);
                        a.pair[c] = end;
                    }
                }
            }
            at = end;
        }
    }
}

// A block per chunk writes its entries' pairs (16-bit tile id inside the view,
// entry), entry after entry. Each warp takes 32 entries at a time, whose pairs go
// to [poff of the first, ..): its work items are (entry, tile row) in order, each
// finding the row's reached columns once; the positions inside the warp's range
// come from a warp scan of the run lengths (an entry's runs add up to its
// tiles_touched), so no two warps wait on each other.
__global__ void __launch_bounds__(256) k_bin_emit(BinArgs a) {
    chain_wait();
    extern __shared__ uint4 bin_smem[];
    uint32_t *cnt = reinterpret_cast<uint32_t *>(bin_smem);
    const unsigned FULL = 0xffffffffu;
    if (a.counters[CNT_STATUS] != (uint64_t)SG_OK) return;   // uniform
    const BinTab &tab = *a.tab;
    const uint32_t c = blockIdx.x;
    if (c >= tab.n_chunks) return;
    const ViewDesc &vw = a.db->view[bin_view_of_chunk(tab, a.n_views, c)];
    const uint32_t T = (uint32_t)vw.tiles_x * (uint32_t)vw.tiles_y, tx = (uint32_t)vw.tiles_x;
    const uint32_t q4 = (T + 3u) / 4u;
    for (uint32_t q = threadIdx.x; q < q4; q += blockDim.x) bin_smem[q] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    const uint32_t V = (uint32_t)min(a.M, a.aux->kept);
    const uint32_t e0 = min(a.start[c], V), e1 = min(a.start[c + 1], V);
    const int lane = threadIdx.x & 31;
    for (uint32_t jb = e0 + (threadIdx.x & ~31u); jb < e1; jb += blockDim.x) {
        const uint32_t j = jb + lane;
        const bool on = j < e1;
        uint32_t e = 0, rows = 0, x01 = 0, y0 = 0;
        TileReach R;
        R.x = R.y = R.B = R.det = R.At = R.ymax = R.m = R.invA = 0.f;
        R.mode = 0;
        if (on) {
            e = a.sorted_ent[j];
            if (e < a.M) {
                const uint2 rc = a.rect[e];
                // the binning reads the record's first 24 bytes: x, y, conic, bound (one sector)
                const float4 ra = a.rec[e].a;
                const float2 rb = *reinterpret_cast<const float2 *>(&a.rec[e].b);
                x01 = rc.x;
                y0 = rc.y & 0xFFFFu;
                rows = (rc.y >> 16) - y0;
                tile_reach_init(ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, R);
            }
        }
        uint32_t pos = __shfl_sync(FULL, on ? a.poff[j] : 0u, 0);   // first pair of the warp's entries
        const uint32_t inc = warp_inclusive(rows), exc = inc - rows;
        const uint32_t n_rows = __shfl_sync(FULL, inc, 31);
        for (uint32_t base = 0; base < n_rows; base += 32) {   // uniform
            // item lane -> its owner: owners that start before this window, and the heads inside it
            const bool own = rows != 0u;
            const uint32_t before = __ballot_sync(FULL, own && exc < base);
            const uint32_t heads = __reduce_or_sync(FULL, own && exc >= base && exc < base + 32u ? 1u << (exc - base) : 0u);
            const uint32_t owners = __ballot_sync(FULL, own);
            const int rank = __popc(before) + __popc(heads & (0xffffffffu >> (31 - lane))) - 1;
            const int o = (owners & (owners + 1u)) == 0u ? rank : (int)__fns(owners, 0, rank + 1);
            const int src = o & 31;
            TileReach S;
            S.x = __shfl_sync(FULL, R.x, src);
            S.y = __shfl_sync(FULL, R.y, src);
            S.B = __shfl_sync(FULL, R.B, src);
            S.det = __shfl_sync(FULL, R.det, src);
            S.At = __shfl_sync(FULL, R.At, src);
            S.ymax = __shfl_sync(FULL, R.ymax, src);
            S.m = __shfl_sync(FULL, R.m, src);
            S.invA = __shfl_sync(FULL, R.invA, src);
            S.mode = __shfl_sync(FULL, R.mode, src);
            const uint32_t sx = __shfl_sync(FULL, x01, src), se = __shfl_sync(FULL, e, src);
            const uint32_t sy = __shfl_sync(FULL, y0, src), s0 = __shfl_sync(FULL, exc, src);
            int c0 = 0, c1 = 0;
            uint32_t row = 0;
            if (base + lane < n_rows) {
                row = sy + (base + lane - s0);
                tile_reach_row(S, (int)row, (int)(sx & 0xFFFFu), (int)(sx >> 16), c0, c1);
            }
            const uint32_t run = (uint32_t)(c1 - c0);
            const uint32_t rinc = warp_inclusive(run);
            uint32_t at = pos + rinc - run;
            for (uint32_t t = row * tx + (uint32_t)c0, te = t + run; t < te; ++t, ++at) {
                if (t < T && at < a.cap) {
                    a.pkey[at] = (uint16_t)t;
                    a.pval[at] = se;
                    atomicAdd(&cnt[t], 1u);
                }
            }
            pos += __shfl_sync(FULL, rinc, 31);
        }
    }
    __syncthreads();
    uint4 *dst = reinterpret_cast<uint4 *>(a.matrix + (uint64_t)c * a.row);
    for (uint32_t q = threadIdx.x; q < q4; q += blockDim.x) dst[q] = bin_smem[q];
}

// Groups of 32 tiles of one view (lane = tile), taken in order from a ticket by
// resident blocks; the view's chunks split into BIN_SCAN_WARPS runs (one per
// warp), whose counts wait in shared memory for the second walk. The sum of
// each tile's counts and the group's total go through a decoupled look-back
// over the groups before it, which gives every tile's first position; the
// second walk replaces each count with its chunk's first position of the tile.
// Also writes every tile's range ((0, 0) when empty) and adds the tile to its
// list-length bucket. words: [0] the ticket, [1 + g] group g's look-back word.
constexpr int BIN_SCAN_WARPS = 32;
__global__ void __launch_bounds__(BIN_SCAN_WARPS * 32, 2) k_bin_scan(BinArgs a, uint32_t spin_limit) {
    chain_wait();
    __shared__ uint32_t part[BIN_SCAN_WARPS][32];
    __shared__ uint32_t s_start[32];
    __shared__ uint32_t s_grp;
    extern __shared__ uint32_t cvs[];   // [longest run][block threads]: the run's counts
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Batch &b = *a.db;
    const bool lists = a.counters[CNT_STATUS] == (uint64_t)SG_OK;   // else no pair is binned
    for (;;) {
        // every thread is past the previous group's reads of the shared words
        __syncthreads();
        if (threadIdx.x == 0) s_grp = (uint32_t)atomicAdd(reinterpret_cast<unsigned long long *>(a.words), 1ull);
        __syncthreads();
        const uint32_t grp = s_grp;
        if (grp >= a.n_groups) break;   // uniform
        int lo = 0, hi = a.n_views - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (b.view[mid].grp_off <= grp) lo = mid; else hi = mid - 1;
        }
        const ViewDesc &vw = b.view[lo];
        const uint32_t t = (grp - vw.grp_off) * 32 + lane;   // tile inside the view
        const bool tv = t < (uint32_t)vw.tiles_x * (uint32_t)vw.tiles_y;
        const uint32_t ca = lists ? a.tab->first_chunk[lo] : 0u, cb = lists ? a.tab->first_chunk[lo + 1] : 0u;
        const uint32_t per = (cb - ca + BIN_SCAN_WARPS - 1) / BIN_SCAN_WARPS;
        const uint32_t c0 = min(cb, ca + warp * per), c1 = min(cb, c0 + per);
        uint32_t *col = a.matrix + t;
        uint32_t sum = 0;
#pragma unroll 8
        for (uint32_t j = 0; j < per; ++j) {
            const uint32_t x = (tv && c0 + j < c1) ? col[(uint64_t)(c0 + j) * a.row] : 0u;
            cvs[j * (BIN_SCAN_WARPS * 32) + threadIdx.x] = x;
            sum += x;
        }
        part[warp][lane] = sum;
        __syncthreads();
        // each warp its runs' prefix over the warps before it; warp 0 the totals
        uint32_t before = 0;
        for (int w = 0; w < warp; ++w) before += part[w][lane];
        if (warp == 0) {
            uint32_t tot = 0;
#pragma unroll
            for (int w = 0; w < BIN_SCAN_WARPS; ++w) tot += part[w][lane];
            const uint32_t inc = warp_inclusive(tot);
            const uint32_t grp_total = __shfl_sync(0xffffffffu, inc, 31);
            if (lane == 0) st_relaxed64(a.words + 1 + grp, DL_AGG | (uint64_t)grp_total);
            const uint64_t excl = block_lookback64(a.words + 1, grp, grp_total, spin_limit, a.counters + CNT_STATUS);
            const uint32_t start = (uint32_t)(excl + inc - tot);
            s_start[lane] = start;
            if (tv) {
                const uint2 rg = tot ? make_uint2(start, start + tot) : make_uint2(0u, 0u);
                a.ranges[vw.tile_off + t] = rg;
                atomicAdd(&a.order_counts[len_bucket(rg)], 1u);
            }
        }
        __syncthreads();
        uint32_t run = s_start[lane] + before;
#pragma unroll 8
        for (uint32_t j = 0; j < per; ++j) {
            if (tv && c0 + j < c1) col[(uint64_t)(c0 + j) * a.row] = run;
            run += cvs[j * (BIN_SCAN_WARPS * 32) + threadIdx.x];
        }
    }
}

// One warp per chunk: its row of first positions in shared memory, then the
// chunk's pairs 32 at a time in order (a pair's tile is the tile whose range
// holds it). Lanes holding the same tile are grouped (match_any); the group's
// first lane takes as many positions from the tile's cursor as the group has
// lanes, and each lane takes the one of its rank in the group. The warp
// barriers order the cursor updates of successive rounds, whose returned
// positions are only read after all U rounds' updates are issued: the rounds'
// shared-memory latencies overlap. Positions at or past cap are not written.
__global__ void __launch_bounds__(32) k_bin_place(BinArgs a) {
    chain_enter();
    extern __shared__ uint4 bin_smem[];
    uint32_t *next = reinterpret_cast<uint32_t *>(bin_smem);
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x;
    const uint64_t status = a.counters[CNT_STATUS];
    if (blockIdx.x == 0 && lane == 0 && a.mirror) a.mirror[1] = status;
    if (status != (uint64_t)SG_OK) return;
    const BinTab &tab = *a.tab;
    const uint32_t c = blockIdx.x;
    if (c >= tab.n_chunks) return;
    const uint32_t K = (uint32_t)min(a.counters[CNT_WRITTEN], a.cap);
    const uint32_t lo = min(a.pair[c], K), hi = min(a.pair[c + 1], K);
    if (lo >= hi) return;
    const ViewDesc &vw = a.db->view[bin_view_of_chunk(tab, a.n_views, c)];
    const uint32_t T = (uint32_t)vw.tiles_x * (uint32_t)vw.tiles_y;
    // the row arrives by asynchronous 16-byte copies while the first batch loads
    const uint4 *src = reinterpret_cast<const uint4 *>(a.matrix + (uint64_t)c * a.row);
    for (uint32_t q = lane; q < (T + 3u) / 4u; q += 32) {
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(bin_smem + q);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src + q) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const uint32_t lt = (1u << lane) - 1u;
    // U rounds of 32 pairs per batch; the next batch's tiles and entries are
    // loaded while this one is placed
    constexpr int U = 8;
    uint32_t tn[U], vn[U];
    auto load = [&](uint32_t base) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t i = base + (uint32_t)(32 * u + lane);
            tn[u] = i < hi ? (uint32_t)a.pkey[i] : 0xFFFFFFFFu;
            vn[u] = i < hi ? a.pval[i] : 0xFFFFFFFFu;
        }
    };
    load(lo);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    for (uint32_t base = lo; base < hi; base += 32 * U) {
        uint32_t t[U], v[U], grp[U], at[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            t[u] = tn[u];
            v[u] = vn[u];
        }
        if (base + 32 * U < hi) load(base + 32 * U);
#pragma unroll
        for (int u = 0; u < U; ++u) grp[u] = __match_any_sync(FULL, t[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            at[u] = 0u;
            if (t[u] < T && (grp[u] & lt) == 0u) at[u] = atomicAdd(&next[t[u]], (uint32_t)__popc(grp[u]));
            __syncwarp();
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t pos = __shfl_sync(FULL, at[u], __ffs(grp[u]) - 1) + (uint32_t)__popc(grp[u] & lt);
            if (t[u] < T && pos < K) a.ovals[pos] = v[u];
        }
    }
}

// The sorted pairs' global tile ids, for layouts that keep them: a warp per tile.
__global__ void __launch_bounds__(256) k_bin_keys(const uint2 *__restrict__ ranges, uint32_t n_tiles,
                                                  uint32_t *__restrict__ okeys) {
    chain_enter();
    const uint32_t nw = gridDim.x * (blockDim.x >> 5);
    for (uint32_t t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < n_tiles; t += nw) {
        const uint2 rg = ranges[t];
        for (uint32_t i = rg.x + (threadIdx.x & 31); i < rg.y; i += 32) okeys[i] = t;
    }
}

cudaError_t launch_bin_pairs(const BinArgs &a, cudaStream_t s) {
    if (a.n_tiles == 0 || a.row == 0 || a.row > BIN_MAX_ROW || a.max_chunks <= (uint32_t)a.n_views ||
        a.max_chunks > BIN_MAX_CHUNKS || a.cap > SORT_MAX_KEYS)
        return cudaErrorInvalidValue;
    const size_t smem = (size_t)a.row * 4;
    cudaError_t e = allow_smem(k_bin_emit, smem, BIN_MAX_ROW * 4);
    if (e != cudaSuccess) return e;
    // larger blocks shorten the look-back over many entries (1M: 20 -> 14 us) but
    // cost the short ones 2 us
    const unsigned cut_threads = a.M > (1u << 19) ? BIN_CUT_THREADS : 256;
    // one block at least: it publishes the zero total of a call without entries;
    // how many of the M entries are in the order is only known on the device
    const uint64_t cut = std::min<uint64_t>(std::max<uint64_t>(div_up(a.M, cut_threads * BIN_ITEMS), 1),
                                            2 * 152 * (1024 / cut_threads));
    e = launch_chain(k_bin_cut, dim3((unsigned)cut), dim3(cut_threads), s, a, sort_wait_polls());
    if (e != cudaSuccess) return refused(e);
    (void)launch_chain_smem(k_bin_emit, dim3(a.max_chunks), dim3(256), smem, s, a);
    count_launches(2);
    return cudaGetLastError();
}

cudaError_t launch_bin_place(const BinArgs &a, cudaStream_t s) {
    const size_t smem = (size_t)a.row * 4;
    auto scan_bytes = [](uint32_t chunks) { return (size_t)div_up(chunks, BIN_SCAN_WARPS) * BIN_SCAN_WARPS * 32 * 4; };
    const size_t scan_smem = scan_bytes(a.max_chunks);
    cudaError_t e = allow_smem(k_bin_place, smem, BIN_MAX_ROW * 4);
    if (e == cudaSuccess) e = allow_smem(k_bin_scan, scan_smem, scan_bytes(BIN_MAX_CHUNKS));
    int dev = 0, sms = 0, per_sm = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    // resident blocks only: a group's look-back may wait on any earlier group
    // (two 1024-thread blocks fill an SM's threads; shared memory decides)
    per_sm = scan_smem <= 100 * 1024 ? 2 : 1;
    const unsigned grid = std::min(a.n_groups, (uint32_t)(sms * per_sm));
    e = launch_chain_smem(k_bin_scan, dim3(grid), dim3(BIN_SCAN_WARPS * 32), scan_smem, s, a, sort_wait_polls());
    if (e != cudaSuccess) return refused(e);   // an unscanned matrix holds no positions
    e = launch_chain_smem(k_bin_place, dim3(a.max_chunks), dim3(32), smem, s, a);
    if (e != cudaSuccess) return refused(e);
    count_launches(2);
    if (a.okeys) {
        (void)launch_chain(k_bin_keys, dim3(std::min(div_up(a.n_tiles, 8), (uint64_t)(sms * 8))), dim3(256), s,
                           (const uint2 *)a.ranges, a.n_tiles, a.okeys);
        count_launches(1);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// duplicateWithKeys: entries in depth order -> (tile, entry) pairs
// ---------------------------------------------------------------------------
// Adds the keys a, a + 1, .., b - 1 to a block's digit histograms: one count
// per key for the lowest digit, one per run of equal digit above it.
__device__ __forceinline__ void hist_key_run(uint32_t (*h)[RS_RADIX], int passes, uint32_t a, uint32_t b) {
    for (uint32_t t = a; t < b; ++t) atomicAdd(&h[0][t & (RS_RADIX - 1)], 1u);
    for (int p = 1; p < passes; ++p) {
        const int sh = 8 * p;
        for (uint32_t t = a; t < b;) {
            const uint64_t next = ((uint64_t)(t >> sh) + 1u) << sh;   // first key of the next digit
            const uint32_t seg = next < (uint64_t)b ? (uint32_t)next : b;
            atomicAdd(&h[p][(t >> sh) & (RS_RADIX - 1)], seg - t);
            t = seg;
        }
    }
}


// One block per 256 depth-sorted entries, in the order the blocks start
// (logical index from counters[CNT_DUP_BLOCK]). The block's pairs go, entry by
// entry and row by row, to [out0, out0 + the block's total), out0 from the
// look-back over the earlier blocks' totals: work items are (entry, tile row);
// each finds its reached columns once and writes that run (row-major inside an
// entry), so a large rectangle is spread over the whole block and the stores
// stay coalesced. Positions at or past cap are not written. The kernel also
// prepares the radix tile sort: it clears its look-back flags and adds exactly
// the keys it writes to the digit histograms of its hist_passes passes.
__global__ void __launch_bounds__(256) k_duplicate(const Batch *__restrict__ bp, uint64_t M,
                                                   const uint32_t *__restrict__ sorted_ent,
                                                   const uint32_t *__restrict__ tiles_touched,
                                                   const uint2 *__restrict__ rect, const Rec *__restrict__ rec,
                                                   const SortAux *__restrict__ depth_aux,
                                                   uint64_t *__restrict__ counters, uint64_t cap,
                                                   uint32_t *__restrict__ pkey,
                                                   uint32_t *__restrict__ pval, int hist_passes,
                                                   SortAux *__restrict__ aux, uint32_t *__restrict__ flags,
                                                   uint64_t flag_words, uint64_t *__restrict__ dflags,
                                                   uint64_t *mirror, uint32_t spin_limit) {
    chain_enter();
    __shared__ uint32_t s_rinc[256], s_e[256], s_rx[256], s_ry[256], s_base[256], s_tx[256];
    __shared__ TileReach s_R[256];
    __shared__ uint32_t shs[33];
    __shared__ uint32_t h[4][RS_RADIX];
    __shared__ unsigned long long s_blk, s_out0;
    // the tile sort's look-back flags start at zero (its passes run after this kernel)
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < flag_words; i += (uint64_t)gridDim.x * 256)
        flags[i] = 0u;
    for (int i = threadIdx.x; i < 4 * RS_RADIX; i += 256) h[i / RS_RADIX][i % RS_RADIX] = 0u;
    // a sort gave up a bounded wait: its order may hold stale words (uniform)
    if (depth_aux->status) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            counters[CNT_STATUS] = depth_aux->status;
            if (mirror) mirror[0] = 0;
        }
        return;
    }
    if (threadIdx.x == 0)
        s_blk = atomicAdd(reinterpret_cast<unsigned long long *>(counters + CNT_DUP_BLOCK), 1ull);
    __syncthreads();
    const uint64_t blk = s_blk;
    const uint64_t j0 = blk * 256;
    const uint64_t j = j0 + threadIdx.x;
    const uint64_t V = min(M, depth_aux->kept);   // entries in depth order with at least one pair
    if (j0 >= V) {   // no entry: only the first block, when there is none at all, reports the zero total
        if (V == 0 && blk == 0 && threadIdx.x == 0 && mirror) mirror[0] = 0;
        return;
    }
    uint32_t e = 0, tt = 0, rows = 0, rx = 0, ry = 0, tbase = 0, tx = 1;
    if (j < V) {
        e = sorted_ent[j];
        tt = e < M ? tiles_touched[e] : 0u;   // an id left by a sort that gave up a wait reaches no tile
    }
    // the block's pair count goes out first; the row bookkeeping below hides the
    // latency of the predecessors' counts
    uint32_t total;
    block_exclusive<uint32_t>(tt, total, shs);
    if (threadIdx.x == 0) st_relaxed64(dflags + blk, DL_AGG | ((uint64_t)total & DL_VAL));
    if (j < V) {
        if (tt) {
            const Batch &b = *bp;
            const ViewDesc &vw = b.view[find_entry_view(b, e)];
            const uint2 rc = rect[e];
            rx = rc.x;
            ry = rc.y;
            rows = (ry >> 16) - (ry & 0xFFFFu);
            tbase = vw.tile_off;
            tx = (uint32_t)vw.tiles_x;
            // the binning reads the record's first 24 bytes: x, y, conic, bound (one sector)
            const float4 ra = rec[e].a;
            const float2 rb = *reinterpret_cast<const float2 *>(&rec[e].b);
            tile_reach_init(ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, s_R[threadIdx.x]);
        }
    }
    uint32_t total_rows;
    const uint32_t rexcl = block_exclusive<uint32_t>(rows, total_rows, shs);
    s_rinc[threadIdx.x] = rexcl + rows;
    s_e[threadIdx.x] = e;
    s_rx[threadIdx.x] = rx;
    s_ry[threadIdx.x] = ry;
    s_base[threadIdx.x] = tbase;
    s_tx[threadIdx.x] = tx;
    if (threadIdx.x < 32) {
        const uint64_t excl = block_lookback64(dflags, blk, total, spin_limit, counters + CNT_STATUS);
        if (threadIdx.x == 0) {
            s_out0 = excl;
            if ((V - 1) / 256 == blk) {   // the last block: the totals
                const uint64_t all = excl + total;
                counters[CNT_PAIRS] = all;
                counters[CNT_WRITTEN] = min(all, cap);
                if (mirror) mirror[0] = all;
                if (all > cap)
                    atomicCAS(reinterpret_cast<unsigned long long *>(counters + CNT_STATUS), 0ull,
                              (unsigned long long)SG_ERR_CAPACITY);
            }
        }
    }
    __syncthreads();
    if (total == 0u) return;
    const uint64_t out0 = s_out0;
    // pairs the block may write: positions below cap only
    const uint32_t lim = out0 >= cap ? 0u : (uint32_t)min((uint64_t)total, cap - out0);
    if (lim == 0u) return;
    uint32_t done = 0u;
    for (uint32_t base = 0; base < total_rows; base += 256) {
        const uint32_t item = base + threadIdx.x;
        int o = 0, row = 0, c0 = 0, c1 = 0;
        if (item < total_rows) {
            // first owner o with s_rinc[o] > item
            int lo = 0, hi = 255;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (s_rinc[mid] > item) hi = mid; else lo = mid + 1;
            }
            o = lo;
            const uint32_t r0 = o ? s_rinc[o - 1] : 0u;
            row = (int)(s_ry[o] & 0xFFFFu) + (int)(item - r0);
            tile_reach_row(s_R[o], row, (int)(s_rx[o] & 0xFFFFu), (int)(s_rx[o] >> 16), c0, c1);
        }
        uint32_t chunk;
        const uint32_t at = done + block_exclusive<uint32_t>((uint32_t)(c1 - c0), chunk, shs);
        const uint32_t key0 = s_base[o] + (uint32_t)row * s_tx[o];
        for (int c = c0; c < c1; ++c) {
            const uint32_t q = at + (uint32_t)(c - c0);
            if (q < lim) {   // rows sum to tiles_touched by construction; never write past the block or cap
                pkey[out0 + q] = key0 + (uint32_t)c;
                pval[out0 + q] = s_e[o];
            }
        }
        if (at < lim)   // the keys written above, no more
            hist_key_run(h, hist_passes, key0 + (uint32_t)c0,
                         key0 + (uint32_t)c0 + min((uint32_t)(c1 - c0), lim - at));
        done += chunk;
    }
    // Rows add up to tiles_touched by construction. Should they ever fall short,
    // the rest of the block's range still gets valid tile ids and entries.
    for (uint32_t q = done + threadIdx.x; q < lim; q += 256) {
        pkey[out0 + q] = s_base[0];
        pval[out0 + q] = s_e[0];
        hist_key_run(h, hist_passes, s_base[0], s_base[0] + 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < hist_passes * RS_RADIX; i += 256) {
        const uint32_t c = h[i / RS_RADIX][i % RS_RADIX];
        if (c) atomicAdd(&aux->hist[i / RS_RADIX][i % RS_RADIX], c);
    }
}

cudaError_t launch_duplicate(const Batch *db, uint64_t M, const uint32_t *sorted_ent, const SortAux *depth_aux,
                             const uint32_t *tiles_touched, const uint2 *rect, const Rec *rec, uint64_t *counters,
                             uint64_t cap, uint32_t *pkey, uint32_t *pval, uint64_t *dup_flags, uint64_t *mirror,
                             cudaStream_t s, int hist_passes, SortAux *sort_aux, uint32_t *flags,
                             uint64_t flag_words) {
    if (hist_passes < 1 || hist_passes > 4) return cudaErrorInvalidValue;
    // one block at least: it reports the zero total of a call without entries
    const uint64_t grid = std::max<uint64_t>(div_up(M, 256), 1);
    // launched in plain stream order: started early, its blocks are placed where the last
    // depth pass leaves room (3840x2160 and three smaller views: 2965 -> 2882 us a forward)
    k_duplicate<<<(unsigned)grid, 256, 0, s>>>(db, M, sorted_ent, tiles_touched, rect, rec, depth_aux, counters, cap,
                                               pkey, pval, hist_passes, sort_aux, flags, flag_words, dup_flags,
                                               mirror, sort_wait_polls());
    count_launches(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// work order of the persistent blend: tiles by descending list length
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_tile_bucket_scatter(const uint2 *__restrict__ ranges, uint32_t n_tiles,
                                                             const uint32_t *__restrict__ counts,
                                                             uint32_t *__restrict__ cursor,
                                                             uint32_t *__restrict__ order) {
    chain_enter();
    __shared__ uint32_t base[TB_BUCKETS];
    __shared__ uint32_t shs[33];
    // longest lists first: exclusive scan over the buckets in reverse
    const uint32_t c = counts[TB_BUCKETS - 1 - threadIdx.x];
    uint32_t tot;
    base[TB_BUCKETS - 1 - threadIdx.x] = block_exclusive<uint32_t>(c, tot, shs);
    __syncthreads();
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n_tiles; t += gridDim.x * blockDim.x) {
        const uint32_t b = len_bucket(ranges[t]);
        order[base[b] + atomicAdd(&cursor[b], 1u)] = t;
    }
}

cudaError_t launch_tile_order(const uint2 *ranges, uint32_t n_tiles, uint32_t *order, uint32_t *scratch,
                              cudaStream_t s) {
    static_assert(TILE_ORDER_WORDS == 2 * TB_BUCKETS, "tile order scratch");
    if (n_tiles == 0) return cudaSuccess;
    uint32_t *counts = scratch, *cursor = scratch + TB_BUCKETS;
    const uint64_t want = div_up(n_tiles, 256);
    const unsigned grid = (unsigned)(want < 608u ? want : 608u);
    (void)launch_chain(k_tile_bucket_scatter, dim3(grid), dim3(256), s, ranges, n_tiles, counts, cursor, order);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace sgk
