// ADMM steps of the memory-constrained optimisation (Alg. 1, Sec. 3.3.2).
//
//  * penalty gradient of the gradient step: grad += delta (x - x~ + lambda)
//  * proximal step (Eq. 7-9): z = x + lambda; keep the kappa entries of z with
//    the largest score, x~ = z there and 0 elsewhere. Scores: the importance
//    I_i (App. A.2) or |z_i| for opacities, the dynamic range
//    D_i = |a_i| |1 - exp(-2 z_i)| (Eq. 10) for lobe sharpness.
//  * dual update: lambda += x - x~
//
// Selection is a radix select over order-preserving keys of the scores (the
// kappa largest, equal scores by lower index): three passes over the key digits,
// most significant first (11, 11 and 10 bits), each histogramming the keys that
// match the threshold digits found so far and picking the next digit where the
// running count reaches kappa (the first histogram is taken while the keys are
// written); then one pass that keeps every key below the threshold and the
// first of its ties in index order (a decoupled look-back over the blocks' tie
// counts), and writes x~ and the new lambda. The steps are bound by their few
// short launches: 11-bit digits need one less than bytes, the final pass's
// eight entries per thread move as 16-byte vectors, and it looks back only where
// some but not all ties are kept (opacity and sharpness step of 1M Gaussians with
// 1.65M lobes: 132 -> 61 us of kernels).
#include "sg_internal.cuh"

#include <algorithm>

namespace sgk {

// Order-preserving key for a DESCENDING order through ascending keys (smaller
// key = larger score). NaN scores come last.
__device__ __forceinline__ uint32_t desc_key(float f) {
    if (isnan(f)) return 0xFFFFFFFFu;
    const uint32_t u = __float_as_uint(f);
    const uint32_t asc = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ~asc;
}

// State of one selection (in the workspace).
struct SelState {
    int64_t kappa;
    int32_t mode;            // 0: select, 1: keep none (kappa <= 0), 2: keep all (kappa >= n)
    int32_t pad;
    uint64_t status;         // SG_ERR_TIMEOUT when the final pass gave up a bounded wait
    uint64_t block_ctr;      // logical blocks of the final pass
};

constexpr int SEL_ITEMS = 8;                     // consecutive entries per thread in the final pass
constexpr int SEL_TILE = 256 * SEL_ITEMS;
constexpr int SEL_BINS = 2048, SEL_PASSES = 3;
constexpr int SEL_PER = SEL_BINS / 256;          // bins per thread
__host__ __device__ constexpr int sel_shift(int p) { return p == 0 ? 21 : p == 1 ? 10 : 0; }
__host__ __device__ constexpr uint32_t sel_mask(int p) { return p == 2 ? 1023u : 2047u; }

// Adds a block's digit counts to the pass's histogram.
__device__ __forceinline__ void sel_flush(uint32_t *h, uint32_t *__restrict__ hist) {
    __syncthreads();
    for (int i = threadIdx.x; i < SEL_BINS; i += 256)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}

__device__ __forceinline__ void sel_clear(uint32_t *h) {
    for (int i = threadIdx.x; i < SEL_BINS; i += 256) h[i] = 0u;
    __syncthreads();
}

// The selection's kappa and mode, by one thread of the score kernel's grid. (Its other
// words, the histograms and the look-back words are zero on entry.)
__device__ __forceinline__ void sel_setup(int64_t n, int64_t kappa, SelState *st) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->kappa = kappa;
        st->mode = kappa <= 0 ? 1 : (kappa >= n ? 2 : 0);
    }
}

__global__ void __launch_bounds__(256) k_score_opacity(int64_t n, const float *__restrict__ x,
                                                       const float *__restrict__ lam,
                                                       const float *__restrict__ score,
                                                       uint32_t *__restrict__ keys, int64_t kappa, SelState *st,
                                                       uint32_t *__restrict__ hist) {
    chain_enter();
    __shared__ uint32_t h[SEL_BINS];
    sel_setup(n, kappa, st);
    sel_clear(h);
    const int64_t nth = (int64_t)gridDim.x * 256;
#pragma unroll 4
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += nth) {
        const uint32_t k = desc_key(score ? score[i] : fabsf(__fadd_rn(x[i], lam[i])));
        keys[i] = k;
        atomicAdd(&h[k >> sel_shift(0)], 1u);
    }
    sel_flush(h, hist);
}

__global__ void __launch_bounds__(256) k_score_sharpness(int64_t L, const float *__restrict__ s,
                                                         const float *__restrict__ lam,
                                                         const float *__restrict__ amp,
                                                         uint32_t *__restrict__ keys, int64_t kappa, SelState *st,
                                                         uint32_t *__restrict__ hist) {
    chain_enter();
    __shared__ uint32_t h[SEL_BINS];
    sel_setup(L, kappa, st);
    sel_clear(h);
    const int64_t nth = (int64_t)gridDim.x * 256;
#pragma unroll 2
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < L; i += nth) {
        const float z = __fadd_rn(s[i], lam[i]);
        const float a0 = amp[i], a1 = amp[L + i], a2 = amp[2 * L + i];
        const float na = sqrtf(a0 * a0 + a1 * a1 + a2 * a2);
        const float D = na * fabsf(1.0f - expf(-2.0f * z));
        const uint32_t k = desc_key(D);
        keys[i] = k;
        atomicAdd(&h[k >> sel_shift(0)], 1u);
    }
    sel_flush(h, hist);
}

// The threshold digits of the first `passes` passes, from their histograms
// (every block of the later kernels redoes these picks; 256 threads, SEL_PER
// bins each). Pass q's digit is the one where the running count of the keys
// matching the earlier digits reaches the entries still to keep.
struct SelPrefix {
    uint32_t prefix, mask;
    int64_t remaining;
    int64_t matching;   // keys that match the digits found
    int32_t mode;
};

__device__ __forceinline__ SelPrefix sel_resolve(const SelState *st, const uint32_t *__restrict__ hist,
                                                 int passes) {
    __shared__ uint64_t shs[33];
    __shared__ uint32_t s_digit;
    __shared__ uint64_t s_below, s_match;
    SelPrefix r{0u, 0u, st->kappa, 0, st->mode};
    for (int q = 0; q < passes && r.mode == 0; ++q) {   // uniform
        uint32_t c[SEL_PER];
        const uint4 *h4 = reinterpret_cast<const uint4 *>(hist + q * SEL_BINS) + threadIdx.x * (SEL_PER / 4);
#pragma unroll
        for (int i = 0; i < SEL_PER / 4; ++i) {
            const uint4 v = h4[i];
            c[4 * i] = v.x; c[4 * i + 1] = v.y; c[4 * i + 2] = v.z; c[4 * i + 3] = v.w;
        }
        uint64_t sum = 0;
#pragma unroll
        for (int i = 0; i < SEL_PER; ++i) sum += c[i];
        uint64_t tot;
        uint64_t excl = block_exclusive<uint64_t>(sum, tot, shs);
        if ((int64_t)excl < r.remaining && r.remaining <= (int64_t)(excl + sum)) {   // one thread
#pragma unroll
            for (int i = 0; i < SEL_PER; ++i) {
                if ((int64_t)excl < r.remaining && r.remaining <= (int64_t)(excl + c[i])) {
                    s_digit = threadIdx.x * SEL_PER + i;
                    s_below = excl;
                    s_match = c[i];
                }
                excl += c[i];
            }
        }
        __syncthreads();
        if ((int64_t)tot < r.remaining) {   // fewer keys than asked (not expected): keep them all
            r.mode = 2;
        } else {
            r.prefix |= s_digit << sel_shift(q);
            r.mask |= sel_mask(q) << sel_shift(q);
            r.remaining -= (int64_t)s_below;
            r.matching = (int64_t)s_match;
        }
        __syncthreads();   // s_digit / s_below are rewritten by the next pass
    }
    return r;
}

// Histogram of pass p's digit over the keys that match the digits of passes
// 0 .. p - 1.
__global__ void __launch_bounds__(256) k_sel_hist(int64_t n, const uint32_t *__restrict__ keys,
                                                  const SelState *st, uint32_t *__restrict__ hist, int p) {
    chain_enter();
    __shared__ uint32_t h[SEL_BINS];
    const SelPrefix r = sel_resolve(st, hist, p);
    if (r.mode != 0) return;   // uniform
    sel_clear(h);
    const int shift = sel_shift(p);
    const uint32_t pre = r.prefix, msk = r.mask, dm = sel_mask(p);
    const int64_t n4 = n / 4;
    const uint4 *k4 = reinterpret_cast<const uint4 *>(keys);
    const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x, nth = (int64_t)gridDim.x * 256;
    for (int64_t j = t; j < n4; j += nth) {
        const uint4 k = k4[j];
        if ((k.x & msk) == pre) atomicAdd(&h[(k.x >> shift) & dm], 1u);
        if ((k.y & msk) == pre) atomicAdd(&h[(k.y >> shift) & dm], 1u);
        if ((k.z & msk) == pre) atomicAdd(&h[(k.z >> shift) & dm], 1u);
        if ((k.w & msk) == pre) atomicAdd(&h[(k.w >> shift) & dm], 1u);
    }
    for (int64_t j = 4 * n4 + t; j < n; j += nth) {
        const uint32_t k = keys[j];
        if ((k & msk) == pre) atomicAdd(&h[(k >> shift) & dm], 1u);
    }
    sel_flush(h, hist + p * SEL_BINS);
}

__global__ void __launch_bounds__(256) k_penalty_grad(int64_t n, const float *__restrict__ x,
                                                      const float *__restrict__ x_tilde,
                                                      const float *__restrict__ lam, float delta,
                                                      float *__restrict__ grad) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float y = __fadd_rn(__fsub_rn(x[i], x_tilde[i]), lam[i]);
    grad[i] = __fadd_rn(grad[i], __fmul_rn(delta, y));
}

// Final pass: thread t of logical block b owns entries b * SEL_TILE + t * SEL_ITEMS
// + 0 .. SEL_ITEMS - 1 (consecutive, so block and thread prefixes of the tie
// counts follow the index order). Keeps the keys below the threshold and the
// first `remaining` keys equal to it; writes x~ = z (kept) or 0 and
// lambda += x - x~. vec: x, lam and x_tilde are 16-byte aligned (a thread's
// eight entries then move as two vectors each).
__global__ void __launch_bounds__(256) k_sel_final(int64_t n, const uint32_t *__restrict__ keys,
                                                   const float *__restrict__ x, float *__restrict__ lam,
                                                   float *__restrict__ x_tilde, SelState *st,
                                                   const uint32_t *__restrict__ hist,
                                                   uint64_t *__restrict__ flags, uint32_t spin_limit, bool vec) {
    chain_enter();
    __shared__ uint32_t shs[33];
    __shared__ uint64_t s_blk, s_excl;
    if (threadIdx.x == 0) s_blk = atomicAdd(reinterpret_cast<unsigned long long *>(&st->block_ctr), 1ull);
    __syncthreads();
    const uint64_t blk = s_blk;
    const SelPrefix r = sel_resolve(st, hist, SEL_PASSES);
    const int32_t mode = r.mode;
    const uint32_t T = r.prefix;          // the threshold key (every digit)
    const int64_t rem = r.remaining;      // its ties to keep
    // all of them (the scores are mostly distinct): no rank among the ties is needed
    const bool ranked = mode == 0 && rem < r.matching;   // uniform over the grid
    const int64_t i0 = (int64_t)blk * SEL_TILE + (int64_t)threadIdx.x * SEL_ITEMS;
    const bool whole = vec && i0 + SEL_ITEMS <= n;
    uint32_t k[SEL_ITEMS];
    float xv[SEL_ITEMS], lv[SEL_ITEMS];
    if (whole) {
        const uint4 *k4 = reinterpret_cast<const uint4 *>(keys + i0);
        const float4 *x4 = reinterpret_cast<const float4 *>(x + i0), *l4 = reinterpret_cast<const float4 *>(lam + i0);
#pragma unroll
        for (int q = 0; q < SEL_ITEMS / 4; ++q) {
            const uint4 kq = k4[q];
            const float4 xq = x4[q], lq = l4[q];
            k[4 * q] = kq.x; k[4 * q + 1] = kq.y; k[4 * q + 2] = kq.z; k[4 * q + 3] = kq.w;
            xv[4 * q] = xq.x; xv[4 * q + 1] = xq.y; xv[4 * q + 2] = xq.z; xv[4 * q + 3] = xq.w;
            lv[4 * q] = lq.x; lv[4 * q + 1] = lq.y; lv[4 * q + 2] = lq.z; lv[4 * q + 3] = lq.w;
        }
    } else {
#pragma unroll
        for (int it = 0; it < SEL_ITEMS; ++it) {
            const bool on = i0 + it < n;
            k[it] = on ? keys[i0 + it] : 0xFFFFFFFFu;
            xv[it] = on ? x[i0 + it] : 0.f;
            lv[it] = on ? lam[i0 + it] : 0.f;
        }
    }
    uint32_t ties = 0u;
#pragma unroll
    for (int it = 0; it < SEL_ITEMS; ++it) ties += (mode == 0 && i0 + it < n && k[it] == T) ? 1u : 0u;
    uint32_t btot, rank = 0u;
    if (ranked) {
        rank = block_exclusive<uint32_t>(ties, btot, shs);   // ties in earlier threads of the block, then blocks
        if (threadIdx.x == 0) st_relaxed64(flags + blk, DL_AGG | ((uint64_t)btot & DL_VAL));
        if (threadIdx.x < 32) {
            const uint64_t excl = block_lookback64(flags, blk, btot, spin_limit, &st->status);
            if (threadIdx.x == 0) s_excl = excl;
        }
        __syncthreads();
    }
    const uint64_t before = ranked ? s_excl : 0ull;
#pragma unroll
    for (int it = 0; it < SEL_ITEMS; ++it) {
        bool keep = mode == 2;
        if (mode == 0) {
            if (k[it] < T) {
                keep = true;
            } else if (k[it] == T && i0 + it < n) {
                keep = !ranked || (int64_t)(before + rank) < rem;
                ++rank;
            }
        }
        const float z = __fadd_rn(xv[it], lv[it]);
        const float xt = keep ? z : 0.0f;
        lv[it] = __fadd_rn(lv[it], __fsub_rn(xv[it], xt));
        xv[it] = xt;
    }
    if (whole) {
        float4 *t4 = reinterpret_cast<float4 *>(x_tilde + i0), *l4 = reinterpret_cast<float4 *>(lam + i0);
#pragma unroll
        for (int q = 0; q < SEL_ITEMS / 4; ++q) {
            t4[q] = make_float4(xv[4 * q], xv[4 * q + 1], xv[4 * q + 2], xv[4 * q + 3]);
            l4[q] = make_float4(lv[4 * q], lv[4 * q + 1], lv[4 * q + 2], lv[4 * q + 3]);
        }
    } else {
#pragma unroll
        for (int it = 0; it < SEL_ITEMS; ++it) {
            if (i0 + it >= n) break;
            x_tilde[i0 + it] = xv[it];
            lam[i0 + it] = lv[it];
        }
    }
}

// Workspace: the selection state, the passes' histograms and the final pass's
// look-back words (zeroed together), and the keys.
struct AdmmLayout {
    size_t state, hist, flags, zeroed, keys, total;
    uint64_t nflags;
};

static size_t al256(size_t x) { return (x + 255) / 256 * 256; }

static AdmmLayout admm_layout(int64_t n) {
    AdmmLayout L{};
    size_t o = 0;
    auto take = [&](size_t b) { size_t r = o; o += al256(b); return r; };
    L.state = take(sizeof(SelState));
    L.hist = take((size_t)SEL_PASSES * SEL_BINS * 4);
    L.nflags = std::max<uint64_t>(div_up((uint64_t)n, SEL_TILE), 1);
    L.flags = take(8 * L.nflags);
    L.zeroed = o;
    L.keys = take(4 * (size_t)n);
    L.total = o;
    return L;
}

size_t admm_workspace_bytes(int64_t n) { return admm_layout(n < 0 ? 0 : n).total; }

// kind 0: opacity (score = importance or |z|), kind 1: sharpness (score = D)
cudaError_t launch_admm_step(int kind, int64_t n, const float *x, const float *score, const float *amp,
                             int64_t kappa, float *lam, float *x_tilde, void *ws, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    if ((uint64_t)n > (uint64_t)UINT32_MAX) return cudaErrorInvalidValue;   // 32-bit histogram counts
    const AdmmLayout L = admm_layout(n);
    char *w = static_cast<char *>(ws);
    SelState *st = reinterpret_cast<SelState *>(w + L.state);
    uint32_t *keys = reinterpret_cast<uint32_t *>(w + L.keys);
    uint32_t *hist = reinterpret_cast<uint32_t *>(w + L.hist);
    uint64_t *flags = reinterpret_cast<uint64_t *>(w + L.flags);
    const cudaError_t e = cudaMemsetAsync(w, 0, L.zeroed, s);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)std::min<uint64_t>(div_up((uint64_t)n, 256 * 8), 4 * 152));
    if (kind == 0)
        (void)launch_chain(k_score_opacity, grid, dim3(256), s, n, x, lam, score, keys, kappa, st, hist);
    else
        (void)launch_chain(k_score_sharpness, grid, dim3(256), s, n, x, lam, amp, keys, kappa, st, hist);
    const unsigned hgrid = (unsigned)std::min<uint64_t>(div_up((uint64_t)n, 256 * 16), 4 * 152);
    for (int p = 1; p < SEL_PASSES; ++p)
        (void)launch_chain(k_sel_hist, dim3(hgrid), dim3(256), s, n, (const uint32_t *)keys, (const SelState *)st,
                           hist, p);
    const bool vec = ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(lam) |
                       reinterpret_cast<uintptr_t>(x_tilde)) & 15u) == 0u;
    (void)launch_chain(k_sel_final, dim3((unsigned)L.nflags), dim3(256), s, n, (const uint32_t *)keys, x, lam,
                       x_tilde, st, (const uint32_t *)hist, flags, sort_wait_polls(), vec);
    count_launches(2 + SEL_PASSES - 1);
    return cudaGetLastError();
}

cudaError_t launch_penalty_grad(int64_t n, const float *x, const float *x_tilde, const float *lam, float delta,
                                float *grad, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_penalty_grad<<<(unsigned)div_up((uint64_t)n, 256), 256, 0, s>>>(n, x, x_tilde, lam, delta, grad);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace sgk
