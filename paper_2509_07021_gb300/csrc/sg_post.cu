// Post-processing after the constrained optimisation (Sec. 3.3.3):
//   1. Gaussians whose opacity m_g o falls below tau_o are removed;
//   2. lobes of the remaining Gaussians whose sharpness falls below tau_s are
//      removed, and each removed lobe's mean over the sphere,
//      m_l a (1 - e^{-2s}) / (2s) (Eq. 12; limit m_l a at s = 0), is added
//      to the diffuse colour c0 (Eq. 13);
//   3. the kept Gaussians and lobes are compacted in their original order.
// The keep decisions are binary32 comparisons (m_g o is one rounded product).
#include "sg_internal.cuh"

namespace sgk {

constexpr uint32_t POST_DROPPED = 0xFFFFFFFFu;   // gidx of a removed Gaussian

__device__ __forceinline__ bool keep_gauss(const sg_scene &sc, int64_t g, float tau_o) {
    const float op = __fmul_rn(sc.gmask[g], static_cast<const float *>(sc.opac)[g]);
    return op >= tau_o;
}

__device__ __forceinline__ void lobe_range(const sg_scene &sc, int64_t g, int &lo, int &hi) {
    hi = min(sc.lobe_off[g + 1], (int)sc.n_lobes);
    lo = max(0, min(sc.lobe_off[g], hi));
}

// Keep flag (bit 0) and kept lobes of every Gaussian.
__global__ void __launch_bounds__(256) k_post_count(const sg_scene sc, float tau_o, float tau_s,
                                                    uint32_t *__restrict__ keep) {
    const int64_t g = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (g >= sc.n) return;
    uint32_t c = 0;
    if (keep_gauss(sc, g, tau_o)) {
        int lo, hi;
        lobe_range(sc, g, lo, hi);
        const float *sh = static_cast<const float *>(sc.sharp);
        for (int k = lo; k < hi; ++k) c += sh[k] >= tau_s ? 1u : 0u;
        c = c << 1 | 1u;
    }
    keep[g] = c;
}

// Every kept Gaussian's output position (over its keep word) and first output
// lobe: each block of POST_BLOCK Gaussians publishes its kept Gaussians and
// lobes in one 64-bit word (31 bits each; both totals are below 2^31) and finds
// its offsets by a decoupled look-back: one launch instead of a three-kernel
// scan for each. The block holding the last Gaussian writes the totals.
constexpr int POST_ITEMS = 8, POST_THREADS = 1024, POST_BLOCK = POST_THREADS * POST_ITEMS;
struct PostState {
    uint64_t totals[2];   // Gaussians, lobes
    uint64_t status;      // SG_ERR_TIMEOUT when a block gave up its bounded wait
    uint64_t block_ctr;
};

__global__ void __launch_bounds__(POST_THREADS) k_post_scan(int64_t n, uint32_t *__restrict__ gidx, uint32_t *__restrict__ loff,
                                                   PostState *__restrict__ st, uint64_t *__restrict__ flags,
                                                   uint32_t spin_limit) {
    __shared__ uint64_t shs[33];
    __shared__ uint64_t s_blk, s_excl;
    if (threadIdx.x == 0) s_blk = atomicAdd(reinterpret_cast<unsigned long long *>(&st->block_ctr), 1ull);
    __syncthreads();
    const uint64_t blk = s_blk;
    const int64_t g0 = (int64_t)blk * POST_BLOCK + (int64_t)threadIdx.x * POST_ITEMS;   // consecutive
    uint32_t w[POST_ITEMS];
    if (g0 + POST_ITEMS <= n) {
        const uint4 a = *reinterpret_cast<const uint4 *>(gidx + g0), b = *reinterpret_cast<const uint4 *>(gidx + g0 + 4);
        w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
    } else {
#pragma unroll
        for (int i = 0; i < POST_ITEMS; ++i) w[i] = g0 + i < n ? gidx[g0 + i] : 0u;
    }
    uint64_t sum = 0;
#pragma unroll
    for (int i = 0; i < POST_ITEMS; ++i) sum += (uint64_t)(w[i] & 1u) | (uint64_t)(w[i] >> 1) << 31;
    uint64_t tot;
    uint64_t at = block_exclusive<uint64_t>(sum, tot, shs);
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0) st_relaxed64(flags + blk, DL_AGG | tot);
        const uint64_t before = block_lookback64(flags, blk, tot, spin_limit, &st->status);
        if (threadIdx.x == 0) {
            s_excl = before;
            if ((int64_t)(blk + 1) * POST_BLOCK >= n) {
                st->totals[0] = (before + tot) & 0x7FFFFFFFull;
                st->totals[1] = (before + tot) >> 31;
            }
        }
    }
    __syncthreads();
    at += s_excl;
    uint32_t gi[POST_ITEMS], lo[POST_ITEMS];
#pragma unroll
    for (int i = 0; i < POST_ITEMS; ++i) {
        gi[i] = (w[i] & 1u) ? (uint32_t)(at & 0x7FFFFFFFull) : POST_DROPPED;
        lo[i] = (uint32_t)(at >> 31);
        at += (uint64_t)(w[i] & 1u) | (uint64_t)(w[i] >> 1) << 31;
    }
    if (g0 + POST_ITEMS <= n) {
#pragma unroll
        for (int i = 0; i < POST_ITEMS; i += 4) {
            *reinterpret_cast<uint4 *>(gidx + g0 + i) = make_uint4(gi[i], gi[i + 1], gi[i + 2], gi[i + 3]);
            *reinterpret_cast<uint4 *>(loff + g0 + i) = make_uint4(lo[i], lo[i + 1], lo[i + 2], lo[i + 3]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < POST_ITEMS; ++i) {
            if (g0 + i >= n) break;
            gidx[g0 + i] = gi[i];
            loff[g0 + i] = lo[i];
        }
    }
}

// mean of a e^{s (mu.v - 1)} over the sphere divided by a: (1 - e^{-2s}) / (2s)
__device__ __forceinline__ float lobe_mean_factor(float s) {
    if (fabsf(s) < 1e-6f) return 1.0f - s;   // series 1 - s + O(s^2)
    return -expm1f(-2.0f * s) / (2.0f * s);
}

struct PostOut {
    float *means, *scales, *quats, *opac, *gmask, *c0, *axis, *sharp, *amp, *lmask;
    int32_t *lobe_off;
    int64_t n_out, l_out;
};

// A block of 256 Gaussians: their fields one thread each; their lobes, a
// contiguous range, one thread each in tiles of POST_TILE (coalesced loads and
// stores instead of one Gaussian's lobes one after the other): kept lobes take the
// next output positions (block scan), removed ones leave amplitude x mean in
// shared memory, which the owner then adds to its diffuse colour in lobe order
// (plan and apply at 1M Gaussians, 1.65M lobes: 87 -> 73 us of kernels in three
// launches instead of eight).
constexpr int POST_TILE = 512;
__global__ void __launch_bounds__(256) k_post_apply(const sg_scene sc, float tau_s,
                                                    const uint32_t *__restrict__ gidx,
                                                    const uint32_t *__restrict__ loff, PostOut o) {
    __shared__ uint16_t s_owner[POST_TILE];
    __shared__ float s_f[POST_TILE], s_a[3][POST_TILE];
    __shared__ uint32_t shs[33];
    __shared__ bool s_kept[256];
    const int64_t g0 = (int64_t)blockIdx.x * 256, g = g0 + threadIdx.x;
    if (g == 0) o.lobe_off[o.n_out] = (int32_t)o.l_out;
    const int64_t n = sc.n, L = sc.n_lobes, N2 = o.n_out, L2 = o.l_out;
    if (n == 0) return;
    const uint32_t i32 = g < n ? gidx[g] : POST_DROPPED;
    const bool kept = i32 != POST_DROPPED;
    const int64_t i = i32;
    int lo = 0, hi = 0;
    if (g < n) lobe_range(sc, g, lo, hi);
    s_kept[threadIdx.x] = kept;
    float c[3] = {0.f, 0.f, 0.f};
    if (kept) {
        const float *mean = static_cast<const float *>(sc.means), *scl = static_cast<const float *>(sc.scales);
        const float *q = static_cast<const float *>(sc.quats), *op = static_cast<const float *>(sc.opac);
        float v[12];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            v[d] = mean[d * n + g];
            v[3 + d] = scl[d * n + g];
            c[d] = sc.c0[d * n + g];
        }
#pragma unroll
        for (int d = 0; d < 4; ++d) v[6 + d] = q[d * n + g];
        v[10] = op[g];
        v[11] = sc.gmask[g];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            o.means[d * N2 + i] = v[d];
            o.scales[d * N2 + i] = v[3 + d];
        }
#pragma unroll
        for (int d = 0; d < 4; ++d) o.quats[d * N2 + i] = v[6 + d];
        o.opac[i] = v[10];
        o.gmask[i] = v[11];
        o.lobe_off[i] = (int32_t)loff[g];
    }
    const int64_t gl = min(g0 + 256, n) - 1;   // the block's last Gaussian
    int b0, b1, t0, t1;
    lobe_range(sc, g0, b0, t0);
    lobe_range(sc, gl, t1, b1);
    const float *ax = static_cast<const float *>(sc.axis), *sh = static_cast<const float *>(sc.sharp);
    const float *am = static_cast<const float *>(sc.amp);
    int64_t base = loff[g0];   // first output lobe of the block
    for (int k0 = b0; k0 < b1; k0 += POST_TILE) {   // uniform
        const int k1 = min(k0 + POST_TILE, b1);
        for (int j = threadIdx.x; j < POST_TILE; j += 256) s_owner[j] = 256;   // a lobe no Gaussian owns
        __syncthreads();
        for (int k = max(lo, k0); k < min(hi, k1); ++k) s_owner[k - k0] = (uint16_t)threadIdx.x;
        __syncthreads();
        for (int h = 0; h < POST_TILE; h += 256) {   // uniform
            const int j = h + threadIdx.x, k = k0 + j;
            const bool mine = k < k1 && s_owner[j] < 256 && s_kept[s_owner[j]];
            float s = 0.f, m = 0.f, a[3] = {0.f, 0.f, 0.f};
            if (mine) {
                s = sh[k];
                m = sc.lmask[k];
#pragma unroll
                for (int d = 0; d < 3; ++d) a[d] = am[d * L + k];
            }
            const bool keep = mine && s >= tau_s;
            uint32_t tot;
            const uint32_t r = block_exclusive<uint32_t>(keep ? 1u : 0u, tot, shs);
            const int64_t p = base + r;
            if (keep && p < L2) {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    o.axis[d * L2 + p] = ax[d * L + k];
                    o.amp[d * L2 + p] = a[d];
                }
                o.sharp[p] = s;
                o.lmask[p] = m;
            }
            s_f[j] = mine && !keep ? m * lobe_mean_factor(s) : 0.f;
            s_owner[j] = mine && !keep ? 1 : 0;   // from here on: a removed lobe
#pragma unroll
            for (int d = 0; d < 3; ++d) s_a[d][j] = a[d];
            base += tot;
        }
        __syncthreads();
        if (kept)
            for (int k = max(lo, k0); k < min(hi, k1); ++k) {
                const int j = k - k0;
                if (!s_owner[j]) continue;
#pragma unroll
                for (int d = 0; d < 3; ++d) c[d] = fmaf(s_a[d][j], s_f[j], c[d]);
            }
        __syncthreads();
    }
    if (kept) {
#pragma unroll
        for (int d = 0; d < 3; ++d) o.c0[d * N2 + i] = c[d];
    }
}

// Workspace: state and look-back words (zeroed together), positions.
struct PostLayout {
    size_t state, flags, zeroed, gidx, loff, total;
};

static size_t al256(size_t x) { return (x + 255) / 256 * 256; }

static PostLayout post_layout(int64_t n) {
    PostLayout L{};
    size_t o = 0;
    auto take = [&](size_t b) { size_t r = o; o += al256(b); return r; };
    L.state = take(sizeof(PostState));
    L.flags = take(8 * div_up((uint64_t)n, POST_BLOCK));
    L.zeroed = o;
    L.gidx = take(4 * (size_t)n);
    L.loff = take(4 * (size_t)n);
    L.total = o;
    return L;
}

size_t post_workspace_bytes(int64_t n) { return post_layout(n < 0 ? 0 : n).total; }

cudaError_t launch_post_plan(const sg_scene &sc, float tau_o, float tau_s, void *ws, uint64_t *totals_host,
                             cudaStream_t s) {
    const PostLayout L = post_layout(sc.n);
    char *w = static_cast<char *>(ws);
    PostState *st = reinterpret_cast<PostState *>(w + L.state);
    cudaError_t e = cudaMemsetAsync(w, 0, L.zeroed, s);
    if (e != cudaSuccess) return e;
    if (sc.n > 0) {
        uint32_t *gidx = reinterpret_cast<uint32_t *>(w + L.gidx);
        k_post_count<<<(unsigned)div_up((uint64_t)sc.n, 256), 256, 0, s>>>(sc, tau_o, tau_s, gidx);
        k_post_scan<<<(unsigned)div_up((uint64_t)sc.n, POST_BLOCK), POST_THREADS, 0, s>>>(
            sc.n, gidx, reinterpret_cast<uint32_t *>(w + L.loff), st, reinterpret_cast<uint64_t *>(w + L.flags),
            sort_wait_polls());
        count_launches(2);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    e = cudaMemcpyAsync(totals_host, st, 24, cudaMemcpyDeviceToHost, s);   // totals and status
    if (e != cudaSuccess) return e;
    return cudaStreamSynchronize(s);
}

cudaError_t launch_post_apply(const sg_scene &sc, float tau_s, const void *ws, const sg_scene &out,
                              int64_t n_out, int64_t l_out, cudaStream_t s) {
    const PostLayout L = post_layout(sc.n);
    const char *w = static_cast<const char *>(ws);
    PostOut o;
    o.means = (float *)out.means; o.scales = (float *)out.scales; o.quats = (float *)out.quats;
    o.opac = (float *)out.opac; o.gmask = (float *)out.gmask; o.c0 = (float *)out.c0;
    o.axis = (float *)out.axis; o.sharp = (float *)out.sharp; o.amp = (float *)out.amp;
    o.lmask = (float *)out.lmask; o.lobe_off = (int32_t *)out.lobe_off;
    o.n_out = n_out; o.l_out = l_out;
    const uint64_t threads = sc.n > 0 ? (uint64_t)sc.n : 1;
    k_post_apply<<<(unsigned)div_up(threads, 256), 256, 0, s>>>(
        sc, tau_s, reinterpret_cast<const uint32_t *>(w + L.gidx), reinterpret_cast<const uint32_t *>(w + L.loff), o);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace sgk
