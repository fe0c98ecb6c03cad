// sort_small.cu -- keys and stable sort of one small system (build.cu has the
// general form: eight onesweep passes, one launch each).
//
// Up to kSmallSortMax particles the eight passes are latency: 68 us at N =
// 1031, 99 at 30011.  Here one cluster of up to sixteen blocks keeps everything
// in its shared memory and sorts in one launch: a stable LSD radix sort by
// 8-bit digits, positions split evenly over the blocks, digit counts read and
// keys sent through distributed shared memory.  Only the top five or six
// digits (40 or 48 bits, 13 or 16 octree levels) are sorted that way; the few
// keys that agree in them are put in order by insertion, since LSD passes
// leave such a run in the order of its particles' indices.  A run of more than
// kRunMax of them sends the cluster through all eight digits instead (a galaxy
// of 65536 has such runs in the top five digits).  Box, keys
// and sort: N = 1031 96 -> 39 us, 30011 129 -> 61, 65536 136 -> 83.  (Eight
// blocks of up to eight keys a thread: 47, 75 and 115; a pass is the keys' way
// through distributed shared memory, which more blocks share.)
#include <cooperative_groups.h>

#include "common.cuh"

namespace treegb {

namespace cg = cooperative_groups;

constexpr int kSmThreads = 1024, kSmWarps = kSmThreads / 32;
constexpr int kSmItems = 4;                           // keys per thread at most
constexpr int kSmBlock = kSmThreads * kSmItems;       // positions per block at most
constexpr int kSmCluster = 16;
constexpr int kRunMax = 32;
constexpr int64_t kTop5Max = 16384;                   // top five digits first up to this size, six above
static_assert((int64_t)kSmBlock * kSmCluster == kSmallSortMax && kSmallSortMax <= 65536, "indices are 16 bits here");

struct SmallSmem {
    uint64_t in_key[kSmBlock];       // this block's positions, written by the cluster
    uint64_t loc_key[kSmBlock];      // this block's keys in digit order
    uint16_t in_idx[kSmBlock], loc_idx[kSmBlock];
    uint16_t whist[kSmWarps][kRadix];
    uint32_t total[kRadix];          // this block's keys per digit (read by the cluster)
    uint32_t lstart[kRadix];         // ... first of them in digit order
    uint32_t gbase[kRadix];          // position of the first of them in the whole order
    uint32_t wt[32];
    uint32_t flag;                   // block 0: some run is too long
};

// Box from the partial minima and maxima (by every block for itself; block 0
// stores it), then the keys.
template <typename Real>
__global__ void __launch_bounds__(256) k_small_keys(const Real *__restrict__ x, int64_t n,
                                                    const double *__restrict__ part, int nparts,
                                                    DevBox *__restrict__ box, uint64_t *__restrict__ key) {
    __shared__ Real sh[6][8];
    __shared__ double res[6];
    __shared__ DevBox sbox;
    // a part without a finite value on an axis holds (DBL_MAX, -DBL_MAX) there
    const Real big = sizeof(Real) == 4 ? (Real)INFINITY : (Real)DBL_MAX;
    Real mn[3] = {big, big, big}, mx[3] = {-big, -big, -big};
    for (int b = threadIdx.x; b < nparts; b += 256) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            mn[d] = min(mn[d], (Real)part[b * 8 + d]);
            mx[d] = max(mx[d], (Real)part[b * 8 + 3 + d]);
        }
    }
    block_minmax<Real>(mn, mx, big, sh, res);
    __syncthreads();
    if (threadIdx.x == 0) {
        double lo[3] = {res[0], res[1], res[2]}, hi[3] = {res[3], res[4], res[5]};
        box_from_minmax(lo, hi, &sbox);
        if (blockIdx.x == 0) *box = sbox;
    }
    __syncthreads();
    for (int64_t i = blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256)
        key[i] = morton3(quantize(x[i], sbox.lo[0], sbox.scale), quantize(x[n + i], sbox.lo[1], sbox.scale),
                         quantize(x[2 * n + i], sbox.lo[2], sbox.scale));
}

// Block r of the cluster holds positions [r Q, min(n, (r + 1) Q)), Q <= kSmBlock.
__global__ void __launch_bounds__(kSmThreads, 1) k_small_sort(const uint64_t *__restrict__ kin, uint64_t *kout,
                                                              uint32_t *vout, uint32_t n, uint32_t Q, int top) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmallSmem &S = *reinterpret_cast<SmallSmem *>(smem_raw);
    cg::cluster_group cl = cg::this_cluster();
    const uint32_t rank = cl.block_rank(), nblk = cl.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = lanemask_lt();
    const uint32_t b0 = rank * Q;
    const uint32_t cnt = b0 < n ? min(Q, n - b0) : 0u;
    // each warp owns `per` consecutive positions, a multiple of 32
    const uint32_t per = ((Q + kSmWarps - 1) / kSmWarps + 31u) & ~31u;
    const int nit = (int)(per / 32u);
    if (tid == 0) S.flag = 0;
    bool done = false;
    for (int first = top; !done; first = 0) {
        for (int pass = first; pass < kSortPasses; ++pass) {
            const int shift = 8 * pass;
            uint64_t k[kSmItems];
            uint32_t v[kSmItems], rk[kSmItems];
            for (int i = tid; i < kSmWarps * kRadix / 2; i += kSmThreads)
                reinterpret_cast<uint32_t *>(&S.whist[0][0])[i] = 0;
#pragma unroll
            for (int i = 0; i < kSmItems; ++i) {
                const uint32_t p = warp * per + i * 32 + lane;
                k[i] = 0;
                v[i] = 0;
                if (i < nit && p < cnt) {
                    if (pass == first) { k[i] = kin[b0 + p]; v[i] = b0 + p; }
                    else { k[i] = S.in_key[p]; v[i] = S.in_idx[p]; }
                }
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kSmItems; ++i) {
                if (i >= nit) break;
                const bool ok = warp * per + i * 32 + lane < cnt;
                const uint32_t d = (uint32_t)(k[i] >> shift) & 0xffu;
                const uint32_t vm = __ballot_sync(0xffffffffu, ok);
                const uint32_t peers = match_digit8(d, ok ? vm : ~vm);
                const uint32_t c = ok ? S.whist[warp][d] : 0u;
                __syncwarp();
                const uint32_t pr = __popc(peers & lt);
                if (ok && pr == 0) S.whist[warp][d] = (uint16_t)(c + __popc(peers));
                __syncwarp();
                rk[i] = c + pr;
            }
            __syncthreads();
            // thread d owns digit d: offsets over the warps, the block's total
            uint32_t mine = 0;
            if (tid < kRadix) {
#pragma unroll 8
                for (int w = 0; w < kSmWarps; ++w) {
                    const uint32_t c = S.whist[w][tid];
                    S.whist[w][tid] = (uint16_t)mine;
                    mine += c;
                }
                S.total[tid] = mine;
            }
            // after this every block has its keys in registers and its totals out
            cl.sync();
            uint32_t all = 0, before = 0;
            if (tid < kRadix)
                for (uint32_t b = 0; b < nblk; ++b) {
                    const uint32_t c = *cl.map_shared_rank(&S.total[tid], b);
                    if (b < rank) before += c;
                    all += c;
                }
            const uint32_t g = block_exclusive_scan(all, S.wt, nullptr);
            const uint32_t l = block_exclusive_scan(mine, S.wt, nullptr);
            if (tid < kRadix) {
                S.lstart[tid] = l;
                S.gbase[tid] = g + before - l;  // position = gbase + place in the block's digit order
            }
            __syncthreads();
#pragma unroll
            for (int i = 0; i < kSmItems; ++i) {
                if (i < nit && warp * per + i * 32 + lane < cnt) {
                    const uint32_t d = (uint32_t)(k[i] >> shift) & 0xffu;
                    const uint32_t p = S.lstart[d] + S.whist[warp][d] + rk[i];
                    S.loc_key[p] = k[i];
                    S.loc_idx[p] = (uint16_t)v[i];
                }
            }
            __syncthreads();
            const bool last = pass == kSortPasses - 1;
            for (uint32_t j = tid; j < cnt; j += kSmThreads) {
                const uint64_t kk = S.loc_key[j];
                const uint32_t o = S.gbase[(uint32_t)(kk >> shift) & 0xffu] + j;
                if (last) {
                    kout[o] = kk;
                    vout[o] = S.loc_idx[j];
                } else {
                    const uint32_t r = o / Q, q = o - r * Q;
                    *cl.map_shared_rank(&S.in_key[q], r) = kk;
                    *cl.map_shared_rank(&S.in_idx[q], r) = S.loc_idx[j];
                }
            }
            cl.sync();
        }
        done = first == 0;
        if (!done) {
            // runs that agree in the sorted digits (the output is this cluster's: seen after the sync)
            const int kLow = 8 * top;
            for (uint32_t j = tid; j < cnt; j += kSmThreads) {
                const uint32_t i = b0 + j;
                const uint64_t h = __ldcg(kout + i) >> kLow;
                if (i > 0 && (__ldcg(kout + i - 1) >> kLow) == h) continue;  // not the run's first
                uint32_t e = i + 1;
                while (e < n && e - i <= kRunMax && (__ldcg(kout + e) >> kLow) == h) ++e;
                if (e - i > kRunMax) { atomicOr(cl.map_shared_rank(&S.flag, 0), 1u); continue; }
                // stable insertion by key: equal keys keep the order of their indices
                for (uint32_t a = i + 1; a < e; ++a) {
                    const uint64_t kk = __ldcg(kout + a);
                    const uint32_t vv = __ldcg(vout + a);
                    uint32_t b = a;
                    while (b > i && __ldcg(kout + b - 1) > kk) {
                        kout[b] = __ldcg(kout + b - 1);
                        vout[b] = __ldcg(vout + b - 1);
                        --b;
                    }
                    if (b != a) { kout[b] = kk; vout[b] = vv; }
                }
            }
            cl.sync();
            done = *cl.map_shared_rank(&S.flag, 0) == 0;
            cl.sync();  // the flag has been read before block 0 can leave
        }
    }
}

cudaError_t launch_small_keys(TreeWorkspace *ws, const void *x, int64_t n, cudaStream_t s) {
    const int nb = grid_for(n, 256, 152 * 2);
    if (ws->p.precision == TREE_F64)
        k_small_keys<double><<<nb, 256, 0, s>>>((const double *)x, n, ws->part, ws->box_parts, ws->box, ws->key_alt);
    else
        k_small_keys<float><<<nb, 256, 0, s>>>((const float *)x, n, ws->part, ws->box_parts, ws->box, ws->key_alt);
    ws->launches += 1;
    return cudaGetLastError();
}

// Launch of n particles: more blocks before more keys per thread (a pass is
// latency, and a block's part of it grows with its keys).
static uint32_t cluster_blocks(int64_t n) {
    return n <= 1024 ? 1 : n <= 2048 ? 2 : n <= 4096 ? 4 : n <= 8192 ? 8 : kSmCluster;
}

static cudaError_t cluster_config(uint32_t C, cudaStream_t s, cudaLaunchConfig_t &cfg, cudaLaunchAttribute &at) {
    cudaError_t e = cudaFuncSetAttribute(k_small_sort, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(SmallSmem));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_small_sort, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(kSmThreads);
    cfg.dynamicSmemBytes = sizeof(SmallSmem);
    cfg.stream = s;
    at = cudaLaunchAttribute{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return e;
}

// A device that is partitioned, or restricted to some of its SMs, may have no
// room for a cluster of sixteen blocks of 100 KB: larger systems then take the
// general passes.
int64_t small_sort_limit(int64_t n_max) {
    for (uint32_t C = cluster_blocks(n_max < kSmallSortMax ? n_max : kSmallSortMax); C > 0; C /= 2) {
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute at;
        int clusters = 0;
        if (cluster_config(C, nullptr, cfg, at) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&clusters, k_small_sort, &cfg) == cudaSuccess && clusters > 0)
            return C == kSmCluster ? kSmallSortMax : 1024 * (int64_t)C;
        cudaGetLastError();
    }
    return 0;
}

cudaError_t launch_small_sort(TreeWorkspace *ws, int64_t n, cudaStream_t s) {
    const uint32_t C = cluster_blocks(n);
    const uint32_t Q = (uint32_t)((n + C - 1) / C);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    cudaError_t e = cluster_config(C, s, cfg, at);
    if (e != cudaSuccess) return e;
    e = cudaLaunchKernelEx(&cfg, k_small_sort, (const uint64_t *)ws->key_alt, ws->key, ws->idx, (uint32_t)n, Q,
                           n <= kTop5Max ? 3 : 2);
    ws->launches += 1;
    return e;
}

}  // namespace treegb
