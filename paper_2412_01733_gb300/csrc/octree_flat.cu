// octree_flat.cu -- the breadth-first octree straight from the sorted keys, in
// three launches (build.cu builds it level by level).
//
// With s(i) the number of leading octal digits that keys i-1 and i share (-1
// where a system starts) and t(j) that of keys j and j + leaf_cap (-1 past the
// end of j's system):
//   - a cell of level L > 0 is a node iff its parent holds more than leaf_cap
//     particles, i.e. iff some leaf_cap + 1 consecutive particles of the
//     parent share L - 1 digits; so the leaf that holds particle i has level
//     lev(i) = min(21, 1 + max t(j), j = i - leaf_cap .. i);
//   - the nodes whose first particle is i are those of levels
//     s(i) + 1 .. lev(i), the last of them a leaf, the others internal, each
//     the first child of the one before; the first one's parent is the latest
//     node of level s(i) that starts before i;
//   - the nodes that end at i are those of levels s(i) + 1 .. lev(i - 1): the
//     latest of their levels that start before i.
// Breadth-first numbers are ranks by (level, first particle), so 22 prefix
// counts over i, one per level, number every node, and everything about a
// node is known where it starts and where it ends, without any search.
//
// Level by level, the octree of a small system is 23 launches of latency
// (with the walk groups: 144 us at N = 1031, 210 at 30011, 380 at 2^20); this
// form is bound by latency too, but of three kernels (31, 31 and 87 us).
// Blocks of kTile positions sum the counts of all blocks before them
// themselves while there are at most kFlatMaxBlocks of them; beyond (2^20
// particles) one more launch scans the blocks' counts, level by level.
#include "common.cuh"

namespace treegb {

constexpr int kFlatThreads = 256;
constexpr int kFlatMaxBlocks = 512;
constexpr int kFlatItemsMax = 8;  // positions per thread
constexpr int kHalo = 16;         // leaf_cap at most

int64_t flat_octree_blocks(int64_t n_max) {
    const int64_t nb = (n_max + kFlatThreads * kFlatItemsMax - 1) / (kFlatThreads * kFlatItemsMax);
    return nb > kFlatMaxBlocks ? nb : kFlatMaxBlocks;
}

// Leading octal digits two keys share (21 if equal).
__device__ __forceinline__ int shared_digits(uint64_t a, uint64_t b) {
    const uint64_t d = a ^ b;
    return d ? (62 - (63 - __clzll((long long)d))) / 3 : kMaxLevel;
}

// First kernel: s(i) + 1 and lev(i) of every particle, and each block's
// number of nodes per level.
template <int ITEMS, bool SEG>
__global__ void __launch_bounds__(kFlatThreads) k_flat_count(const uint64_t *__restrict__ skey, int64_t n, int lcap,
                                                             const int64_t *__restrict__ seg_off, int64_t nseg,
                                                             uint8_t *__restrict__ sdig, uint8_t *__restrict__ plev,
                                                             uint32_t *__restrict__ cnt, const uint32_t *ctr) {
    constexpr int kTile = kFlatThreads * ITEMS;
    __shared__ uint64_t key[kTile + 2 * kHalo + 1];  // key[k]: particle b0 - kHalo + k
    __shared__ int8_t t[kTile + kHalo];              // t[k]: of particle b0 - kHalo + k
    __shared__ uint8_t bnd[SEG ? kTile + 2 * kHalo + 1 : 1];  // a system starts at particle b0 - kHalo + k
    __shared__ uint32_t diff[24];
    if (aborted(ctr, kStageAfter)) return;
    const int64_t b0 = (int64_t)blockIdx.x * kTile;
    if constexpr (SEG) {
        for (int k = threadIdx.x; k < kTile + 2 * kHalo + 1; k += kFlatThreads) bnd[k] = 0;
        __syncthreads();
        // the systems that start inside the tile and its halo
        const int64_t lo = b0 - kHalo, hi = b0 + kTile + kHalo;
        for (int64_t b = (lo > 0 ? seg_find(seg_off, nseg, lo < n ? lo : n - 1) : 0) + threadIdx.x; b < nseg;
             b += kFlatThreads) {
            const int64_t o = seg_off[b];
            if (o >= hi) break;
            if (o >= lo) bnd[o - lo] = 1;
        }
    }
    if (threadIdx.x < 24) diff[threadIdx.x] = 0;
    for (int k = threadIdx.x; k < kTile + 2 * kHalo; k += kFlatThreads) {
        const int64_t i = b0 - kHalo + k;
        key[k] = i >= 0 && i < n ? skey[i] : 0u;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < kTile + kHalo; k += kFlatThreads) {
        const int64_t j = b0 - kHalo + k;
        bool same = j >= 0 && j + lcap < n;
        if constexpr (SEG)
            for (int o = 1; o <= lcap; ++o) same &= bnd[k + o] == 0;
        t[k] = same ? (int8_t)shared_digits(key[k], key[k + lcap]) : (int8_t)-1;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
        const int k = q * kFlatThreads + threadIdx.x;
        const int64_t i = b0 + k;
        if (i >= n) continue;
        int m = -1;
        for (int o = 0; o <= lcap; ++o) m = max(m, (int)t[k + kHalo - o]);
        const int lev = min(kMaxLevel, 1 + m);
        bool head = i == 0;
        if constexpr (SEG) head = bnd[k + kHalo] != 0;
        const int sd = head ? 0 : shared_digits(key[k + kHalo - 1], key[k + kHalo]) + 1;
        sdig[i] = (uint8_t)sd;
        plev[i] = (uint8_t)lev;
        if (sd <= lev) {  // nodes start here at levels sd .. lev
            atomicAdd(&diff[sd], 1u);
            atomicSub(&diff[lev + 1], 1u);
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        // level counts: running sums of the interval ends
        uint32_t v = threadIdx.x < 24 ? diff[threadIdx.x] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
            if ((int)threadIdx.x >= o) v += y;
        }
        if (threadIdx.x < kLevels) cnt[(size_t)blockIdx.x * kLevels + threadIdx.x] = v;
    }
}

// Scan of the blocks' counts of one level per block (many blocks): counts
// become the numbers of nodes of the level in the blocks before; cnt[nblocks]
// holds the totals.
__global__ void __launch_bounds__(1024) k_flat_scan(uint32_t *__restrict__ cnt, int nblocks, const uint32_t *ctr) {
    __shared__ uint32_t wt[32];
    if (aborted(ctr, kStageAfter)) return;
    uint32_t *c = cnt + blockIdx.x;  // level
    const int per = (nblocks + 1023) / 1024;
    const int b0 = threadIdx.x * per, b1 = min(nblocks, b0 + per);
    uint32_t sum = 0;
#pragma unroll 8
    for (int b = b0; b < b1; ++b) sum += c[(size_t)b * kLevels];
    uint32_t total;
    uint32_t run = block_exclusive_scan(sum, wt, &total);
#pragma unroll 8
    for (int b = b0; b < b1; ++b) {
        const uint32_t v = c[(size_t)b * kLevels];
        c[(size_t)b * kLevels] = run;
        run += v;
    }
    if (threadIdx.x == 0) c[(size_t)nblocks * kLevels] = total;
}

// The tree when the node array is too small for it: one block builds it level
// by level, children of a node numbered only while they fit (as k_level).
__device__ __noinline__ void flat_overflow(const uint64_t *__restrict__ skey, int64_t n,
                                           const int64_t *__restrict__ seg_off, int64_t nseg, uint32_t *nfirst,
                                           uint32_t *ncount, uint4 *ngeo, uint2 *nlink, uint32_t *nparent,
                                           uint32_t *ctr, uint32_t lcap, uint32_t node_cap, int32_t *dstatus) {
    __shared__ uint32_t wt[32], s_trunc;
    const uint32_t tid = threadIdx.x;
    for (int64_t b = tid; b < nseg; b += kFlatThreads) {
        nfirst[b] = nseg > 1 ? (uint32_t)seg_off[b] : 0u;
        ncount[b] = nseg > 1 ? (uint32_t)(seg_off[b + 1] - seg_off[b]) : (uint32_t)n;
        nparent[b] = (uint32_t)b;
    }
    if (tid == 0) ctr[kCtrLevelStart] = 0;
    uint32_t start = 0, end = (uint32_t)nseg;
    for (int L = 0; L < kLevels; ++L) {
        if (tid == 0) s_trunc = 0xffffffffu;
        __syncthreads();
        const int shift = 3 * (kMaxLevel - 1 - L);
        const uint32_t cmask = ~((1u << (kBits - L)) - 1u);
        uint32_t base = end;  // first free node
        for (uint32_t t0 = start; t0 < end; t0 += kFlatThreads) {
            const uint32_t node = t0 + tid;
            const bool valid = node < end;
            const uint32_t first = valid ? nfirst[node] : 0u, count = valid ? ncount[node] : 0u;
            const uint64_t k0 = valid ? skey[first] : 0u;
            bool internal = valid && count > lcap && L < kMaxLevel;
            uint32_t b[9], nch = 0;
            if (internal) {
                octant_bounds(skey, first, count, shift, b);
#pragma unroll
                for (int o = 0; o < 8; ++o) nch += b[o + 1] > b[o] ? 1u : 0u;
            }
            uint32_t tot;
            const uint32_t cf = base + block_exclusive_scan(nch, wt, &tot);
            if (internal && (uint64_t)cf + nch > node_cap) {
                internal = false;
                atomicMin(&s_trunc, cf);
                set_status(dstatus, TREE_DEV_NODES);
            }
            if (valid) {
                ngeo[node] = make_uint4(compact3(k0 >> 2) & cmask, compact3(k0 >> 1) & cmask, compact3(k0) & cmask,
                                        (uint32_t)L | (internal ? 0u : 0x100u));
                nlink[node] = internal ? make_uint2(cf, nch) : make_uint2(first, count);
            }
            if (internal) {
                uint32_t c = cf;
#pragma unroll
                for (int o = 0; o < 8; ++o)
                    if (b[o + 1] > b[o]) {
                        nfirst[c] = b[o];
                        ncount[c] = b[o + 1] - b[o];
                        nparent[c] = node;
                        ++c;
                    }
            }
            base += tot;
            __syncthreads();
        }
        const uint32_t next = min(base, s_trunc);
        start = end;
        end = next;
        if (tid == 0) ctr[kCtrLevelStart + L + 1] = start;
        __syncthreads();
    }
}

// Second kernel: numbers, starts, parents and geometry of the nodes that
// start in the block's positions; ends of the nodes that end there; leaf of
// every particle.  raw[node] = {first child or first particle, its end}.
// SCANNED: cnt comes from k_flat_scan.
template <int ITEMS, bool SCANNED>
__global__ void __launch_bounds__(kFlatThreads) k_flat_nodes(
    const uint64_t *__restrict__ skey, int64_t n, const uint8_t *__restrict__ sdig,
    const uint8_t *__restrict__ plev, const uint32_t *__restrict__ cnt, int nblocks, uint32_t *__restrict__ nfirst, uint32_t *__restrict__ ncount,
    uint4 *__restrict__ ngeo, uint2 *__restrict__ nlink, uint2 *__restrict__ raw, uint32_t *__restrict__ nparent,
    uint32_t *__restrict__ pleaf, uint32_t *ctr, uint32_t lcap, uint32_t node_cap, int32_t *dstatus,
    const int64_t *__restrict__ seg_off, int64_t nseg) {
    constexpr int kTile = kFlatThreads * ITEMS;
    constexpr int kChunks = kTile / 32, kWarps = kFlatThreads / 32;
    __shared__ uint32_t base[kChunks][24];  // per chunk of 32 positions: number of its first node of each level
    __shared__ uint32_t part[kWarps][2][24];
    __shared__ uint32_t s_end;
    if (aborted(ctr, kStageAfter)) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lt = lanemask_lt();
    // nodes per level in the blocks before this one, and in all
    {
        uint32_t before = 0, all = 0;
        if (SCANNED) {
            if (warp == 0 && lane < kLevels) {
                before = cnt[(size_t)blockIdx.x * kLevels + lane];  // (position n's own block: the totals)
                all = cnt[(size_t)nblocks * kLevels + lane];
            }
        } else if (lane < kLevels)
            for (int b = warp; b < nblocks; b += kWarps) {
                const uint32_t c = cnt[(size_t)b * kLevels + lane];
                all += c;
                if (b < (int)blockIdx.x) before += c;
            }
        if (lane < 24) { part[warp][0][lane] = before; part[warp][1][lane] = all; }
    }
    __syncthreads();
    uint32_t myoff = 0;  // warp 0, lane L: first node of level L in this block
    if (warp == 0) {
        uint32_t before = 0, all = 0;
        if (lane < kLevels)
            for (int w = 0; w < kWarps; ++w) { before += part[w][0][lane]; all += part[w][1][lane]; }
        uint32_t incl = all;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        myoff = incl - all + before;
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        if (lane == 0) s_end = total;
        if (blockIdx.x == 0 && total <= node_cap && lane <= kLevels)
            ctr[kCtrLevelStart + lane] = lane < kLevels ? incl - all : total;
    }
    __syncthreads();
    if (s_end > node_cap) {
        if (blockIdx.x == 0) {
            if (tid == 0) ctr[kCtrFlatFull] = 1;  // the links below are final; the leaves' particles follow
            flat_overflow(skey, n, seg_off, nseg, nfirst, ncount, ngeo, nlink, nparent, ctr, lcap, node_cap, dstatus);
        }
        return;
    }
    const int64_t b0 = (int64_t)blockIdx.x * kTile;
    const int64_t last = min((int64_t)kTile, n + 1 - b0);  // position n ends what is still open
    int sd[ITEMS], lv[ITEMS], pv[ITEMS];
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
        const int chunk = warp * ITEMS + q, k = chunk * 32 + lane;
        const int64_t i = b0 + k;
        sd[q] = 64; lv[q] = -1; pv[q] = -1;
        if (k < last) {
            sd[q] = i < n ? sdig[i] : 0;
            lv[q] = i < n ? plev[i] : -1;
            pv[q] = i > 0 ? plev[i - 1] : -1;
        }
        uint32_t mine = 0;
#pragma unroll
        for (int L = 0; L < kLevels; ++L) {
            const uint32_t c = __popc(__ballot_sync(0xffffffffu, sd[q] <= L && L <= lv[q]));
            if (lane == L) mine = c;
        }
        if (lane < 24) base[chunk][lane] = mine;
    }
    __syncthreads();
    if (warp == 0 && lane < kLevels) {
        uint32_t run = myoff;
        for (int c = 0; c < kChunks; ++c) {
            const uint32_t v = base[c][lane];
            base[c][lane] = run;
            run += v;
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
        const int chunk = warp * ITEMS + q, k = chunk * 32 + lane;
        const int64_t i = b0 + k;
        const uint64_t k0 = k < last && i < n ? skey[i] : 0u;
        const uint32_t qx = compact3(k0 >> 2), qy = compact3(k0 >> 1), qz = compact3(k0);
        uint32_t prev = 0;        // number of the next node of level L - 1 at i
        uint32_t up = 0;          // node of level L - 1 that starts at i
        uint32_t closing = 0;     // node of level L - 1 that ends at i
        // the levels at which something starts or ends among the warp's positions, or is a leaf, and
        // the level before them
        const int top = max(lv[q], pv[q]);
        const int l0 = (int)__reduce_min_sync(0xffffffffu, (unsigned)min(sd[q], lv[q] >= 0 ? lv[q] : 64));
        const int l1 = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(top, 0));
#pragma unroll 1
        for (int L = max(l0 - 1, 0); L <= l1; ++L) {
            const bool starts = sd[q] <= L && L <= lv[q];
            const bool ends = sd[q] <= L && L <= pv[q];
            const uint32_t b = __ballot_sync(0xffffffffu, starts);
            const uint32_t id = base[chunk][L] + __popc(b & lt);
            if (ends) {
                const uint32_t c = id - 1u;
                if (L > sd[q]) raw[closing].y = id;       // the children of the node above end here too
                if (L == pv[q]) raw[c].y = (uint32_t)i;   // a leaf: its particles end
                ncount[c] = (uint32_t)i;                  // (its end; k_flat_links subtracts the start)
                closing = c;
            }
            if (starts) {
                const uint32_t cmask = ~((1u << (kBits - L)) - 1u);
                nfirst[id] = (uint32_t)i;
                nparent[id] = L == 0 ? id : L == sd[q] ? prev - 1u : up;
                ngeo[id] = make_uint4(qx & cmask, qy & cmask, qz & cmask, (uint32_t)L | (L == lv[q] ? 0x100u : 0u));
                if (L > sd[q]) raw[up].x = id;
                if (L == lv[q]) raw[id].x = (uint32_t)i;
                up = id;
            }
            if (L == lv[q]) pleaf[i] = starts ? id : id - 1u;
            prev = id;
        }
    }
}

// Third kernel: ends become counts.  (When the node array was too small, the
// counts are there, and the particles learn their leaves: a warp per leaf.)
__global__ void __launch_bounds__(256) k_flat_links(const uint32_t *__restrict__ ctr, const uint2 *__restrict__ raw,
                                                    const uint32_t *__restrict__ nfirst, uint32_t *__restrict__ ncount,
                                                    const uint4 *__restrict__ ngeo, uint2 *__restrict__ nlink,
                                                    uint8_t *__restrict__ plev, uint32_t *__restrict__ pleaf) {
    if (aborted(ctr, kStageAfter)) return;
    const uint32_t nn = ctr[kCtrLevelStart + kLevels];
    if (ctr[kCtrFlatFull]) {
        for (uint32_t c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < nn; c += (gridDim.x * blockDim.x) >> 5) {
            const uint32_t w = ngeo[c].w;
            if (!((w >> 8) & 1u)) continue;
            const uint2 l = nlink[c];
            for (uint32_t j = l.x + (threadIdx.x & 31); j < l.x + l.y; j += 32) {
                plev[j] = (uint8_t)(w & 0xffu);
                pleaf[j] = c;
            }
        }
        return;
    }
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < nn; c += gridDim.x * blockDim.x) {
        const uint2 r = raw[c];
        nlink[c] = make_uint2(r.x, r.y - r.x);
        ncount[c] -= nfirst[c];
    }
}

template <int ITEMS, bool SCANNED>
static void flat_launch(TreeWorkspace *ws, int64_t n, cudaStream_t s) {
    const int nb = (int)((n + kFlatThreads * ITEMS - 1) / (kFlatThreads * ITEMS));
    if (ws->nseg > 1)
        k_flat_count<ITEMS, true><<<nb, kFlatThreads, 0, s>>>(ws->key, n, ws->p.leaf_cap, ws->seg_off, ws->nseg,
                                                             ws->sdig, ws->plev, ws->flat_cnt, ws->ctr);
    else
        k_flat_count<ITEMS, false><<<nb, kFlatThreads, 0, s>>>(ws->key, n, ws->p.leaf_cap, nullptr, 1, ws->sdig,
                                                              ws->plev, ws->flat_cnt, ws->ctr);
    if (SCANNED) k_flat_scan<<<kLevels, 1024, 0, s>>>(ws->flat_cnt, nb, ws->ctr);
    ws->launches += SCANNED ? 3 : 2;
    // position n may need a block of its own
    const int nb1 = (int)((n + kFlatThreads * ITEMS) / (kFlatThreads * ITEMS));
    k_flat_nodes<ITEMS, SCANNED><<<nb1, kFlatThreads, 0, s>>>(ws->key, n, ws->sdig, ws->plev, ws->flat_cnt, nb, ws->nfirst,
                                                    ws->ncount, ws->ngeo, ws->nlink, ws->nraw, ws->nparent, ws->pleaf,
                                                    ws->ctr, (uint32_t)ws->p.leaf_cap, (uint32_t)ws->node_cap,
                                                    ws->dstatus, ws->seg_off, ws->nseg);
}

cudaError_t launch_octree_flat(TreeWorkspace *ws, int64_t n, cudaStream_t s) {
    // as few positions per thread as give at most kFlatMaxBlocks blocks
    const int64_t one = (int64_t)kFlatMaxBlocks * kFlatThreads;
    if (n <= one) flat_launch<1, false>(ws, n, s);
    else if (n <= 2 * one) flat_launch<2, false>(ws, n, s);
    else if (n <= 4 * one) flat_launch<4, false>(ws, n, s);
    else if (n <= kFlatItemsMax * one) flat_launch<kFlatItemsMax, false>(ws, n, s);
    else flat_launch<kFlatItemsMax, true>(ws, n, s);
    k_flat_links<<<grid_for(ws->node_cap, 256, 152 * 8), 256, 0, s>>>(ws->ctr, ws->nraw, ws->nfirst, ws->ncount,
                                                                      ws->ngeo, ws->nlink, ws->plev, ws->pleaf);
    ws->launches += 1;
    return cudaGetLastError();
}

}  // namespace treegb
