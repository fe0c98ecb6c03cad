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
//
// A node array that is too small cuts the tree as the level-by-level build
// does: children are numbered in order while they fit, and a cell whose
// children do not stays a leaf.  With X the first level whose nodes do not all
// fit, the levels before it are whole, and level X keeps the children of the
// cells before P, the parent of the node whose number is the array's capacity:
// numbers below `trunc`, P's first child.  At most seven slots are left, for
// the children of the first cells of level X (the first kCutKids nodes of
// level X + 1 tell which) and theirs in turn; everything else of level X is a
// leaf.  So the same kernels cut the tree, in parallel too; one thread follows
// the last seven.  Build of tight pairs with leaf_cap 1, which need 1.2 times
// the default array: N = 1048577 0.39 ms (level by level 0.90; one block
// building the whole tree 31.7), 1e7 2.4 (4.8).
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

// A cut tree (see above): what k_flat_nodes leaves for k_flat_links.
constexpr int kCutKids = 8;
struct FlatCut {
    uint32_t first[kCutKids], parent[kCutKids];  // the first nodes of level X + 1: first particle, parent
    uint32_t kids;                               // how many of them there are
    uint32_t P;
};
static_assert(sizeof(FlatCut) <= kLevels * sizeof(uint32_t), "kept in the row of flat_cnt after the totals");
constexpr uint32_t kCutInParent = 1u << 31;      // leaf of a particle: not its node of level X, but the one above

// A thread's positions: s, lev and lev of the position before.
template <int ITEMS>
struct FlatItems {
    int sd[ITEMS], lv[ITEMS], pv[ITEMS];
};

// Numbers, starts, parents and geometry of the nodes that start in the block's
// positions; ends of the nodes that end there; leaf of every particle.
// raw[node] = {first child or first particle, its end}.  CUT: the tree is cut
// at level X (nodes of that level are leaves here, T: number of the first one
// of the next level).
template <int ITEMS, bool CUT>
__device__ __forceinline__ void flat_number(const FlatItems<ITEMS> &it, const uint32_t (*base)[24], int64_t b0,
                                            int64_t last, int64_t n, const uint64_t *__restrict__ skey,
                                            uint32_t *__restrict__ nfirst, uint32_t *__restrict__ ncount,
                                            uint4 *__restrict__ ngeo, uint2 *__restrict__ raw,
                                            uint32_t *__restrict__ nparent, uint32_t *__restrict__ pleaf, int X,
                                            uint32_t T, uint32_t cap, FlatCut *cut) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = lanemask_lt();
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
        const int sd = it.sd[q], lv = it.lv[q], pv = it.pv[q];
        const int chunk = warp * ITEMS + q, k = chunk * 32 + lane;
        const int64_t i = b0 + k;
        const uint64_t k0 = k < last && i < n ? skey[i] : 0u;
        const uint32_t qx = compact3(k0 >> 2), qy = compact3(k0 >> 1), qz = compact3(k0);
        uint32_t prev = 0;        // number of the next node of level L - 1 at i
        uint32_t up = 0;          // node of level L - 1 that starts at i
        uint32_t closing = 0;     // node of level L - 1 that ends at i
        uint32_t above = 0;       // CUT: node of level L - 1 that holds i
        // the levels at which something starts or ends among the warp's positions, or is a leaf, and
        // the level before them
        const int top = max(lv, pv);
        int l0 = (int)__reduce_min_sync(0xffffffffu, (unsigned)min(sd, lv >= 0 ? lv : 64));
        int l1 = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(top, 0));
        if (CUT) { l0 = min(l0, X); l1 = min(l1, X + 1); }
#pragma unroll 1
        for (int L = max(l0 - 1, 0); L <= l1; ++L) {
            const bool starts = sd <= L && L <= lv;
            const bool ends = sd <= L && L <= pv;
            const uint32_t b = __ballot_sync(0xffffffffu, starts);
            const uint32_t id = base[chunk][L] + __popc(b & lt);
            const uint32_t par = L == sd ? prev - 1u : up;  // (of a node that starts here, L > 0)
            if (CUT && L > X) {
                if (starts && id - T < (uint32_t)kCutKids) {
                    cut->first[id - T] = (uint32_t)i;
                    cut->parent[id - T] = par;
                }
                break;
            }
            if (ends) {
                const uint32_t c = id - 1u;
                if (L > sd) raw[closing].y = id;       // the children of the node above end here too
                if (!CUT || c < cap) {
                    if (L == pv || (CUT && L == X)) raw[c].y = (uint32_t)i;  // a leaf: its particles end
                    ncount[c] = (uint32_t)i;           // (its end; k_flat_links subtracts the start)
                }
                closing = c;
            }
            const bool leaf = L == lv || (CUT && L == X);
            if (starts) {
                const uint32_t cmask = ~((1u << (kBits - L)) - 1u);
                if (!CUT || id < cap) {
                    nfirst[id] = (uint32_t)i;
                    nparent[id] = L == 0 ? id : par;
                    ngeo[id] = make_uint4(qx & cmask, qy & cmask, qz & cmask, (uint32_t)L | (leaf ? 0x100u : 0u));
                    if (leaf) raw[id].x = (uint32_t)i;
                }
                if (L > sd) raw[up].x = id;
                if (CUT && id == cap) cut->P = par;    // (level X: the numbers before it fit)
                up = id;
            }
            const uint32_t in = starts ? id : id - 1u;
            if (L == (CUT ? min(lv, X) : lv)) pleaf[i] = CUT && in >= cap ? above | kCutInParent : in;
            if (CUT) above = in;
            prev = id;
        }
    }
}

// Second kernel: the nodes (flat_number).  SCANNED: cnt comes from k_flat_scan.
template <int ITEMS, bool SCANNED>
__global__ void __launch_bounds__(kFlatThreads) k_flat_nodes(
    const uint64_t *__restrict__ skey, int64_t n, const uint8_t *__restrict__ sdig,
    const uint8_t *__restrict__ plev, const uint32_t *__restrict__ cnt, int nblocks, uint32_t *__restrict__ nfirst,
    uint32_t *__restrict__ ncount, uint4 *__restrict__ ngeo, uint2 *__restrict__ raw, uint32_t *__restrict__ nparent,
    uint32_t *__restrict__ pleaf, uint32_t *ctr, uint32_t node_cap, FlatCut *cut) {
    constexpr int kTile = kFlatThreads * ITEMS;
    constexpr int kChunks = kTile / 32, kWarps = kFlatThreads / 32;
    __shared__ uint32_t base[kChunks][24];  // per chunk of 32 positions: number of its first node of each level
    __shared__ uint32_t part[kWarps][2][24];
    __shared__ uint32_t s_cut, s_next;      // level at which the tree is cut (kLevels: it fits), T of flat_number
    if (aborted(ctr, kStageAfter)) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
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
        // (levels after the first one that does not fit play no part)
        const uint32_t over = __ballot_sync(0xffffffffu, incl > node_cap);
        const int X = over ? __ffs(over) - 1 : kLevels;
        if (lane == 0) s_cut = (uint32_t)X;
        if (lane == X) s_next = incl;
        if (blockIdx.x == 0) {
            if (lane <= min(X, kLevels)) ctr[kCtrLevelStart + lane] = lane < kLevels ? incl - all : total;
            const uint32_t kids = __shfl_down_sync(0xffffffffu, all, 1);  // nodes of the next level
            if (lane == X && over) {
                ctr[kCtrFlatCut] = (uint32_t)X;
                cut->kids = min(kids, (uint32_t)kCutKids);
            }
        }
    }
    __syncthreads();
    const int64_t b0 = (int64_t)blockIdx.x * kTile;
    const int64_t last = min((int64_t)kTile, n + 1 - b0);  // position n ends what is still open
    FlatItems<ITEMS> it;
#pragma unroll
    for (int q = 0; q < ITEMS; ++q) {
        const int chunk = warp * ITEMS + q, k = chunk * 32 + lane;
        const int64_t i = b0 + k;
        it.sd[q] = 64; it.lv[q] = -1; it.pv[q] = -1;
        if (k < last) {
            it.sd[q] = i < n ? sdig[i] : 0;
            it.lv[q] = i < n ? plev[i] : -1;
            it.pv[q] = i > 0 ? plev[i - 1] : -1;
        }
        uint32_t mine = 0;
#pragma unroll
        for (int L = 0; L < kLevels; ++L) {
            const uint32_t c = __popc(__ballot_sync(0xffffffffu, it.sd[q] <= L && L <= it.lv[q]));
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
    if (s_cut == (uint32_t)kLevels)
        flat_number<ITEMS, false>(it, base, b0, last, n, skey, nfirst, ncount, ngeo, raw, nparent, pleaf, 0, 0u, 0u,
                                  nullptr);
    else
        flat_number<ITEMS, true>(it, base, b0, last, n, skey, nfirst, ncount, ngeo, raw, nparent, pleaf, (int)s_cut,
                                 s_next, node_cap, cut);
}

// Third kernel for a tree that is cut at level X: links, leaf flags, the nodes
// in the slots that are left, and the leaves of the particles.
__device__ __noinline__ void flat_links_cut(const uint64_t *__restrict__ skey, int64_t n, uint32_t *ctr,
                                            const FlatCut *cut, const uint2 *raw, uint32_t *nfirst, uint32_t *ncount,
                                            uint4 *ngeo, uint2 *nlink, uint32_t *nparent, uint8_t *plev,
                                            uint32_t *pleaf, uint32_t lcap, uint32_t cap, int32_t *dstatus) {
    // the last nodes, numbers trunc + q, in order, and the cells of level X that have children
    struct Node { uint32_t first, end, parent, level, child, nchild; };
    __shared__ Node tail[kCutKids];
    __shared__ uint32_t s_cell[kCutKids], s_child[kCutKids], s_nchild[kCutKids], s_tail, s_cells;
    const uint32_t X = ctr[kCtrFlatCut], P = cut->P, trunc = raw[P].x;
    if (threadIdx.x == 0) {
        const bool store = blockIdx.x == 0;
        uint32_t free = trunc, cells = 0;
        for (uint32_t k = 0; k < cut->kids;) {
            const uint32_t p = cut->parent[k];
            uint32_t m = 1;
            while (k + m < cut->kids && cut->parent[k + m] == p) ++m;
            if (p >= trunc || free + m > cap) break;
            s_cell[cells] = p; s_child[cells] = free; s_nchild[cells] = m;
            ++cells;
            for (uint32_t j = 0; j < m; ++j)
                tail[free - trunc + j] =
                    Node{cut->first[k + j], j + 1 < m ? cut->first[k + j + 1] : raw[p].y, p, X + 1u, 0u, 0u};
            free += m;
            k += m;
        }
        if (store) ctr[kCtrLevelStart + X + 1] = trunc;
        uint32_t q = 0;
        for (uint32_t L = X + 1; L < (uint32_t)kLevels; ++L) {
            const uint32_t end = free - trunc;
            if (store) ctr[kCtrLevelStart + L + 1] = free;
            bool fits = true;
            for (; q < end; ++q) {
                const Node c = tail[q];
                if (!fits || c.end - c.first <= lcap || L == (uint32_t)kMaxLevel) continue;
                uint32_t b[9], m = 0;
                octant_bounds(skey, c.first, c.end - c.first, 3 * (kMaxLevel - 1 - (int)L), b);
                for (int o = 0; o < 8; ++o) m += b[o + 1] > b[o] ? 1u : 0u;
                if (free + m > cap) { fits = false; continue; }
                tail[q].child = free;
                tail[q].nchild = m;
                for (int o = 0; o < 8; ++o)
                    if (b[o + 1] > b[o]) tail[free++ - trunc] = Node{b[o], b[o + 1], trunc + q, L + 1u, 0u, 0u};
            }
        }
        s_tail = free - trunc;
        s_cells = cells;
        if (store) set_status(dstatus, TREE_DEV_NODES);
    }
    __syncthreads();
    const uint32_t ntail = s_tail, ncells = s_cells;
    const uint32_t t0 = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    if (t0 < ntail) {
        const Node c = tail[t0];
        const uint32_t id = trunc + t0, cmask = ~((1u << (kBits - c.level)) - 1u);
        const uint64_t k0 = skey[c.first];
        nfirst[id] = c.first;
        ncount[id] = c.end - c.first;
        nparent[id] = c.parent;
        ngeo[id] = make_uint4(compact3(k0 >> 2) & cmask, compact3(k0 >> 1) & cmask, compact3(k0) & cmask,
                              c.level | (c.nchild ? 0u : 0x100u));
        nlink[id] = c.nchild ? make_uint2(c.child, c.nchild) : make_uint2(c.first, c.end - c.first);
    }
    for (uint32_t c = t0; c < trunc; c += stride) {
        const uint2 r = raw[c];
        const uint32_t w = ngeo[c].w, lev = w & 0xffu, first = nfirst[c], count = ncount[c] - first;
        ncount[c] = count;
        uint2 l = make_uint2(r.x, r.y - r.x);
        if (lev == X) {
            for (uint32_t k = 0; k < ncells; ++k)
                if (s_cell[k] == c) {
                    l = make_uint2(s_child[k], s_nchild[k]);
                    ngeo[c].w = lev;
                }
        } else if (!(w & 0x100u) && lev + 1u == X && r.x >= trunc) {
            l = make_uint2(first, count);  // P and the cells after it
            ngeo[c].w = w | 0x100u;
        }
        nlink[c] = l;
    }
    for (int64_t i = t0; i < n; i += stride) {
        if (plev[i] < X) continue;
        uint32_t a = pleaf[i], lev = X;
        if (a >= trunc) {  // (numbers from trunc to the capacity: children of P)
            a = a & kCutInParent ? a & ~kCutInParent : P;
            lev = X - 1u;
        } else {
            for (uint32_t q = 0; q < ntail; ++q)
                if (tail[q].parent == a && tail[q].first <= i && i < tail[q].end) { a = trunc + q; lev = tail[q].level; }
        }
        pleaf[i] = a;
        plev[i] = (uint8_t)lev;
    }
}

// Third kernel: ends become counts.
__global__ void __launch_bounds__(256) k_flat_links(const uint64_t *__restrict__ skey, int64_t n, uint32_t *ctr,
                                                    const FlatCut *cut, const uint2 *raw, uint32_t *nfirst,
                                                    uint32_t *ncount, uint4 *ngeo, uint2 *nlink, uint32_t *nparent,
                                                    uint8_t *plev, uint32_t *pleaf, uint32_t lcap, uint32_t node_cap,
                                                    int32_t *dstatus) {
    if (aborted(ctr, kStageAfter)) return;
    if (ctr[kCtrFlatCut]) {
        flat_links_cut(skey, n, ctr, cut, raw, nfirst, ncount, ngeo, nlink, nparent, plev, pleaf, lcap, node_cap,
                       dstatus);
        return;
    }
    const uint32_t nn = ctr[kCtrLevelStart + kLevels];
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < nn; c += gridDim.x * blockDim.x) {
        const uint2 r = raw[c];
        nlink[c] = make_uint2(r.x, r.y - r.x);
        ncount[c] -= nfirst[c];
    }
}

static FlatCut *flat_cut(TreeWorkspace *ws) {
    return reinterpret_cast<FlatCut *>(ws->flat_cnt + (size_t)(flat_octree_blocks(ws->n_max) + 1) * kLevels);
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
    k_flat_nodes<ITEMS, SCANNED><<<nb1, kFlatThreads, 0, s>>>(ws->key, n, ws->sdig, ws->plev, ws->flat_cnt, nb,
                                                              ws->nfirst, ws->ncount, ws->ngeo, ws->nraw, ws->nparent,
                                                              ws->pleaf, ws->ctr, (uint32_t)ws->node_cap, flat_cut(ws));
}

cudaError_t launch_octree_flat(TreeWorkspace *ws, int64_t n, cudaStream_t s) {
    // as few positions per thread as give at most kFlatMaxBlocks blocks
    const int64_t one = (int64_t)kFlatMaxBlocks * kFlatThreads;
    if (n <= one) flat_launch<1, false>(ws, n, s);
    else if (n <= 2 * one) flat_launch<2, false>(ws, n, s);
    else if (n <= 4 * one) flat_launch<4, false>(ws, n, s);
    else if (n <= kFlatItemsMax * one) flat_launch<kFlatItemsMax, false>(ws, n, s);
    else flat_launch<kFlatItemsMax, true>(ws, n, s);
    k_flat_links<<<grid_for(ws->node_cap, 256, 152 * 8), 256, 0, s>>>(
        ws->key, n, ws->ctr, flat_cut(ws), ws->nraw, ws->nfirst, ws->ncount, ws->ngeo, ws->nlink, ws->nparent, ws->plev,
        ws->pleaf, (uint32_t)ws->p.leaf_cap, (uint32_t)ws->node_cap, ws->dstatus);
    ws->launches += 1;
    return cudaGetLastError();
}

}  // namespace treegb
