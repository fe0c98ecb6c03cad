// moments.cu -- cell moments in FP64 (Sec. 2: a far cell acts through its
// total mass at its centre of mass; the quadrupole is the next term of the
// expansion).
//
// Every cell sums its sources k (its particles, or its children as point
// masses at their centres of mass R_k) about a fixed point c near the cell's
// geometric centre (u_k = r_k - c, |u_k| <= sqrt(3) s, so no large
// cancellation):
//   M = sum m_k,  S = sum m_k u_k,  T = sum m_k u_k u_k^T,
//   R = c + S / M,  T_R = T - S S^T / M  (= sum m_k d_k d_k^T, d_k = r_k - R),
//   Q = sum_k Q_k + 3 T_R - tr(T_R) I,
// Q_k = 0 for particles: the parallel-axis theorem of the traceless
// quadrupole.  Massless cells get R = c, Q = 0.  M, S, T and Q are
// accumulated in FP64; rounded copies in the walk's precision are packed for
// the walk (FP32: -Q).
//
// Work order.  The FP64 pipe runs at 1/64 of the FP32 rate, and a warp
// issues its FP64 loop for its longest cell, so cells are first bucketed:
// leaves by particle count (one launch for all leaves, since they only need
// particles), internal cells by (level, number of children) (one launch per
// level, finest first).  A warp then mostly holds cells with equal trip
// counts.  The order inside a bucket is arbitrary; every cell's arithmetic
// is its own, so the results do not depend on it.
//
// Given-up waits.  The walk groups are made beside the moments, which do not
// need them, so a wait of the group scan may give up while these kernels run.
// They run on then (aborted(ctr, kStageGroupScan)): returning half-way would
// leave arrival counters behind that the next build's climb starts from, and
// slots of `order` unwritten.  The waits of the sort and the octree are over
// before the moments start; after one of those gave up, none of these kernels
// does anything.
#include "common.cuh"

namespace treegb {

// bucket of a node: leaves 0..kMomLeafBuckets-1 by min(count, 17) (count 0
// with count 1), internal cells kMomLeafBuckets + 8 level + (nchild - 1)
__device__ __forceinline__ uint32_t mom_bucket(uint4 g, uint2 l) {
    if ((g.w >> 8) & 1u) return min(max(l.y, 1u), (uint32_t)kMomLeafBuckets) - 1u;
    return (uint32_t)kMomLeafBuckets + 8u * (g.w & 0xffu) + (l.y - 1u);
}

// Bucket counts of all nodes.
__global__ void __launch_bounds__(256) k_mom_hist(const uint32_t *__restrict__ ctr, const uint4 *__restrict__ ngeo,
                                                  const uint2 *__restrict__ nlink, uint32_t *__restrict__ cnt) {
    // after a given-up wait of the sort or the octree the buckets stay empty, so no later moment kernel does any work
    if (aborted(ctr, kStageGroupScan)) return;
    __shared__ uint32_t sh[kMomBuckets];
    for (int i = threadIdx.x; i < kMomBuckets; i += blockDim.x) sh[i] = 0;
    __syncthreads();
    const uint32_t nn = ctr[kCtrLevelStart + kLevels];
    for (uint32_t node = blockIdx.x * blockDim.x + threadIdx.x; node < nn; node += gridDim.x * blockDim.x)
        atomicAdd(&sh[mom_bucket(ngeo[node], nlink[node])], 1u);
    __syncthreads();
    for (int i = threadIdx.x; i < kMomBuckets; i += blockDim.x)
        if (sh[i]) atomicAdd(cnt + i, sh[i]);
}

// Bucket offsets (every block scans the counts; block 0 stores them, with
// the total at [kMomBuckets]), then each tile of 256 nodes reserves its
// slots per bucket with one atomic per bucket and writes the node indices.
__global__ void __launch_bounds__(256) k_mom_scatter(const uint32_t *__restrict__ ctr, const uint4 *__restrict__ ngeo,
                                                     const uint2 *__restrict__ nlink, const uint32_t *__restrict__ cnt,
                                                     uint32_t *__restrict__ off, uint32_t *__restrict__ cursor,
                                                     uint32_t *__restrict__ order) {
    if (aborted(ctr, kStageGroupScan)) return;
    __shared__ uint32_t s_off[kMomBuckets + 1], s_cnt[kMomBuckets], s_base[kMomBuckets];
    for (int b = threadIdx.x; b < kMomBuckets; b += blockDim.x) s_cnt[b] = cnt[b];
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        for (int b = 0; b < kMomBuckets; ++b) {
            s_off[b] = run;
            run += s_cnt[b];
        }
        s_off[kMomBuckets] = run;
    }
    __syncthreads();
    if (blockIdx.x == 0)
        for (int b = threadIdx.x; b <= kMomBuckets; b += blockDim.x) off[b] = s_off[b];
    const uint32_t nn = ctr[kCtrLevelStart + kLevels];
    for (uint32_t base = blockIdx.x * blockDim.x; base < nn; base += gridDim.x * blockDim.x) {
        for (int b = threadIdx.x; b < kMomBuckets; b += blockDim.x) s_cnt[b] = 0;
        __syncthreads();
        const uint32_t node = base + threadIdx.x;
        const bool valid = node < nn;
        uint32_t b = 0, rank = 0;
        if (valid) {
            b = mom_bucket(ngeo[node], nlink[node]);
            rank = atomicAdd(&s_cnt[b], 1u);
        }
        __syncthreads();
        for (int q = threadIdx.x; q < kMomBuckets; q += blockDim.x)
            if (s_cnt[q]) s_base[q] = atomicAdd(cursor + q, s_cnt[q]);
        __syncthreads();
        if (valid) order[s_off[b] + s_base[b] + rank] = node;
        __syncthreads();
    }
}

// FP64 sums of one cell about c and its finished moments.
struct MomSums {
    double M = 0, sx = 0, sy = 0, sz = 0, txx = 0, tyy = 0, tzz = 0, txy = 0, txz = 0, tyz = 0;
    double qxx = 0, qyy = 0, qzz = 0, qxy = 0, qxz = 0, qyz = 0;  // sum of the sources' own Q
    __device__ __forceinline__ void add(double m, double ux, double uy, double uz) {
        // every rounding explicit: the kernels that sum cells round alike
        M += m;
        const double mx = __dmul_rn(m, ux), my = __dmul_rn(m, uy), mz = __dmul_rn(m, uz);
        sx = __dadd_rn(sx, mx); sy = __dadd_rn(sy, my); sz = __dadd_rn(sz, mz);
        txx = fma(mx, ux, txx); tyy = fma(my, uy, tyy); tzz = fma(mz, uz, tzz);
        txy = fma(mx, uy, txy); txz = fma(mx, uz, txz); tyz = fma(my, uz, tyz);
    }
};

template <typename Real>
__device__ __forceinline__ void mom_store(const MomSums &a, double cx, double cy, double cz, uint32_t node,
                                          double *__restrict__ mom64, int64_t cap,
                                          typename Vec4<Real>::T *__restrict__ mom_a,
                                          typename Vec4<Real>::T *__restrict__ mom_b,
                                          typename Vec2<Real>::T *__restrict__ mom_c) {
    double Rx = cx, Ry = cy, Rz = cz, qxx = 0, qyy = 0, qzz = 0, qxy = 0, qxz = 0, qyz = 0;
    if (a.M != 0.0) {
        const double iM = 1.0 / a.M;
        Rx = fma(a.sx, iM, cx); Ry = fma(a.sy, iM, cy); Rz = fma(a.sz, iM, cz);
        const double nx = -a.sx, ny = -a.sy, nz = -a.sz;
        const double txx = fma(__dmul_rn(nx, a.sx), iM, a.txx), tyy = fma(__dmul_rn(ny, a.sy), iM, a.tyy);
        const double tzz = fma(__dmul_rn(nz, a.sz), iM, a.tzz), txy = fma(__dmul_rn(nx, a.sy), iM, a.txy);
        const double txz = fma(__dmul_rn(nx, a.sz), iM, a.txz), tyz = fma(__dmul_rn(ny, a.sz), iM, a.tyz);
        const double tr = txx + tyy + tzz;
        qxx = a.qxx + fma(3.0, txx, -tr); qyy = a.qyy + fma(3.0, tyy, -tr); qzz = a.qzz + fma(3.0, tzz, -tr);
        qxy = fma(3.0, txy, a.qxy); qxz = fma(3.0, txz, a.qxz); qyz = fma(3.0, tyz, a.qyz);
    }
    mom64[node] = a.M; mom64[cap + node] = Rx; mom64[2 * cap + node] = Ry; mom64[3 * cap + node] = Rz;
    mom64[4 * cap + node] = qxx; mom64[5 * cap + node] = qyy; mom64[6 * cap + node] = qzz;
    mom64[7 * cap + node] = qxy; mom64[8 * cap + node] = qxz; mom64[9 * cap + node] = qyz;
    // the FP32 walk copies hold -Q (the sign its packed pair terms want)
    const double qs = sizeof(Real) == 4 ? -1.0 : 1.0;
    typename Vec4<Real>::T A, B;
    typename Vec2<Real>::T C;
    A.x = (Real)Rx; A.y = (Real)Ry; A.z = (Real)Rz; A.w = (Real)a.M;
    B.x = (Real)(qs * qxx); B.y = (Real)(qs * qyy); B.z = (Real)(qs * qzz); B.w = (Real)(qs * qxy);
    C.x = (Real)(qs * qxz); C.y = (Real)(qs * qyz);
    mom_a[node] = A; mom_b[node] = B; mom_c[node] = C;
}

// Expansion point c of a node: its geometric centre, in the frame of the
// node's own segment.  The FP32 path rounds it to FP32 with one FP32 fused
// multiply-add (any point near the cell serves; the FP32 particle
// coordinates then differ from it by exactly representable FP64 values).
template <typename Real>
__device__ __forceinline__ void mom_centre(uint4 g, uint32_t node, const DevBox *__restrict__ box,
                                           const uint32_t *__restrict__ nfirst, const int64_t *__restrict__ seg_off,
                                           int64_t nseg, double &cx, double &cy, double &cz) {
    const DevBox *bx = nseg > 1 ? box + seg_find(seg_off, nseg, nfirst[node]) : box;
    const int lvl = (int)(g.w & 0xffu);
    if (sizeof(Real) == 4) {
        const float half = 0.5f * (float)(1u << (kBits - lvl)), unit = (float)bx->unit;
        cx = (double)__fmaf_rn((float)g.x + half, unit, (float)bx->lo[0]);
        cy = (double)__fmaf_rn((float)g.y + half, unit, (float)bx->lo[1]);
        cz = (double)__fmaf_rn((float)g.z + half, unit, (float)bx->lo[2]);
    } else {
        const double half = 0.5 * (double)(1u << (kBits - lvl)), unit = bx->unit;
        cx = fma((double)g.x + half, unit, bx->lo[0]);
        cy = fma((double)g.y + half, unit, bx->lo[1]);
        cz = fma((double)g.z + half, unit, bx->lo[2]);
    }
}

// Sums over the particles [first, end) of a leaf.  Four loads are in flight at
// a time; the sums keep the particles' order.
template <typename Real>
__device__ __forceinline__ void mom_leaf(MomSums &a, const typename Vec4<Real>::T *__restrict__ spos, uint32_t first,
                                         uint32_t end, double cx, double cy, double cz) {
    for (uint32_t j = first; j < end; j += 4) {
        typename Vec4<Real>::T p[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (j + k < end) p[k] = spos[j + k];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (j + k < end) a.add((double)p[k].w, (double)p[k].x - cx, (double)p[k].y - cy, (double)p[k].z - cz);
    }
}

// Moments of internal cell `nd` by a half-warp (c = lane & 15), one of the
// sixteen sums per lane:
//   c = 0: M;  1..3: S;  4..9: T (xx yy zz xy xz yz);  10..15: sum of the
//   children's Q (same order).
// Every sum is acc = fma(m ua, ub, acc) with ones in the places of missing
// factors, which rounds as MomSums::add does, so the results are those of one
// thread doing all sixteen.  All 32 lanes call it together; has: this half
// has a cell.
template <typename Real>
__device__ __forceinline__ void mom_cell_half(uint32_t nd, bool has, int lane, const uint4 *__restrict__ ngeo,
                                              const uint2 *__restrict__ nlink, DevBox *__restrict__ box,
                                              const uint32_t *__restrict__ nfirst, const int64_t *__restrict__ seg_off,
                                              int64_t nseg, double *mom64, int64_t cap, Real *__restrict__ mom_a,
                                              Real *__restrict__ mom_b, Real *__restrict__ mom_c) {
    const int c = lane & 15, hb = lane & 16;
    const uint2 lk = nlink[nd];
    const uint4 g = ngeo[nd];
    // axes (0 x, 1 y, 2 z) of this lane's factors; 3: one
    const int aa = c == 0 ? 3 : c <= 3 ? c - 1 : c <= 6 ? c - 4 : c <= 8 ? 0 : c == 9 ? 1 : 3;
    const int ab = c <= 3 ? 3 : c <= 6 ? c - 4 : c == 7 ? 1 : c <= 9 ? 2 : 3;
    // rows of mom64 this lane's factors come from
    const double *rm = mom64, *ra = mom64 + (c >= 10 ? c - 6 : 1 + (aa & 3)) * cap, *rb = mom64 + (1 + (ab & 3)) * cap;
    const bool lm = c < 10, la = aa < 3 || c >= 10, lb = ab < 3;
    const int nch = has ? (int)lk.y : 0;
    double vm[8], va[8], vb[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        vm[k] = va[k] = vb[k] = 1.0;
        if (k < nch) {
            if (lm) vm[k] = __ldcg(rm + lk.x + k);
            if (la) va[k] = __ldcg(ra + lk.x + k);
            if (lb) vb[k] = __ldcg(rb + lk.x + k);
        }
    }
    double cx, cy, cz;
    mom_centre<Real>(g, nd, box, nfirst, seg_off, nseg, cx, cy, cz);
    const double ca = aa == 0 ? cx : aa == 1 ? cy : cz, cb = ab == 0 ? cx : ab == 1 ? cy : cz;
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        if (k < nch) {
            const double ua = aa < 3 ? va[k] - ca : va[k], ub = ab < 3 ? vb[k] - cb : vb[k];
            acc = fma(__dmul_rn(vm[k], ua), ub, acc);
        }
    }
    const double M = __shfl_sync(0xffffffffu, acc, hb);
    const double sx = __shfl_sync(0xffffffffu, acc, hb + 1), sy = __shfl_sync(0xffffffffu, acc, hb + 2),
                 sz = __shfl_sync(0xffffffffu, acc, hb + 3);
    const double iM = M != 0.0 ? 1.0 / M : 0.0;
    // T about the centre of mass, in the lanes of T
    const double sa = aa == 0 ? sx : aa == 1 ? sy : sz, sb = ab == 0 ? sx : ab == 1 ? sy : sz;
    const double T = fma(__dmul_rn(-sa, sb), iM, acc);
    const double txx = __shfl_sync(0xffffffffu, T, hb + 4), tyy = __shfl_sync(0xffffffffu, T, hb + 5),
                 tzz = __shfl_sync(0xffffffffu, T, hb + 6);
    const double Tc = __shfl_sync(0xffffffffu, T, hb + (c >= 10 ? c - 6 : c));  // Q lane <- its T lane
    double out = acc;  // M
    if (c >= 1 && c <= 3) out = M != 0.0 ? fma(acc, iM, ca) : ca;
    if (c >= 10) {
        const double tr = txx + tyy + tzz;
        out = M == 0.0 ? 0.0 : c <= 12 ? acc + fma(3.0, Tc, -tr) : fma(3.0, Tc, acc);
    }
    if (has && (c <= 3 || c >= 10)) {
        mom64[(c <= 3 ? c : c - 6) * cap + nd] = out;
        const double qs = sizeof(Real) == 4 ? -1.0 : 1.0;  // the FP32 walk copies hold -Q
        if (c <= 3) mom_a[4 * (size_t)nd + (c == 0 ? 3 : c - 1)] = (Real)out;
        else if (c <= 13) mom_b[4 * (size_t)nd + (c - 10)] = (Real)(qs * out);
        else mom_c[2 * (size_t)nd + (c - 14)] = (Real)(qs * out);
        if (c == 0 && nd < (uint32_t)nseg) box[nd].r5fit = pc_r5_fits(box[nd].k, (Real)M) ? 1 : 0;
    }
}

// The whole moment tree in one launch: a lane takes a leaf, and whoever
// finishes the last child of a cell goes on with that cell, up to the root
// (one arrival counter per cell, back at zero when the cell's children are
// done, so the next pass finds it clear).  Nobody waits for anybody.  The
// same sums in the same order as level by level (k_moments_level), which is
// 21 launches of latency for a small system; here the latency is that of one
// path of about ten cells, and most of it is FP64 latency (ncu: 60 % of a
// warp's time in fixed-latency waits).  So what a cell needs is loaded before
// it is needed, and while a warp has one or two cells left (the upper part of
// every path) sixteen lanes share each; with more cells to a warp, a lane
// does its own (sixteen lanes for all of them took longer, 144 us against 104
// at N = 30011, the cells of a warp then following one another).  BUCKETS:
// leaves in bucket order.
template <typename Real, bool BUCKETS>
__global__ void __launch_bounds__(64) k_moments_climb(
    const uint32_t *__restrict__ ctr, const uint32_t *__restrict__ off, const uint32_t *__restrict__ order,
    const uint4 *__restrict__ ngeo, const uint2 *__restrict__ nlink, const uint32_t *__restrict__ nparent,
    uint32_t *__restrict__ arrived, const typename Vec4<Real>::T *__restrict__ spos, DevBox *__restrict__ box,
    const uint32_t *__restrict__ nfirst, const int64_t *__restrict__ seg_off, int64_t nseg, double *mom64, int64_t cap,
    typename Vec4<Real>::T *__restrict__ mom_a, typename Vec4<Real>::T *__restrict__ mom_b,
    typename Vec2<Real>::T *__restrict__ mom_c) {
    if (aborted(ctr, kStageGroupScan)) return;
    const int lane = threadIdx.x & 31;
    const uint32_t end = BUCKETS ? off[kMomLeafBuckets] : ctr[kCtrLevelStart + kLevels];
    const uint32_t stride = gridDim.x * blockDim.x;
    for (uint32_t t0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); t0 < end; t0 += stride) {
        const uint32_t t = t0 + lane;
        bool active = t < end;  // this lane has finished cell `node`
        // node's parent, and the parent's children
        uint32_t node = 0, par = 0;
        uint2 lk = make_uint2(0, 0);
        double cx, cy, cz;
        if (active) {
            node = BUCKETS ? order[t] : t;
            const uint4 g = ngeo[node];
            active = BUCKETS || ((g.w >> 8) & 1u);
            if (active) {
                lk = nlink[node];
                par = nparent[node];
                mom_centre<Real>(g, node, box, nfirst, seg_off, nseg, cx, cy, cz);
                MomSums a;
                mom_leaf<Real>(a, spos, lk.x, lk.x + lk.y, cx, cy, cz);
                lk = nlink[par];
                mom_store<Real>(a, cx, cy, cz, node, mom64, cap, mom_a, mom_b, mom_c);
                if (node < (uint32_t)nseg) box[node].r5fit = pc_r5_fits(box[node].k, (Real)a.M) ? 1 : 0;
            }
        }
        for (;;) {
            __threadfence();  // the finished cells' moments before their arrivals
            __syncwarp();
            bool ready = false;
            if (active && node >= (uint32_t)nseg) ready = atomicAdd(arrived + par, 1u) + 1u == lk.y;
            const uint32_t todo = __ballot_sync(0xffffffffu, ready);
            if (!todo) break;
            __threadfence();  // the other children's arrivals before their moments
            active = ready;
            if (ready) {
                node = par;
                arrived[node] = 0;
                par = nparent[node];
            }
            if (__popc(todo) <= 2) {
                const int l0 = __ffs(todo) - 1, l1 = 31 - __clz(todo);
                const uint32_t nd = __shfl_sync(0xffffffffu, node, lane < 16 ? l0 : l1);
                if (ready) lk = nlink[par];
                mom_cell_half<Real>(nd, lane < 16 || l1 != l0, lane, ngeo, nlink, box, nfirst, seg_off, nseg, mom64,
                                    cap, reinterpret_cast<Real *>(mom_a), reinterpret_cast<Real *>(mom_b),
                                    reinterpret_cast<Real *>(mom_c));
            } else if (ready) {
                mom_centre<Real>(ngeo[node], node, box, nfirst, seg_off, nseg, cx, cy, cz);
                MomSums b;
                const uint32_t k1 = lk.x + lk.y;
                for (uint32_t k0 = lk.x; k0 < k1; k0 += 4) {
                    double r[4][10];
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int c = 0; c < 10; ++c)
                            if (k0 + j < k1) r[j][c] = __ldcg(mom64 + c * cap + k0 + j);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (k0 + j < k1) {
                            b.add(r[j][0], r[j][1] - cx, r[j][2] - cy, r[j][3] - cz);
                            b.qxx += r[j][4]; b.qyy += r[j][5]; b.qzz += r[j][6];
                            b.qxy += r[j][7]; b.qxz += r[j][8]; b.qyz += r[j][9];
                        }
                }
                lk = nlink[par];
                mom_store<Real>(b, cx, cy, cz, node, mom64, cap, mom_a, mom_b, mom_c);
                if (node < (uint32_t)nseg) box[node].r5fit = pc_r5_fits(box[node].k, (Real)b.M) ? 1 : 0;
            }
        }
    }
}

// All leaves, in bucket order: sums over the cell's particles.
template <typename Real>
__global__ void __launch_bounds__(256) k_moments_leaves(
    const uint32_t *__restrict__ off, const uint32_t *__restrict__ order, const uint4 *__restrict__ ngeo,
    const uint2 *__restrict__ nlink, const typename Vec4<Real>::T *__restrict__ spos, const DevBox *__restrict__ box,
    const uint32_t *__restrict__ nfirst, const int64_t *__restrict__ seg_off, int64_t nseg, double *__restrict__ mom64,
    int64_t cap, typename Vec4<Real>::T *__restrict__ mom_a, typename Vec4<Real>::T *__restrict__ mom_b,
    typename Vec2<Real>::T *__restrict__ mom_c) {
    const uint32_t end = off[kMomLeafBuckets];
    for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < end; t += gridDim.x * blockDim.x) {
        const uint32_t node = order[t];
        const uint4 g = ngeo[node];
        const uint2 lk = nlink[node];
        double cx, cy, cz;
        mom_centre<Real>(g, node, box, nfirst, seg_off, nseg, cx, cy, cz);
        MomSums a;
        mom_leaf<Real>(a, spos, lk.x, lk.x + lk.y, cx, cy, cz);
        mom_store<Real>(a, cx, cy, cz, node, mom64, cap, mom_a, mom_b, mom_c);
    }
}

// Internal cells of level L: sums over the children's (M_k, R_k, Q_k).
template <typename Real>
__global__ void __launch_bounds__(256) k_moments_level(
    int L, const uint32_t *__restrict__ off, const uint32_t *__restrict__ order, const uint4 *__restrict__ ngeo,
    const uint2 *__restrict__ nlink, const DevBox *__restrict__ box, const uint32_t *__restrict__ nfirst,
    const int64_t *__restrict__ seg_off, int64_t nseg, double *__restrict__ mom64, int64_t cap,
    typename Vec4<Real>::T *__restrict__ mom_a, typename Vec4<Real>::T *__restrict__ mom_b,
    typename Vec2<Real>::T *__restrict__ mom_c) {
    const uint32_t b0 = kMomLeafBuckets + 8 * L;
    const uint32_t start = off[b0], end = off[b0 + 8];
    const double *M_ = mom64, *Rx_ = mom64 + cap, *Ry_ = mom64 + 2 * cap, *Rz_ = mom64 + 3 * cap;
    for (uint32_t t = start + blockIdx.x * blockDim.x + threadIdx.x; t < end; t += gridDim.x * blockDim.x) {
        const uint32_t node = order[t];
        const uint4 g = ngeo[node];
        const uint2 lk = nlink[node];
        double cx, cy, cz;
        mom_centre<Real>(g, node, box, nfirst, seg_off, nseg, cx, cy, cz);
        MomSums a;
        for (uint32_t k = lk.x; k < lk.x + lk.y; ++k) {
            a.add(M_[k], Rx_[k] - cx, Ry_[k] - cy, Rz_[k] - cz);
            a.qxx += mom64[4 * cap + k]; a.qyy += mom64[5 * cap + k]; a.qzz += mom64[6 * cap + k];
            a.qxy += mom64[7 * cap + k]; a.qxz += mom64[8 * cap + k]; a.qyz += mom64[9 * cap + k];
        }
        mom_store<Real>(a, cx, cy, cz, node, mom64, cap, mom_a, mom_b, mom_c);
    }
}

// Per segment b (its root is node b), whether the walk may take its r^-5
// far-cell form: pc_r5_fits of the segment's cube and root mass.
template <typename V4, typename Real>
__global__ void __launch_bounds__(256) k_r5_flags(const uint32_t *__restrict__ ctr, DevBox *box,
                                                  const V4 *__restrict__ mom_a, int64_t nseg) {
    if (aborted(ctr, kStageGroupScan)) return;
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < nseg; b += (int64_t)gridDim.x * blockDim.x)
        box[b].r5fit = pc_r5_fits(box[b].k, (Real)mom_a[b].w) ? 1 : 0;
}

template <typename Real>
static cudaError_t moments_impl(TreeWorkspace *ws, cudaStream_t s) {
    using V4 = typename Vec4<Real>::T;
    using V2 = typename Vec2<Real>::T;
    uint32_t *cnt = ws->mbucket, *off = ws->mbucket + kMomBuckets, *cursor = ws->mbucket + 2 * kMomBuckets + 1;
    const int64_t cap = ws->node_cap;
    const bool climb = ws->n <= kClimbMaxN, buckets = !climb || ws->n > kClimbPlainN;
    if (climb && !buckets) {
        k_moments_climb<Real, false><<<grid_for(cap, 64, 152 * 16), 64, 0, s>>>(
            ws->ctr, off, ws->morder, ws->ngeo, ws->nlink, ws->nparent, ws->marrived, (const V4 *)ws->spos, ws->box,
            ws->nfirst, ws->seg_off, ws->nseg, ws->mom64, cap, (V4 *)ws->mom_a, (V4 *)ws->mom_b, (V2 *)ws->mom_c);
        ws->launches += 1;
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(ws->mbucket, 0, (3 * kMomBuckets + 1) * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    k_mom_hist<<<grid_for(cap, 256, 152 * 8), 256, 0, s>>>(ws->ctr, ws->ngeo, ws->nlink, cnt);
    k_mom_scatter<<<grid_for(cap, 256, 152 * 8), 256, 0, s>>>(ws->ctr, ws->ngeo, ws->nlink, cnt, off,
                                                                             cursor, ws->morder);
    if (climb) {
        k_moments_climb<Real, true><<<grid_for(cap, 64, 152 * 16), 64, 0, s>>>(
            ws->ctr, off, ws->morder, ws->ngeo, ws->nlink, ws->nparent, ws->marrived, (const V4 *)ws->spos, ws->box,
            ws->nfirst, ws->seg_off, ws->nseg, ws->mom64, cap, (V4 *)ws->mom_a, (V4 *)ws->mom_b, (V2 *)ws->mom_c);
        ws->launches += 3;
        return cudaGetLastError();
    }
    k_moments_leaves<Real><<<grid_for(cap, 256, 152 * 8), 256, 0, s>>>(
        off, ws->morder, ws->ngeo, ws->nlink, (const V4 *)ws->spos, ws->box, ws->nfirst, ws->seg_off, ws->nseg,
        ws->mom64, cap, (V4 *)ws->mom_a, (V4 *)ws->mom_b, (V2 *)ws->mom_c);
    const int nbl = grid_for(cap, 256, 152 * 8);
    for (int L = kMaxLevel - 1; L >= 0; --L)
        k_moments_level<Real><<<nbl, 256, 0, s>>>(L, off, ws->morder, ws->ngeo, ws->nlink, ws->box, ws->nfirst,
                                                 ws->seg_off, ws->nseg, ws->mom64, ws->node_cap, (V4 *)ws->mom_a,
                                                 (V4 *)ws->mom_b, (V2 *)ws->mom_c);
    ws->launches += 3 + kMaxLevel;
    k_r5_flags<V4, Real><<<grid_for(ws->nseg, 256, 152), 256, 0, s>>>(ws->ctr, ws->box, (const V4 *)ws->mom_a, ws->nseg);
    ws->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_moments(TreeWorkspace *ws, cudaStream_t s) {
    if (ws->p.precision == TREE_F64) return moments_impl<double>(ws, s);
    return moments_impl<float>(ws, s);
}

}  // namespace treegb
