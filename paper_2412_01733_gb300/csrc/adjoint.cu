// adjoint.cu -- vector-Jacobian product of the tree force (Sec. 2 TreeCode,
// Eq. 1) with the tree structure of the last build held fixed: key order,
// cells, walk groups and the stored interaction lists.  Moments are
// functions of (x, m), so cell cotangents are carried back to the particles.
//
// Given cotangents abar (of the accelerations) and phibar (of the
// potentials), adds to xbar and mbar:
//   PP pair (source j, target i, d = r_j - r_i, s^2 = |d|^2 + eps^2):
//     g = G m_j (abar_i s^-3 - 3 d (d.abar_i) s^-5) + G m_j phibar_i d s^-3,
//     xbar_j += g, xbar_i -= g, mbar_j += G (d.abar_i) s^-3 - G phibar_i s^-1.
//   PC pair (cell C, y = r_i - R): derivative of the cell expansion with
//     respect to y (xbar_i += ybar, Rbar_C -= ybar), M and the six stored
//     quadrupole components.
//   Cell cotangents reach the particles of the cell: with d = r_j - R, Qf the
//     symmetric matrix of the stored-component cotangent (off-diagonals
//     halved) and f(d) = 3 d.Qf.d - |d|^2 tr Qf:
//       mbar_j += Mbar + d.Rbar / M + f(d),
//       xbar_j += m_j (Rbar / M + 6 Qf d - 2 tr(Qf) d);
//     a massless cell passes only Mbar (k_cot_paths).
// One warp per group walks the group's stored lists, 32 sources (cells or
// particles) at a time, one source per lane.  Each (target, source) pair is
// evaluated once: the source-side cotangents (cell or particle) are summed in
// the lane and added to global FP64 accumulators with one atomic per
// quantity per source per group; the target-side sums rotate through the
// lanes with the targets.
#include <type_traits>

#include "pairs.cuh"

namespace treegb {

constexpr int kAdjWarps = 4;
constexpr int kAdjMaxParts = 8;   // warps sharing a group's lists, at most

struct AdjArgs {
    int64_t n;
    int64_t ngroups;
    int32_t parts;         // warps per group: part p takes every parts-th tile of the lists
    const uint32_t *gfirst;
    const void *spos;      // Vec4 (x, y, z, m), key order
    const void *cot;       // Vec4 (abar, phibar), key order
    const uint2 *nlink;
    const void *mom_a, *mom_b, *mom_c;
    const int64_t *list_off;  // [2][ngroups + 1]
    const int32_t *pc_list, *pp_list;
    double eps2;
    double *xg;            // [3][n] xbar / G (atomics), key order
    double *mg;            // [n]    mbar / G (atomics), key order
    double *ccot;          // [10][cap] cell cotangents / G: Mbar, Rbar(3), Qbar(6)
    int64_t cap;
};

// One quantity of the targets a lane meets at a time: two in FP32 (packed
// instructions), one in FP64.
template <typename Real> struct Pack;
template <> struct Pack<float> {
    using V = float2;
    static constexpr int kW = 2;
    static __device__ __forceinline__ V dup(float a) { return make_float2(a, a); }
    static __device__ __forceinline__ V add(V a, V b) { return __fadd2_rn(a, b); }
    static __device__ __forceinline__ V mul(V a, V b) { return __fmul2_rn(a, b); }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
    static __device__ __forceinline__ V pick(bool ox, bool oy, V a) { return make_float2(ox ? 0.f : a.x, oy ? 0.f : a.y); }
    static __device__ __forceinline__ float total(V a) { return a.x + a.y; }
    template <bool SOFT> static __device__ __forceinline__ V rsqrt(V a) { return rsqrt_pair<SOFT>(a); }
    static __device__ __forceinline__ V shfl(V a, int src) {
        return make_float2(__shfl_sync(0xffffffffu, a.x, src), __shfl_sync(0xffffffffu, a.y, src));
    }
};
template <> struct Pack<double> {
    using V = double;
    static constexpr int kW = 1;
    static __device__ __forceinline__ V dup(double a) { return a; }
    static __device__ __forceinline__ V add(V a, V b) { return a + b; }
    static __device__ __forceinline__ V mul(V a, V b) { return a * b; }
    static __device__ __forceinline__ V fma(V a, V b, V c) { return ::fma(a, b, c); }
    static __device__ __forceinline__ V pick(bool ox, bool, V a) { return ox ? 0.0 : a; }
    static __device__ __forceinline__ double total(V a) { return a; }
    // r^2 = 0 contributes nothing, in the softened case too (eps^2 may underflow)
    template <bool SOFT> static __device__ __forceinline__ V rsqrt(V a) { return a > 0.0 ? ::rsqrt(a) : 0.0; }
    static __device__ __forceinline__ V shfl(V a, int src) { return __shfl_sync(0xffffffffu, a, src); }
};

// What a lane knows of its source (a cell, or a particle with no quadrupole).
template <typename Real>
struct AdjSource {
    typename Pack<Real>::V x, y, z, nm, q[6];  // position, -M, -Q (xx yy zz xy xz yz)
};

// Adds the derivatives of f = abar.a + phibar phi of (target, source) pairs to
// the source's sums and to the targets'.  With u = R - x, b = abar, p = phibar:
//   e = -(u.b)/r^2, k = -5/2 e - p/2, h = -(b/r^5 + k u/r^5)... in the signs that
// need no subtraction; -b, -p, -p/2 and -x are staged, -M and -Q held:
//   df/du = C u + D (-b) + 2 c (-Q u) - r^-5 Q b,
//     c = -k/r^5,  D = -M/r^3 - 5/2 (u.Q u)/r^7,
//     C = M/r^3 (3e + p) + 5/r^7 [(Q u).b - (u.Q u)(k - e)];
//   df/dM = -(u.(-b))/r^3 - p/r;   df/dQ_ij = -(u_i h_j + u_j h_i) (once on the
//     diagonal), h = b/r^5 (signs as staged) + c u.
// acc: 0, 1 the two parts of df/dM; 2-4 df/du; 5-10 -df/dQ.  85 operations for
// a cell with quadrupole, 29 without.  own: the pair leaves the source itself
// out (ox, oy: which of the lane's targets it is).
template <typename Real, bool QUAD, bool SOFT>
__device__ __forceinline__ void pair_vjp(const AdjSource<Real> &S, typename Pack<Real>::V nx, typename Pack<Real>::V ny,
                                         typename Pack<Real>::V nz, typename Pack<Real>::V bx,
                                         typename Pack<Real>::V by, typename Pack<Real>::V bz,
                                         typename Pack<Real>::V np, typename Pack<Real>::V eps2, bool own, bool ox,
                                         bool oy, typename Pack<Real>::V (&acc)[11], typename Pack<Real>::V (&t)[3]) {
    using P = Pack<Real>;
    using V = typename P::V;
    const V ux = P::add(S.x, nx), uy = P::add(S.y, ny), uz = P::add(S.z, nz);
    const V r2 = P::fma(ux, ux, P::fma(uy, uy, P::fma(uz, uz, eps2)));
    V i1 = P::template rsqrt<SOFT>(r2);
    if (own) i1 = P::pick(ox, oy, i1);
    const V i2 = P::mul(i1, i1);
    const V i3 = P::mul(i1, i2);
    const V ub = P::fma(ux, bx, P::fma(uy, by, P::mul(uz, bz)));  // u.(-b)
    const V e = P::mul(ub, i2);
    const V nmi3 = P::mul(S.nm, i3);
    const V s = P::fma(P::dup(Real(-3)), e, np);  // -(3e + p)
    V C = P::mul(nmi3, s), D = nmi3;
    acc[0] = P::fma(np, i1, acc[0]);
    acc[1] = P::fma(ub, i3, acc[1]);
    V gx, gy, gz;
    if (QUAD) {
        const V ni2 = P::mul(i2, P::dup(Real(-1)));
        const V ni5 = P::mul(i3, ni2);
        const V k5 = P::mul(ni5, P::mul(ni2, P::dup(Real(5))));  // 5 / r^7
        const V wx = P::fma(S.q[0], ux, P::fma(S.q[3], uy, P::mul(S.q[4], uz)));
        const V wy = P::fma(S.q[3], ux, P::fma(S.q[1], uy, P::mul(S.q[5], uz)));
        const V wz = P::fma(S.q[4], ux, P::fma(S.q[5], uy, P::mul(S.q[2], uz)));
        const V vx = P::fma(S.q[0], bx, P::fma(S.q[3], by, P::mul(S.q[4], bz)));
        const V vy = P::fma(S.q[3], bx, P::fma(S.q[1], by, P::mul(S.q[5], bz)));
        const V vz = P::fma(S.q[4], bx, P::fma(S.q[5], by, P::mul(S.q[2], bz)));
        const V uw = P::fma(ux, wx, P::fma(uy, wy, P::mul(uz, wz)));
        const V wb = P::fma(bx, wx, P::fma(by, wy, P::mul(bz, wz)));
        const V hp = P::mul(np, P::dup(Real(0.5)));               // -p/2
        const V k = P::fma(P::dup(Real(-2.5)), e, hp);
        const V d = P::fma(P::dup(Real(-3.5)), e, hp);
        const V uwk = P::mul(uw, k5);
        C = P::add(C, P::fma(uwk, d, P::mul(k5, wb)));
        D = P::fma(P::dup(Real(0.5)), uwk, D);
        const V c = P::mul(ni5, k), c2 = P::add(c, c);
        gx = P::fma(C, ux, P::fma(D, bx, P::fma(c2, wx, P::mul(ni5, vx))));
        gy = P::fma(C, uy, P::fma(D, by, P::fma(c2, wy, P::mul(ni5, vy))));
        gz = P::fma(C, uz, P::fma(D, bz, P::fma(c2, wz, P::mul(ni5, vz))));
        const V hx = P::fma(ni5, bx, P::mul(c, ux)), hy = P::fma(ni5, by, P::mul(c, uy)),
                hz = P::fma(ni5, bz, P::mul(c, uz));
        acc[5] = P::fma(ux, hx, acc[5]);
        acc[6] = P::fma(uy, hy, acc[6]);
        acc[7] = P::fma(uz, hz, acc[7]);
        acc[8] = P::fma(ux, hy, P::fma(uy, hx, acc[8]));
        acc[9] = P::fma(ux, hz, P::fma(uz, hx, acc[9]));
        acc[10] = P::fma(uy, hz, P::fma(uz, hy, acc[10]));
    } else {
        gx = P::fma(C, ux, P::mul(D, bx));
        gy = P::fma(C, uy, P::mul(D, by));
        gz = P::fma(C, uz, P::mul(D, bz));
    }
    acc[2] = P::add(acc[2], gx); acc[3] = P::add(acc[3], gy); acc[4] = P::add(acc[4], gz);
    t[0] = P::add(t[0], gx); t[1] = P::add(t[1], gy); t[2] = P::add(t[2], gz);
}

// A warp (one of A.parts sharing the group) walks its share of the group's
// stored lists, 32 sources at a time, one source per lane.  Bound by the FMA
// pipe; in FP32 a lane meets two targets at a time in packed instructions:
// targets j and j + 16 of a half of the group travel as a pair through
// sixteen lanes, the warp's two halves holding one copy of the targets' sums
// each.  Plummer sphere, N = 262144: 5.3 ms with one pair at a time, 2.9 in
// twos, 2.7 with two steps in flight and G left to the scatter (the FP64 pipe
// was 40 % busy with the totals); five blocks per SM (96 registers, spills)
// +3 %.  Up to kAdjMaxParts warps share a group where there are few groups:
// N = 65536 1.9 -> 0.63 ms.
template <typename Real, bool QUAD, bool SOFT>
__global__ void __launch_bounds__(kAdjWarps * 32, 4) k_force_vjp(const AdjArgs A) {
    using P = Pack<Real>;
    using V = typename P::V;
    using V4 = typename Vec4<Real>::T;
    using V2 = typename Vec2<Real>::T;
    constexpr int W = P::kW, L = 32 / W;  // targets met at a time, and steps to meet a half
    // per warp and half: -x, -y, -z, -bx, -by, -bz, -p of the targets, packed
    __shared__ V s_t[kAdjWarps][2][7][L];
    __shared__ uint32_t s_buf[kAdjWarps][32 + 32 * kMaxLeafSmall];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int next = (lane & ~(L - 1)) | ((lane + 1) & (L - 1));
    const int64_t item = (int64_t)blockIdx.x * kAdjWarps + w;
    const int64_t g = item / A.parts;
    const int part = (int)(item - g * A.parts);
    if (g >= A.ngroups) return;
    const V4 *spos = reinterpret_cast<const V4 *>(A.spos);
    const V4 *cot = reinterpret_cast<const V4 *>(A.cot);
    const V4 *momA = reinterpret_cast<const V4 *>(A.mom_a);
    const V4 *momB = reinterpret_cast<const V4 *>(A.mom_b);
    const V2 *momC = reinterpret_cast<const V2 *>(A.mom_c);
    const V eps2 = P::dup((Real)A.eps2);
    const uint32_t s0 = A.gfirst[g];
    const int cnt = (int)(A.gfirst[g + 1] - s0);
    const int halves = cnt > 32 ? 2 : 1;
    for (int t = lane; t < 32 * halves; t += 32) {
        // places past the group's end: its first particle without a cotangent, which adds nothing
        const V4 p = spos[s0 + (t < cnt ? t : 0)];
        V4 b{};
        if (t < cnt) b = cot[s0 + t];
        const int at = W * (t & (L - 1)) + ((t & 31) >= L ? 1 : 0);  // target j + 16 is the second of pair j
        Real *st = reinterpret_cast<Real *>(&s_t[w][t >> 5][0][0]);
        const Real v[7] = {-p.x, -p.y, -p.z, -b.x, -b.y, -b.z, -b.w};
#pragma unroll
        for (int c = 0; c < 7; ++c) st[c * 32 + at] = v[c];
    }
    __syncwarp();
    double xt[2][3] = {{0, 0, 0}, {0, 0, 0}};

    // All pairs of the lanes' sources with the group's targets: the source-side
    // sums stay in the lane, the targets' partial sums travel with them (one
    // shuffle per step passes each on to the lane that meets it next).  Lanes
    // without a source and places without a target take part with zero weights,
    // at the position of the tile's first source and of the group's first
    // particle: pairs that are there anyway, so a stand-in's powers of 1/r are
    // finite (and its terms zero) wherever theirs are.  At a distance of their
    // own they might not be: at r = 3e-6 a cell's 5/r^7 is past the FP32 range,
    // and 0 times it a NaN.  The self pair, which nothing else meets, is left
    // out for stand-ins too.
    auto meet = [&](const AdjSource<Real> &S, auto quad, bool own, uint32_t sj, V(&acc)[11]) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h >= halves) break;
            V t[3] = {P::dup(Real(0)), P::dup(Real(0)), P::dup(Real(0))};
            const V(*st)[L] = s_t[w][h];
            auto target = [&](int j) { return s0 + (uint32_t)(32 * h + j < cnt ? 32 * h + j : 0); };
#pragma unroll W
            for (int k = 0; k < L; ++k) {
                if (k > 0) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) t[c] = P::shfl(t[c], next);
                }
                const int j = (lane + k) & (L - 1);
                pair_vjp<Real, decltype(quad)::value, SOFT>(S, st[0][j], st[1][j], st[2][j], st[3][j], st[4][j],
                                                            st[5][j], st[6][j], eps2, own, target(j) == sj,
                                                            target(j + L) == sj, acc, t);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                t[c] = P::shfl(t[c], next);
                if constexpr (W == 2) {
                    // both halves of the warp hold a share of pair (lane & 15)
                    t[c] = P::add(t[c], P::shfl(t[c], lane ^ 16));
                    xt[h][c] += (double)(lane < 16 ? t[c].x : t[c].y);
                } else {
                    xt[h][c] += t[c];
                }
            }
        }
    };

    // ---- far cells ----
    const int64_t pc0 = A.list_off[g], pc1 = A.list_off[g + 1];
    for (int64_t base = pc0 + 32 * part; base < pc1; base += 32 * A.parts) {
        const int nt = (int)min((int64_t)32, pc1 - base);
        const uint32_t cid = (uint32_t)A.pc_list[base + (lane < nt ? lane : 0)];
        const V4 a = momA[cid];
        AdjSource<Real> S;
        S.x = P::dup(a.x); S.y = P::dup(a.y); S.z = P::dup(a.z); S.nm = P::dup(lane < nt ? -a.w : Real(0));
#pragma unroll
        for (int q = 0; q < 6; ++q) S.q[q] = P::dup(Real(0));
        if (QUAD && lane < nt) {
            const V4 b = momB[cid];
            const V2 c = momC[cid];
            const Real qs = sizeof(Real) == 4 ? Real(1) : Real(-1);  // the FP32 walk copies hold -Q
            S.q[0] = P::dup(qs * b.x); S.q[1] = P::dup(qs * b.y); S.q[2] = P::dup(qs * b.z);
            S.q[3] = P::dup(qs * b.w); S.q[4] = P::dup(qs * c.x); S.q[5] = P::dup(qs * c.y);
        }
        // the group's (at most 64) targets are summed in the working precision;
        // the per-group totals go to the FP64 accumulators (G comes with the scatter)
        V acc[11];
#pragma unroll
        for (int q = 0; q < 11; ++q) acc[q] = P::dup(Real(0));
        meet(S, std::bool_constant<QUAD>{}, false, 0u, acc);
        if (lane < nt) {
            const Real mb = P::total(acc[0]) - P::total(acc[1]);
            if (mb != Real(0)) atomicAdd(A.ccot + cid, (double)mb);
#pragma unroll
            for (int q = 2; q < (QUAD ? 11 : 5); ++q) {
                const Real v = P::total(acc[q]);
                if (v != Real(0)) atomicAdd(A.ccot + (int64_t)(q - 1) * A.cap + cid, (double)(q < 5 ? v : -v));
            }
        }
    }

    // ---- near leaves: expand particles into the buffer, tiles of 32 ----
    const int64_t pp0 = A.list_off[A.ngroups + 1 + g], pp1 = A.list_off[A.ngroups + 1 + g + 1];
    auto pp_tile = [&](uint32_t sj, int nt) {
        const uint32_t s1 = __shfl_sync(0xffffffffu, sj, 0);
        if (lane >= nt) sj = s1;
        const V4 a = spos[sj];
        AdjSource<Real> S;
        S.x = P::dup(a.x); S.y = P::dup(a.y); S.z = P::dup(a.z); S.nm = P::dup(lane < nt ? -a.w : Real(0));
        const bool own = __any_sync(0xffffffffu, sj - s0 < (uint32_t)cnt);
        V acc[11];
#pragma unroll
        for (int q = 0; q < 5; ++q) acc[q] = P::dup(Real(0));
        // the self pair is excluded by index
        if (own) meet(S, std::false_type{}, true, sj, acc);
        else meet(S, std::false_type{}, false, 0u, acc);
        if (lane < nt) {
            atomicAdd(A.xg + sj, (double)P::total(acc[2]));
            atomicAdd(A.xg + A.n + sj, (double)P::total(acc[3]));
            atomicAdd(A.xg + 2 * A.n + sj, (double)P::total(acc[4]));
            atomicAdd(A.mg + sj, (double)(P::total(acc[0]) - P::total(acc[1])));
        }
    };
    uint32_t *buf = s_buf[w];
    int nb = 0;
    for (int64_t base = pp0 + 32 * part; base < pp1; base += 32 * A.parts) {
        const int nl = (int)min((int64_t)32, pp1 - base);
        uint2 lk = make_uint2(0, 0);
        if (lane < nl) lk = A.nlink[(uint32_t)A.pp_list[base + lane]];
        const bool big = lk.y > (uint32_t)kMaxLeafSmall;
        const uint32_t sc = big ? 0u : lk.y;
        uint32_t incl = sc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t tot = __shfl_sync(0xffffffffu, incl, 31);
        for (uint32_t c = 0; c < sc; ++c) buf[nb + (incl - sc) + c] = lk.x + c;
        nb += (int)tot;
        __syncwarp();
        uint32_t bm = __ballot_sync(0xffffffffu, big);
        while (bm) {
            const int b = __ffs(bm) - 1;
            bm &= bm - 1;
            const uint32_t f = __shfl_sync(0xffffffffu, lk.x, b), c = __shfl_sync(0xffffffffu, lk.y, b);
            for (uint32_t o = 0; o < c; o += 32) pp_tile(f + o + (uint32_t)lane, (int)min(32u, c - o));
        }
        int done = 0;
        while (nb - done >= 32) {
            pp_tile(buf[done + lane], 32);
            done += 32;
        }
        const int r = nb - done;
        const uint32_t keep = lane < r ? buf[done + lane] : 0u;
        __syncwarp();
        if (lane < r) buf[lane] = keep;
        __syncwarp();
        nb = r;
    }
    if (nb > 0) pp_tile(lane < nb ? buf[lane] : 0u, nb);

    for (int h = 0; h < halves; ++h) {
        const int t = lane + 32 * h;
        if (t < cnt) {
#pragma unroll
            for (int c = 0; c < 3; ++c) atomicAdd(A.xg + c * A.n + s0 + t, -xt[h][c]);
        }
    }
}

// Cotangents (abar, phibar) from the caller's order into key order.
template <typename Real>
__global__ void __launch_bounds__(256) k_cot_gather(const Real *__restrict__ abar, const Real *__restrict__ phibar,
                                                    const uint32_t *__restrict__ perm, int64_t n,
                                                    typename Vec4<Real>::T *__restrict__ cot,
                                                    const uint32_t *__restrict__ ctr) {
    if (aborted(ctr, kStageAfter)) return;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t i = perm[s];
        typename Vec4<Real>::T c;
        c.x = abar[i]; c.y = abar[n + i]; c.z = abar[2 * n + i];
        c.w = phibar ? phibar[i] : Real(0);
        cot[s] = c;
    }
}

// Cell cotangents back to the particles.  What a cell's cotangents give a
// particle at r is a quadratic polynomial, with d = r - R:
//   P(d) = Mbar + d.Rbar / M + 3 d.Qf.d - |d|^2 tr Qf,
// P itself to mbar and m grad P to xbar (the chain of the moment tree, cell by
// cell, composes to just that, the moments being exact sums over the cell's
// particles).  A massless cell passes only Mbar on, so what is above one acts
// through its value at that cell's R.  So a leaf adds up the polynomials of
// its ancestors, shifted to its own R, in one launch without order (top-down,
// level by level, this was 22 launches and 0.83 ms at N = 262144), and leaves
// the sum in its own row: a; gx, gy, gz; hxx, hyy, hzz, hxy, hxz, hyz with
// P = a + g.d + d.h.d (h symmetric).
__global__ void __launch_bounds__(128) k_cot_paths(const uint32_t *__restrict__ ctr, const uint4 *__restrict__ ngeo,
                                                   const uint32_t *__restrict__ nparent,
                                                   const double *__restrict__ mom64, int64_t cap, int64_t nseg,
                                                   double *ccot) {
    if (aborted(ctr, kStageAfter)) return;
    const uint32_t nn = ctr[kCtrLevelStart + kLevels];
    for (uint32_t leaf = blockIdx.x * blockDim.x + threadIdx.x; leaf < nn; leaf += gridDim.x * blockDim.x) {
        if (!((ngeo[leaf].w >> 8) & 1u)) continue;
        const double *R = mom64 + cap;
        double px = R[leaf], py = R[cap + leaf], pz = R[2 * cap + leaf];  // where the sum is centred
        double a = 0, gx = 0, gy = 0, gz = 0, hxx = 0, hyy = 0, hzz = 0, hxy = 0, hxz = 0, hyz = 0;
        bool value = false;  // below a massless cell: only the value at its R counts
        for (uint32_t c = leaf;;) {
            const uint32_t up = nparent[c];
            double q[10];
            bool any = false;
#pragma unroll
            for (int k = 0; k < 10; ++k) {
                q[k] = ccot[(int64_t)k * cap + c];
                any |= q[k] != 0.0;
            }
            const double M = mom64[c];
            if (any) {
                a += q[0];
                if (M != 0.0) {
                    const double iM = 1.0 / M;
                    const double bx = q[1] * iM, by = q[2] * iM, bz = q[3] * iM;
                    const double tr = q[4] + q[5] + q[6];
                    const double sxx = 3.0 * q[4] - tr, syy = 3.0 * q[5] - tr, szz = 3.0 * q[6] - tr;
                    const double sxy = 1.5 * q[7], sxz = 1.5 * q[8], syz = 1.5 * q[9];
                    const double dx = px - R[c], dy = py - R[cap + c], dz = pz - R[2 * cap + c];
                    const double fx = sxx * dx + sxy * dy + sxz * dz, fy = sxy * dx + syy * dy + syz * dz,
                                 fz = sxz * dx + syz * dy + szz * dz;
                    a += dx * (bx + fx) + dy * (by + fy) + dz * (bz + fz);
                    if (!value) {
                        gx += bx + 2.0 * fx; gy += by + 2.0 * fy; gz += bz + 2.0 * fz;
                        hxx += sxx; hyy += syy; hzz += szz;
                        hxy += sxy; hxz += sxz; hyz += syz;
                    }
                }
            }
            if (M == 0.0) {
                value = true;
                px = R[c]; py = R[cap + c]; pz = R[2 * cap + c];
            }
            if (c < (uint32_t)nseg) break;
            c = up;
        }
        const double out[10] = {a, gx, gy, gz, hxx, hyy, hzz, hxy, hxz, hyz};
#pragma unroll
        for (int k = 0; k < 10; ++k) ccot[(int64_t)k * cap + leaf] = out[k];
    }
}

// xbar[i] += G (xg + m grad P), mbar[i] += G (mg + P) (key order -> caller order), P of
// the particle's leaf.
template <typename Real>
__global__ void __launch_bounds__(256) k_grad_scatter(const double *__restrict__ xg, const double *__restrict__ mg,
                                                      const double *__restrict__ ccot,
                                                      const double *__restrict__ mom64, int64_t cap,
                                                      const uint32_t *__restrict__ pleaf,
                                                      const typename Vec4<Real>::T *__restrict__ spos,
                                                      const uint32_t *__restrict__ perm, int64_t n, double G,
                                                      Real *__restrict__ xbar, Real *__restrict__ mbar,
                                                      const uint32_t *__restrict__ ctr) {
    if (aborted(ctr, kStageAfter)) return;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t i = perm[s], c = pleaf[s];
        const typename Vec4<Real>::T p = spos[s];
        double q[10];
#pragma unroll
        for (int k = 0; k < 10; ++k) q[k] = ccot[(int64_t)k * cap + c];
        const double dx = (double)p.x - mom64[cap + c], dy = (double)p.y - mom64[2 * cap + c],
                     dz = (double)p.z - mom64[3 * cap + c], m = (double)p.w;
        const double fx = q[4] * dx + q[7] * dy + q[8] * dz, fy = q[7] * dx + q[5] * dy + q[9] * dz,
                     fz = q[8] * dx + q[9] * dy + q[6] * dz;
        if (xbar) {
            xbar[i] += (Real)(G * (xg[s] + m * (q[1] + 2.0 * fx)));
            xbar[n + i] += (Real)(G * (xg[n + s] + m * (q[2] + 2.0 * fy)));
            xbar[2 * n + i] += (Real)(G * (xg[2 * n + s] + m * (q[3] + 2.0 * fz)));
        }
        if (mbar) mbar[i] += (Real)(G * (mg[s] + q[0] + dx * (q[1] + fx) + dy * (q[2] + fy) + dz * (q[3] + fz)));
    }
}

template <typename Real>
static cudaError_t adjoint_impl(TreeWorkspace *ws, const void *abar, const void *phibar, void *xbar, void *mbar,
                                cudaStream_t s) {
    const int64_t n = ws->n, cap = ws->node_cap;
    cudaError_t e;
    if ((e = cudaMemsetAsync(ws->adj_xg, 0, 3 * n * sizeof(double), s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ws->adj_mg, 0, n * sizeof(double), s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ws->adj_ccot, 0, 10 * cap * sizeof(double), s)) != cudaSuccess) return e;
    const int nb = grid_for(n, 256, 152 * 8);
    k_cot_gather<Real><<<nb, 256, 0, s>>>((const Real *)abar, (const Real *)phibar, ws->idx, n,
                                          (typename Vec4<Real>::T *)ws->adj_cot, ws->ctr);
    AdjArgs A;
    A.n = n;
    A.ngroups = ws->list_groups;
    A.gfirst = ws->gfirst;
    A.spos = ws->spos;
    A.cot = ws->adj_cot;
    A.nlink = ws->nlink;
    A.mom_a = ws->mom_a; A.mom_b = ws->mom_b; A.mom_c = ws->mom_c;
    A.list_off = ws->list_cnt;
    A.pc_list = ws->pc_list; A.pp_list = ws->pp_list;
    A.eps2 = ws->p.eps * ws->p.eps;
    A.xg = ws->adj_xg; A.mg = ws->adj_mg; A.ccot = ws->adj_ccot;
    A.cap = cap;
    // enough warps for several rounds of the chip also when there are few groups
    const int64_t want = 152 * 64;
    A.parts = A.ngroups > 0 ? (int)((want + A.ngroups - 1) / A.ngroups) : 1;
    if (A.parts > kAdjMaxParts) A.parts = kAdjMaxParts;
    const unsigned gb = (unsigned)((A.ngroups * A.parts + kAdjWarps - 1) / kAdjWarps);
    if (A.ngroups > 0) {
        const bool quad = ws->p.order == 2, soft = sizeof(Real) == 8 || walk_soft_f32(ws->p.eps);
        if (quad) {
            if (soft) k_force_vjp<Real, true, true><<<gb, kAdjWarps * 32, 0, s>>>(A);
            else k_force_vjp<Real, true, false><<<gb, kAdjWarps * 32, 0, s>>>(A);
        } else {
            if (soft) k_force_vjp<Real, false, true><<<gb, kAdjWarps * 32, 0, s>>>(A);
            else k_force_vjp<Real, false, false><<<gb, kAdjWarps * 32, 0, s>>>(A);
        }
    }
    k_cot_paths<<<grid_for(cap, 128, 152 * 16), 128, 0, s>>>(ws->ctr, ws->ngeo, ws->nparent, ws->mom64, cap, ws->nseg,
                                                              ws->adj_ccot);
    k_grad_scatter<Real><<<nb, 256, 0, s>>>(ws->adj_xg, ws->adj_mg, ws->adj_ccot, ws->mom64, cap, ws->pleaf,
                                            (const typename Vec4<Real>::T *)ws->spos, ws->idx, n, ws->p.G, (Real *)xbar,
                                            (Real *)mbar, ws->ctr);
    ws->launches += 4;
    return cudaGetLastError();
}

// One reverse step of Eqs. 2-5 (see leapfrog_adjoint_step in treegb.h).
template <typename Real>
__global__ void __launch_bounds__(256) k_adj_kick(Real *__restrict__ abar, const Real *__restrict__ vbar, Real h,
                                                  int64_t n3) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n3; i += (int64_t)gridDim.x * blockDim.x)
        abar[i] += h * vbar[i];
}
template <typename Real>
__global__ void __launch_bounds__(256) k_adj_drift(Real *__restrict__ abar, Real *__restrict__ vbar,
                                                   const Real *__restrict__ xbar, Real h, Real tau, int64_t n3) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n3; i += (int64_t)gridDim.x * blockDim.x) {
        const Real vb = vbar[i] + tau * xbar[i];
        vbar[i] = vb;
        abar[i] = h * vb;
    }
}

template <typename Real>
static cudaError_t adjoint_step_impl(TreeWorkspace *ws, Real *xbar, Real *vbar, Real *abar, Real *mbar,
                                     const Real *phibar, double tau, cudaStream_t s) {
    const int64_t n3 = 3 * ws->n;
    const int nb = grid_for(n3, 256, 152 * 8);
    k_adj_kick<Real><<<nb, 256, 0, s>>>(abar, vbar, (Real)(0.5 * tau), n3);
    cudaError_t e = adjoint_impl<Real>(ws, abar, phibar, xbar, mbar, s);
    if (e != cudaSuccess) return e;
    k_adj_drift<Real><<<nb, 256, 0, s>>>(abar, vbar, xbar, (Real)(0.5 * tau), (Real)tau, n3);
    ws->launches += 2;
    return cudaGetLastError();
}

cudaError_t launch_adjoint_step(TreeWorkspace *ws, void *xbar, void *vbar, void *abar, void *mbar,
                                const void *phibar, double tau, cudaStream_t s) {
    if (ws->p.precision == TREE_F64)
        return adjoint_step_impl<double>(ws, (double *)xbar, (double *)vbar, (double *)abar, (double *)mbar,
                                         (const double *)phibar, tau, s);
    return adjoint_step_impl<float>(ws, (float *)xbar, (float *)vbar, (float *)abar, (float *)mbar,
                                    (const float *)phibar, tau, s);
}

// Cotangents of W = 1/2 sum m phi (tree_energy_vjp): phi_bar = w_bar m / 2,
// m_bar += w_bar phi / 2.
template <typename Real>
__global__ void __launch_bounds__(256) k_energy_vjp(const Real *__restrict__ m, const Real *__restrict__ phi,
                                                    const double *__restrict__ wbar, int64_t n,
                                                    Real *__restrict__ phibar, Real *__restrict__ mbar) {
    const Real h = (Real)(0.5 * wbar[0]);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (phibar) phibar[i] = h * m[i];
        if (mbar) mbar[i] += h * phi[i];
    }
}

cudaError_t launch_energy_vjp(TreeWorkspace *ws, const void *m, const void *phi, const double *wbar, int64_t n,
                              void *phibar, void *mbar, cudaStream_t s) {
    const int nb = grid_for(n, 256, 152 * 8);
    if (ws->p.precision == TREE_F64)
        k_energy_vjp<double><<<nb, 256, 0, s>>>((const double *)m, (const double *)phi, wbar, n, (double *)phibar,
                                                (double *)mbar);
    else
        k_energy_vjp<float><<<nb, 256, 0, s>>>((const float *)m, (const float *)phi, wbar, n, (float *)phibar,
                                               (float *)mbar);
    ws->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_adjoint(TreeWorkspace *ws, const void *abar, const void *phibar, void *xbar, void *mbar,
                           cudaStream_t s) {
    if (ws->p.precision == TREE_F64) return adjoint_impl<double>(ws, abar, phibar, xbar, mbar, s);
    return adjoint_impl<float>(ws, abar, phibar, xbar, mbar, s);
}

}  // namespace treegb
