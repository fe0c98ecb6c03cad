// walk.cuh -- the tree walk and force evaluation (Sec. 2 TreeCode; Eq. 1 for
// the near part), one warp per group of Gs key-ordered particles.
//
// Small systems leave most of the chip idle in this form: a group is one
// warp's serial chain (at N = 30011 there are 989 groups for 3648 resident
// warps, and the group with the longest lists sets the time), and in FP64 one
// SM's pipe does 2 lanes a clock.  They take the split walk, three kernels:
// the traversal writes each group's tiles of 32 sources, in the order in which
// it would have evaluated them, into tile slots (kWalkTiles); every slot is
// then evaluated by whichever warp of the chip comes to it (k_eval_tiles); and
// the partial sums are folded, group by group, in the order of the tiles
// (kWalkFold).  Each tile's partial sums and the order of the folds are those
// of the one-warp walk, so the results are the same bits, alone or in an
// ensemble.  Force on a Plummer sphere, theta = 0.7, in ms (one-warp -> split,
// the moments then beside the traversal): FP32 N = 16384 0.455 -> 0.221, 65537
// 0.659 -> 0.558, 100000 0.749 -> 0.712, 131072 0.872 -> 0.919, 200000 1.21 ->
// 1.29 (1.25 KB of slot traffic per tile, and the traversal no longer hides
// behind the arithmetic: the two cross near 115000); FP64 16384 12.8 -> 2.7
// (walk alone), 65537 19.7 -> 12.9, 131072 29.7 -> 27.2, 200000 45.7 -> 43.8,
// 262144 58.6 -> 57.8, 400000 91.6 -> 93.0 (above 2^17 a few percent for twice
// the slots and more).  walk_splits() draws the lines, at 2^17 in both.
//
// Traversal (per warp, depth first, stack in shared memory):
//   the stack holds ranges of sibling nodes (children are contiguous in the
//   breadth-first numbering), one entry per opened cell.  Each step pops up
//   to 32 nodes from the top ranges (splitting the last one if needed), one
//   node per lane, and tests each against the group box with the integer
//   opening criterion d2 >= D[level] (D from tree_mac_table): far nodes go
//   to the PC buffer, near leaves' particles to the PP buffer, near internal
//   nodes push their child range.  Compaction uses warp ballots and scans.
// Evaluation: whenever a buffer holds 32 entries, the warp stages the 32
//   sources (float4 position+mass, or the cell's mass, COM and quadrupole)
//   in shared memory and every lane applies all 32 to its own target(s)
//   (each source is a broadcast shared-memory read; the arithmetic is plain
//   FP32 FMA plus one rsqrt per pair).  Per-tile partial sums are folded into
//   the running sums with Kahan compensation.
// The self pair i = j is excluded by index: a tile of near particles that
// holds some of the group's own particles is evaluated with the mass of each
// lane's own particle set to zero (removing -m_i/eps afterwards instead would
// cancel in FP32 against a potential that can be far smaller than m_i/eps);
// with eps = 0 a guarded variant also skips other r = 0 pairs.
#pragma once

#include "pairs.cuh"

namespace treegb {

constexpr int kWalkWarps = 4;                      // warps per block
constexpr int kPPCap = 32 + 32 * kMaxLeafSmall;    // PP buffer entries per warp
constexpr int kPCCap = 32 + 32 * 8;                // PC buffer entries per warp (a step adds <= 32 x 8)

struct WalkArgs {
    int64_t n;
    int32_t gs;
    int64_t ngroups;
    const void *spos;
    const uint64_t *skey;
    const uint32_t *perm;
    const uint4 *ngeo;
    const uint2 *nlink;
    const void *mom_a, *mom_b, *mom_c;
    const int64_t *dmac;
    double G, eps, eps2;
    void *a, *phi, *v;
    double half_tau;
    void *v2, *phi2;      // mirrors of the kicked v and of phi, or NULL
    int32_t stack_depth;
    uint4 *gstat;          // per group: {n_pc cells, n_pp particles, max stack, n_pp leaves}
    int32_t *dstatus;
    const int64_t *list_off;  // [2][ngroups+1] (emit mode)
    int32_t *pc_list, *pp_list;
    const uint32_t *order;    // processing order of the groups (widest boxes first), or NULL
    const uint32_t *gfirst;   // group g = sorted particles [gfirst[g], gfirst[g+1])
    uint32_t *ctr;            // counter block: group count and the walk's group ticket
    const int64_t *seg_off;   // segment offsets (nseg > 1): a group walks its own segment's tree
    int64_t nseg;
    const DevBox *box;        // per segment: the tree's cube (side 2^k)
    // split walk (kWalkTiles, k_eval_tiles, kWalkFold): tile slots and the groups' chains of them
    uint2 *tile_hdr;          // per slot: {group, sources | far cells << 8}; 0 sources: unused
    uint32_t *tile_idx;       // per slot: 32 source indices
    void *tile_part;          // per slot: Vec4 partial sums of 32 TPL targets
    uint32_t *tile_next;      // per chunk of kTileChunk slots: first slot of the group's next chunk
    uint32_t tile_cap;        // slots, a multiple of kTileChunk
    uint32_t *ghead, *gtiles; // per group: first slot; tiles, or kTilesFull
};

template <typename Real> __device__ __forceinline__ Real rsqrt_r(Real x);
template <> __device__ __forceinline__ float rsqrt_r<float>(float x) { return rsqrtf(x); }
template <> __device__ __forceinline__ double rsqrt_r<double>(double x) { return rsqrt(x); }

// Source staging per warp: FP32 uses 16 source pairs x 5 float4 (pair-
// interleaved, see pp_pair / pc_pair); FP64 uses 32 x (double4, double4, double2).
template <typename Real>
__host__ __device__ constexpr size_t walk_stage_bytes() {
    return sizeof(Real) == 4 ? 80 * sizeof(float4)
                             : 32 * (sizeof(typename Vec4<Real>::T) * 2 + sizeof(typename Vec2<Real>::T));
}

// Per-warp shared-memory slice, rounded up to 32 bytes so that every warp's
// staging arrays (float4 / 32-byte double4) stay aligned.
template <typename Real>
__host__ __device__ constexpr size_t walk_warp_bytes(int stack_depth) {
    return (((size_t)(stack_depth + kPPCap + kPCCap + 32) * 4 + walk_stage_bytes<Real>()) + 31) & ~(size_t)31;
}

// --- pair terms ------------------------------------------------------------
// PP: source s = (x, y, z, m); d = r_s - r_i; accumulates m d / r^3 and -m / r.
template <typename Real, bool SOFT>
__device__ __forceinline__ void pp_term(Real px, Real py, Real pz, const typename Vec4<Real>::T &s,
                                        Real eps2, Real (&acc)[4]) {
    const Real dx = s.x - px, dy = s.y - py, dz = s.z - pz;
    const Real r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2)));
    Real rinv = rsqrt_r<Real>(r2);
    if (!SOFT) rinv = r2 > Real(0) ? rinv : Real(0);
    const Real mr = s.w * rinv;
    const Real mr3 = mr * (rinv * rinv);
    acc[0] = fma(mr3, dx, acc[0]);
    acc[1] = fma(mr3, dy, acc[1]);
    acc[2] = fma(mr3, dz, acc[2]);
    acc[3] = fma(-s.w, rinv, acc[3]);  // explicit: every kernel rounds it alike
}

// PC: y = r_i - R, r_s^2 = |y|^2 + eps^2;
//   a += -M y / r_s^3 + Q y / r_s^5 - 5/2 (y.Q.y) y / r_s^7
//   phi += -M / r_s - 1/2 (y.Q.y) / r_s^5
// A = (Rx, Ry, Rz, M), B = (Qxx, Qyy, Qzz, Qxy), C = (Qxz, Qyz).
// R5 (quadrupole only): r^-5 taken out of the acceleration, as in pc_pair: with
// u = R - r_i, t = (u.Q.u)/r^4, k = r^2 (M + 5/2 t), a = r^-5 (k u - Q u) and
// phi = -(M + 1/2 t)/r; 32 operations and the rsqrt instead of 34 (FP64:
// 42.7 pipe slots a pair instead of 45.4).
template <typename Real, bool QUAD, bool SOFT, bool R5 = false>
__device__ __forceinline__ void pc_term(Real px, Real py, Real pz, const typename Vec4<Real>::T &A,
                                        const typename Vec4<Real>::T &B, const typename Vec2<Real>::T &C,
                                        Real eps2, Real (&acc)[4]) {
    if constexpr (QUAD && R5) {
        const Real ux = A.x - px, uy = A.y - py, uz = A.z - pz;
        const Real r2 = fma(ux, ux, fma(uy, uy, fma(uz, uz, eps2)));
        Real ri = rsqrt_r<Real>(r2);
        if (!SOFT) ri = r2 > Real(0) ? ri : Real(0);
        const Real ri2 = ri * ri, ri4 = ri2 * ri2, r5 = ri4 * ri;
        const Real wx = fma(B.x, ux, fma(B.w, uy, C.x * uz)), wy = fma(B.w, ux, fma(B.y, uy, C.y * uz)),
                   wz = fma(C.x, ux, fma(C.y, uy, B.z * uz));
        const Real t = fma(ux, wx, fma(uy, wy, uz * wz)) * ri4;
        const Real k = r2 * fma(Real(2.5), t, A.w);
        acc[0] = fma(r5, fma(k, ux, -wx), acc[0]);
        acc[1] = fma(r5, fma(k, uy, -wy), acc[1]);
        acc[2] = fma(r5, fma(k, uz, -wz), acc[2]);
        acc[3] = fma(-ri, fma(Real(0.5), t, A.w), acc[3]);
        return;
    }
    const Real yx = px - A.x, yy = py - A.y, yz = pz - A.z;
    const Real r2 = fma(yx, yx, fma(yy, yy, fma(yz, yz, eps2)));
    Real rinv = rsqrt_r<Real>(r2);
    if (!SOFT) rinv = r2 > Real(0) ? rinv : Real(0);
    const Real rinv2 = rinv * rinv;
    const Real Mr = A.w * rinv;
    const Real Mr3 = Mr * rinv2;
    if (QUAD) {
        const Real Qx = fma(B.x, yx, fma(B.w, yy, C.x * yz));
        const Real Qy = fma(B.w, yx, fma(B.y, yy, C.y * yz));
        const Real Qz = fma(C.x, yx, fma(C.y, yy, B.z * yz));
        const Real yQy = fma(yx, Qx, fma(yy, Qy, yz * Qz));
        const Real r3 = rinv * rinv2;
        const Real r5 = r3 * rinv2;
        const Real qr5 = yQy * r5;
        const Real c = fma(Real(-2.5) * qr5, rinv2, -Mr3);
        acc[0] = fma(c, yx, fma(r5, Qx, acc[0]));
        acc[1] = fma(c, yy, fma(r5, Qy, acc[1]));
        acc[2] = fma(c, yz, fma(r5, Qz, acc[2]));
        acc[3] -= fma(Real(0.5), qr5, Mr);
    } else {
        acc[0] = fma(-Mr3, yx, acc[0]);
        acc[1] = fma(-Mr3, yy, acc[1]);
        acc[2] = fma(-Mr3, yz, acc[2]);
        acc[3] = fma(-A.w, rinv, acc[3]);
    }
}

// Inclusive prefix of v < 2^B over the (full) warp and the warp's total.  A
// warp that is alone on its scheduler (BALLOTS: the split walk's traversal)
// waits less for B independent ballots than for five dependent shuffles; among
// many warps the shuffles cost less issue (large walk: ballots +0.5 %).
template <int B, bool BALLOTS>
__device__ __forceinline__ uint32_t warp_prefix(uint32_t v, int lane, uint32_t &total) {
    if constexpr (BALLOTS) {
        uint32_t ex = 0, tot = 0;
        const uint32_t lt = lanemask_lt();
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const uint32_t m = __ballot_sync(0xffffffffu, (v >> b) & 1u);
            ex += (uint32_t)__popc(m & lt) << b;
            tot += (uint32_t)__popc(m) << b;
        }
        total = tot;
        return ex + v;
    } else {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        total = __shfl_sync(0xffffffffu, v, 31);
        return v;
    }
}

// --- evaluation of one tile (whole warp) -----------------------------------
// A warp's targets: its group's particles, lane l holding l (and l + 32).
template <typename Real, int TPL>
struct Targets {
    Real px[TPL], py[TPL], pz[TPL];
    float2 nX[TPL], nY[TPL], nZ[TPL];  // negated and duplicated (packed FP32 terms)
    __device__ __forceinline__ void set_packed() {
#pragma unroll
        for (int t = 0; t < TPL; ++t) {
            nX[t] = make_float2(-(float)px[t], -(float)px[t]);
            nY[t] = make_float2(-(float)py[t], -(float)py[t]);
            nZ[t] = make_float2(-(float)pz[t], -(float)pz[t]);
        }
    }
};

// A warp's staging area.  FP32: sources are staged as pairs, pair k in
// F[5k .. 5k+4]:
//   PP: (x0, x1, y0, y1), (z0, z1, m0, m1)
//   PC: (Rx0, Rx1, Ry0, Ry1), (Rz0, Rz1, M0, M1), -(Qxx, Qyy), -(Qzz, Qxy), -(Qxz, Qyz)
// with an odd count padded by a massless source at the origin.  FP64: A, B, C
// one record per source.
template <typename Real>
struct Stage {
    float4 *F;
    typename Vec4<Real>::T *A, *B;
    typename Vec2<Real>::T *C;
    uint32_t *sidx;  // sorted index of each staged near source
    __device__ __forceinline__ Stage(unsigned char *wb, uint32_t *si) : sidx(si) {
        F = reinterpret_cast<float4 *>(wb);
        A = reinterpret_cast<typename Vec4<Real>::T *>(wb);
        B = A + 32;
        C = reinterpret_cast<typename Vec2<Real>::T *>(B + 32);
    }
};

// Stages ns near sources (lane l: src, sorted index si); true when some of
// them is one of the group's own particles [s0, s0 + cnt).
template <typename Real>
__device__ __forceinline__ bool stage_pp(const Stage<Real> &S, int lane, const typename Vec4<Real>::T &src,
                                         uint32_t si, int ns, uint32_t s0, int cnt) {
    S.sidx[lane] = lane < ns ? si : 0xffffffffu;
    const bool own = __any_sync(0xffffffffu, lane < ns && si - s0 < (uint32_t)cnt);
    if constexpr (sizeof(Real) == 4) {
        const int ne = (ns + 1) & ~1;
        if (lane < ne) {
            float *a = reinterpret_cast<float *>(S.F + 5 * (lane >> 1));
            const int sl = lane & 1;
            const bool v = lane < ns;
            a[sl] = v ? (float)src.x : 0.f;
            a[2 + sl] = v ? (float)src.y : 0.f;
            a[4 + sl] = v ? (float)src.z : 0.f;
            a[6 + sl] = v ? (float)src.w : 0.f;
        }
    } else {
        if (lane < ns) S.A[lane] = src;
    }
    return own;
}

// Partial sums of the staged near sources.  UNROLL: the full tile's loop.
template <typename Real, int TPL, bool SOFT, int UNROLL>
__device__ __forceinline__ void part_pp(const Stage<Real> &S, const Targets<Real, TPL> &T, int lane, int ns, bool own,
                                        uint32_t s0, Real eps2, float2 eps2v, Real (&p1)[TPL][4]) {
    using V4 = typename Vec4<Real>::T;
    if constexpr (sizeof(Real) == 4) {
        const float2 neg1 = make_float2(-1.f, -1.f);
        const float4 *stF = S.F;
        const uint32_t *sidx = S.sidx;
        float2 part[TPL][4];
#pragma unroll
        for (int t = 0; t < TPL; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) part[t][c] = make_float2(0.f, 0.f);
        const int np = (ns + 1) >> 1;
        if (own) {
            // the group's own particles are in this tile: each lane drops its own index
            for (int k = 0; k < np; ++k) {
                const float4 a = stF[5 * k], b = stF[5 * k + 1];
                const uint32_t i0 = sidx[2 * k], i1 = sidx[2 * k + 1];
#pragma unroll
                for (int t = 0; t < TPL; ++t) {
                    const uint32_t me = s0 + (uint32_t)(lane + 32 * t);
                    const float2 mm = make_float2(i0 == me ? 0.f : b.z, i1 == me ? 0.f : b.w);
                    pp_pair<SOFT>(T.nX[t], T.nY[t], T.nZ[t], make_float2(a.x, a.y), make_float2(a.z, a.w),
                                  make_float2(b.x, b.y), mm, eps2v, neg1, part[t]);
                }
            }
        } else if (np == 16) {
#pragma unroll UNROLL
            for (int k = 0; k < 16; ++k) {
                const float4 a = stF[5 * k], b = stF[5 * k + 1];
#pragma unroll
                for (int t = 0; t < TPL; ++t)
                    pp_pair<SOFT>(T.nX[t], T.nY[t], T.nZ[t], make_float2(a.x, a.y), make_float2(a.z, a.w),
                                  make_float2(b.x, b.y), make_float2(b.z, b.w), eps2v, neg1, part[t]);
            }
        } else {
            for (int k = 0; k < np; ++k) {
                const float4 a = stF[5 * k], b = stF[5 * k + 1];
#pragma unroll
                for (int t = 0; t < TPL; ++t)
                    pp_pair<SOFT>(T.nX[t], T.nY[t], T.nZ[t], make_float2(a.x, a.y), make_float2(a.z, a.w),
                                  make_float2(b.x, b.y), make_float2(b.z, b.w), eps2v, neg1, part[t]);
            }
        }
#pragma unroll
        for (int t = 0; t < TPL; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) p1[t][c] = (Real)(part[t][c].x + part[t][c].y);
    } else {
#pragma unroll
        for (int t = 0; t < TPL; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) p1[t][c] = Real(0);
        for (int j = 0; j < ns; ++j) {
            const V4 s = S.A[j];
            const uint32_t sj = S.sidx[j];
#pragma unroll
            for (int t = 0; t < TPL; ++t) {
                V4 st = s;
                if (own && sj == s0 + (uint32_t)(lane + 32 * t)) st.w = Real(0);
                pp_term<Real, SOFT>(T.px[t], T.py[t], T.pz[t], st, eps2, p1[t]);
            }
        }
    }
}

// Stages ns far cells (lane l: cell index `cell`).
template <typename Real, bool QUAD>
__device__ __forceinline__ void stage_pc(const Stage<Real> &S, int lane, uint32_t cell, int ns,
                                         const typename Vec4<Real>::T *__restrict__ momA,
                                         const typename Vec4<Real>::T *__restrict__ momB,
                                         const typename Vec2<Real>::T *__restrict__ momC) {
    using V4 = typename Vec4<Real>::T;
    using V2 = typename Vec2<Real>::T;
    if constexpr (sizeof(Real) == 4) {
        const int ne = (ns + 1) & ~1;
        if (lane < ne) {
            float *q = reinterpret_cast<float *>(S.F + 5 * (lane >> 1));
            const int sl = lane & 1;
            V4 a{};
            V4 b{};
            V2 c{};
            if (lane < ns) {
                a = momA[cell];
                if (QUAD) { b = momB[cell]; c = momC[cell]; }
            }
            q[sl] = a.x; q[2 + sl] = a.y; q[4 + sl] = a.z; q[6 + sl] = a.w;
            if (QUAD) {  // the FP32 cell copies already hold -Q
                q[8 + sl] = b.x; q[10 + sl] = b.y; q[12 + sl] = b.z; q[14 + sl] = b.w;
                q[16 + sl] = c.x; q[18 + sl] = c.y;
            }
        }
    } else {
        if (lane < ns) {
            S.A[lane] = momA[cell];
            if (QUAD) { S.B[lane] = momB[cell]; S.C[lane] = momC[cell]; }
        }
    }
}

// Partial sums of the staged far cells; r5: they take the r^-5 form (FP32: full tiles).
template <typename Real, int TPL, bool QUAD, bool SOFT, int UNROLL5, int UNROLL>
__device__ __forceinline__ void part_pc(const Stage<Real> &S, const Targets<Real, TPL> &T, int ns, bool r5, Real eps2,
                                        float2 eps2v, Real (&p1)[TPL][4]) {
    using V4 = typename Vec4<Real>::T;
    using V2 = typename Vec2<Real>::T;
    if constexpr (sizeof(Real) == 4) {
        const float2 neg1 = make_float2(-1.f, -1.f), halfv = make_float2(0.5f, 0.5f), m25 = make_float2(-2.5f, -2.5f),
                     mhalf = make_float2(-0.5f, -0.5f);
        const float4 *stF = S.F;
        float2 part[TPL][4];
#pragma unroll
        for (int t = 0; t < TPL; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) part[t][c] = make_float2(0.f, 0.f);
        const int np = (ns + 1) >> 1;
        const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
        const bool tile_r5 = np == 16 && r5;  // part[t][3] then holds -phi
        if (tile_r5) {
#pragma unroll UNROLL5
            for (int k = 0; k < 16; ++k) {
                const float4 a = stF[5 * k], b = stF[5 * k + 1];
                const float4 c = stF[5 * k + 2], d = stF[5 * k + 3], e = stF[5 * k + 4];
#pragma unroll
                for (int t = 0; t < TPL; ++t)
                    pc_pair<QUAD, SOFT, true>(T.nX[t], T.nY[t], T.nZ[t], a, b, c, d, e, eps2v, mhalf, halfv, m25,
                                              part[t]);
            }
        } else if (np == 16) {
#pragma unroll UNROLL
            for (int k = 0; k < 16; ++k) {
                const float4 a = stF[5 * k], b = stF[5 * k + 1];
                const float4 c = QUAD ? stF[5 * k + 2] : z4, d = QUAD ? stF[5 * k + 3] : z4,
                             e = QUAD ? stF[5 * k + 4] : z4;
#pragma unroll
                for (int t = 0; t < TPL; ++t)
                    pc_pair<QUAD, SOFT>(T.nX[t], T.nY[t], T.nZ[t], a, b, c, d, e, eps2v, neg1, halfv, m25, part[t]);
            }
        } else {
            for (int k = 0; k < np; ++k) {
                const float4 a = stF[5 * k], b = stF[5 * k + 1];
                const float4 c = QUAD ? stF[5 * k + 2] : z4, d = QUAD ? stF[5 * k + 3] : z4,
                             e = QUAD ? stF[5 * k + 4] : z4;
#pragma unroll
                for (int t = 0; t < TPL; ++t)
                    pc_pair<QUAD, SOFT>(T.nX[t], T.nY[t], T.nZ[t], a, b, c, d, e, eps2v, neg1, halfv, m25, part[t]);
            }
        }
#pragma unroll
        for (int t = 0; t < TPL; ++t) {
#pragma unroll
            for (int c = 0; c < 4; ++c) p1[t][c] = (Real)(part[t][c].x + part[t][c].y);
            if (tile_r5) p1[t][3] = -p1[t][3];
        }
    } else {
#pragma unroll
        for (int t = 0; t < TPL; ++t)
#pragma unroll
            for (int c = 0; c < 4; ++c) p1[t][c] = Real(0);
        V4 b0{};
        V2 c0{};
        if (QUAD && r5) {
            for (int j = 0; j < ns; ++j) {
                const V4 a = S.A[j], b = S.B[j];
                const V2 c = S.C[j];
#pragma unroll
                for (int t = 0; t < TPL; ++t)
                    pc_term<Real, QUAD, SOFT, true>(T.px[t], T.py[t], T.pz[t], a, b, c, eps2, p1[t]);
            }
        } else {
            for (int j = 0; j < ns; ++j) {
                const V4 a = S.A[j];
                const V4 b = QUAD ? S.B[j] : b0;
                const V2 c = QUAD ? S.C[j] : c0;
#pragma unroll
                for (int t = 0; t < TPL; ++t)
                    pc_term<Real, QUAD, SOFT>(T.px[t], T.py[t], T.pz[t], a, b, c, eps2, p1[t]);
            }
        }
    }
}

// Resident blocks per SM the registers are held to.  FP32: 5 (96 registers, no
// spills): galaxy of 1e7 41.8 ms against 42.0 at 6 blocks (80) and 42.4 at 4,
// Plummer 2^20 at theta = 0.5 7.25 against 7.33 and 7.27.  kWalkFold keeps two
// batches of partial sums in registers (the fold of the longest group is a
// chain of loads: 65 us at N = 16384 with one batch that spilled, 20 with two
// that fit) and runs few groups: 3 blocks.
constexpr int walk_blocks(int mode, int tpl) {
    return mode == kWalkFold ? 3 : tpl == 2 ? 4 : 5;
}

template <typename Real, int TPL, bool QUAD, bool KAHAN, bool SOFT, int MODE>
__global__ void __launch_bounds__(kWalkWarps * 32, walk_blocks(MODE, TPL)) k_walk(const WalkArgs A) {
    using V4 = typename Vec4<Real>::T;
    using V2 = typename Vec2<Real>::T;
    extern __shared__ __align__(32) unsigned char smem[];
    __shared__ long long sD[kLevels];
    if (aborted(A.ctr, kStageAfter)) return;  // the build gave up a wait: no valid tree
    if (threadIdx.x < kLevels) sD[threadIdx.x] = A.dmac[threadIdx.x];
    __syncthreads();

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int SD = A.stack_depth;
    unsigned char *wb = smem + (size_t)warp * walk_warp_bytes<Real>(SD);
    uint32_t *stack = reinterpret_cast<uint32_t *>(wb + walk_stage_bytes<Real>());
    uint32_t *ppbuf = stack + SD;
    uint32_t *pcbuf = ppbuf + kPPCap;
    const Stage<Real> S(wb, pcbuf + kPCCap);
    const uint32_t lt = lanemask_lt();

    const V4 *__restrict__ spos = reinterpret_cast<const V4 *>(A.spos);
    const V4 *__restrict__ momA = reinterpret_cast<const V4 *>(A.mom_a);
    const V4 *__restrict__ momB = reinterpret_cast<const V4 *>(A.mom_b);
    const V2 *__restrict__ momC = reinterpret_cast<const V2 *>(A.mom_c);
    const Real eps2 = (Real)A.eps2;

    // far cells take the R5 form where it fits the segment's cube (flag set per
    // segment after the moments); in FP32, full tiles of one-target-per-lane groups
    constexpr bool kR5 = QUAD && (sizeof(Real) == 8 || TPL == 1);
    // tiles are filled and consumed (evaluated or emitted)
    constexpr bool kTiles = MODE == kWalkForce || MODE == kWalkFold || MODE == kWalkTiles;
    // few warps, each with its scheduler to itself: shorter chains of instructions before fewer of them
    // (the list walks serve gradients, at sizes where that holds too)
    constexpr bool kAlone = MODE == kWalkTiles || MODE == kWalkCount || MODE == kWalkEmit;

    // persistent warps: each takes the next group slot until all are done
    const uint32_t ngroups = A.ctr[kCtrGroups];
    for (;;) {
    uint32_t slot = 0;
    if (lane == 0) slot = atomicAdd(A.ctr + kCtrWalkTicket, 1u);
    slot = __shfl_sync(0xffffffffu, slot, 0);
    if (slot >= ngroups) break;
    const int64_t g = A.order ? (int64_t)A.order[slot] : (int64_t)slot;
    const int64_t s0 = A.gfirst[g];
    const int cnt = (int)(A.gfirst[g + 1] - A.gfirst[g]);
    // the group's segment b (its tree's root is node b)
    const uint32_t gseg = A.nseg > 1 ? seg_find(A.seg_off, A.nseg, s0) : 0u;

    // targets and the group's integer box
    Targets<Real, TPL> T;
    uint32_t lo0 = 0xffffffffu, lo1 = 0xffffffffu, lo2 = 0xffffffffu, hi0 = 0, hi1 = 0, hi2 = 0;
#pragma unroll
    for (int t = 0; t < TPL; ++t) {
        const int li = lane + 32 * t;
        T.px[t] = T.py[t] = T.pz[t] = Real(0);
        if (li < cnt) {
            const V4 p = spos[s0 + li];
            T.px[t] = p.x; T.py[t] = p.y; T.pz[t] = p.z;
            const uint64_t k = A.skey[s0 + li];
            const uint32_t qx = compact3(k >> 2), qy = compact3(k >> 1), qz = compact3(k);
            lo0 = min(lo0, qx); lo1 = min(lo1, qy); lo2 = min(lo2, qz);
            hi0 = max(hi0, qx); hi1 = max(hi1, qy); hi2 = max(hi2, qz);
        }
    }
    const int glo0 = (int)__reduce_min_sync(0xffffffffu, lo0), glo1 = (int)__reduce_min_sync(0xffffffffu, lo1),
              glo2 = (int)__reduce_min_sync(0xffffffffu, lo2);
    const int ghi0 = (int)__reduce_max_sync(0xffffffffu, hi0) + 1, ghi1 = (int)__reduce_max_sync(0xffffffffu, hi1) + 1,
              ghi2 = (int)__reduce_max_sync(0xffffffffu, hi2) + 1;

    Real sum[TPL][4], cmp[TPL][4];
#pragma unroll
    for (int t = 0; t < TPL; ++t)
#pragma unroll
        for (int c = 0; c < 4; ++c) { sum[t][c] = Real(0); cmp[t][c] = Real(0); }

    T.set_packed();
    const float2 eps2v = make_float2((float)A.eps2, (float)A.eps2);
    const bool r5 = kR5 && A.box[gseg].r5fit != 0;

    // --- evaluation (whole warp) ---
    auto fold_tile = [&](const Real(&p1)[TPL][4]) {
#pragma unroll
        for (int t = 0; t < TPL; ++t) fold<Real, KAHAN>(sum[t], cmp[t], p1[t]);
    };
    auto eval_pp = [&](uint32_t si, int ns) {
        V4 s{};
        if (lane < ns) s = spos[si];
        __syncwarp();
        const bool own = stage_pp<Real>(S, lane, s, si, ns, (uint32_t)s0, cnt);
        __syncwarp();
        Real p1[TPL][4];
        part_pp<Real, TPL, SOFT, 16>(S, T, lane, ns, own, (uint32_t)s0, eps2, eps2v, p1);
        fold_tile(p1);
        __syncwarp();
    };
    auto eval_pc = [&](const uint32_t *buf, int ns) {
        stage_pc<Real, QUAD>(S, lane, lane < ns ? buf[lane] : 0u, ns, momA, momB, momC);
        __syncwarp();
        Real p1[TPL][4];
        part_pc<Real, TPL, QUAD, SOFT, 16, 4>(S, T, ns, r5, eps2, eps2v, p1);
        fold_tile(p1);
        __syncwarp();
    };
    // --- split walk: the same tiles, in the same order, into tile slots ---
    // (a chunk is asked for half a chunk before it is needed, so that the
    // atomic's latency passes behind the tiles in between)
    uint32_t ntile = 0, tbase = 0, tnext = 0;
    bool full = false;  // out of slots: kWalkFold walks this group itself
    if (MODE == kWalkTiles && lane == 0) tnext = atomicAdd(A.ctr + kCtrTiles, (uint32_t)kTileChunk);
    // room for the next tile's chunk; false when the slots have run out
    auto open_chunk = [&]() {
        const uint32_t base = __shfl_sync(0xffffffffu, tnext, 0);
        if (base > A.tile_cap - kTileChunk) { full = true; return; }
        if (lane == 0) {
            if (ntile == 0) A.ghead[g] = base;
            else A.tile_next[tbase / kTileChunk] = base;
        }
        tbase = base;
    };
    auto emit_tile = [&](uint32_t src, int ns, uint32_t far) {
        if (full) return;
        const uint32_t k = ntile & (kTileChunk - 1);
        if (k == 0) open_chunk();
        if (full) return;
        if (k == kTileChunk / 2 && lane == 0) tnext = atomicAdd(A.ctr + kCtrTiles, (uint32_t)kTileChunk);
        const uint32_t slot = tbase + k;
        if (lane == 0) A.tile_hdr[slot] = make_uint2((uint32_t)g, (uint32_t)ns | (far << 8));
        A.tile_idx[(size_t)slot * 32 + lane] = lane < ns ? src : 0u;
        ++ntile;
    };
    // `count` full tiles from a buffer: as many at a time as their chunk holds
    auto emit_tiles = [&](const uint32_t *buf, int count, uint32_t far) {
        while (count > 0 && !full) {
            const uint32_t k = ntile & (kTileChunk - 1);
            if (k == 0) open_chunk();
            if (full) return;
            const int m = min(count, (int)(kTileChunk - k));
            if (k <= kTileChunk / 2 && k + m > kTileChunk / 2 && lane == 0)
                tnext = atomicAdd(A.ctr + kCtrTiles, (uint32_t)kTileChunk);
            const uint32_t slot = tbase + k;
            if (lane < m) A.tile_hdr[slot + lane] = make_uint2((uint32_t)g, 32u | (far << 8));
            uint32_t *dst = A.tile_idx + (size_t)slot * 32 + lane;
#pragma unroll 4
            for (int t = 0; t < m; ++t) dst[32 * t] = buf[32 * t + lane];
            buf += 32 * m;
            ntile += (uint32_t)m;
            count -= m;
        }
    };
    auto pc_tile = [&](const uint32_t *buf, int ns) {
        if (MODE == kWalkTiles) emit_tile(lane < ns ? buf[lane] : 0u, ns, 1u);
        else eval_pc(buf, ns);
    };
    auto pp_tile = [&](uint32_t si, int ns) {
        if (MODE == kWalkTiles) emit_tile(si, ns, 0u);
        else eval_pp(si, ns);
    };

    // --- traversal ---
    int64_t pc_base = 0, pp_base = 0;
    if (MODE == kWalkEmit) {
        pc_base = A.list_off[g];
        pp_base = A.list_off[A.ngroups + 1 + g];
    }
    uint32_t n_pc = 0, n_pp = 0, n_ppl = 0, max_top = 1;
    int top = 1, npc = 0, npp = 0;
    bool folded = false;
    if (MODE == kWalkFold) {
        // the group's tiles have been evaluated: fold their partial sums in the
        // order in which the one-warp walk would have evaluated them
        const uint32_t nt = A.gtiles[g];
        folded = nt != kTilesFull;
        if (folded) {
            const V4 *__restrict__ tp = reinterpret_cast<const V4 *>(A.tile_part);
            // two batches of 32 registers: one is folded while the next is loaded
            constexpr int kB = 128 / (int)(sizeof(V4) * TPL);
            static_assert(kTileChunk % kB == 0, "a batch stays inside one chunk");
            V4 q[kB][TPL], r[kB][TPL];
            uint32_t base = nt ? A.ghead[g] : 0u;
            uint32_t next = nt > kTileChunk ? A.tile_next[base / kTileChunk] : 0u;
            auto load = [&](V4(&d)[kB][TPL], uint32_t b) {
                if (b >= nt) return;
                if (b != 0 && (b & (kTileChunk - 1)) == 0) {
                    base = next;
                    next = b + kTileChunk < nt ? A.tile_next[base / kTileChunk] : 0u;
                }
#pragma unroll
                for (int k = 0; k < kB; ++k)
#pragma unroll
                    for (int t = 0; t < TPL; ++t)
                        if (b + k < nt) d[k][t] = tp[((size_t)(base + (b & (kTileChunk - 1)) + k) * TPL + t) * 32 + lane];
            };
            auto fold_batch = [&](const V4(&d)[kB][TPL], uint32_t b) {
#pragma unroll
                for (int k = 0; k < kB; ++k) {
                    if (b + k >= nt) break;
                    Real p1[TPL][4];
#pragma unroll
                    for (int t = 0; t < TPL; ++t) {
                        p1[t][0] = d[k][t].x; p1[t][1] = d[k][t].y;
                        p1[t][2] = d[k][t].z; p1[t][3] = d[k][t].w;
                    }
                    fold_tile(p1);
                }
            };
            load(q, 0);
#pragma unroll 1
            for (uint32_t b = 0; b < nt; b += 2 * kB) {
                load(r, b + kB);
                fold_batch(q, b);
                load(q, b + 2 * kB);
                fold_batch(r, b + kB);
            }
            top = 0;  // nothing left to walk
        }
    }
    // Stack entries are child ranges: first node | (count - 1) << 29.
    // the root of the group's segment (node b at level 0): range (node b, 1 node)
    if (lane == 0) stack[0] = gseg;
    __syncwarp();
    bool overflow = false;
    while (top > 0 && !(MODE == kWalkTiles && full)) {
        // pop up to 32 nodes from the top ranges; the last range may be split
        const int nr = top < 32 ? top : 32;
        uint32_t e = 0, sz = 0;
        if (lane < nr) {
            e = stack[top - 1 - lane];
            sz = (e >> 29) + 1u;
        }
        uint32_t avail;
        const uint32_t incl0 = warp_prefix<4, kAlone>(sz, lane, avail);
        const uint32_t excl0 = incl0 - sz;
        const uint32_t take = avail < 32u ? avail : 32u;
        const bool contrib = lane < nr && excl0 < take;
        const int nfull = __popc(__ballot_sync(0xffffffffu, lane < nr && incl0 <= take));
        // the contributing ranges are lanes 0..k-1 with increasing starts excl0:
        // lane t belongs to the last one whose start is <= t
        const uint32_t starts = __reduce_or_sync(0xffffffffu, contrib ? (1u << excl0) : 0u);
        const int owner = __popc(starts & (lt | (1u << lane))) - 1;
        const uint32_t e_own = __shfl_sync(0xffffffffu, e, owner & 31);
        const uint32_t x_own = __shfl_sync(0xffffffffu, excl0, owner & 31);
        const bool act = (uint32_t)lane < take;
        const uint32_t node = act ? (e_own & 0x1fffffffu) + ((uint32_t)lane - x_own) : 0u;
        if (contrib && incl0 > take) {
            // partially used range (lane == nfull): keep its unused tail on the stack
            const uint32_t used = take - excl0;
            stack[top - 1 - lane] = ((e & 0x1fffffffu) + used) | ((sz - used - 1u) << 29);
        }
        top -= nfull;
        __syncwarp();
        uint4 geo = make_uint4(0, 0, 0, 0);
        uint2 lk = make_uint2(0, 0);
        if (act) { geo = A.ngeo[node]; lk = A.nlink[node]; }
        const int level = (int)(geo.w & 0xffu);
        const bool leaf = (geo.w >> 8) & 1u;
        const int s = 1 << (kBits - level);
        const int cx = (int)geo.x, cy = (int)geo.y, cz = (int)geo.z;
        const int gx = max(0, max(cx - ghi0, glo0 - (cx + s)));
        const int gy = max(0, max(cy - ghi1, glo1 - (cy + s)));
        const int gz = max(0, max(cz - ghi2, glo2 - (cz + s)));
        const long long d2 = (long long)gx * gx + (long long)gy * gy + (long long)gz * gz;
        const bool far = act && d2 >= sD[level];
        const bool nleaf = act && !far && leaf;
        const bool open = act && !far && !leaf;
        // A child's box lies inside its parent's, so it is at least as far from
        // the group: when an opened cell already meets its children's threshold
        // (d2 >= D[level + 1]), all its children are far and go to the far list
        // without being popped and tested one by one.
        const bool allfar = open && d2 >= sD[min(level + 1, kMaxLevel)];

        // far cells
        const uint32_t fm = __ballot_sync(0xffffffffu, far);
        const uint32_t nf = __popc(fm);
        if (kTiles) {
            if (far) pcbuf[npc + __popc(fm & lt)] = node;
            npc += nf;
        } else if (MODE == kWalkEmit) {
            if (far) A.pc_list[pc_base + n_pc + __popc(fm & lt)] = (int32_t)node;
        }
        n_pc += nf;
        const uint32_t am = __ballot_sync(0xffffffffu, allfar);
        if (am) {
            const uint32_t cc = allfar ? lk.y : 0u;
            uint32_t tot;
            const uint32_t incl = warp_prefix<4, kAlone>(cc, lane, tot);
            if (kTiles) {
                uint32_t *dst = pcbuf + npc + (incl - cc);
                if constexpr (kAlone) {
#pragma unroll
                    for (uint32_t c = 0; c < 8; ++c)
                        if (c < cc) dst[c] = lk.x + c;
                } else {
                    if (allfar)
                        for (uint32_t c = 0; c < cc; ++c) dst[c] = lk.x + c;
                }
                npc += (int)tot;
            } else if (MODE == kWalkEmit) {
                int32_t *dst = A.pc_list + pc_base + n_pc + (incl - cc);
#pragma unroll
                for (uint32_t c = 0; c < 8; ++c)
                    if (c < cc) dst[c] = (int32_t)(lk.x + c);
            }
            n_pc += tot;
        }

        // children of the other opened cells: one stack entry per opened cell
        const bool push = open && !allfar;
        const uint32_t om = __ballot_sync(0xffffffffu, push);
        if (om) {
            const int no = __popc(om);
            if (top + no > SD) {
                overflow = true;
            } else {
                if (push) stack[top + __popc(om & lt)] = lk.x | ((lk.y - 1u) << 29);
                top += no;
            }
            max_top = max(max_top, (uint32_t)top);
        }

        // near leaves (most steps of a deep walk have none)
        const uint32_t lm = __ballot_sync(0xffffffffu, nleaf);
        if (lm) {
            if (MODE == kWalkEmit) {
                if (nleaf) A.pp_list[pp_base + n_ppl + __popc(lm & lt)] = (int32_t)node;
            }
            n_ppl += __popc(lm);
            const uint32_t lc = nleaf ? lk.y : 0u;
            const bool big = lc > (uint32_t)kMaxLeafSmall;
            const uint32_t sc = big ? 0u : lc;
            uint32_t tot2;
            const uint32_t incl2 = warp_prefix<5, kAlone>(sc, lane, tot2);
            n_pp += __reduce_add_sync(0xffffffffu, lc);
            if (kTiles) {
                uint32_t *dst = ppbuf + npp + (incl2 - sc);
                if constexpr (kAlone) {
#pragma unroll
                    for (uint32_t c = 0; c < (uint32_t)kMaxLeafSmall; ++c)
                        if (c < sc) dst[c] = lk.x + c;
                } else {
                    if (nleaf && !big)
                        for (uint32_t c = 0; c < lc; ++c) dst[c] = lk.x + c;
                }
                npp += (int)tot2;
                __syncwarp();
                uint32_t bm = __ballot_sync(0xffffffffu, big);
                while (bm) {
                    const int b = __ffs(bm) - 1;
                    bm &= bm - 1;
                    const uint32_t f = __shfl_sync(0xffffffffu, lk.x, b);
                    const uint32_t c = __shfl_sync(0xffffffffu, lk.y, b);
                    for (uint32_t o = 0; o < c; o += 32) pp_tile(f + o + (uint32_t)lane, (int)min(32u, c - o));
                }
            }
        }
        if (kTiles) {
            if (npc >= 32) {
                __syncwarp();
                const int nfull = npc >> 5;
                if (MODE == kWalkTiles) emit_tiles(pcbuf, nfull, 1u);
                else
                    for (int t = 0; t < nfull; ++t) pc_tile(pcbuf + 32 * t, 32);
                const int r = npc & 31;
                uint32_t t = lane < r ? pcbuf[32 * nfull + lane] : 0;
                __syncwarp();
                if (lane < r) pcbuf[lane] = t;
                __syncwarp();
                npc = r;
            }
            if (npp >= 32) {
                const int nfull = npp >> 5;
                if (MODE == kWalkTiles) emit_tiles(ppbuf, nfull, 0u);
                else
                    for (int t = 0; t < nfull; ++t) pp_tile(ppbuf[32 * t + lane], 32);
                const int r = npp & 31;
                uint32_t t = lane < r ? ppbuf[32 * nfull + lane] : 0;
                __syncwarp();
                if (lane < r) ppbuf[lane] = t;
                __syncwarp();
                npp = r;
            }
        } else {
            __syncwarp();
        }
    }
    if (kTiles) {
        // every traversal step evaluates the whole tiles, so fewer than 32
        // entries are left here: the staging holds at most 32 sources
        if (npc > 0) pc_tile(pcbuf, npc);
        if (npp > 0) pp_tile(lane < npp ? ppbuf[lane] : 0xffffffffu, npp);
    }
    if (MODE == kWalkTiles) {
        if (lane == 0) A.gtiles[g] = full ? kTilesFull : ntile;
        // unused slots hold no sources: the rest of the last chunk, and a chunk asked for but not begun
        const uint32_t used = ntile & (kTileChunk - 1);
        const uint32_t ahead = __shfl_sync(0xffffffffu, tnext, 0);
        if (used && lane >= (int)used && lane < kTileChunk) A.tile_hdr[tbase + lane] = make_uint2(0u, 0u);
        if ((ntile == 0 || used == 0 || used > kTileChunk / 2) && ahead <= A.tile_cap - kTileChunk && lane < kTileChunk)
            A.tile_hdr[ahead + lane] = make_uint2(0u, 0u);
    }
    if (overflow && lane == 0) set_status(A.dstatus, TREE_DEV_STACK);
    if (lane == 0 && A.gstat && !folded) A.gstat[g] = make_uint4(n_pc, n_pp, max_top, n_ppl);

    if (MODE == kWalkForce || MODE == kWalkFold) {
        const Real G = (Real)A.G;
#pragma unroll
        for (int t = 0; t < TPL; ++t) {
            const int li = lane + 32 * t;
            if (li < cnt) {
                const uint32_t i = A.perm[s0 + li];
                Real ax, ay, az, ph;
                if (KAHAN) {
                    ax = sum[t][0] - cmp[t][0]; ay = sum[t][1] - cmp[t][1];
                    az = sum[t][2] - cmp[t][2]; ph = sum[t][3] - cmp[t][3];
                } else {
                    ax = sum[t][0]; ay = sum[t][1]; az = sum[t][2]; ph = sum[t][3];
                }
                ax *= G; ay *= G; az *= G; ph *= G;
                Real *a = reinterpret_cast<Real *>(A.a);
                const int64_t n = A.n;
                a[i] = ax; a[n + i] = ay; a[2 * n + i] = az;
                if (A.phi) reinterpret_cast<Real *>(A.phi)[i] = ph;
                if (A.phi2) reinterpret_cast<Real *>(A.phi2)[i] = ph;
                if (A.v) {
                    Real *v = reinterpret_cast<Real *>(A.v);
                    const Real ht = (Real)A.half_tau;
                    const Real vx = fma(ht, ax, v[i]), vy = fma(ht, ay, v[n + i]), vz = fma(ht, az, v[2 * n + i]);
                    v[i] = vx; v[n + i] = vy; v[2 * n + i] = vz;
                    if (A.v2) {
                        Real *w = reinterpret_cast<Real *>(A.v2);
                        w[i] = vx; w[n + i] = vy; w[2 * n + i] = vz;
                    }
                }
            }
        }
    }
    }  // group loop
}

// Split walk, second kernel: one warp per tile slot stages and evaluates the
// slot's 32 sources for its group's targets and stores the partial sums.
template <typename Real, int TPL, bool QUAD, bool SOFT>
__global__ void __launch_bounds__(kWalkWarps * 32) k_eval_tiles(const WalkArgs A) {
    using V4 = typename Vec4<Real>::T;
    using V2 = typename Vec2<Real>::T;
    __shared__ __align__(32) unsigned char s_stage[kWalkWarps][walk_stage_bytes<Real>()];
    __shared__ uint32_t s_idx[kWalkWarps][32];
    constexpr bool kR5 = QUAD && (sizeof(Real) == 8 || TPL == 1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (blockIdx.x == 0 && threadIdx.x == 0) A.ctr[kCtrWalkTicket] = 0;  // kWalkFold takes the groups again
    if (aborted(A.ctr, kStageAfter)) return;
    const Stage<Real> S(s_stage[warp], s_idx[warp]);
    const V4 *__restrict__ spos = reinterpret_cast<const V4 *>(A.spos);
    const V4 *__restrict__ momA = reinterpret_cast<const V4 *>(A.mom_a);
    const V4 *__restrict__ momB = reinterpret_cast<const V4 *>(A.mom_b);
    const V2 *__restrict__ momC = reinterpret_cast<const V2 *>(A.mom_c);
    const Real eps2 = (Real)A.eps2;
    const float2 eps2v = make_float2((float)A.eps2, (float)A.eps2);
    const uint32_t total = min(A.ctr[kCtrTiles], A.tile_cap);
    for (uint32_t slot = blockIdx.x * kWalkWarps + warp; slot < total; slot += gridDim.x * kWalkWarps) {
        const uint2 h = A.tile_hdr[slot];
        const uint32_t si = A.tile_idx[(size_t)slot * 32 + lane];
        const int ns = (int)(h.y & 0xffu);
        if (ns == 0) continue;
        const uint32_t s0 = A.gfirst[h.x];
        const int cnt = (int)(A.gfirst[h.x + 1] - s0);
        Targets<Real, TPL> T;
#pragma unroll
        for (int t = 0; t < TPL; ++t) {
            V4 p{};
            if (lane + 32 * t < cnt) p = spos[s0 + lane + 32 * t];
            T.px[t] = p.x; T.py[t] = p.y; T.pz[t] = p.z;
        }
        T.set_packed();
        Real p1[TPL][4];
        if (h.y >> 8) {
            const bool r5 = kR5 && A.box[A.nseg > 1 ? seg_find(A.seg_off, A.nseg, s0) : 0u].r5fit != 0;
            stage_pc<Real, QUAD>(S, lane, si, ns, momA, momB, momC);
            __syncwarp();
            part_pc<Real, TPL, QUAD, SOFT, 16, 4>(S, T, ns, r5, eps2, eps2v, p1);
        } else {
            V4 s{};
            if (lane < ns) s = spos[si];
            const bool own = stage_pp<Real>(S, lane, s, si, ns, s0, cnt);
            __syncwarp();
            part_pp<Real, TPL, SOFT, 16>(S, T, lane, ns, own, s0, eps2, eps2v, p1);
        }
        V4 *tp = reinterpret_cast<V4 *>(A.tile_part);
#pragma unroll
        for (int t = 0; t < TPL; ++t) {
            V4 q;
            q.x = p1[t][0]; q.y = p1[t][1]; q.z = p1[t][2]; q.w = p1[t][3];
            tp[((size_t)slot * TPL + t) * 32 + lane] = q;
        }
        __syncwarp();
    }
}

}  // namespace treegb

namespace treegb {

// Host: walk arguments from the workspace.
inline WalkArgs make_walk_args(TreeWorkspace *ws, const WalkOut &out) {
    WalkArgs a;
    a.n = ws->n;
    a.gs = ws->p.group_size;
    a.ngroups = ws->list_groups_host;  // host copy of the group count (list emission only)
    a.spos = ws->spos;
    a.skey = ws->key;
    a.perm = ws->idx;
    a.ngeo = ws->ngeo;
    a.nlink = ws->nlink;
    a.mom_a = ws->mom_a;
    a.mom_b = ws->mom_b;
    a.mom_c = ws->mom_c;
    a.dmac = ws->dmac;
    a.G = ws->p.G;
    a.eps = ws->p.eps;
    a.eps2 = ws->p.eps * ws->p.eps;
    a.a = out.a;
    a.phi = out.phi;
    a.v = out.v;
    a.half_tau = out.half_tau;
    a.v2 = out.v_mirror;
    a.phi2 = out.phi_mirror;
    a.stack_depth = ws->p.stack_depth;
    a.gstat = ws->gstat;
    a.dstatus = ws->dstatus;
    a.list_off = ws->list_cnt;
    a.pc_list = ws->pc_list;
    a.pp_list = ws->pp_list;
    a.order = out.ordered ? ws->gorder : nullptr;
    a.gfirst = ws->gfirst;
    a.ctr = ws->ctr;
    a.seg_off = ws->seg_off;
    a.nseg = ws->nseg;
    a.box = ws->box;
    a.tile_hdr = ws->tile_hdr;
    a.tile_idx = ws->tile_idx;
    a.tile_part = ws->tile_part;
    a.tile_next = ws->tile_next;
    // the partial sums of two targets per lane take twice the room
    a.tile_cap = ws->p.group_size > 32 ? (ws->tile_cap / 2) & ~(uint32_t)(kTileChunk - 1) : ws->tile_cap;
    a.ghead = ws->ghead;
    a.gtiles = ws->gtiles;
    return a;
}

template <typename Real, int TPL, bool QUAD, bool KAHAN, bool SOFT, int MODE>
cudaError_t walk_run(TreeWorkspace *ws, const WalkArgs &a, cudaStream_t s) {
    if (ws->n <= 0) return cudaSuccess;
    auto k = k_walk<Real, TPL, QUAD, KAHAN, SOFT, MODE>;
    const size_t smem = kWalkWarps * walk_warp_bytes<Real>(a.stack_depth);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // persistent grid: the resident blocks, never more than the groups need
    int per_sm = 0, sms = 0, dev = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kWalkWarps * 32, smem);
    if (e != cudaSuccess) return e;
    const int64_t ng_bound = (ws->n + kWalkWarps - 1) / kWalkWarps;
    int64_t nb = (int64_t)(per_sm > 0 ? per_sm : 1) * sms;
    if (nb > ng_bound) nb = ng_bound;
    if (nb < 1) nb = 1;
    if (MODE != kWalkFold) {  // (k_eval_tiles has reset the ticket for kWalkFold)
        e = cudaMemsetAsync(ws->ctr + kCtrWalkTicket, 0, 2 * sizeof(uint32_t), s);
        if (e != cudaSuccess) return e;
    }
    k<<<(unsigned)nb, kWalkWarps * 32, smem, s>>>(a);
    ws->launches += 1;
    return cudaGetLastError();
}

// The split walk's traversal into tile slots (kWalkTiles; the precision and the
// pair terms play no part in it), or the evaluation of the slots and the fold.
template <typename Real, int TPL, bool QUAD, bool KAHAN, bool SOFT>
cudaError_t walk_split(TreeWorkspace *ws, WalkMode part, const WalkArgs &a, cudaStream_t s) {
    if (ws->n <= 0) return cudaSuccess;
    if (part == kWalkTiles) return walk_run<Real, TPL, false, false, true, kWalkTiles>(ws, a, s);
    auto k = k_eval_tiles<Real, TPL, QUAD, SOFT>;
    k<<<wave_grid(k, (int64_t)ws->tile_cap * 32, kWalkWarps * 32, 1 << 20), kWalkWarps * 32, 0, s>>>(a);
    ws->launches += 1;
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return walk_run<Real, TPL, QUAD, KAHAN, SOFT, kWalkFold>(ws, a, s);
}

}  // namespace treegb
