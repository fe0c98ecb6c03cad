// walk_split_f32.cu -- the split walk (walk.cuh) in FP32.
#include "walk.cuh"

namespace treegb {

template <int TPL, bool QUAD>
static cudaError_t dispatch(TreeWorkspace *ws, WalkMode part, const WalkArgs &a, bool kahan, bool soft, cudaStream_t s) {
    if (kahan)
        return soft ? walk_split<float, TPL, QUAD, true, true>(ws, part, a, s)
                    : walk_split<float, TPL, QUAD, true, false>(ws, part, a, s);
    return soft ? walk_split<float, TPL, QUAD, false, true>(ws, part, a, s)
                : walk_split<float, TPL, QUAD, false, false>(ws, part, a, s);
}

cudaError_t launch_walk_split_f32(TreeWorkspace *ws, WalkMode part, const WalkOut &out, cudaStream_t s) {
    const WalkArgs a = make_walk_args(ws, out);
    const bool kahan = ws->p.kahan != 0, soft = walk_soft_f32(ws->p.eps);
    if (ws->p.group_size > 32)
        return ws->p.order == 2 ? dispatch<2, true>(ws, part, a, kahan, soft, s) : dispatch<2, false>(ws, part, a, kahan, soft, s);
    return ws->p.order == 2 ? dispatch<1, true>(ws, part, a, kahan, soft, s) : dispatch<1, false>(ws, part, a, kahan, soft, s);
}

}  // namespace treegb
