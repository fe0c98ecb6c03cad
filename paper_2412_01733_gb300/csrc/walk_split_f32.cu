// walk_split_f32.cu -- the split walk (walk.cuh) in FP32.
#include "walk.cuh"

namespace treegb {

template <int TPL, bool QUAD>
static cudaError_t dispatch(TreeWorkspace *ws, const WalkArgs &a, bool kahan, bool soft, cudaStream_t s) {
    if (kahan)
        return soft ? walk_split<float, TPL, QUAD, true, true>(ws, a, s)
                    : walk_split<float, TPL, QUAD, true, false>(ws, a, s);
    return soft ? walk_split<float, TPL, QUAD, false, true>(ws, a, s)
                : walk_split<float, TPL, QUAD, false, false>(ws, a, s);
}

cudaError_t launch_walk_split_f32(TreeWorkspace *ws, const WalkOut &out, cudaStream_t s) {
    const WalkArgs a = make_walk_args(ws, out);
    const bool kahan = ws->p.kahan != 0, soft = walk_soft_f32(ws->p.eps);
    if (ws->p.group_size > 32)
        return ws->p.order == 2 ? dispatch<2, true>(ws, a, kahan, soft, s) : dispatch<2, false>(ws, a, kahan, soft, s);
    return ws->p.order == 2 ? dispatch<1, true>(ws, a, kahan, soft, s) : dispatch<1, false>(ws, a, kahan, soft, s);
}

}  // namespace treegb
