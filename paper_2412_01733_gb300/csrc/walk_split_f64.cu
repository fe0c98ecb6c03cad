// walk_split_f64.cu -- the split walk (walk.cuh) in FP64.
#include "walk.cuh"

namespace treegb {

template <int TPL, bool QUAD>
static cudaError_t dispatch(TreeWorkspace *ws, WalkMode part, const WalkArgs &a, bool soft, cudaStream_t s) {
    return soft ? walk_split<double, TPL, QUAD, false, true>(ws, part, a, s)
                : walk_split<double, TPL, QUAD, false, false>(ws, part, a, s);
}

cudaError_t launch_walk_split_f64(TreeWorkspace *ws, WalkMode part, const WalkOut &out, cudaStream_t s) {
    const WalkArgs a = make_walk_args(ws, out);
    const bool soft = ws->p.eps > 0.0;
    if (ws->p.group_size > 32)
        return ws->p.order == 2 ? dispatch<2, true>(ws, part, a, soft, s) : dispatch<2, false>(ws, part, a, soft, s);
    return ws->p.order == 2 ? dispatch<1, true>(ws, part, a, soft, s) : dispatch<1, false>(ws, part, a, soft, s);
}

}  // namespace treegb
