// T fused D2Q9 steps, FP32 storage: kernel instantiations.
#include "lbm_walk_d2q9.cuh"

namespace lbm {

cudaError_t launch_walk_d2q9_f32(int T, bool field, bool save, WalkArgs& p, cudaStream_t st)
{
    if (save) {
        if (T == 4) return field ? walk_w<ST_F32, true, 4, true>(p, st) : walk_w<ST_F32, false, 4, true>(p, st);
        return field ? walk_w<ST_F32, true, 2, true>(p, st) : walk_w<ST_F32, false, 2, true>(p, st);
    }
    if (T == 4) return field ? walk_w<ST_F32, true, 4, false>(p, st) : walk_w<ST_F32, false, 4, false>(p, st);
    return field ? walk_w<ST_F32, true, 2, false>(p, st) : walk_w<ST_F32, false, 2, false>(p, st);
}

}  // namespace lbm
