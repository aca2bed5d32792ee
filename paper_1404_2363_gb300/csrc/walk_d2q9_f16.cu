// T fused D2Q9 steps, FP16 storage: kernel instantiations.
#include "lbm_walk_d2q9.cuh"

namespace lbm {

cudaError_t launch_walk_d2q9_f16(int T, bool field, bool, WalkArgs& p, cudaStream_t st)
{
    if (T == 4) return field ? walk_w<ST_F16, true, 4, false>(p, st) : walk_w<ST_F16, false, 4, false>(p, st);
    return field ? walk_w<ST_F16, true, 2, false>(p, st) : walk_w<ST_F16, false, 2, false>(p, st);
}

}  // namespace lbm
