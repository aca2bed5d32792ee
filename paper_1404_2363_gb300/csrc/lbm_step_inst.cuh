// Launch dispatch for one (lattice, storage) pair of the fused step kernel.
// Each step_*.cu translation unit includes this with LBM_LAT / LBM_STORE /
// LBM_FN defined, so the template instantiations compile in parallel.
#include "lbm_device.cuh"
#include "lbm_pair.cuh"
#include "lbm_pair_d3q15.cuh"
#include "lbm_tma_d2q9.cuh"
#include "lbm_zwalk_d3q15.cuh"

namespace lbm {

// Whether a one-step launch may start while the previous one drains (LD_ORDERED or
// LD_PLAIN) or is an ordinary one (LD_READONLY). The overlap saves about 2 us a launch,
// but blocks that execute the wait and the trigger start at no more than one a ns: with
// 64 threads a block, D2Q9 4096^2 FP32 takes 263 us a step instead of 175 (262144
// blocks). So not where starting the blocks takes longer than the nodes, at the rates the
// kernels reach, and the 2 us (3 with D3Q15's longer chain: 41 x 62 x 192 FP32 15.4 us a
// step overlapping, 16.6 not). Rates measured with 64 (pairs: 32) threads a block, in TB/s:
// FP32 6; 16 bit: D2Q9 5, D3Q15 with one node per thread 3.7 (at rest, periodic; else 2.6),
// pairs 5, less by what lanes past the row's end take (FP16 and periodic: 3.2, where the
// ordered loads are also the faster ones, 290 x 200 x 200 at rest 219 us against 237).
inline bool overlap_pays(dim3 grid, int block, const StepArgs& a, int q, int store, int uk, bool walls, bool pairs)
{
    const double blocks = (double)grid.x * grid.y * grid.z;
    const int dim = q == 9 ? 2 : 3;
    const int bytes = (store == ST_F32 ? 8 * q : 4 * q + 8) + (uk == U_FIELD ? 4 * dim : 0);
    double rate = 6.0e6;   // bytes a us
    if (store != ST_F32) {
        if (q == 9) rate = 5.0e6;
        else if (pairs) rate = store == ST_F16 && !walls ? 3.2e6 : 5.0e6 * a.nx / (2.0 * block * grid.x);
        else rate = uk == U_NONE && !walls ? 3.7e6 : 2.6e6;
    }
    return blocks * 1e-3 + 1.0 <= (double)a.ncell * bytes / rate + (q == 9 ? 2.0 : 3.0);
}

template <class L, int STORE, int UK, bool WALLS>
static cudaError_t step_vec(LaunchCfg cfg, const StepArgs& a, cudaStream_t st)
{
    if (a.bcx_lo != BC_PERIODIC || a.bcz_lo != BC_PERIODIC) {
        // walls on the x or z faces: the general one-node kernel, whatever the launch shape
        const dim3 grid((unsigned)((a.nx + 255) / 256), (unsigned)a.ny, (unsigned)a.nz);
        const bool ov = overlap_pays(grid, 256, a, L::Q, STORE, UK, true, false);
        auto launch = [&](auto kernel) { return launch_dependent(kernel, grid, dim3(256), 0, st, a, ov); };
        if ((long long)(L::Q + 3) * a.ncell < (1LL << 31))
            return launch(ov ? k_step_box<L, STORE, UK, int, LD_PLAIN> : k_step_box<L, STORE, UK, int, LD_READONLY>);
        return launch(ov ? k_step_box<L, STORE, UK, long long, LD_PLAIN> : k_step_box<L, STORE, UK, long long, LD_READONLY>);
    }
    if constexpr (L::Q == 9) {
        if (cfg.vec == 6 && quad_ok(a, UK)) {
            // node-quad variant: 128-bit / 64-bit vector loads and stores, four nodes per thread
            const int per = 4 * cfg.block;
            dim3 grid((unsigned)((a.nx + per - 1) / per), (unsigned)a.ny, 1);
            k_step_quad_d2q9<STORE, UK, WALLS><<<grid, cfg.block, 0, st>>>(a);
            return cudaGetLastError();
        }
    }
    if constexpr (L::Q == 15 && STORE != ST_F32) {
        // phi, the velocity factors and the offsets staged in shared memory along a walk in z
        if (cfg.vec == 9 && cfg.block == 256 && zw_ok(a, UK, 8)) return launch_zw_d3q15<STORE, UK, WALLS, 8>(a, st);
        if (cfg.vec == 9 && cfg.block == 128 && zw_ok(a, UK, 4)) return launch_zw_d3q15<STORE, UK, WALLS, 4>(a, st);
        if (cfg.vec == 5 && pair_ok(a, UK, L::Q)) {
            // node-pair variant (paired FP32 arithmetic, two adjacent nodes per thread)
            const int per = 2 * cfg.block;
            dim3 grid((unsigned)((a.nx + per - 1) / per), (unsigned)a.ny, (unsigned)a.nz);
            // Large launches gain nothing from the overlap, and these instances lose more by its loads (us a
            // step, LD_ORDERED against LD_READONLY): walls and a field 256 x 256 x 256 BF16 477 / 363, 128 x
            // 128 x 64 26.3 / 23.3; FP16 between walls at rest 290 x 200 x 200 191.6 / 181.7; BF16 with a field
            // 142 x 194 x 246 174 / 167 (but 64 x 225 x 163 56.3 / 57.6)
            long long most = 1LL << 62;
            if (UK == U_FIELD && WALLS) most = 1LL << 19;
            else if (UK == U_NONE && WALLS && STORE == ST_F16) most = 3LL << 20;
            else if (UK == U_FIELD && STORE == ST_BF16) most = 5LL << 19;
            const bool ov = a.ncell <= most && overlap_pays(grid, cfg.block, a, L::Q, STORE, UK, WALLS, true);
            return launch_dependent(ov ? k_step_pair_d3q15<STORE, UK, WALLS, LD_ORDERED> : k_step_pair_d3q15<STORE, UK, WALLS, LD_READONLY>,
                                    grid, dim3((unsigned)cfg.block), 0, st, a, ov);
        }
    }
    if constexpr (L::Q == 9 && STORE != ST_F32) {
        // TMA-staged rows: two rows per iteration and six stages, or one row and four
        if (cfg.vec == 7 && tma_ok(a, UK)) return launch_tma_d2q9<STORE, UK, WALLS, 2, 6>(a, st);
        if (cfg.vec == 8 && tma_ok(a, UK)) return launch_tma_d2q9<STORE, UK, WALLS, 1, 4>(a, st);
        if (cfg.vec == 5 && a.nz == 1 && pair_ok(a, UK, L::Q)) {
            // node-pair variant (paired FP32 arithmetic, two adjacent nodes per thread)
            const int per = 2 * cfg.block;
            dim3 grid((unsigned)((a.nx + per - 1) / per), (unsigned)a.ny, 1);
            k_step_pair_d2q9<STORE, UK, WALLS><<<grid, cfg.block, 0, st>>>(a);
            return cudaGetLastError();
        }
    }
    const int vec = cfg.vec == 2 ? 2 : 1;
    const int per = cfg.block * vec;
    dim3 grid((unsigned)((a.nx + per - 1) / per), (unsigned)a.ny, (unsigned)a.nz);
    // between walls with a field, the D2Q9 16-bit forms lose more by the ordered loads than large launches gain
    // (4096^2 FP16, LD_ORDERED against LD_READONLY: two nodes per thread 245 / 213 us a step, one 220 / 214)
    constexpr bool slow = L::Q == 9 && STORE != ST_F32 && UK == U_FIELD && WALLS;
    const bool ov = !(slow && a.ncell >= (vec == 2 ? 1LL << 21 : 1LL << 23)) &&
                    overlap_pays(grid, cfg.block, a, L::Q, STORE, UK, WALLS, false);
    auto launch = [&](auto kernel) { return launch_dependent(kernel, grid, dim3((unsigned)cfg.block), 0, st, a, ov); };
    // 32-bit offsets when every plane and velocity offset fits
    if ((long long)(L::Q + 3) * a.ncell < (1LL << 31)) {
        if (vec == 2)
            return launch(ov ? k_step<L, STORE, UK, WALLS, 2, int, LD_ORDERED> : k_step<L, STORE, UK, WALLS, 2, int, LD_READONLY>);
        return launch(ov ? k_step<L, STORE, UK, WALLS, 1, int, LD_ORDERED> : k_step<L, STORE, UK, WALLS, 1, int, LD_READONLY>);
    }
    if (vec == 2)
        return launch(ov ? k_step<L, STORE, UK, WALLS, 2, long long, LD_ORDERED> : k_step<L, STORE, UK, WALLS, 2, long long, LD_READONLY>);
    return launch(ov ? k_step<L, STORE, UK, WALLS, 1, long long, LD_ORDERED> : k_step<L, STORE, UK, WALLS, 1, long long, LD_READONLY>);
}

template <class L, int STORE, int UK>
static cudaError_t step_w(bool walls, LaunchCfg cfg, const StepArgs& a, cudaStream_t st)
{
    return walls ? step_vec<L, STORE, UK, true>(cfg, a, st) : step_vec<L, STORE, UK, false>(cfg, a, st);
}

cudaError_t LBM_FN(int uk, bool walls, LaunchCfg cfg, const StepArgs& a, cudaStream_t st)
{
    switch (uk) {
        case U_FIELD: return step_w<LBM_LAT, LBM_STORE, U_FIELD>(walls, cfg, a, st);
        case U_ROW: return step_w<LBM_LAT, LBM_STORE, U_ROW>(walls, cfg, a, st);
        default: return step_w<LBM_LAT, LBM_STORE, U_NONE>(walls, cfg, a, st);
    }
}

}  // namespace lbm
