// Several D2Q9 steps per launch: the choice between the kernels and their launch.
#include <algorithm>

#include "lbm_tile_d2q9.cuh"

namespace lbm {

cudaError_t launch_walk_d2q9_f32(int, bool, bool, WalkArgs&, cudaStream_t);
cudaError_t launch_walk_d2q9_f16(int, bool, bool, WalkArgs&, cudaStream_t);
cudaError_t launch_walk_d2q9_bf16(int, bool, bool, WalkArgs&, cudaStream_t);

int walk_ranges(int strips, int ny, int T, int sms, int warps, double* cost)
{
    const int most = sms * warps / strips;
    double best = 1e300;
    int ranges = 1;
    for (int b = 1; b <= ny && (b <= most || b == 1); ++b) {
        const double k = (double)strips * b / (4 * sms);
        const double c = ((ny + b - 1) / b + 2 * T) * (0.45 + 0.47 * (k > 1.0 ? k : 1.0));
        if (c < best) {
            best = c;
            ranges = b;
        }
    }
    if (cost) *cost = best * (T == 4 ? 1.0 : 0.85) + 1.5;
    return ranges;
}

// Times of one launch in us, measured on GB300 (FP32; the 16-bit forms cost the
// fused kernels about 1.2 times as much, and the one-step kernel as well):
//   one step: 4.1 us from launch to launch, 80 bytes a node at 6.8 TB/s when that is more;
//   walk:     walk_ranges; rows whose length allows no 16-byte copies take 1.1 (FP32) or
//             1.5 (16-bit) times as long;
//   tile:     2.3 us + per wave of one tile per SM: 1 us to load and 0.03 us a row beyond 32
//             (300 x 4000: 13.8 us a step in three waves of two steps, walk 11.9), 0.2 us a step and
//             0.05 us a row and step (128^2: 6.2 us for 6 steps on 16-row tiles; 256^2: 8.7 on
//             24 rows; 512^2: 15.7 on 48 rows); on grids whose two states do not fit in L2 a tile's
//             loads and stores come from HBM, which nothing overlaps with one CTA per SM (FP16 2913 x 2240:
//             77 us a step; without this term the plan took it for 47 and the walk, 52, for slower).
// Walls: the walk's T = 4 instances hold 8 warps per SM instead of 12 (and T = 2 is charged alike). The strips with an x wall (1.6 times a row's
// time, with ranges of their own) and the tiles with one (1.5 times) change neither kernel's place: their figures are
// left out. Over 18 grids (333 x 33 to 4096 x 4096), FP32 and BF16, with a field, a row profile and five wall pairs, the
// choice takes 1.011 times the fastest of the three in the mean, at most 1.25 times (1280 x 900 BF16 periodic: walk 13.0,
// tile 10.4).
// The tile kernel wins below about 1M nodes (us a step: 512^2 2.7, walk 5.3, one step 4.1; 896^2 6.6, 9.1,
// 8.8), the walk above (1024^2: 7.7 against 9.0 and 10.5; 2049^2: 23, 37, 52; 4096^2: 71, 141, 190).
FusePlan plan_fused(int store, int nx, int ny, bool walls, int sms, long long left, int kinds)
{
    const double n = (double)nx * ny;
    const double single = n * 80 / 6.8e6;
    const double slow = store == ST_F32 ? (nx % 4 ? 1.1 : 1.0) : (nx % 8 ? 1.5 : 1.0);
    const double bytes = store == ST_F32 ? 80 : 52;   // a node's, read and written
    const double fetch = n * bytes > 1e8 ? 64 * bytes * sms / 6.8e6 : 0;   // us a row of every SM's tile
    double best = kinds != FUSE_ANY ? 1e300 : (single > 4.1 ? single : 4.1);
    FusePlan p{1, 0};
    for (int T = 2; T <= 4 && T <= left && (kinds & FUSE_WALK); T += 2) {
        double c;
        walk_ranges((nx + WALK_COLS - 1) / WALK_COLS, ny, T, sms, walls ? 8 : 12, &c);
        if (c * slow / T < best) {
            best = c * slow / T;
            p = {T, 0};
        }
    }
    for (int T = 2; T <= TILE_T && T <= left && (kinds & FUSE_TILE); ++T)
        for (int rows = 2 * T + 2; rows <= TILE_ROWS; rows += 2) {
            const int h = rows - 2 * T;
            const long long tiles = (long long)((nx + 63 - 2 * T) / (64 - 2 * T)) * ((ny + h - 1) / h);
            const double load = 1.0 + (fetch > 0 ? fetch * rows : 0.03 * std::max(0, rows - 32));
            const double c = 2.3 + (double)((tiles + sms - 1) / sms) * (load + 0.2 * T + 0.05 * T * (h + T - 1));
            if (c / T < best) {
                best = c / T;
                p = {T, rows};
            }
        }
    return p;
}

cudaError_t launch_walk(int store, int ukind, int T, const StepArgs& a, void* const* mid, cudaStream_t st)
{
    WalkArgs p{};
    p.a = a;
    if (ukind == U_NONE) p.a.ua = nullptr;
    for (int j = 0; j <= T; ++j) p.srow[j] = sched_row(a.k - 1 + j, a.sched && ukind != U_NONE ? a.sched_len : 0);
    for (int j = 0; mid != nullptr && j < T - 1; ++j) p.mid[j] = mid[j];
    uintptr_t mis = reinterpret_cast<uintptr_t>(a.src) | reinterpret_cast<uintptr_t>(a.dst) |
                    reinterpret_cast<uintptr_t>(a.phi_src) | reinterpret_cast<uintptr_t>(a.phi_dst) |
                    (ukind == U_FIELD ? reinterpret_cast<uintptr_t>(a.ua) : 0);
    for (void* m : p.mid) mis |= reinterpret_cast<uintptr_t>(m);
    p.vec = a.nx % 2 == 0 && (mis & 7) == 0;
    p.wide = a.nx % (store == ST_F32 ? 4 : 8) == 0 && (mis & 15) == 0;
    const bool field = ukind == U_FIELD;
    if (store == ST_F16) return launch_walk_d2q9_f16(T, field, false, p, st);
    if (store == ST_BF16) return launch_walk_d2q9_bf16(T, field, false, p, st);
    return launch_walk_d2q9_f32(T, field, mid != nullptr, p, st);
}

cudaError_t launch_tile(int store, int ukind, int T, int rows, const StepArgs& a, void* const* mid, cudaStream_t st)
{
    TileArgs p{};
    p.a = a;
    if (ukind == U_NONE) p.a.ua = nullptr;
    p.field = ukind == U_FIELD;
    p.T = T;
    p.rows = rows;
    for (int j = 0; j <= T; ++j) p.srow[j] = sched_row(a.k - 1 + j, a.sched && ukind != U_NONE ? a.sched_len : 0);
    for (int j = 0; mid != nullptr && j < T - 1; ++j) p.mid[j] = mid[j];
    const bool walls = a.bc_lo != BC_PERIODIC || a.bcx_lo != BC_PERIODIC;
    if (store == ST_F16) return walls ? tile_d2q9<ST_F16, true>(p, st) : tile_d2q9<ST_F16, false>(p, st);
    if (store == ST_BF16) return walls ? tile_d2q9<ST_BF16, true>(p, st) : tile_d2q9<ST_BF16, false>(p, st);
    return walls ? tile_d2q9<ST_F32, true>(p, st) : tile_d2q9<ST_F32, false>(p, st);
}

}  // namespace lbm
