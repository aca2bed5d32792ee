// T <= 8 time steps of the D2Q9 model on tiles held in shared memory (all storage
// forms, walls on any face), for small and middle grids.
//
// There one step a launch is bound by the launch itself (4.1 us from launch to
// launch up to 256^2, 6.2 at 512^2). Here a CTA loads 64 columns x `rows` rows of
// the state, takes T steps in shared memory (a row and a column are lost on each
// side per step) and stores the rest: neighbouring CTAs repeat each other's
// halo instead of talking. The steps run in place, in pairs (gather, local), with
// one block barrier each, so a tile costs 36 B a node and one copy of it.
// A lane owns the columns l and l + 32 of a row: every shared access is one
// conflict-free wavefront at any shift, and the two nodes form the operands of the
// paired arithmetic without a move.
//
// us a step: 128^2 0.92, 256^2 1.3, 512^2 2.7 (one step a launch: 2.1, 2.2, 4.1; not overlapping 4.1, 4.1, 6.2).
// Bound by the launch and the load (about 3.5 us a launch) on small grids, by
// issue on larger ones (278 instructions a row of 64 nodes and step at 64
// registers, 53 % issue active; at 128 registers, one CTA of 16 warps per SM, the
// constants stay in registers: 2.6 instead of 2.75 us at 512^2). 1024-thread
// CTAs: 1.1 / 1.5 / 2.85 us.
#pragma once
#include "lbm_walk_d2q9.cuh"

namespace lbm {

constexpr int TILE_THREADS = 512;
constexpr int TILE_PAD = 32;     // floats around every plane of a tile
constexpr int tile_smem(int rows) { return (TILE_PAD + 11 * (64 * rows + TILE_PAD)) * 4; }   // nine populations, two velocity factors
static_assert(tile_smem(TILE_ROWS) <= 227 * 1024 - 128, "a tile fits in shared memory");

template <int STORE, bool WALLS>
__global__ void __launch_bounds__(TILE_THREADS, 1) k_tile_d2q9(const __grid_constant__ TileArgs p)
{
    using L = D2Q9;
    constexpr bool NEQ = STORE != ST_F32;
    constexpr float SC = STORE == ST_F16 ? F16_SCALE : 1.f;   // working units of the 16-bit forms
    const StepArgs& a = p.a;
    const Coef& c = a.c;
    const int nx = a.nx, ny = a.ny, N = (int)a.ncell;
    const int T = p.T, H = p.rows, P = 64;
    extern __shared__ float tile_sm[];
    const int plane = H * P + TILE_PAD;
    float* const sm = tile_sm + TILE_PAD;
    __shared__ float sched[TILE_T + 1][2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // this CTA's nodes: columns [xv, xv + P - 2T), rows [yv, yv + H - 2T)
    const int xv = blockIdx.x * (P - 2 * T), yv = blockIdx.y * (H - 2 * T);
    const int xe = min(xv + P - 2 * T, nx), ye = min(yv + H - 2 * T, ny);
    const bool xwall = WALLS && a.bcx_lo != BC_PERIODIC, ywall = WALLS && a.bc_lo != BC_PERIODIC;
    grid_dep_sync();
    const void* const asrc = after_dep(a.src);
    const float* const aua = after_dep(a.ua);
    const float* const aphi = after_dep(a.phi_src);
    if (threadIdx.x <= T) {
        float s[3];
        sched_row_at(after_dep(a.sched), p.srow[threadIdx.x], 2, s);
        sched[threadIdx.x][0] = s[0];
        sched[threadIdx.x][1] = s[1];
    }
    if (NEQ) __syncthreads();

    // a warp takes every WARPS-th row, a lane the nodes lane and lane + 32 of it
    constexpr int WARPS = TILE_THREADS / 32;
#pragma unroll NEQ ? 2 : 1
    for (int ty = warp; ty < H; ty += WARPS) {
        int y = yv - T + ty;
        // rows that no step needs, or beyond a wall, are not loaded
        if (y >= ye + T || (ywall && (y < 0 || y >= ny))) continue;
        if (!ywall) {
            y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
            if (y < 0 || y >= ny) y = ((y % ny) + ny) % ny;
        }
        int x[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            int xx = xv - T + lane + 32 * h;
            if (xwall) xx = min(max(xx, 0), nx - 1);
            else {
                xx = xx < 0 ? xx + nx : (xx >= nx ? xx - nx : xx);
                if (xx < 0 || xx >= nx) xx = ((xx % nx) + nx) % nx;
            }
            x[h] = xx + y * nx;
        }
        float* d = sm + ty * P + lane;
        if constexpr (NEQ) {
            float2 ax = sp2(0.f), ay = sp2(0.f);
            if (p.field) {
                ax = make_float2(__ldg(aua + x[0]), __ldg(aua + x[1]));
                ay = make_float2(__ldg(aua + N + x[0]), __ldg(aua + N + x[1]));
            } else if (aua != nullptr) {
                ax = sp2(__ldg(aua + y));
                ay = sp2(__ldg(aua + ny + y));
            }
            const unsigned short* q = static_cast<const unsigned short*>(asrc);
            unsigned g[9];
#pragma unroll
            for (int i = 0; i < 9; ++i)
                g[i] = (unsigned)ld_dep(q + i * N + x[0]) | (unsigned)ld_dep(q + i * N + x[1]) << 16;
            const float2 phi = xmul2(make_float2(ld_dep(aphi + x[0]), ld_dep(aphi + x[1])), sp2(SC));
            float2 e[9];
            walk_feq(c, xmul2(ax, sp2(sched[0][0])), xmul2(ay, sp2(sched[0][1])), e);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const float2 f = fma2(phi, e[i], Pair<STORE>::to_f_raw(QuadH<STORE>::as_t2(g[i])));
                d[i * plane] = f.x, d[i * plane + 32] = f.y;
            }
            d[9 * plane] = ax.x, d[9 * plane + 32] = ax.y;
            d[10 * plane] = ay.x, d[10 * plane + 32] = ay.y;
        } else {
            const float* q = static_cast<const float*>(asrc);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                walk_copy<4>(d + i * plane, q + i * N + x[0]);
                walk_copy<4>(d + i * plane + 32, q + i * N + x[1]);
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                float* du = d + (9 + k) * plane;
                if (p.field) {
                    walk_copy<4>(du, aua + k * N + x[0]);
                    walk_copy<4>(du + 32, aua + k * N + x[1]);
                } else {
                    const float v = aua != nullptr ? __ldg(aua + k * ny + y) : 0.f;
                    du[0] = v, du[32] = v;
                }
            }
        }
    }
    if (!NEQ) asm volatile("cp.async.wait_all;" ::: "memory");

    // Steps in place, in pairs. A tile slot (i, x) first holds f'_i(x). The odd
    // step gathers f_i(x) from the slots (i, x - e_i), which no other node
    // reads, and writes f'_opp(i)(x) back to them: slot (i, y) then holds the
    // population opp(i) that streams to y. The even step takes its populations
    // from the node's own slots and leaves f'_i(x) in slot (i, x). The last step
    // goes to global memory.
    auto row_step = [&](int s, int ty, auto odd, auto slow) {   // slow: a row or a tile with a wall
        constexpr bool gather = decltype(odd)::value;
        const int y = yv - T + ty;
        float* const d = sm + ty * P + lane;
        const float2 uax = make_float2(d[9 * plane], d[9 * plane + 32]);
        const float2 uay = make_float2(d[10 * plane], d[10 * plane + 32]);
        auto slot = [&](int i) { return d + (gather ? i * plane - L::ey(i) * P - L::ex(i) : opposite<L>(i) * plane); };
        float2 f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const float* q = slot(i);
            f[i] = make_float2(q[0], q[32]);
        }
        bool in0 = true, in1 = true;   // the lane's nodes inside the domain (x walls)
        if constexpr (decltype(slow)::value) {
            const int x = xv - T + lane;
            in0 = !xwall || (x >= 0 && x < nx);
            in1 = !xwall || (x + 32 >= 0 && x + 32 < nx);
            const bool l0 = xwall && x == 0, l1 = xwall && x + 32 == 0, r0 = xwall && x == nx - 1,
                       r1 = xwall && x + 32 == nx - 1;
            const bool edge = __any_sync(0xffffffffu, l0 || l1 || r0 || r1);
            const bool lo = ywall && y == 0, hi = ywall && y == ny - 1;
            const int kind = lo ? a.bc_lo : a.bc_hi;
            // the node's own f'_opp(i) of the last step: its own slot, or the one it was pushed to
            auto own = [&](int i) { return d + (gather ? opposite<L>(i) * plane : i * plane - L::ey(i) * P - L::ex(i)); };
            if ((lo || hi) && kind == BC_BOUNCE) {
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    if (L::ey(i) != 0 && (L::ey(i) == 1) == lo) f[i] = make_float2(own(i)[0], own(i)[32]);
            }
            if (edge) {
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    if (L::ex(i) == 1 && a.bcx_lo == BC_BOUNCE) {
                        if (l0) f[i].x = own(i)[0];
                        if (l1) f[i].y = own(i)[32];
                    }
                    if (L::ex(i) == -1 && a.bcx_hi == BC_BOUNCE) {
                        if (r0) f[i].x = own(i)[0];
                        if (r1) f[i].y = own(i)[32];
                    }
                }
                if (a.bcx_lo == BC_NOFLUX) {
                    if (l0) f[1].x = f[3].x, f[5].x = f[6].x, f[8].x = f[7].x;
                    if (l1) f[1].y = f[3].y, f[5].y = f[6].y, f[8].y = f[7].y;
                }
                if (a.bcx_hi == BC_NOFLUX) {
                    if (r0) f[3].x = f[1].x, f[6].x = f[5].x, f[7].x = f[8].x;
                    if (r1) f[3].y = f[1].y, f[6].y = f[5].y, f[7].y = f[8].y;
                }
            }
            if (lo || hi) {
                if (kind == BC_NOFLUX) {
                    if (lo) f[2] = f[4], f[5] = f[8], f[6] = f[7];
                    else f[4] = f[2], f[8] = f[5], f[7] = f[6];
                } else if (kind == BC_DIRICHLET) {
                    float2 e[9];
                    walk_feq(c, xmul2(uax, sp2(sched[s - 1][0])), xmul2(uay, sp2(sched[s - 1][1])), e);
                    const int inward = lo ? 1 : -1;
                    float2 known = sp2(0.f), wk = sp2(0.f);
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        if (L::ey(i) == inward) wk = add2(wk, e[i]);
                        else known = add2(known, f[i]);
                    }
                    const float phiw = (lo ? a.phiw_lo : a.phiw_hi) * SC;
                    const float2 ps = make_float2((phiw - known.x) / wk.x, (phiw - known.y) / wk.y);
#pragma unroll
                    for (int i = 0; i < 9; ++i)
                        if (L::ey(i) == inward) f[i] = xmul2(ps, e[i]);
                }
            }
        }
        const float2 ux = NEQ ? xmul2(uax, sp2(sched[s][0])) : mul2(uax, sp2(sched[s][0]));
        const float2 uy = NEQ ? xmul2(uay, sp2(sched[s][1])) : mul2(uay, sp2(sched[s][1]));
        const float2 phi = walk_collide<NEQ>(f, ux, uy, c);
        const int x = xv - T + lane;
        const bool keep = y >= yv && y < ye;
        const bool k0 = keep && x >= xv && x < xe, k1 = keep && x + 32 >= xv && x + 32 < xe;
        const int cell = y * nx + x;
        if constexpr (NEQ) {
            unsigned g[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) g[i] = QuadH<STORE>::as_u(Pair<STORE>::from_f_raw(f[i]));
            if (s == T) {
                unsigned short* q = static_cast<unsigned short*>(a.dst) + cell;
                const float2 ph = xmul2(phi, sp2(1.f / SC));
                if (k0) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) q[i * N] = (unsigned short)(g[i] & 0xffffu);
                    a.phi_dst[cell] = ph.x;
                }
                if (k1) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) q[i * N + 32] = (unsigned short)(g[i] >> 16);
                    a.phi_dst[cell + 32] = ph.y;
                }
                return;
            }
            float2 e[9];
            walk_feq(c, ux, uy, e);   // the offsets as they would be stored, decoded with u of this step
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = fma2(phi, e[i], Pair<STORE>::to_f_raw(QuadH<STORE>::as_t2(g[i])));
        } else {
            float* q = static_cast<float*>(s == T ? a.dst : p.mid[s - 1]);
            if (q != nullptr) {
                q += cell;
                if (k0) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) q[i * N] = f[i].x;
                }
                if (k1) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) q[i * N + 32] = f[i].y;
                }
            }
            if (s == T) return;
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            float* q = gather ? slot(i) : d + i * plane;
            const float2 v = gather ? f[opposite<L>(i)] : f[i];
            if (in0) q[0] = v.x;
            if (in1) q[32] = v.y;
        }
    };
    const bool xedge = xwall && (xv - T <= 0 || xv + 64 - T >= nx);   // the tile has columns at or past an x wall
    auto step = [&](int t, auto odd) {
        __syncthreads();
#pragma unroll 1
        for (int ty = warp; ty < H; ty += WARPS) {
            const int y = yv - T + ty;
            // the rows that later steps still need, inside the domain
            if (y < yv - (T - t) || y >= ye + (T - t) || (ywall && (y < 0 || y >= ny))) continue;
            if (WALLS && (xedge || (ywall && (y == 0 || y == ny - 1)))) row_step(t, ty, odd, std::integral_constant<bool, WALLS>{});
            else row_step(t, ty, odd, std::false_type{});
        }
    };
#pragma unroll 1
    for (int t = 1; t <= T; t += 2) {
        step(t, std::true_type{});
        if (t < T) step(t + 1, std::false_type{});
    }
}

template <int STORE, bool WALLS>
cudaError_t tile_d2q9(const TileArgs& p, cudaStream_t st)
{
    static std::atomic<unsigned> known[64];
    KernelFit fit;
    const cudaError_t fe = kernel_fit(known, k_tile_d2q9<STORE, WALLS>, TILE_THREADS, tile_smem(TILE_ROWS), fit);
    if (fe != cudaSuccess) return fe;
    const dim3 grid((unsigned)((p.a.nx + 64 - 2 * p.T - 1) / (64 - 2 * p.T)),
                    (unsigned)((p.a.ny + p.rows - 2 * p.T - 1) / (p.rows - 2 * p.T)));
    return launch_dependent(k_tile_d2q9<STORE, WALLS>, grid, dim3(TILE_THREADS), tile_smem(p.rows), st, p);
}

}  // namespace lbm
