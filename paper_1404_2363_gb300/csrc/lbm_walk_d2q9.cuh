// T = 2 or 4 time steps of the D2Q9 model in one pass over the grid (all storage
// forms, walls on any face), for grids that do not fit in a few waves of tiles.
//
// One step a launch is bound by HBM: 80 B a node and step for FP32, 193 us at
// 4096^2. Here a warp owns a strip of 64 columns (a node pair per lane) and walks
// down a range of rows. Every level of the walk takes one row of the state of its
// step and gives the row above it one step later: the e_y = +-1 pulls come from
// what the warp keeps of its last two rows in registers (18 a level and node
// pair), the e_x = +-1 pulls from the neighbouring lanes by shuffles, so a state
// between the levels never leaves the register file, and a warp waits for no other.
// The price is redundant work: of the 64 columns 56 are kept (a column is lost on
// each side per step), and a range walks 2 T more rows than it stores.
// Rows enter through a ring in shared memory, three in flight, by 16-byte cp.async
// (register prefetch of one row: 105 us a step; 8-byte copies through L1: 74).
//
// FP32, 4096^2, T = 4: 71 us a step (1.34 GB a launch of four steps, what one step
// moves, at 4.7 TB/s; issue 60 %, 12 warps per SM); 16-bit forms 86 to 88 us against
// 207 (one node per thread) and 120 (TMA-staged), 1024^2 FP32 7.7 against 12.3. Measured and
// not kept: T = 3 at 12 or 16 warps per SM (81 / 102 us), T = 4 at 14 warps per SM
// (100: spills), T = 2 (130), scalar instead of paired arithmetic (84).
#pragma once
#include <type_traits>

#include "lbm_pair.cuh"

namespace lbm {

// A product that feeds an addition, rounded on its own in every build, so that
// the fused steps give the bits of k_step (which uses __fmul_rn): a paired
// product may be fused into a paired addition that follows it, with any rounding
// suffix.
__device__ __forceinline__ float2 xmul2(float2 a, float2 b)
{
    return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y));
}

// collide<D2Q9, OFFSET> for a node pair, bit for bit: post-collision
// populations (FP32 storage) or offsets (16-bit forms). Returns phi.
template <bool OFFSET>
__device__ __forceinline__ float2 walk_collide(float2 (&v)[9], float2 ux, float2 uy, const Coef& c)
{
    const float2 sx = add2(v[1], v[3]), ax = sub2(v[1], v[3]);
    const float2 sy = add2(v[2], v[4]), ay = sub2(v[2], v[4]);
    const float2 p57 = add2(v[5], v[7]), d57 = sub2(v[5], v[7]);
    const float2 p68 = add2(v[6], v[8]), d68 = sub2(v[6], v[8]);
    const float2 sa = add2(sx, sy), sd = add2(p57, p68);
    const float2 dx = sub2(d57, d68), dy = add2(d57, d68);
    const float2 phi = add2(add2(v[0], sa), sd);
    const float2 m7 = sub2(sx, sy), m8 = sub2(p57, p68);
    float2 A, B, AP, AM, BP, BM, X, Xd, Y, Yd;
    if constexpr (OFFSET) {
        const float2 d1 = fma2(sp2(-c.meq1), phi, fma2(sp2(2.f), sd, fma2(sp2(-4.f), v[0], neg2(sa))));
        const float2 d2 = fma2(sp2(-c.meq2), phi, fma2(sp2(-2.f), sa, fma2(sp2(4.f), v[0], sd)));
        const float2 d3 = fma2(neg2(phi), ux, add2(ax, dx)), d4 = fma2(phi, ux, fma2(sp2(-2.f), ax, dx));
        const float2 d5 = fma2(neg2(phi), uy, add2(ay, dy)), d6 = fma2(phi, uy, fma2(sp2(-2.f), ay, dy));
        const float2 a1 = mul2(d1, sp2(c.ro[1])), a2 = mul2(d2, sp2(c.ro[2]));
        const float2 a4 = mul2(d4, sp2(c.ro[4])), a6 = mul2(d6, sp2(c.ro[6]));
        const float2 a3 = fma2(sp2(c.fr[0]), d3, fma2(sp2(c.fr[1]), d4, fma2(sp2(c.fr[2]), d5, mul2(sp2(c.fr[3]), d6))));
        const float2 a5 = fma2(sp2(c.fr[4]), d3, fma2(sp2(c.fr[5]), d4, fma2(sp2(c.fr[6]), d5, mul2(sp2(c.fr[7]), d6))));
        A = fma2(sp2(-2.f), a2, neg2(a1));
        B = fma2(sp2(2.f), a1, a2);
        AP = fma2(sp2(c.ro[7]), m7, A), AM = fma2(sp2(-c.ro[7]), m7, A);
        BP = fma2(sp2(c.ro[8]), m8, B), BM = fma2(sp2(-c.ro[8]), m8, B);
        X = fma2(sp2(-2.f), a4, a3), Xd = fma2(sp2(c.ro[4]), d4, a3);
        Y = fma2(sp2(-2.f), a6, a5), Yd = fma2(sp2(c.ro[6]), d6, a5);
    } else {
        const float2 m1 = fma2(sp2(2.f), sd, fma2(sp2(-4.f), v[0], neg2(sa)));
        const float2 m2 = fma2(sp2(-2.f), sa, fma2(sp2(4.f), v[0], sd));
        const float2 m3 = add2(ax, dx), m4 = fma2(sp2(-2.f), ax, dx);
        const float2 m5 = add2(ay, dy), m6 = fma2(sp2(-2.f), ay, dy);
        float2 d1 = fma2(sp2(-c.meq1), phi, m1), d2 = fma2(sp2(-c.meq2), phi, m2);
        const float2 d3 = fma2(neg2(phi), ux, m3), d4 = fma2(phi, ux, m4);
        const float2 d5 = fma2(neg2(phi), uy, m5), d6 = fma2(phi, uy, m6);
        float2 d7 = m7, d8 = m8;
        if (c.b1 != 0.f || c.b2 != 0.f || c.g7 != 0.f || c.g8 != 0.f) {   // MRT-B1/B2 only
            const float2 uyy = xmul2(uy, uy);
            const float2 u2 = fma2(ux, ux, uyy);
            d1 = fma2(xmul2(sp2(-c.b1), u2), phi, d1);
            d2 = fma2(xmul2(sp2(-c.b2), u2), phi, d2);
            d7 = fma2(xmul2(sp2(-c.g7), fma2(ux, ux, neg2(uyy))), phi, d7);
            d8 = fma2(xmul2(sp2(-c.g8), xmul2(ux, uy)), phi, d8);
        }
        float2 r0 = xmul2(sp2(c.A[0]), d3);
        r0 = fma2(sp2(c.C[0]), d4, r0);
        r0 = fma2(sp2(c.A[1]), d5, r0);
        r0 = fma2(sp2(c.C[1]), d6, r0);
        float2 r1 = xmul2(sp2(c.A[2]), d3);
        r1 = fma2(sp2(c.C[2]), d4, r1);
        r1 = fma2(sp2(c.A[3]), d5, r1);
        r1 = fma2(sp2(c.C[3]), d6, r1);
        const float2 a0 = xmul2(phi, sp2(1.f / 9.f));
        const float2 a1 = xmul2(fma2(sp2(-c.s[1]), d1, m1), sp2(1.f / 36.f));
        const float2 a2 = xmul2(fma2(sp2(-c.s[2]), d2, m2), sp2(1.f / 36.f));
        const float2 a3 = xmul2(sub2(m3, r0), sp2(1.f / 6.f));
        const float2 a4 = xmul2(fma2(sp2(-c.s[4]), d4, m4), sp2(1.f / 12.f));
        const float2 a5 = xmul2(sub2(m5, r1), sp2(1.f / 6.f));
        const float2 a6 = xmul2(fma2(sp2(-c.s[6]), d6, m6), sp2(1.f / 12.f));
        // 1/|M_7|^2 = 1/|M_8|^2 = 1/4: exact products, so fused below
        const float2 q7 = fma2(sp2(-c.s[7]), d7, m7), q8 = fma2(sp2(-c.s[8]), d8, m8);
        A = fma2(sp2(-2.f), a2, sub2(a0, a1));
        B = fma2(sp2(2.f), a1, add2(a0, a2));
        AP = fma2(sp2(0.25f), q7, A), AM = fma2(sp2(-0.25f), q7, A);
        BP = fma2(sp2(0.25f), q8, B), BM = fma2(sp2(-0.25f), q8, B);
        X = fma2(sp2(-2.f), a4, a3), Xd = add2(a3, a4);
        Y = fma2(sp2(-2.f), a6, a5), Yd = add2(a5, a6);
    }
    const float2 XY = add2(Xd, Yd), XmY = sub2(Xd, Yd);
    v[1] = add2(AP, X);
    v[3] = sub2(AP, X);
    v[2] = add2(AM, Y);
    v[4] = sub2(AM, Y);
    v[5] = add2(BP, XY);
    v[7] = sub2(BP, XY);
    v[6] = sub2(BM, XmY);
    v[8] = add2(BM, XmY);
    const float2 AB = add2(A, B);
    if constexpr (OFFSET) v[0] = fma2(sp2(-c.eps0), phi, mul2(sp2(-4.f), AB));   // Coef::eps0
    else v[0] = fma2(sp2(-4.f), AB, phi);                                         // 4 x exact
    return phi;
}

// f_i = g_i + phi f^eq_i(1, u) for a node pair (feq_unit<D2Q9>)
__device__ __forceinline__ void walk_feq(const Coef& c, float2 ux, float2 uy, float2 (&e)[9])
{
    const float2 s = add2(ux, uy), d = sub2(ux, uy);
    e[0] = sp2(c.w0);
    e[1] = fma2(sp2(c.ka), ux, sp2(c.wa));
    e[3] = fma2(sp2(-c.ka), ux, sp2(c.wa));
    e[2] = fma2(sp2(c.ka), uy, sp2(c.wa));
    e[4] = fma2(sp2(-c.ka), uy, sp2(c.wa));
    e[5] = fma2(sp2(c.kd), s, sp2(c.wd));
    e[7] = fma2(sp2(-c.kd), s, sp2(c.wd));
    e[8] = fma2(sp2(c.kd), d, sp2(c.wd));
    e[6] = fma2(sp2(-c.kd), d, sp2(c.wd));
}

constexpr int WALK_WARPS = 4;    // independent warps per CTA
__host__ __device__ constexpr int walk_minb(int T, bool walls) { return T <= 2 ? 4 : (walls ? 2 : 3); }   // 128 / 168 / up to 255 (walls) registers

// What a level keeps of its last two rows for the rows that still pull from
// them, unshifted: the e_y = 0 populations {0, 1, 3} of the last row and the
// e_y = +1 populations {2, 5, 6} of the last two (pa / pb, which change roles
// with every row, so that a row enters in place).
struct WalkLevel {
    float2 c0[3], pa[3], pb[3];
    float sb;   // x walls: the last row's e_y = -1 population that a bounce-back on x returns
};

__device__ __forceinline__ float2 walk_from_left(float2 v)    // the pair's values one column to the left
{
    return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x);
}
__device__ __forceinline__ float2 walk_from_right(float2 v)
{
    return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1));
}

// Shared memory of one warp: a ring of WALK_ROWS source rows and one of
// WALK_UROWS rows of the velocity factors. A source row is nine FP32 planes of
// 64 columns, or nine 16-bit planes of 72 columns (four more on each side, so
// that their 16-byte copies are aligned) and 64 columns of phi.
constexpr int WALK_ROWS = 4, WALK_AHEAD = 3;   // rows r .. r + 3: three in flight
constexpr int WALK_UROWS = 8;                  // rows r - 4 .. r + 3
template <int STORE>
struct WalkSlot {
    static constexpr bool neq = STORE != ST_F32;
    static constexpr int plane = neq ? 144 : 256;                   // bytes of a plane's staged row
    static constexpr int first = neq ? 8 : 0;                       // column 0 of the warp within it
    static constexpr int state = 9 * plane + (neq ? 256 : 0);       // bytes of a staged row
    static constexpr int gchunks = 9 * (plane / 16);                // 16-byte copies of the nine planes
    static constexpr int schunks = state / 16;                      // with phi
    __host__ __device__ static constexpr int chunks(bool field) { return schunks + (field ? 32 : 0); }
    __host__ __device__ static constexpr int warp(bool field) { return WALK_ROWS * state + (field ? WALK_UROWS * 512 : 0); }
};

template <int BYTES>
__device__ __forceinline__ void walk_copy(void* dst, const void* src)   // asynchronous, no registers held
{
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}

// SAVE: the FP32 states between are stored too (p.mid), for the reverse sweep.
// At T = 4 the levels need 168 registers: 12 warps per SM.
template <int STORE, bool FIELD, bool WALLS, int T, bool SAVE>
__global__ void __launch_bounds__(32 * WALK_WARPS, walk_minb(T, WALLS)) k_walk_d2q9(const __grid_constant__ WalkArgs p)
{
    using L = D2Q9;
    constexpr bool NEQ = STORE != ST_F32;
    static_assert(!SAVE || !NEQ, "only FP32 states are kept between the fused steps");
    static_assert(T + WALK_AHEAD < WALK_UROWS, "the ring holds the rows r - T .. r + WALK_AHEAD");
    constexpr float SC = STORE == ST_F16 ? F16_SCALE : 1.f;   // working units of the 16-bit forms (k_step_quad_d2q9)
    constexpr int HALO = WALK_HALO, COLS = WALK_COLS;
    static_assert(T <= HALO, "T columns on each side are lost");
    const StepArgs& a = p.a;
    const Coef& c = a.c;
    const int nx = a.nx, ny = a.ny;
    const int N = (int)a.ncell;
    extern __shared__ __align__(16) unsigned char walk_sm[];
    __shared__ float sched[T + 1][2];
    grid_dep_sync();
    const void* const asrc = after_dep(a.src);
    const float* const aua = after_dep(a.ua);
    if (threadIdx.x <= T) {
        float s[3];
        sched_row_at(after_dep(a.sched), p.srow[threadIdx.x], 2, s);
        sched[threadIdx.x][0] = s[0];
        sched[threadIdx.x][1] = s[1];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int w = blockIdx.x * WALK_WARPS + (threadIdx.x >> 5);
    int strip, range, ranges = p.ranges;
    if (WALLS && p.eranges > 0) {   // the strips with an x wall have more ranges
        const int inner = p.strips - 2, e = w - inner * p.ranges;
        if (e >= 2 * p.eranges) return;
        range = e < 0 ? w / inner : e >> 1;
        strip = e < 0 ? 1 + w - range * inner : ((e & 1) ? p.strips - 1 : 0);
        if (e >= 0) ranges = p.eranges;
    } else {
        if (w >= p.strips * p.ranges) return;
        range = w / p.strips, strip = w - range * p.strips;
    }
    const int ya = (int)((long long)range * ny / ranges), yb = (int)((long long)(range + 1) * ny / ranges);
    if (ya >= yb) return;
    const int x0 = strip * COLS - HALO + 2 * lane;   // even
    const bool xwall = WALLS && a.bcx_lo != BC_PERIODIC;
    int c0, c1;                                      // columns the lane loads
    if (xwall) {
        c0 = min(max(x0, 0), nx - 1);
        c1 = min(max(x0 + 1, 0), nx - 1);
    } else {
        c0 = x0 % nx;
        c0 = c0 < 0 ? c0 + nx : c0;
        c1 = c0 + 1 == nx ? 0 : c0 + 1;
    }
    const bool mine = lane >= HALO / 2 && lane < 32 - HALO / 2 && x0 < nx;
    const bool left = xwall && x0 == 0;
    const bool rx = xwall && x0 == nx - 1, ry = xwall && x0 + 1 == nx - 1;
    const bool edge = WALLS && __any_sync(0xffffffffu, left || rx || ry);
    const bool lb = left && a.bcx_lo == BC_BOUNCE, ln = left && a.bcx_lo == BC_NOFLUX, hb = a.bcx_hi == BC_BOUNCE;
    const bool ywall = WALLS && a.bc_lo != BC_PERIODIC;
    const int rs = ywall ? max(ya - T, 0) : ya - T, re = yb - 1 + T;

    using Slot = WalkSlot<STORE>;
    unsigned char* const sm = walk_sm + (threadIdx.x >> 5) * Slot::warp(FIELD);
    unsigned char* const smu = sm + WALK_ROWS * Slot::state;
    auto wrap = [&](int y) {   // grid row of walk row y
        if (ywall) return min(max(y, 0), ny - 1);
        y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
        if (y < 0 || y >= ny) y = ((y % ny) + ny) % ny;   // grids of fewer rows than the walk's halo
        return y;
    };
    // wide rows: the lane's 16-byte copies lane, lane + 32, ... of a staged row, their sources in row 0
    constexpr int CH = (Slot::chunks(FIELD) + 31) / 32;
    const unsigned char* from[CH];
#pragma unroll
    for (int k = 0; k < CH; ++k) {
        const int ch = lane + 32 * k;
        constexpr int per = Slot::plane / 16;
        const bool g16 = NEQ && ch < Slot::gchunks;
        int plane, col;                                        // columns relative to the strip's lane 0
        if (ch < Slot::gchunks) plane = ch / per, col = g16 ? 8 * (ch % per) - 4 : 4 * (ch % per);
        else plane = (ch - Slot::gchunks) / 16, col = 4 * ((ch - Slot::gchunks) % 16);
        col += strip * COLS - HALO;
        const int wide = g16 ? 8 : 4;
        if (xwall) col = min(max(col, 0), nx - wide);
        else {
            col %= nx;
            if (col < 0) col += nx;
        }
        const float* fp = NEQ ? a.phi_src : static_cast<const float*>(asrc);
        if (FIELD && ch >= Slot::schunks) fp = aua + (ch >= Slot::schunks + 16 ? N : 0);
        else if (!NEQ) fp += plane * N;
        from[k] = g16 ? reinterpret_cast<const unsigned char*>(static_cast<const unsigned short*>(asrc) + plane * N + col)
                      : reinterpret_cast<const unsigned char*>(fp + col);
    }
    auto issue = [&](int r) {   // stage walk row r
        if (r <= re) {
            const int row = wrap(r) * nx;
            unsigned char* st = sm + (r & (WALK_ROWS - 1)) * Slot::state;
            unsigned char* su = smu + (r & (WALK_UROWS - 1)) * 512;
            if (p.wide) {
#pragma unroll
                for (int k = 0; k < CH; ++k) {
                    const int ch = lane + 32 * k;
                    const bool g16 = NEQ && ch < Slot::gchunks;
                    if (32 * k + 31 < Slot::chunks(FIELD) || ch < Slot::chunks(FIELD))
                        walk_copy<16>(FIELD && ch >= Slot::schunks ? su + (ch - Slot::schunks) * 16 : st + ch * 16,
                                      from[k] + (size_t)(unsigned)(g16 ? 2 * row : 4 * row));
                }
            } else {
                auto copy_pair = [&](unsigned char* d, const float* q) {
                    walk_copy<4>(d, q + row + c0);
                    walk_copy<4>(d + 4, q + row + c1);
                };
                if constexpr (NEQ) {   // no 4-byte copy can start at an odd 16-bit word
                    const unsigned short* q = static_cast<const unsigned short*>(asrc);
                    unsigned g[9];
#pragma unroll
                    for (int i = 0; i < 9; ++i)
                        g[i] = (unsigned)ld_dep(q + i * N + row + c0) | (unsigned)ld_dep(q + i * N + row + c1) << 16;
#pragma unroll
                    for (int i = 0; i < 9; ++i)
                        *reinterpret_cast<unsigned*>(st + Slot::plane * i + Slot::first + 4 * lane) = g[i];
                    copy_pair(st + 9 * Slot::plane + 8 * lane, a.phi_src);
                } else {
#pragma unroll
                    for (int i = 0; i < 9; ++i)
                        copy_pair(st + Slot::plane * i + 8 * lane, static_cast<const float*>(asrc) + i * N);
                }
                if (FIELD) {
                    copy_pair(su + 8 * lane, aua);
                    copy_pair(su + 256 + 8 * lane, aua + N);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float rux[T + 1], ruy[T + 1];   // row profile: the velocity factors of the rows r .. r - T
#pragma unroll
    for (int s = 0; s <= T; ++s) rux[s] = ruy[s] = 0.f;
    auto velocity = [&](int y, int s, float2& ux, float2& uy) {   // velocity factors of walk row y = r - s
        if (!FIELD) {
            ux = sp2(rux[s]);
            uy = sp2(ruy[s]);
        } else {
            const unsigned char* su = smu + (y & (WALK_UROWS - 1)) * 512 + 8 * lane;
            ux = *reinterpret_cast<const float2*>(su);
            uy = *reinterpret_cast<const float2*>(su + 256);
        }
    };

    WalkLevel lv[T];
#pragma unroll
    for (int s = 0; s < T; ++s) {
        lv[s].sb = 0.f;
#pragma unroll
        for (int j = 0; j < 3; ++j) lv[s].c0[j] = lv[s].pa[j] = lv[s].pb[j] = sp2(0.f);
    }

#pragma unroll 1
    for (int j = 0; j < WALK_AHEAD; ++j) issue(rs + j);

    // Rows next to a y wall, and the strips with an x wall, run their own instances: the branches of the wall
    // rules between the levels cost all other rows their overlap (4096^2 between Neumann walls: 125 us a
    // step with them in place, 77 without)
    auto row_step = [&](int r, auto par, auto rule) {   // rule: 0 none, 1 x walls, 2 y walls (x walls if edge)
        constexpr bool SLOW = decltype(rule)::value == 2, EDGE = WALLS && decltype(rule)::value > 0;
        constexpr bool ODD = decltype(par)::value != 0;
        float2 n[9];
        asm volatile("cp.async.wait_group %0;" ::"n"(WALK_AHEAD - 1) : "memory");
        if (!FIELD && aua != nullptr) {
#pragma unroll
            for (int s = T; s > 0; --s) rux[s] = rux[s - 1], ruy[s] = ruy[s - 1];
            const int y = wrap(r);
            rux[0] = __ldg(aua + y);
            ruy[0] = __ldg(aua + ny + y);
        }
        __syncwarp();   // row r has landed for every lane, and every lane is done with row r - 1
        {
            const unsigned char* st = sm + (r & (WALK_ROWS - 1)) * Slot::state;
            if constexpr (NEQ) {
                using P = Pair<STORE>;
                using Q = QuadH<STORE>;
                float2 ax, ay, e[9];
                velocity(r, 0, ax, ay);
                walk_feq(c, xmul2(ax, sp2(sched[0][0])), xmul2(ay, sp2(sched[0][1])), e);
                const float2 phi = xmul2(*reinterpret_cast<const float2*>(st + 9 * Slot::plane + 8 * lane), sp2(SC));
#pragma unroll
                for (int i = 0; i < 9; ++i)
                    n[i] = fma2(phi, e[i], P::to_f_raw(Q::as_t2(*reinterpret_cast<const unsigned*>(st + Slot::plane * i + Slot::first + 4 * lane))));
            } else {
#pragma unroll
                for (int i = 0; i < 9; ++i) n[i] = *reinterpret_cast<const float2*>(st + Slot::plane * i + 8 * lane);
            }
        }
        issue(r + WALK_AHEAD);
#pragma unroll
        for (int s = 1; s <= T; ++s) {
            // row r - s + 1 of level s - 1 has come in (n); level s computes row y
            WalkLevel& lw = lv[s - 1];
            float2(&p1)[3] = ODD ? lw.pb : lw.pa;   // e_y = +1 populations of row y, and of row y - 1
            float2(&p2)[3] = ODD ? lw.pa : lw.pb;
            const int y = r - s;
            float2 ax, ay;
            velocity(y, s, ax, ay);
            float2 f[9];
            f[0] = lw.c0[0];
            f[1] = walk_from_left(lw.c0[1]);
            f[3] = walk_from_right(lw.c0[2]);
            f[2] = p2[0];
            f[5] = walk_from_left(p2[1]);
            f[6] = walk_from_right(p2[2]);
            f[4] = n[4];
            f[7] = walk_from_right(n[7]);
            f[8] = walk_from_left(n[8]);
            if constexpr (SLOW || EDGE) {
                // the rules of k_step_box, in its order of precedence: bounce-back on y, on x, then the
                // mirror rule on x, on y, then Dirichlet
                const bool lo = SLOW && ywall && y == 0, hi = SLOW && ywall && y == ny - 1;
                const int kind = lo ? a.bc_lo : a.bc_hi;
                if ((lo || hi) && kind == BC_BOUNCE) {
                    if (lo) {      // stashed when row 0 came in
                        f[2] = p2[0];
                        f[5] = p2[1];
                        f[6] = p2[2];
                    } else {
                        f[4] = p1[0];
                        f[7] = p1[1];
                        f[8] = p1[2];
                    }
                }
                if (EDGE) {   // selects, no branches
                    f[1].x = lb ? lw.c0[2].x : (ln ? f[3].x : f[1].x);
                    f[5].x = lb ? lw.sb : (ln ? f[6].x : f[5].x);
                    f[8].x = lb ? p1[2].x : (ln ? f[7].x : f[8].x);
                    const float3 rv = rx ? make_float3(hb ? lw.c0[1].x : f[1].x, hb ? lw.sb : f[5].x, hb ? p1[1].x : f[8].x)
                                         : make_float3(hb ? lw.c0[1].y : f[1].y, hb ? lw.sb : f[5].y, hb ? p1[1].y : f[8].y);
                    f[3].x = rx ? rv.x : f[3].x, f[6].x = rx ? rv.y : f[6].x, f[7].x = rx ? rv.z : f[7].x;
                    f[3].y = ry ? rv.x : f[3].y, f[6].y = ry ? rv.y : f[6].y, f[7].y = ry ? rv.z : f[7].y;
                    lw.sb = left ? n[7].x : (rx ? n[8].x : n[8].y);
                }
                if (lo || hi) {
                    if (kind == BC_NOFLUX) {
                        if (lo) f[2] = f[4], f[5] = f[8], f[6] = f[7];
                        else f[4] = f[2], f[8] = f[5], f[7] = f[6];
                    } else if (kind == BC_DIRICHLET) {
                        float2 e[9];
                        walk_feq(c, xmul2(ax, sp2(sched[s - 1][0])), xmul2(ay, sp2(sched[s - 1][1])), e);
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
            p2[0] = n[2], p2[1] = n[5], p2[2] = n[6];   // the next row's p1
            lw.c0[0] = n[0], lw.c0[1] = n[1], lw.c0[2] = n[3];
            if (SLOW && ywall && y == -1 && a.bc_lo == BC_BOUNCE) p1[0] = n[4], p1[1] = n[7], p1[2] = n[8];

            // a product that only feeds products may be paired; u also feeds sums in the 16-bit decode
            const float2 ux = NEQ ? xmul2(ax, sp2(sched[s][0])) : mul2(ax, sp2(sched[s][0]));
            const float2 uy = NEQ ? xmul2(ay, sp2(sched[s][1])) : mul2(ay, sp2(sched[s][1]));
            const float2 phi = walk_collide<NEQ>(f, ux, uy, c);
            const bool keep = mine && y >= ya && y < yb;
            if constexpr (NEQ) {
                using P = Pair<STORE>;
                using Q = QuadH<STORE>;
                unsigned g[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) g[i] = Q::as_u(P::from_f_raw(f[i]));
                if (s < T) {       // the offsets as they would be stored, decoded with u of this step
                    float2 e[9];
                    walk_feq(c, ux, uy, e);
#pragma unroll
                    for (int i = 0; i < 9; ++i) n[i] = fma2(phi, e[i], P::to_f_raw(Q::as_t2(g[i])));
                } else if (keep) {
                    unsigned short* q = static_cast<unsigned short*>(a.dst) + y * nx + x0;
                    float* pq = a.phi_dst + y * nx + x0;
                    const float2 ph = xmul2(phi, sp2(1.f / SC));
                    if (p.vec) {
#pragma unroll
                        for (int i = 0; i < 9; ++i) *reinterpret_cast<unsigned*>(q + i * N) = g[i];
                        *reinterpret_cast<float2*>(pq) = ph;
                    } else {
                        const bool two = x0 + 1 < nx;
#pragma unroll
                        for (int i = 0; i < 9; ++i) {
                            q[i * N] = (unsigned short)(g[i] & 0xffffu);
                            if (two) q[i * N + 1] = (unsigned short)(g[i] >> 16);
                        }
                        pq[0] = ph.x;
                        if (two) pq[1] = ph.y;
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < 9; ++i) n[i] = f[i];
                if ((s == T || SAVE) && keep) {
                    float* q = static_cast<float*>(s == T ? a.dst : p.mid[s < 4 ? s - 1 : 0]) + y * nx + x0;
                    if (p.vec) {
#pragma unroll
                        for (int i = 0; i < 9; ++i) *reinterpret_cast<float2*>(q + i * N) = f[i];
                    } else {
                        const bool two = x0 + 1 < nx;
#pragma unroll
                        for (int i = 0; i < 9; ++i) {
                            q[i * N] = f[i].x;
                            if (two) q[i * N + 1] = f[i].y;
                        }
                    }
                }
            }
        }
    };
#pragma unroll 1
    for (int r = rs; r <= re; r += 2) {   // the row past re, where there is one, computes nothing that is kept
        auto two = [&](auto rule) {
            row_step(r, std::integral_constant<int, 0>{}, rule);
            row_step(r + 1, std::integral_constant<int, 1>{}, rule);
        };
        if (WALLS && ywall && (r - T <= 0 || r >= ny - 1)) two(std::integral_constant<int, WALLS ? 2 : 0>{});
        else if (edge) two(std::integral_constant<int, WALLS ? 1 : 0>{});
        else two(std::integral_constant<int, 0>{});
    }
}

template <int STORE, bool FIELD, bool WALLS, int T, bool SAVE>
cudaError_t walk_d2q9(WalkArgs& p, cudaStream_t st)
{
    constexpr int smem = WALK_WARPS * WalkSlot<STORE>::warp(FIELD);
    static std::atomic<unsigned> known[64];
    KernelFit fit;
    const cudaError_t fe = kernel_fit(known, k_walk_d2q9<STORE, FIELD, WALLS, T, SAVE>, 32 * WALK_WARPS, smem, fit);
    if (fe != cudaSuccess) return fe;
    p.strips = (p.a.nx + WALK_COLS - 1) / WALK_COLS;
    p.ranges = walk_ranges(p.strips, p.a.ny, T, fit.sms, fit.per_sm * WALK_WARPS, nullptr);
    int warps = p.strips * p.ranges;
    if (WALLS && p.a.bcx_lo != BC_PERIODIC && p.strips >= 3) {
        // a row of a strip with an x wall takes about 1.6 times as long (selects in every level)
        const int most = fit.sms * fit.per_sm * WALK_WARPS;
        auto total = [&] { return (p.strips - 2) * p.ranges + 2 * p.eranges; };
        p.eranges = (8 * p.ranges + 4) / 5;
        while (p.ranges > 1 && total() > most) p.eranges = (8 * --p.ranges + 4) / 5;
        if (p.eranges > p.a.ny) p.eranges = p.a.ny;
        warps = total();
    }
    const int ctas = (warps + WALK_WARPS - 1) / WALK_WARPS;
    return launch_dependent(k_walk_d2q9<STORE, FIELD, WALLS, T, SAVE>, dim3((unsigned)ctas), dim3(32 * WALK_WARPS), smem, st, p);
}

template <int STORE, bool FIELD, int T, bool SAVE>
cudaError_t walk_w(WalkArgs& p, cudaStream_t st)
{
    const bool walls = p.a.bc_lo != BC_PERIODIC || p.a.bcx_lo != BC_PERIODIC;
    return walls ? walk_d2q9<STORE, FIELD, true, T, SAVE>(p, st)
                 : walk_d2q9<STORE, FIELD, false, T, SAVE>(p, st);
}

}  // namespace lbm
