// Internal declarations shared by the CUDA translation units of the solver.
// Not part of the public C ABI (include/lbm_cde.h).
#pragma once

#include <cuda.h>            // CUtensorMap (tensor maps of the TMA-staged step)
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <atomic>
#include <type_traits>

namespace lbm {

enum Store { ST_F32 = 0, ST_F16 = 1, ST_BF16 = 2 };
enum UKind { U_NONE = 0, U_FIELD = 1, U_ROW = 2 };
enum Bc { BC_PERIODIC = 0, BC_NOFLUX = 1, BC_BOUNCE = 2, BC_DIRICHLET = 3 };

// Relaxation and equilibrium constants of one solver, passed by value to
// every kernel (they live in the kernel parameter bank, i.e. constant cache).
struct Coef {
    // m^eq per unit phi for the two scalar moments:
    //   D2Q9  (Eq. 15b-c): m1 = alpha1/4, m2 = alpha2/4
    //   D3Q15 (Eq. A.3b-c): m1 = 5 alpha1/6, m2 = alpha2/24
    float meq1, meq2;
    float s[15];   // diagonal rates (entries 3, 5, 7 unused)
    float A[9];    // flux block (row-major dim x dim)
    // Coupling of flux row a to q-moment column b (Eq. 30a-b, A.5):
    //   (A_ab / 2 - delta_ab) * s_{q-row of b}
    float C[9];
    // f^eq_i = phi * (w_i + k_i e_i.u), Eq. 17 / its D3Q15 counterpart
    float w0, wa, wd, ka, kd;
    // u^2 terms of the MRT-B1/B2 equilibria (Eq. 38-39), zero for MRT-A/B3:
    //   m1 += b1 |u|^2 phi, m2 += b2 |u|^2 phi, m7 = g7 (ux^2 - uy^2) phi, m8 = g8 ux uy phi
    float b1, b2, g7, g8;
    // Offset forms (linear equilibria): the relaxation and the 1/|M_k|^2
    // scaling folded together, a_k = (m' - m^eq)_k / |M_k|^2 from dl = m - m^eq:
    //   ro[k] = (1 - s_k) / |M_k|^2 for the diagonal rows;
    //   D2Q9: fr[4 r + j], flux row 3 + 2 r on dl_3, dl_4, dl_5, dl_6
    //         ((delta_r0 - A_r0) / 6, -C_r0 / 6, (delta_r1 - A_r1) / 6, -C_r1 / 6);
    //   D3Q15: fr[6 r + 2 b + j], flux row 3 + 2 r on dl_{3 + 2 b} (j = 0) and
    //         dl_{4 + 2 b} (j = 1): (delta_rb - A_rb) / |M_3|^2, -C_rb / |M_3|^2
    float ro[15];
    float fr[18];
    // sum_i w_i - 1 with the FP32 weights the 16-bit decode adds back (w0 + 4 wa
    // + 4 wd for D2Q9, w0 + 6 wa + 8 wd for D3Q15): the rest offset g_0 carries
    // -phi eps0 so that decode and store conserve mass in FP32 as they do exactly
    float eps0;
};

// Fills ro and fr from s, A and C (D2Q9 or D3Q15; host side).
inline void fold_offset_coef(Coef& c, int q = 9)
{
    if (q == 9) {
        const double n2[9] = {9, 36, 36, 6, 12, 6, 12, 4, 4};
        for (int k = 0; k < 9; ++k) c.ro[k] = (float)((1.0 - (double)c.s[k]) / n2[k]);
        for (int r = 0; r < 2; ++r) {
            c.fr[4 * r + 0] = (float)(((r == 0 ? 1.0 : 0.0) - (double)c.A[2 * r + 0]) / 6.0);
            c.fr[4 * r + 1] = (float)(-(double)c.C[2 * r + 0] / 6.0);
            c.fr[4 * r + 2] = (float)(((r == 1 ? 1.0 : 0.0) - (double)c.A[2 * r + 1]) / 6.0);
            c.fr[4 * r + 3] = (float)(-(double)c.C[2 * r + 1] / 6.0);
        }
        return;
    }
    // D3Q15 row norms |M_k|^2 of Eq. A.2
    const double n2[15] = {15, 18, 360, 10, 40, 10, 40, 10, 40, 12, 4, 8, 8, 8, 8};
    for (int k = 0; k < 15; ++k) c.ro[k] = (float)((1.0 - (double)c.s[k]) / n2[k]);
    for (int r = 0; r < 3; ++r)
        for (int b = 0; b < 3; ++b) {
            c.fr[6 * r + 2 * b] = (float)(((r == b ? 1.0 : 0.0) - (double)c.A[3 * r + b]) / n2[3]);
            c.fr[6 * r + 2 * b + 1] = (float)(-(double)c.C[3 * r + b] / n2[3]);
        }
}

// Tensor maps of the TMA-staged D2Q9 step (k_step_tma_d2q9) for one source
// buffer: each pair is the 256-column box of one grid row and its halo box.
struct TmaMaps {
    CUtensorMap g, gh;    // 16-bit offsets [9][ny][nx]: boxes (256, 1, 9) and (8, 1, 9)
    CUtensorMap p, ph;    // phi [ny][nx]: boxes (256, 1) and (4, 1)
    CUtensorMap u, uh;    // velocity factors [2][ny][nx]: boxes (256, 1, 2) and (4, 1, 2)
};

struct StepArgs {
    const void* src;      // state planes [q][ncell] (float or 16-bit)
    void* dst;
    const float* phi_src; // phi planes of the 16-bit forms
    float* phi_dst;
    const float* ua;      // velocity a(x) (FIELD: [dim][ncell], ROW: [dim][ny])
    const float* sched;   // [sched_len][dim] or nullptr
    long long sched_len;
    long long k;          // this step computes f(k) and collides with u(k)
    int srow_now;         // schedule rows of u(k) and u(k-1): k mod sched_len,
    int srow_prev;        // (k-1) mod sched_len, or -1 without a schedule
    int nx, ny, nz;
    long long ncell;
    int bc_lo, bc_hi;     // y faces
    float phiw_lo, phiw_hi;
    int bcx_lo, bcx_hi;   // x faces (k_step_box only)
    int bcz_lo, bcz_hi;   // z faces (k_step_box only)
    Coef c;
    int* status;          // device status word (LBM_E_TIMEOUT from a bounded wait) or nullptr
    long long spin_limit; // SM clock cycles a bounded wait may take (0: give up at once)
    const TmaMaps* tma;   // host pointer: tensor maps of src / phi_src / ua, or nullptr
    int zwalk;            // D3Q15 z-walk kernel: planes per CTA (0: chosen by the launcher)
};

// Several fused D2Q9 steps (lbm_walk_d2q9.cuh).
struct WalkArgs {
    StepArgs a;          // src: state k - 1; dst: state k - 1 + T
    int srow[5];         // schedule rows of u(k - 1) .. u(k - 1 + T), or -1
    void* mid[3];        // SAVE: the states k .. k + T - 2 (FP32)
    int strips, ranges;  // strips of WALK_COLS columns x ranges of rows
    int eranges;         // ranges of the first and the last strip where they have an x wall, or 0
    int vec;             // pairs are stored as one word (nx even, aligned planes)
    int wide;            // rows are staged by 16-byte copies (nx a multiple of 4, or 8 for 16-bit planes; aligned)
};

// Steps of the D2Q9 model on tiles in shared memory (lbm_tile_d2q9.cuh).
constexpr int TILE_T = 8;        // most steps of one launch
constexpr int TILE_ROWS = 64;    // most rows of a tile
struct TileArgs {
    StepArgs a;              // src: state k - 1; dst: state k - 1 + T
    int srow[TILE_T + 1];    // schedule rows of u(k - 1) .. u(k - 1 + T), or -1
    void* mid[TILE_T - 1];   // FP32: where the states between go, or NULL
    int T;                   // steps
    int rows;                // tile: 64 columns x rows, the halo of T on each side included
    int field;               // a.ua is a field (else a row profile, or NULL)
};

// The fused D2Q9 steps need int offsets.
inline bool fused_ok(int q, long long ncell) { return q == 9 && 12LL * ncell < (1LL << 31); }

constexpr int WALK_HALO = 4;     // columns of a warp's 64 lost on each side: at least T, and a multiple of 4 so
                                 // that strips start on 16-byte boundaries
constexpr int WALK_COLS = 64 - 2 * WALK_HALO;

// Ranges of rows of the walk kernel for at most `warps` resident warps per SM,
// and its time of one launch in us (cost, may be NULL). Measured on GB300: a row
// takes about 0.45 us + 0.47 us k at T = 4 with k >= 1 warps per scheduler
// (1024^2: 0.92, 1.33, 1.87 us at k = 1, 2, 3); a range of R rows walks R + 2 T.
int walk_ranges(int strips, int ny, int T, int sms, int warps, double* cost);

// How the next of `left` D2Q9 steps run: T steps by one launch of the one-step
// kernel (T = 1), of the walk kernel (rows = 0) or of the tile kernel (rows of a tile).
struct FusePlan { int T, rows; };
enum { FUSE_WALK = 1, FUSE_TILE = 2, FUSE_ANY = 3 };   // kernels the plan may take (one: at least two steps by it)
FusePlan plan_fused(int store, int nx, int ny, bool walls, int sms, long long left, int kinds = FUSE_ANY);

// One reverse-time step (lbm_adjoint.cu).
struct AdjArgs {
    const float* mu_in;   // adjoint of the post-collision state B_k [q][ncell]
    float* mu_out;        // adjoint of B_{k-1}
    const float* fprev;   // forward state B_{k-1} (FP32) [q][ncell]
    const float* ua;
    const float* sched;
    long long sched_len;
    long long k;          // the forward step being reversed (collision with u(k))
    int srow;             // k mod sched_len, or -1 without a schedule
    int srow_prev;        // (k - 1) mod sched_len, or -1: u(k - 1) of the Dirichlet fill
    float phiw_lo, phiw_hi;   // Dirichlet wall values (y faces)
    int rows;             // grid rows per row of threads of a block (adjoint_rows)
    int nx, ny, nz;
    long long ncell;
    int bc_lo, bc_hi;     // y faces
    int bcx_lo, bcx_hi;   // x faces (wall mode 2)
    int bcz_lo, bcz_hi;   // z faces (wall mode 2)
    Coef c;
    float* du_acc;        // dL/da accumulator [dim][ncell] (FIELD velocity) or nullptr
    float* partials;      // per-block gradient partials [ngrad][nblocks] (one slice per step)
    float2* grad_acc;     // [ngrad] running compensated sums (value = x + y): G_A[dim][dim],
                          // G_AC[dim][dim], G_diag[q]
};

// Row of a schedule of length len for step k (k mod len), -1 without one;
// computed on the host so that no kernel divides by the schedule length.
inline int sched_row(long long k, long long len)
{
    if (len <= 0) return -1;
    long long r = k % len;
    return (int)(r < 0 ? r + len : r);
}

inline void set_step(StepArgs& a, long long k)
{
    a.k = k;
    a.srow_now = sched_row(k, a.sched ? a.sched_len : 0);
    a.srow_prev = sched_row(k - 1, a.sched ? a.sched_len : 0);
}

// The node-quad D2Q9 kernel needs nx % 4 == 0, int offsets and a 16-byte
// aligned velocity field (it reads four nodes per vector load).
inline bool quad_ok(const StepArgs& a, int ukind)
{
    return a.nx % 4 == 0 && a.nz == 1 && 12LL * a.ncell < (1LL << 31) &&
           (ukind != U_FIELD || (reinterpret_cast<uintptr_t>(a.ua) & 15) == 0);
}

// The node-pair kernels need nx even, int offsets ((q + 3) ncell < 2^31) and
// an 8-byte aligned velocity field (they read two nodes per vector load).
inline bool pair_ok(const StepArgs& a, int ukind, int q)
{
    return a.nx % 2 == 0 && (long long)(q + 3) * a.ncell < (1LL << 31) &&
           (ukind != U_FIELD || (reinterpret_cast<uintptr_t>(a.ua) & 7) == 0);
}

// The TMA-staged D2Q9 kernel needs 256-column strips (nx % 256 == 0), int
// offsets, a 16-byte aligned velocity field and the tensor maps of the source.
inline bool tma_ok(const StepArgs& a, int ukind)
{
    return a.tma != nullptr && a.nx % 256 == 0 && a.nz == 1 && 12LL * a.ncell < (1LL << 31) &&
           (ukind != U_FIELD || (reinterpret_cast<uintptr_t>(a.ua) & 15) == 0);
}

// The D3Q15 z-walk kernel needs 64-column tiles (nx % 64 == 0), ty-row tiles
// (ny % ty == 0), int offsets and 16-byte aligned offsets, phi and velocity
// fields (its shared-memory fills are 16-byte copies).
inline bool zw_ok(const StepArgs& a, int ukind, int ty)
{
    return a.nx % 64 == 0 && a.ny % ty == 0 && 18LL * a.ncell < (1LL << 31) &&
           (reinterpret_cast<uintptr_t>(a.phi_src) & 15) == 0 && (reinterpret_cast<uintptr_t>(a.src) & 15) == 0 &&
           (ukind != U_FIELD || (reinterpret_cast<uintptr_t>(a.ua) & 15) == 0);
}

// Encode the tensor maps for one source buffer (lbm_tma.cu); false if the
// driver entry point is missing or the layout breaks a tensor-map rule.
bool encode_tma_maps(const void* g, const float* phi, const float* ua, int nx, int ny, TmaMaps* out);

struct LaunchCfg {
    int block;   // threads per block (multiple of 32)
    int vec;     // cells per thread along x (1, 2 or 4)
};

// Programmatic dependent launch. A kernel waits for the one before it before its
// first read, and only then lets the next one start, so that no more than two are
// in flight: the next one's launch drops what the L1 caches held from before the
// kernel that is still writing. What that kernel writes is read with ld_dep (or
// cp.async): __ldg and the loads the compiler makes of it promise data that nothing
// writes while the kernel exists, and were seen to return the state of two steps before.
__device__ __forceinline__ void grid_dep_sync()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ float ld_dep(const float* p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 ld_dep(const float2* p)
{
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned ld_dep(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned short ld_dep(const unsigned short* p)
{
    unsigned short v;
    asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}
// A pointer whose read-only loads (__ldg, for what the caller owns) stay behind grid_dep_sync().
template <class P>
__device__ __forceinline__ P after_dep(P p)
{
    unsigned long long v = reinterpret_cast<unsigned long long>(p);
    asm volatile("" : "+l"(v)::"memory");
    return reinterpret_cast<P>(v);
}

// The forms a one-step kernel reads its source in. The first two are for dependent
// launches; which one a kernel takes was measured (the compiler places, merges and
// addresses their loads differently): see the launchers.
//   LD_ORDERED:  ld_dep, and __ldg of pointers that went through after_dep()
//   LD_PLAIN:    plain loads (velocity too). They stay behind grid_dep_sync(), which clobbers
//                memory, and no pointer in the kernel is __restrict__ or read in another type than
//                it is written in, so that nothing tells the compiler that the data is read-only
//   LD_READONLY: __ldg throughout, no wait: for ordinary launches, which start when the
//                previous kernel has ended
enum { LD_ORDERED = 0, LD_PLAIN = 1, LD_READONLY = 2 };

template <int LD, class T>
__device__ __forceinline__ T ld_src(const T* p)
{
    if constexpr (LD == LD_ORDERED) return ld_dep(p);
    else if constexpr (LD == LD_PLAIN) return *p;
    else return __ldg(p);
}
template <int LD, class T>
__device__ __forceinline__ T ld_vel(const T* p)   // what the caller owns
{
    if constexpr (LD == LD_PLAIN) return *p;
    else return __ldg(p);
}

// The arguments a kernel of form LD works with: a copy whose pointers went through
// after_dep(), or the kernel parameters themselves (as uniform operands).
template <int LD>
using StepArgsLD = typename std::conditional<LD == LD_ORDERED, StepArgs, const StepArgs&>::type;
template <int LD>
__device__ __forceinline__ void step_after_dep(StepArgsLD<LD>& a)
{
    if constexpr (LD != LD_READONLY) grid_dep_sync();
    if constexpr (LD == LD_ORDERED) {
        a.src = after_dep(a.src);
        a.phi_src = after_dep(a.phi_src);
        a.ua = after_dep(a.ua);
        a.sched = after_dep(a.sched);
    }
}

// A launch that may start while the stream's previous kernel drains: it waits
// in grid_dep_sync() before it reads anything. From launch to launch of dependent
// kernels: D3Q15 40^3 4.6 -> 3.4 us a step, 64^3 8.2 -> 5.8, 97 x 80 x 66 12.4 -> 10.2.
// overlap = false: an ordinary launch (LD_READONLY).
template <class A>
cudaError_t launch_dependent(void (*kernel)(A), dim3 grid, dim3 block, int smem, cudaStream_t st, const A& args,
                             bool overlap = true)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args);
}

// How a kernel with dynamic shared memory fits the current device: its multiprocessors and the CTAs each holds. Asked
// once per kernel and device (`known`, one per instantiation) and published as one word, so that threads with handles
// of their own see all of it or ask themselves; an error is returned and nothing remembered.
struct KernelFit { int sms, per_sm; };
template <class K>
cudaError_t kernel_fit(std::atomic<unsigned> (&known)[64], K* kernel, int threads, int smem, KernelFit& fit)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    unsigned w = dev < 64 ? known[dev].load(std::memory_order_acquire) : 0;
    if (w == 0) {
        int sms = 0, per_sm = 0;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
        if (e != cudaSuccess) {
            cudaGetLastError();   // returned, not left for the next call
            return e;
        }
        w = (unsigned)(sms > 0 ? sms : 1) << 16 | (unsigned)(per_sm > 0 ? per_sm : 1);
        if (dev < 64) known[dev].store(w, std::memory_order_release);
    }
    fit = {(int)(w >> 16), (int)(w & 0xffffu)};
    return cudaSuccess;
}

// Kernel launchers (lbm_kernels.cu). Each returns the cudaError_t of the launch.
cudaError_t launch_step(int q, int store, int ukind, bool walls, LaunchCfg cfg,
                        const StepArgs& a, cudaStream_t st);
// T (2 or 4) fused D2Q9 steps from a.src to a.dst; mid: the T - 1 states between
// (FP32 storage), or nullptr
cudaError_t launch_walk(int store, int ukind, int T, const StepArgs& a, void* const* mid, cudaStream_t st);
// T (1 .. TILE_T) D2Q9 steps on tiles of the given rows in shared memory, likewise
cudaError_t launch_tile(int store, int ukind, int T, int rows, const StepArgs& a, void* const* mid, cudaStream_t st);
cudaError_t launch_init(int q, int store, int ukind, const float* phi0, const StepArgs& a,
                        cudaStream_t st);
cudaError_t launch_phi(int q, int store, const StepArgs& a, float* phi_out, cudaStream_t st);
cudaError_t launch_sum(int q, int store, const StepArgs& a, double* partials, int nblocks,
                       double* out_dev, cudaStream_t st);

// reduce = true: also add the block partials to grad_acc (one step at a time);
// a backward sweep writes the partials of up to ADJ_SLICES consecutive steps to
// separate slices (AdjArgs::partials = base + slice * adjoint_slice_size) and
// reduces them together with launch_grad_reduce.
// wmode: 0 periodic, 1 walls on the y faces only, 2 walls on x or z faces (any face)
cudaError_t launch_adjoint(int q, int ukind, int wmode, const AdjArgs& a, cudaStream_t st, bool reduce);
cudaError_t launch_grad_reduce(int q, const AdjArgs& a, float* base, int nslice, long long slice, cudaStream_t st);
long long adjoint_slice_size(int q, long long nx, long long ny, long long nz, int sms);
constexpr int ADJ_SLICES = 16;   // reverse steps whose block partials are kept apart before one reduction
cudaError_t launch_adjoint_init(int q, int ukind, const AdjArgs& a, const float* phi0, float* dphi0,
                                cudaStream_t st);
cudaError_t launch_adjoint_seed(const float* g, float* mu, long long ncell, int q, cudaStream_t st);
long long adjoint_partials_size(int q, long long nx, long long ny, long long nz, int sms);   // in floats
struct AdjBlock { int w, h; };   // threads of a block: columns x rows
AdjBlock adjoint_block(long long nx);
int adjoint_rows(long long nx, long long ny, long long nz, int sms);
int adjoint_ngrad(int q);

}  // namespace lbm
