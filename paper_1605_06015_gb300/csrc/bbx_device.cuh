// Device-side building blocks of the sm_103a monodomain step: TMA/mbarrier
// wrappers (inline PTX), the cell models, and the fused step kernel template.
//
// The step kernel is one pass of the paper's unsplit scheme (section
// "Computation of intermediate expressions": diff followed by euler /
// rushlarsen) for every tissue node of a brick list:
//   - 2.5D z-marching over columns of 64 x TY nodes; a producer warp stages each
//     z-plane of V (with a one-node halo, widened in x to the 16-byte TMA rule)
//     in one ring of shared memory and each computed plane's own fibres, W-tilde
//     sums, other variables and (masked grids) neighbour words in a second one,
//     by cp.async.bulk.tensor on mbarriers, ahead of the consumer warps;
//   - the operator of Eq. (Lu) is formed from differences of V, the node's unit
//     fibre, Eq. (sigma), and the W-tilde sums, computed once per grid; its
//     weights are not stored;
//   - the arithmetic runs on pairs of x-adjacent nodes (packed FP32: one issue
//     slot a pair), every operation with its rounding named, so that a node's
//     result does not depend on the tile shape or the kernel variant;
//   - the reaction update (Eq. (Euler) for V and non-gates, Eq. (RL) for
//     gates) is fused, the new state is stored straight from registers;
//   - the activation map is written on the first upward crossing only;
//   - the sum of the new V over tissue nodes is reduced in the same pass
//     (compensated float pairs per thread and warp, one double per piece;
//     the fixed-order sum of the pieces when the total is read, or at the
//     end of a batch launch).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

#include "../../include/bbx.h"

namespace bbx {

// ---------------------------------------------------------------------------
// launch arguments
// ---------------------------------------------------------------------------

enum : int { ERRBIT_TIMEOUT = 1, ERRBIT_NAN = 2, ERRBIT_HINT = 4 };

// Device-updated state of one grid: written once per launch, by the CTA that
// takes the last start ticket (single-grid launch) or by the last CTA to
// finish (batch launch), and by the on-demand sum of a pending total.
struct TissueDyn {
    double t;       // model time t_n
    double total;   // tissue sum of V after the most recent step
    long long n;    // steps taken
    int cur;        // buffer holding the current state (0 or 1)
    int total_pending;  // not 0: total is still to be summed from the per-piece
                        // partials of the grid's last single-grid launch (1, 2:
                        // of which of the grid's plans)
};

// Host-written description of one grid for the step kernel (in device memory,
// so that one launch, or one graph node, can serve any number of grids).
struct TissueArgs {  // (CUtensorMap members impose its alignment)
    CUtensorMap tm_u[2];  // V of buffer b with halo (box TX+8 x TY+2)
    CUtensorMap tm_s[2];  // non-diffusing variables of buffer b (box TX x TY x S-1; with 16-bit gates: Ca only)
    CUtensorMap tm_g[2];  // 16-bit gates of buffer b (box TX x TY x 6 uint16), when stored so
    CUtensorMap tm_f;     // unit fibres (box TX x TY x 3, no halo)
    CUtensorMap tm_d;     // the W-tilde sums of every node (box TX x TY x 3)
    CUtensorMap tm_m;     // neighbour words of a masked grid (box TX x TY, no halo)
    float* state[2];      // the ping-pong buffers, var v at state[b] + v*vol (32-bit variables)
    uint16_t* gate16[2];  // 16-bit gates: gate g (variable 2 + g) at gate16[b] + g*vol, or nullptr
    int32_t* act;         // activation steps
    const uint8_t* stim;  // stimulus region (nullptr: none)
    TissueDyn* dyn;
    long long plane, vol;  // px*ny, px*ny*nz
    double t_on, t_off;    // stimulus window, compared with t_n
    double dt_d;           // time step, for t_{n+1} = t_n + dt
    int nx, ny, nz, px;
    float dt, theta, stim_amp;
    int split;  // 1: Lie operator splitting (diffusion substep, then kinetics); 0: unsplit
    int rk4;    // kinetics solver: 1 classical RK4 (right-hand-side models), 0 forward Euler / Rush-Larsen
    int wsum_zero;  // 1: every W-tilde sum of the grid is exactly 0 (a single-grid launch then skips their copies)
    // diffusion constants over h^2: anisotropic D = Dperp I + (Dpar-Dperp) f f^T
    // gives c_perp = Dperp/h^2, c_d = (Dpar-Dperp)/h^2, c_s = c_d/4 (Wtilde); isotropic D gives c_iso = D/h^2.
    float c_perp, c_d, c_s, c_iso;
    float mp[8];  // model parameters in kernel form
    const struct SurrogateData* surr;  // reaction surrogate (Beeler-Reuter), or nullptr
    const float4* tab;                 // V-table of the model (kTabN x 4 float4), or nullptr
};

// Where the done flags of a piece's column are (a launch of several steps over
// unmasked grids): the flag of computed plane z (a sheet: tile row z) at
// base + z; len planes from z0 on; the columns one tile further in y lie `row`
// flags away, those in x len flags; which of them exist.
struct PieceFlags {
    long long base;
    int row, len, z0;
    int has;  // bit 0, 1: column at x - 1, x + 1; bit 2, 3: at y - 1, y + 1
};

// One launch: a balanced schedule of pieces over the grids of one kernel type.
// CTA c marches through the slots c*cta_stride .. c*cta_stride + cta_count[c]
// of pieces[]; a piece (x0, y0, z0, z1) is one 64 x TY column of grid
// piece_tissue[i] over the z-range [z0, z1).  A fixed stride lets a CTA find
// its first piece with one load.
//
// A launch over one grid (`single`) carries that grid's TissueArgs in the
// kernel parameters (t0): its tensor maps, constants and the pointer to its
// TissueDyn are then read from parameter space instead of through a chain of
// dependent global loads at the start of every CTA.
struct LaunchArgs {
    TissueArgs t0;             // the grid of a single-grid launch
    const TissueArgs* tissues;
    const int4* pieces;        // ctas x cta_stride slots
    const int* piece_tissue;   // per slot
    const int* cta_count;      // pieces of each CTA
    const int* tissue_off;     // grid t owns slots tissue_pieces[tissue_off[t] .. tissue_off[t+1])
    const int* tissue_pieces;  // (for the per-grid sums, in a fixed order)
    int n_tissues;
    int single;                // one grid: t0 is valid and slots are summed in index order
    int cta_stride;
    int n_slots;               // ctas x cta_stride; unused slots keep a zero partial
    double* partials;          // one per slot
    unsigned int* ticket;      // zero between launches
    unsigned int* tissue_done; // per grid: pieces finished in this launch (zero between launches)
    const int* empty_tissues;  // the grids with no piece (their time still advances)
    int n_empty;
    int* err;                  // sticky error bits
    long long wait_limit;      // clock64 cycles a wait may spin before giving up
    int poison_first_load;     // fault injection: CTA 0's first plane never completes
    // Single-grid launch: the buffer parity the host expects (-1: read it),
    // and for an unmasked 3D grid the schedule's shape, from which a CTA finds
    // its first piece without a memory read (reg_len = 0: read the list).  A
    // CTA then issues its first plane copies before any global load returns;
    // both are checked against device memory (ERRBIT_HINT on a mismatch).
    int cur_hint;
    int reg_len, reg_nbx, reg_ty, reg_ctas;  // column length (nz), columns in x, tile rows, CTAs
    long long reg_planes;                    // column-planes of the schedule
    int reg_z0;                              // first computed plane of every column (0; 1 below a halo plane)
    int n_steps;         // time steps of this launch (more than one: unmasked grids only, all CTAs resident)
    const PieceFlags* piece_flags;  // per slot
    int* flags;          // per grid column and computed plane: the last step done, as a running number
    int epoch;           // that number before this launch's first step
    int total_mark;      // single-grid launch: total_pending after it
};

struct Coef {
    float c_perp, c_d, c_s, c_iso;
};

// ---------------------------------------------------------------------------
// PTX wrappers: shared-memory barriers and tensor-map bulk copies
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Expect bytes on the barrier without arriving (the arrival comes later).
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// The same without waiting (a try_wait that fails has waited for a
// system-dependent time, several microseconds here).
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the barrier phase with the given parity; gives up (returns false)
// after `limit` SM clock cycles instead of spinning forever.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, long long limit) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > limit) return false;
    }
    return true;
}

// Stores of the new state: st.global states the address space, so the
// compiler need not assume they overwrite the shared-memory piece context
// (which it would otherwise reload after every store).
__device__ __forceinline__ void st_global(float* p, float2 v) {
    asm volatile("st.global.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v.x), "f"(v.y));
}
__device__ __forceinline__ void st_global(float* p, float v) { asm volatile("st.global.f32 [%0], %1;" ::"l"(p), "f"(v)); }

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int x, int y, int z, int w,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_addr(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_addr(bar))
        : "memory");
}

// Done flags of a launch of several steps.
__device__ __forceinline__ int ld_flag(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_flag(int* p, int v) {
    asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ int ld_shared_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.cta.shared::cta.s32 %0, [%1];" : "=r"(v) : "r"(smem_addr(p)) : "memory");
    return v;
}
__device__ __forceinline__ void st_shared_release(int* p, int v) {
    asm volatile("st.release.cta.shared::cta.s32 [%0], %1;" ::"r"(smem_addr(p)), "r"(v) : "memory");
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// ---------------------------------------------------------------------------
// compensated float accumulation (Knuth's TwoSum) for the V reduction
// ---------------------------------------------------------------------------

struct F2 {
    float hi, lo;
};

// Packed FP32 pairs (the two x-adjacent nodes of a thread): one instruction
// slot per pair.  The FP32 pipe runs them at the rate of two scalar
// operations (measured: 2.2 cycles a warp against 1.1), but the step kernels
// are bound by instruction issue, where a pair costs one slot instead of two;
// broadcast scalars, immediates and negated operands are free.  Every
// operation is rounded on its own (no contraction), so a node's result does
// not depend on the kernel variant it is computed in.
__device__ __forceinline__ float2 splat2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// TwoSum of a running pair of sums: the rounding error of each addition goes
// to lo, as two_sum_add does for one.
__device__ __forceinline__ void two_sum_add2(float2& hi, float2& lo, float2 b) {
    const float2 s = add2(hi, b);
    const float2 bb = sub2(s, hi);
    lo = add2(lo, add2(sub2(hi, sub2(s, bb)), sub2(b, bb)));
    hi = s;
}

__device__ __forceinline__ void two_sum_add(F2& a, float b) {
    float s = a.hi + b;
    float bb = s - a.hi;
    float err = (a.hi - (s - bb)) + (b - bb);
    a.hi = s;
    a.lo += err;
}

// Sum a per-thread double over the block (any blockDim that is a multiple of
// 32, at most 1024); result valid in thread 0.
__device__ __forceinline__ double block_sum_double(double v, double* scratch32) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) scratch32[warp] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        for (int w = 0; w < nw; ++w) s += scratch32[w];
    }
    return s;
}

// Per-CTA partial -> deterministic grid total by the last CTA to finish.  The
// last CTA sums the partials with all its threads (fixed strided order, then
// a fixed tree), so the result does not depend on which CTA finished last.
__device__ __forceinline__ void grid_total_finalize(double block_partial, double* partials,
                                                    unsigned int* ticket, double* out, int* err,
                                                    bool flag_nonfinite, double* scratch32) {
    __shared__ bool last;
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = block_partial;
        if (flag_nonfinite && !isfinite(block_partial)) atomicOr(err, ERRBIT_NAN);
        __threadfence();
        unsigned int t = atomicAdd(ticket, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double s = 0.0;
    for (unsigned int b = threadIdx.x; b < gridDim.x; b += blockDim.x) s += __ldcg(&partials[b]);
    __syncthreads();  // scratch32 may still be read by the caller's block sum
    const double total = block_sum_double(s, scratch32);
    if (threadIdx.x == 0) {
        *out = total;
        *ticket = 0u;
    }
}

// Single-grid launch, producer lane of every CTA, once its t, n and parity
// are read: the CTA that arrives last (all others have read them too)
// advances them, marks the total as pending and resets the ticket.
__device__ __forceinline__ void start_ticket(const LaunchArgs& L, const TissueDyn& d0) {
    __threadfence();
    const unsigned int t = atomicAdd(L.ticket, 1u);
    if (t == gridDim.x - 1) {
        TissueDyn* d = L.t0.dyn;
        double tn = d0.t;
        for (int s = 0; s < L.n_steps; ++s) tn = tn + L.t0.dt_d;
        d->t = tn;
        d->n = d0.n + L.n_steps;
        d->cur = d0.cur ^ (L.n_steps & 1);
        d->total_pending = L.total_mark;
        *L.ticket = 0u;
    }
}

// The fixed-order sum of a grid's per-piece partials tissue_pieces[k0 .. k1):
// each of `stride` threads takes every stride-th piece from `first`, four
// loads at a time so their L2 latencies overlap; then a shuffle tree over
// the warp (the caller adds the warps' results in order).
__device__ __forceinline__ double grid_partials_sum(const LaunchArgs& L, int k0, int k1, int first, int stride) {
    double s = 0.0;
    for (int k = k0 + first; k < k1; k += 4 * stride) {
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int kk = k + u * stride;
            v[u] = kk < k1 ? __ldcg(&L.partials[__ldcg(&L.tissue_pieces[kk])]) : 0.0;
        }
        s += (v[0] + v[1]) + (v[2] + v[3]);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// The end of a grid's step in a launch over several grids: its total, then
// t += dt, n += 1 and the buffer parity flip.
__device__ __forceinline__ void finish_grid(const LaunchArgs& L, int ti, double s) {
    const TissueArgs* T = L.tissues + ti;
    TissueDyn* d = T->dyn;
    if (!isfinite(s)) atomicOr(L.err, ERRBIT_NAN);
    d->total = s;
    double tn = d->t;
    for (int k = 0; k < L.n_steps; ++k) tn = tn + T->dt_d;
    d->t = tn;
    d->n = d->n + L.n_steps;
    d->cur = d->cur ^ (L.n_steps & 1);
    d->total_pending = 0;
}

// Launch over several grids, one warp of the CTA that has just written the
// partial of piece pi (lane 0 wrote it): the piece counts towards its grid,
// and the CTA that completes a grid finishes it at once (per-grid sums spread
// over the CTAs while the others still compute, instead of one CTA summing
// every grid at the end).  A grid's pieces all precede its finish, so no
// producer reads the grid's parity after it flips.
__device__ __forceinline__ void grid_piece_done(const LaunchArgs& L, int pi, int lane) {
    int fin = -1;
    if (lane == 0) {
        __threadfence();  // the piece's partial before its count
        const int ti = L.piece_tissue[pi];
        const unsigned int npc = (unsigned int)(L.tissue_off[ti + 1] - L.tissue_off[ti]);
        if (atomicAdd(&L.tissue_done[ti], 1u) == npc - 1u) fin = ti;
    }
    fin = __shfl_sync(0xffffffffu, fin, 0);
    if (fin < 0) return;
    __threadfence();
    const double s = grid_partials_sum(L, __ldcg(&L.tissue_off[fin]), __ldcg(&L.tissue_off[fin + 1]), lane, 32);
    if (lane == 0) {
        finish_grid(L, fin, s);
        L.tissue_done[fin] = 0u;
    }
}

// End of a launch over several grids: the grids without pieces (no tissue)
// advance t, n and the parity in the last CTA to finish; the others were
// finished by grid_piece_done.  A single-grid launch has no end step: its
// producers advance t, n and the parity as soon as every CTA has read them
// (start_ticket), and the grid's total is summed from the partials when it
// is asked for.
__device__ __forceinline__ void step_finalize(const LaunchArgs& L) {
    __shared__ bool last;
    if (L.single || L.n_empty == 0) return;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const unsigned int t = atomicAdd(L.ticket, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return;
    for (int e = threadIdx.x; e < L.n_empty; e += blockDim.x) finish_grid(L, __ldcg(&L.empty_tissues[e]), 0.0);
    __syncthreads();
    if (threadIdx.x == 0) *L.ticket = 0u;
}

// ---------------------------------------------------------------------------
// cell models (kernel form of the parameters is prepared on the host)
// ---------------------------------------------------------------------------

template <int MODEL>
struct Model;

// FitzHugh-Nagumo, Eq. (FHN) with the cubic: mp = {1/eps, eps, beta, gamma}.
template <>
struct Model<BBX_FHN> {
    static constexpr int S = 2;
    __device__ static __forceinline__ void update(const float* mp, float* y, float L, float Is, float dt) {
        const float u = y[0], v = y[1];
        const float du = (u - u * u * u * (1.0f / 3.0f) - v) * mp[0] + L + Is;
        const float dv = mp[1] * (u + mp[2] - mp[3] * v);
        y[0] = u + dt * du;
        y[1] = v + dt * dv;
    }
    // the same for a pair of nodes, L the diffusion term plus the stimulus
    __device__ static __forceinline__ void update2(const float* mp, float2* y, float2 L, float dt) {
        const float2 u = y[0], v = y[1];
        const float2 c = fma2(mul2(u, u), splat2(-1.0f / 3.0f), splat2(1.0f));
        const float2 du = fma2(sub2(mul2(u, c), v), splat2(mp[0]), L);
        const float2 dv = mul2(fma2(v, splat2(-mp[3]), add2(u, splat2(mp[2]))), splat2(mp[1]));
        y[0] = fma2(splat2(dt), du, u);
        y[1] = fma2(splat2(dt), dv, v);
    }
    // right-hand side with the source I (diffusion term + stimulus) on u
    __device__ static __forceinline__ void rhs(const float* mp, const float* y, float I, float* dy) {
        const float u = y[0], v = y[1];
        dy[0] = (u - u * u * u * (1.0f / 3.0f) - v) * mp[0] + I;
        dy[1] = mp[1] * (u + mp[2] - mp[3] * v);
    }
};

// Barkley (1991): mp = {1/a, b, 1/eps}.
template <>
struct Model<BBX_BARKLEY> {
    static constexpr int S = 2;
    __device__ static __forceinline__ void update(const float* mp, float* y, float L, float Is, float dt) {
        const float u = y[0], v = y[1];
        const float du = u * (1.0f - u) * (u - (v + mp[1]) * mp[0]) * mp[2] + L + Is;
        y[0] = u + dt * du;
        y[1] = v + dt * (u - v);
    }
    __device__ static __forceinline__ void update2(const float* mp, float2* y, float2 L, float dt) {
        const float2 u = y[0], v = y[1];
        const float2 q = mul2(u, sub2(splat2(1.0f), u));
        const float2 w = fma2(add2(v, splat2(mp[1])), splat2(-mp[0]), u);
        const float2 du = fma2(mul2(q, w), splat2(mp[2]), L);
        y[0] = fma2(splat2(dt), du, u);
        y[1] = fma2(splat2(dt), sub2(u, v), v);
    }
    __device__ static __forceinline__ void rhs(const float* mp, const float* y, float I, float* dy) {
        const float u = y[0], v = y[1];
        dy[0] = u * (1.0f - u) * (u - (v + mp[1]) * mp[0]) * mp[2] + I;
        dy[1] = u - v;
    }
};

// ZFK / Nagumo reaction of Eq. (ZFKbidomV): mp = {alpha}.
template <>
struct Model<BBX_ZFK> {
    static constexpr int S = 1;
    __device__ static __forceinline__ void update(const float* mp, float* y, float L, float Is, float dt) {
        const float u = y[0];
        y[0] = u + dt * (u * (u - mp[0]) * (1.0f - u) + L + Is);
    }
    __device__ static __forceinline__ void update2(const float* mp, float2* y, float2 L, float dt) {
        const float2 u = y[0];
        const float2 q = mul2(u, sub2(u, splat2(mp[0])));
        y[0] = fma2(splat2(dt), fma2(q, sub2(splat2(1.0f), u), L), u);
    }
    __device__ static __forceinline__ void rhs(const float* mp, const float* y, float I, float* dy) {
        const float u = y[0];
        dy[0] = u * (u - mp[0]) * (1.0f - u) + I;
    }
};

// Diffusion equation alone.
template <>
struct Model<BBX_DIFFUSION> {
    static constexpr int S = 1;
    __device__ static __forceinline__ void update(const float*, float* y, float L, float Is, float dt) {
        y[0] = y[0] + dt * (L + Is);
    }
    __device__ static __forceinline__ void update2(const float*, float2* y, float2 L, float dt) {
        y[0] = fma2(splat2(dt), L, y[0]);
    }
    __device__ static __forceinline__ void rhs(const float*, const float*, float I, float* dy) { dy[0] = I; }
};

// One classical fourth-order Runge-Kutta step (the rk4 kinetics solver of
// section "Explicit solvers") of a model given by its right-hand side, with
// the diffusion term and stimulus held fixed over the step as a source on the
// first variable: stages at t, t + dt/2, t + dt/2, t + dt; weights 1, 2, 2, 1
// over 6.
template <int MODEL>
__device__ __forceinline__ void rk4_update(const float* mp, float* y, float L, float Is, float dt) {
    constexpr int S = Model<MODEL>::S;
    const float I = L + Is, h2 = 0.5f * dt;
    float k1[S], k2[S], k3[S], k4[S], t[S];
    Model<MODEL>::rhs(mp, y, I, k1);
#pragma unroll
    for (int v = 0; v < S; ++v) t[v] = y[v] + h2 * k1[v];
    Model<MODEL>::rhs(mp, t, I, k2);
#pragma unroll
    for (int v = 0; v < S; ++v) t[v] = y[v] + h2 * k2[v];
    Model<MODEL>::rhs(mp, t, I, k3);
#pragma unroll
    for (int v = 0; v < S; ++v) t[v] = y[v] + dt * k3[v];
    Model<MODEL>::rhs(mp, t, I, k4);
#pragma unroll
    for (int v = 0; v < S; ++v) y[v] += (dt * (1.0f / 6.0f)) * ((k1[v] + k4[v]) + 2.0f * (k2[v] + k3[v]));
}

// Beeler-Reuter (1977).  State (V, Ca, x1, m, h, j, d, f); mp = {gNa, gNaC,
// ENa, gs}.  V in mV, t in ms, Ca in mol/L, currents in uA/cm^2, Cm = 1.
// Rate constants of the 1977 publication, written out per gate.
__device__ __forceinline__ float br_ratio(float num, float den) { return __fdividef(num, den); }

// e^x - 1 in FP32: near 0 the Taylor series of e^x - 1 about 0 up to x^7/5040
// (|x| < 0.25: the first omitted term is below 2e-9 of the value), elsewhere
// the difference e^x - 1, whose cancellation is bounded there (e^x - 1 >= 0.22
// for x >= 0.25, <= -0.22 for x <= -0.25).
__device__ __forceinline__ float expm1_br(float x) {
    if (fabsf(x) < 0.25f) {
        float p = fmaf(x, 1.0f / 5040.0f, 1.0f / 720.0f);
        p = fmaf(x, p, 1.0f / 120.0f);
        p = fmaf(x, p, 1.0f / 24.0f);
        p = fmaf(x, p, 1.0f / 6.0f);
        p = fmaf(x, p, 0.5f);
        p = fmaf(x, p, 1.0f);
        return x * p;
    }
    return __expf(x) - 1.0f;
}

// Powers of two, logarithm and reciprocal by the special-function unit, for
// pairs; results below the normal range are 0.
__device__ __forceinline__ float2 ex2_pair(float2 a) {
    float2 r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(a.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 lg2_pair(float2 a) {
    float2 r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(a.x));
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 rcp_pair(float2 a) {
    float2 r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(a.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(a.y));
    return r;
}
// a e^{k (V + c)} with log2a = log2(a): one multiply-add and one power of two.
__device__ __forceinline__ float2 exp_rate(float2 V, double k, double c, double log2a) {
    constexpr double l2e = 1.4426950408889634;
    return ex2_pair(fma2(V, splat2((float)(k * l2e)), splat2((float)(k * c * l2e + log2a))));
}
// 1 / a and 1 / b by one reciprocal.
__device__ __forceinline__ void rcp_both(float2 a, float2 b, float2* ra, float2* rb) {
    const float2 i = rcp_pair(mul2(a, b));
    *ra = mul2(i, b);
    *rb = mul2(i, a);
}
// (1 - e^{-z}) / z for |z| < 1/4: its Taylor series to z^5/720 (the first
// omitted term is below 5e-8).
__device__ __forceinline__ float2 phi_series(float2 z) {
    float2 p = fma2(z, splat2(-1.0f / 720.0f), splat2(1.0f / 120.0f));
    p = fma2(z, p, splat2(-1.0f / 24.0f));
    p = fma2(z, p, splat2(1.0f / 6.0f));
    p = fma2(z, p, splat2(-0.5f));
    return fma2(z, p, splat2(1.0f));
}
// The same for any z >= 0: by the power of two where z >= 1/4 (1 - e^{-z} >= 0.22 there).
__device__ __forceinline__ float2 phi_any(float2 z) {
    const float2 q = phi_series(z);
    const float2 e = ex2_pair(mul2(z, splat2(-1.44269504f)));
    const float2 r = mul2(sub2(splat2(1.0f), e), rcp_pair(z));
    return make_float2(z.x < 0.25f ? q.x : r.x, z.y < 0.25f ? q.y : r.y);
}

// Voltage tables of the Beeler-Reuter models: kTabN entries kTabDv mV apart
// from kTabVmin (-120 to +80 mV), 16 floats (4 float4) each; V outside the
// range takes the end entry.  Entry index and interpolation weight of V.
constexpr float kTabVmin = -120.0f, kTabDv = 0.025f, kTabInvDv = 40.0f;
constexpr int kTabN = 8001;
__device__ __forceinline__ int tab_index(float V, float* w) {
    float xi = (V - kTabVmin) * kTabInvDv;
    xi = fminf(fmaxf(xi, 0.0f), (float)(kTabN - 1));
    int i = (int)xi;
    if (i > kTabN - 2) i = kTabN - 2;
    *w = xi - (float)i;
    return i;
}

// The interpolated table entry c at V.
__device__ __forceinline__ void tab_entry(const float4* __restrict__ tab, float V, float* c) {
    float w;
    const int i = tab_index(V, &w);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 a = __ldg(tab + 4 * i + q), b = __ldg(tab + 4 * i + 4 + q);
        c[4 * q + 0] = fmaf(w, b.x - a.x, a.x);
        c[4 * q + 1] = fmaf(w, b.y - a.y, a.y);
        c[4 * q + 2] = fmaf(w, b.z - a.z, a.z);
        c[4 * q + 3] = fmaf(w, b.w - a.w, a.w);
    }
}

// The same for every lane's V, the 32 lanes of a warp together: four lanes
// read one node's two entries as 2 x 64 consecutive bytes, interpolate four
// coefficients each and hand them to the node's lane through shared memory
// (buf: 32 nodes x 64 bytes, the 16-byte parts swapped so that eight lanes
// touch every bank once).  What bounds a tabulated step is the wavefronts of
// these loads: where V differs from node to node, a lane reading its own
// node's entries takes eight loads of 32 separate lines, this eight loads of
// eight 64-byte segments, and half as many wavefronts again for the exchange.
// In waves (V different everywhere), each lane its own entries / gathered, us a
// step: 256x256x64 slab 104 / 79, Markov sodium 197 / 128, 256^3 shell 131 / 106,
// with 16-bit gates 127 / 104, 1024x1024 sheet 30.7 / 23.1.  Where the warp's V
// lie within a few entries (tissue at rest) each lane reads its own: its loads
// are then a line or two for the whole warp (slab at rest gathered 68, so 58;
// Markov sodium 103 and 75).  A slab at rest but for one front is slower with
// it, 63 / 66, with 16-bit gates 55 / 60: few warps look up, and each waits for
// two exchanges (with a cold L2 72 / 80 and 65 / 76, Markov sodium 117 / 127).
__device__ __forceinline__ void tab_entry_warp(const float4* __restrict__ tab, float V, float4* buf, float* c) {
    const int lane = threadIdx.x & 31, p = lane & 3;
    float w;
    const int i = tab_index(V, &w);
    if (__reduce_max_sync(0xffffffffu, i) - __reduce_min_sync(0xffffffffu, i) <= 3) {
        tab_entry(tab, V, c);
        return;
    }
    float4 a[4], b[4];
    float wn[4];
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int n = 8 * it + (lane >> 2);
        const float4* e = tab + 4 * __shfl_sync(0xffffffffu, i, n) + p;
        wn[it] = __shfl_sync(0xffffffffu, w, n);
        a[it] = __ldg(e);
        b[it] = __ldg(e + 4);
    }
    __syncwarp();  // the entries handed over before have been read
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int n = 8 * it + (lane >> 2);
        buf[4 * n + (p ^ ((n >> 1) & 3))] =
            make_float4(fmaf(wn[it], b[it].x - a[it].x, a[it].x), fmaf(wn[it], b[it].y - a[it].y, a[it].y),
                        fmaf(wn[it], b[it].z - a[it].z, a[it].z), fmaf(wn[it], b[it].w - a[it].w, a[it].w));
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 v = buf[4 * lane + (q ^ ((lane >> 1) & 3))];
        c[4 * q + 0] = v.x;
        c[4 * q + 1] = v.y;
        c[4 * q + 2] = v.z;
        c[4 * q + 3] = v.w;
    }
}

template <>
struct Model<BBX_BR> {
    static constexpr int S = 8;


    // The change of every variable over one step (the update is y + d): the
    // Euler increments of V and Ca, and the Rush-Larsen increments of the
    // gates, Eq. (RL) read as y' = A y + B, i.e. d = (1 - A)(y_inf - y) with
    // 1 - A by expm1_br (no cancellation when (alpha+beta) dt is small).
    __device__ static __forceinline__ void increment(const float* mp, const float* y, float L, float Is, float dt,
                                                     float* d) {
        increment_m3(mp, y, y[3] * y[3] * y[3], L, Is, dt, d);
    }

    // The same with the open probability m3 of the sodium activation given
    // (y[3] only feeds the m-gate increment d[3]).
    __device__ static __forceinline__ void increment_m3(const float* mp, const float* y, float m3, float L,
                                                        float Is, float dt, float* d) {
        const float V = y[0], Ca = y[1];
        const float x1 = y[2], m = y[3], h = y[4], j = y[5], dd = y[6], f = y[7];

        // membrane currents
        const float INa = (mp[0] * m3 * h * j + mp[1]) * (V - mp[2]);
        const float Es = -82.3f - 13.0287f * __logf(Ca);
        const float Is_ = mp[3] * dd * f * (V - Es);
        const float Ix1 = x1 * 0.8f * (__expf(0.04f * (V + 77.0f)) - 1.0f) * __expf(-0.04f * (V + 35.0f));
        const float w = V + 23.0f;
        const float lin = (w == 0.0f) ? 5.0f : br_ratio(0.2f * w, -expm1_br(-0.04f * w));
        const float IK1 = 0.35f * (br_ratio(4.0f * (__expf(0.04f * (V + 85.0f)) - 1.0f),
                                            __expf(0.08f * (V + 53.0f)) + __expf(0.04f * (V + 53.0f))) +
                                   lin);
        const float Iion = INa + Is_ + Ix1 + IK1;
        const float dCa = -1e-7f * Is_ + 0.07f * (1e-7f - Ca);

        // gate rates, 1/ms
        const float a_x1 = br_ratio(0.0005f * __expf(0.083f * (V + 50.0f)), __expf(0.057f * (V + 50.0f)) + 1.0f);
        const float b_x1 = br_ratio(0.0013f * __expf(-0.06f * (V + 20.0f)), __expf(-0.04f * (V + 20.0f)) + 1.0f);
        const float xm = V + 47.0f;
        const float a_m = (xm == 0.0f) ? 10.0f : br_ratio(-xm, expm1_br(-0.1f * xm));
        const float b_m = 40.0f * __expf(-0.056f * (V + 72.0f));
        const float a_h = 0.126f * __expf(-0.25f * (V + 77.0f));
        const float b_h = br_ratio(1.7f, __expf(-0.082f * (V + 22.5f)) + 1.0f);
        const float a_j = br_ratio(0.055f * __expf(-0.25f * (V + 78.0f)), __expf(-0.2f * (V + 78.0f)) + 1.0f);
        const float b_j = br_ratio(0.3f, __expf(-0.1f * (V + 32.0f)) + 1.0f);
        const float a_d = br_ratio(0.095f * __expf(-0.01f * (V - 5.0f)), __expf(-0.072f * (V - 5.0f)) + 1.0f);
        const float b_d = br_ratio(0.07f * __expf(-0.017f * (V + 44.0f)), __expf(0.05f * (V + 44.0f)) + 1.0f);
        float a_f, b_f;
        f_rates(V, &a_f, &b_f);

        d[0] = dt * (-(Iion - Is) + L);  // Cm = 1
        d[1] = dt * dCa;
        d[2] = rl_inc(x1, a_x1, b_x1, dt);
        d[3] = rl_inc(m, a_m, b_m, dt);
        d[4] = rl_inc(h, a_h, b_h, dt);
        d[5] = rl_inc(j, a_j, b_j, dt);
        d[6] = rl_inc(dd, a_d, b_d, dt);
        d[7] = rl_inc(f, a_f, b_f, dt);
    }

    // alpha_f and beta_f, the rates of the slow inward current's inactivation
    __device__ static __forceinline__ void f_rates(float V, float* a_f, float* b_f) {
        *a_f = br_ratio(0.012f * __expf(-0.008f * (V + 28.0f)), __expf(0.15f * (V + 28.0f)) + 1.0f);
        *b_f = br_ratio(0.0065f * __expf(-0.02f * (V + 30.0f)), __expf(-0.2f * (V + 30.0f)) + 1.0f);
    }

    __device__ static __forceinline__ float rl_inc(float y, float al, float be, float dt) {
        const float s = al + be;
        const float one_minus_A = -expm1_br(-s * dt);
        return one_minus_A * (__fdividef(al, s) - y);
    }

    __device__ static __forceinline__ void update(const float* mp, float* y, float L, float Is, float dt) {
        float d[8];
        increment(mp, y, L, Is, dt, d);
#pragma unroll
        for (int v = 0; v < 8; ++v) y[v] = y[v] + d[v];
    }

    // The same for a pair of nodes (Is the stimulus).  What bounds it is the
    // number of instructions: update() takes about 470 per node (each
    // exponential, logarithm and division carries the scaling of its denormal
    // range), this about 110.  Exponents are one multiply-add; exponentials
    // that are powers of one another (0.02, 0.04, 0.06 and 0.1, 0.2 per mV)
    // share one; the two rates of a gate share one reciprocal; and the
    // Rush-Larsen increment (1 - e^{-s dt}) (alpha/s - y), s = alpha + beta,
    // is taken as dt phi(s dt) (alpha - s y), phi(z) = (1 - e^{-z})/z, which
    // needs no division.  For V in (-140, 120) mV and dt <= 0.19 ms, where no
    // exponential leaves the range and s dt < 1/4 for x1, j, d, f; update()
    // elsewhere.
    __device__ static __forceinline__ void update2(const float* mp, float2* y, float2 L, float2 Is, float dt) {
        const float2 V = y[0], Ca = y[1];
        if (!(fminf(V.x, V.y) > -140.0f && fmaxf(V.x, V.y) < 120.0f && dt <= 0.19f)) {
            float a[8], b[8];
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                a[v] = y[v].x;
                b[v] = y[v].y;
            }
            update(mp, a, L.x, Is.x, dt);
            update(mp, b, L.y, Is.y, dt);
#pragma unroll
            for (int v = 0; v < 8; ++v) y[v] = make_float2(a[v], b[v]);
            return;
        }
        const float2 one = splat2(1.0f);
        const float2 R = exp_rate(V, -0.02, 20.0, 0.0);  // e^{-0.02 (V + 20)}
        const float2 R2 = mul2(R, R);                    // e^{-0.04 (V + 20)}
        const float2 P = exp_rate(V, -0.1, 47.0, 0.0);   // e^{-0.1 (V + 47)}
        const float2 P2 = mul2(P, P);                    // e^{-0.2 (V + 47)}

        // the removable singularities w / (1 - e^{-z}), z = k w: alpha_m (w = V + 47, k = 0.1) and
        // the linear part of I_K1 (w = V + 23, k = 0.04); 1 / (k phi(z)) near 0
        float2 nm = add2(V, splat2(47.0f)), dm = sub2(one, P);
        float2 nl = add2(V, splat2(23.0f)), dl = fma2(R2, splat2(-0.8869204367f), one);  // e^{-0.12}
        if (fminf(fabsf(nm.x), fabsf(nm.y)) < 2.5f) {
            const float2 q = phi_series(mul2(nm, splat2(0.1f)));
            if (fabsf(nm.x) < 2.5f) { nm.x = 10.0f; dm.x = q.x; }
            if (fabsf(nm.y) < 2.5f) { nm.y = 10.0f; dm.y = q.y; }
        }
        if (fminf(fabsf(nl.x), fabsf(nl.y)) < 6.25f) {
            const float2 q = phi_series(mul2(nl, splat2(0.04f)));
            if (fabsf(nl.x) < 6.25f) { nl.x = 25.0f; dl.x = q.x; }
            if (fabsf(nl.y) < 6.25f) { nl.y = 25.0f; dl.y = q.y; }
        }
        float2 im, il;
        rcp_both(dm, dl, &im, &il);
        const float2 a_m = mul2(nm, im);
        const float2 lin = mul2(nl, il);  // (0.2 w / (1 - e^{-z}) = 0.2 lin)

        // membrane currents
        const float2 V_ENa = add2(V, splat2(-mp[2]));
        const float2 m3hj = mul2(mul2(mul2(y[3], y[3]), y[3]), mul2(y[4], y[5]));
        const float2 INa = mul2(fma2(m3hj, splat2(mp[0]), splat2(mp[1])), V_ENa);
        // V - E_s = V + 82.3 + 13.0287 ln Ca
        const float2 V_Es = fma2(lg2_pair(Ca), splat2(9.03080667f), add2(V, splat2(82.3f)));
        const float2 Is_ = mul2(mul2(mul2(y[6], y[7]), splat2(mp[3])), V_Es);
        // 0.8 (e^{0.04 (V + 77)} - 1) e^{-0.04 (V + 35)}
        const float2 Ix1 = mul2(y[2], fma2(R2, splat2(-0.439049309f), splat2(4.29244478f)));
        // 4 (e^{0.04 (V + 85)} - 1) / (e^{0.08 (V + 53)} + e^{0.04 (V + 53)}), r = e^{-0.04 (V + 53)}
        const float2 r = mul2(R2, splat2(0.267135302f));
        const float2 Eh = exp_rate(V, -0.082, 22.5, 0.0);
        float2 ik, bh;
        rcp_both(add2(one, r), add2(one, Eh), &ik, &bh);
        const float2 k1 = mul2(mul2(r, sub2(splat2(3.59663973f), r)), ik);
        const float2 IK1 = fma2(k1, splat2(1.4f), mul2(lin, splat2(0.07f)));
        const float2 Iion = add2(add2(INa, Is_), add2(Ix1, IK1));
        const float2 dCa = fma2(Is_, splat2(-1e-7f), fma2(Ca, splat2(-0.07f), splat2(7e-9f)));

        // the gates: alpha and beta, 1/ms
        auto gate = [&](int v, float2 al, float2 be, bool any) {
            const float2 s = add2(al, be), z = mul2(s, splat2(dt));
            const float2 t = fma2(s, make_float2(-y[v].x, -y[v].y), al);
            y[v] = fma2(mul2(any ? phi_any(z) : phi_series(z), t), splat2(dt), y[v]);
        };
        auto gate2 = [&](int v, float2 n1, float2 d1, float2 n2, float2 d2) {
            float2 i1, i2;
            rcp_both(d1, d2, &i1, &i2);
            gate(v, mul2(n1, i1), mul2(n2, i2), false);
        };
        const float2 a_h = exp_rate(V, -0.25, 77.0, -2.9885043611621702);
        gate2(2, exp_rate(V, 0.026, 50.0, -10.965784284662087), add2(one, exp_rate(V, -0.057, 50.0, 0.0)),
              mul2(mul2(R2, R), splat2(0.0013f)), add2(R2, one));
        gate(3, a_m, exp_rate(V, -0.056, 72.0, 5.321928094887363), true);
        gate(4, a_h, mul2(bh, splat2(1.7f)), true);
        gate2(5, mul2(a_h, splat2(0.339952723f)), fma2(P2, splat2(0.00202943064f), one), splat2(0.3f),
              fma2(P, splat2(4.48168907f), one));
        gate2(6, exp_rate(V, -0.01, -5.0, -3.3959286763311392), add2(one, exp_rate(V, -0.072, -5.0, 0.0)),
              exp_rate(V, -0.017, 44.0, -3.8365012677171206), add2(one, exp_rate(V, 0.05, 44.0, 0.0)));
        gate2(7, exp_rate(V, -0.008, 28.0, -6.380821783940931), add2(one, exp_rate(V, 0.15, 28.0, 0.0)),
              mul2(R, splat2(0.00532174991f)), fma2(P2, splat2(29.9641000f), one));
        y[0] = fma2(splat2(dt), add2(sub2(Is, Iion), L), V);  // Cm = 1
        y[1] = fma2(splat2(dt), dCa, Ca);
    }

    // The same step with the Rush-Larsen coefficients tabulated in V (the
    // rushlarsen device's tabulation, section "Exponential solvers"): per
    // entry A and B of Eq. (RL) for x1, m, h, j, d, f, then the V factors of
    // I_x1 (I_x1 = x1 K(V)) and I_K1, interpolated linearly; gates by
    // y' = A y + B.  The table is built for the grid's dt; entry(k, V, c): the
    // interpolated entry c of the model's table k at V.
    template <typename E>
    __device__ static __forceinline__ void update_tab(const float* mp, E entry, float* y, float L, float Is,
                                                      float dt) {
        const float V = y[0], Ca = y[1];
        float c[16];
        entry(0, V, c);
        const float m = y[3];
        const float INa = (mp[0] * m * m * m * y[4] * y[5] + mp[1]) * (V - mp[2]);
        const float Es = -82.3f - 13.0287f * __logf(Ca);
        const float Is_ = mp[3] * y[6] * y[7] * (V - Es);
        const float Iion = INa + Is_ + y[2] * c[12] + c[13];
        const float dCa = -1e-7f * Is_ + 0.07f * (1e-7f - Ca);
        y[0] = V + dt * (-(Iion - Is) + L);  // Cm = 1
        y[1] = Ca + dt * dCa;
#pragma unroll
        for (int g = 0; g < 6; ++g) y[2 + g] = fmaf(c[2 * g], y[2 + g], c[2 * g + 1]);
    }
};

// Beeler-Reuter with the sodium activation m^3 in its Markov form: the
// probabilities P0..P3 that k = 0..3 of the three activation subunits are
// open (P3 in place of m^3), du/dt = A(V) u with k -> k+1 at (3-k) alpha_m
// and k -> k-1 at k beta_m, advanced by the matrix Rush-Larsen scheme
// u_{n+1} = T(V_n) u_n, T = exp(dt A) (section "Exponential solvers").  T is
// tabulated in V (kTabN entries kTabDv mV apart from kTabVmin, 16 floats
// each, row-major; built on the device for the grid's dt) and interpolated
// linearly; V outside the table takes the end entry.  x1, h, j, d, f by
// Eq. (RL) with tabulated coefficients (as Model<BBX_BR>::update_tab), V and
// Ca by Eq. (Euler).
// State: V, Ca, x1, h, j, d, f, P0, P1, P2, P3.

template <>
struct Model<BBX_BR_MRL> {
    static constexpr int S = 11;

    // Table 0: the Rush-Larsen table of Model<BBX_BR>::update_tab (kTabN x 4
    // float4), followed by table 1, the chain's transition matrices (kTabN x 4
    // float4).
    template <typename E>
    __device__ static __forceinline__ void update_tab(const float* mp, E entry, float* y, float L, float Is,
                                                      float dt) {
        const float V = y[0], Ca = y[1];
        // the chain, from V at the start of the step
        float c[16], pn[4];
        entry(1, V, c);
#pragma unroll
        for (int r = 0; r < 4; ++r)
            pn[r] = fmaf(c[4 * r], y[7], fmaf(c[4 * r + 1], y[8], fmaf(c[4 * r + 2], y[9], c[4 * r + 3] * y[10])));
        entry(0, V, c);
        // currents with P3 in place of m^3; x1, h, j, d, f by y' = A y + B
        const float INa = (mp[0] * y[10] * y[3] * y[4] + mp[1]) * (V - mp[2]);
        const float Es = -82.3f - 13.0287f * __logf(Ca);
        const float Is_ = mp[3] * y[5] * y[6] * (V - Es);
        const float Iion = INa + Is_ + y[2] * c[12] + c[13];
        const float dCa = -1e-7f * Is_ + 0.07f * (1e-7f - Ca);
        y[0] = V + dt * (-(Iion - Is) + L);  // Cm = 1
        y[1] = Ca + dt * dCa;
        y[2] = fmaf(c[0], y[2], c[1]);  // x1
#pragma unroll
        for (int g = 0; g < 4; ++g) y[3 + g] = fmaf(c[4 + 2 * g], y[3 + g], c[5 + 2 * g]);  // h, j, d, f
#pragma unroll
        for (int r = 0; r < 4; ++r) y[7 + r] = pn[r];
    }
};

// Beeler-Reuter with the slow inward current's inactivation as a two-gate
// channel: the voltage gate f (alpha_f, beta_f of the 1977 model) and a
// calcium gate c (closed -> open at c_inf / tau_c, open -> closed at
// (1 - c_inf) / tau_c, c_inf = Kc / (Kc + Ca)), the four states q = f + 2 c
// with probabilities Q0..Q3, and a small direct transition (f open, c
// closed) -> (f closed, c open) at eps alpha_f (1 - c_inf).  The generator
// A(V, Ca) of Eq. (markov-generic) is the sum of a V-univariate matrix (the
// f gate), a Ca-univariate matrix (the c gate) and that multivariate
// remainder; section "Exponential solvers" advances such a chain by Lie
// splitting: each univariate part by its exact step from the values of V
// and Ca at the start of the step, the remainder by forward Euler.  The f
// gate's step comes from the Rush-Larsen V-table; the c gate's rates sum to
// 1/tau_c at every Ca, so its step has the closed form open' = open +
// (1 - e^{-dt/tau_c}) (c_inf total - open) with one constant.  Both gate steps
// move probability within pairs of states (total of the pair kept exactly).
// With the parameter onfly set, the channel takes the step the same section
// gives for a generator with no such decomposition instead: the exponential
// of the whole A(V, Ca) applied at run time, with no table and no splitting.
// I_s = g_s d Q3 (V - E_s); x1, m, h, j, d by Rush-Larsen; V, Ca by Euler.
// State: V, Ca, x1, m, h, j, d, Q0, Q1, Q2, Q3.
// Kernel parameters mp: gNa, gNaC, ENa, gs, Kc, eps, 1/tau_c, onfly (0 or 1).

template <>
struct Model<BBX_BR_FCA> {
    static constexpr int S = 11;

    // the channel step (u = Q0..Q3): f gate by open' = A_f open + B_f total,
    // c gate as above with omc = 1 - e^{-dt/tau_c}, then the remainder
    __device__ static __forceinline__ void channel(const float* mp, float A_f, float B_f, float a_f, float omc,
                                                   float Ca, float dt, float* u) {
        const float pc0 = u[0] + u[1], pc1 = u[2] + u[3];  // c closed, c open
        const float fo0 = fmaf(A_f, u[1], B_f * pc0), fo1 = fmaf(A_f, u[3], B_f * pc1);
        u[0] = pc0 - fo0;
        u[1] = fo0;
        u[2] = pc1 - fo1;
        u[3] = fo1;
        const float inv = __fdividef(1.0f, mp[4] + Ca);
        const float ci = mp[4] * inv, one_minus_ci = Ca * inv;
        const float pf0 = u[0] + u[2], pf1 = u[1] + u[3];  // f closed, f open
        const float co0 = fmaf(omc, fmaf(ci, pf0, -u[2]), u[2]), co1 = fmaf(omc, fmaf(ci, pf1, -u[3]), u[3]);
        u[0] = pf0 - co0;
        u[2] = co0;
        u[1] = pf1 - co1;
        u[3] = co1;
        const float flow = dt * mp[5] * a_f * one_minus_ci * u[1];
        u[1] -= flow;
        u[2] += flow;
    }

    // u <- exp(dt A(V, Ca)) u with every rate evaluated at the node: the
    // Taylor series of the exponential's action on u to nine terms, on 2^s
    // substeps, s the smallest (at most 6) that brings dt / 2^s times the
    // largest absolute column sum of A (twice the largest outflow) to 1/2.
    __device__ static __forceinline__ void channel_onfly(const float* mp, float V, float Ca, float dt, float* u) {
        float a_f, b_f;
        Model<BBX_BR>::f_rates(V, &a_f, &b_f);
        const float inv = __fdividef(1.0f, mp[4] + Ca);
        const float a_c = mp[4] * inv * mp[6], b_c = Ca * inv * mp[6];
        const float r = mp[5] * a_f * (Ca * inv);
        // outflow of each state q = f + 2 c
        const float o0 = a_f + a_c, o1 = b_f + a_c + r, o2 = a_f + b_c, o3 = b_f + b_c;
        float nrm = 2.0f * dt * fmaxf(fmaxf(o0, o1), fmaxf(o2, o3)), h = dt;
        int s = 0;
        while (nrm > 0.5f && s < 6) {
            nrm *= 0.5f;
            h *= 0.5f;
            ++s;
        }
        for (int k = 0; k < (1 << s); ++k) {
            float t0 = u[0], t1 = u[1], t2 = u[2], t3 = u[3];
            float s0 = t0, s1 = t1, s2 = t2, s3 = t3;
#pragma unroll
            for (int n = 1; n <= 9; ++n) {
                const float c = h * (1.0f / (float)n);
                const float n0 = fmaf(-o0, t0, fmaf(b_f, t1, b_c * t2));
                const float n1 = fmaf(a_f, t0, fmaf(-o1, t1, b_c * t3));
                const float n2 = fmaf(a_c, t0, fmaf(r, t1, fmaf(-o2, t2, b_f * t3)));
                const float n3 = fmaf(a_c, t1, fmaf(a_f, t2, -o3 * t3));
                t0 = c * n0;
                t1 = c * n1;
                t2 = c * n2;
                t3 = c * n3;
                s0 += t0;
                s1 += t1;
                s2 += t2;
                s3 += t3;
            }
            u[0] = s0;
            u[1] = s1;
            u[2] = s2;
            u[3] = s3;
        }
    }

    // Table 0: the Rush-Larsen table of Model<BBX_BR>::update_tab (kTabN x 4
    // float4) with entry 14 = alpha_f(V) and entry 15 = 1 - e^{-dt/tau_c}.
    template <typename E>
    __device__ static __forceinline__ void update_tab(const float* mp, E entry, float* y, float L, float Is,
                                                      float dt) {
        const float V = y[0], Ca = y[1];
        float c[16];
        entry(0, V, c);
        const float m = y[3];
        const float INa = (mp[0] * m * m * m * y[4] * y[5] + mp[1]) * (V - mp[2]);
        const float Es = -82.3f - 13.0287f * __logf(Ca);
        const float Is_ = mp[3] * y[6] * y[10] * (V - Es);
        const float Iion = INa + Is_ + y[2] * c[12] + c[13];
        const float dCa = -1e-7f * Is_ + 0.07f * (1e-7f - Ca);
        y[0] = V + dt * (-(Iion - Is) + L);  // Cm = 1
        y[1] = Ca + dt * dCa;
#pragma unroll
        for (int g = 0; g < 5; ++g) y[2 + g] = fmaf(c[2 * g], y[2 + g], c[2 * g + 1]);  // x1, m, h, j, d
        if (mp[7] != 0.0f)
            channel_onfly(mp, V, Ca, dt, y + 7);
        else
            channel(mp, c[10], c[11], c[14], c[15], Ca, dt, y + 7);
    }

    // The same step with every rate evaluated at V (no table): the rest-state
    // integration uses it.
    __device__ static __forceinline__ void update(const float* mp, float* y, float L, float Is, float dt) {
        const float V = y[0], Ca = y[1];
        float y8[8] = {y[0], y[1], y[2], y[3], y[4], y[5], y[6], y[10]};  // Q3 in the place of f
        float d[8];
        Model<BBX_BR>::increment_m3(mp, y8, y[3] * y[3] * y[3], L, Is, dt, d);
        float a_f, b_f;
        Model<BBX_BR>::f_rates(V, &a_f, &b_f);
        const float omA = -expm1_br(-(a_f + b_f) * dt);
        const float omc = -expm1_br(-dt * mp[6]);
#pragma unroll
        for (int v = 0; v < 7; ++v) y[v] += d[v];
        if (mp[7] != 0.0f)
            channel_onfly(mp, V, Ca, dt, y + 7);
        else
            channel(mp, 1.0f - omA, __fdividef(a_f, a_f + b_f) * omA, a_f, omc, Ca, dt, y + 7);
    }
};

// ---------------------------------------------------------------------------
// shared-memory plan of the step kernel
// ---------------------------------------------------------------------------

constexpr int kTileX = 64;  // nodes per brick along x: 32 threads x 2 nodes
// Several steps in one launch (FLOW variants): unmasked grids of the light
// models (the others' steps are long next to a launch, and the further warp it
// takes would cost the registers their consumers need).  The same grids run the
// variants without the sync warp at one launch a step where that is faster (in
// a batch of several kernel types, and by size when alone: bbx_grid's plans):
// four CTAs per SM instead of three when isotropic (192 sheets and 64 blocks 337
// us a step against 365).
__host__ __device__ constexpr bool has_flow(bool masked, int s) { return !masked && s <= 2; }
// Consumer warps per CTA (plus the producer warp, plus the sync warp) for a
// tile of TY rows: 7 warps of 1 or 2 rows each for TY = 7, 14; for 28 rows 7
// warps of 4 rows, or 14 warps of 2 rows (one CTA of 480 threads per SM, whose
// warps share one ring of planes and so finish together) without a sync warp.
// (8 warps and 16 rows with the sync warp, which load the four schedulers
// evenly, were slower: 256x256x64 slab 24.9 -> 29.5 us, sheets 60 -> 73 us.)
__host__ __device__ constexpr int rows_of_threads(int ty, bool flow) { return ty == 28 && !flow ? 14 : 7; }
__host__ __device__ constexpr int step_threads(int ty, bool flow) {
    return 32 * rows_of_threads(ty, flow) + 32 + (flow ? 32 : 0);
}

// Anisotropy of a step kernel variant: isotropic (c_iso only), anisotropic
// with the W-tilde sums read from memory, or anisotropic for grids whose
// W-tilde sums all vanish (no sums in the stage ring, no W-tilde arithmetic).
enum : int { AN_ISO = 0, AN_SUMS = 1, AN_NO_SUMS = 2 };

// Resident CTAs per SM a kernel variant is built for (the register budget:
// two CTAs of 256 threads allow 128 registers a thread; the masked
// anisotropic stencil with 2 rows a thread and the surrogate need more; the
// unmasked isotropic variants of the light models fit in 64, so four CTAs hide
// more latency (Beeler-Reuter spilled 216 bytes there: 83 us a step of a
// 256x256x64 slab, 54 with two CTAs); with
// a sync warp, 288 threads: 96 registers at two CTAs, 72 at three).
__host__ __device__ constexpr int ctas_per_sm(bool masked, bool aniso, int ty, bool surr, bool flow, int s) {
    if (flow) return aniso ? (ty == 28 ? 1 : 2) : 3;
    return (masked && aniso && ty != 7) || ty == 28 || (surr && ty != 7) ? 1 : (!masked && !aniso && s <= 2 ? 4 : 2);
}
constexpr int align128(int b) { return (b + 127) & ~127; }

// Tissue-mask byte on the device: bit 0 = tissue, bit 1 = tissue node whose
// 18 stencil neighbours are all tissue inside the array ("interior").
enum : uint8_t { MASK_TISSUE = 1, MASK_INTERIOR = 2 };

// Per-node word of a masked grid, as the step reads it (a tile's own words,
// 4 B a node, instead of three planes of mask bytes with their halo and a
// byte load and a test for each neighbour): the grid indicator psi of the 18
// stencil neighbours, then the node's own two mask bits.
enum : uint32_t {
    PSI_XP = 1u << 0, PSI_XM = 1u << 1, PSI_YP = 1u << 2, PSI_YM = 1u << 3, PSI_ZP = 1u << 4, PSI_ZM = 1u << 5,
    PSI_XPYP = 1u << 6, PSI_XMYM = 1u << 7, PSI_XPYM = 1u << 8, PSI_XMYP = 1u << 9,
    PSI_XPZP = 1u << 10, PSI_XMZM = 1u << 11, PSI_XPZM = 1u << 12, PSI_XMZP = 1u << 13,
    PSI_YPZP = 1u << 14, PSI_YMZM = 1u << 15, PSI_YPZM = 1u << 16, PSI_YMZP = 1u << 17,
    PSI_TISSUE = 1u << 18, PSI_INTERIOR = 1u << 19
};

// Storage of the Beeler-Reuter gates (variables 2..7) between steps: FP32
// (default), IEEE binary16, or 16-bit unsigned fixed point y = u / 65535
// (uniform steps of 1.5e-5 over [0, 1]); arithmetic is FP32 in every case,
// the new values rounded to nearest when stored.
enum : int { GATES_F32 = 0, GATES_F16 = 1, GATES_U16 = 2 };

template <int GATES>
__device__ __forceinline__ float2 gate_decode2(uint32_t w) {
    if (GATES == GATES_F16) {
        __half2 h = *reinterpret_cast<__half2*>(&w);
        return __half22float2(h);
    }
    constexpr float k = 1.0f / 65535.0f;
    return make_float2((float)(w & 0xffffu) * k, (float)(w >> 16) * k);
}

template <int GATES>
__device__ __forceinline__ uint16_t gate_encode(float y) {
    if (GATES == GATES_F16) return __half_as_ushort(__float2half_rn(y));
    return (uint16_t)__float2uint_rn(__saturatef(y) * 65535.0f);
}

template <int GATES>
__device__ __forceinline__ uint32_t gate_encode2(float lo, float hi) {
    return (uint32_t)gate_encode<GATES>(lo) | ((uint32_t)gate_encode<GATES>(hi) << 16);
}

__device__ __forceinline__ void st_global_u32(uint16_t* p, uint32_t v) {
    asm volatile("st.global.u32 [%0], %1;" ::"l"(p), "r"(v));
}
__device__ __forceinline__ void st_global_u16(uint16_t* p, uint16_t v) {
    asm volatile("st.global.u16 [%0], %1;" ::"l"(p), "h"(v));
}

template <int MODEL, bool MASKED, int ANISO, int TY, bool SURR = false, int GATES = GATES_F32,
          bool FL = has_flow(MASKED, Model<MODEL>::S), bool GEN = false>
struct Plan {
    static constexpr int S = Model<MODEL>::S;
    static constexpr int NG = GATES ? 6 : 0;  // variables stored in 16 bits (the gates, last in the state)
    static constexpr int TX = kTileX;
    static constexpr int RY = rows_of_threads(TY, FL);
    static constexpr int CTAS = ctas_per_sm(MASKED, ANISO != AN_ISO, TY, SURR, FL, Model<MODEL>::S);
    static constexpr int CY = TY / RY;  // nodes per thread along y (each a pair in x)
    static constexpr bool FLOW = FL;
    static constexpr int THREADS = step_threads(TY, FL);  // consumer warps + producer warp (+ sync warp)
    static constexpr int UW = TX + 8;   // x from x0-4 to x0+TX+3 (16-byte aligned start)
    static constexpr int UH = TY + 2;   // y from y0-1 to y0+TY
    // ring A, one stage per loaded plane (the computed planes and the z-halo
    // planes): V with its one-node halo
    static constexpr int U_RAW = UW * UH * 4;
    static constexpr int U_OFF = 0;
    // (each stage ends with its two mbarriers, so a stage's address gives them)
    static constexpr int A_BAR = U_OFF + align128(U_RAW);
    static constexpr int A_STAGE = A_BAR + 128;
    static constexpr uint32_t A_BYTES = U_RAW;
    // ring B, one stage per computed plane: the node's own unit fibre and
    // W-tilde sums (3 x TX x TY floats each), the other variables, the
    // neighbour words of a masked grid
    static constexpr int F_RAW = ANISO ? 3 * TX * TY * 4 : 0;
    static constexpr int D_RAW = ANISO == AN_SUMS ? 3 * TX * TY * 4 : 0;
    static constexpr int S32_RAW = (S > 1) ? (S - 1 - NG) * TX * TY * 4 : 0;  // 32-bit non-diffusing variables
    static constexpr int G_RAW = NG * TX * TY * 2;                              // 16-bit gates
    static constexpr int S_RAW = S32_RAW + G_RAW;
    static constexpr int F_OFF = 0;
    static constexpr int D_OFF = F_OFF + F_RAW;    // (each part a multiple of 128 bytes)
    static constexpr int S_OFF = D_OFF + D_RAW;
    static constexpr int G_OFF = S_OFF + S32_RAW;
    static constexpr int M_RAW = MASKED ? TX * TY * 4 : 0;
    static constexpr int M_OFF = G_OFF + G_RAW;
    static constexpr int B_BAR = align128(F_RAW + D_RAW + S_RAW + M_RAW);
    static constexpr int B_STAGE = B_BAR + 128;
    static constexpr uint32_t B_BYTES = F_RAW + D_RAW + S_RAW + M_RAW;
    static constexpr bool HAS_B = B_BYTES > 0;
    static constexpr int ROOM = (CTAS == 1 ? 200 : (CTAS == 2 ? 112 : (CTAS == 3 ? 72 : 54))) * 1024;  // dynamic shared memory per CTA
    // A kernel that gathers from a V-table (TAB) takes at most three stages of
    // ring B and leaves the rest to the L1 cache (Markov model, 181x428x43
    // slab: 204 us a step with four, 155 with three); its warps gather
    // together (tab_entry_warp) where their buffers cost none of these stages
    // (256^3 tabulated shell, when it was chosen: 110 us, 132 with two stages, 129
    // with four and without the buffers).
    static constexpr bool TAB = MODEL == BBX_BR_MRL || MODEL == BBX_BR_FCA || (MODEL == BBX_BR && GEN && !SURR);
    static constexpr int NB_TAB = ROOM >= 3 * B_STAGE + 5 * A_STAGE ? 3 : 2;
    static constexpr int TABW_BYTES = RY * 2048 + 2048;  // (2 KB: barriers and piece contexts)
    static constexpr bool TABW = TAB && TABW_BYTES + NB_TAB * B_STAGE + 4 * A_STAGE <= ROOM;
    // per consumer warp: the surrogate's 64 rows of 32 bytes, or 32 table entries of 64 bytes
    static constexpr int WBUF = SURR || TABW ? RY * 2048 : 0;
    static constexpr int BUDGET = ROOM - (TABW ? TABW_BYTES : 0);
    static constexpr int NB_FIT = HAS_B ? (BUDGET - 5 * A_STAGE) / B_STAGE : 0;
    static constexpr int NB_MAX = TAB ? NB_TAB : 5;
    static constexpr int NB = !HAS_B ? 0 : (TABW ? NB_TAB : (NB_FIT > NB_MAX ? NB_MAX : (NB_FIT < 2 ? 2 : NB_FIT)));
    // (two CTAs: 228 KB an SM, 1 KB of it per CTA the system's)
    static constexpr int NA_TWO = CTAS == 2 ? (114 * 1024 - 1024 - 128 - WBUF - NB * B_STAGE) / (A_STAGE + 176) : 8;
    static constexpr int NA_ROOM = (BUDGET - NB * B_STAGE) / A_STAGE, NA_FIT = NA_ROOM < NA_TWO ? NA_ROOM : NA_TWO;
    static constexpr int NA = NA_FIT > 8 ? 8 : (NA_FIT < 4 ? 4 : NA_FIT);
    static constexpr int RING_OFF = NA * A_STAGE + NB * B_STAGE + WBUF;
    // stages with their barriers, warp buffers, piece contexts
    static constexpr int SMEM = 128 + RING_OFF + NA * 176;
    static_assert(TY % RY == 0 && CY >= 1, "tile rows must be a multiple of the thread rows");
    static_assert(U_RAW % 16 == 0 && F_RAW % 128 == 0 && D_RAW % 128 == 0 && S32_RAW % 128 == 0 && G_RAW % 128 == 0, "stage layout");
};

// The precomputed ingredients of Eq. (Lu) at a node: the unit fibre f (D =
// Dperp I + (Dpar - Dperp) f f^T, Eq. (sigma)) and the W-tilde sums sd_k =
// sum_j (f_j f_k at p + q_j minus at p - q_j), with a void neighbour's fibre
// replaced by f at p (computed once per grid, k_divergence).

// The differences of V around a pair of nodes from which (L u)_p is formed:
// second differences along the axes (void neighbours counted out), the
// four-point cross differences, and the central differences for W-tilde.
struct Diffs {
    float2 xx, yy, zz;  // u(+) + u(-) - (psi(+) + psi(-)) u0
    float2 xy, xz, yz;  // (u(+,+) - u(+,-)) - (u(-,+) - u(-,-))
    float2 x1, y1, z1;  // u(+) - u(-)
};

// (L u)_p of Eq. (Lu) for the pair, from the unit fibres f: with D = Dperp I +
// (Dpar - Dperp) f f^T the weights sum to
//   c_perp (xx + yy + zz) + c_d f.(H f), H_kk the second differences and
//   H_jk a quarter of the cross differences, plus c_s times the W-tilde sums'
// dot product with the central differences.  c_perp = Dperp/h^2, c_d =
// (Dpar-Dperp)/h^2, c_s = c_d/4.  PLANAR: no z terms (a sheet).  Adding a
// vanishing W-tilde term leaves L as it is, so the variants with and without
// the sums agree bitwise where they all vanish.
template <int ANISO, bool PLANAR>
__device__ __forceinline__ float2 lap_pair(const Coef& a, const Diffs& d, const float2* f, const float2* sd) {
    const float2 hy = mul2(splat2(0.5f), f[1]);
    float2 t1 = fma2(hy, d.xy, mul2(f[0], d.xx));
    float2 t2 = mul2(f[1], d.yy);
    float2 lap = add2(d.xx, d.yy);
    float2 q;
    if (PLANAR) {
        q = fma2(f[1], t2, mul2(f[0], t1));
    } else {
        const float2 hz = mul2(splat2(0.5f), f[2]);
        t1 = fma2(hz, d.xz, t1);
        t2 = fma2(hz, d.yz, t2);
        lap = add2(d.xx, add2(d.yy, d.zz));
        q = fma2(f[2], mul2(f[2], d.zz), fma2(f[1], t2, mul2(f[0], t1)));
    }
    float2 L = fma2(splat2(a.c_d), q, mul2(splat2(a.c_perp), lap));
    if (ANISO == AN_SUMS) {
        float2 dv = fma2(sd[1], d.y1, mul2(sd[0], d.x1));
        if (!PLANAR) dv = fma2(sd[2], d.z1, dv);
        L = fma2(splat2(a.c_s), dv, L);
    }
    return L;
}

// ---------------------------------------------------------------------------
// the fused step kernel
// ---------------------------------------------------------------------------

// The reaction surrogate as the step kernel uses it (built on the device from
// a trained network, bbx_set_surrogate): BF16 weights laid out row-major
// [out][in] as 32-bit pairs (W1 padded to 16 inputs), FP32 biases, the
// normalisation and envelope, and the upstroke threshold.
struct SurrogateData {
    // BF16 pairs in MMA-fragment order: for output row n and lane t (of
    // the 4 lanes sharing a row group), the words holding input columns
    // (2t, 2t+1) and (2t+8, 2t+9) of each 16-wide k-step are adjacent.
    uint32_t W1[64 * 8];   // [64 rows][4 lanes][b0, b1]      (inputs padded to 16)
    uint32_t W2[64 * 32];  // [64 rows][4 lanes][4 k-steps][b0, b1]
    uint32_t W3[8 * 32];   // [8 rows][4 lanes][4 k-steps][b0, b1]
    float b1[64], b2[64], b3[8];
    float norm[48];        // mu_in, sd_in, mu_out, sd_out, lo, hi (8 each)
    float inv_sd_in[8];    // 1 / sd_in
    float v_up;            // the exact model runs where V >= v_up
};

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// ReLU and BF16 packing of two FP32 values in one instruction (lo in the low
// half, as the MMA fragments expect).
__device__ __forceinline__ uint32_t relu_pack_bf16(float lo, float hi) {
    uint32_t d;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// The network on the 64 nodes of one warp row (2 per lane) with tensor-core
// MMAs (m16n8k16, BF16 inputs, FP32 accumulation), four m-tiles of 16 nodes.
// Hidden activations stay in registers: the accumulators of two adjacent
// 8-column tiles are the A fragment of the next layer's 16-wide k-tile.  The
// accumulators start from the bias, ReLU and BF16 packing are one instruction
// per pair, and each lane's B fragments are stored contiguously
// (k_build_surrogate), one 64- or 128-bit load per MMA or pair of MMAs.
// wbuf: this warp's 2 KB of shared memory (64 rows of 32 bytes), first the
// BF16 inputs of a row, then, row by row, its 8 FP32 outputs.  All 32 lanes
// must call it.  s: the two nodes' raw states; d: their raw increments.
__device__ __forceinline__ void surrogate_warp64(const SurrogateData* __restrict__ W, unsigned char* wbuf,
                                                 const float (*s)[8], float (*d)[8]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const float* nrm = W->norm;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        uint32_t* row = reinterpret_cast<uint32_t*>(wbuf + (lane * 2 + e) * 32);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            row[k] = pack_bf16((s[e][2 * k] - nrm[2 * k]) * W->inv_sd_in[2 * k],
                               (s[e][2 * k + 1] - nrm[2 * k + 1]) * W->inv_sd_in[2 * k + 1]);
#pragma unroll
        for (int k = 4; k < 8; ++k) row[k] = 0u;
    }
    __syncwarp();
    const uint2* W1 = reinterpret_cast<const uint2*>(W->W1);  // [row][lane t]: (b0, b1)
    const uint4* W2 = reinterpret_cast<const uint4*>(W->W2);  // [row][lane t][kk pair]: (b0, b1, b0', b1')
    const uint4* W3 = reinterpret_cast<const uint4*>(W->W3);
#pragma unroll 1
    for (int q = 0; q < 4; ++q) {
        uint32_t* X = reinterpret_cast<uint32_t*>(wbuf + q * 16 * 32);
        uint32_t a[4] = {X[g * 8 + t], X[(g + 8) * 8 + t], X[g * 8 + t + 4], X[(g + 8) * 8 + t + 4]};
        __syncwarp();  // every lane holds its fragment before the rows are overwritten
        uint32_t h[4][4];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float2 bias = *reinterpret_cast<const float2*>(W->b1 + 8 * j + 2 * t);
            float c[4] = {bias.x, bias.y, bias.x, bias.y};
            const uint2 b = W1[(8 * j + g) * 4 + t];
            mma_bf16(c, a, b.x, b.y);
            const uint32_t lo = relu_pack_bf16(c[0], c[1]), hi = relu_pack_bf16(c[2], c[3]);
            if (j & 1) { h[j >> 1][2] = lo; h[j >> 1][3] = hi; }
            else { h[j >> 1][0] = lo; h[j >> 1][1] = hi; }
        }
        uint32_t h2[4][4];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float2 bias = *reinterpret_cast<const float2*>(W->b2 + 8 * j + 2 * t);
            float c[4] = {bias.x, bias.y, bias.x, bias.y};
            const uint4 b01 = W2[((8 * j + g) * 4 + t) * 2], b23 = W2[((8 * j + g) * 4 + t) * 2 + 1];
            mma_bf16(c, h[0], b01.x, b01.y);
            mma_bf16(c, h[1], b01.z, b01.w);
            mma_bf16(c, h[2], b23.x, b23.y);
            mma_bf16(c, h[3], b23.z, b23.w);
            const uint32_t lo = relu_pack_bf16(c[0], c[1]), hi = relu_pack_bf16(c[2], c[3]);
            if (j & 1) { h2[j >> 1][2] = lo; h2[j >> 1][3] = hi; }
            else { h2[j >> 1][0] = lo; h2[j >> 1][1] = hi; }
        }
        const float2 b3 = *reinterpret_cast<const float2*>(W->b3 + 2 * t);
        float c[4] = {b3.x, b3.y, b3.x, b3.y};
        const uint4 b01 = W3[(g * 4 + t) * 2], b23 = W3[(g * 4 + t) * 2 + 1];
        mma_bf16(c, h2[0], b01.x, b01.y);
        mma_bf16(c, h2[1], b01.z, b01.w);
        mma_bf16(c, h2[2], b23.x, b23.y);
        mma_bf16(c, h2[3], b23.z, b23.w);
        float* Y = reinterpret_cast<float*>(X);
        *reinterpret_cast<float2*>(Y + g * 8 + 2 * t) = make_float2(c[0], c[1]);
        *reinterpret_cast<float2*>(Y + (g + 8) * 8 + 2 * t) = make_float2(c[2], c[3]);
    }
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float4* y = reinterpret_cast<const float4*>(wbuf + (lane * 2 + e) * 32);
        const float4 y0 = y[0], y1 = y[1];
        const float yy[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
#pragma unroll
        for (int k = 0; k < 8; ++k) d[e][k] = fmaf(yy[k], nrm[24 + k], nrm[16 + k]);
    }
    __syncwarp();  // the buffer is reused by the next row
}

// Per-piece context, written into a shared ring by the producer warp when it
// issues the piece's first plane load, and read by the consumer warps once
// that load has landed (the mbarrier orders the two).
struct PieceSlot : Coef {
    int x0, y0, z0, z1;
    int nx, ny, nz, px;
    long long plane, vol;
    float* dst;
    uint16_t* dst16;  // the 16-bit gates of the buffer written (nullptr: all variables 32-bit)
    int32_t* act;
    const uint8_t* stim;
    float stim_amp, dt, theta;
    int step_next;
    int split, rk4;
    const SurrogateData* surr;  // nullptr: exact reaction everywhere
    const float4* tab;          // V-table of the model, or nullptr
    float mp[8];
};
static_assert(sizeof(PieceSlot) <= 176, "piece ring slot size");


// The kinetics step of a pair of nodes: y the state at the start of the step
// (the half-step voltage under Lie splitting), L the diffusion term (0 then),
// Is the stimulus.  All 32 lanes of a warp call it.
template <int MODEL, bool SURR, bool GEN, bool TABW>
__device__ __forceinline__ void react_pair(const PieceSlot& a, const float* mp, float dt, unsigned char* wbufs,
                                           const bool* live, float2* y, float2 L, float2 Is) {
    constexpr int S = Model<MODEL>::S;
    if constexpr (MODEL == BBX_BR && SURR) {
        // the surrogate where the state is inside the training envelope and V
        // below the upstroke threshold; the exact model elsewhere
        const SurrogateData* W = a.surr;
        float ys[2][S];
#pragma unroll
        for (int v = 0; v < S; ++v) {
            ys[0][v] = y[v].x;
            ys[1][v] = y[v].y;
        }
        bool want[2] = {false, false};
        if (W) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                bool in = live[e] && ys[e][0] < W->v_up;
#pragma unroll
                for (int v = 0; v < S; ++v) in = in && ys[e][v] >= W->norm[32 + v] && ys[e][v] <= W->norm[40 + v];
                want[e] = in;
            }
        }
        const bool some = __any_sync(0xffffffffu, want[0] || want[1]);
        if (!(want[0] && want[1])) Model<MODEL>::update2(mp, y, L, Is, dt);
        if (some) {
            float dsur[2][8];
            surrogate_warp64(W, wbufs + (threadIdx.x >> 5) * 2048, ys, dsur);
            if (want[0]) {
#pragma unroll
                for (int v = 0; v < S; ++v) y[v].x = ys[0][v] + dsur[0][v];
                y[0].x += dt * (L.x + Is.x);
            }
            if (want[1]) {
#pragma unroll
                for (int v = 0; v < S; ++v) y[v].y = ys[1][v] + dsur[1][v];
                y[0].y += dt * (L.y + Is.y);
            }
        }
    } else if constexpr (MODEL == BBX_BR || MODEL == BBX_BR_MRL || MODEL == BBX_BR_FCA) {
        // tabulated Rush-Larsen coefficients (of BBX_BR in the general
        // variants only, so the default kernel carries no code for them)
        if (MODEL != BBX_BR || (GEN && a.tab)) {
            float ys[2][S];
#pragma unroll
            for (int v = 0; v < S; ++v) {
                ys[0][v] = y[v].x;
                ys[1][v] = y[v].y;
            }
            auto entry = [&](int k, float V, float* c) {
                const float4* t = a.tab + 4 * kTabN * k;
                if constexpr (TABW)
                    tab_entry_warp(t, V, reinterpret_cast<float4*>(wbufs + (threadIdx.x >> 5) * 2048), c);
                else
                    tab_entry(t, V, c);
            };
            Model<MODEL>::update_tab(mp, entry, ys[0], L.x, Is.x, dt);
            Model<MODEL>::update_tab(mp, entry, ys[1], L.y, Is.y, dt);
#pragma unroll
            for (int v = 0; v < S; ++v) y[v] = make_float2(ys[0][v], ys[1][v]);
        } else if constexpr (MODEL == BBX_BR) {
            Model<MODEL>::update2(mp, y, L, Is, dt);
        }
    } else {
        const float2 src = add2(L, Is);
        if (GEN && a.rk4) {
            float ys[2][S];
#pragma unroll
            for (int v = 0; v < S; ++v) {
                ys[0][v] = y[v].x;
                ys[1][v] = y[v].y;
            }
            rk4_update<MODEL>(mp, ys[0], src.x, 0.0f, dt);
            rk4_update<MODEL>(mp, ys[1], src.y, 0.0f, dt);
#pragma unroll
            for (int v = 0; v < S; ++v) y[v] = make_float2(ys[0][v], ys[1][v]);
        } else {
            Model<MODEL>::update2(mp, y, src, dt);
        }
    }
}


// Barrier over the consumer warps only (named barrier 1), returning the OR of
// a per-thread predicate.
__device__ __forceinline__ bool consumers_sync_or(bool p, int nthreads) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred pi, po;\n\t"
        "setp.ne.u32 pi, %1, 0;\n\t"
        "bar.red.or.pred po, 1, %2, pi;\n\t"
        "selp.u32 %0, 1, 0, po;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)p), "r"(nthreads)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ void consumers_sync(int nthreads) {
    asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

// First row of the tile of load off of a piece: a 3D piece keeps its tile
// (pc.y); a sheet's piece is a run of tile rows pc.z .. pc.w of a column.
template <bool PLANAR, int TY>
__device__ __forceinline__ int tile_row_of(int4 pc, int off) {
    return PLANAR ? (pc.z + off) * TY : pc.y;
}

// Warp-specialised step kernel: warps 0..RY-1 compute (2 x CY nodes per
// thread), warp RY is the producer, warp RY + 1 (FL) tells the producer which
// planes of the neighbouring columns have finished the step before.
//
// GEN: the variant that honours the per-grid scheme and solver settings (Lie
// splitting, RK4 kinetics); the default variant (unsplit, Euler/Rush-Larsen)
// carries no code for them.
//
// PLANAR (grids with nz = 1): a piece is a run of tiles down one column of
// the sheet, pieces[i] = (x0, -, first tile, end tile); each stage holds one
// tile with its one-row halo and the consumers march along y.  The z
// terms of the stencil are left out, which is the 5-point (isotropic) or
// 9-point (anisotropic) sheet operator.  A stage's full barrier completes when
// the plane's bulk copies have landed, its empty barrier when all RY consumer
// warps are done with the plane.  No CTA-wide barrier is taken per plane.
template <int MODEL, bool MASKED, int ANISO, int TY, bool SURR = false, bool PLANAR = false, bool GEN = false,
          int GATES = GATES_F32, bool FL = has_flow(MASKED, Model<MODEL>::S)>
__global__ void __launch_bounds__(step_threads(TY, FL), ctas_per_sm(MASKED, ANISO != AN_ISO, TY, SURR, FL, Model<MODEL>::S))
step_kernel(const __grid_constant__ LaunchArgs L) {
    using P = Plan<MODEL, MASKED, ANISO, TY, SURR, GATES, FL, GEN>;
    static_assert(GATES == GATES_F32 || (MODEL == BBX_BR && !SURR), "16-bit gates: Beeler-Reuter without surrogate");
    constexpr int NG = P::NG, S32 = P::S - NG;  // 16-bit variables last
    constexpr int S = P::S, TX = P::TX, UW = P::UW, CY = P::CY;
    constexpr int NS = P::NA;            // ring A: loaded planes
    constexpr int NB = P::NB;            // ring B: computed planes (0: nothing beyond V)
    constexpr bool HB = P::HAS_B;
    constexpr int NCW = P::RY;  // consumer warps
    constexpr int NCT = 32 * NCW;        // consumer threads
    static_assert(TX == 64, "pair mapping assumes 64-node rows");
    constexpr int CB = TX * TY;  // component stride in a ring-B stage

    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u);
    unsigned char* bstages = smem + NS * P::A_STAGE;    // ring B
    unsigned char* wbufs = bstages + NB * P::B_STAGE;   // per consumer warp: the surrogate's, or table entries'
    PieceSlot* ring = reinterpret_cast<PieceSlot*>(smem + P::RING_OFF);
    // full (the copies have landed) and empty (the consumer warps are done)
    // barriers of a stage of ring A and of ring B
    auto full = [&](int slot) { return reinterpret_cast<uint64_t*>(smem + slot * P::A_STAGE + P::A_BAR); };
    auto empty = [&](int slot) { return full(slot) + 1; };
    auto fullb = [&](int slot) { return reinterpret_cast<uint64_t*>(bstages + slot * P::B_STAGE + P::B_BAR); };
    auto emptyb = [&](int slot) { return fullb(slot) + 1; };
    __shared__ double red_scratch[32];
    __shared__ volatile int abort_flag;
    // launch of several steps: planes each consumer warp has left, loads allowed
    __shared__ int sync_done[P::RY], sync_allowed;

    const int tid = threadIdx.x;
    const int warp = tid / 32, lane = tid % 32;

    // W-tilde sums that vanish at every node of the grid (a fibre field whose
    // tensor does not change along the directions the sums difference, e.g.
    // fibres in the x-y plane turning with z only, or uniform fibres), in a
    // variant that keeps them (masked grids, the general, surrogate and
    // 16-bit-gate kernels; unmasked plain kernels run AN_NO_SUMS instead): a
    // single-grid launch does not copy them, and their part of every ring-B
    // stage holds zeros for the whole launch, so the arithmetic is unchanged
    // and the result is bitwise the one with the sums loaded.  (Batch launches
    // share stages between grids and always copy them.)
    const bool skip_d = ANISO == AN_SUMS && L.single && L.t0.wsum_zero;
    if (skip_d) {
        for (int s = 0; s < NB; ++s) {
            float4* zd = reinterpret_cast<float4*>(bstages + s * P::B_STAGE + P::D_OFF);
            for (int i = tid; i < P::D_RAW / 16; i += P::THREADS) zd[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
    const uint32_t b_bytes = skip_d ? P::B_BYTES - P::D_RAW : P::B_BYTES;
    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(full(s), 1);
            mbar_init(empty(s), NCW);
        }
        for (int s = 0; s < NB; ++s) {
            mbar_init(fullb(s), 1);
            mbar_init(emptyb(s), NCW);
        }
        abort_flag = 0;
        for (int w = 0; w < NCW; ++w) sync_done[w] = 0;
        sync_allowed = 0;
        mbar_init_fence();
    }
    __syncthreads();
    // Programmatic dependent launch: the next step's grid may be scheduled from
    // here on (its CTAs take the SMs this grid's CTAs leave), and every thread
    // waits until the previous grid on the stream has completed and its writes
    // are visible before it touches memory that grid wrote (state, t, n,
    // parity, activation map); with no such grid the wait returns at once.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const int piece_begin = blockIdx.x * L.cta_stride, piece_end = piece_begin + L.cta_count[blockIdx.x];
    int issued = 0;   // producer: plane loads issued (ring A)
    int issuedb = 0;  // producer: computed planes issued (ring B)
    const int n_pieces = piece_end - piece_begin;
    // A launch of several steps: odd CTAs walk their share (a range of the
    // schedule's planes) from its end, so that neighbours along z begin every
    // step at their common border and no CTA waits there for planes that its
    // neighbour has only just done.
    const bool down = P::FLOW && L.n_steps > 1 && (blockIdx.x & 1);

    auto piece_slot = [&](int i) { return down ? piece_end - 1 - i : piece_begin + i; };

    if (warp == NCW) {
        // ---------------- producer warp ----------------
        bool stop = false;
        int lp = 0;
        // the loads the first plane waits for, issued together: the first
        // piece (its slot always exists) and, for one grid, its t, n, parity
        // (a share walked upwards starts with its first slot, whose load need not wait for the count)
        int4 pc_next;
        if (down && n_pieces > 0) pc_next = L.pieces[piece_slot(0)];
        else pc_next = L.pieces[piece_begin];
        TissueDyn d0 = {};
        bool ticketed = !L.single;  // a single-grid launch takes one start ticket per CTA
        if (L.single) {
            const TissueDyn* D = L.t0.dyn;
            d0.t = D->t;
            d0.n = D->n;
            d0.cur = D->cur;
        }
        // ring B copies of the computed plane z (tile rows from y0) of grid T
        auto load_b = [&](const TissueArgs* T, int src, int x0, int y0, int z, int bslot, uint64_t* bar) {
            unsigned char* sb = bstages + bslot * P::B_STAGE;
            if (ANISO) {
                tma_load_4d(sb + P::F_OFF, &T->tm_f, x0, y0, z, 0, bar);
                if (ANISO == AN_SUMS && !skip_d) tma_load_4d(sb + P::D_OFF, &T->tm_d, x0, y0, z, 0, bar);
            }
            if (S > 1 && S32 > 1) tma_load_4d(sb + P::S_OFF, &T->tm_s[src], x0, y0, z, 1, bar);
            if (NG) tma_load_4d(sb + P::G_OFF, &T->tm_g[src], x0, y0, z, 0, bar);
            if (MASKED) tma_load_3d(sb + P::M_OFF, &T->tm_m, x0, y0, z, bar);
        };
        // Single-grid launch of an unmasked grid with a known parity: the
        // first piece from the schedule's shape and its first plane copies
        // (three planes; two tile rows of a sheet) issued now, expected on
        // their barriers but not yet arrived on (the arrival follows the
        // piece context, below).
        bool early = false;
        int n_early = 0;
        int4 pc_early = make_int4(0, 0, 0, 0);
        if (L.single && L.cur_hint >= 0 && L.reg_len > 0 && !L.poison_first_load && !down) {
            const long long p0 = (long long)blockIdx.x * L.reg_planes / L.reg_ctas;
            const long long p1 = ((long long)blockIdx.x + 1) * L.reg_planes / L.reg_ctas;
            if (p1 > p0) {
                const int col = (int)(p0 / L.reg_len), z0 = L.reg_z0 + (int)(p0 % L.reg_len);
                const int z1 = (int)min((long long)(L.reg_z0 + L.reg_len), z0 + (p1 - p0));
                pc_early = make_int4((col % L.reg_nbx) * TX, (col / L.reg_nbx) * L.reg_ty, z0, z1);
                early = true;
                const TissueArgs* T = &L.t0;
                const int src = L.cur_hint;
                const int nl = PLANAR ? z1 - z0 : z1 - z0 + 2;
                n_early = PLANAR ? min(nl, 2) : 3;  // (3D: at most 2 computed planes; NB >= 2)
                if (HB && PLANAR && n_early > NB) n_early = NB;
                if (lane == 0) {
#pragma unroll 1
                    for (int off = 0; off < n_early; ++off) {
                        const int z = PLANAR ? 0 : z0 - 1 + off;  // (outside the array: the copy fills zeros)
                        const int y0 = tile_row_of<PLANAR, TY>(pc_early, off);
                        uint64_t* bar = full(off);
                        unsigned char* st = smem + off * P::A_STAGE;
                        const bool halo = !PLANAR && ((off == 0) || (off == nl - 1));
                        mbar_expect_tx(bar, P::A_BYTES);
                        tma_load_3d(st + P::U_OFF, &T->tm_u[src], pc_early.x - 4, y0 - 1, z, bar);
                        if (HB && !halo) {  // computed plane b = off - 1 (3D) or off (sheet): slot b
                            const int b = PLANAR ? off : off - 1;
                            mbar_expect_tx(fullb(b), b_bytes);
                            load_b(T, src, pc_early.x, y0, z, b, fullb(b));
                        }
                    }
                }
            }
        }
        if (lane == 0 && L.single && L.cur_hint >= 0 &&
            (d0.cur != L.cur_hint ||
             (early && (pc_early.x != pc_next.x || pc_early.y != pc_next.y || pc_early.z != pc_next.z ||
                        pc_early.w != pc_next.w))))
            atomicOr(L.err, ERRBIT_HINT);

        if (lane == 0) {
            const bool stim_s = L.t0.stim && L.t0.stim_amp != 0.0f;
            double t_now = d0.t;  // start time of the step (single-grid launch)
            // the slots and the parities of the empty phases to wait for (a
            // fresh barrier's preceding phase counts as complete)
            int as = 0, ap = 1, bs = 0, bp = 1;
            int n_ready = 0;  // loads the sync warp allows (launch of several steps)
            for (int s = 0; s < L.n_steps && !stop; ++s) {
                for (int i = 0; i < n_pieces && !stop; ++i, ++lp) {
                    const int pi = piece_slot(i);
                    const int4 pc = pc_next;
                    if (n_pieces > 1) pc_next = L.pieces[piece_slot(i + 1 < n_pieces ? i + 1 : 0)];
                    const TissueArgs* T = L.single ? &L.t0 : L.tissues + L.piece_tissue[pi];
                    const TissueDyn* D = L.single ? nullptr : T->dyn;
                    const int src = (L.single ? (L.cur_hint >= 0 ? L.cur_hint : d0.cur) : D->cur) ^ (s & 1);
                    const int nz = MASKED ? (L.single ? L.t0.nz : T->nz) : 0;
                    const int ncomp = pc.w - pc.z, nload = PLANAR ? ncomp : ncomp + 2;
                    // plane of the next load (a sheet: its tile row), walked by dir
                    const int dir = down ? -1 : 1;
                    int zt = down ? (PLANAR ? pc.w - 1 : pc.w) : (PLANAR ? pc.z : pc.z - 1);
                    for (int off = 0; off < nload; ++off, zt += dir) {
                        const bool comp = PLANAR || (off >= 1 && off <= ncomp);  // a computed plane: ring B too
                        if (!ticketed && issued == NS) {
                            // the ring is full: the ticket's round trip overlaps the copies
                            start_ticket(L, d0);
                            ticketed = true;
                        }
                        if (L.poison_first_load && blockIdx.x == 0 && issued == 0) {
                            // fault injection: wait for an empty-slot phase that no
                            // consumer completes; the bounded wait runs out
                            (void)mbar_wait_bounded(empty(0), 0, L.wait_limit);
                            stop = true;
                        } else if (!mbar_wait_bounded(empty(as), ap, L.wait_limit)) {
                            stop = true;
                        } else if (HB && comp && !mbar_wait_bounded(emptyb(bs), bp, L.wait_limit)) {
                            stop = true;
                        }
                        if (P::FLOW && s > 0 && issued >= n_ready && !stop) {
                            const long long t0 = clock64();
                            while ((n_ready = ld_shared_acquire(&sync_allowed)) <= issued) {
                                if (abort_flag || clock64() - t0 > L.wait_limit) {
                                    stop = true;
                                    break;
                                }
                            }
                        }
                        if (stop || abort_flag) {
                            stop = true;
                            break;
                        }
                        if (off == 0) {
                            PieceSlot& r = ring[lp % NS];
                            r.x0 = pc.x; r.y0 = pc.y; r.z0 = pc.z; r.z1 = pc.w;
                            r.dst = L.single ? (src ? L.t0.state[0] : L.t0.state[1]) : T->state[src ^ 1];
                            r.dst16 = L.single ? (src ? L.t0.gate16[0] : L.t0.gate16[1]) : T->gate16[src ^ 1];
                            r.stim_amp = 0.0f;
                            if (L.single ? stim_s : T->stim && T->stim_amp != 0.0f) {
                                double tn = L.single ? t_now : D->t;
                                if (!L.single)
                                    for (int q = 0; q < s; ++q) tn = tn + T->dt_d;
                                if (tn >= T->t_on && tn < T->t_off) r.stim_amp = T->stim_amp;
                            }
                            r.step_next = (int)((L.single ? d0.n : D->n) + s + 1);
                            if (!L.single || lp < NS) {  // the rest of a single grid's contexts stays in the ring
                                r.nx = T->nx; r.ny = T->ny; r.nz = T->nz; r.px = T->px;
                                r.plane = T->plane; r.vol = T->vol;
                                r.act = T->act;
                                r.stim = T->stim;
                                r.dt = T->dt;
                                r.theta = T->theta;
                                r.split = T->split;
                                r.rk4 = T->rk4;
                                r.c_perp = T->c_perp; r.c_d = T->c_d; r.c_s = T->c_s; r.c_iso = T->c_iso;
                                r.surr = T->surr;
                                r.tab = T->tab;
#pragma unroll
                                for (int q = 0; q < 8; ++q) r.mp[q] = T->mp[q];
                            }
                        }
                        const int z = PLANAR ? 0 : zt;
                        const int y0 = PLANAR ? zt * TY : pc.y;  // first row of the tile
                        uint64_t* bar = full(as);
                        unsigned char* st = smem + as * P::A_STAGE;
                        if (early && issued < n_early) {
                            mbar_arrive(bar);  // its copies were issued at the start
                            if (HB && comp) mbar_arrive(fullb(bs));
                        } else if (MASKED && (z < 0 || z >= nz)) {
                            mbar_arrive(bar);  // plane outside the array: not read (never a computed one)
                        } else {
                            // (an unmasked grid's plane outside the array: the copy fills zeros)
                            mbar_arrive_expect_tx(bar, P::A_BYTES);
                            tma_load_3d(st + P::U_OFF, &T->tm_u[src], pc.x - 4, y0 - 1, z, bar);
                            if (HB && comp) {
                                mbar_arrive_expect_tx(fullb(bs), b_bytes);
                                load_b(T, src, pc.x, y0, z, bs, fullb(bs));
                            }
                        }
                        ++issued;
                        if (++as == NS) {
                            as = 0;
                            ap ^= 1;
                        }
                        if (HB && comp) {
                            ++issuedb;
                            if (++bs == NB) {
                                bs = 0;
                                bp ^= 1;
                            }
                        }
                    }
                }
                if (L.single) t_now = t_now + L.t0.dt_d;
            }
            if (!ticketed) start_ticket(L, d0);  // every CTA takes it, also on a short or aborted run
            if (stop) abort_flag = 1;
        }
        __syncwarp();
    } else if (P::FLOW && warp == NCW + 1) {
        // ---------------- sync warp (launch of several steps) ----------------
        // flags[] holds, per column and computed plane, the running number of
        // the last step done there.  A plane of V may be copied for step s
        // (after the first) once the step before is done at that plane in the
        // 3 x 3 columns around it (the box's halo; a sheet: the 3 x 3 tiles):
        // the copies of planes z-1 .. z+1 then also show that no CTA still
        // reads, for the step before, the plane z that step s overwrites in
        // the other buffer.  This warp sets the flags of the planes its CTA
        // has done and tells the producer how many loads may go; in the
        // producer itself the fence before a flag (1100 to 2300 cycles, the
        // SM's stores in flight) and the flags' round trips would each stall
        // the copies (512x512x256 slab: 2970 cycles a plane against 2420).
        if (L.n_steps > 1 && n_pieces > 0) {
            int4 fg_pc = L.pieces[piece_slot(0)], al_pc = fg_pc;
            PieceFlags fg_pf = L.piece_flags[piece_slot(0)], al_pf = fg_pf;
            // next flag to set, next load to allow: the piece and the place in it
            int fg_i = 0, fg_t = 0, fg_step = 0, n_flag = 0;
            int al_i = 0, al_off = 0, al_step = 1, n_allow = 0;
            int planes = 0;  // computed planes of a step
            for (int i = 0; i < n_pieces; ++i) {
                const int4 q = n_pieces > 1 ? L.pieces[piece_slot(i)] : fg_pc;
                planes += q.w - q.z;
                n_allow += q.w - q.z + (PLANAR ? 0 : 2);
            }
            const int n_all = planes * (L.n_steps - 1);
            const int j = lane / 9, c = lane - 9 * j, dx = c % 3 - 1, dy = c / 3 - 1;
            long long t0 = clock64();
            while (n_flag < n_all || al_step < L.n_steps) {
                bool moved = false;
                // planes that every consumer warp has left (the counts are released after the warp's stores)
                int done = lane < NCW ? ld_shared_acquire(&sync_done[lane]) : 0x7fffffff;
                done = min(__reduce_min_sync(0xffffffffu, done), n_all);
                if (done > n_flag) {
                    __syncwarp();
                    if (lane == 0) asm volatile("fence.acq_rel.gpu;" ::: "memory");
                    while (n_flag < done) {
                        const int n = min(done - n_flag, fg_pc.w - fg_pc.z - fg_t);  // planes of one column
                        int* f = L.flags + fg_pf.base + (down ? fg_pc.w - 1 - fg_t : fg_pc.z + fg_t);
                        if (lane == 0)
                            for (int q = 0; q < n; ++q) st_flag(f + (down ? -q : q), L.epoch + fg_step + 1);
                        n_flag += n;
                        fg_t += n;
                        if (fg_t == fg_pc.w - fg_pc.z) {
                            fg_t = 0;
                            if (++fg_i == n_pieces) {
                                fg_i = 0;
                                ++fg_step;
                            }
                            if (n_pieces > 1) {
                                fg_pc = L.pieces[piece_slot(fg_i)];
                                fg_pf = L.piece_flags[piece_slot(fg_i)];
                            }
                        }
                    }
                    moved = true;
                }
                if (al_step < L.n_steps) {
                    // nine flags of each of the next 12 loads' planes
                    const int nload = al_pc.w - al_pc.z + (PLANAR ? 0 : 2);
                    const bool col_in = lane < 27 && (dx == 0 || (al_pf.has & (dx < 0 ? 1 : 2))) &&
                                        (PLANAR || dy == 0 || (al_pf.has & (dy < 0 ? 4 : 8)));
                    const int* fl = L.flags + al_pf.base + dx * al_pf.len + (PLANAR ? 0 : dy * al_pf.row);
                    const int want = L.epoch + al_step;
                    int v[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int o = al_off + j + 3 * q;
                        const int z = (down ? al_pc.w - (PLANAR ? 1 : 0) - o : al_pc.z - (PLANAR ? 0 : 1) + o) + (PLANAR ? dy : 0);
                        v[q] = want;
                        if (col_in && o < nload && z >= al_pf.z0 && z < al_pf.z0 + al_pf.len) v[q] = ld_flag(fl + z);
                    }
                    int ok = 0;
                    bool run = true;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const unsigned m = __ballot_sync(0xffffffffu, (int)((unsigned)v[q] - (unsigned)want) >= 0);
#pragma unroll
                        for (int e = 0; e < 3; ++e) {
                            run = run && ((m >> (9 * e)) & 0x1ffu) == 0x1ffu;
                            if (run) ok = 3 * q + e + 1;
                        }
                    }
                    ok = min(ok, nload - al_off);
                    if (ok > 0) {
                        // the other CTAs' stores (acquired with the flags) before this CTA's copies of them
                        __syncwarp();
                        asm volatile("fence.proxy.async;" ::: "memory");
                        __syncwarp();
                        n_allow += ok;
                        if (lane == 0) st_shared_release(&sync_allowed, n_allow);
                        al_off += ok;
                        if (al_off == nload) {
                            al_off = 0;
                            if (++al_i == n_pieces) {
                                al_i = 0;
                                ++al_step;
                            }
                            if (n_pieces > 1) {
                                al_pc = L.pieces[piece_slot(al_i)];
                                al_pf = L.piece_flags[piece_slot(al_i)];
                            }
                        }
                        moved = true;
                    }
                }
                if (moved) t0 = clock64();
                if (__any_sync(0xffffffffu, abort_flag || clock64() - t0 > L.wait_limit)) {
                    abort_flag = 1;
                    break;
                }
            }
        }
    } else {
        // ---------------- consumer warps ----------------
        const int tx = tid % 32, row0 = (tid / 32) * CY;  // node pair (x, x+1) = x0 + 2 tx
        float2 vhi = splat2(0.0f), vlo = splat2(0.0f);  // the tissue sums of the pair's two columns
        bool timed_out = false;
        int lr = 0;                // slot of the piece's context
        int aw = 0, apar = 0;  // ring A: byte offset and phase parity of the next plane to wait for
        int bw = 0, bpar = 0;  // ring B: the same
        // The wait for a phase; false when it ran out (or another part of the CTA gave up).
        auto wait_bar = [&](uint64_t* bar, int parity) {
            if (mbar_try_wait(bar, parity)) return true;
            const long long t0 = clock64();
            while (!mbar_try_wait(bar, parity)) {
                if (abort_flag || clock64() - t0 > L.wait_limit) {
                    abort_flag = 1;
                    return false;
                }
            }
            return true;
        };
        auto bar_a = [&](int off) { return reinterpret_cast<uint64_t*>(smem + off + P::A_BAR); };
        // Wait for the next plane of ring A; its stage's byte offset.
        auto next_plane = [&]() {
            const int o = aw;
            if (!timed_out && !wait_bar(bar_a(o), apar)) timed_out = true;
            aw += P::A_STAGE;
            if (aw == NS * P::A_STAGE) {
                aw = 0;
                apar ^= 1;
            }
            return o;
        };
        auto ld2 = [&](const float* U, int o) { return *reinterpret_cast<const float2*>(U + o); };
        const int toff = row0 * UW + (2 * tx + 4);  // stage index of node (x, yb - 1), even
        const int boff = row0 * TX + 2 * tx;        // ring-B index of node (x, yb)
        const int n_walk = (P::FLOW ? L.n_steps : 1) * n_pieces;  // the pieces of every step in order
        int n_left = 0;  // planes this warp has left
        for (int pw = 0; pw < n_walk; ++pw) {
            const bool last_step = pw >= n_walk - n_pieces;
            int op = PLANAR ? 0 : next_plane();  // the piece's first load carries its context
            int oc = next_plane();
            const PieceSlot& a = ring[lr];
            lr = lr + 1 == NS ? 0 : lr + 1;
            const int ncomp = timed_out ? 0 : a.z1 - a.z0;  // (a context that never came is not read further)
            Coef co;
            co.c_perp = a.c_perp; co.c_d = a.c_d; co.c_s = a.c_s; co.c_iso = a.c_iso;
            float mp[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) mp[i] = a.mp[i];
            const float theta = a.theta, dt = a.dt;
            const bool stim_on = a.stim_amp != 0.0f;
            const int nx = a.nx, ny = a.ny, nz = a.nz, px = a.px;
            const int x = a.x0 + 2 * tx;  // first node of this thread's pair
            const bool x_in = x < nx, x1_in = x + 1 < nx;
            // unmasked grids: minus the number of x neighbours, and psi(x+1) - psi(x-1), of the two nodes
            const float px0 = x1_in ? 1.0f : 0.0f, mx0 = x > 0 ? 1.0f : 0.0f, px1 = x + 2 < nx ? 1.0f : 0.0f;
            const float2 ncx = MASKED ? splat2(-2.0f) : make_float2(-(px0 + mx0), -(px1 + 1.0f));
            const float2 ex = make_float2(px0 - mx0, px1 - 1.0f);
            // marched upwards, or downwards (then the plane before the current one lies above it)
            const int first = down ? a.z1 - 1 : a.z0, dir = down ? -1 : 1;
            int yb = (PLANAR ? first * TY : a.y0) + row0;  // y of this thread's first row
            int k = PLANAR ? 0 : first;
            float* pd = a.dst + (long long)k * a.plane + (long long)yb * px + x;  // node (x, yb) of plane k (even)
            const long long gstep = (PLANAR ? (long long)TY * px : a.plane) * dir;
            float* const dst = a.dst;
            const long long vol = a.vol;
            for (int t = 0; t < ncomp; ++t) {
                const int on = PLANAR ? (t ? (oc = next_plane()) : oc) : next_plane();
                uint64_t* barb = reinterpret_cast<uint64_t*>(bstages + bw + P::B_BAR);
                if (HB && !timed_out && !wait_bar(barb, bpar)) timed_out = true;
                if (timed_out) break;
                const float* Uc = reinterpret_cast<const float*>(smem + oc + P::U_OFF) + toff;
                const int ozm = down ? on : op, ozp = down ? op : on;  // planes k-1 and k+1
                const float* Up = reinterpret_cast<const float*>(smem + ozm + P::U_OFF) + toff;
                const float* Un = reinterpret_cast<const float*>(smem + ozp + P::U_OFF) + toff;
                const unsigned char* stb = bstages + bw;
                const float* Fb = reinterpret_cast<const float*>(stb + P::F_OFF) + boff;  // [3][TY][TX]
                const float* Db = reinterpret_cast<const float*>(stb + P::D_OFF) + boff;  // [3][TY][TX]
                const float* Sv = reinterpret_cast<const float*>(stb + P::S_OFF) + boff;
                const uint32_t* Mb = reinterpret_cast<const uint32_t*>(stb + P::M_OFF) + boff;
                const bool zn_ok = k + 1 < nz, zp_ok = k > 0;
                const int nrows = ny - yb;  // rows of this thread inside the array
                const float ncz = MASKED || (zn_ok && zp_ok) ? -2.0f : (zn_ok || zp_ok ? -1.0f : 0.0f);
                // unmasked: this thread's rows touch the array's border in y
                const bool yborder = !MASKED && (yb == 0 || nrows <= CY);
                const float2 ncp = add2(ncx, splat2(-2.0f + (PLANAR ? 0.0f : ncz)));  // (isotropic: all axes)
                // unmasked: some cross difference misses a neighbour on one side only (a row or plane at
                // the array's border)
                const bool border = !MASKED && ANISO && (yborder || (!PLANAR && !(zn_ok && zp_ok)));

                // Sliding window down the rows: plane k at x-1..x+2, the own pair of planes k+-1.
                float2 wB[CY + 2], wN[CY + 2], wP[CY + 2];
                float wA[CY + 2], wC[CY + 2];
                auto load_row = [&](int w) {  // row w - 1 of the window
                    const int o = w * UW;
                    wB[w] = ld2(Uc, o);
                    if (ANISO || (w > 0 && w <= CY)) {
                        wA[w] = Uc[o - 1];
                        wC[w] = Uc[o + 2];
                    }
                    if (!PLANAR && (ANISO || (w > 0 && w <= CY))) {
                        wN[w] = ld2(Un, o);
                        wP[w] = ld2(Up, o);
                    }
                };
                load_row(0);
                load_row(1);
#pragma unroll
                for (int r = 0; r < CY; ++r) {
                    load_row(r + 2);
                    if (r >= nrows) continue;  // (warp-uniform)
                    const int w = r + 1;
                    const float2 u0 = wB[w];
                    bool live[2] = {x_in, x1_in};
                    uint2 psi = make_uint2(0u, 0u);
                    bool edge = false;  // a tissue node of the pair has a void neighbour
                    if (MASKED) {
                        psi = *reinterpret_cast<const uint2*>(Mb + r * TX);
                        live[0] = (psi.x & PSI_TISSUE) != 0;
                        live[1] = (psi.y & PSI_TISSUE) != 0;
                        edge = (live[0] && !(psi.x & PSI_INTERIOR)) || (live[1] && !(psi.y & PSI_INTERIOR));
                    }
                    float2 Lr;
                    float miss = 0.0f;  // y neighbours outside the array
                    if (!MASKED && yborder) miss = (r == 0 && yb == 0 ? 1.0f : 0.0f) + (r + 1 == nrows ? 1.0f : 0.0f);
                    // a neighbour's value, u0 in place of a void one (every difference with it then vanishes)
                    auto nb = [&](uint32_t bit, float a0, float a1) {
                        return make_float2(psi.x & bit ? a0 : u0.x, psi.y & bit ? a1 : u0.y);
                    };
                    float2 sx = make_float2(__fadd_rn(u0.y, wA[w]), __fadd_rn(wC[w], u0.x));
                    float2 sy = add2(wB[w + 1], wB[w - 1]), sz;
                    if (!PLANAR) sz = add2(wN[w], wP[w]);
                    if (MASKED && edge) {
                        sx = add2(nb(PSI_XP, u0.y, wC[w]), nb(PSI_XM, wA[w], u0.x));
                        sy = add2(nb(PSI_YP, wB[w + 1].x, wB[w + 1].y), nb(PSI_YM, wB[w - 1].x, wB[w - 1].y));
                        if (!PLANAR) sz = add2(nb(PSI_ZP, wN[w].x, wN[w].y), nb(PSI_ZM, wP[w].x, wP[w].y));
                    }
                    if (!ANISO) {
                        float2 sum = add2(sx, sy);
                        if (!PLANAR) sum = add2(sum, sz);
                        float2 nc = ncp;
                        if (!MASKED && yborder) nc = add2(nc, splat2(miss));
                        Lr = mul2(splat2(co.c_iso), fma2(nc, u0, sum));
                    } else {
                        Diffs d;
                        d.xx = fma2(ncx, u0, sx);
                        d.yy = fma2(splat2(miss - 2.0f), u0, sy);
                        d.y1 = sub2(wB[w + 1], wB[w - 1]);
                        const float ya = __fsub_rn(wA[w + 1], wA[w - 1]), yc = __fsub_rn(wC[w + 1], wC[w - 1]);
                        d.xy = make_float2(__fsub_rn(d.y1.y, ya), __fsub_rn(yc, d.y1.x));
                        float nA, nC, pA, pC;
                        if (!PLANAR) {
                            nA = Un[w * UW - 1], nC = Un[w * UW + 2], pA = Up[w * UW - 1], pC = Up[w * UW + 2];
                            d.zz = fma2(splat2(ncz), u0, sz);
                            d.z1 = sub2(wN[w], wP[w]);
                            d.xz = make_float2(__fsub_rn(d.z1.y, __fsub_rn(nA, pA)), __fsub_rn(__fsub_rn(nC, pC), d.z1.x));
                            d.yz = sub2(sub2(wN[w + 1], wP[w + 1]), sub2(wN[w - 1], wP[w - 1]));
                        }
                        if (ANISO == AN_SUMS)
                            d.x1 = make_float2(__fsub_rn(u0.y, wA[w]), __fsub_rn(wC[w], u0.x));
                        if (MASKED && edge) {
                            d.xy = sub2(sub2(nb(PSI_XPYP, wB[w + 1].y, wC[w + 1]), nb(PSI_XPYM, wB[w - 1].y, wC[w - 1])),
                                        sub2(nb(PSI_XMYP, wA[w + 1], wB[w + 1].x), nb(PSI_XMYM, wA[w - 1], wB[w - 1].x)));
                            if (!PLANAR) {
                                d.xz = sub2(sub2(nb(PSI_XPZP, wN[w].y, nC), nb(PSI_XPZM, wP[w].y, pC)),
                                            sub2(nb(PSI_XMZP, nA, wN[w].x), nb(PSI_XMZM, pA, wP[w].x)));
                                d.yz = sub2(sub2(nb(PSI_YPZP, wN[w + 1].x, wN[w + 1].y), nb(PSI_YPZM, wP[w + 1].x, wP[w + 1].y)),
                                            sub2(nb(PSI_YMZP, wN[w - 1].x, wN[w - 1].y), nb(PSI_YMZM, wP[w - 1].x, wP[w - 1].y)));
                            }
                            // (a W-tilde sum is 0 where its axis misses a neighbour, whose value may be anything)
                            if (ANISO == AN_SUMS) {
                                d.x1 = sub2(nb(PSI_XP, u0.y, wC[w]), nb(PSI_XM, wA[w], u0.x));
                                d.y1 = sub2(nb(PSI_YP, wB[w + 1].x, wB[w + 1].y), nb(PSI_YM, wB[w - 1].x, wB[w - 1].y));
                                if (!PLANAR) d.z1 = sub2(nb(PSI_ZP, wN[w].x, wN[w].y), nb(PSI_ZM, wP[w].x, wP[w].y));
                            }
                        }
                        if (border) {
                            // psi = 0 on one side only leaves a cross difference short of u0 where both
                            // axes end (the array's edges)
                            const float ey = (r + 1 == nrows ? 0.0f : 1.0f) - (r == 0 && yb == 0 ? 0.0f : 1.0f);
                            const float ez = (zn_ok ? 1.0f : 0.0f) - (zp_ok ? 1.0f : 0.0f);
                            d.xy = fma2(mul2(ex, splat2(-ey)), u0, d.xy);
                            if (!PLANAR) {
                                d.xz = fma2(mul2(ex, splat2(-ez)), u0, d.xz);
                                d.yz = fma2(splat2(-ey * ez), u0, d.yz);
                            }
                        }
                        const float2 f[3] = {ld2(Fb, r * TX), ld2(Fb, r * TX + CB), ld2(Fb, r * TX + 2 * CB)};
                        float2 sd[3];
                        if (ANISO == AN_SUMS) {
#pragma unroll
                            for (int c = 0; c < 3; ++c) sd[c] = ld2(Db, r * TX + c * CB);
                        }
                        Lr = lap_pair<ANISO, PLANAR>(co, d, f, sd);
                    }

                    // reaction, stores, activation, tissue sum (predicated)
                    float* const pr = pd + r * px;
                    float2 y[S];
                    y[0] = u0;
#pragma unroll
                    for (int v = 1; v < S32; ++v) y[v] = ld2(Sv, (v - 1) * CB + r * TX);
#pragma unroll
                    for (int v = S32; v < S; ++v) {  // 16-bit gates, decoded to FP32
                        const uint32_t w16 = *reinterpret_cast<const uint32_t*>(
                            stb + P::G_OFF + 2 * ((v - S32) * CB + boff + r * TX));
                        y[v] = gate_decode2<GATES>(w16);
                    }
                    float2 Is = splat2(0.0f);
                    if (stim_on) {
                        const long long gr = pr - dst;
                        if (live[0] && a.stim[gr]) Is.x = a.stim_amp;
                        if (live[1] && a.stim[gr + 1]) Is.y = a.stim_amp;
                    }
                    if (GEN && a.split) {
                        // Lie splitting: the diffusion substep on its own, then
                        // the kinetics step from the half-step voltage
                        y[0] = fma2(splat2(dt), Lr, y[0]);
                        Lr = splat2(0.0f);
                    }
                    react_pair<MODEL, SURR, GEN, P::TABW>(a, mp, dt, wbufs, live, y, Lr, Is);
                    if (live[0] && live[1]) {
                        float* q = pr;
#pragma unroll
                        for (int v = 0; v < S32; ++v) {
                            st_global(q, y[v]);
                            q += vol;
                        }
#pragma unroll
                        for (int v = S32; v < S; ++v)
                            st_global_u32(a.dst16 + (long long)(v - S32) * vol + (pr - dst), gate_encode2<GATES>(y[v].x, y[v].y));
                    } else if (live[0] || live[1]) {
#pragma unroll
                        for (int e = 0; e < 2; ++e)
                            if (live[e]) {
#pragma unroll
                                for (int v = 0; v < S32; ++v)
                                    st_global(pr + (long long)v * vol + e, e ? y[v].y : y[v].x);
#pragma unroll
                                for (int v = S32; v < S; ++v)
                                    st_global_u16(a.dst16 + (long long)(v - S32) * vol + (pr - dst) + e,
                                                  gate_encode<GATES>(e ? y[v].y : y[v].x));
                            }
                    }
                    const bool up0 = u0.x < theta && theta <= y[0].x, up1 = u0.y < theta && theta <= y[0].y;
                    if (up0 || up1) {
                        const long long gr = pr - dst;
                        if (up0 && live[0] && a.act[gr] == BBX_ACT_NONE) a.act[gr] = a.step_next;
                        if (up1 && live[1] && a.act[gr + 1] == BBX_ACT_NONE) a.act[gr + 1] = a.step_next;
                    }
                    // (columns outside an unmasked array are left out of the piece's sum)
                    if (last_step) two_sum_add2(vhi, vlo, MASKED ? make_float2(live[0] ? y[0].x : 0.0f, live[1] ? y[0].y : 0.0f) : y[0]);
                }

                __syncwarp();
                if (P::FLOW) ++n_left;
                if (lane == 0) {
                    if (P::FLOW && !last_step) st_shared_release(&sync_done[warp], n_left);
                    mbar_arrive(bar_a(PLANAR ? oc : op) + 1);
                    if (HB) mbar_arrive(barb + 1);
                }
                if (HB) {
                    bw += P::B_STAGE;
                    if (bw == NB * P::B_STAGE) {
                        bw = 0;
                        bpar ^= 1;
                    }
                }
                op = oc;
                oc = on;
                if (PLANAR) yb += dir * TY;
                else k += dir;
                pd += gstep;
            }
            __syncwarp();
            if (!PLANAR && lane == 0) {  // release the piece's last two planes
                mbar_arrive(bar_a(op) + 1);
                mbar_arrive(bar_a(oc) + 1);
            }
            if (!last_step) continue;
            // per-piece partial of the tissue sum, and a vote on timeouts
            const int pi = down ? piece_end - 1 - (pw - (n_walk - n_pieces)) : piece_begin + (pw - (n_walk - n_pieces));
            // The two columns are joined in FP32, by TwoSum, before FP64: the FP64 pipe takes an SM's warps one
            // after the other (a warp's instruction some 16 cycles), and joined in FP64, with four more
            // instructions a warp, a one-step launch took 0.3 us longer with one CTA on an SM, 1 us with four
            // (FHN sheets in 7-row tiles: 64x64 5.7 -> 6.0 us, 400x400 7.6 -> 8.7 us; as here 5.7 and 7.6).
            F2 vs = {x_in ? vhi.x : 0.0f, x_in ? vlo.x : 0.0f};
            two_sum_add(vs, x1_in ? vhi.y : 0.0f);
            vs.lo += x1_in ? vlo.y : 0.0f;
            double v = (double)vs.hi + (double)vs.lo;
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) red_scratch[warp] = v;
            const bool any_to = consumers_sync_or(timed_out, NCT);
            if (tid == 0) {
                double s = 0.0;
                for (int w = 0; w < NCW; ++w) s += red_scratch[w];
                L.partials[pi] = s;
                if (!isfinite(s)) atomicOr(L.err, ERRBIT_NAN);
            }
            consumers_sync(NCT);
            if (!L.single && warp == 0 && !any_to) grid_piece_done(L, pi, lane);
            vhi = vlo = splat2(0.0f);
            if (any_to) break;
        }
        if (timed_out) abort_flag = 1;
    }
    __syncthreads();

    if (abort_flag && warp == NCW && lane == 0) {
        // Give the loads that may still be in flight a bounded chance to land.
        atomicOr(L.err, ERRBIT_TIMEOUT);
        for (int j = issued > NS ? issued - NS : 0; j < issued; ++j)
            (void)mbar_wait_bounded(full(j % NS), (j / NS) & 1, L.wait_limit);
        for (int j = issuedb > NB ? issuedb - NB : 0; j < issuedb; ++j)
            (void)mbar_wait_bounded(fullb(j % NB), (j / NB) & 1, L.wait_limit);
    }
    step_finalize(L);
}

// host-visible description of one compiled step kernel
struct StepKernel {
    const void* fn;
    int smem;
    int threads;
    int ty;
    bool flow = false;    // may take several steps in one launch
    bool gather = false;  // its warps gather table entries together
};

}  // namespace bbx
