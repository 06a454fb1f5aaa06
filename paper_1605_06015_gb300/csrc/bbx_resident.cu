// Resident multi-step kernel for small sheets: a cluster of CTAs holds the
// whole sheet in distributed shared memory and advances many time steps in
// one launch.  Each CTA owns a band of rows; the stencil reads the rows next
// to its band from the neighbouring CTAs' shared memory, and one cluster
// barrier per step separates a step's writes from the next step's reads.
// Nothing goes through global memory between steps except activation events,
// so a step costs neither a launch nor a DRAM round trip: the unsplit step of
// section "Computation of intermediate expressions" with the 5-point
// operator of an isotropic sheet (faces only; no-flux edges: a missing
// neighbour contributes nothing).
#include <limits.h>

#include <cooperative_groups.h>

#include "bbx_device.cuh"

namespace cg = cooperative_groups;

namespace bbx {

namespace {

// CTAs in the cluster: 16 (a non-portable cluster size the launch asks for),
// else the portable 8
constexpr int kResCtasLarge = 16, kResCtasPortable = 8;
constexpr int kResThreads = 1024;
constexpr int kResMaxSmem = 200 * 1024;
constexpr long long kWaitLimit = 4000000000LL;  // SM cycles a wait may spin (about 2 s)

__device__ __forceinline__ void res_two_sum(double& hi, double& lo, double b) {
    const double s = hi + b, bb = s - hi;
    lo += (hi - (s - bb)) + (b - bb);
    hi = s;
}

// Launched with NC CTAs forming one cluster.  Shared memory per CTA:
// two buffers of the band's V (maxr rows of nx) and S-1 buffers of the other
// variables, updated in place (only V is read by neighbours).
template <int MODEL, int NC>
__global__ void __cluster_dims__(NC, 1, 1) __launch_bounds__(kResThreads, 1)
    k_resident_sheet(const TissueArgs* __restrict__ T, int n_steps, int* __restrict__ err) {
    constexpr int S = Model<MODEL>::S;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    extern __shared__ float sm[];
    __shared__ double red_hi[kResThreads / 32];
    __shared__ double cl_part[NC];

    const int nx = T->nx, ny = T->ny, px = T->px;
    const long long vol = T->vol;
    const int maxr = (ny + NC - 1) / NC;
    const int rb0 = (int)((long long)ny * rank / NC), rb1 = (int)((long long)ny * (rank + 1) / NC);
    const int nr = rb1 - rb0;
    const int nb = nr * nx;
    float* V[2] = {sm, sm + maxr * nx};
    float* Wv = sm + 2 * maxr * nx;  // the other variables, (S-1) x maxr x nx
    // the neighbouring bands' V buffers (rows rb0-1 and rb1 live there)
    const int up = rank > 0 ? rank - 1 : rank, dn = rank + 1 < NC ? rank + 1 : rank;
    const int nr_up = rb0 - (int)((long long)ny * up / NC);
    float* Vu[2] = {cl.map_shared_rank(V[0], up), cl.map_shared_rank(V[1], up)};
    float* Vd[2] = {cl.map_shared_rank(V[0], dn), cl.map_shared_rank(V[1], dn)};

    TissueDyn* D = T->dyn;
    const int cur0 = D->cur;
    double t = D->t;
    long long n = D->n;
    const float* src = T->state[cur0];
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        const int r = i / nx, x = i - r * nx;
        const long long gi = (long long)(rb0 + r) * px + x;
        V[0][i] = src[gi];
#pragma unroll
        for (int v = 1; v < S; ++v) Wv[(v - 1) * maxr * nx + i] = src[v * vol + gi];
    }
    cl.sync();

    const float c = T->c_iso, dt = T->dt, theta = T->theta;
    float mp[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) mp[k] = T->mp[k];
    const int dr = (int)blockDim.x / nx, dx = (int)blockDim.x - dr * nx;
    int p = 0;
    for (int s = 0; s < n_steps; ++s) {
        const bool stim_on = T->stim && T->stim_amp != 0.0f && t >= T->t_on && t < T->t_off;
        const float* Vo = V[p];
        float* Vn = V[p ^ 1];
        const float* Vup = Vu[p];
        const float* Vdn = Vd[p];
        // node i = r nx + x of the band, advanced by blockDim without divisions
        int r = (int)threadIdx.x / nx, x = (int)threadIdx.x - r * nx;
        for (int i = threadIdx.x; i < nb; i += blockDim.x) {
            const int y = rb0 + r;
            const float u0 = Vo[i];
            const float xp = x + 1 < nx ? Vo[i + 1] : u0;
            const float xm = x > 0 ? Vo[i - 1] : u0;
            const float ym = r > 0 ? Vo[i - nx] : (y > 0 ? Vup[(nr_up - 1) * nx + x] : u0);
            const float yp = r + 1 < nr ? Vo[i + nx] : (y + 1 < ny ? Vdn[x] : u0);
            const float L = c * (((xp - u0) + (xm - u0)) + ((yp - u0) + (ym - u0)));
            float yv[S];
            yv[0] = u0;
#pragma unroll
            for (int v = 1; v < S; ++v) yv[v] = Wv[(v - 1) * maxr * nx + i];
            const long long gi = (long long)y * px + x;
            const float Is = (stim_on && T->stim[gi]) ? T->stim_amp : 0.0f;
            Model<MODEL>::update(mp, yv, L, Is, dt);
            Vn[i] = yv[0];
#pragma unroll
            for (int v = 1; v < S; ++v) Wv[(v - 1) * maxr * nx + i] = yv[v];
            if (u0 < theta && theta <= yv[0] && T->act[gi] == BBX_ACT_NONE) T->act[gi] = (int32_t)(n + 1);
            x += dx;
            r += dr;
            if (x >= nx) {
                x -= nx;
                ++r;
            }
        }
        cl.sync();  // every band's new V is written before any band reads it
        p ^= 1;
        t = t + T->dt_d;
        n += 1;
    }

    // the new state into the buffer that becomes current, and the FP64 total of V
    const int cur1 = cur0 ^ (n_steps & 1);
    float* dst = T->state[cur1];
    double hi = 0.0, lo = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        const int r = i / nx, x = i - r * nx;
        const long long gi = (long long)(rb0 + r) * px + x;
        const float u = V[p][i];
        dst[gi] = u;
#pragma unroll
        for (int v = 1; v < S; ++v) dst[v * vol + gi] = Wv[(v - 1) * maxr * nx + i];
        res_two_sum(hi, lo, (double)u);
    }
    double part = hi + lo;
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((threadIdx.x & 31) == 0) red_hi[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        double b = 0.0;
        for (int w = 0; w < kResThreads / 32; ++w) b += red_hi[w];
        double* root = cl.map_shared_rank(cl_part, 0);
        root[rank] = b;
    }
    cl.sync();
    if (rank == 0 && threadIdx.x == 0) {
        double tot = 0.0;
        for (int k = 0; k < NC; ++k) tot += cl_part[k];
        if (!isfinite(tot)) atomicOr(err, ERRBIT_NAN);
        D->total = tot;
        D->total_pending = 0;
        D->t = t;
        D->n = n;
        D->cur = cur1;
    }
    cl.sync();  // no CTA leaves while its shared memory may still be read
}

// ---------------------------------------------------------------------------
// the same sheet with each thread's nodes in registers
// ---------------------------------------------------------------------------
//
// A thread owns R rows of one pair of columns for all steps: V (and for R <= 4
// the other variables) stay in its registers, and only V goes through shared
// memory, once per step for the neighbours.  The rows at a band's ends are also
// written into the neighbour CTA's halo row, so every read is local.  A step
// waits on an mbarrier: the arrivals of the CTA's own warps and of the
// neighbours' warps that wrote its halo rows.  V has two buffers and there are
// two barriers, used in turn: a neighbour may be one step ahead (its arrival
// for step s+1 can come before this CTA's last warp has arrived for step s),
// never two, since its step s+2 waits for this CTA's border warps of step s+1;
// by then they have read step s's halo values and passed its barrier.  The arithmetic of a node is the tiled
// step kernel's, operation for operation, so results are bitwise the same, in both state buffers: the state
// before the last step is written too (a program that owns the buffers may look at both).
// What bounded the kernel above: 82 instructions a node (16 CTAs of 32 warps,
// three quarters of the issue slots) and a cluster-wide barrier a step.

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void arrive_cluster(uint32_t addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ bool try_wait_cluster(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// A sum of floats kept in three (TwoSum of the value into hi, of its rounding
// error into lo, of that one's into lo2: about 70 bits).  The FP64 pipe takes
// an SM's warps one after the other, a warp's instruction some 16 cycles; seven
// of them a node and six a warp bounded short calls: 2 steps on a 200x200
// sheet 16.6 us a call, 10.4 so, on 400x400 41.2 and 19.8.
struct F3 {
    float hi, lo, lo2;
};
__device__ __forceinline__ float res_two_sum_f(float a, float b, float* err) {
    const float s = a + b, bb = s - a;
    *err = (a - (s - bb)) + (b - bb);
    return s;
}
__device__ __forceinline__ void f3_add(F3& a, F3 b) {
    float e, f, g;
    a.hi = res_two_sum_f(a.hi, b.hi, &e);
    const float t = res_two_sum_f(a.lo, b.lo, &f);
    a.lo = res_two_sum_f(t, e, &g);
    a.lo2 += b.lo2 + (f + g);
}
__device__ __forceinline__ void f3_add(F3& a, float b) { f3_add(a, F3{b, 0.0f, 0.0f}); }

// Warps of a CTA with np pairs of columns whose threads own row r of the band.
__host__ __device__ __forceinline__ int row_warp0(int np, int R, int r) { return (r / R * np) / 32; }
__host__ __device__ __forceinline__ int row_warps(int np, int R, int r) {
    return (r / R * np + np - 1) / 32 - row_warp0(np, R, r) + 1;
}

constexpr int kPairPad = 4;  // zero columns of a V row: two before x = 0, two after the last pair
constexpr int kPairMaxSmem = 220 * 1024;
__host__ __device__ constexpr bool pair_regs(int R) { return R <= 4; }

template <int MODEL, int NC, int R>
__global__ void __cluster_dims__(NC, 1, 1) __launch_bounds__(kResThreads, 1)
    k_resident_pairs(const TissueArgs* __restrict__ T, int n_steps, int* __restrict__ err, long long wait_limit) {
    constexpr int S = Model<MODEL>::S;
    constexpr bool VREG = pair_regs(R);
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    extern __shared__ float sm[];
    __shared__ float red[3][kResThreads / 32];
    __shared__ double cl_part[NC];
    __shared__ alignas(8) uint64_t bar[2];

    const int nx = T->nx, ny = T->ny, px = T->px;
    const long long vol = T->vol;
    const int np = (nx + 1) / 2, pitch = 2 * np + kPairPad;
    const int maxr = (ny + NC - 1) / NC;
    const int rb0 = (int)((long long)ny * rank / NC), rb1 = (int)((long long)ny * (rank + 1) / NC);
    const int nr = rb1 - rb0;
    float* V[2] = {sm, sm + (maxr + 2) * pitch};   // rows -1 .. nr of the band
    float* Wv = sm + 2 * (maxr + 2) * pitch;       // (!VREG) the other variables, (S-1) x maxr x 2 np
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
    const int q = tid / np, pc = tid - q * np;  // row group, pair
    const int r0 = q * R, rows = min(R, nr - r0), x = 2 * pc;  // (rows <= 0: a thread without nodes)
    const bool has_up = rank > 0, has_dn = rank + 1 < NC;
    const int nr_up = has_up ? rb0 - (int)((long long)ny * (rank - 1) / NC) : 0;
    // the neighbours' halo rows for this band's first and last row, and their barriers
    const uint32_t vbuf = smem_addr(sm), vstep = (uint32_t)((maxr + 2) * pitch * 4), bar_a = smem_addr(bar);
    const uint32_t col = (uint32_t)((2 + x) * 4);
    const uint32_t up_halo = has_up ? map_rank(vbuf, rank - 1) + (uint32_t)((nr_up + 1) * pitch * 4) + col : 0u;
    const uint32_t dn_halo = has_dn ? map_rank(vbuf, rank + 1) + col : 0u;
    const uint32_t up_bar = has_up ? map_rank(bar_a, rank - 1) : 0u, dn_bar = has_dn ? map_rank(bar_a, rank + 1) : 0u;
    const bool warp_up = has_up && warp < row_warps(np, R, 0);
    const bool warp_dn = has_dn && warp >= row_warp0(np, R, nr - 1) &&
                         warp < row_warp0(np, R, nr - 1) + row_warps(np, R, nr - 1);

    TissueDyn* D = T->dyn;
    const int cur0 = D->cur;
    double t = D->t;
    long long n = D->n;
    const float* src = T->state[cur0];
    for (int i = tid; i < 2 * (maxr + 2) * pitch; i += blockDim.x) sm[i] = 0.0f;
    if (tid == 0) {
        int count = nwarp;
        if (has_up) count += row_warps(np, R, nr_up - 1);  // the band above: its last row's warps
        if (has_dn) count += row_warps(np, R, 0);
        mbar_init(&bar[0], count);
        mbar_init(&bar[1], count);
        mbar_init_fence();
    }
    __syncthreads();
    float2 u[R], w[VREG ? R * (S > 1 ? S - 1 : 1) : 1];
    const bool x1_in = x + 1 < nx;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        if (k >= rows) continue;
        const long long gi = (long long)(rb0 + r0 + k) * px + x;
        u[k] = make_float2(src[gi], x1_in ? src[gi + 1] : 0.0f);
        *reinterpret_cast<float2*>(V[0] + (r0 + k + 1) * pitch + 2 + x) = u[k];
#pragma unroll
        for (int v = 1; v < S; ++v) {
            const float2 z = make_float2(src[v * vol + gi], x1_in ? src[v * vol + gi + 1] : 0.0f);
            if (VREG) w[k * (S - 1) + v - 1] = z;
            else *reinterpret_cast<float2*>(Wv + ((v - 1) * maxr + r0 + k) * 2 * np + x) = z;
        }
    }
    if (rows > 0 && r0 == 0 && has_up) {
        const long long gi = (long long)(rb0 - 1) * px + x;
        *reinterpret_cast<float2*>(V[0] + 2 + x) = make_float2(src[gi], x1_in ? src[gi + 1] : 0.0f);
    }
    if (rows > 0 && r0 + rows == nr && has_dn) {
        const long long gi = (long long)rb1 * px + x;
        *reinterpret_cast<float2*>(V[0] + (nr + 1) * pitch + 2 + x) = make_float2(src[gi], x1_in ? src[gi + 1] : 0.0f);
    }
    cl.sync();  // barriers initialised, buffers cleared and loaded everywhere

    const float c = T->c_iso, dt = T->dt, theta = T->theta;
    float mp[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) mp[k] = T->mp[k];
    // minus the number of x neighbours of the two nodes
    const float2 ncx = make_float2(-((x1_in ? 1.0f : 0.0f) + (x > 0 ? 1.0f : 0.0f)), -((x + 2 < nx ? 1.0f : 0.0f) + 1.0f));
    const bool stim_any = T->stim && T->stim_amp != 0.0f;
    const bool keep_t = stim_any || warp == 0;  // (FP64 additions are slow: only where the time is used)
    bool timed_out = false;
    int p = 0;
    for (int s = 0; s < n_steps; ++s) {
        if (s + 1 == n_steps) {
            // The buffer that does not become current gets the state of the step before the last one, as when
            // every step writes its buffer (the initial state, where it held that, was read before the first
            // cl.sync).  (`here` is 0: it keeps these addresses out of the registers of the other steps.)
            int here;
            asm volatile("mov.u32 %0, 0;" : "=r"(here));
            float* const other = T->state[cur0 ^ 1 ^ (n_steps & 1)] + here;
            const long long g0 = (long long)(rb0 + r0 + here) * px + x;
#pragma unroll
            for (int k = 0; k < R; ++k) {
                if (k >= rows) continue;
                float* o = other + g0 + (long long)k * px;
#pragma unroll
                for (int v = 0; v < S; ++v) {
                    const float2 z = v == 0 ? u[k]
                                     : VREG ? w[VREG && v > 0 ? k * (S - 1) + v - 1 : 0]
                                            : *reinterpret_cast<const float2*>(Wv + ((v - 1) * maxr + r0 + k) * 2 * np + x);
                    o[v * vol] = z.x;
                    if (x1_in) o[v * vol + 1] = z.y;
                }
            }
        }
        const uint32_t prev = bar_a + 8u * (uint32_t)((s - 1) & 1), phase = (uint32_t)((s - 1) >> 1) & 1u;
        if (s > 0 && !timed_out && !try_wait_cluster(prev, phase)) {
            const long long c0 = clock64();
            while (!try_wait_cluster(prev, phase)) {
                if (clock64() - c0 > wait_limit) {
                    timed_out = true;
                    break;
                }
            }
        }
        const bool stim_on = stim_any && t >= T->t_on && t < T->t_off;
        const float* Vo = V[p] + (r0 + 1) * pitch + 2 + x;
        float* Vn = V[p ^ 1] + (r0 + 1) * pitch + 2 + x;
        if (rows > 0) {
            float2 above = *reinterpret_cast<const float2*>(Vo - pitch);
#pragma unroll
            for (int k = 0; k < R; ++k) {
                if (k >= rows) continue;
                const int y = rb0 + r0 + k;
                const float2 u0 = u[k];
                const float2 below = k + 1 < R && k + 1 < rows ? u[k + 1 < R ? k + 1 : k]
                                                               : *reinterpret_cast<const float2*>(Vo + (k + 1) * pitch);
                const float2 sx = make_float2(__fadd_rn(u0.y, Vo[k * pitch - 1]), __fadd_rn(Vo[k * pitch + 2], u0.x));
                const float ncy = -2.0f + (y == 0 ? 1.0f : 0.0f) + (y + 1 == ny ? 1.0f : 0.0f);
                const float2 L = mul2(splat2(c), fma2(add2(ncx, splat2(ncy)), u0, add2(sx, add2(below, above))));
                float2 yv[S];
                yv[0] = u0;
#pragma unroll
                for (int v = 1; v < S; ++v)
                    yv[v] = VREG ? w[VREG ? k * (S - 1) + v - 1 : 0]
                                 : *reinterpret_cast<const float2*>(Wv + ((v - 1) * maxr + r0 + k) * 2 * np + x);
                float2 Is = splat2(0.0f);
                const long long gi = (long long)y * px + x;
                if (stim_on) {
                    if (T->stim[gi]) Is.x = T->stim_amp;
                    if (x1_in && T->stim[gi + 1]) Is.y = T->stim_amp;
                }
                Model<MODEL>::update2(mp, yv, add2(L, Is), dt);
                if (!x1_in) yv[0].y = 0.0f;  // (read as the absent neighbour's value)
                *reinterpret_cast<float2*>(Vn + k * pitch) = yv[0];
#pragma unroll
                for (int v = 1; v < S; ++v) {
                    if (VREG) w[VREG ? k * (S - 1) + v - 1 : 0] = yv[v];
                    else *reinterpret_cast<float2*>(Wv + ((v - 1) * maxr + r0 + k) * 2 * np + x) = yv[v];
                }
                if (k == 0 && r0 == 0 && has_up) st_cluster(up_halo + (p ? 0u : vstep), yv[0]);
                if (r0 + k + 1 == nr && has_dn) st_cluster(dn_halo + (p ? 0u : vstep), yv[0]);
                const bool c0 = u0.x < theta && theta <= yv[0].x, c1 = x1_in && u0.y < theta && theta <= yv[0].y;
                if (c0 || c1) {
                    if (c0 && T->act[gi] == BBX_ACT_NONE) T->act[gi] = (int32_t)(n + 1);
                    if (c1 && T->act[gi + 1] == BBX_ACT_NONE) T->act[gi + 1] = (int32_t)(n + 1);
                }
                above = u0;
                u[k] = yv[0];
            }
        }
        __syncwarp();
        if (lane == 0) {
            const uint32_t o = 8u * (uint32_t)(s & 1);
            mbar_arrive(&bar[s & 1]);
            if (warp_up) arrive_cluster(up_bar + o);
            if (warp_dn) arrive_cluster(dn_bar + o);
        }
        p ^= 1;
        if (keep_t) t = t + T->dt_d;
        n += 1;
    }
    if (timed_out) atomicOr(err, ERRBIT_TIMEOUT);

    // the new state into the buffer that becomes current, and the FP64 total of V
    const int cur1 = cur0 ^ (n_steps & 1);
    float* dst = T->state[cur1];
    F3 sum = {0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < R; ++k) {
        if (k >= rows) continue;
        const long long gi = (long long)(rb0 + r0 + k) * px + x;
        dst[gi] = u[k].x;
        f3_add(sum, u[k].x);
        if (x1_in) {
            dst[gi + 1] = u[k].y;
            f3_add(sum, u[k].y);
        }
#pragma unroll
        for (int v = 1; v < S; ++v) {
            const float2 z = VREG ? w[VREG ? k * (S - 1) + v - 1 : 0]
                                  : *reinterpret_cast<const float2*>(Wv + ((v - 1) * maxr + r0 + k) * 2 * np + x);
            dst[v * vol + gi] = z.x;
            if (x1_in) dst[v * vol + gi + 1] = z.y;
        }
    }
    for (int o = 16; o > 0; o >>= 1)
        f3_add(sum, F3{__shfl_xor_sync(0xffffffffu, sum.hi, o), __shfl_xor_sync(0xffffffffu, sum.lo, o),
                       __shfl_xor_sync(0xffffffffu, sum.lo2, o)});
    if (lane == 0) {
        red[0][warp] = sum.hi;
        red[1][warp] = sum.lo;
        red[2][warp] = sum.lo2;
    }
    __syncthreads();
    if (warp == 0) {
        double b = lane < nwarp ? (double)red[0][lane] + ((double)red[1][lane] + (double)red[2][lane]) : 0.0;
        for (int o = 16; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
        if (lane == 0) cl.map_shared_rank(cl_part, 0)[rank] = b;
    }
    cl.sync();
    if (rank == 0 && tid == 0) {
        double tot = 0.0;
        for (int k = 0; k < NC; ++k) tot += cl_part[k];
        if (!isfinite(tot)) atomicOr(err, ERRBIT_NAN);
        D->total = tot;
        D->total_pending = 0;
        D->t = t;
        D->n = n;
        D->cur = cur1;
    }
    cl.sync();  // no CTA leaves while its shared memory may still be written or read
}

// Rows a thread takes: the least that leaves at most 1024 threads (0: none fits).
inline int pair_rows(int nx, int ny, int NC) {
    const int np = (nx + 1) / 2, maxr = (ny + NC - 1) / NC;
    for (int R : {1, 2, 3, 4, 6, 8, 12})
        if ((long long)np * ((maxr + R - 1) / R) <= kResThreads) return R;
    return 0;
}

// From how many steps of a call this kernel is the faster route (the call's
// fixed cost, 16 SMs loading and storing the sheet, against one launch a step).
// Measured, us a call of n steps here and by tiles with the fastest height:
// 200x200 n = 2 11.7 / 11.9; 256x256 n = 2 12.4 / 11.9, n = 3 14.5 / 17.8;
// 340x340 n = 2 16.6 / 13.2, n = 3 18.6 / 19.8; one variable 512x512 n = 4
// 25.8 / 25.2, n = 6 32 / 38.  With more than four rows a thread the second
// variable is in shared memory, and registers spill, more with more rows:
// 362x362 n = 3 22.6 / 20.2, n = 4 24.8 / 27.1; 400x400 n = 4 26.8 / 27.2, n = 6
// 32 / 41; 450x450 n = 10 67 / 70; 512x512 n = 10 72 / 65, n = 20 124 / 128;
// twelve rows: one variable 560x560 n = 10 68 / 67, n = 16 99 / 107, two
// variables 520x520 n = 20 159 / 140.
inline int pairs_from(int S, int R, int nx, int ny) {
    const int n = nx * ny;  // (at most 16 x 1024 x 12 x 2)
    if (R > 8) return S == 1 ? 11 : INT_MAX;
    return 2 + n / (S == 1 || R <= 4 ? 65536 : (R <= 6 ? 50000 : 19000));
}

template <int MODEL, int NC, int R>
cudaError_t pairs_try(const TissueArgs* d_t, int nx, int ny, int n_steps, int* d_err, cudaStream_t s, bool check_only,
                      bool* ok, int* from) {
    const int np = (nx + 1) / 2, maxr = (ny + NC - 1) / NC, pitch = 2 * np + kPairPad;
    const size_t smem = sizeof(float) * (2 * (size_t)(maxr + 2) * pitch +
                                         (pair_regs(R) ? 0 : (size_t)(Model<MODEL>::S - 1) * maxr * 2 * np));
    *ok = false;
    if (smem > (size_t)kPairMaxSmem || ny < NC) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(NC);
    cfg.blockDim = dim3((unsigned)((np * ((maxr + R - 1) / R) + 31) / 32 * 32));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    if (check_only) {
        if (cudaFuncSetAttribute(k_resident_pairs<MODEL, NC, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kPairMaxSmem) != cudaSuccess ||
            cudaFuncSetAttribute(k_resident_pairs<MODEL, NC, R>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                cudaSuccess) {
            cudaGetLastError();  // not offered here
            return cudaSuccess;
        }
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, k_resident_pairs<MODEL, NC, R>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            return cudaSuccess;
        }
        *ok = clusters >= 1;
        *from = pairs_from(Model<MODEL>::S, R, nx, ny);
        return cudaSuccess;
    }
    *ok = true;
    k_resident_pairs<MODEL, NC, R><<<cfg.gridDim, cfg.blockDim, smem, s>>>(d_t, n_steps, d_err, kWaitLimit);
    return cudaGetLastError();
}

template <int MODEL>
cudaError_t pairs_launch(const TissueArgs* d_t, int nx, int ny, int n_steps, int* d_err, cudaStream_t s,
                         bool check_only, bool* ok, int* from) {
    constexpr int NC = kResCtasLarge;
    *ok = false;
    switch (pair_rows(nx, ny, NC)) {
        case 1: return pairs_try<MODEL, NC, 1>(d_t, nx, ny, n_steps, d_err, s, check_only, ok, from);
        case 2: return pairs_try<MODEL, NC, 2>(d_t, nx, ny, n_steps, d_err, s, check_only, ok, from);
        case 3: return pairs_try<MODEL, NC, 3>(d_t, nx, ny, n_steps, d_err, s, check_only, ok, from);
        case 4: return pairs_try<MODEL, NC, 4>(d_t, nx, ny, n_steps, d_err, s, check_only, ok, from);
        case 6: return pairs_try<MODEL, NC, 6>(d_t, nx, ny, n_steps, d_err, s, check_only, ok, from);
        case 8: return pairs_try<MODEL, NC, 8>(d_t, nx, ny, n_steps, d_err, s, check_only, ok, from);
        case 12: return pairs_try<MODEL, NC, 12>(d_t, nx, ny, n_steps, d_err, s, check_only, ok, from);
    }
    return cudaSuccess;
}

template <int MODEL, int NC>
int resident_smem(int nx, int ny) {
    const int maxr = (ny + NC - 1) / NC;
    return (int)(sizeof(float) * (size_t)(Model<MODEL>::S + 1) * maxr * nx);
}

// One cluster of NC CTAs, if the grid fits and the GPU can hold such a
// cluster (*ok); returns launch errors.
template <int MODEL, int NC>
cudaError_t resident_try(const TissueArgs* d_t, int nx, int ny, int n_steps, int* d_err, cudaStream_t s,
                         bool check_only, bool* ok) {
    const int smem = resident_smem<MODEL, NC>(nx, ny);
    *ok = false;
    if (smem > kResMaxSmem || ny < NC) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_resident_sheet<MODEL, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    if (NC > kResCtasPortable &&
        cudaFuncSetAttribute(k_resident_sheet<MODEL, NC>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess) {
        cudaGetLastError();  // not offered here: the caller tries the portable size
        return cudaSuccess;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(NC);
    cfg.blockDim = dim3(kResThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, k_resident_sheet<MODEL, NC>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return cudaSuccess;
    }
    if (clusters < 1) return cudaSuccess;
    *ok = true;
    if (check_only) return cudaSuccess;
    k_resident_sheet<MODEL, NC><<<NC, kResThreads, smem, s>>>(d_t, n_steps, d_err);
    return cudaGetLastError();
}

template <int MODEL>
cudaError_t resident_launch(const TissueArgs* d_t, int nx, int ny, int n_steps, int* d_err, cudaStream_t s,
                            bool check_only, bool* ok) {
    cudaError_t e = resident_try<MODEL, kResCtasLarge>(d_t, nx, ny, n_steps, d_err, s, check_only, ok);
    if (e != cudaSuccess || *ok) return e;
    return resident_try<MODEL, kResCtasPortable>(d_t, nx, ny, n_steps, d_err, s, check_only, ok);
}

}  // namespace

// n_steps on a small isotropic, unmasked sheet with the register-resident
// kernel, bitwise as the tiled kernel steps it.  check_only: report in *ok
// whether the grid's shape runs there (and make the kernel ready for it; a
// launch needs an earlier check of the same shape) and in *from from how many
// steps of a call it is the faster route.
cudaError_t resident_pair_steps(int model, const TissueArgs* d_t, int nx, int ny, int n_steps, int* d_err,
                                cudaStream_t s, bool check_only, bool* ok, int* from) {
    switch (model) {
        case BBX_FHN: return pairs_launch<BBX_FHN>(d_t, nx, ny, n_steps, d_err, s, check_only, ok, from);
        case BBX_BARKLEY: return pairs_launch<BBX_BARKLEY>(d_t, nx, ny, n_steps, d_err, s, check_only, ok, from);
        case BBX_ZFK: return pairs_launch<BBX_ZFK>(d_t, nx, ny, n_steps, d_err, s, check_only, ok, from);
        case BBX_DIFFUSION: return pairs_launch<BBX_DIFFUSION>(d_t, nx, ny, n_steps, d_err, s, check_only, ok, from);
    }
    *ok = false;
    return cudaSuccess;
}

// Run n_steps on a small isotropic, unmasked sheet with the resident kernel.
// check_only: only report (in *ok) whether this grid shape can run resident.
cudaError_t resident_sheet_steps(int model, const TissueArgs* d_t, int nx, int ny, int n_steps, int* d_err,
                                 cudaStream_t s, bool check_only, bool* ok) {
    switch (model) {
        case BBX_FHN: return resident_launch<BBX_FHN>(d_t, nx, ny, n_steps, d_err, s, check_only, ok);
        case BBX_BARKLEY: return resident_launch<BBX_BARKLEY>(d_t, nx, ny, n_steps, d_err, s, check_only, ok);
        case BBX_ZFK: return resident_launch<BBX_ZFK>(d_t, nx, ny, n_steps, d_err, s, check_only, ok);
        case BBX_DIFFUSION: return resident_launch<BBX_DIFFUSION>(d_t, nx, ny, n_steps, d_err, s, check_only, ok);
    }
    *ok = false;
    return cudaSuccess;
}

}  // namespace bbx
