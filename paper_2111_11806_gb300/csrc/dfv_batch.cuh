// dfv_batch.cuh -- many independent 2-D instances (own grid size, body and
// time step) advanced together: every kernel is a persistent launch over a
// work list of (instance, tile) items, so one launch per phase serves the whole
// batch.  The per-tile work is the single-grid stage_tile / seeding code.
#pragma once

#include <algorithm>

#include "dfv_kernels.cuh"

namespace dfv {

struct BatchInst {
    GridP g;            // the instance's grid and materials (pitch: its own)
    long long off;      // element offset of its planes in the state arrays
    int tiles_x, tiles_y, ntiles, rest;   // rest: its body does not move
    Ctl *ctl;           // its control block (dt, t, smax, error word)
};

struct BatchArgs {
    const void *in;          // stage input, read with halo
    const void *un;          // U^n
    void *out;               // stage output
    const BatchInst *inst;
    const int2 *items;       // (instance, tile) in the order of the schedule
    long long nitems;
    int final_mode;          // mode of the finalize phase (after stage 3 or a CFL reduction)
    unsigned int *queue;     // dynamic schedule: next item counter (nullptr: static round-robin)
};

// Next work item of this CTA: static round-robin or a shared counter.
__device__ __forceinline__ long long next_item(const BatchArgs &b, long long cur, long long *s_item)
{
    if (!b.queue) return cur < 0 ? (long long)blockIdx.x : cur + gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) *s_item = (long long)atomicAdd(b.queue, 1u);
    __syncthreads();
    return *s_item;
}

// Copy the instance record into shared memory (GridP is read all through the
// tile code; shared memory keeps those reads off the global path).
__device__ __forceinline__ void load_inst(const BatchInst *src, BatchInst *dst)
{
    const int *s = reinterpret_cast<const int *>(src);
    int *d = reinterpret_cast<int *>(dst);
    constexpr int NW = (int)(sizeof(BatchInst) / sizeof(int));
    for (int k = threadIdx.x; k < NW; k += blockDim.x) d[k] = s[k];
}

// Register bound: five CTAs per SM for the FP32 single-material form (40
// registers, a few dozen bytes of spills; 1 % faster than four on the
// 256-ellipse batch), two otherwise.
template <class R, int NMAT, int STAGE>
__global__ void __launch_bounds__(Tile<2, 0>::THREADS, (sizeof(R) == 4 && NMAT == 1) ? 5 : 2)
    k_batch_stage(BatchArgs b)
{
    pdl_enter();
    __shared__ BatchInst s_inst;
    __shared__ long long s_item;
    __shared__ int s_cur;
    if (threadIdx.x == 0) s_cur = -1;
    for (long long it = next_item(b, -1, &s_item); it < b.nitems; it = next_item(b, it, &s_item)) {
        const int2 w = b.items[it];
        __syncthreads();
        if (s_cur != w.x) {
            load_inst(&b.inst[w.x], &s_inst);
            __syncthreads();
            if (threadIdx.x == 0) s_cur = w.x;
        }
        __syncthreads();
        const BatchInst &I = s_inst;
        StageArgs a;
        a.in = reinterpret_cast<const R *>(b.in) + I.off;
        a.un = reinterpret_cast<const R *>(b.un) + I.off;
        a.out = reinterpret_cast<R *>(b.out) + I.off;
        a.ctl = I.ctl;
        a.partials = nullptr;   // no force is wanted
        a.want_force = 0;
        a.rest = I.rest;
        a.early = 0;
        a.next = 0;
        a.late = 0;
        stage_tile<R, 2, NMAT, 0, STAGE, 0>(I.g, a, w.y % I.tiles_x, w.y / I.tiles_x, 0, w.y);
    }
}

// Rigid seeding of every instance: SEED_CTAS CTAs of 256 threads per
// instance stride over the cells of its rigid box (the whole grid until its
// first stage 3); the instance record is read through the cache.
// MODE 0: in place; 1: seeded states into the scratch planes b.out; 2: the
// scratch into U (the fixed probe reads the step-start state only).
constexpr int SEED_CTAS = 32;

template <class R, int NMAT, int MODE, int OPT>
__global__ void __launch_bounds__(256) k_batch_seed(BatchArgs b)
{
    pdl_enter();
    const BatchInst &I = b.inst[blockIdx.x / SEED_CTAS];
    R *U = reinterpret_cast<R *>(const_cast<void *>(b.in)) + I.off;
    R *S = reinterpret_cast<R *>(b.out) + I.off;
    seed_box_cells<R, 2, NMAT, false, OPT, MODE>(U, S, I.ctl, I.g,
                                                 (int)(blockIdx.x % SEED_CTAS), SEED_CTAS, false);
}

// CFL wave speed of every instance's stored state: blockIdx.y the instance,
// blockIdx.x its CFL_CELLS cells, the block's maximum folded into the
// instance's running maximum as stage 3 does; the finalize launch that follows
// sets its dt.  (One CTA for each 256 cells with a ticket for the last of an
// instance, which reduced their partials, took 826 us on 26 million cells;
// read once they are 525 MB.)
constexpr int CFL_CELLS = 4096;

template <class R, int NMAT>
__global__ void __launch_bounds__(256) k_batch_cfl(const BatchInst *inst, const void *Uv)
{
    using L = Lay<2, NMAT, 0>;
    __shared__ R sred[32];
    const BatchInst &I = inst[blockIdx.y];
    const long long n = I.g.ncell, P = I.g.pitch, c0 = (long long)blockIdx.x * CFL_CELLS;
    if (c0 >= n) return;
    const R *U = reinterpret_cast<const R *>(Uv) + I.off;
    const long long c1 = min(n, c0 + CFL_CELLS);
    R top = R(0);
    bool bad = false;
    for (long long c = c0 + threadIdx.x; c < c1; c += 256) {
        R q[L::NVAR], cs;
#pragma unroll
        for (int v = 0; v < L::NVAR; v++) q[v] = U[v * P + c];
        const R s = cell_speed<R, 2, NMAT, 0>(I.g, q, cs);
        bad = bad || !(s == s);
        top = nan_max(top, s);
    }
    top = block_max<256, R>(top, sred);
    const int nan = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        double m = (double)top;
        if (nan || !(m >= 0.0)) m = __longlong_as_double(0x7ff0000000000000LL);   // NaN -> +inf: dt = 0
        atomicMax(&I.ctl->smax_acc, (unsigned long long)__double_as_longlong(m));
    }
}

template <class R, int NMAT>
cudaError_t batch_cfl(int count, long long max_cells, const BatchInst *inst, const void *U, cudaStream_t st)
{
    const unsigned bx = (unsigned)((max_cells + CFL_CELLS - 1) / CFL_CELLS);
    for (int i0 = 0; i0 < count; i0 += 65535)
        k_batch_cfl<R, NMAT><<<dim3(bx, (unsigned)std::min(count - i0, 65535)), 256, 0, st>>>(inst + i0, U);
    return cudaGetLastError();
}

// Finalize of every instance after stage 3, one block per instance: its CFL
// maximum (folded by its stage-3 tiles), time, step count and next dt.
template <int THREADS>
__global__ void __launch_bounds__(THREADS) k_batch_finalize(BatchArgs b)
{
    pdl_enter();
    __shared__ double sred[4 * 32];
    const BatchInst &I = b.inst[blockIdx.x];
    finalize_block<THREADS>(I.ctl, nullptr, 0, 0, b.final_mode, 2, I.g.dx[0], I.g.dx[1], I.g.dx[2], sred);
    // the stages of this step are complete: reset the dynamic-schedule counters
    if (blockIdx.x == 0 && threadIdx.x == 0 && b.queue)
        for (int k = 1; k <= 3; k++) b.queue[k] = 0u;
}

static __global__ void k_batch_init_ctl(Ctl *ctl, int count, const double *v_body /* 3 per instance */)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        Ctl *c = ctl + i;
        memset(c, 0, sizeof(Ctl));
        ctl_box_reset(c);
        for (int d = 0; d < 3; d++) c->v[d] = v_body[3 * i + d];
        ctl_sync_v(c);
    }
}

static __global__ void k_batch_set_run(Ctl *ctl, int count, double cfl, double t_end)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        ctl[i].cfl = cfl;
        ctl[i].t_end = t_end;
    }
}

// Field conversion of every instance in one launch: blockIdx.y the instance,
// blockIdx.x its FIELD_CELLS cells (blocks past its end return).  ptr: the
// caller's FP64 planes of each instance, in memory the device can address,
// passed with the launch (nothing of the host is read later).  One
// launch for FIELD_INST instances instead of one for each (256 of them left the
// chip idle between and at the end of each).  MODE 0: primitives in (and the rigid box
// unknown), 1: conserved out, 2: primitives out.
constexpr int FIELD_CELLS = 2048, FIELD_INST = 256;

struct FieldPtrs {
    double *p[FIELD_INST];
};

template <class R, int NMAT, int MODE>
__global__ void __launch_bounds__(256) k_batch_fields(const BatchInst *inst, const __grid_constant__ FieldPtrs ptr, void *Uv)
{
    using L = Lay<2, NMAT, 0>;
    const BatchInst &I = inst[blockIdx.y];
    const long long n = I.g.ncell, P = I.g.pitch, c0 = (long long)blockIdx.x * FIELD_CELLS;
    if (MODE == 0 && blockIdx.x == 0 && threadIdx.x == 0) I.ctl->rbox_valid = 0;
    if (c0 >= n) return;
    R *U = reinterpret_cast<R *>(Uv) + I.off;
    double *f = ptr.p[blockIdx.y];
    const long long c1 = min(n, c0 + FIELD_CELLS);
    for (long long c = c0 + threadIdx.x; c < c1; c += 256) {
        double a[L::NVAR], b[L::NVAR];
        if constexpr (MODE == 0) {
#pragma unroll
            for (int v = 0; v < L::NVAR; v++) a[v] = f[v * n + c];
            prim_to_cons<double, 2, NMAT, 0>(I.g, a, b);
#pragma unroll
            for (int v = 0; v < L::NVAR; v++) U[v * P + c] = m_store<R>(b[v]);
        } else {
#pragma unroll
            for (int v = 0; v < L::NVAR; v++) a[v] = m_widen(U[v * P + c]);
            if constexpr (MODE == 2) cons_to_prim_ct<double, 2, NMAT, 0>(I.g, a, b);
#pragma unroll
            for (int v = 0; v < L::NVAR; v++) f[v * n + c] = MODE == 2 ? b[v] : a[v];
        }
    }
}

// Launch table of the batch kernels of one precision.
template <class R, int NMAT>
struct BK {
    static constexpr int threads = Tile<2, 0>::THREADS;
    static constexpr size_t smem = StageSmem<R, 2, NMAT, 0, 0>::bytes;
    static cudaError_t prepare()
    {
        cudaError_t e = cudaFuncSetAttribute(k_batch_stage<R, NMAT, 1>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_batch_stage<R, NMAT, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_batch_stage<R, NMAT, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem);
        return e;
    }
    static int max_ctas_per_sm()
    {
        int a = 0, b = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_batch_stage<R, NMAT, 2>, threads, smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_batch_stage<R, NMAT, 3>, threads, smem);
        return std::max(1, std::min(a, b));
    }
    template <int MODE>
    static void seed(int opt, int grid, const BatchArgs &a, cudaStream_t st)
    {
        switch (opt) {
        case 0: launch_pdl(k_batch_seed<R, NMAT, MODE, 0>, dim3(grid * SEED_CTAS), dim3(256), 0, st, a); break;
        case 1: launch_pdl(k_batch_seed<R, NMAT, MODE, 1>, dim3(grid * SEED_CTAS), dim3(256), 0, st, a); break;
        case 2: launch_pdl(k_batch_seed<R, NMAT, MODE, 2>, dim3(grid * SEED_CTAS), dim3(256), 0, st, a); break;
        default: launch_pdl(k_batch_seed<R, NMAT, MODE, 3>, dim3(grid * SEED_CTAS), dim3(256), 0, st, a); break;
        }
    }
    // phase: 0 seed in place, 1..3 stages, 5 / 6 seed to scratch / apply,
    // 7 finalize after stage 3;
    // opt: the seeding option set (seed_opt)
    static cudaError_t launch(int phase, int grid, const BatchArgs &a, int opt, cudaStream_t st)
    {
        switch (phase) {
        case 0: seed<0>(opt, grid, a, st); break;
        case 5: seed<1>(opt, grid, a, st); break;
        case 6: launch_pdl(k_batch_seed<R, NMAT, 2, 0>, dim3(grid * SEED_CTAS), dim3(256), 0, st, a); break;
        case 7: launch_pdl(k_batch_finalize<32>, dim3(grid), dim3(32), 0, st, a); break;
        case 1: launch_pdl(k_batch_stage<R, NMAT, 1>, dim3(grid), dim3(threads), smem, st, a); break;
        case 2: launch_pdl(k_batch_stage<R, NMAT, 2>, dim3(grid), dim3(threads), smem, st, a); break;
        default: launch_pdl(k_batch_stage<R, NMAT, 3>, dim3(grid), dim3(threads), smem, st, a); break;
        }
        return cudaGetLastError();
    }
};

// Field conversion of every instance (mode as k_batch_fields); max_cells: of
// the largest instance.
template <class R, int NMAT>
cudaError_t batch_fields(int mode, int count, long long max_cells, const BatchInst *inst, double *const *ptr, void *U,
                         cudaStream_t st)
{
    const unsigned bx = (unsigned)((max_cells + FIELD_CELLS - 1) / FIELD_CELLS);
    for (int i0 = 0; i0 < count; i0 += FIELD_INST) {
        const int n = std::min(count - i0, FIELD_INST);
        FieldPtrs p;
        for (int i = 0; i < FIELD_INST; i++) p.p[i] = i < n ? ptr[i0 + i] : nullptr;
        const dim3 g(bx, (unsigned)n);
        if (mode == 0) k_batch_fields<R, NMAT, 0><<<g, 256, 0, st>>>(inst + i0, p, U);
        else if (mode == 1) k_batch_fields<R, NMAT, 1><<<g, 256, 0, st>>>(inst + i0, p, U);
        else k_batch_fields<R, NMAT, 2><<<g, 256, 0, st>>>(inst + i0, p, U);
    }
    return cudaGetLastError();
}

struct Kern {
    cudaError_t (*prepare)();
    int (*max_ctas_per_sm)();
    cudaError_t (*launch)(int, int, const BatchArgs &, int, cudaStream_t);
    cudaError_t (*fields)(int, int, long long, const BatchInst *, double *const *, void *, cudaStream_t);
    cudaError_t (*cfl)(int, long long, const BatchInst *, const void *, cudaStream_t);
};

template <class R>
Kern batch_kernels(int nmat)
{
    return nmat == 1   ? Kern{BK<R, 1>::prepare, BK<R, 1>::max_ctas_per_sm, BK<R, 1>::launch, batch_fields<R, 1>, batch_cfl<R, 1>}
           : nmat == 2 ? Kern{BK<R, 2>::prepare, BK<R, 2>::max_ctas_per_sm, BK<R, 2>::launch, batch_fields<R, 2>, batch_cfl<R, 2>}
                       : Kern{BK<R, 3>::prepare, BK<R, 3>::max_ctas_per_sm, BK<R, 3>::launch, batch_fields<R, 3>, batch_cfl<R, 3>};
}

// One translation unit per precision (the FP32 one is built with the fast
// single-precision divide, like the single-grid FP32 kernels).
Kern batch_kernels_f32(int nmat);
Kern batch_kernels_f64(int nmat);


}  // namespace dfv
