// dfv_gas3.cuh -- the SSP-RK3 stage (Sec. 3.1) of 3-D single-gas grids in
// FP32 (one ideal or stiffened gas, static body, transmissive or reflective
// sides): the form of the sphere workload.
//
// A CTA owns a 32 x 8 column of cells and marches through a chunk of planes
// in z.  A ring of three planes of primitives (z, z+1, z+2, each with its x
// and y halo of 2) sits in shared memory; per plane z:
//   1. plane z+2 is converted from the conserved values that arrived in the
//      shared fetch slot during the previous plane (one TMA tensor copy of
//      the plane's box, or per-thread asynchronous copies when rows are not
//      16-byte multiples); then plane z+3 is fetched into the slot, and the
//      cell's own values of plane z+1 are prefetched into L1;
//   2. slopes: every cell of plane z its van Leer slopes in x and y (face
//      values to shared memory, one warp the halo), every cell of plane z+1
//      its slope in z;
//   3. faces: every thread the HLLC fluxes of its cell's left x face, bottom
//      y face and top z face; the bottom z face and the top z-face value of
//      plane z were carried in shared memory from the previous plane;
//   4. update of plane z: divergence, rigid
//      mask, RK combination; in stage 3 the CFL maximum and the rigid box.
// Each primitive is converted once per chunk and each slope computed once;
// the arithmetic per face is that of the 2-D gas kernel (dfv_gas.cuh) with
// two tangential velocities.  Halo of 2: without a moving body the upwind r
// flux vanishes and r is not reconstructed (MUSCL only).
#pragma once

#include <cuda.h>

#include "dfv_gas.cuh"

namespace dfv {

// ------------------------------------------------------------ TMA, mbarrier

__device__ __forceinline__ unsigned smem_u32(const void *p)
{
    return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// Bounded wait for the phase of parity `parity` to complete; false when the
// iteration limit ran out (the caller reports it and stops).
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity)
{
    const unsigned a = smem_u32(bar);
    for (int it = 0; it < (1 << 22); it++) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (ok) return true;
    }
    return false;
}

struct Gas3T {
    static constexpr int TX = 32, TY = 8, H = 2;
    static constexpr int PX = TX + 2 * H, PY = TY + 2 * H;   // a plane with its x, y halo
    static constexpr int CELLS = TX * TY;
    static constexpr int THREADS = CELLS + 32;
    static constexpr int NCONV = TY * PX + 2 * H * TX;       // loaded cells of a plane (corners not)
    static constexpr int K = (NCONV + THREADS - 1) / THREADS; // loaded cells per thread
    static constexpr int RING = 3;
    static constexpr int NP = 6;                             // rho, rho u, rho v, rho w, rho E, r
    static constexpr int FXS = TX + 1, FYS = TY + 1;
    // planes per CTA of large grids (256^3 sphere, us a step at 16 / 24 / 32 /
    // 48 / 64 planes: 1602 / 1590 / 1621 / 1589 / 1611); gas3_planes otherwise
    static constexpr int ZCHUNK = 24;
    static constexpr int CTAS = 3;   // resident per SM
    // the TMA box of a plane: x from ox-4 (a 16-byte boundary) to ox+35, y
    // from oy-2 to oy+9, the five conserved planes rho .. rho E
    static constexpr int BX = TX + 8, BY = PY, BV = 5;
    static constexpr int BOXF = BX * BY * BV;
    static constexpr int XFER = K * 5 * THREADS > BOXF ? K * 5 * THREADS : BOXF;   // floats of the fetch slot
};
static_assert((Gas3T::BOXF * 4) % 128 == 0, "the TMA box keeps 128-byte multiples");

// primitives (rho, u, v, w) and p of one cell or face value
struct __align__(128) Gas3Smem {
    // the fetch slot of the next plane, first (a tensor copy's destination
    // is 128-byte aligned): its TMA box [v][y][x], or per thread the conserved
    // values of its cells (asynchronous copies read back by the same thread)
    float xfer[Gas3T::XFER];
    unsigned long long mbar;                             // completion of the slot's tensor copy
    float4 pa[Gas3T::RING][Gas3T::PY][Gas3T::PX + 1];   // odd row length: column reads conflict-free
    float pp[Gas3T::RING][Gas3T::PY][Gas3T::PX + 1];
    float4 fvxa[Gas3T::TY][Gas3T::FXS];                  // right-face values, column -1 .. TX-1
    float fvxp[Gas3T::TY][Gas3T::FXS];
    float4 fvya[Gas3T::FYS][Gas3T::TX];                  // top-face values, row -1 .. TY-1
    float fvyp[Gas3T::FYS][Gas3T::TX];
    float4 hrxa[Gas3T::TY];                              // left-face values of column TX
    float hrxp[Gas3T::TY];
    float4 hrya[Gas3T::TX];                              // bottom-face values of row TY
    float hryp[Gas3T::TX];
    float4 fxa[Gas3T::TY][Gas3T::FXS];                   // x-face fluxes (rho, rho u, rho v, rho w)
    float fxe[Gas3T::TY][Gas3T::FXS];                    //  and rho E
    float4 fya[Gas3T::FYS][Gas3T::TX];
    float fye[Gas3T::FYS][Gas3T::TX];
    // per column: the carried top z-face value and bottom z-face flux
    float4 zqa[Gas3T::CELLS], zfa[Gas3T::CELLS];
    float zqp[Gas3T::CELLS], zfe[Gas3T::CELLS];
    double red[32];
};

struct Gas3Args {
    const float *in;    // stage input
    const float *un;    // U^n
    float *out;         // stage output
    Ctl *ctl;
    int n0, n1, n2;
    long long pitch;
    float idx, idy, idz;
    int wall[3][2];     // reflective sides
    int zc;             // planes per CTA
    float Gam, invGam, pref0;
};

// HLLC flux of the gas with normal velocity un and tangential ut1, ut2
// (Sec. 3.1: Toro's HLLC, Davis wave speeds); F = (rho, normal momentum,
// tangential momenta 1 and 2, energy).
__device__ __forceinline__ void gas_hllc3(const Gas3Args &a, const float L[5], const float R[5], float F[5])
{
    // L, R: (rho, un, ut1, ut2, p)
    float SL, SR, Ss;
    float2 d2, m2;
    gas_waves(a, L[0], L[1], L[4], R[0], R[1], R[4], SL, SR, Ss, d2, m2);
    const int region = SL >= 0.f ? 0 : (Ss >= 0.f ? 1 : (SR > 0.f ? 2 : 3));
    const bool left = region <= 1;
    // the upwind side's state, element by element (a pointer choice would
    // put both arrays in local memory)
    const float r = left ? L[0] : R[0], un = left ? L[1] : R[1], u1 = left ? L[2] : R[2];
    const float u2 = left ? L[3] : R[3], p = left ? L[4] : R[4];
    const float S = left ? SL : SR, d = left ? d2.x : d2.y, m = left ? m2.x : m2.y;
    const float E = fmaf(0.5f * r, fmaf(u2, u2, fmaf(u1, u1, un * un)), (p - a.pref0) * a.invGam);
    float us = un, ps = p, cS = un, FE = (E + p) * un;
    if (region == 1 || region == 2) {
        // the star state's own flux (gas_hllc)
        const float2 dd = gas_sub2(gas_f2(S, Ss), gas_f2(Ss, un));   // (S_K - S*, S* - u_K)
        const float iD = gas_rcp(dd.x);
        us = Ss;
        cS = __fmul_rn(__fmul_rn(d, iD), Ss);
        ps = fmaf(m, dd.y, p);
        FE = (fmaf(d, E, fmaf(ps, Ss, -__fmul_rn(p, un))) * iD + ps) * Ss;
    }
    const float M = __fmul_rn(r, cS);
    F[0] = M;
    F[1] = fmaf(M, us, ps);
    F[2] = M * u1;
    F[3] = M * u2;
    F[4] = FE;
}

// A plane (with its x, y halo) in flight: its conserved values arrive in the
// fetch slot, by one tensor copy (TMA) or by every thread's asynchronous
// copies; the mirror flags of a thread's cells (3 bits each, cp.async path)
// or of the plane (TMA path) and the copy's mbarrier phase stay in registers.
struct Gas3Plane {
    unsigned flip;
    int gz;           // plane read
    unsigned phase;   // tensor copies issued so far (TMA path)
    // of each cell that the thread converts: its place in the fetch slot's box
    // (low half) and in a ring plane (high half), the same for every plane, and
    // its x and y mirror flags (2 bits a cell; TMA path)
    unsigned at[Gas3T::K];
    unsigned mirror;
};

__device__ __forceinline__ void gas3_cp4(float *dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// One 4-D tensor copy (x, y, plane z, variable) of a box into shared memory.
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, int x, int y, int z, int v,
                                            unsigned long long *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z), "r"(v), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ int gas3_map(int i, int n, int wlo, int whi, bool *flip)
{
    if (i < 0) {
        if (wlo) {
            *flip = true;
            const int m = -1 - i;
            return m > n - 1 ? n - 1 : m;
        }
        return 0;
    }
    if (i > n - 1) {
        if (whi) {
            *flip = true;
            const int m = 2 * n - 1 - i;
            return m < 0 ? 0 : m;
        }
        return n - 1;
    }
    return i;
}

// loaded cell q of a plane -> (lx, ly) relative to the column's corner
__device__ __forceinline__ void gas3_cell(int q, int &lx, int &ly)
{
    using T = Gas3T;
    if (q < T::TY * T::PX) {
        ly = q / T::PX;
        lx = q - ly * T::PX - T::H;
    } else {
        const int r = q - T::TY * T::PX;
        const int row = r / T::TX;
        lx = r - row * T::TX;
        ly = row < 2 ? row - 2 : T::TY + (row - 2);
    }
}

// Start the fetch of plane z into the slot.  TMA: thread 0 issues one tensor
// copy of the box (the slot's previous contents have been read: the caller
// fetches after a barrier); otherwise every thread copies its own cells.
template <bool TMA>
__device__ __forceinline__ void gas3_fetch(const Gas3Args &a, const CUtensorMap *map, Gas3Smem &S, Gas3Plane &f,
                                           int ox, int oy, int z, bool interior)
{
    using T = Gas3T;
    bool fz = false;
    const int gz = gas3_map(z, a.n2, a.wall[2][0], a.wall[2][1], &fz);
    if constexpr (TMA) {
        f.flip = fz ? 4u : 0u;
        f.gz = gz;
        if (threadIdx.x == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect_tx(&S.mbar, 4u * T::BOXF);
            tma_load_4d(S.xfer, map, ox - 4, oy - T::H, gz, 0, &S.mbar);
        }
        return;
    }
    f.flip = 0u;
#pragma unroll
    for (int k = 0; k < T::K; k++) {
        const int q = threadIdx.x + k * T::THREADS;
        if (q >= T::NCONV) continue;
        int lx, ly;
        gas3_cell(q, lx, ly);
        bool fx = false, fy = false;
        int gx = ox + lx, gy = oy + ly;
        if (!interior) {
            gx = gas3_map(gx, a.n0, a.wall[0][0], a.wall[0][1], &fx);
            gy = gas3_map(gy, a.n1, a.wall[1][0], a.wall[1][1], &fy);
        }
        f.flip |= ((fx ? 1u : 0u) | (fy ? 2u : 0u) | (fz ? 4u : 0u)) << (3 * k);
        const long long c = gx + (long long)a.n0 * (gy + (long long)a.n1 * gz);
#pragma unroll
        for (int v = 0; v < 5; v++) gas3_cp4(&S.xfer[(k * 5 + v) * T::THREADS + threadIdx.x], a.in + c + v * a.pitch);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ void gas3_prim(const Gas3Args &a, const float q[5], unsigned flip, float w[5])
{
    const float ir = __fdividef(1.f, q[0]);
    const float u = q[1] * ir, v = q[2] * ir, ww = q[3] * ir;
    const float ke = 0.5f * q[0] * u * u + 0.5f * q[0] * v * v + 0.5f * q[0] * ww * ww;
    w[0] = q[0];
    w[1] = (flip & 1u) ? -u : u;
    w[2] = (flip & 2u) ? -v : v;
    w[3] = (flip & 4u) ? -ww : ww;
    w[4] = a.pref0 + a.Gam * (q[4] - ke);
}

// Convert the fetched plane into ring slot `slot`; false when a tensor copy
// never completed (bounded wait).
template <bool TMA>
__device__ __forceinline__ bool gas3_commit(const Gas3Args &a, Gas3Plane &f, Gas3Smem &S, int slot)
{
    using T = Gas3T;
    if constexpr (TMA) {
        const bool ok = mbar_wait(&S.mbar, f.phase & 1u);
        f.phase++;
        if (!ok) return false;
    } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");   // this thread's copies have landed
    }
    float4 *pa = &S.pa[slot][0][0];
    float *pp = &S.pp[slot][0][0];
#pragma unroll
    for (int k = 0; k < T::K; k++) {
        if (threadIdx.x + k * T::THREADS >= T::NCONV) continue;
        const unsigned at = f.at[k] & 0xffffu, to = f.at[k] >> 16;
        float c5[5], w[5];
        unsigned flip;
        if constexpr (TMA) {
#pragma unroll
            for (int v = 0; v < 5; v++) c5[v] = S.xfer[v * T::BY * T::BX + at];
            flip = (f.mirror >> (2 * k) & 3u) | f.flip;
        } else {
#pragma unroll
            for (int v = 0; v < 5; v++) c5[v] = S.xfer[(k * 5 + v) * T::THREADS + threadIdx.x];
            flip = (f.flip >> (3 * k)) & 7u;
        }
        gas3_prim(a, c5, flip, w);
        pa[to] = make_float4(w[0], w[1], w[2], w[3]);
        pp[to] = w[4];
    }
    return true;
}

// The places of the thread's cells (Gas3Plane::at, mirror).
__device__ __forceinline__ void gas3_places(const Gas3Args &a, Gas3Plane &f, int ox, int oy, bool interior)
{
    using T = Gas3T;
    f.mirror = 0u;
#pragma unroll
    for (int k = 0; k < T::K; k++) {
        const int q = threadIdx.x + k * T::THREADS;
        f.at[k] = 0u;
        if (q >= T::NCONV) continue;
        int lx, ly;
        gas3_cell(q, lx, ly);
        // the cell's place in the box: the halo beyond a side is the
        // nearest cell or the mirror image (flip), clamped into the box
        // (cells far outside a small grid feed only faces outside it)
        bool fx = false, fy = false;
        int gx = ox + lx, gy = oy + ly;
        if (!interior) {
            gx = gas3_map(gx, a.n0, a.wall[0][0], a.wall[0][1], &fx);
            gy = gas3_map(gy, a.n1, a.wall[1][0], a.wall[1][1], &fy);
        }
        const int bx = min(max(gx - (ox - 4), 0), T::BX - 1), by = min(max(gy - (oy - T::H), 0), T::BY - 1);
        f.at[k] = (unsigned)(by * T::BX + bx) | (unsigned)((ly + T::H) * (T::PX + 1) + lx + T::H) << 16;
        f.mirror |= ((fx ? 1u : 0u) | (fy ? 2u : 0u)) << (2 * k);
    }
}

// (rho, u, v, w) and p, or the fluxes of (rho, rho u, rho v, rho w) and rho E:
// the four by twos on the packed FP32 units
struct Gas3S {
    float4 a;
    float p;
};

// primitives of the column's own cell in a ring slot
__device__ __forceinline__ Gas3S gas3_own(const Gas3Smem &S, int slot, int px, int py)
{
    return {S.pa[slot][py][px], S.pp[slot][py][px]};
}

// primitives of the own column's cell at plane z, loaded and converted
// directly (the planes below the chunk, needed for its first z slopes only)
__device__ __forceinline__ Gas3S gas3_column(const Gas3Args &a, int gx, int gy, int z)
{
    bool fz = false, fx = false, fy = false;
    const int gz = gas3_map(z, a.n2, a.wall[2][0], a.wall[2][1], &fz);
    const int cx = gas3_map(gx, a.n0, 0, 0, &fx), cy = gas3_map(gy, a.n1, 0, 0, &fy);
    const long long c = cx + (long long)a.n0 * (cy + (long long)a.n1 * gz);
    float q[5], w[5];
#pragma unroll
    for (int v = 0; v < 5; v++) q[v] = a.in[c + v * a.pitch];
    gas3_prim(a, q, fz ? 4u : 0u, w);
    return {make_float4(w[0], w[1], w[2], w[3]), w[4]};
}

// half the limited slope of four values
__device__ __forceinline__ float4 gas3_half(const float4 &m, const float4 &c, const float4 &p)
{
    const float4 d = gasw_sub(c, m), e = gasw_sub(p, c);
    return gasw_cat(gas_half_slope2(gasw_lo(d), gasw_lo(e)), gas_half_slope2(gasw_hi(d), gasw_hi(e)));
}
__device__ __forceinline__ float4 gas3_add(const float4 &x, const float4 &y)
{
    return gasw_cat(__fadd2_rn(gasw_lo(x), gasw_lo(y)), __fadd2_rn(gasw_hi(x), gasw_hi(y)));
}

// face values of cell c from its neighbours m and p: lo towards m, hi towards p
__device__ __forceinline__ void gas3_slope(const Gas3S &m, const Gas3S &c, const Gas3S &p, Gas3S &lo, Gas3S &hi)
{
    const float4 h = gas3_half(m.a, c.a, p.a);
    const float hp = gas_half_slope(c.p - m.p, p.p - c.p);
    lo.a = gasw_sub(c.a, h);
    hi.a = gas3_add(c.a, h);
    lo.p = c.p - hp;
    hi.p = c.p + hp;
}

// the same in x and y at once (the two pressures as a pair)
__device__ __forceinline__ void gas3_slope_xy(const Gas3S &xm, const Gas3S &xp, const Gas3S &ym, const Gas3S &yp,
                                              const Gas3S &c, Gas3S &xlo, Gas3S &xhi, Gas3S &ylo, Gas3S &yhi)
{
    const float4 hx = gas3_half(xm.a, c.a, xp.a), hy = gas3_half(ym.a, c.a, yp.a);
    xlo.a = gasw_sub(c.a, hx);
    xhi.a = gas3_add(c.a, hx);
    ylo.a = gasw_sub(c.a, hy);
    yhi.a = gas3_add(c.a, hy);
    const float2 cp = gas_f2(c.p, c.p);
    const float2 h = gas_half_slope2(gas_sub2(cp, gas_f2(xm.p, ym.p)), gas_sub2(gas_f2(xp.p, yp.p), cp));
    const float2 lo = gas_sub2(cp, h), hi = __fadd2_rn(cp, h);
    xlo.p = lo.x;
    ylo.p = lo.y;
    xhi.p = hi.x;
    yhi.p = hi.y;
}

// HLLC flux of a face normal to direction D (0, 1, 2)
template <int D>
__device__ __forceinline__ Gas3S gas3_face(const Gas3Args &a, const Gas3S &l, const Gas3S &r)
{
    float L[5] = {l.a.x, l.a.y, l.a.z, l.a.w, l.p}, R[5] = {r.a.x, r.a.y, r.a.z, r.a.w, r.p}, F[5];
    if (D == 1) {
        L[1] = l.a.z, L[2] = l.a.w, L[3] = l.a.y;
        R[1] = r.a.z, R[2] = r.a.w, R[3] = r.a.y;
    } else if (D == 2) {
        L[1] = l.a.w, L[2] = l.a.y, L[3] = l.a.z;
        R[1] = r.a.w, R[2] = r.a.y, R[3] = r.a.z;
    }
    gas_hllc3(a, L, R, F);
    return {D == 0 ? make_float4(F[0], F[1], F[2], F[3])
                   : (D == 1 ? make_float4(F[0], F[3], F[1], F[2]) : make_float4(F[0], F[2], F[3], F[1])),
            F[4]};
}

// A tensor copy that did not complete in the bounded wait: report it, and
// give it one more bounded wait before the CTA's shared memory is released.
__device__ __forceinline__ void gas3_fail(const Gas3Args &a, Gas3Smem &S, const Gas3Plane &f)
{
    if (threadIdx.x == 0) {
        atomicOr(&a.ctl->err, (unsigned)ERR_TIMEOUT);
        (void)mbar_wait(&S.mbar, (f.phase - 1u) & 1u);
    }
}

// a column's carried top z-face value and bottom z-face flux
__device__ __forceinline__ void gas3_carry(Gas3Smem &S, int tid, const Gas3S &q, const Gas3S &F)
{
    S.zqa[tid] = q.a;
    S.zqp[tid] = q.p;
    S.zfa[tid] = F.a;
    S.zfe[tid] = F.p;
}

// TMA: the plane boxes come by tensor copies through `map` (over the stage
// input's first five planes); else by per-thread asynchronous copies.
template <int STAGE, bool TMA>
__global__ void __launch_bounds__(Gas3T::THREADS, Gas3T::CTAS) k_gas3_stage(Gas3Args a, const __grid_constant__ CUtensorMap map)
{
    pdl_enter();
    using T = Gas3T;
    // the dynamic shared memory is the kernel's only shared memory and starts
    // the CTA's shared window; a tensor copy needs its slot 128-byte aligned
    extern __shared__ __align__(128) unsigned char gas3_smem_raw[];
    Gas3Smem &S = *reinterpret_cast<Gas3Smem *>(gas3_smem_raw);
    const int tid = threadIdx.x;
    if (TMA) {
        if ((smem_u32(S.xfer) & 127u) != 0) {
            // never issue a misaligned tensor copy: report and stop
            if (tid == 0) atomicOr(&a.ctl->err, (unsigned)ERR_TIMEOUT);
            return;
        }
        if (tid == 0) {
            mbar_init(&S.mbar, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        __syncthreads();
    }
    const int ox = blockIdx.x * T::TX, oy = blockIdx.y * T::TY;
    const int z0 = blockIdx.z * a.zc, z1 = min(z0 + a.zc, a.n2);
    const bool interior = ox >= T::H && ox + T::TX + T::H <= a.n0 && oy >= T::H && oy + T::TY + T::H <= a.n1;
    const bool own = tid < T::CELLS;
    const int ci = tid & 31, cj = tid >> 5;
    const int gx = ox + ci, gy = oy + cj;
    const bool col = own && gx < a.n0 && gy < a.n1;
    const int px = ci + T::H, py = cj + T::H;
    const float dt = ctl_dt<float>(a.ctl);
    const float ca = STAGE == 2 ? 0.75f : (STAGE == 3 ? 1.f / 3.f : 0.f);
    const float cb = STAGE == 2 ? 0.25f : (STAGE == 3 ? 2.f / 3.f : 1.f);
    if (STAGE == 2 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && tid == 0) ctl_box_reset(a.ctl);

    // prologue: planes z0, z0+1 into the ring, plane z0+2 into registers
    // (committed by the first plane's step 1);
    // the column's planes z0-2, z0-1 for its first z slopes
    Gas3Plane fp;
    fp.phase = 0u;
    gas3_places(a, fp, ox, oy, interior);
    gas3_fetch<TMA>(a, &map, S, fp, ox, oy, z0, interior);
    if (__syncthreads_or(!gas3_commit<TMA>(a, fp, S, z0 % T::RING))) {
        gas3_fail(a, S, fp);
        return;
    }
    gas3_fetch<TMA>(a, &map, S, fp, ox, oy, z0 + 1, interior);
    if (__syncthreads_or(!gas3_commit<TMA>(a, fp, S, (z0 + 1) % T::RING))) {
        gas3_fail(a, S, fp);
        return;
    }
    gas3_fetch<TMA>(a, &map, S, fp, ox, oy, z0 + 2, interior);
    if (own) {
        const Gas3S wm2 = gas3_column(a, gx, gy, z0 - 2), wm1 = gas3_column(a, gx, gy, z0 - 1);
        const Gas3S w0 = gas3_own(S, z0 % T::RING, px, py), w1 = gas3_own(S, (z0 + 1) % T::RING, px, py);
        Gas3S lo, hi, hm;
        gas3_slope(wm2, wm1, w0, lo, hm);    // plane z0-1: its top-face value hm
        gas3_slope(wm1, w0, w1, lo, hi);     // plane z0: bottom-face value lo, top-face value hi
        const Gas3S F = gas3_face<2>(a, hm, lo);   // the bottom z face of plane z0
        gas3_carry(S, tid, hi, F);
    }

    float smax_cell = 0.f;
    int zlo = 0x7fffffff, zhi = -1;
    for (int z = z0; z < z1; z++) {
        const int sz = z % T::RING, s1 = (z + 1) % T::RING, s2 = (z + 2) % T::RING;
        // 1. plane z+2 into the ring (its slot held plane z-1, whose last
        // readers are behind the previous plane's barriers); then, with the
        // fetch slot read by every thread, plane z+3 fetched into it
        if (__syncthreads_or(!gas3_commit<TMA>(a, fp, S, s2))) {
            gas3_fail(a, S, fp);
            return;
        }
        if (z + 3 <= z1 + 1) gas3_fetch<TMA>(a, &map, S, fp, ox, oy, z + 3, interior);
        if (col && z + 1 < z1) {
            // the cell's stage input and U^n at the next plane into L1 (read
            // at that plane's update; no register or shared slot holds them)
            const unsigned cn = gx + (unsigned)a.n0 * (gy + (unsigned)a.n1 * (z + 1));
#pragma unroll
            for (int v = 0; v < 6; v++) {
                asm volatile("prefetch.global.L1 [%0];" ::"l"((a.in + v * a.pitch) + cn));
                if (STAGE > 1) asm volatile("prefetch.global.L1 [%0];" ::"l"((a.un + v * a.pitch) + cn));
            }
        }

        // 2. slopes: x and y of plane z (face values to shared memory), z of plane z+1
        Gas3S qRx, qRy, qRz1, qLz1;
        if (own) {
            const Gas3S wc = gas3_own(S, sz, px, py);
            Gas3S hx, hy;
            gas3_slope_xy(gas3_own(S, sz, px - 1, py), gas3_own(S, sz, px + 1, py), gas3_own(S, sz, px, py - 1),
                          gas3_own(S, sz, px, py + 1), wc, qRx, hx, qRy, hy);
            S.fvxa[cj][ci + 1] = hx.a;
            S.fvxp[cj][ci + 1] = hx.p;
            S.fvya[cj + 1][ci] = hy.a;
            S.fvyp[cj + 1][ci] = hy.p;
            gas3_slope(wc, gas3_own(S, s1, px, py), gas3_own(S, s2, px, py), qRz1, qLz1);
        } else {
            // the extra warp: lanes 0-7 the right-face values of column -1,
            // lanes 8-15 the left-face values of column TX; every lane the
            // top-face value of row -1 and the bottom-face value of row TY
            const int l = tid - T::CELLS;
            const bool west = l < T::TY, east = !west && l < 2 * T::TY;
            const int jh = west ? l : (east ? l - T::TY : 0);
            const int cx = west ? T::H - 1 : T::TX + T::H;
            Gas3S lo, hi;
            gas3_slope(gas3_own(S, sz, cx - 1, jh + T::H), gas3_own(S, sz, cx, jh + T::H),
                       gas3_own(S, sz, cx + 1, jh + T::H), lo, hi);
            if (west) {
                S.fvxa[jh][0] = hi.a;
                S.fvxp[jh][0] = hi.p;
            } else if (east) {
                S.hrxa[jh] = lo.a;
                S.hrxp[jh] = lo.p;
            }
            gas3_slope(gas3_own(S, sz, l + T::H, T::H - 2), gas3_own(S, sz, l + T::H, T::H - 1),
                       gas3_own(S, sz, l + T::H, T::H), lo, hi);
            S.fvya[0][l] = hi.a;
            S.fvyp[0][l] = hi.p;
            gas3_slope(gas3_own(S, sz, l + T::H, T::TY + T::H - 1), gas3_own(S, sz, l + T::H, T::TY + T::H),
                       gas3_own(S, sz, l + T::H, T::TY + T::H + 1), lo, hi);
            S.hrya[l] = lo.a;
            S.hryp[l] = lo.p;
        }
        __syncthreads();

        // 3. faces: left x, bottom y, top z of the cell
        Gas3S Fxl, Fyl, Fzhi;
        if (own) {
            Fxl = gas3_face<0>(a, {S.fvxa[cj][ci], S.fvxp[cj][ci]}, qRx);
            Fyl = gas3_face<1>(a, {S.fvya[cj][ci], S.fvyp[cj][ci]}, qRy);
            Fzhi = gas3_face<2>(a, {S.zqa[tid], S.zqp[tid]}, qRz1);
            S.fxa[cj][ci] = Fxl.a;
            S.fxe[cj][ci] = Fxl.p;
            S.fya[cj][ci] = Fyl.a;
            S.fye[cj][ci] = Fyl.p;
        } else {
            const int l = tid - T::CELLS, jh = l < T::TY ? l : 0;
            if (l < T::TY) {
                const Gas3S F = gas3_face<0>(a, {S.fvxa[jh][T::TX], S.fvxp[jh][T::TX]}, {S.hrxa[jh], S.hrxp[jh]});
                S.fxa[jh][T::TX] = F.a;
                S.fxe[jh][T::TX] = F.p;
            }
            const Gas3S F = gas3_face<1>(a, {S.fvya[T::TY][l], S.fvyp[T::TY][l]}, {S.hrya[l], S.hryp[l]});
            S.fya[T::TY][l] = F.a;
            S.fye[T::TY][l] = F.p;
        }
        __syncthreads();

        // 4. update of plane z: the cell's stage input and step-start values
        // (loaded here, not held through the faces: three CTAs fit an SM)
        // (a 32-bit index from each plane's address: cells are fewer than 2^32)
        const unsigned c = gx + (unsigned)a.n0 * (gy + (unsigned)a.n1 * z);
        if (col) {
            float cin[6], cun[6];
#pragma unroll
            for (int v = 0; v < 6; v++) {
                cin[v] = (a.in + v * a.pitch)[c];
                cun[v] = (a.un + v * a.pitch)[c];
            }
            const bool masked = cun[5] > 0.5f;
            float o[6];
            // D = dFx/dx + dFy/dy + dFz/dz; out = ca un + cb (in - dt D), D rounded three
            // times, as the products of a compensated sum are (gasw_update2); that spills
            // at 72 registers: 256^3 9.1 ms a pass against 8.5, with errors after 150
            // steps within 0.1 % of these (momenta 0.3 %)
            const float4 dx = gasw_sub(S.fxa[cj][ci + 1], Fxl.a), dy = gasw_sub(S.fya[cj + 1][ci], Fyl.a),
                         dz = gasw_sub(Fzhi.a, S.zfa[tid]);
            const float2 ix = gas_f2(a.idx, a.idx), iy = gas_f2(a.idy, a.idy), iz = gas_f2(a.idz, a.idz);
            const float2 mdt = gas_f2(-dt, -dt), ca2 = gas_f2(ca, ca), cb2 = gas_f2(cb, cb);
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const float2 D = __ffma2_rn(h ? gasw_hi(dz) : gasw_lo(dz), iz,
                                            __ffma2_rn(h ? gasw_hi(dy) : gasw_lo(dy), iy,
                                                       __fmul2_rn(h ? gasw_hi(dx) : gasw_lo(dx), ix)));
                const float2 y = __ffma2_rn(mdt, D, gas_f2(cin[2 * h], cin[2 * h + 1]));
                const float2 n = gas_f2(cun[2 * h], cun[2 * h + 1]);
                const float2 t = STAGE == 1 ? y : __ffma2_rn(cb2, y, __fmul2_rn(ca2, n));
                o[2 * h] = masked ? n.x : t.x;
                o[2 * h + 1] = masked ? n.y : t.y;
            }
            {
                const float D = fmaf(Fzhi.p - S.zfe[tid], a.idz,
                                     fmaf(S.fye[cj + 1][ci] - Fyl.p, a.idy, (S.fxe[cj][ci + 1] - Fxl.p) * a.idx));
                const float y = fmaf(-dt, D, cin[4]);
                o[4] = masked ? cun[4] : (STAGE == 1 ? y : fmaf(cb, y, __fmul_rn(ca, cun[4])));
            }
            // r: no flux without a moving body
            o[5] = STAGE == 1 ? cin[5] : fmaf(cb, cin[5], __fmul_rn(ca, cun[5]));
#pragma unroll
            for (int v = 0; v < 6; v++) (a.out + v * a.pitch)[c] = o[v];
            if (!(o[0] > 0.f) || !(o[4] == o[4])) atomicOr(&a.ctl->err, (unsigned)ERR_STATE);
            if (STAGE == 3) {
                if (o[5] > 0.5f) {
                    zlo = min(zlo, z);
                    zhi = max(zhi, z);
                }
                const float inv[3] = {a.idx, a.idy, a.idz};
                float c2;
                smax_cell = fmaxf(smax_cell, gas_speed<3>(a.Gam, a.pref0, o, inv, c2));
                if (!(c2 > 0.f)) atomicOr(&a.ctl->err, (unsigned)ERR_SOUND);
            }
        }
        if (own) gas3_carry(S, tid, qLz1, Fzhi);
    }
    if (STAGE == 3) {
        // the column's rigid cells into the box of the next seeding, the
        // chunk's CFL maximum into the launch's running maximum
        const bool rig = zhi >= 0;
        if (__any_sync(0xffffffffu, rig)) {
            const int big = 0x7fffffff;
            const int b[6] = {rig ? gx : big, rig ? gy : big, rig ? zlo : big, rig ? gx : -1, rig ? gy : -1,
                              rig ? zhi : -1};
            int m[6];
#pragma unroll
            for (int k = 0; k < 3; k++) {
                m[k] = __reduce_min_sync(0xffffffffu, b[k]);
                m[3 + k] = __reduce_max_sync(0xffffffffu, b[3 + k]);
            }
            if ((tid & 31) == 0) {
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    atomicMin(&a.ctl->rnext[k], m[k]);
                    atomicMax(&a.ctl->rnext[3 + k], m[3 + k]);
                }
            }
        }
        float *sr = reinterpret_cast<float *>(S.red);
        const float mx = block_max<T::THREADS, float>(smax_cell, sr);
        if (tid == 0) {
            double md = (double)mx;
            if (!(md >= 0.0)) md = __longlong_as_double(0x7ff0000000000000LL);   // NaN -> +inf: dt = 0
            atomicMax(&a.ctl->smax_acc, (unsigned long long)__double_as_longlong(md));
        }
    }
}

// Host side (dfv_gas_f32_k.cu).
cudaError_t gas3_prepare();
// The tensor map of a stage input's first five planes (rho .. rho E) with the
// plane box of the kernel: 4-D (x, y, z, variable) over n0 x n1 x n2 x 5
// floats at base, row stride n0, plane stride n0 n1, variable stride pitch.
// False when the grid does not allow it (rows or planes not a multiple of 16
// bytes, a misaligned base); the kernel then copies per thread.
int gas3_planes(int n0, int n1, int n2);   // planes per CTA
bool gas3_encode_map(CUtensorMap *map, const void *base, int n0, int n1, int n2, long long pitch);
// map: the stage input's tensor map, or nullptr for the per-thread copies.
cudaError_t gas3_stage(int stage, const Gas3Args &a, const CUtensorMap *map, cudaStream_t st);

}  // namespace dfv
