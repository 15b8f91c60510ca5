// dfv_kernels_z.cuh -- the 3-D single-material stage kernel that marches along
// z (2.5-D blocking), for the grids that the FP32 gas kernel (dfv_gas3.cuh)
// does not take: every FP64 one, and in FP32 moving bodies, periodic sides,
// HLLC-LM and solids' equations of state.  A CTA owns a column of 256 cells and
// advances through zc planes; the primitives of three planes (z, z+1, z+2,
// each with its x and y halo, corners unused) sit in a ring in shared memory,
// so every plane is converted once per chunk, every slope formed once and
// every face solved once (the tiled kernel converts 5.7 cells per cell and
// solves 3.8 faces).  What the z direction carries from plane to plane, the
// upper face value and the flux of the face below, stays in the thread of the
// column; r, which the BVD rule needs two planes further, is read from global
// memory.  Same arithmetic per face and per cell as k_stage (Sec. 3.1).
#pragma once

#include "dfv_kernels.cuh"

namespace dfv {

// Column of 32 x 8 cells in FP32, 16 x 16 in FP64: there the time is the number
// of FP64 instructions of whole warps, and the square column has the smaller
// halo (384 against 416 conversions per 256 cells) and wastes less on grids
// that are no multiple of 32 wide.
template <class R>
struct ZGeo {
    static constexpr int TX = sizeof(R) == 8 ? 16 : 32, TY = 256 / TX;
    static constexpr int HX = 3, HY = 3;
    static constexpr int BX = TX + 2 * HX, BY = TY + 2 * HY;  // one plane with halo
    static constexpr int SN = BX * BY;
    static constexpr int RING = 3;                            // planes z, z+1, z+2
    static constexpr int CELLS = TX * TY;
    static constexpr int THREADS = CELLS + 32;                // + a warp for the closing x and y faces
    static constexpr int FX = (TX + 1) * TY, FY = TX * (TY + 1);
    static constexpr int MAXF = FX > FY ? FX : FY;
    static_assert(TX <= 32 && TY <= 32, "one lane of the extra warp per pencil");
};

template <class R, int NMAT>
struct ZSmem {
    using L = Lay<3, NMAT, 0>;
    using Z = ZGeo<R>;
    static constexpr size_t floats = (size_t)Z::RING * L::NVAR * Z::SN + 2 * (size_t)L::NF * Z::MAXF;
    static constexpr size_t bytes = ((sizeof(R) * floats + 7) & ~(size_t)7) + 4 * 32 * sizeof(double);
};

// Primitives of one cell of plane z (mapped beyond the sides as in the tiled
// kernel: nearest cell, periodic image or mirror image).
template <class R, int NMAT>
__device__ __forceinline__ void z_cell(const GridP &g, const R *in, int x, int y, int z, bool interior, R *w)
{
    using L = Lay<3, NMAT, 0>;
    bool fl[3] = {false, false, false};
    int gx = x, gy = y;
    if (!interior) {
        gx = halo_idx(g, 0, x, &fl[0]);
        gy = halo_idx(g, 1, y, &fl[1]);
    }
    const int gz = halo_idx(g, 2, z, &fl[2]);
    const long long c = gx + (long long)g.n[0] * (gy + (long long)g.n[1] * gz);
    R q[L::NVAR];
#pragma unroll
    for (int v = 0; v < L::NVAR; v++) q[v] = in[v * g.pitch + c];
    cons_to_prim<R, 3, NMAT, 0>(g, q, w);
#pragma unroll
    for (int d = 0; d < 3; d++)
        if (fl[d]) w[L::IMOM + d] = -w[L::IMOM + d];
}

// plane z with its halo of hw into a ring slot
template <class R, int NMAT>
__device__ __forceinline__ void z_plane(const GridP &g, const R *in, R *dst, int ox, int oy, int z, int hw,
                                        bool interior)
{
    using L = Lay<3, NMAT, 0>;
    using Z = ZGeo<R>;
    const int px = Z::TX + 2 * hw, n1 = px * Z::TY, n2 = n1 + 2 * hw * Z::TX;
    for (int i = threadIdx.x; i < n2; i += Z::THREADS) {
        int lx, ly;
        if (i < n1) {
            ly = hw == 2 ? i / (Z::TX + 4) : i / (Z::TX + 6);
            lx = i - ly * px - hw;
        } else {
            const int k = i - n1, h = k / Z::TX;
            lx = k % Z::TX;
            ly = h < hw ? h - hw : Z::TY + h - hw;
        }
        R w[L::NVAR];
        z_cell<R, NMAT>(g, in, ox + lx, oy + ly, z, interior, w);
        const int ib = (ly + Z::HY) * Z::BX + (lx + Z::HX);
#pragma unroll
        for (int v = 0; v < L::NVAR; v++) dst[v * Z::SN + ib] = w[v];
    }
}

// Reconstruction of direction D (0, 1) of a plane, as slope_pass of the tiled
// kernel; the extra warp's lane e does pencil e.
template <class R, int NMAT, int D>
__device__ __forceinline__ void z_slopes(const GridP &g, const R *pl, R *sQ, R vr, R *lo)
{
    using L = Lay<3, NMAT, 0>;
    using Z = ZGeo<R>;
    constexpr int T = D == 0 ? Z::TX : Z::TY, SB = D == 0 ? 1 : Z::BX, EX = Z::TX + (D == 0), SF = D == 0 ? 1 : EX;
    const int t = threadIdx.x, e = t - Z::CELLS;
    const bool own = t < Z::CELLS;
    if (!own && e >= Z::CELLS / T) return;
    const int lx = own ? t % Z::TX : (D == 0 ? 0 : e), ly = own ? t / Z::TX : (D == 0 ? e : 0);
    const R *w0 = pl + (ly + Z::HY) * Z::BX + (lx + Z::HX);
    R *q0 = sQ + ly * EX + lx;
#pragma unroll
    for (int v = 0; v < L::NVAR; v++) {
        const bool frac = (v >= L::IPHI && v < L::IPHI + NMAT - 1) || v == L::IR;
        if (v == L::IR && vr == R(0)) {
            lo[v] = R(0);
            continue;
        }
        const R *w = w0 + v * Z::SN;
        R *q = q0 + v * Z::MAXF;
        R s[5], hi, dummy;
        if (own) {
#pragma unroll
            for (int k = 0; k < 5; k++) s[k] = (frac || (k > 0 && k < 4)) ? w[(k - 2) * SB] : R(0);
            recon_form<R, NMAT, 0>(g, s, frac, lo[v], hi);
            q[SF] = hi;
        } else {
#pragma unroll
            for (int k = 0; k < 5; k++) s[k] = (frac || (k > 0 && k < 4)) ? w[(k - 3) * SB] : R(0);
            recon_form<R, NMAT, 0>(g, s, frac, dummy, hi);
            q[0] = hi;
#pragma unroll
            for (int k = 0; k < 5; k++) s[k] = (frac || (k > 0 && k < 4)) ? w[(k - 2 + T) * SB] : R(0);
            recon_form<R, NMAT, 0>(g, s, frac, lo[v], dummy);
        }
    }
}

// the face fluxes of direction D (0, 1) of the plane, in place (face_pass)
template <class R, int NMAT, int D>
__device__ __forceinline__ void z_faces(const GridP &g, R *sQ, R vr, const R *lo)
{
    using L = Lay<3, NMAT, 0>;
    using Z = ZGeo<R>;
    constexpr int T = D == 0 ? Z::TX : Z::TY, EX = Z::TX + (D == 0), SF = D == 0 ? 1 : EX;
    const int t = threadIdx.x, e = t - Z::CELLS;
    const bool own = t < Z::CELLS;
    if (!own && e >= Z::CELLS / T) return;
    const int lx = own ? t % Z::TX : (D == 0 ? 0 : e), ly = own ? t / Z::TX : (D == 0 ? e : 0);
    R *q = sQ + ly * EX + lx + (own ? 0 : T * SF);
    R wL[L::NVAR], F[L::NF];
#pragma unroll
    for (int v = 0; v < L::NVAR; v++) wL[v] = (v == L::IR && vr == R(0)) ? R(0) : q[v * Z::MAXF];
    riemann<R, 3, NMAT, 0, D>(g, wL, lo, vr, F);
#pragma unroll
    for (int k = 0; k < L::NF; k++) q[k * Z::MAXF] = F[k];
}

// divergence of direction D (0, 1) of the thread's cell (accum_pass)
template <class R, int NMAT, int D>
__device__ __forceinline__ void z_accum(const GridP &g, const R *sQ, const R *w, bool rest, Acc<R> *Dacc)
{
    using L = Lay<3, NMAT, 0>;
    using Z = ZGeo<R>;
    constexpr int EX = Z::TX + (D == 0), SF = D == 0 ? 1 : EX;
    const R *q = sQ + (threadIdx.x / Z::TX) * EX + threadIdx.x % Z::TX;
    const R inv = gridc<R>(g).inv_dx[D];
    const R dus = NMAT > 1 ? q[L::NVAR * Z::MAXF + SF] - q[L::NVAR * Z::MAXF] : R(0);
#pragma unroll
    for (int v = 0; v < L::NVAR; v++) {
        if (sizeof(R) == 8 && v >= NMAT - 1) {
            // FP64: as accum_pass
            if (v == L::IR && rest) continue;
            const R df = q[v * Z::MAXF + SF] - q[v * Z::MAXF];
            Dacc[v].hi = D == 0 ? df * inv : m_fma(df, inv, Dacc[v].hi);
            continue;
        }
        const R div = (q[v * Z::MAXF + SF] - q[v * Z::MAXF]) * inv;
        const R snc = (v >= L::IPHI && v < L::IPHI + NMAT - 1) ? w[v] * dus * inv : R(0);
        if (D == 0) Dacc[v].set(div - snc);
        else Dacc[v].add(div - snc);
    }
}

// r (or a volume fraction: plane v, a primitive as it is stored) of the
// thread's column at plane z
template <class R>
__device__ __forceinline__ R z_raw(const GridP &g, const R *in, int v, int gx, int gy, int z)
{
    bool fl = false;
    const int gz = halo_idx(g, 2, z, &fl);
    return in[v * g.pitch + gx + (long long)g.n[0] * (gy + (long long)g.n[1] * gz)];
}

// Face values in z of plane z of the thread's column from its primitives at
// planes z-1, z, z+1 (fractions: read at z-2 .. z+2).
template <class R, int NMAT>
__device__ __forceinline__ void z_slope_z(const GridP &g, const R *in, const R *wm, const R *w0, const R *wp, int gx,
                                          int gy, int z, R vr, R *lo, R *hi)
{
    using L = Lay<3, NMAT, 0>;
#pragma unroll
    for (int v = 0; v < L::NVAR; v++) {
        const bool frac = (v >= L::IPHI && v < L::IPHI + NMAT - 1) || v == L::IR;
        if (v == L::IR && vr == R(0)) {
            lo[v] = hi[v] = R(0);
            continue;
        }
        R s[5] = {R(0), wm[v], w0[v], wp[v], R(0)};
        if (frac) {
            s[0] = z_raw(g, in, v, gx, gy, z - 2);
            s[4] = z_raw(g, in, v, gx, gy, z + 2);
        }
        recon_form<R, NMAT, 0>(g, s, frac, lo[v], hi[v]);
    }
}

// REST: the body is at rest (no r to reconstruct).  Two CTAs per SM in FP64
// (ring and face arrays 106 KB), three in FP32; a moving body's FP64 kernel
// takes the registers of one CTA instead, since with the BVD choice of r it
// would spill 600 bytes a thread (105 in stage 3 as it is, 300 at rest, of the
// 168 and 96 registers that the CTAs leave).  Measured in FP64 over two steps: sphere
// 52 x 70 x 59 moving 7172 us with two CTAs, 4500 with one; 97 x 90 x 101 at
// rest 7236 with one, 6668 with two, 6385 since REST is known at compile time.
template <class R, int NMAT, int STAGE, bool REST>
__global__ void __launch_bounds__(ZGeo<R>::THREADS, sizeof(R) == 8 ? (REST ? 2 : 1) : 3)
    k_stage_z(StageArgs a, GridP g, int zc)
{
    pdl_enter();
    using L = Lay<3, NMAT, 0>;
    using Z = ZGeo<R>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using SM = ZSmem<R, NMAT>;
    R *ring = reinterpret_cast<R *>(smem_raw);
    R *sQx = ring + (size_t)Z::RING * L::NVAR * Z::SN;
    R *sQy = sQx + (size_t)L::NF * Z::MAXF;
    double *sred = reinterpret_cast<double *>(smem_raw + ((sizeof(R) * SM::floats + 7) & ~(size_t)7));
    const R *in = reinterpret_cast<const R *>(a.in);
    const R *un = reinterpret_cast<const R *>(a.un);
    R *out = reinterpret_cast<R *>(a.out);
    const long long P = g.pitch;
    const int ox = blockIdx.x * Z::TX, oy = blockIdx.y * Z::TY;
    const int z0 = blockIdx.z * zc, z1 = min(z0 + zc, g.n[2]);
    constexpr int hw = NMAT == 1 && REST ? 2 : 3;
    const bool interior = ox >= hw && ox + Z::TX + hw <= g.n[0] && oy >= hw && oy + Z::TY + hw <= g.n[1];
    const bool own = threadIdx.x < Z::CELLS;
    const int lx = threadIdx.x % Z::TX, ly = threadIdx.x / Z::TX;
    const int gx = ox + lx, gy = oy + ly;
    const bool col = own && gx < g.n[0] && gy < g.n[1];
    const int cell = own ? (ly + Z::HY) * Z::BX + (lx + Z::HX) : 0;
    R vr[3];
#pragma unroll
    for (int d = 0; d < 3; d++) vr[d] = REST ? R(0) : ctl_v<R>(a.ctl, d);
    const R dt = ctl_dt<R>(a.ctl);
    const R ca = STAGE == 2 ? R(0.75) : (STAGE == 3 ? R(1.0 / 3.0) : R(0));
    const R cb = STAGE == 2 ? R(0.25) : (STAGE == 3 ? R(2.0 / 3.0) : R(1));
    const GridC<R> &gc = gridc<R>(g);
    if (STAGE == 2 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && threadIdx.x == 0) ctl_box_reset(a.ctl);

    // planes z0, z0+1; the column's first z face and upper face value
    z_plane<R, NMAT>(g, in, ring + (size_t)(z0 % Z::RING) * L::NVAR * Z::SN, ox, oy, z0, hw, interior);
    z_plane<R, NMAT>(g, in, ring + (size_t)((z0 + 1) % Z::RING) * L::NVAR * Z::SN, ox, oy, z0 + 1, hw, interior);
    __syncthreads();
    R hz[L::NVAR], Flo[L::NF];   // upper face value of plane z, flux of the face below it
    if (col) {
        R wm2[L::NVAR], wm1[L::NVAR], w0[L::NVAR], w1[L::NVAR], lo[L::NVAR], hm[L::NVAR], dummy[L::NVAR];
        z_cell<R, NMAT>(g, in, gx, gy, z0 - 2, true, wm2);
        z_cell<R, NMAT>(g, in, gx, gy, z0 - 1, true, wm1);
#pragma unroll
        for (int v = 0; v < L::NVAR; v++) {
            w0[v] = ring[((size_t)(z0 % Z::RING) * L::NVAR + v) * Z::SN + cell];
            w1[v] = ring[((size_t)((z0 + 1) % Z::RING) * L::NVAR + v) * Z::SN + cell];
        }
        z_slope_z<R, NMAT>(g, in, wm2, wm1, w0, gx, gy, z0 - 1, vr[2], dummy, hm);
        z_slope_z<R, NMAT>(g, in, wm1, w0, w1, gx, gy, z0, vr[2], lo, hz);
        riemann<R, 3, NMAT, 0, 2>(g, hm, lo, vr[2], Flo);
    }

    R smax_cell = R(0);
    int zlo = 0x7fffffff, zhi = -1;
    for (int z = z0; z < z1; z++) {
        const R *p0 = ring + (size_t)(z % Z::RING) * L::NVAR * Z::SN;
        const R *p1 = ring + (size_t)((z + 1) % Z::RING) * L::NVAR * Z::SN;
        R *p2 = ring + (size_t)((z + 2) % Z::RING) * L::NVAR * Z::SN;
        // plane z+2 (its slot held plane z-1, last read before the barrier
        // between slopes and faces of the previous plane)
        z_plane<R, NMAT>(g, in, p2, ox, oy, z + 2, hw, interior);
        __syncthreads();
        R lox[L::NVAR], loy[L::NVAR], loz[L::NVAR], hz1[L::NVAR];
        z_slopes<R, NMAT, 0>(g, p0, sQx, vr[0], lox);
        z_slopes<R, NMAT, 1>(g, p0, sQy, vr[1], loy);
        R w0[L::NVAR];
        if (col) {
            R w1[L::NVAR], w2[L::NVAR];
#pragma unroll
            for (int v = 0; v < L::NVAR; v++) {
                w0[v] = p0[v * Z::SN + cell];
                w1[v] = p1[v * Z::SN + cell];
                w2[v] = p2[v * Z::SN + cell];
            }
            z_slope_z<R, NMAT>(g, in, w0, w1, w2, gx, gy, z + 1, vr[2], loz, hz1);
        }
        __syncthreads();
        z_faces<R, NMAT, 0>(g, sQx, vr[0], lox);
        z_faces<R, NMAT, 1>(g, sQy, vr[1], loy);
        R Fhi[L::NF];
        if (col) riemann<R, 3, NMAT, 0, 2>(g, hz, loz, vr[2], Fhi);
        __syncthreads();
        if (col) {
            const long long c = gx + (long long)g.n[0] * (gy + (long long)g.n[1] * z);
            Acc<R> Dacc[L::NVAR];
            // x, then y, then z, in the order of the tiled kernel
            z_accum<R, NMAT, 0>(g, sQx, w0, REST, Dacc);
            z_accum<R, NMAT, 1>(g, sQy, w0, REST, Dacc);
            const R inv = gc.inv_dx[2];
            const R dus = Fhi[L::NVAR] - Flo[L::NVAR];
            R cun[L::NVAR], o[L::NVAR];
#pragma unroll
            for (int v = 0; v < L::NVAR; v++) cun[v] = un[v * P + c];
            const bool masked = cun[L::IR] > R(0.5);
#pragma unroll
            for (int v = 0; v < L::NVAR; v++) {
                if (sizeof(R) == 8 && v >= NMAT - 1) {
                    if (v == L::IR && REST) {
                        o[v] = STAGE == 1 ? in[v * P + c] : ca * cun[v] + cb * in[v * P + c];
                        continue;
                    }
                    Dacc[v].hi = m_fma(Fhi[v] - Flo[v], inv, Dacc[v].hi);
                    o[v] = (masked && v != L::IR) ? cun[v]
                                                  : rk_combine<R>(STAGE, cun[v], in[v * P + c], Dacc[v], dt, ca, cb);
                    continue;
                }
                const R div = (Fhi[v] - Flo[v]) * inv;
                const R snc = (v >= L::IPHI && v < L::IPHI + NMAT - 1) ? w0[v] * dus * inv : R(0);
                Dacc[v].add(div - snc);
                o[v] = (masked && v != L::IR) ? cun[v] : rk_combine<R>(STAGE, cun[v], in[v * P + c], Dacc[v], dt, ca, cb);
            }
#pragma unroll
            for (int v = 0; v < L::NVAR; v++) out[v * P + c] = o[v];
            if (!(o[L::IAR] + (NMAT > 1 ? o[L::IAR + NMAT - 1] : R(0)) > R(0)) || !(o[L::IE] == o[L::IE]))
                atomicOr(&a.ctl->err, (unsigned)ERR_STATE);
            if (STAGE == 3) {
                if (o[L::IR] > R(0.5)) {
                    zlo = min(zlo, z);
                    zhi = max(zhi, z);
                }
                R cs;
                const R sum = cell_speed<R, 3, NMAT, 0>(g, o, cs);
                if (!(cs > R(0))) atomicOr(&a.ctl->err, (unsigned)ERR_SOUND);
                smax_cell = nan_max(smax_cell, sum);
            }
#pragma unroll
            for (int k = 0; k < L::NF; k++) Flo[k] = Fhi[k];
#pragma unroll
            for (int v = 0; v < L::NVAR; v++) hz[v] = hz1[v];
        }
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
            if ((threadIdx.x & 31) == 0) {
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    atomicMin(&a.ctl->rnext[k], m[k]);
                    atomicMax(&a.ctl->rnext[3 + k], m[3 + k]);
                }
            }
        }
        R *sr = reinterpret_cast<R *>(sred);
        const R mx = block_max<Z::THREADS, R>(smax_cell, sr);
        if (threadIdx.x == 0) {
            double md = (double)mx;
            if (!(md >= 0.0)) md = __longlong_as_double(0x7ff0000000000000LL);   // NaN -> +inf: dt = 0
            atomicMax(&a.ctl->smax_acc, (unsigned long long)__double_as_longlong(md));
        }
    }
}

}  // namespace dfv
