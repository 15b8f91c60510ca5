// dfv_device.cuh -- device-side physics of the diffuse rigid-body
// finite-volume update (arXiv:2111.11806), written for sm_103a.
//
// Everything here is a __device__ function templated on the compute type T
// (double for the plain FP64 form, float for the FP32 bulk form) and on the
// system shape (dimension, number of materials, solid or fluid), so that every
// index into the per-cell state is a compile-time constant and lives in
// registers.  The stretch-tensor logarithm and the plastic return are always
// evaluated in FP64.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

namespace dfv {

// ------------------------------------------------------------------ params

struct MatP {
    int kind;                 // 0 ideal, 1 stiffened, 2 Romenskii
    double gamma, pinf;
    double rho0, K0, G0, alpha, beta, Gamma0;
    double sigY;
    int jc;                   // 1: Johnson-Cook flow stress instead of sigY
    double jc_c1, jc_c2, jc_c3, jc_n, jc_m, jc_tmelt, jc_cv;
};

// Material and grid constants in the compute precision, derived on the host
// (finish_params) so that the FP32 form does no double-precision arithmetic
// or conversion in its face and cell loops.
template <class T>
struct MatC {
    int kind;
    T Gam;          // Grueneisen coefficient (gamma - 1 for the gases)
    T invGam;       // 1 / Gam
    T pref0;        // constant p_ref of the gases (-gamma p_inf, 0)
    T rho0, K0, G0, alpha, beta, sigY;
    // products of the constants that the closures use, so that they divide by
    // nothing: 1 + 1/Gam, p_ref/Gam (gases), 1/rho0, K0/(2 alpha^2), K0/alpha,
    // 1/alpha, beta + 1, beta (beta + 1)
    T Gam1;         // 1 + Gam
    T kA, kB, irho0, kE, kP, ialpha, beta1, bb;
    int n_alpha, n_beta1;   // alpha, beta + 1 where they are whole numbers 1..8, else 0
    int has_rho0;
};

template <class T>
struct GridC {
    T lo[3], dx[3], inv_dx[3];
    T dxmin, dV;
    T beta, cosh_b, sinh_b, tanh_b;   // THINC constants
    T inv_sinh_b;
    T phi_guard;
};

struct GridP {
    int dim;
    int n[3];
    int periodic[3];
    double lo[3], dx[3], inv_dx[3];
    long long ncell, pitch;   // cells, elements between planes
    double dV, dxmin;
    MatP mat[3];
    int use_thinc;
    int hllc_lm;        // 1: low-Mach HLLC-LM dissipation in the star regions
    int seed_variant;   // 0: reflected state (Sec. 3.2), 1: Riemann-problem star state
    int normal_method;  // 0: Youngs, 1: ELVIRA (2-D) (Sec. 3.3)
    int probe_mode;     // 0: stepped probe 1.0..4.0 dx, 1: fixed 1.5 dx (Sec. 3.2)
    int wall[3][2];     // reflective wall on the low / high side of direction d
    double beta, cosh_b, sinh_b, tanh_b;   // THINC constants
    double phi_guard;
    MatC<double> mc_d[3];
    MatC<float> mc_f[3];
    GridC<double> gc_d;
    GridC<float> gc_f;
    int any_jc;         // some material has a Johnson-Cook flow stress
};

// an exponent that is one of the whole numbers 1..8, else 0
__host__ inline int whole_power(double e)
{
    return e >= 1.0 && e <= 8.0 && e == std::floor(e) ? (int)e : 0;
}

template <class T>
__host__ inline void fill_consts(const GridP &g, MatC<T> *mc, GridC<T> &gc)
{
    for (int l = 0; l < 3; l++) {
        const MatP &m = g.mat[l];
        mc[l].kind = m.kind;
        mc[l].Gam = (T)(m.kind == 2 ? m.Gamma0 : m.gamma - 1.0);
        mc[l].invGam = (T)(1.0 / (m.kind == 2 ? m.Gamma0 : m.gamma - 1.0));
        mc[l].pref0 = (m.kind == 1) ? (T)(-m.gamma * m.pinf) : T(0);
        mc[l].rho0 = (T)m.rho0;
        mc[l].K0 = (T)m.K0;
        mc[l].G0 = (T)m.G0;
        mc[l].alpha = (T)m.alpha;
        mc[l].beta = (T)m.beta;
        mc[l].sigY = (T)m.sigY;
        mc[l].has_rho0 = m.rho0 > 0.0;
        const double iG = 1.0 / (m.kind == 2 ? m.Gamma0 : m.gamma - 1.0);
        mc[l].Gam1 = (T)(1.0 + (m.kind == 2 ? m.Gamma0 : m.gamma - 1.0));
        mc[l].kA = (T)(1.0 + iG);
        mc[l].kB = m.kind == 1 ? (T)(-m.gamma * m.pinf * iG) : T(0);
        mc[l].irho0 = m.rho0 > 0.0 ? (T)(1.0 / m.rho0) : T(0);
        mc[l].kE = m.alpha != 0.0 ? (T)(m.K0 / (2.0 * m.alpha * m.alpha)) : T(0);
        mc[l].kP = m.alpha != 0.0 ? (T)(m.K0 / m.alpha) : T(0);
        mc[l].ialpha = m.alpha != 0.0 ? (T)(1.0 / m.alpha) : T(0);
        mc[l].beta1 = (T)(m.beta + 1.0);
        mc[l].bb = (T)(m.beta * (m.beta + 1.0));
        mc[l].n_alpha = whole_power(m.alpha);
        mc[l].n_beta1 = whole_power(m.beta + 1.0);
    }
    for (int d = 0; d < 3; d++) {
        gc.lo[d] = (T)g.lo[d];
        gc.dx[d] = (T)g.dx[d];
        gc.inv_dx[d] = (T)g.inv_dx[d];
    }
    gc.dxmin = (T)g.dxmin;
    gc.dV = (T)g.dV;
    gc.beta = (T)g.beta;
    gc.cosh_b = (T)g.cosh_b;
    gc.sinh_b = (T)g.sinh_b;
    gc.tanh_b = (T)g.tanh_b;
    gc.inv_sinh_b = (T)(1.0 / g.sinh_b);
    gc.phi_guard = (T)g.phi_guard;
}

// The scheme options of a grid: THINC on/off and its steepness (default 1.6),
// the HLLC-LM flux, the seeding variant, the normal method and the probe.
__host__ inline void apply_options(GridP &g, int use_thinc, double thinc_beta, int hllc_lm, int seed_variant,
                                   int normal_method, int probe_mode)
{
    g.normal_method = normal_method == 1 ? 1 : 0;
    g.probe_mode = probe_mode == 1 ? 1 : 0;
    g.use_thinc = use_thinc ? 1 : 0;
    g.beta = thinc_beta > 0.0 ? thinc_beta : 1.6;
    g.cosh_b = std::cosh(g.beta);
    g.sinh_b = std::sinh(g.beta);
    g.tanh_b = std::tanh(g.beta);
    g.hllc_lm = hllc_lm ? 1 : 0;
    g.seed_variant = seed_variant == 1 ? 1 : 0;
    g.phi_guard = 1e-14;
}

// The checks of one material's parameters (kind 0 ideal, 1 stiffened, 2
// Romenskii), shared by every entry point that takes materials: nullptr when
// valid, else what is wrong.  Gases need gamma > 1 (Gamma = gamma - 1 > 0);
// the Romenskii solid needs rho0 > 0, Gamma0 > 0 and alpha != 0 (Sec. 2.1.3,
// eq:Romenskii divides by both).
__host__ inline const char *material_problem(int kind, double gamma, double rho0, double Gamma0, double alpha,
                                             double jc_c1 = 0.0, double jc_c2 = 0.0, double jc_n = 0.0,
                                             double jc_tmelt = 0.0, double jc_cv = 0.0)
{
    if (kind < 0 || kind > 2) return "bad material kind";
    if (kind != 2 && !(gamma > 1.0)) return "gamma <= 1";
    if (kind == 2 && !(rho0 > 0.0 && Gamma0 > 0.0 && alpha != 0.0)) return "bad Romenskii parameters";
    if ((jc_c1 > 0.0 || jc_c2 > 0.0) && !(jc_tmelt > 298.0 && jc_cv > 0.0 && jc_n >= 0.0 && jc_c1 >= 0.0 &&
                                         jc_c2 >= 0.0))
        return "bad Johnson-Cook parameters";
    return nullptr;
}

// Copy the caller's material parameters (dfvrb.h) into a MatP.
template <class P>
__host__ inline void set_material(MatP &m, int kind, const P &p)
{
    m.kind = kind;
    m.gamma = p.gamma;
    m.pinf = p.pinf;
    m.rho0 = p.rho0;
    m.K0 = p.K0;
    m.G0 = p.G0;
    m.alpha = p.alpha;
    m.beta = p.beta;
    m.Gamma0 = p.Gamma0;
    m.sigY = p.sigma_y;
    m.jc = (p.jc_c1 > 0.0 || p.jc_c2 > 0.0) ? 1 : 0;
    m.jc_c1 = p.jc_c1;
    m.jc_c2 = p.jc_c2;
    m.jc_c3 = p.jc_c3;
    m.jc_n = p.jc_n;
    m.jc_m = p.jc_m;
    m.jc_tmelt = p.jc_tmelt;
    m.jc_cv = p.jc_cv;
}

// Derive the per-precision constants from the double parameters; call after
// every change of the grid or of a material.
__host__ inline void finish_params(GridP &g)
{
    fill_consts<double>(g, g.mc_d, g.gc_d);
    fill_consts<float>(g, g.mc_f, g.gc_f);
    g.any_jc = 0;
    for (int l = 0; l < 3; l++) g.any_jc |= g.mat[l].jc;
}

template <class T>
__device__ __forceinline__ const MatC<T> &matc(const GridP &g, int l);
template <>
__device__ __forceinline__ const MatC<double> &matc<double>(const GridP &g, int l) { return g.mc_d[l]; }
template <>
__device__ __forceinline__ const MatC<float> &matc<float>(const GridP &g, int l) { return g.mc_f[l]; }

template <class T>
__device__ __forceinline__ const GridC<T> &gridc(const GridP &g);
template <>
__device__ __forceinline__ const GridC<double> &gridc<double>(const GridP &g) { return g.gc_d; }
template <>
__device__ __forceinline__ const GridC<float> &gridc<float>(const GridP &g) { return g.gc_f; }

// Device-resident control block: time step, time, body state and the error
// word.  Kernels read dt and the body velocity from here so that a whole step
// can be replayed from a CUDA graph without host involvement.
struct Ctl {
    double dt, t, t_end, cfl;
    double smax;              // max_cells sum_d (|u_d|+c)/dx_d of the last reduction
    unsigned long long smax_acc;  // running maximum of the tiles of a stage-3 launch, as
                                  // the bits of a non-negative double (0 between launches)
    double force[3];
    double v[3];
    double x[3];
    double mass;
    int dynamic;
    int auto_dt;              // 1: the finalize kernel sets the next dt from cfl
    unsigned int err;         // bit 0: rho<=0/NaN in an update, bit 1: c^2<=0/NaN
    int steps;
    unsigned int pad;
    float dtf, vf[3];         // dt and v in single precision, kept equal to (float)dt, (float)v
    int rbox_valid;           // 1: rbox bounds every cell with r > 0.5 of the stored state
    int rbox[6];              // inclusive cell-index box lo x, y, z, hi x, y, z (empty: lo > hi)
    int rnext[6];             // the same for the state stage 3 produces (atomic min / max)
};

// Empty box for rnext, and a fresh control block's fields that are not 0.
__host__ __device__ inline void ctl_box_reset(Ctl *c)
{
    for (int d = 0; d < 3; d++) {
        c->rnext[d] = 0x7fffffff;
        c->rnext[3 + d] = -1;
    }
}

// dt and body velocity in the compute precision
template <class T>
__device__ __forceinline__ T ctl_dt(const Ctl *c);
template <>
__device__ __forceinline__ double ctl_dt<double>(const Ctl *c) { return c->dt; }
template <>
__device__ __forceinline__ float ctl_dt<float>(const Ctl *c) { return c->dtf; }
template <class T>
__device__ __forceinline__ T ctl_v(const Ctl *c, int d);
template <>
__device__ __forceinline__ double ctl_v<double>(const Ctl *c, int d) { return c->v[d]; }
template <>
__device__ __forceinline__ float ctl_v<float>(const Ctl *c, int d) { return c->vf[d]; }
// the same read from L2 (bypassing a possibly stale L1 line)
template <class T>
__device__ __forceinline__ T ctl_v_cg(const Ctl *c, int d);
template <>
__device__ __forceinline__ double ctl_v_cg<double>(const Ctl *c, int d) { return __ldcg(&c->v[d]); }
template <>
__device__ __forceinline__ float ctl_v_cg<float>(const Ctl *c, int d) { return __ldcg(&c->vf[d]); }

__device__ __forceinline__ void ctl_set_dt(Ctl *c, double dt)
{
    c->dt = dt;
    c->dtf = (float)dt;
}
__device__ __forceinline__ void ctl_sync_v(Ctl *c)
{
    for (int d = 0; d < 3; d++) c->vf[d] = (float)c->v[d];
}

enum { ERR_STATE = 1u, ERR_SOUND = 2u, ERR_TIMEOUT = 4u };   // ERR_TIMEOUT: a bounded device wait ran out

// Programmatic dependent launch: the kernels of a step are launched with
// launch_pdl, so a kernel's CTAs may be scheduled while the previous kernel
// on the stream is still finishing.  Each such kernel first waits for its
// predecessor to complete with its memory visible (griddepcontrol.wait; a
// no-op without a programmatic predecessor), then lets its own successor be
// scheduled (griddepcontrol.launch_dependents): the successor's CTAs take SM
// slots only after every CTA of this grid has started, and they wait in turn.
__device__ __forceinline__ void pdl_enter()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// The two halves, for a kernel that does work not depending on its
// predecessor before it waits.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
__host__ inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                       cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ------------------------------------------------------------------ layout

template <int DIM, int NMAT, int SOLID>
struct Lay {
    static constexpr int NV = SOLID ? (DIM == 1 ? 3 : (DIM == 2 ? 5 : 9)) : 0;
    static constexpr int IPHI = 0;
    static constexpr int IAR = NMAT - 1;
    static constexpr int IMOM = 2 * NMAT - 1;
    static constexpr int IE = IMOM + DIM;
    static constexpr int IV = IE + 1;
    static constexpr int IR = IV + NV;
    static constexpr int NH = SOLID == 2 ? NMAT : 0;   // plastic-strain planes (phi rho eps)_l
    static constexpr int IH = IR + 1;
    static constexpr int NVAR = IR + 1 + NH;
    static constexpr int NB = SOLID ? DIM : 0;   // V*_{d b} entries kept per face
    static constexpr int NF = NVAR + 1 + NB;     // per-face record: fluxes, u*_d, V*_{d.}
};

// FP32 mixtures of fluids.  Their phasic density (phi rho)_l/phi_l beside an
// interface, where phi_l is some 1e-6, carries the rounding noise of its two
// transported factors magnified (1e-3 of the density at single cells), so
// that any other order of rounding gives another noise; their closures, fluxes
// and reconstruction keep one fixed order of operations, apart from those of
// the other forms.
template <class T, int NMAT, int SOLID>
__host__ __device__ constexpr bool mix32()
{
    return sizeof(T) == 4 && NMAT >= 2 && SOLID == 0;
}

// stored stretch component c -> tensor indices (a, b)
__host__ __device__ constexpr int v_row(int dim, int c)
{
    return dim == 1 ? c : (dim == 2 ? (c < 2 ? 0 : (c < 4 ? 1 : 2)) : c / 3);
}
__host__ __device__ constexpr int v_col(int dim, int c)
{
    return dim == 1 ? c : (dim == 2 ? (c == 0 ? 0 : (c == 1 ? 1 : (c == 2 ? 0 : (c == 3 ? 1 : 2)))) : c % 3);
}

// ------------------------------------------------------------------ math

__device__ __forceinline__ float m_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double m_exp(double x) { return exp(x); }
__device__ __forceinline__ float m_exp(float x) { return expf(x); }
__device__ __forceinline__ double m_sin(double x) { return sin(x); }
// products and sums rounded one by one (never fused into an FMA)
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float m_sin(float x) { return sinf(x); }
__device__ __forceinline__ double m_log(double x) { return log(x); }
__device__ __forceinline__ float m_log(float x) { return logf(x); }
__device__ __forceinline__ double m_pow(double x, double y) { return pow(x, y); }
__device__ __forceinline__ float m_pow(float x, float y) { return powf(x, y); }
__device__ __forceinline__ double m_abs(double x) { return fabs(x); }
__device__ __forceinline__ float m_abs(float x) { return fabsf(x); }
__device__ __forceinline__ double m_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float m_fma(float a, float b, float c) { return fmaf(a, b, c); }

// The FP64 pipe is what bounds the FP64 form (two lanes per SM and clock: an
// FP64 instruction of a warp takes the time of 64 others), so what can be done
// elsewhere is: reciprocals and roots start from the special-function unit's
// approximation and take one third-order step (Chebyshev's iteration: the
// relative error e of the start becomes e^3; e < 2^-19), and comparisons and
// selections work on the bits.

// Conversions between the precisions by integer arithmetic, the same values as
// the conversion instructions, which go through the FP64 pipe: exact to FP64,
// to nearest (ties to even) to FP32.  Subnormals, infinities, NaNs and
// overflows take the instruction (volatile: else it is executed for all and its
// result selected).
__device__ __forceinline__ double m_widen(float x)
{
    const unsigned u = __float_as_uint(x);
    if ((u << 1) == 0u) return __hiloint2double((int)u, 0);
    if ((((u >> 23) + 1u) & 0xffu) <= 1u) {   // exponent 0 or 255
        double r;
        asm volatile("cvt.f64.f32 %0, %1;" : "=d"(r) : "f"(x));
        return r;
    }
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}
__device__ __forceinline__ double m_widen(double x) { return x; }
__device__ __forceinline__ float m_narrow(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
    const unsigned e = (unsigned)(b >> 52);
    if (b == 0ull) return __uint_as_float((unsigned)__double2hiint(x));
    if (e - 897u > 252u) {   // outside the normal range below the last binade
        float r;
        asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(r) : "d"(x));
        return r;
    }
    const unsigned q = (unsigned)(b >> 29), rem = (unsigned)b & 0x1fffffffu;
    const unsigned r = q - 0xc0000000u + ((rem + 0x0fffffffu + (q & 1u)) >> 29);
    return __uint_as_float(r | ((unsigned)__double2hiint(x) & 0x80000000u));
}
// to the storage type
template <class R>
__device__ __forceinline__ R m_store(double x);
template <>
__device__ __forceinline__ double m_store<double>(double x) { return x; }
template <>
__device__ __forceinline__ float m_store<float>(double x) { return m_narrow(x); }

// 1/x: y (1 + e + e^2), e = 1 - x y; to one unit in the last place for
// 2^-1022 <= |x| <= 2^1022.  m_rcp: where the start is 0 or infinite it is the
// result: infinity for 0 and the subnormals (from 2^-1024 on 1/x would still be
// a number, see m_quot), 0 for infinity and |x| > 2^1022.  m_rcp_normal: NaN
// there, for a cell's density and the differences of a face's wave speeds, from
// which a 0 makes no state either way (1-D grids, where few warps wait for each
// other's chains, 2113 us a pass of tube 400 against 2176 with m_rcp).
__device__ __forceinline__ double m_rcp_step(double x, double &y)
{
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double m_rcp_normal(double x)
{
    double y;
    return m_rcp_step(x, y);
}
__device__ __forceinline__ double m_rcp(double x)
{
    double y;
    const double r = m_rcp_step(x, y);
    const bool edge = ((__double2hiint(y) + 0x00100000) & 0x7fe00000) == 0;   // exponent 0 or all ones
    return __longlong_as_double(edge ? __double_as_longlong(y) : __double_as_longlong(r));
}
__device__ __forceinline__ float m_rcp(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float m_rcp_normal(float x) { return m_rcp(x); }

// a/b (FP32: the product with the approximate reciprocal, rounded on its own --
// what the fast division gives over the normal range, without its range fix-up)
__device__ __forceinline__ float m_div(float a, float b) { return __fmul_rn(a, m_rcp(b)); }
__device__ __forceinline__ double m_div(double a, double b) { return a * m_rcp(b); }

// a/b for a b of any size: the partial density of a material that spreads
// through cells it was absent from falls by orders of magnitude a cell, down
// through the subnormals, whose reciprocal overflows
__device__ __forceinline__ double m_quot(double a, double b)
{
    if ((__double2hiint(b) & 0x7fffffff) < 0x00400000) return a / b;   // |b| < 2^-1019
    return m_div(a, b);
}
__device__ __forceinline__ float m_quot(float a, float b) { return m_div(a, b); }

// comparisons on the bits, with those of the ordinary operators: false for a
// NaN, zero of either sign equal to zero
__device__ __forceinline__ unsigned long long m_bits(double x) { return (unsigned long long)__double_as_longlong(x); }
constexpr unsigned long long M_INF = 0x7ff0000000000000ull, M_SIGN = 0x8000000000000000ull;
__device__ __forceinline__ bool m_pos(double x) { return m_bits(x) - 1ull < M_INF; }                  // x > 0
__device__ __forceinline__ bool m_pos(float x) { return x > 0.f; }
__device__ __forceinline__ bool m_neg(double x) { return m_bits(x) - (M_SIGN + 1ull) < M_INF; }       // x < 0
__device__ __forceinline__ bool m_neg(float x) { return x < 0.f; }
__device__ __forceinline__ bool m_ge0(double x) { return m_bits(x) <= M_INF || m_bits(x) == M_SIGN; }  // x >= 0
__device__ __forceinline__ bool m_ge0(float x) { return x >= 0.f; }
__device__ __forceinline__ bool m_zero(double x) { return (m_bits(x) << 1) == 0ull; }                 // x == 0
__device__ __forceinline__ bool m_over1(double x)                                                     // x > 1
{
    return m_bits(x) - 0x3ff0000000000001ull < M_INF - 0x3ff0000000000000ull;
}
__device__ __forceinline__ bool m_over1(float x) { return x > 1.f; }
__device__ __forceinline__ bool m_nan(double x) { return (__double2hiint(x) & 0x7fffffff) >= 0x7ff80000; }  // quiet NaN
__device__ __forceinline__ bool m_nan(float x) { return x != x; }
// whether a < b, neither a NaN; the bits of doubles, negative ones with their magnitude inverted, order like them
__device__ __forceinline__ long long m_key(double x)
{
    const long long k = __double_as_longlong(x);
    return k ^ ((k >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ bool m_less(double a, double b) { return m_key(a) < m_key(b); }
__device__ __forceinline__ bool m_less(float a, float b) { return a < b; }
__device__ __forceinline__ double m_sel(bool c, double a, double b)
{
    return __longlong_as_double(c ? __double_as_longlong(a) : __double_as_longlong(b));
}
__device__ __forceinline__ float m_sel(bool c, float a, float b) { return c ? a : b; }
// minimum and maximum that pass over a NaN, as fmin and fmax do: a state of
// negative c^2 then leaves the wave speeds to the other side of its face
__device__ __forceinline__ double m_min(double a, double b)
{
    return m_sel(m_nan(b) || (!m_nan(a) && m_less(a, b)), a, b);
}
__device__ __forceinline__ float m_min(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double m_max(double a, double b)
{
    return m_sel(m_nan(b) || (!m_nan(a) && m_less(b, a)), a, b);
}
__device__ __forceinline__ float m_max(float a, float b) { return fmaxf(a, b); }

// sqrt(x): x/sqrt(x), the reciprocal root with the third-order step y (1 + e/2 + 3 e^2/8), e = 1 - x y^2;
// to one unit in the last place for every x >= 0
__device__ __forceinline__ double m_sqrt(double x)
{
    if (m_pos(x) && m_less(x, 1e-290)) return sqrt(x);   // the start flushes subnormals to 0
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double c = x * y;
    const double e = fma(-c, y, 1.0);
    const double r = fma(c, e * fma(e, 0.375, 0.5), c);
    return m_sel(m_zero(x) || m_bits(x) == M_INF, x, r);
}

// sqrt(a/b): a / sqrt(a b) with the reciprocal root's start y and its
// third-order step y (1 + e/2 + 3 e^2/8), e = 1 - a b y^2; to two units in the
// last place.  Products outside 2^-959 .. 2^993 (and a = 0) take the quotient.
__device__ __forceinline__ double m_sqrt_ratio(double a, double b)
{
    const double x = a * b;
    if ((unsigned)(__double2hiint(x) & 0x7fffffff) - 0x04000000u >= 0x7a000000u) return m_sqrt(m_div(a, b));
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-(x * y), y, 1.0);
    const double c = a * y;
    return fma(c, e * fma(e, 0.375, 0.5), c);
}
__device__ __forceinline__ float m_sqrt_ratio(float a, float b) { return sqrtf(a * m_rcp(b)); }

// x^n for a whole number n = 1..8
template <class T>
__device__ __forceinline__ T m_whole_pow(T x, int n)
{
    const T x2 = x * x, x4 = x2 * x2;
    T r = n & 1 ? x : T(1);
    if (n & 2) r *= x2;
    if (n & 4) r *= x4;
    if (n & 8) r *= x4 * x4;
    return r;
}

__device__ __forceinline__ int map_idx(int i, int n, int periodic)
{
    if (periodic) {
        int m = i % n;
        return m < 0 ? m + n : m;
    }
    return i < 0 ? 0 : (i > n - 1 ? n - 1 : i);
}

// Halo index of direction d with reflective walls: a wall side mirrors (cell
// -1-i below, 2n-1-i above, clamped into the grid when n < 3); *flip is set
// when the cell is a mirror image.
__device__ __forceinline__ int halo_idx(const GridP &g, int d, int i, bool *flip)
{
    const int n = g.n[d];
    if ((i < 0 && g.wall[d][0]) || (i > n - 1 && g.wall[d][1])) {
        *flip = true;
        const int m = i < 0 ? -1 - i : 2 * n - 1 - i;
        return m < 0 ? 0 : (m > n - 1 ? n - 1 : m);
    }
    return map_idx(i, n, g.periodic[d]);
}

// ------------------------------------------------------ material closure

template <class T>
struct Ref {
    T re, pref, rdp, G;   // rho e_ref, p_ref, rho dp_ref/drho, shear modulus
};

// Mie-Grueneisen reference curves p = p_ref + rho Gamma (e - e_ref) of one
// material (Sec. 2.1.2-2.1.3): ideal gas (p_ref = e_ref = 0), stiffened gas
// (e_ref = 0, p_ref = -gamma p_inf), Romenskii solid (eq:Romenskii, cold term
// K0/(2 rho alpha^2)(x^alpha - 1)^2 as printed, shear energy G J^2/rho with
// G = G0 x^(beta+1), x = rho/rho0, and p_ref = rho^2 de_ref/drho).  Written
// for rho e_ref and rho dp_ref/drho, which need no division.  The two powers
// share one logarithm, and take products where the exponents are whole
// numbers (copper: 1 and 4); at rho = rho0, where every absent solid is set,
// both are 1.
template <class T>
__device__ __forceinline__ Ref<T> mat_ref(const MatC<T> &m, T rho, T J2)
{
    Ref<T> r;
    if (m.kind == 2) {
        T xa = T(1), xg = T(1);
        if (rho != m.rho0) {
            const T x = rho * m.irho0;
            const T lx = (m.n_alpha && m.n_beta1) ? T(0) : m_log(x);
            xa = m.n_alpha ? m_whole_pow(x, m.n_alpha) : m_exp(m.alpha * lx);
            xg = m.n_beta1 ? m_whole_pow(x, m.n_beta1) : m_exp(m.beta1 * lx);
        }
        const T xm1 = add_rn(xa, T(-1));
        const T rc = mul_rn(mul_rn(m.kE, xm1), xm1);          // rho e_c
        r.G = mul_rn(m.G0, xg);
        const T GJ = mul_rn(r.G, J2);
        r.re = add_rn(rc, GJ);
        r.pref = m_fma(m.beta, GJ, m_fma(mul_rn(m.kP, xm1), xa, -rc));
        r.rdp = m_fma(mul_rn(m.K0, xa), m_fma(-m.ialpha, xm1, m_fma(T(2), xa, T(-1))), mul_rn(m.bb, GJ));
    } else {
        r.re = T(0);
        r.pref = m.pref0;
        r.rdp = T(0);
        r.G = T(0);
    }
    return r;
}

// ------------------------------------------------------ stretch tensor

// artanh(z)/z of z^2 (>= 0): its series to 2^-53 (FP64) or 2^-24 (FP32) below
// z^2 = 0.01, the closed form above.  An elastic metal's stretches differ by
// the yield strain, some 0.1 to 1 %, so its cells take the series; a gas may
// shear without limit.
__device__ __forceinline__ double artanh_ratio(double z2)
{
    if (m_less(z2, 0.01)) {
        double s = 1.0 / 17.0;
        s = fma(s, z2, 1.0 / 15.0);
        s = fma(s, z2, 1.0 / 13.0);
        s = fma(s, z2, 1.0 / 11.0);
        s = fma(s, z2, 1.0 / 9.0);
        s = fma(s, z2, 1.0 / 7.0);
        s = fma(s, z2, 1.0 / 5.0);
        s = fma(s, z2, 1.0 / 3.0);
        return fma(s, z2, 1.0);
    }
    const double z = sqrt(z2);
    return 0.5 * log((1.0 + z) / (1.0 - z)) / z;
}
__device__ __forceinline__ float artanh_ratio(float z2)
{
    if (z2 < 0.01f) {
        float s = 1.f / 9.f;
        s = fmaf(s, z2, 1.f / 7.f);
        s = fmaf(s, z2, 1.f / 5.f);
        s = fmaf(s, z2, 1.f / 3.f);
        return fmaf(s, z2, 1.f);
    }
    const float z = sqrtf(z2);
    return 0.5f * logf((1.f + z) / (1.f - z)) / z;
}

// The logarithm of the stretch, dev(H) = dev ln V with V^2 = A A^T (Sec.
// 2.1.2), in 2-D, where A A^T = B is block diagonal, and 1-D, where it is
// diagonal.  The in-plane block's log-stretches are mean +- k/2 about a mean
// that, made traceless, is -d2/2, with
//   d2 = (1/3) ln(A_zz^2/|det A_2|) = (2/3) artanh(s), s = (A_zz^2 - |det A_2|)/(A_zz^2 + |det A_2|),
//   k = artanh(z), z = |(half, b01)|/mid of B's mean and deviator,
// so that in place of three logarithms, a root and two divisions there are
// two values of artanh(z)/z, an even function; k c_2 and k s_2 (2 theta the
// doubled angle of the eigenvectors) are then q half and q b01 with
// q = artanh(z)/(z mid).
template <class T>
struct StretchLog {
    T d2, q, half, b01;   // see above (2-D); 1-D: dev log-stretches d0 = half, d1 = b01, d2
    T k2, J2;             // k^2; |dev H|^2
};

template <class T, int DIM>
__device__ __forceinline__ void stretch_log(const T A[3][3], StretchLog<T> &e)
{
    if (DIM == 1) {
        const T h0 = m_log(m_abs(A[0][0])), h1 = m_log(m_abs(A[1][1])), h2 = m_log(m_abs(A[2][2]));
        const T hm = (h0 + h1 + h2) * (T(1) / T(3));
        e.half = h0 - hm;
        e.b01 = h1 - hm;
        e.d2 = h2 - hm;
        e.q = e.k2 = T(0);
        e.J2 = e.half * e.half + e.b01 * e.b01 + e.d2 * e.d2;
    } else {
        const T b00 = m_fma(A[0][0], A[0][0], mul_rn(A[0][1], A[0][1]));
        const T b11 = m_fma(A[1][1], A[1][1], mul_rn(A[1][0], A[1][0]));
        e.b01 = m_fma(A[0][0], A[1][0], mul_rn(A[0][1], A[1][1]));
        e.half = T(0.5) * (b00 - b11);
        const T imid = m_rcp(T(0.5) * (b00 + b11));
        const T det = m_abs(m_fma(A[0][0], A[1][1], -mul_rn(A[0][1], A[1][0]))), zz = mul_rn(A[2][2], A[2][2]);
        const T s = mul_rn(zz - det, m_rcp(add_rn(zz, det)));
        const T h = e.half * imid, b = e.b01 * imid, z2 = m_fma(h, h, mul_rn(b, b));
        const T F = artanh_ratio(z2);
        e.d2 = mul_rn(mul_rn(T(2) / T(3), s), artanh_ratio(s * s));
        e.q = mul_rn(F, imid);
        e.k2 = mul_rn(mul_rn(z2, F), F);
        e.J2 = m_fma(mul_rn(T(1.5), e.d2), e.d2, mul_rn(T(0.5), e.k2));
    }
}

// dev(H), in-plane block (and the other entries a closure reads)
template <class T, int DIM>
__device__ __forceinline__ void stretch_dev(const StretchLog<T> &e, T H[DIM][DIM])
{
    if constexpr (DIM == 1) {
        H[0][0] = e.half;
    } else {
        const T qh = T(0.5) * e.q, m = T(-0.5) * e.d2;
#pragma unroll
        for (int a = 0; a < DIM; a++)
#pragma unroll
            for (int b = 0; b < DIM; b++) H[a][b] = T(0);
        H[0][0] = m_fma(qh, e.half, m);
        H[1][1] = m_fma(-qh, e.half, m);
        H[0][1] = H[1][0] = qh * e.b01;
    }
}

// ------------------------------------------------------------- thermo

// Closure weight of a transported volume fraction: clipped to [0, 1].
template <class T>
__device__ __forceinline__ T phi_clip(T f)
{
    return m_sel(m_neg(f), T(0), m_sel(m_over1(f), T(1), f));
}

// Phasic density (phi rho)_l / phi_l (Sec. 2.2); a material whose clipped
// fraction is below 1e-6 is absent from the cell and takes its reference
// density rho0 (when one is given) -- the ratio of two round-off-sized numbers
// would otherwise set the pressure through a stiff cold curve.
template <class T>
__device__ __forceinline__ T phasic_density(const GridP &g, int l, T ar, T phc)
{
    const MatC<T> &m = matc<T>(g, l);
    if (m_less(phc, T(1e-6)) && m.has_rho0) return m.rho0;
    const T guard = gridc<T>(g).phi_guard;
    const T f = m_less(guard, phc) ? phc : guard;
    return m_div(ar, f);
}

// Mixture sums over the materials at phasic densities rhol (Sec. 2.2), all
// with the weights phi_l/Gamma_l: den = sum of the weights, Q such that
// rho e = p den - Q, Yn = rho c^2 den (one material: rho c^2), and the sums
// of G and sigma_Y.
template <class T, int NMAT>
struct Mix {
    T phi[NMAT], ar[NMAT];
    T rho, den, Q, Yn, Gn, Sn;
};

template <class T, int NMAT, int SOLID>
__device__ __forceinline__ void mix_sums(const GridP &g, const T *phi, const T *rhol, T p, T J2, Mix<T, NMAT> &x)
{
    T fsum = T(0);
#pragma unroll
    for (int l = 0; l < NMAT - 1; l++) {
        x.phi[l] = phi[l];
        fsum += phi[l];
    }
    x.phi[NMAT - 1] = T(1) - fsum;
    x.rho = x.den = x.Q = x.Yn = x.Gn = x.Sn = T(0);
#pragma unroll
    for (int l = 0; l < NMAT; l++) {
        const MatC<T> &m = matc<T>(g, l);
        const T f = NMAT == 1 ? T(1) : phi_clip(x.phi[l]);
        x.phi[l] = f;
        x.ar[l] = NMAT == 1 ? rhol[l] : mul_rn(f, rhol[l]);
        x.rho = l == 0 ? x.ar[0] : add_rn(x.rho, x.ar[l]);
        const T w = mul_rn(f, m.invGam);
        x.den = l == 0 ? w : add_rn(x.den, w);
        // a material without mass has no reference energy and no part in the sound speed
        const bool mass = x.ar[l] != T(0);
        if (m.kind == 2) {
            const Ref<T> r = mat_ref<T>(m, rhol[l], J2);
            x.Q = m_fma(w, r.pref, m_fma(-(mass ? f : T(0)), r.re, x.Q));
            // (Gam + 1)(p - p_ref) + rho dp_ref/drho + 4/3 G   (rho^2 de_ref/drho = p_ref)
            const T y = m_fma(m.kA, p - r.pref, mul_rn(m.invGam, m_fma(T(4) / T(3), r.G, r.rdp)));
            if (NMAT == 1) x.Yn = mul_rn(y, m.Gam);
            else if (mass) x.Yn = m_fma(f, y, x.Yn);
            x.Gn = m_fma(w, r.G, x.Gn);
            x.Sn = m_fma(w, m.sigY, x.Sn);
        } else {
            x.Q = m_fma(f, m.kB, x.Q);
            if (NMAT == 1) {
                x.Yn = m_fma(p, m.Gam1, -m.pref0);
            } else {
                const T y = m_fma(p, m.kA, -m.kB);   // (Gam p + p - p_ref)/Gam
                if (mass) x.Yn = m_fma(f, y, x.Yn);
            }
        }
    }
}

template <class T, int DIM, int NMAT, int SOLID>
struct State {
    T phi[NMAT], ar[NMAT];
    T rho, u[DIM], p, c;   // c: sound speed
    T den, Q;              // rho E = p den - Q + rho |u|^2/2
    T c2, rhoE;            // FP32 fluid mixtures: c^2 and rho E in place of c, den, Q
    T G, sigY;
    T H[DIM][DIM];     // dev(H), in-plane block
    T eps[NMAT];       // equivalent plastic strain (SOLID == 2)
};

template <class T, int DIM, int NMAT, int SOLID>
__device__ __forceinline__ void unpack_A_ct(const T *w, T A[3][3])
{
    using L = Lay<DIM, NMAT, SOLID>;
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) A[a][b] = T(0);
#pragma unroll
    for (int c = 0; c < L::NV; c++) A[v_row(DIM, c)][v_col(DIM, c)] = w[L::IV + c];
}

template <class T, int DIM, int NMAT, int SOLID>
__device__ __forceinline__ void unpack_A(const T *w, double A[3][3])
{
    using L = Lay<DIM, NMAT, SOLID>;
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) A[a][b] = 0.0;
#pragma unroll
    for (int c = 0; c < L::NV; c++) A[v_row(DIM, c)][v_col(DIM, c)] = m_widen(w[L::IV + c]);
}

// The closure of the FP32 fluid mixtures: the same rules, material by material.
template <class T, int DIM, int NMAT>
__device__ __forceinline__ void mix32_state(const GridP &g, const T *w, State<T, DIM, NMAT, 0> &s)
{
    using L = Lay<DIM, NMAT, 0>;
    T fsum = T(0);
#pragma unroll
    for (int l = 0; l < NMAT - 1; l++) {
        s.phi[l] = w[L::IPHI + l];
        fsum += s.phi[l];
    }
    s.phi[NMAT - 1] = T(1) - fsum;
    T rhol[NMAT];
    s.rho = T(0);
#pragma unroll
    for (int l = 0; l < NMAT; l++) {
        s.phi[l] = phi_clip(s.phi[l]);
        rhol[l] = w[L::IAR + l];
        s.ar[l] = s.phi[l] * rhol[l];
        s.rho += s.ar[l];
    }
#pragma unroll
    for (int a = 0; a < DIM; a++) s.u[a] = w[L::IMOM + a];
    s.p = w[L::IE];
    T rhoe = T(0), den = T(0), Yn = T(0);
#pragma unroll
    for (int l = 0; l < NMAT; l++) {
        const MatC<T> &m = matc<T>(g, l);
        const T iG = m.invGam;
        const T irl = m_rcp(rhol[l]);
        if (m.kind == 2) {
            // a solid's equation of state in a fluid run (no stretch: J^2 = 0)
            const Ref<T> r = mat_ref<T>(m, rhol[l], T(0));
            if (s.ar[l] != T(0)) rhoe += s.ar[l] * (r.re * irl);
            rhoe += s.phi[l] * (s.p - r.pref) * iG;
            den += s.phi[l] * iG;
            const T c2l = ((m.Gam + T(1)) * (s.p - r.pref) + r.rdp + T(4) / T(3) * r.G) * irl;
            if (s.ar[l] != T(0)) Yn += s.ar[l] * c2l * iG;
            continue;
        }
        rhoe += s.phi[l] * (s.p - m.pref0) * iG;
        den += s.phi[l] * iG;
        const T c2l = (m.Gam * s.p + (s.p - m.pref0)) * irl;
        if (s.ar[l] != T(0)) Yn += s.ar[l] * c2l * iG;
    }
    T ke = T(0);
#pragma unroll
    for (int a = 0; a < DIM; a++) ke += T(0.5) * s.rho * s.u[a] * s.u[a];
    const T iden = m_rcp(den);
    s.rhoE = rhoe + ke;
    s.c2 = m_div(Yn, s.rho) * iden;
    s.c = m_sqrt(s.c2);
    s.G = s.sigY = T(0);
}

// Full state from primitives w (mixture rules of Sec. 2.2): rho = sum phi_l rho_l,
// rho e = sum [ (phi rho)_l e_ref,l + phi_l (p - p_ref,l)/Gamma_l ],
// G = sum(phi_l G_l/Gamma_l)/sum(phi_l/Gamma_l) (sigma_Y with the same weights),
// c^2 = sum(Y_l c_l^2/Gamma_l)/sum(phi_l/Gamma_l) with c_l^2 = a_l^2 + 4/3 G_l/rho_l.
template <class T, int DIM, int NMAT, int SOLID>
__device__ __forceinline__ void state_from_prim_ct(const GridP &g, const T *w, State<T, DIM, NMAT, SOLID> &s)
{
    using L = Lay<DIM, NMAT, SOLID>;
#pragma unroll
    for (int l = 0; l < NMAT; l++) s.eps[l] = T(0);
    if constexpr (mix32<T, NMAT, SOLID>()) {
        mix32_state<T, DIM, NMAT>(g, w, s);
        return;
    }
#pragma unroll
    for (int a = 0; a < DIM; a++) s.u[a] = w[L::IMOM + a];
    s.p = w[L::IE];
    if constexpr (SOLID == 2) {
#pragma unroll
        for (int l = 0; l < NMAT; l++) s.eps[l] = w[L::IH + l];
    }
    T J2 = T(0);
    if (SOLID) {
        T A[3][3];
        StretchLog<T> e;
        unpack_A_ct<T, DIM, NMAT, SOLID>(w, A);
        stretch_log<T, DIM>(A, e);
        stretch_dev<T, DIM>(e, s.H);
        J2 = e.J2;
    }
    Mix<T, NMAT> x;
    mix_sums<T, NMAT, SOLID>(g, w + L::IPHI, w + L::IAR, s.p, J2, x);
#pragma unroll
    for (int l = 0; l < NMAT; l++) {
        s.phi[l] = x.phi[l];
        s.ar[l] = x.ar[l];
    }
    s.rho = x.rho;
    s.den = x.den;
    s.Q = x.Q;
    s.c = m_sqrt_ratio(x.Yn, NMAT == 1 ? x.rho : mul_rn(x.rho, x.den));
    s.G = s.sigY = T(0);
    if (SOLID) {
        const T iden = m_rcp(x.den);
        s.G = mul_rn(x.Gn, iden);
        s.sigY = mul_rn(x.Sn, iden);
    }
}

// rho E of a state
template <class T, int DIM, int NMAT, int SOLID>
__device__ __forceinline__ T state_energy(const State<T, DIM, NMAT, SOLID> &s)
{
    if (mix32<T, NMAT, SOLID>()) return s.rhoE;
    T uu = T(0);
#pragma unroll
    for (int a = 0; a < DIM; a++) uu = m_fma(s.u[a], s.u[a], uu);
    return m_fma(T(0.5) * s.rho, uu, m_fma(s.p, s.den, -s.Q));
}

// The FP32 form's precision rule: the closure of a mixed cell -- at least two
// materials present (fraction >= 1e-6) -- in which another material's fraction
// is below 1e-6 runs in FP64.  A material below 1e-6 is absent (it takes its
// reference density, reading of Sec. 2.2), so with two materials such a cell
// does not exist; the rule acts from three materials on.
template <class T, int NMAT>
__device__ __forceinline__ bool needs_fp64(const T *phi_first)
{
    if (NMAT < 3) return false;
    T fsum = T(0), mn = T(1);
    int present = 0;
#pragma unroll
    for (int l = 0; l < NMAT - 1; l++) {
        mn = m_min(mn, phi_first[l]);
        fsum += phi_first[l];
        present += phi_first[l] >= T(1e-6);
    }
    const T last = T(1) - fsum;
    mn = m_min(mn, last);
    present += last >= T(1e-6);
    return present >= 2 && mn < T(1e-6);
}

template <class T, int NMAT>
__device__ __forceinline__ bool fp64_closure(const T *phi_first)
{
    return sizeof(T) == 4 && needs_fp64<T, NMAT>(phi_first);
}

// State from primitives in the compute type T; the FP32 form switches to FP64
// for cells whose smallest volume fraction is below 1e-6.
template <class T, int DIM, int NMAT, int SOLID>
__device__ __forceinline__ void state_from_prim(const GridP &g, const T *w, State<T, DIM, NMAT, SOLID> &s)
{
    using L = Lay<DIM, NMAT, SOLID>;
    if (sizeof(T) == 4 && needs_fp64<T, NMAT>(w + L::IPHI)) {
        double wd[L::NVAR];
#pragma unroll
        for (int v = 0; v < L::NVAR; v++) wd[v] = (double)w[v];
        State<double, DIM, NMAT, SOLID> sd;
        state_from_prim_ct<double, DIM, NMAT, SOLID>(g, wd, sd);
#pragma unroll
        for (int l = 0; l < NMAT; l++) {
            s.phi[l] = (T)sd.phi[l];
            s.ar[l] = (T)sd.ar[l];
        }
        s.rho = (T)sd.rho;
#pragma unroll
        for (int a = 0; a < DIM; a++) s.u[a] = (T)sd.u[a];
        s.p = (T)sd.p;
        s.c = (T)sd.c;
        s.den = (T)sd.den;
        s.Q = (T)sd.Q;
        s.c2 = (T)(sd.c * sd.c);
        s.rhoE = (T)state_energy<double, DIM, NMAT, SOLID>(sd);
        s.G = (T)sd.G;
        s.sigY = (T)sd.sigY;
#pragma unroll
        for (int l = 0; l < NMAT; l++) s.eps[l] = (T)sd.eps[l];
        if (SOLID) {
#pragma unroll
            for (int a = 0; a < DIM; a++)
#pragma unroll
                for (int b = 0; b < DIM; b++) s.H[a][b] = (T)sd.H[a][b];
        }
        return;
    }
    state_from_prim_ct<T, DIM, NMAT, SOLID>(g, w, s);
}

// Conserved -> primitive (Sec. 2.2): rho_l = (phi rho)_l / max(phi_l, guard),
// u = (rho u)/rho and the mixture pressure
// p = (rho E - rho|u|^2/2 - sum[(phi rho)_l e_ref,l - phi_l p_ref,l/Gamma_l]) / sum phi_l/Gamma_l.
template <class T, int DIM, int NMAT, int SOLID>
__device__ __forceinline__ void cons_to_prim_ct(const GridP &g, const T *q, T *w)
{
    using L = Lay<DIM, NMAT, SOLID>;
    T phi[NMAT], ar[NMAT], rho = T(0), fsum = T(0);
#pragma unroll
    for (int l = 0; l < NMAT - 1; l++) {
        phi[l] = q[L::IPHI + l];
        fsum += phi[l];
    }
    phi[NMAT - 1] = T(1) - fsum;
#pragma unroll
    for (int l = 0; l < NMAT; l++) {
        ar[l] = q[L::IAR + l];
        rho += ar[l];
    }
    if constexpr (mix32<T, NMAT, SOLID>()) {
        T u[DIM];
        const T irho = m_rcp(rho);
#pragma unroll
        for (int a = 0; a < DIM; a++) u[a] = q[L::IMOM + a] * irho;
        T ke = T(0);
#pragma unroll
        for (int a = 0; a < DIM; a++) ke += T(0.5) * rho * u[a] * u[a];
        T num = q[L::IE] - ke, den = T(0);
        T rhol[NMAT];
#pragma unroll
        for (int l = 0; l < NMAT; l++) {
            const T phc = phi_clip(phi[l]);
            rhol[l] = phasic_density<T>(g, l, ar[l], phc);
            const MatC<T> &m = matc<T>(g, l);
            T pref = m.pref0;
            if (m.kind == 2) {
                const Ref<T> r = mat_ref<T>(m, rhol[l], T(0));
                pref = r.pref;
                if (ar[l] != T(0)) num -= ar[l] * m_div(r.re, rhol[l]);
            }
            num += phc * pref * m.invGam;
            den += phc * m.invGam;
        }
#pragma unroll
        for (int l = 0; l < NMAT - 1; l++) w[L::IPHI + l] = phi[l];
#pragma unroll
        for (int l = 0; l < NMAT; l++) w[L::IAR + l] = rhol[l];
#pragma unroll
        for (int a = 0; a < DIM; a++) w[L::IMOM + a] = u[a];
        w[L::IE] = m_div(num, den);
        w[L::IR] = q[L::IR];
        return;
    }
    T u[DIM], mu = T(0);
    const T irho = m_rcp_normal(rho);
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        u[a] = q[L::IMOM + a] * irho;
        mu = m_fma(q[L::IMOM + a], u[a], mu);
    }
    T J2 = T(0);
    if (SOLID) {
        T A[3][3];
        StretchLog<T> e;
        unpack_A_ct<T, DIM, NMAT, SOLID>(q, A);
        stretch_log<T, DIM>(A, e);
        J2 = e.J2;
    }
    T num = m_fma(T(-0.5), mu, q[L::IE]), den = T(0);
    T rhol[NMAT];
    if constexpr (NMAT == 1) {
        // p = p_ref + Gamma (rho e - rho e_ref)   (eq:MieGruneisenEOS)
        const MatC<T> &m = matc<T>(g, 0);
        rhol[0] = rho;
        if (m.kind == 2) {
            const Ref<T> r = mat_ref<T>(m, rho, J2);
            w[L::IE] = m_fma(m.Gam, num - r.re, r.pref);
        } else {
            w[L::IE] = m_fma(m.Gam, num, m.pref0);
        }
    } else {
#pragma unroll
        for (int l = 0; l < NMAT; l++) {
            const T f = phi_clip(phi[l]);
            rhol[l] = phasic_density<T>(g, l, ar[l], f);
            const MatC<T> &m = matc<T>(g, l);
            if (m.kind == 2) {
                // (phi rho) e_ref is phi (rho e_ref), and for an absent material at rho0 its mass over rho0
                const Ref<T> r = mat_ref<T>(m, rhol[l], J2);
                num -= (m_less(f, T(1e-6)) ? ar[l] * m.irho0 : f) * r.re;
                num += f * m.invGam * r.pref;
            } else {
                num = m_fma(f, m.kB, num);
            }
            den = m_fma(f, m.invGam, den);
        }
        w[L::IE] = num * m_rcp(den);
    }
#pragma unroll
    for (int l = 0; l < NMAT - 1; l++) w[L::IPHI + l] = phi[l];
#pragma unroll
    for (int l = 0; l < NMAT; l++) w[L::IAR + l] = rhol[l];
#pragma unroll
    for (int a = 0; a < DIM; a++) w[L::IMOM + a] = u[a];
#pragma unroll
    for (int c = 0; c < L::NV; c++) w[L::IV + c] = q[L::IV + c];
    w[L::IR] = q[L::IR];
    // history: specific eps_l = (phi rho eps)_l / (phi rho)_l, 0 without mass
    if constexpr (SOLID == 2) {
#pragma unroll
        for (int l = 0; l < NMAT; l++) w[L::IH + l] = ar[l] != T(0) ? m_quot(q[L::IH + l], ar[l]) : T(0);
    }
}

// Wave speed sum_d (|u_d| + c)/dx_d of one gas cell from its conserved values
// (FP32; momenta q[1..DIM]); every operation rounded as written, so that
// the stage kernels and the standalone reduction agree to the bit.  c2: c^2.
template <int DIM>
__device__ __forceinline__ float gas_speed(float Gam, float pref0, const float *q, const float *inv_dx, float &c2)
{
    const float ir = m_rcp(q[0]), hr = __fmul_rn(0.5f, q[0]);
    float u[DIM], ke = 0.f;
#pragma unroll
    for (int d = 0; d < DIM; d++) {
        u[d] = __fmul_rn(q[1 + d], ir);
        const float h = __fmul_rn(hr, u[d]);
        ke = d == 0 ? __fmul_rn(h, u[d]) : fmaf(h, u[d], ke);
    }
    const float p = fmaf(Gam, __fadd_rn(q[1 + DIM], -ke), pref0);
    c2 = __fmul_rn(fmaf(Gam, p, __fadd_rn(p, -pref0)), ir);
    const float c = sqrtf(c2);
    float s = __fmul_rn(__fadd_rn(fabsf(u[DIM - 1]), c), inv_dx[DIM - 1]);
#pragma unroll
    for (int d = DIM - 2; d >= 0; d--) s = fmaf(__fadd_rn(fabsf(u[d]), c), inv_dx[d], s);
    return s;
}

template <class T, int DIM, int NMAT, int SOLID>
__device__ __forceinline__ void cons_to_prim(const GridP &g, const T *q, T *w)
{
    using L = Lay<DIM, NMAT, SOLID>;
    if (sizeof(T) == 4 && needs_fp64<T, NMAT>(q + L::IPHI)) {
        double qd[L::NVAR], wd[L::NVAR];
#pragma unroll
        for (int v = 0; v < L::NVAR; v++) qd[v] = (double)q[v];
        cons_to_prim_ct<double, DIM, NMAT, SOLID>(g, qd, wd);
#pragma unroll
        for (int v = 0; v < L::NVAR; v++) w[v] = (T)wd[v];
        return;
    }
    cons_to_prim_ct<T, DIM, NMAT, SOLID>(g, q, w);
}

// Wave speed sum_d (|u_d| + c)/dx_d of a cell from its conserved values; c: its
// sound speed or its square (not positive where c^2 <= 0).
template <class T, int DIM, int NMAT, int SOLID>
__device__ __forceinline__ T cell_speed(const GridP &g, const T *q, T &c)
{
    using L = Lay<DIM, NMAT, SOLID>;
    if constexpr (sizeof(T) == 4 && NMAT == 1 && SOLID == 0) {
        if (g.mc_f[0].kind != 2) {
            float c2;
            const T s = gas_speed<DIM>(g.mc_f[0].Gam, g.mc_f[0].pref0, q + L::IAR, g.gc_f.inv_dx, c2);
            c = c2;
            return s;
        }
    }
    T w[L::NVAR];
    cons_to_prim<T, DIM, NMAT, SOLID>(g, q, w);
    State<T, DIM, NMAT, SOLID> s;
    state_from_prim<T, DIM, NMAT, SOLID>(g, w, s);
    T sum = T(0);
#pragma unroll
    for (int d = 0; d < DIM; d++)
        sum += mix32<T, NMAT, SOLID>() ? (m_abs(s.u[d]) + s.c) / gridc<T>(g).dx[d]
                                       : (m_abs(s.u[d]) + s.c) * gridc<T>(g).inv_dx[d];
    c = s.c;
    return sum;
}

template <class T, int DIM, int NMAT, int SOLID>
__device__ __forceinline__ void prim_to_cons(const GridP &g, const T *w, T *q)
{
    using L = Lay<DIM, NMAT, SOLID>;
    State<T, DIM, NMAT, SOLID> s;
    state_from_prim<T, DIM, NMAT, SOLID>(g, w, s);
#pragma unroll
    for (int l = 0; l < NMAT - 1; l++) q[L::IPHI + l] = s.phi[l];
#pragma unroll
    for (int l = 0; l < NMAT; l++) q[L::IAR + l] = s.ar[l];
#pragma unroll
    for (int a = 0; a < DIM; a++) q[L::IMOM + a] = s.rho * s.u[a];
    q[L::IE] = state_energy<T, DIM, NMAT, SOLID>(s);
#pragma unroll
    for (int c = 0; c < L::NV; c++) q[L::IV + c] = w[L::IV + c];
    q[L::IR] = w[L::IR];
    if constexpr (SOLID == 2) {
#pragma unroll
        for (int l = 0; l < NMAT; l++) q[L::IH + l] = s.ar[l] * s.eps[l];
    }
}

// ------------------------------------------------------- reconstruction

// The slope, THINC and reconstruction of the FP32 fluid mixtures, and of
// the volume fractions and r of every FP32 form (recon_cell below says what
// they do), in one fixed order of operations: where MUSCL's and THINC's
// boundary variations agree to round-off, the choice between them, and with it
// the face value, would otherwise change with the order of rounding.
template <class T>
__device__ __forceinline__ T vanleer(T a, T b)
{
    return (a * b <= T(0)) ? T(0) : m_div(T(2) * a * b, a + b);
}

template <class T>
__device__ __forceinline__ bool mix32_thinc(const GridP &g, T qm, T q0, T qp, T &fm, T &fp)
{
    if ((qp - q0) * (q0 - qm) <= T(0)) return false;
    const T qmin = m_min(qm, qp), qmax = m_max(qm, qp);
    const T dq = qmax - qmin;
    const T th = (qp - qm) >= T(0) ? T(1) : T(-1);
    const T C = (q0 - qmin) / dq;
    if (!(C > T(1e-8) && C < T(1) - T(1e-8))) return false;
    const GridC<T> &gc = gridc<T>(g);
    const T B = m_exp(th * gc.beta * (T(2) * C - T(1)));
    const T ty = (gc.cosh_b - B) * gc.inv_sinh_b;
    const T tb = gc.tanh_b;
    const T t1 = (tb - ty) / (T(1) - tb * ty);
    fm = qmin + T(0.5) * dq * (T(1) - th * ty);
    fp = qmin + T(0.5) * dq * (T(1) + th * t1);
    return true;
}

// face values lo (towards i-1) and hi (towards i+1) of cell i, s[0..4] = q_{i-2} .. q_{i+2}
template <class T>
__device__ __forceinline__ void mix32_recon_cell(const GridP &g, const T *s, bool frac, T &lo, T &hi)
{
    const T slB = vanleer(s[2] - s[1], s[3] - s[2]);
    const T Bm = s[2] - T(0.5) * slB, Bp = s[2] + T(0.5) * slB;
    lo = Bm;
    hi = Bp;
    if (!frac || !g.use_thinc) return;
    const T slA = vanleer(s[1] - s[0], s[2] - s[1]);
    const T slC = vanleer(s[3] - s[2], s[4] - s[3]);
    const T Ap = s[1] + T(0.5) * slA, Cm = s[3] - T(0.5) * slC;
    T tAm = s[1] - T(0.5) * slA, tAp = Ap, tBm = Bm, tBp = Bp, tCm = Cm, tCp = s[3] + T(0.5) * slC;
    if (!mix32_thinc<T>(g, s[1], s[2], s[3], tBm, tBp)) return;   // MUSCL's values either way
    mix32_thinc<T>(g, s[0], s[1], s[2], tAm, tAp);
    mix32_thinc<T>(g, s[2], s[3], s[4], tCm, tCp);
    const T tbvBM = m_abs(Ap - Bm) + m_abs(Bp - Cm);
    const T tbvBT = m_abs(tAp - tBm) + m_abs(tBp - tCm);
    if (tbvBT < tbvBM) {
        lo = tBm;
        hi = tBp;
    }
}

// half the van Leer slope 2ab/(a+b) of a cell from its backward and forward
// differences.  (Here and in the closures the products and sums are rounded as
// written, fused only where fma says so: the two sides of a wall face, mirror
// images, then go through the same roundings and S* there is exactly 0.)
template <class T>
__device__ __forceinline__ T half_slope(T a, T b)
{
    const T ab = a * b;
    return m_pos(ab) ? mul_rn(ab, m_rcp(a + b)) : T(0);
}

// THINC face values of a cell (Sec. 3.1, MUSCL-BVD-THINC): the tanh profile
// q_min + dq/2 (1 + theta tanh(beta (x - x_c))) on [0,1] whose cell average is
// q0 has tanh(beta x_c) = (cosh beta - exp(theta beta (2C-1)))/sinh beta with
// C = (q0 - q_min)/dq; its end values are returned.  Only monotone cells with
// 1e-8 < C < 1 - 1e-8.
template <class T>
__device__ __forceinline__ bool thinc(const GridP &g, T qm, T q0, T qp, T &fm, T &fp)
{
    if (!m_pos((qp - q0) * (q0 - qm))) return false;
    const bool up = !m_less(qp, qm);
    const T qmin = m_sel(up, qm, qp);
    const T d = qp - qm, dq = m_abs(d);
    const T C = (q0 - qmin) * m_rcp(dq);
    if (!(m_less(T(1e-8), C) && m_less(C, T(1) - T(1e-8)))) return false;
    const GridC<T> &gc = gridc<T>(g);
    const T th = m_sel(up, T(1), T(-1));
    const T B = m_exp(th * gc.beta * (T(2) * C - T(1)));
    const T ty = (gc.cosh_b - B) * gc.inv_sinh_b;
    const T tb = gc.tanh_b;
    const T t1 = (tb - ty) * m_rcp(T(1) - tb * ty);
    const T hd = T(0.5) * d;                     // theta dq/2
    const T mid = m_fma(T(0.5), dq, qmin);
    fm = m_fma(-hd, ty, mid);
    fp = m_fma(hd, t1, mid);
    return true;
}

// Face values of cell i of a pencil, s[0..4] = q_{i-2} .. q_{i+2}: lo at its face
// towards i-1, hi at its face towards i+1.  MUSCL (van Leer) for every
// primitive (s[1..3] only); for a volume fraction (frac = true) the BVD rule
// keeps the cell's THINC face values only where its total boundary variation
// is strictly below MUSCL's (where the cell has none, nothing is to choose).
template <class T>
__device__ __forceinline__ void recon_cell(const GridP &g, const T *s, bool frac, T &lo, T &hi)
{
    if (sizeof(T) == 4 && frac) {
        mix32_recon_cell<T>(g, s, frac, lo, hi);
        return;
    }
    const T hB = half_slope(s[2] - s[1], s[3] - s[2]);
    const T Bm = s[2] - hB, Bp = s[2] + hB;
    lo = Bm;
    hi = Bp;
    if (!frac || !g.use_thinc) return;
    T tBm, tBp;
    if (!thinc<T>(g, s[1], s[2], s[3], tBm, tBp)) return;
    const T hA = half_slope(s[1] - s[0], s[2] - s[1]);
    const T hC = half_slope(s[3] - s[2], s[4] - s[3]);
    const T Ap = s[1] + hA, Cm = s[3] - hC;
    T tAm = Ap, tAp = Ap, tCm = Cm, tCp = Cm;
    thinc<T>(g, s[0], s[1], s[2], tAm, tAp);
    thinc<T>(g, s[2], s[3], s[4], tCm, tCp);
    const T tbvBM = m_abs(Ap - Bm) + m_abs(Bp - Cm);
    const T tbvBT = m_abs(tAp - tBm) + m_abs(tBp - tCm);
    // (at a steepness from about 19 on tanh beta is 1 in FP64 and a profile's end value can be 0/0: the variation is
    // then a NaN, and MUSCL's values stand)
    if (!m_nan(tbvBT) && m_less(tbvBT, tbvBM)) {
        lo = tBm;
        hi = tBp;
    }
}

// the same in the order of operations of a form
template <class T, int NMAT, int SOLID>
__device__ __forceinline__ void recon_form(const GridP &g, const T *s, bool frac, T &lo, T &hi)
{
    if constexpr (mix32<T, NMAT, SOLID>()) mix32_recon_cell<T>(g, s, frac, lo, hi);
    else recon_cell<T>(g, s, frac, lo, hi);
}

// ------------------------------------------------------------- Riemann

// Left value where the contact moves right (sgn > 0), right value where it
// moves left, the mean of both where it stands.
template <class T>
__device__ __forceinline__ T upwind_mix(int sgn, T xl, T xr)
{
    T v = m_sel(sgn > 0, xl, xr);
    if (sgn == 0) v = T(0.5) * (xl + xr);
    return v;
}

// out += a (U*_K - U_K) on the partial densities, momenta and energy, for the
// HLLC star state of side K (wave speed SK, normal traction TK, contact Ss).
template <class T, int DIM, int NMAT, int SOLID, int D>
__device__ __forceinline__ void star_jump(const State<T, DIM, NMAT, SOLID> &K, T SK, T TK, T Ss, T a, T *out)
{
    using L = Lay<DIM, NMAT, SOLID>;
    const T uK = K.u[D], EK = state_energy<T, DIM, NMAT, SOLID>(K);
    const T iD = m_rcp(SK - Ss);
    const T chi = (SK - uK) * iD;
#pragma unroll
    for (int l = 0; l < NMAT; l++) out[L::IAR + l] += a * (K.ar[l] * chi - K.ar[l]);
    if constexpr (SOLID == 2) {
#pragma unroll
        for (int l = 0; l < NMAT; l++) out[L::IH + l] += a * (K.ar[l] * K.eps[l] * chi - K.ar[l] * K.eps[l]);
    }
#pragma unroll
    for (int b = 0; b < DIM; b++) out[L::IMOM + b] += a * (K.rho * chi * (b == D ? Ss : K.u[b]) - K.rho * K.u[b]);
    out[L::IE] += a * (chi * EK + (Ss - uK) * (K.rho * chi * Ss + TK * iD) - EK);
}

template <class T>
__device__ __forceinline__ T mix32_upwind(T w, T xl, T xr)
{
    return w == T(1) ? xl : (w == T(0) ? xr : T(0.5) * (xl + xr));
}

// out += a (U*_K - U_K) on the partial densities, momenta and energy, for the
// HLLC star state of side K (wave speed SK, normal traction TK, contact Ss).
template <class T, int DIM, int NMAT, int D>
__device__ __forceinline__ void mix32_star_jump(const State<T, DIM, NMAT, 0> &K, T SK, T TK, T Ss, T a, T *out)
{
    using L = Lay<DIM, NMAT, 0>;
    const T uK = K.u[D];
    const T chi = (SK - uK) / (SK - Ss);
#pragma unroll
    for (int l = 0; l < NMAT; l++) out[L::IAR + l] += a * (K.ar[l] * chi - K.ar[l]);
#pragma unroll
    for (int b = 0; b < DIM; b++) out[L::IMOM + b] += a * (K.rho * chi * (b == D ? Ss : K.u[b]) - K.rho * K.u[b]);
    const T EK = K.rhoE / K.rho;
    out[L::IE] += a * (K.rho * chi * (EK + (Ss - uK) * (Ss + TK / (K.rho * (SK - uK)))) - K.rhoE);
}

// HLLC flux of the FP32 fluid mixtures in their fixed order of operations: the
// flux of the upwind side plus the jump to its star state.
template <class T, int DIM, int NMAT, int D>
__device__ __forceinline__ void mix32_riemann(const GridP &g, const T *wL, const T *wR, T vr, T *out)
{
    using L = Lay<DIM, NMAT, 0>;
    State<T, DIM, NMAT, 0> sl, sr;
    state_from_prim<T, DIM, NMAT, 0>(g, wL, sl);
    state_from_prim<T, DIM, NMAT, 0>(g, wR, sr);
    const T cL = m_sqrt(sl.c2), cR = m_sqrt(sr.c2);
    const T uL = sl.u[D], uR = sr.u[D];
    const T TL = sl.p, TR = sr.p;
    const T SL = m_min(uL - cL, uR - cR);
    const T SR = m_max(uL + cL, uR + cR);
    const T num = add_rn(add_rn(TR - TL, mul_rn(mul_rn(sl.rho, uL), SL - uL)),
                         -mul_rn(mul_rn(sr.rho, uR), SR - uR));
    const T Ss = m_div(num, sl.rho * (SL - uL) - sr.rho * (SR - uR));
    int region;
    if (SL >= T(0)) region = 0;
    else if (Ss >= T(0)) region = 1;
    else if (SR > T(0)) region = 2;
    else region = 3;
    const State<T, DIM, NMAT, 0> &K = (region <= 1) ? sl : sr;
    const T SK = (region <= 1) ? SL : SR;
    const T TK = (region <= 1) ? TL : TR;
    const T uK = K.u[D];
    const bool star = (region == 1 || region == 2);
    const T wlf = Ss > T(0) ? T(1) : (Ss < T(0) ? T(0) : T(0.5));
    T ut[DIM];
#pragma unroll
    for (int a = 0; a < DIM; a++) ut[a] = mix32_upwind(wlf, sl.u[a], sr.u[a]);
    T sig[DIM];
#pragma unroll
    for (int a = 0; a < DIM; a++) sig[a] = (a == D ? -K.p : T(0));
    T work = T(0), work_n = T(0);
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        work += K.u[a] * sig[a];
        if (a == D) work_n += K.u[a] * sig[a];
    }
    const T chi = star ? m_div(SK - uK, SK - Ss) : T(0);
#pragma unroll
    for (int l = 0; l < NMAT; l++) {
        const T F = K.ar[l] * uK;
        out[L::IAR + l] = star ? F + SK * (K.ar[l] * chi - K.ar[l]) : F;
    }
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        const T m = K.rho * K.u[a];
        const T Us = K.rho * chi * (a == D ? Ss : K.u[a]);
        if (star) {
            const T Fa = m * uK - (a == D ? sig[a] : T(0));
            out[L::IMOM + a] = Fa + SK * (Us - m);
        } else {
            out[L::IMOM + a] = m * uK - sig[a];
        }
    }
    {
        const T EK = m_div(K.rhoE, K.rho);
        const T Us = K.rho * chi * (EK + (Ss - uK) * (Ss + m_div(TK, K.rho * (SK - uK))));
        out[L::IE] = star ? (K.rhoE * uK - work_n) + SK * (Us - K.rhoE) : K.rhoE * uK - work;
    }
    if (star && g.hllc_lm) {
        const T Ma = m_max(m_abs(uL) / cL, m_abs(uR) / cR);
        const T ph = m_sin(m_min(T(1), Ma / T(0.1)) * T(3.14159265358979323846) / T(2));
        const T k = T(-0.5) * (T(1) - ph);
        mix32_star_jump<T, DIM, NMAT, D>(sl, SL, TL, Ss, k * SL, out);
        mix32_star_jump<T, DIM, NMAT, D>(sr, SR, TR, Ss, k * SR, out);
    }
    const T us = (region == 0) ? uL : ((region == 3) ? uR : Ss);
#pragma unroll
    for (int l = 0; l < NMAT - 1; l++) out[L::IPHI + l] = mix32_upwind(wlf, wL[L::IPHI + l], wR[L::IPHI + l]) * us;
    out[L::IR] = (vr > T(0)) ? wL[L::IR] * vr : ((vr < T(0)) ? wR[L::IR] * vr : T(0));
    out[L::NVAR] = us;
}

// HLLC flux across a face normal to direction D (Sec. 3.1: Toro's HLLC; the
// fluid pressure replaced by the normal traction T = p - 2G devH_DD for solids;
// Davis wave speeds; partial densities scaled like the mixture density).
// out[0..NVAR-1]: flux of every plane (r: upwind with the body velocity vr),
// out[NVAR]: face velocity u*_D, out[NVAR+1+b]: V*_{D b} (upwind by S*).
//
// In the star regions F_K + S_K (U*_K - U_K) is, by the jump conditions across
// S_K, the flux of the star state itself: with d = S_K - u_K, the mass flux
// M = rho d S*/(S_K - S*), T* = T_K + rho d (S* - u_K), the normal momentum's
// M S* + T* and the energy's S* (E* + T*), E* = (d E - T_K u_K + T* S*)/(S_K - S*):
// half the operations, and no differences of large terms at low Mach numbers.
// The energy is formed for the upwind side only.
template <class T, int DIM, int NMAT, int SOLID, int D>
__device__ __forceinline__ void riemann(const GridP &g, const T *wL, const T *wR, T vr, T *out)
{
    using L = Lay<DIM, NMAT, SOLID>;
    if constexpr (mix32<T, NMAT, SOLID>()) {
        mix32_riemann<T, DIM, NMAT, D>(g, wL, wR, vr, out);
        return;
    }
    State<T, DIM, NMAT, SOLID> sl, sr;
    state_from_prim<T, DIM, NMAT, SOLID>(g, wL, sl);
    state_from_prim<T, DIM, NMAT, SOLID>(g, wR, sr);
    const T uL = sl.u[D], uR = sr.u[D];
    const T TL = SOLID ? m_fma(T(-2) * sl.G, sl.H[D][D], sl.p) : sl.p;
    const T TR = SOLID ? m_fma(T(-2) * sr.G, sr.H[D][D], sr.p) : sr.p;
    const T SL = m_min(uL - sl.c, uR - sr.c);
    const T SR = m_max(uL + sl.c, uR + sr.c);
    // contact speed; the numerator's products are rounded one by one and
    // summed left to right, so that mirror-image states (a wall face) give
    // S* = 0 exactly
    const T dL = SL - uL, dR = SR - uR;
    const T mL = mul_rn(sl.rho, dL), mR = mul_rn(sr.rho, dR);
    const T num = add_rn(add_rn(TR - TL, mul_rn(mL, uL)), -mul_rn(mR, uR));
    const T Ss = num * m_rcp_normal(mL - mR);
    // regions: left of S_L, left star, right star, right of S_R
    const bool all_left = m_ge0(SL);
    const bool left = all_left || m_ge0(Ss);
    const bool star = !all_left && (left || m_pos(SR));
    // quantities carried by the contact take the left value for S* > 0, the
    // right one for S* < 0 and the mean of both at S* = 0 (mirror-symmetric
    // at a wall face)
    const int sgn = m_pos(Ss) ? 1 : (m_neg(Ss) ? -1 : 0);
    State<T, DIM, NMAT, SOLID> K;
#pragma unroll
    for (int l = 0; l < NMAT; l++) {
        K.ar[l] = m_sel(left, sl.ar[l], sr.ar[l]);
        if (SOLID == 2) K.eps[l] = m_sel(left, sl.eps[l], sr.eps[l]);
    }
#pragma unroll
    for (int a = 0; a < DIM; a++) K.u[a] = m_sel(left, sl.u[a], sr.u[a]);
    K.rho = m_sel(left, sl.rho, sr.rho);
    K.p = m_sel(left, sl.p, sr.p);
    K.den = NMAT == 1 ? sl.den : m_sel(left, sl.den, sr.den);
    K.Q = (NMAT == 1 && SOLID == 0) && matc<T>(g, 0).kind != 2 ? sl.Q : m_sel(left, sl.Q, sr.Q);
    const T SK = m_sel(left, SL, SR), TK = m_sel(left, TL, TR), dK = m_sel(left, dL, dR), mK = m_sel(left, mL, mR);
    const T uK = K.u[D];
    const T EK = state_energy<T, DIM, NMAT, SOLID>(K);
    // Tangential traction and velocity at the face: the linear shear-wave
    // Riemann problem (sigma -/+ Z u constant along the shear characteristics,
    // Z = sqrt(rho G)); a gas (Z = 0) transmits no shear.  Without shear
    // stiffness on either side the tangential velocity is upwind by S*.  Right
    // and left of all waves it is the upwind side's own.
    T sig_t[DIM], us[DIM];
    T work_s = T(0);
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        sig_t[a] = T(0);
        us[a] = a == D ? m_sel(star, Ss, uK) : K.u[a];
        // (a solid's stretch flux alone reads the tangential velocity of a standing contact)
        if (SOLID && a != D && star && sgn == 0) us[a] = T(0.5) * (sl.u[a] + sr.u[a]);
    }
    if (SOLID) {
        const T ZL = m_sqrt(sl.rho * sl.G), ZR = m_sqrt(sr.rho * sr.G);
        const bool stiff = m_pos(ZL + ZR);
        const T iZ = m_rcp(ZL + ZR);
#pragma unroll
        for (int a = 0; a < DIM; a++) {
            if (a == D) continue;
            const T sL = T(2) * sl.G * sl.H[a][D], sR = T(2) * sr.G * sr.H[a][D];
            if (!star) {
                sig_t[a] = m_sel(left, sL, sR);
            } else if (stiff) {
                sig_t[a] = (ZR * sL + ZL * sR + ZL * ZR * (sr.u[a] - sl.u[a])) * iZ;
                us[a] = (ZL * sl.u[a] + ZR * sr.u[a] + sR - sL) * iZ;
            }
            work_s += us[a] * sig_t[a];
        }
    }
    // cS: transport velocity of the upwind side's contents (rho* S*/rho_K, or u_K)
    T cS, Tf, EF;
    if (star) {
        const T iD = m_rcp_normal(SK - Ss);
        cS = dK * iD * Ss;
        Tf = m_fma(mK, Ss - uK, TK);
        const T Es = m_fma(dK, EK, m_fma(Tf, Ss, -(TK * uK))) * iD;
        EF = Ss * (Es + Tf);
    } else {
        cS = uK;
        Tf = TK;
        EF = uK * (EK + TK);
    }
    const T M = K.rho * cS;
#pragma unroll
    for (int l = 0; l < NMAT; l++) out[L::IAR + l] = NMAT == 1 ? M : K.ar[l] * cS;
    if constexpr (SOLID == 2) {
        // plastic-strain planes: carried like the partial densities
#pragma unroll
        for (int l = 0; l < NMAT; l++) out[L::IH + l] = K.eps[l] * out[L::IAR + l];
    }
#pragma unroll
    for (int a = 0; a < DIM; a++)
        out[L::IMOM + a] = a == D ? m_fma(M, us[D], Tf) : (SOLID ? M * K.u[a] - sig_t[a] : M * K.u[a]);
    out[L::IE] = SOLID ? EF - work_s : EF;
    if (star && g.hllc_lm) {
        // HLLC-LM (the published low-Mach form): the centred flux
        // (F_L + F_R)/2 + [phi S_L (U*_L - U_L) + |S*| (U*_L - U*_R) + phi S_R (U*_R - U_R)]/2
        // with phi = sin(min(1, Ma/0.1) pi/2), Ma the larger face-normal Mach
        // number.  With the jump conditions across the three waves this is
        // the HLLC flux above minus (1 - phi)/2 [S_L (U*_L - U_L) + S_R (U*_R - U_R)]
        // on the partial densities, momenta and energy.
        const T Ma = m_max(m_abs(uL) * m_rcp(sl.c), m_abs(uR) * m_rcp(sr.c));
        const T ph = m_sin(m_min(T(1), Ma / T(0.1)) * T(3.14159265358979323846) / T(2));
        const T k = T(-0.5) * (T(1) - ph);
        star_jump<T, DIM, NMAT, SOLID, D>(sl, SL, TL, Ss, k * SL, out);
        star_jump<T, DIM, NMAT, SOLID, D>(sr, SR, TR, Ss, k * SR, out);
    }
#pragma unroll
    for (int l = 0; l < NMAT - 1; l++) out[L::IPHI + l] = upwind_mix(sgn, wL[L::IPHI + l], wR[L::IPHI + l]) * us[D];
    // V*: upwind by S*; F(V_ab) = V*_ab u*_D - V*_Db u*_a, V*_Db stored whenever b < DIM or (D,b) = (2,2)
    T vs[L::NV > 0 ? L::NV : 1];
#pragma unroll
    for (int c = 0; c < L::NV; c++) vs[c] = upwind_mix(sgn, wL[L::IV + c], wR[L::IV + c]);
#pragma unroll
    for (int c = 0; c < L::NV; c++) {
        const int a = v_row(DIM, c), b = v_col(DIM, c);
        T F = vs[c] * us[D];
#pragma unroll
        for (int cc = 0; cc < L::NV; cc++)
            if (v_row(DIM, cc) == D && v_col(DIM, cc) == b && a < DIM) F -= vs[cc] * us[a];
        // the row of D itself: V*_Db u*_D - V*_Db u*_D
        out[L::IV + c] = a == D ? T(0) : F;
    }
    out[L::IR] = m_pos(vr) ? wL[L::IR] * vr : (m_neg(vr) ? wR[L::IR] * vr : T(0));
    out[L::NVAR] = us[D];
#pragma unroll
    for (int b = 0; b < L::NB; b++) {
        T vdb = T(0);
#pragma unroll
        for (int cc = 0; cc < L::NV; cc++)
            if (v_row(DIM, cc) == D && v_col(DIM, cc) == b) vdb = vs[cc];
        out[L::NVAR + 1 + b] = vdb;
    }
}

// -------------------------------------------------------- plastic return

// cosh(y) - 1 and sinh(y)/y of y^2 (>= 0), FP64: their series to 2^-53 below
// y^2 = 0.02 (elastic metals: y is half the yield strain), exp above.
__device__ __forceinline__ void coshm1_sinhc(double y2, double &ch, double &sh)
{
    if (m_less(y2, 0.02)) {
        double c = 1.0 / 3628800.0;                      // 1/10!
        c = fma(c, y2, 1.0 / 40320.0);
        c = fma(c, y2, 1.0 / 720.0);
        c = fma(c, y2, 1.0 / 24.0);
        c = fma(c, y2, 0.5);
        ch = c * y2;
        double s = 1.0 / 39916800.0;                     // 1/11!
        s = fma(s, y2, 1.0 / 362880.0);
        s = fma(s, y2, 1.0 / 5040.0);
        s = fma(s, y2, 1.0 / 120.0);
        s = fma(s, y2, 1.0 / 6.0);
        sh = fma(s, y2, 1.0);
        return;
    }
    const double y = sqrt(y2), e = exp(y), i = 1.0 / e;
    ch = fma(0.5, e + i, -1.0);
    sh = 0.5 * (e - i) / y;
}

// exp(x) - 1 for |x| < 0.0625: its series to 2^-53
__device__ __forceinline__ double expm1_near0(double x)
{
    double e = 1.0 / 362880.0;                           // 1/9!
    e = fma(e, x, 1.0 / 40320.0);
    e = fma(e, x, 1.0 / 5040.0);
    e = fma(e, x, 1.0 / 720.0);
    e = fma(e, x, 1.0 / 120.0);
    e = fma(e, x, 1.0 / 24.0);
    e = fma(e, x, 1.0 / 6.0);
    e = fma(e, x, 0.5);
    e = fma(e, x, 1.0);
    return e * x;
}

// Perfect plasticity by instantaneous radial return, in FP64: the stored A is
// replaced by its symmetric unimodular stretch Q diag(exp(s d_k)) Q^T with d_k
// the deviatoric log-stretches and s = min(1, sigma_Y/sigma_vm),
// sigma_vm = sqrt(3/2) 2 G |d| (mixture G and sigma_Y).  Energy, masses and
// momenta are untouched.  Returns the equivalent plastic strain increment
// sqrt(2/3) (1 - s) |d| (0 below yield).
// yield(svm, |d|, J2) gives the yield stress for the trial von Mises stress
// svm and deviatoric log-stretch norm |d| (Johnson-Cook: plastic strain,
// temperature and rate); the constant-sigma_Y form ignores its arguments.
//
// In 2-D the in-plane log-stretches are -d2/2 +- k/2 (stretch_log), so the new
// in-plane block is e^{-s d2/2} [cosh(s k/2) I + sinh(s k/2) (c_2, s_2)]: the
// FP64 pipe does some 75 operations for an elastic or yielding metal cell in
// place of three logarithms, three exponentials, a root and divisions.
// e: the stretch logarithm of A; sc: the scale s.
template <int DIM, class Y>
__device__ __forceinline__ double plastic_return_y(const StretchLog<double> &e, double A[3][3], double G, Y yield,
                                                   double &sc)
{
    const double nd = m_sqrt(e.J2);
    const double svm = sqrt(6.0) * G * nd;
    const double sigY = yield(svm, nd, e.J2);
    double deps = 0.0;
    sc = 1.0;
    if (svm > sigY) {
        sc = sigY / svm;
        // equivalent plastic strain of the removed deviatoric log-strain (1 - s)|d|
        deps = sqrt(2.0 / 3.0) * (1.0 - sc) * nd;
    }
    if (DIM == 1) {
        A[0][0] = exp(sc * e.half);
        A[1][1] = exp(sc * e.b01);
        A[2][2] = exp(sc * e.d2);
        A[0][1] = A[1][0] = 0.0;
    } else {
        const double h = 0.5 * sc, x = -h * e.d2;
        double ch, sh, q;
        coshm1_sinhc(h * h * e.k2, ch, sh);
        // q: sinh(s k/2)/|(half, b01)|, times the mean stretch e^x
        if (m_less(m_abs(x), 0.03125)) {
            // stretches near 1 by what they differ from it, each rounded once
            const double m = expm1_near0(x), s = fma(ch, m, ch + m);   // e^x cosh - 1
            q = (1.0 + m) * sh * (h * e.q);
            A[0][0] = 1.0 + fma(q, e.half, s);
            A[1][1] = 1.0 + fma(-q, e.half, s);
            A[2][2] = 1.0 + expm1_near0(-2.0 * x);
        } else {
            const double m = exp(x);
            q = m * sh * (h * e.q);
            ch = fma(ch, m, m);
            A[0][0] = fma(q, e.half, ch);
            A[1][1] = fma(-q, e.half, ch);
            A[2][2] = exp(-2.0 * x);
        }
        A[0][1] = A[1][0] = q * e.b01;
    }
    A[0][2] = A[2][0] = A[1][2] = A[2][1] = 0.0;
    return deps;
}

// Johnson-Cook flow stress of material m (the law, the reference temperature
// 298 K and rate 1/s are readings of Table 2, which lists the constants only):
// (c1 + c2 eps^n)(1 + c3 ln max(rate, 1))(1 - T*^m), T* = (T - 298)/(T_melt - 298)
// clipped to [0, 1]: its first and last factors.
__device__ __forceinline__ double jc_yield0(const MatP &m, double eps, double T)
{
    double ts = (T - 298.0) / (m.jc_tmelt - 298.0);
    ts = ts < 0.0 ? 0.0 : (ts > 1.0 ? 1.0 : ts);
    const double e = eps > 0.0 ? eps : 0.0;
    return (m.jc_c1 + m.jc_c2 * pow(e, m.jc_n)) * (1.0 - pow(ts, m.jc_m));
}

// Mixture yield stress of a cell with Johnson-Cook materials (weights
// phi_l/Gamma_l, Sec. 2.2), each at its plastic strain and at the temperature
// of its Mie-Grueneisen thermal energy, 298 K + (p - p_ref)/(rho_l Gamma_l C_V);
// w: the cell's primitives, J2: its |dev ln V|^2.  The rate enters through its
// logarithm only: the yield stress is y0 + y1 ln max(rate, 1), one evaluation
// of the powers for the rate-free and the final stress.
template <class R, int DIM, int NMAT, int SOLID>
__device__ __forceinline__ void jc_mixture_yield(const GridP &g, const R *w, double J2, double &y0, double &y1)
{
    using L = Lay<DIM, NMAT, SOLID>;
    double fsum = 0.0, phi[NMAT];
#pragma unroll
    for (int l = 0; l < NMAT - 1; l++) {
        phi[l] = (double)w[L::IPHI + l];
        fsum += phi[l];
    }
    phi[NMAT - 1] = 1.0 - fsum;
    double n0 = 0.0, n1 = 0.0, den = 0.0;
    const double p = (double)w[L::IE];
#pragma unroll
    for (int l = 0; l < NMAT; l++) {
        const double f = phi_clip(phi[l]) * g.mc_d[l].invGam;
        double sy = g.mat[l].sigY;
        if (g.mat[l].jc) {
            const double rl = (double)w[L::IAR + l];
            const Ref<double> r = mat_ref<double>(g.mc_d[l], rl, J2);
            double eps = 0.0;
            if constexpr (SOLID == 2) eps = (double)w[L::IH + l];
            sy = jc_yield0(g.mat[l], eps, 298.0 + (p - r.pref) * m_rcp(rl * g.mc_d[l].Gam * g.mat[l].jc_cv));
            n1 += f * sy * g.mat[l].jc_c3;
        }
        n0 += f * sy;
        den += f;
    }
    const double i = m_rcp(den);
    y0 = n0 * i;
    y1 = n1 * i;
}

// The return of a cell below yield (s = 1) in 2-D: A becomes the unimodular
// stretch of A A^T = B itself.  A 2 x 2 block's root is (B + d I)/sqrt(T), d its
// own root's determinant |det A_2| and T = tr B + 2 d, so that with the scale to
// determinant one the block is (B + d I) X^(-1/6), X = (d |A_zz|)^2 T^3: some 33
// operations of the FP64 pipe in place of 95 by way of the logarithm.  The
// sixth root starts in FP32 and takes one third-order step; false (nothing
// written) where X leaves FP32's middle range.
__device__ __forceinline__ bool elastic_stretch(double A[3][3])
{
    const double b00 = fma(A[0][0], A[0][0], A[0][1] * A[0][1]);
    const double b11 = fma(A[1][1], A[1][1], A[1][0] * A[1][0]);
    const double b01 = fma(A[0][0], A[1][0], A[0][1] * A[1][1]);
    const double d = m_abs(fma(A[0][0], A[1][1], -(A[0][1] * A[1][0])));
    const double T = fma(2.0, d, b00 + b11), m = d * m_abs(A[2][2]);
    const double X = (m * m) * (T * T * T);
    const float xf = m_narrow(X);
    if (!(xf > 1e-25f && xf < 1e25f)) return false;
    const double y = m_widen(exp2f(log2f(xf) * (-1.f / 6.f)));
    const double y2 = y * y, e = fma(-X, y2 * y2 * y2, 1.0);
    const double q = fma(y * e, fma(e, 7.0 / 72.0, 1.0 / 6.0), y);
    A[2][2] = m_rcp(d * (q * q) * T);
    A[0][0] = (b00 + d) * q;
    A[1][1] = (b11 + d) * q;
    A[0][1] = A[1][0] = b01 * q;
    A[0][2] = A[2][0] = A[1][2] = A[2][1] = 0.0;
    return true;
}

// End of a step for a cell of a solid's grid (Sec. 2.1.1): the plastic return
// of the new conserved state o, and the wave speed of the state it leaves
// (cell_speed).  The reference curves are linear in J^2 (p_ref and rho e_ref
// by G J^2), and the return scales J^2 by s^2, so that pressure, shear modulus
// and sound speed before and after it come from one stretch logarithm and one
// evaluation of the curves (FP64 form: five and four before).  Decomposition
// and return are FP64 in both forms; the FP32 form first asks its own stretch
// logarithm whether the cell is clearly below yield, where the return is a root.
template <class R, int DIM, int NMAT, int SOLID>
__device__ __forceinline__ R solid_finish(const GridP &g, double dt, R *o, R &c)
{
    using L = Lay<DIM, NMAT, SOLID>;
    R A[3][3];
    unpack_A_ct<R, DIM, NMAT, SOLID>(o, A);
    StretchLog<R> e;
    stretch_log<R, DIM>(A, e);
    // sums over the materials: num = num0 + J^2 numJ (over den, the pressure),
    // Yn = p K1 - K0 + J^2 KJ (mix_sums), G and sigma_Y
    R phi[NMAT], rhol[NMAT], rho = R(0), rhos = R(0), fsum = R(0);
#pragma unroll
    for (int l = 0; l < NMAT - 1; l++) {
        phi[l] = o[L::IPHI + l];
        fsum += phi[l];
    }
    phi[NMAT - 1] = R(1) - fsum;
#pragma unroll
    for (int l = 0; l < NMAT; l++) rho += o[L::IAR + l];
    const R irho = m_rcp(rho);
    R u[DIM], mu = R(0);
#pragma unroll
    for (int a = 0; a < DIM; a++) {
        u[a] = o[L::IMOM + a] * irho;
        mu = m_fma(o[L::IMOM + a], u[a], mu);
    }
    R num0 = m_fma(R(-0.5), mu, o[L::IE]), numJ = R(0), den = R(0), K1 = R(0), K0 = R(0), KJ = R(0), Gn = R(0), Sn = R(0);
#pragma unroll
    for (int l = 0; l < NMAT; l++) {
        const MatC<R> &m = matc<R>(g, l);
        const R ar = o[L::IAR + l], f = NMAT == 1 ? R(1) : phi_clip(phi[l]);
        rhol[l] = NMAT == 1 ? rho : phasic_density<R>(g, l, ar, f);
        const R w = f * m.invGam, as = f * rhol[l];
        rhos += as;
        den += w;
        const R fy = as != R(0) ? f : R(0);   // a material without mass has no part in the sound speed
        K1 = m_fma(fy, m.kA, K1);
        if (m.kind == 2) {
            const Ref<R> r = mat_ref<R>(m, rhol[l], R(0));
            const R fe = NMAT > 1 && m_less(f, R(1e-6)) ? ar * m.irho0 : f;
            num0 += w * r.pref - fe * r.re;
            numJ += (w * m.beta - fe) * r.G;
            const R ky = fy * m.kA, wy = fy * m.invGam;
            K0 += ky * r.pref - wy * m_fma(R(4) / R(3), r.G, r.rdp);
            KJ += (wy * m.bb - ky * m.beta) * r.G;
            Gn = m_fma(w, r.G, Gn);
            Sn = m_fma(w, m.sigY, Sn);
        } else {
            num0 = m_fma(f, m.kB, num0);
            K0 = m_fma(fy, m.kB, K0);
        }
    }
    const R iden = m_rcp(den);
    // the return
    double Ad[3][3], sc = 1.0, deps = 0.0;
    StretchLog<double> ed;
    bool elastic = false;
    if constexpr (sizeof(R) == 8) {
        ed = e;
    } else {
        unpack_A<R, DIM, NMAT, SOLID>(o, Ad);
        // below yield by more than the error of the FP32 stretch: 1 % and 5e-7, twice
        // what the roundings of A A^T's terms leave of |dev H| (2e-7 in all), so that
        // a yield strain of that size takes the FP64 decomposition in every cell
        if (DIM == 2 && !g.any_jc && R(2.4494897) * Gn * (m_sqrt(e.J2) + R(5e-7)) <= R(0.99) * Sn && e.J2 < R(0.25))
            elastic = elastic_stretch(Ad);
        if (!elastic) stretch_log<double, DIM>(Ad, ed);
    }
    const double G = m_widen(Gn * iden), sigY = m_widen(Sn * iden);
    if (elastic) {
    } else if (g.any_jc) {
        // Johnson-Cook: the rate is that of a return at the rate-free
        // yield stress over the step (one explicit predictor)
        deps = plastic_return_y<DIM>(ed, Ad, G, [&](double svm, double nd, double J2) {
            R w[L::NVAR];
#pragma unroll
            for (int l = 0; l < NMAT - 1; l++) w[L::IPHI + l] = phi[l];
#pragma unroll
            for (int l = 0; l < NMAT; l++) {
                w[L::IAR + l] = rhol[l];
                const R ar = o[L::IAR + l];
                if constexpr (SOLID == 2) w[L::IH + l] = ar != R(0) ? m_quot(o[L::IH + l], ar) : R(0);
            }
            w[L::IE] = m_fma(numJ, e.J2, num0) * iden;
            double y0, y1;
            jc_mixture_yield<R, DIM, NMAT, SOLID>(g, w, J2, y0, y1);
            if (!(svm > y0 && dt > 0.0)) return y0;
            const double rate = sqrt(2.0 / 3.0) * (1.0 - y0 / svm) * nd / dt;
            return rate > 1.0 ? y0 + y1 * log(rate) : y0;
        }, sc);
    } else {
        deps = plastic_return_y<DIM>(ed, Ad, G, [sigY](double, double, double) { return sigY; }, sc);
    }
#pragma unroll
    for (int k = 0; k < L::NV; k++) o[L::IV + k] = m_store<R>(Ad[v_row(DIM, k)][v_col(DIM, k)]);
    if constexpr (SOLID == 2) {
        // the strain removed by the return, added to every material with a yield stress
#pragma unroll
        for (int l = 0; l < NMAT; l++)
            if ((matc<R>(g, l).sigY > R(0) || g.mat[l].jc) && deps > 0.0)
                o[L::IH + l] = (R)((double)o[L::IH + l] + (double)o[L::IAR + l] * deps);
    }
    // wave speed of the state after the return
    const R s2 = (R)sc, J2 = s2 * s2 * e.J2;
    const R p = m_fma(numJ, J2, num0) * iden;
    const R Yn = m_fma(p, K1, m_fma(J2, KJ, -K0));
    c = NMAT == 1 ? m_sqrt_ratio(Yn * matc<R>(g, 0).Gam, rhos) : m_sqrt_ratio(Yn, rhos * den);
    R sum = R(0);
#pragma unroll
    for (int d = 0; d < DIM; d++) sum += (m_abs(u[d]) + c) * gridc<R>(g).inv_dx[d];
    return sum;
}

}  // namespace dfv
