// idugks_kernels.cu -- sm_103a kernels of one IDUGKS iteration
// (arXiv 1709.01819, Section 2).
//
// Storage.  The distribution f~ (Eq. 10) of every (cell, discrete velocity) is
// kept as a pair {G, H} (Eq. 5) relative to one global reference Maxwellian
// M_ref: dev = f~ - M_ref.  All per-velocity operations of the scheme are
// linear in f~ except the equilibria, which are evaluated directly in deviation
// form (dev_equilibrium), so float32 storage rounds relative to the deviation
// and not to f.  The flux of M_ref through the closed surface of a cell
// vanishes (sum_f n_f S_f = 0), so stored face fluxes are fluxes of
// (f_face - M_ref); the macroscopic face moments add M_ref's float64 moments
// back.  Layouts are velocity-contiguous: [cell][velocity]{G,H}.
//
// Precision.  GB300 runs float64 at 1/64 of the float32 rate (a warp-wide
// float64 instruction occupies an SM for ~16 cycles), so in mixed precision
// every per-velocity operation is float32 and the velocity sums are
// accumulated in float32 over at most 8 terms per lane, then in a compensated
// float-float pair (about 48 significant bits) across lanes; the pair is
// widened to float64 by the lane-parallel per-cell / per-face kernels, which
// do all scalar physics (state from moments, tau, equilibrium coefficients)
// in float64.  In FP64 mode the same code runs in float64 throughout.
//
// One iteration, in launch order on the caller's stream:
//   k_cell_moments   warp per cell: raw moments of f~                     [a1]
//   k_cell_params    thread per cell: heat flux (q of Eq. 20), tau,
//                    equilibrium at W^n, coefficients of fb+ (Eq. 10, 12)
//   k_fbp            per (cell, velocity): fb+ = c1 f~ + c2 f^S
//   k_cell_recon     per (cell, velocity): least-squares gradient (Eq. 14-15),
//                    limiter (Eq. 16-17) and fb at the half step (Eq. 11, 13)
//                    at the faces the velocity leaves the cell by          [a2]
//   k_face_moments   warp per face: wall density (Eq. 35) and the incoming
//                    part at boundary faces, raw moments of fb; with the
//                    linearised wall the ghost density increment of Eq. (35) [a3]
//   k_face_params    thread per face: face state, tau, q, equilibrium, and
//                    the weights of Eq. (18)                              [a4]
//   k_face_flux      warp per face: f at the face (Eq. 18), flux (Eq. 19),
//                    flux moments; with the linearised wall the ghost term
//                    of Eq. (34) on the incoming velocities of wall faces
//   k_face_phi       thread per face: Phi_f = sum_k w psi F_k (Eq. 27)
//   k_macro_pre, k_macro_sweep, k_macro_post: macroscopic LU-SGS          [a5]
//                    (k_macro_sweep_sched on an unstructured mesh; with the
//                    point-relaxation predictor k_record_residual and n
//                    launches of k_macro_relax in place of the sweep)
//   k_micro_residual, then the micro LU-SGS sweeps and update: k_sweep_lines
//                    (lines of cells of a structured block) or k_sweep (level
//                    schedules of an unstructured mesh)              [a6-a7]
// Explicit DUGKS (Eq. 21) runs the cell and face kernels, then
// k_explicit_update, k_cell_moments, k_explicit_w and k_record_residual.
// Data are laid out per cell in four face slots (a triangle's fourth slot is
// unused: sign 0, no neighbour, no geometry).
#include "idugks_internal.h"
#include "wavefront.cuh"

#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

namespace idg {

// ---------------------------------------------------------------------------
// precision helpers
// ---------------------------------------------------------------------------
template <class T> struct V2;
template <> struct V2<float> { using t = float2; };
template <> struct V2<double> { using t = double2; };

__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
// a b + c in one rounding.  This file is compiled without contraction
// (-fmad=false) and says where it fuses: a kernel's instances for one problem
// and for a batch then round alike, whatever the compiler makes of each.
__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }
// correctly rounded reciprocals: the same value as 1 / x in IEEE division,
// without the general division routine
__device__ __forceinline__ float rcp_rn(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double rcp_rn(double x) { return __drcp_rn(x); }
// 1/x in the line macroscopic sweep's flux increments: one approximate
// reciprocal in float32 -- the predictor's increments set the convergence
// path, not the fixed point, which the residual alone fixes -- and correctly
// rounded in float64 (FP64 parity with the oracle)
__device__ __forceinline__ float rcp_line(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ double rcp_line(double x) { return __drcp_rn(x); }
// e^x - 1 for |x| < 1/2 by its Taylor series in Horner form (every x^k / k! up
// to k = 9 in float32, 15 in float64: the terms left out sum to at most 5.7e-10
// and 1.51e-18 of x; in float32 0.29 to 0.30 ulp rms and 0.82 at most, where
// expm1f measures 0.29 to 0.51 and 1.33): half the instructions of the general
// function, which reduces the range first.  (Taking
// it up to |x| = 1 raised the float32 residual floor of a Ma 5 flow by half: the
// exponent difference carries the rounding of its large terms.)
__device__ __forceinline__ float expm1_near(float x)
{
    float q = 1.0f / 362880.0f;
    q = fmaf(q, x, 1.0f / 40320.0f);
    q = fmaf(q, x, 1.0f / 5040.0f);
    q = fmaf(q, x, 1.0f / 720.0f);
    q = fmaf(q, x, 1.0f / 120.0f);
    q = fmaf(q, x, 1.0f / 24.0f);
    q = fmaf(q, x, 1.0f / 6.0f);
    q = fmaf(q, x, 0.5f);
    return fmaf(x * x, q, x);
}
__device__ __forceinline__ double expm1_near(double x)
{
    double q = 1.0 / 1307674368000.0;
    q = fma(q, x, 1.0 / 87178291200.0);
    q = fma(q, x, 1.0 / 6227020800.0);
    q = fma(q, x, 1.0 / 479001600.0);
    q = fma(q, x, 1.0 / 39916800.0);
    q = fma(q, x, 1.0 / 3628800.0);
    q = fma(q, x, 1.0 / 362880.0);
    q = fma(q, x, 1.0 / 40320.0);
    q = fma(q, x, 1.0 / 5040.0);
    q = fma(q, x, 1.0 / 720.0);
    q = fma(q, x, 1.0 / 120.0);
    q = fma(q, x, 1.0 / 24.0);
    q = fma(q, x, 1.0 / 6.0);
    q = fma(q, x, 0.5);
    return fma(x * x, q, x);
}
__device__ __forceinline__ float t_exp(float x) { return expf(x); }
__device__ __forceinline__ double t_exp(double x) { return exp(x); }

template <class T> __device__ __forceinline__ T vx(const KParams &p, int k);
template <> __device__ __forceinline__ float vx<float>(const KParams &p, int k) { return p.uxf[k]; }
template <> __device__ __forceinline__ double vx<double>(const KParams &p, int k) { return p.ux[k]; }
template <class T> __device__ __forceinline__ T vy(const KParams &p, int k);
template <> __device__ __forceinline__ float vy<float>(const KParams &p, int k) { return p.uyf[k]; }
template <> __device__ __forceinline__ double vy<double>(const KParams &p, int k) { return p.uy[k]; }
template <class T> __device__ __forceinline__ T vw(const KParams &p, int k);
template <> __device__ __forceinline__ float vw<float>(const KParams &p, int k) { return p.wf[k]; }
template <> __device__ __forceinline__ double vw<double>(const KParams &p, int k) { return p.w[k]; }
template <class T> __device__ __forceinline__ T vgref(const KParams &p, int k);
template <> __device__ __forceinline__ float vgref<float>(const KParams &p, int k) { return p.greff[k]; }
template <> __device__ __forceinline__ double vgref<double>(const KParams &p, int k) { return p.gref[k]; }

// xi . n without contraction, so the sign decision matches a plain
// multiply-add evaluation bit for bit in float64
template <class T> __device__ __forceinline__ T xi_dot_n(T ux, T uy, T nx, T ny)
{
    return add_rn(mul_rn(ux, nx), mul_rn(uy, ny));
}

// ---------------------------------------------------------------------------
// accumulators: float-float pairs in mixed precision, double in FP64
// ---------------------------------------------------------------------------
struct FF {
    float hi, lo;
};
// error-free sum of two floats (Knuth's two-sum)
__device__ __forceinline__ FF two_sum(float a, float b)
{
    float s = a + b;
    float bb = s - a;
    float e = (a - (s - bb)) + (b - bb);
    return {s, e};
}
__device__ __forceinline__ FF ff_add(FF a, FF b)
{
    FF s = two_sum(a.hi, b.hi);
    float e = s.lo + (a.lo + b.lo);
    float hi = s.hi + e;
    return {hi, e - (hi - s.hi)};
}

template <class T> struct Acc;
template <> struct alignas(8) Acc<float> {
    FF v;
    __device__ __forceinline__ void zero() { v = {0.f, 0.f}; }
    // (the error terms collect in lo: renormalised once, by warp_sum)
    __device__ __forceinline__ void add(float x)
    {
        const FF s = two_sum(v.hi, x);
        v.hi = s.hi;
        v.lo += s.lo;
    }
    __device__ __forceinline__ void warp_sum()
    {
        for (int o = 16; o > 0; o >>= 1) {
            FF u{__shfl_down_sync(0xffffffffu, v.hi, o), __shfl_down_sync(0xffffffffu, v.lo, o)};
            v = ff_add(v, u);
        }
    }
    __device__ __forceinline__ void store(void *base, size_t i) const { ((float2 *)base)[i] = make_float2(v.hi, v.lo); }
    __device__ __forceinline__ double value() const { return (double)v.hi + (double)v.lo; }
};
template <> struct Acc<double> {
    double v;
    __device__ __forceinline__ void zero() { v = 0.0; }
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ void warp_sum()
    {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    __device__ __forceinline__ void store(void *base, size_t i) const { ((double *)base)[i] = v; }
    __device__ __forceinline__ double value() const { return v; }
};

// Sums of NA <= 16 accumulators over the 32 lanes, stored at base[q], q < NA.
// Lanes halve the set of sums they carry at each exchange (16, 8, 4, 2, 1 lanes
// apart), so that 16 sums take 16 exchanges instead of 16 x 5; lane pairs meet
// in the same order as in warp_sum.
__device__ __forceinline__ FF shfl_xor_acc(FF a, int o)
{
    return {__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}
__device__ __forceinline__ double shfl_xor_acc(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ FF sum_acc(FF a, FF b) { return ff_add(a, b); }
__device__ __forceinline__ double sum_acc(double a, double b) { return a + b; }
// One to four warps share a row (row_warps): with more than one their sums meet
// in shared memory behind a barrier of those warps and are added in order.
constexpr int kRowSums = 8 * 16;  // shared sums of a 256-thread block
struct Row {
    int sub, warps;  // this warp of the row's warps
};
__device__ __forceinline__ Row row_of(const KParams &p, int blk, int &row)
{
    Row r;
    r.warps = p.row_warps;
    const int w = threadIdx.x >> 5;
    row = blk * (8 / r.warps) + w / r.warps;
    r.sub = w & (r.warps - 1);
    return r;
}
__device__ __forceinline__ void row_barrier(const Row &r)
{
    asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)(threadIdx.x >> 5) / r.warps), "r"(32 * r.warps) : "memory");
}
template <int NA, class T>
__device__ __forceinline__ void row_sum_store(const Acc<T> (&acc)[NA], int lane, const Row &r, Acc<T> *sums, void *base, size_t i0)
{
    constexpr int NP = NA <= 4 ? 4 : 16;  // sums carried, the ones past NA zero
    decltype(acc[0].v) x[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) {
        if (q < NA) x[q] = acc[q].v;
        else x[q] = decltype(acc[0].v){};
    }
    int mine = 0;
#pragma unroll
    for (int o = 16, n = NP; o > 0; o >>= 1) {
        if (n > 1) {
            // the upper lane of a pair keeps the upper half of the sums
            n >>= 1;
            const bool up = lane & o;
#pragma unroll
            for (int q = 0; q < n; ++q) {
                const auto keep = up ? x[q + n] : x[q], give = up ? x[q] : x[q + n];
                x[q] = sum_acc(keep, shfl_xor_acc(give, o));
            }
            if (up) mine += n;
        } else {
            x[0] = sum_acc(x[0], shfl_xor_acc(x[0], o));
        }
    }
    // lanes that differ in the last log2(32 / NP) bits carry the same sum
    const bool owner = (lane & (32 / NP - 1)) == 0 && mine < NA;
    Acc<T> a;
    a.v = x[0];
    if (r.warps > 1) {
        Acc<T> *s = sums + 16 * (threadIdx.x >> 5) + mine;
        if (owner) *s = a;
        row_barrier(r);
        if (r.sub > 0) return;
        if (owner)
            for (int w = 1; w < r.warps; ++w) a.v = sum_acc(a.v, s[16 * w].v);
    }
    if (owner) a.store(base, i0 + mine);
}

// an accumulator entry widened to float64
template <class T> __device__ __forceinline__ double acc_load(const void *base, size_t i);
template <> __device__ __forceinline__ double acc_load<float>(const void *base, size_t i)
{
    float2 a = ((const float2 *)base)[i];
    return (double)a.x + (double)a.y;
}
template <> __device__ __forceinline__ double acc_load<double>(const void *base, size_t i)
{
    return ((const double *)base)[i];
}

// block sum of float64 values (fixed tree: deterministic); result in thread 0
template <int NV>
__device__ void block_sum(double (&v)[NV], double *sm /* >= 32*NV */)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q)
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < NV; ++q) sm[wid * NV + q] = v[q];
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 0; q < NV; ++q) {
            double a = 0.0;
            for (int u = 0; u < nw; ++u) a += sm[u * NV + q];
            v[q] = a;
        }
    }
}

// ---------------------------------------------------------------------------
// launches over one or many problem instances
// ---------------------------------------------------------------------------
// Every iteration kernel takes a Launch: the instances' parameters in device
// memory, the prefix sums of blocks per instance for this kernel (null for a
// single instance) and per-instance activity flags (converged instances of a
// batch are skipped).  A block finds its instance by binary search.
struct Launch {
    const KParams *params;
    const int *off;     // [ninst + 1] or null
    const int *active;  // [ninst] or null
    int ninst;
};

__device__ __forceinline__ bool locate(const Launch &L, const KParams *&pp, int &blk)
{
    int b = blockIdx.x, inst = 0;
    if (L.off) {
        int lo = 0, hi = L.ninst;
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (L.off[mid] <= b) lo = mid;
            else hi = mid;
        }
        inst = lo;
        b -= L.off[lo];
    }
    pp = L.params + inst;
    blk = b;
    return !L.active || L.active[inst];
}

// one instance's launch: its parameters by value (the kernel's constant bank),
// which saves every block a chain of dependent loads before its first data
struct LaunchOne {
    KParams p;
};
__device__ __forceinline__ bool locate(const LaunchOne &L, const KParams *&pp, int &blk)
{
    pp = &L.p;
    blk = blockIdx.x;
    return true;
}

#define IDG_LOCATE()                                   \
    const KParams *pp_;                                \
    int blk;                                           \
    if (!locate(L, pp_, blk)) return;                  \
    const KParams &__restrict__ p = *pp_;

// ---------------------------------------------------------------------------
// kinetic model in float64 (per cell / per face quantities)
// ---------------------------------------------------------------------------
__device__ __forceinline__ double viscosity(const KParams &p, double RT)
{
    return p.mu_ref * pow(RT * p.iRT_ref, p.omega);
}

// The power law of the viscosity for tau in the iteration's kernels: with
// float32 storage tau only sets float32 coefficients (fb+ weights, Eq. 18
// weights, the collision rate, the Shakhov factor) and the float32
// preconditioner, so the power is taken in float32; float64 keeps float64.
template <class T> __device__ __forceinline__ double viscosity_t(const KParams &p, double RT);
template <> __device__ __forceinline__ double viscosity_t<double>(const KParams &p, double RT)
{
    return viscosity(p, RT);
}
template <> __device__ __forceinline__ double viscosity_t<float>(const KParams &p, double RT)
{
    return p.mu_ref * (double)powf((float)(RT * p.iRT_ref), (float)p.omega);
}

// heat flux q = 1/2 sum w c (c^2 G + H) about (U, V) from raw moments
// (G: 1,x,y,xx,xy,yy,x|xi|^2,y|xi|^2; H: 1,x,y), Eq. (4)-(5)
__device__ __forceinline__ void raw_heat_flux(const double *r, double U, double V, double &qx,
                                              double &qy)
{
    const double U2 = mad(U, U, V * V), e = r[3] + r[5] + r[8];
    // the energy-weighted sums less U e, plus 2 U (U . m) and U2 (m - U rho), where
    // m = (r1, r2), less the shear part 2 (r3, r4; r4, r5) U
    const double um = mad(U, r[1], V * r[2]);
    const double cx = mad(-U, r[0], r[1]), cy = mad(-V, r[0], r[2]);
    const double sx = mad(U2, cx, mad(2.0 * U, um, mad(-U, e, r[6] + r[9])));
    const double sy = mad(U2, cy, mad(2.0 * V, um, mad(-V, e, r[7] + r[10])));
    qx = 0.5 * mad(-2.0, mad(U, r[3], V * r[4]), sx);
    qy = 0.5 * mad(-2.0, mad(U, r[4], V * r[5]), sy);
}

__device__ __forceinline__ void raw_to_state(const KParams &p, const double *r, double &rho, double &irho, double &U,
                                             double &V, double &RT, double &qx, double &qy)
{
    rho = r[0];
    irho = rcp_rn(rho);
    U = r[1] * irho;
    V = r[2] * irho;
    const double rhoE2 = r[3] + r[5] + r[8];  // twice the energy density
    RT = mad(-V, V, mad(-U, U, rhoE2 * irho)) * p.iK2;
    raw_heat_flux(r, U, V, qx, qy);
}

// Coefficients of the deviation equilibrium at (rho, U, V, RT, q):
// reduced Maxwellian (Eq. 2, 5) with the Shakhov factor (Eq. 20 read for
// D = 2 + K dof: G factor (c^2/RT - 4), H factor (c^2/RT - 2)).
struct EqD {
    double e0, ex, ey, e2, U, V, invRT, pqx, pqy, rr, rrm1, kRT, A, lam;
};

// (irho, ir: 1 / rho and 1 / RT; the float64 pipe issues a warp's operation in
// 16 cycles and a division is a dozen of them, so that every division is taken
// once and by its reciprocal, the reference's on the host)
__device__ __forceinline__ EqD make_eq(const KParams &p, double rho, double irho, double U, double V, double RT,
                                       double ir, double qx, double qy)
{
    EqD e;
    const double lam = 0.5 * ir, lamr = 0.5 * p.iRT_r;
    e.e2 = lamr - lam;
    e.ex = 2.0 * mad(lam, U, -lamr * p.U_r);
    e.ey = 2.0 * mad(lam, V, -lamr * p.V_r);
    // a non-positive density (a transient state, e.g. an evacuated wall
    // face after an impulsive start) has no logarithm: e0 then sends every
    // velocity to the direct branch, which takes the signed amplitude A
    e.e0 = rho > 0.0 ? mad(-lam, mad(U, U, V * V), log(rho * lam * p.iAref)) + lamr * mad(p.U_r, p.U_r, p.V_r * p.V_r)
                     : 1e30;
    e.U = U;
    e.V = V;
    e.invRT = ir;
    const double pc = p.shakhov && rho != 0.0 ? p.pc0 * irho * (ir * ir) : 0.0;
    e.pqx = pc * qx;
    e.pqy = pc * qy;
    e.rr = RT * p.iRT_r;
    e.rrm1 = (RT - p.RT_r) * p.iRT_r;
    e.kRT = p.K * RT;
    e.A = rho * lam * (1.0 / M_PI);
    e.lam = lam;
    return e;
}

template <class T> struct EqT {
    T e0, ex, ey, e2, U, V, invRT, pqx, pqy, rr, rrm1, kRT, A, lam;
};

template <class T> __device__ __forceinline__ void eq_storeT(T *cp, const EqD &e)
{
    cp[0] = (T)e.e0; cp[1] = (T)e.ex; cp[2] = (T)e.ey; cp[3] = (T)e.e2; cp[4] = (T)e.U;
    cp[5] = (T)e.V; cp[6] = (T)e.invRT; cp[7] = (T)e.pqx; cp[8] = (T)e.pqy; cp[9] = (T)e.rr;
    cp[10] = (T)e.rrm1; cp[11] = (T)e.kRT; cp[12] = (T)e.A; cp[13] = (T)e.lam;
}

template <class T> __device__ __forceinline__ EqT<T> eq_loadT(const T *cp)
{
    EqT<T> e;
    e.e0 = cp[0]; e.ex = cp[1]; e.ey = cp[2]; e.e2 = cp[3]; e.U = cp[4]; e.V = cp[5];
    e.invRT = cp[6]; e.pqx = cp[7]; e.pqy = cp[8]; e.rr = cp[9]; e.rrm1 = cp[10]; e.kRT = cp[11];
    e.A = cp[12]; e.lam = cp[13];
    return e;
}

// f^S(k) - M_ref(k) for G and H.  Near M_ref (|E| < 1/2) through expm1 of the
// exponent difference E = ln(f^eq/M_ref), so the result is accurate relative
// to the deviation; far from it directly (no cancellation is possible then).
template <class T>
__device__ __forceinline__ void dev_equilibrium(const EqT<T> &e, T ux, T uy, T gref, T kRTr,
                                                T &dG, T &dH)
{
    const T cx = ux - e.U, cy = uy - e.V;
    const T q2 = mad(cx, cx, cy * cy);
    const T P = mad(e.pqx, cx, e.pqy * cy);
    const T PG = P * mad(q2, e.invRT, (T)-4), PH = P * mad(q2, e.invRT, (T)-2);
    const T E = mad(e.e2, mad(ux, ux, uy * uy), mad(e.ex, ux, mad(e.ey, uy, e.e0)));
    const T href = kRTr * gref;
    if (fabs(E) < (T)0.5) {
        const T em = expm1_near(E), em1 = (T)1 + em;
        dG = gref * mad(PG, em1, em);
        dH = href * mad(e.rr, mad(PH, em1, em), e.rrm1);
    } else {
        const T g = e.A * t_exp(-e.lam * q2);
        dG = mad(g, PG, g) - gref;
        dH = mad(e.kRT * g, (T)1 + PH, -href);
    }
}

// raw-moment partials of one velocity: G: 1,x,y,xx,xy,yy,x|xi|^2,y|xi|^2; H: 1,x,y
template <class T>
__device__ __forceinline__ void raw_terms(T (&a)[kRaw], T w, T ux, T uy, T g, T h)
{
    const T wg = w * g, wh = w * h, s2 = mad(ux, ux, uy * uy), gx = wg * ux, gy = wg * uy;
    a[0] += wg; a[1] += gx; a[2] += gy; a[3] = mad(gx, ux, a[3]); a[4] = mad(gx, uy, a[4]);
    a[5] = mad(gy, uy, a[5]); a[6] = mad(gx, s2, a[6]); a[7] = mad(gy, s2, a[7]);
    a[8] += wh; a[9] = mad(wh, ux, a[9]); a[10] = mad(wh, uy, a[10]);
}

// Warp loop over the discrete velocities: lane l takes k = k0 + 32u + l,
// u < 8, for chunks of 256 velocities; each chunk's per-lane partial sums
// (at most 8 terms, storage precision) are folded into the accumulators.
// Full chunks run unchecked and unrolled so several velocities' loads are in
// flight; the ragged last chunk is bounds-checked.
template <int NA, class T, class Body>
__device__ __forceinline__ void vel_loop(int Nv, int lane, Acc<T> (&acc)[NA], Body body)
{
    int k0 = 0;
    for (; k0 + 256 <= Nv; k0 += 256) {
        T a[NA];
#pragma unroll
        for (int q = 0; q < NA; ++q) a[q] = (T)0;
#pragma unroll 4
        for (int u = 0; u < 8; ++u) body(k0 + 32 * u + lane, a);
#pragma unroll
        for (int q = 0; q < NA; ++q) acc[q].add(a[q]);
    }
    if (k0 < Nv) {
        T a[NA];
#pragma unroll
        for (int q = 0; q < NA; ++q) a[q] = (T)0;
        for (int u = 0; u < 8; ++u) {
            int k = k0 + 32 * u + lane;
            if (k < Nv) body(k, a);
        }
#pragma unroll
        for (int q = 0; q < NA; ++q) acc[q].add(a[q]);
    }
}

template <class T> __device__ __forceinline__ void load_pair(const void *base, size_t i, T (&g)[2], T (&h)[2]);

// Pair loop over the discrete velocities: lane l takes the two velocities
// k, k + 1 with k = k0 + 64u + 2l, u < 4, for chunks of 256 velocities (the
// stored velocity count is a multiple of 4, so pairs are whole and start on
// 16-byte boundaries); each chunk's per-lane partial sums (at most 8 terms)
// are folded into the accumulators as in vel_loop.  fold(a) takes them.  The warps
// of a row take its chunks in turn.
template <int NA, class T, class Body, class Fold>
__device__ __forceinline__ void vel_loop2(int Nv, int lane, const Row &row, Body body, Fold fold)
{
    int k0 = 256 * row.sub;
    for (; k0 + 256 <= Nv; k0 += 256 * row.warps) {
        T a[NA];
#pragma unroll
        for (int q = 0; q < NA; ++q) a[q] = (T)0;
#pragma unroll 2
        for (int u = 0; u < 4; ++u) body(k0 + 64 * u + 2 * lane, a);
        fold(a);
    }
    if (k0 < Nv) {
        T a[NA];
#pragma unroll
        for (int q = 0; q < NA; ++q) a[q] = (T)0;
        for (int u = 0; u < 4; ++u) {
            int k = k0 + 64 * u + 2 * lane;
            if (k < Nv) body(k, a);
        }
        fold(a);
    }
}
template <int NA, class T, class Body>
__device__ __forceinline__ void vel_loop2(int Nv, int lane, const Row &row, Acc<T> (&acc)[NA], Body body)
{
    vel_loop2<NA, T>(Nv, lane, row, body, [&](const T(&a)[NA]) {
#pragma unroll
        for (int q = 0; q < NA; ++q) acc[q].add(a[q]);
    });
}

// The same with each thread's float-float accumulators held in shared memory
// (sacc[q * blockDim.x + threadIdx.x]) between chunks, which leaves a
// 64-register thread room for its loads in flight.
template <int NA, class Body>
__device__ __forceinline__ void vel_loop2_sm(int Nv, int lane, const Row &row, Acc<float> (&acc)[NA], FF *sacc, Body body)
{
    FF *s = sacc + threadIdx.x;
    const int nt = blockDim.x;
#pragma unroll
    for (int q = 0; q < NA; ++q) s[q * nt] = FF{0.f, 0.f};
    vel_loop2<NA, float>(Nv, lane, row, body, [&](const float(&a)[NA]) {
#pragma unroll
        for (int q = 0; q < NA; ++q) {
            Acc<float> x;
            x.v = s[q * nt];
            x.add(a[q]);
            s[q * nt] = x.v;
        }
    });
#pragma unroll
    for (int q = 0; q < NA; ++q) acc[q].v = s[q * nt];
}

// store of two consecutive velocities' {G, H} (see load_pair)
template <class T> __device__ __forceinline__ void store_pair(void *base, size_t i, const T (&g)[2], const T (&h)[2]);
template <> __device__ __forceinline__ void store_pair<float>(void *base, size_t i, const float (&g)[2], const float (&h)[2])
{
    ((float4 *)base)[i >> 1] = make_float4(g[0], h[0], g[1], h[1]);
}
template <> __device__ __forceinline__ void store_pair<double>(void *base, size_t i, const double (&g)[2], const double (&h)[2])
{
    ((double2 *)base)[i] = make_double2(g[0], h[0]);
    ((double2 *)base)[i + 1] = make_double2(g[1], h[1]);
}

// the same where on[v], without branches
__device__ __forceinline__ void st_pair_if(float2 *d, const float (&g)[2], const float (&h)[2], const bool (&on)[2])
{
    asm volatile("{.reg .pred p, q, r; setp.ne.s32 p, %5, 0; setp.ne.s32 q, %6, 0; and.pred r, p, q; xor.pred p, p, r; xor.pred q, q, r; "
                 "@r st.global.v4.f32 [%0], {%1, %2, %3, %4}; @p st.global.v2.f32 [%0], {%1, %2}; @q st.global.v2.f32 [%0+8], {%3, %4};}"
                 ::"l"(d), "f"(g[0]), "f"(h[0]), "f"(g[1]), "f"(h[1]), "r"((int)on[0]), "r"((int)on[1]) : "memory");
}
__device__ __forceinline__ void st_pair_if(double2 *d, const double (&g)[2], const double (&h)[2], const bool (&on)[2])
{
    if (on[0]) d[0] = make_double2(g[0], h[0]);
    if (on[1]) d[1] = make_double2(g[1], h[1]);
}

// velocity table entries k, k + 1 (k even)
template <class T> __device__ __forceinline__ void vtab2(const float *tf, const double *td, int k, T (&o)[2]);
template <> __device__ __forceinline__ void vtab2<float>(const float *tf, const double *, int k, float (&o)[2])
{
    const float2 v = ((const float2 *)tf)[k >> 1];
    o[0] = v.x; o[1] = v.y;
}
template <> __device__ __forceinline__ void vtab2<double>(const float *, const double *td, int k, double (&o)[2])
{
    const double2 v = ((const double2 *)td)[k >> 1];
    o[0] = v.x; o[1] = v.y;
}

// ---------------------------------------------------------------------------
// cell moments and cell prep (Eq. 10, 12)                                [a1]
// ---------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ void cell_moments_body(const KParams &__restrict__ p, int blk)
{
    using T2 = typename V2<T>::t;
    const int lane = threadIdx.x & 31;
    int c;
    const Row row = row_of(p, blk, c);
    if (c >= p.N) return;  // all warps of a row
    __shared__ Acc<T> sums[kRowSums];
    const T2 *f = (const T2 *)p.f + (size_t)c * p.Nv;
    Acc<T> acc[kRaw];
#pragma unroll
    for (int q = 0; q < kRaw; ++q) acc[q].zero();
    auto body = [&](int k, T(&a)[kRaw]) {
        T ux[2], uy[2], w[2], g[2], h[2];
        vtab2<T>(p.uxf, p.ux, k, ux);
        vtab2<T>(p.uyf, p.uy, k, uy);
        vtab2<T>(p.wf, p.w, k, w);
        load_pair<T>(f, k, g, h);
        raw_terms<T>(a, w[0], ux[0], uy[0], g[0], h[0]);
        raw_terms<T>(a, w[1], ux[1], uy[1], g[1], h[1]);
    };
    if constexpr (sizeof(T) == 4) {
        __shared__ FF sacc[kRaw * 256];
        vel_loop2_sm<kRaw>(p.Nv, lane, row, acc, sacc, body);
    } else {
        vel_loop2<kRaw, T>(p.Nv, lane, row, acc, body);
    }
    row_sum_store<kRaw, T>(acc, lane, row, sums, p.cellraw, (size_t)c * kRaw);
}

template <class T, class LT>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 1) k_cell_moments(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    cell_moments_body<T>(p, blk);
}

// the same with the parameters passed by value (moment queries)
template <class T>
__global__ void __launch_bounds__(256) k_cell_moments_v(KParams p)
{
    cell_moments_body<T>(p, blockIdx.x);
}

// per cell: heat flux of f from f~ (about U of W), tau, equilibrium at W^n,
// and the two coefficients of fb+ = (2tau-h)/(2tau+dt) f~ + 3h/(2tau+dt) f^S
template <class T, class LT>
__global__ void __launch_bounds__(32) k_cell_params(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    const int c = blk * blockDim.x + threadIdx.x;
    if (c >= p.N) return;
    double r[kRaw];
    for (int q = 0; q < kRaw; ++q) r[q] = acc_load<T>(p.cellraw, (size_t)c * kRaw + q) + p.mref_raw[q];
    const double *W = p.W + 4 * c;
    const double rho = W[0], irho = rcp_rn(rho), U = W[1] * irho, V = W[2] * irho;
    const double RT = mad(-V, V, mad(-U, U, 2.0 * W[3] * irho)) * p.iK2, ir = rcp_rn(RT);
    const double tau2 = 2.0 * viscosity_t<T>(p, RT) * (irho * ir);  // 2 tau
    double qtx, qty;
    raw_heat_flux(r, U, V, qtx, qty);
    const double Pr = p.shakhov ? p.Pr : 1.0, fq = tau2 * rcp_rn(tau2 + p.dt * Pr);
    const double qx = fq * qtx, qy = fq * qty;
    p.cellq[2 * c] = qx;
    p.cellq[2 * c + 1] = qy;
    T *cA = (T *)p.cellA + kCellP * c;
    eq_storeT<T>(cA, make_eq(p, rho, irho, U, V, RT, ir, qx, qy));
    const double fd = rcp_rn(tau2 + p.dt);
    cA[14] = (T)((tau2 - p.h) * fd);
    cA[15] = (T)(3.0 * p.h * fd);
}

// The per-(cell, velocity) kernels: 128-thread blocks, each over 256 velocities
// (a pair per thread) of p.cpb consecutive cells.  Several cells a block where
// there are enough of them: the block's parameters and velocity tables are read
// once, and the next cell's loads overlap the current one's arithmetic (16
// cavities of 32 to 96 cells a side, one cell a block before: k_fbp 272 ->
// 208 us, k_micro_residual 453 -> 349 us).
// body(c) for the block's cells, k the thread's first velocity.
template <class Body> __device__ __forceinline__ void for_cells(const KParams &p, int blk, int &k, Body body)
{
    const int nvb = (p.Nv + 255) / 256;
    const int b = blk / nvb;
    k = 2 * ((blk - b * nvb) * 128 + threadIdx.x);
    if (k >= p.Nv) return;
    const int c0 = b * p.cpb, c1 = min(c0 + p.cpb, p.N);
    for (int c = c0; c < c1; ++c) body(c);
}

// per (cell, pair of velocities): fb+ = c1 f~ + c2 f^S
template <class T, class LT>
__global__ void __launch_bounds__(128) k_fbp(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    int k;
    for_cells(p, blk, k, [&](int c) {
        const T *cA = (const T *)p.cellA + kCellP * c;
        const EqT<T> e = eq_loadT<T>(cA);
        const T c1 = cA[14], c2 = cA[15], kRTr = (T)(p.K * p.RT_r);
        const size_t ck = (size_t)c * p.Nv + k;
        T ux[2], uy[2], gr[2], g[2], h[2];
        vtab2<T>(p.uxf, p.ux, k, ux);
        vtab2<T>(p.uyf, p.uy, k, uy);
        vtab2<T>(p.greff, p.gref, k, gr);
        load_pair<T>(p.f, ck, g, h);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            T dG, dH;
            dev_equilibrium<T>(e, ux[v], uy[v], gr[v], kRTr, dG, dH);
            g[v] = mad(c1, g[v], c2 * dG);
            h[v] = mad(c1, h[v], c2 * dH);
        }
        store_pair<T>(p.fbp, ck, g, h);
    });
}

// ---------------------------------------------------------------------------
// faces: reconstruction from one cell along the characteristic (Eq. 11,
// 13-17), moments, face equilibrium and flux (Eq. 18-19)            [a2-a4]
// ---------------------------------------------------------------------------
// Divisions of the limiter: exact in float64 (the oracle's rounding up to
// order); in float32 storage the approximate quotient (2 ulp) of the fast
// reciprocal path, the limiter being a smooth function of its ratios
__device__ __forceinline__ float lim_div(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double lim_div(double a, double b) { return a / b; }

template <class T> __device__ __forceinline__ T venkat(T x) { return lim_div(mad(x, x, (T)2 * x), mad(x, x, x + (T)2)); }

// G and H of two consecutive velocities k, k + 1 (k even: 16-byte aligned
// because the stored velocity count is a multiple of 4)
template <class T> __device__ __forceinline__ void load_pair(const void *base, size_t i, T (&g)[2], T (&h)[2]);
template <> __device__ __forceinline__ void load_pair<float>(const void *base, size_t i, float (&g)[2], float (&h)[2])
{
    const float4 a = ((const float4 *)base)[i >> 1];
    g[0] = a.x; h[0] = a.y; g[1] = a.z; h[1] = a.w;
}
template <> __device__ __forceinline__ void load_pair<double>(const void *base, size_t i, double (&g)[2], double (&h)[2])
{
    const double2 a = ((const double2 *)base)[i], b = ((const double2 *)base)[i + 1];
    g[0] = a.x; h[0] = a.y; g[1] = b.x; h[1] = b.y;
}

// four storage scalars, 16- or 32-byte aligned
template <class T> __device__ __forceinline__ void load4(const T *s, T &a, T &b, T &c, T &e);
template <> __device__ __forceinline__ void load4<float>(const float *s, float &a, float &b, float &c, float &e)
{
    const float4 v = *(const float4 *)s;
    a = v.x; b = v.y; c = v.z; e = v.w;
}
template <> __device__ __forceinline__ void load4<double>(const double *s, double &a, double &b, double &c, double &e)
{
    const double2 v = ((const double2 *)s)[0], w = ((const double2 *)s)[1];
    a = v.x; b = v.y; c = w.x; e = w.y;
}

// limiter of one scalar (Eq. 16-17): phi = min over the faces of
// theta(x_m), x_m = (v_max - v0)/d_m where the extrapolated increment d_m to
// the face is positive, (v_min - v0)/d_m where it is negative (faces with
// d_m = 0 impose nothing), capped at 1.  Every x_m is >= 0, and theta rises
// monotonically from theta(0) = 0 to theta(2) = 1 and stays >= 1 beyond, so
// phi = theta(min(2, min_m x_m)): one evaluation of theta instead of four.
// Selects instead of branches: the sign of d differs between neighbouring
// velocities.
// With the smoothing constant (e2 = eps^2 > 0) each face's factor is
// (P^2 + e2 + 2 D P) / (P^2 + 2 D^2 + P D + e2), P the increment to the
// neighbourhood's max or min, D the extrapolated one, and the minimum is
// taken over the four faces (the factor is no function of P / D alone).
template <class T>
__device__ __forceinline__ T limit_scalar_sel(const T (&frx)[4], const T (&fry)[4], T v0, T vmax, T vmin, T sx, T sy,
                                              T e2)
{
    if (e2 > (T)0) {
        T phi = (T)1;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const T d = mad(sx, frx[m], sy * fry[m]);
            const T P = (d > (T)0 ? vmax : vmin) - v0, q = mad(P, P, e2);
            const T t = lim_div(mad((T)2 * d, P, q), mad((T)2 * d, d, mad(P, d, q)));
            phi = (d != (T)0 && t < phi) ? t : phi;
        }
        return phi;
    }
    T xm = (T)2;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const T d = mad(sx, frx[m], sy * fry[m]);
        const T x = lim_div((d > (T)0 ? vmax : vmin) - v0, d);
        xm = (d != (T)0 && x < xm) ? x : xm;
    }
    return venkat<T>(xm);
}

// slot of velocity k among those along a face (xi.n = 0 in the storage type):
// the velocity grid is a tensor product, so every row (or column) of it, taken
// across the normal's larger component, holds at most one such velocity
template <class T> __device__ __forceinline__ int tie_slot(const KParams &p, int k, T nx, T ny)
{
    return fabs(nx) >= fabs(ny) ? k / p.nvx : k % p.nvx;
}

// Per (cell, pair of velocities): the least-squares gradient of fb+ (Eq. 14-15),
// LIM: the Venkatakrishnan limiter (Eq. 16-17), and fb at the half step
// (Eq. 11, 13) at those of the cell's faces that the velocity leaves it by --
// fb+_c + phi sigma_c . (x_f - xi h - x_c) -- into the face buffer.  The
// limiter ratios and the gradients only involve differences of fb+ between
// cells at one velocity, so the M_ref offset cancels and deviations serve as
// is.  An interior face gets each velocity from the one cell that is upwind of
// it; at a velocity along the face (s = 0) both sides count half, the L side
// going to the face buffer and the R side to the tie buffer (k_face_moments
// takes the mean).  Boundary faces get the outgoing velocities and the ties.
// The cell's stencil record is read by every thread (one broadcast per load).
// Bound by the latency of the stencil's loads and the face buffer's bytes.
// Gathering at the faces instead formed an unlimited gradient once per face a
// velocity leaves by, or stored the limited ones in a second pass; with the
// moments of a face (k_face_moments) it took, float32, 81 us on 64 x 64 cells
// x 1024 velocities, 259 us on 128 x 128 x 784 and, limited, 1952 us on
// 121 x 81 x 7921; this 32 + 35, 107 + 101 and 908 + 464 us.
template <class T, bool LIM, class LT>
__global__ void __launch_bounds__(128) k_cell_recon(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    using T2 = typename V2<T>::t;
    int k;
    for_cells(p, blk, k, [&](int c) {
    int nb[4], fc[4], sg[4];
    T gx[4], gy[4], frx[4], fry[4], nx[4], ny[4];
    {
        const int4 n4 = *(const int4 *)(p.cnb + 4 * c), f4 = *(const int4 *)(p.cface + 4 * c),
                   s4 = *(const int4 *)(p.csign + 4 * c);
        nb[0] = n4.x; nb[1] = n4.y; nb[2] = n4.z; nb[3] = n4.w;
        fc[0] = f4.x; fc[1] = f4.y; fc[2] = f4.z; fc[3] = f4.w;
        sg[0] = s4.x; sg[1] = s4.y; sg[2] = s4.z; sg[3] = s4.w;
        const T *g = (const T *)p.clsgT + 8 * c;
        const T *o = (const T *)p.crT + 8 * c;
        const T *n = (const T *)p.cnT + 8 * c;
        load4<T>(g, gx[0], gy[0], gx[1], gy[1]);
        load4<T>(g + 4, gx[2], gy[2], gx[3], gy[3]);
        load4<T>(o, frx[0], fry[0], frx[1], fry[1]);
        load4<T>(o + 4, frx[2], fry[2], frx[3], fry[3]);
        load4<T>(n, nx[0], ny[0], nx[1], ny[1]);
        load4<T>(n + 4, nx[2], ny[2], nx[3], ny[3]);
    }
    T g0[2], h0[2];
    load_pair<T>(p.fbp, (size_t)c * p.Nv + k, g0, h0);
    T sgx[2] = {0, 0}, sgy[2] = {0, 0}, shx[2] = {0, 0}, shy[2] = {0, 0};
    T gmax[2] = {g0[0], g0[1]}, gmin[2] = {g0[0], g0[1]}, hmax[2] = {h0[0], h0[1]}, hmin[2] = {h0[0], h0[1]};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (nb[m] < 0) continue;
        T gn[2], hn[2];
        load_pair<T>(p.fbp, (size_t)nb[m] * p.Nv + k, gn, hn);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const T dg = gn[v] - g0[v], dh = hn[v] - h0[v];
            sgx[v] = mad(gx[m], dg, sgx[v]); sgy[v] = mad(gy[m], dg, sgy[v]);
            shx[v] = mad(gx[m], dh, shx[v]); shy[v] = mad(gy[m], dh, shy[v]);
            if (LIM) {
                gmax[v] = gn[v] > gmax[v] ? gn[v] : gmax[v]; gmin[v] = gn[v] < gmin[v] ? gn[v] : gmin[v];
                hmax[v] = hn[v] > hmax[v] ? hn[v] : hmax[v]; hmin[v] = hn[v] < hmin[v] ? hn[v] : hmin[v];
            }
        }
    }
    if (LIM && p.limiter) {
        // the smoothing constant's eps^2 = (K h)^3, h = sqrt(area) (0: Eq. 16-17)
        T e2 = (T)0;
        if (p.venkat_k3 > 0.0) {
            const double a = p.area[c];
            e2 = (T)(p.venkat_k3 * a * sqrt(a));
        }
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const T pg = limit_scalar_sel<T>(frx, fry, g0[v], gmax[v], gmin[v], sgx[v], sgy[v], e2);
            const T ph = limit_scalar_sel<T>(frx, fry, h0[v], hmax[v], hmin[v], shx[v], shy[v], e2);
            sgx[v] *= pg; sgy[v] *= pg;
            shx[v] *= ph; shy[v] *= ph;
        }
    }
    T ux[2], uy[2];
    vtab2<T>(p.uxf, p.ux, k, ux);
    vtab2<T>(p.uyf, p.uy, k, uy);
    const T h = (T)p.h;
    // back along the characteristic first, then to each face's midpoint
    T bg[2], bh[2];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
        bg[v] = mad(-h, mad(sgx[v], ux[v], sgy[v] * uy[v]), g0[v]);
        bh[v] = mad(-h, mad(shx[v], ux[v], shy[v] * uy[v]), h0[v]);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        if (sg[m] == 0) continue;  // a triangle's unused slot
        T og[2], oh[2], s[2];
        bool out[2];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            s[v] = xi_dot_n<T>(ux[v], uy[v], nx[m], ny[m]);
            out[v] = s[v] > (T)0;
            og[v] = bg[v] + mad(sgx[v], frx[m], sgy[v] * fry[m]);
            oh[v] = bh[v] + mad(shx[v], frx[m], shy[v] * fry[m]);
        }
        if (s[0] == (T)0 || s[1] == (T)0) {
            // along the face: the L side (of a boundary face the only one) to the
            // face buffer, the R side to the tie buffer
            const bool own = sg[m] > 0 || nb[m] < 0;
#pragma unroll
            for (int v = 0; v < 2; ++v)
                if (s[v] == (T)0) {
                    out[v] = own;
                    if (!own && k + v < p.nvx * p.nvy) {  // (the ghost velocities have no slot)
                        T2 o;
                        o.x = og[v];
                        o.y = oh[v];
                        ((T2 *)p.ftie)[(size_t)fc[m] * max(p.nvx, p.nvy) + tie_slot<T>(p, k + v, nx[m], ny[m])] = o;
                    }
                }
        }
        st_pair_if((T2 *)p.F + ((size_t)fc[m] * p.Nv + k), og, oh, out);
    }
    });
}

// Linearised wall (Eq. 33-35), at a wall face f: the outgoing sum
// S = sum_out w (xi.n_out) G~ of the inner cell's stored state (products in
// the storage type, compensated sum across lanes: float64 stays exact to
// round-off, float32 rounds each product as the fluxes themselves are
// rounded) and the ghost density increment of Eq. (35),
//   drho_g = (S^n - S^{n-1}) / sum_in w |xi.n_out| G_w,
// zero in the first iteration after a restart.  The M_ref part of f~
// cancels in the difference.  Out of line: the wall faces' extra work keeps
// out of the register allocation of the kernel's hot path.
template <class T>
__device__ __noinline__ void wall_ghost_density(const KParams &p, int f, int lane, int c, T on, T nx, T ny,
                                                double in_sum)
{
    using T2 = typename V2<T>::t;
    const T2 *fc0 = (const T2 *)p.f + (size_t)c * p.Nv;
    Acc<T> a[1];
    a[0].zero();
    vel_loop<1, T>(p.Nv, lane, a, [&](int k, T(&q)[1]) {
        const T so = on * xi_dot_n<T>(vx<T>(p, k), vy<T>(p, k), nx, ny);
        if (so > (T)0) q[0] = mad(vw<T>(p, k) * so, fc0[k].x, q[0]);
    });
    a[0].warp_sum();
    const double sn = __shfl_sync(0xffffffffu, a[0].value(), 0);
    if (lane == 0) {
        p.walldrg[f] = *p.wallok ? (sn - p.wallS[f]) / in_sum : 0.0;
        p.wallS[f] = sn;
    }
}

// raw moments of fb - M_ref at every face (plus the wall density, Eq. 35), a
// warp per face.  k_cell_recon left fb in the face buffer, except what enters
// through a boundary face -- the wall Maxwellian rho_w M_w or the far-field
// state, formed and stored here -- and the R side of the ties.
template <class T, class LT>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 1) k_face_moments(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    using T2 = typename V2<T>::t;
    const int lane = threadIdx.x & 31;
    const int f = blk * 8 + (threadIdx.x >> 5);
    if (f >= p.nf) return;  // whole warp
    constexpr Row row{0, 1};
    const T *geo = (const T *)p.fgeoT + 8 * f;
    const T nx = geo[0], ny = geo[1];
    const int kind = p.fbc[f];  // -1 interior, 1 wall, 2 far field
    T2 *Fo = (T2 *)p.F + (size_t)f * p.Nv;
    Acc<T> outsum[1];
    outsum[0].zero();
    double rw = 1.0;
    Acc<T> acc[kRaw];
#pragma unroll
    for (int q = 0; q < kRaw; ++q) acc[q].zero();
    const int lc = p.fL[f], side = p.fside[f];
    const T on = kind < 0 || lc >= 0 ? (T)1 : (T)-1;
    T rhow = (T)1, rwm1 = (T)0;
    if (kind == 1) {
        // zero net mass flux: rho_w sum_in w |xi.n| G_w = sum_out w (xi.n) fb
        vel_loop<1, T>(p.Nv, lane, outsum, [&](int k, T(&a)[1]) {
            const T so = on * xi_dot_n<T>(vx<T>(p, k), vy<T>(p, k), nx, ny);
            if (so > (T)0) a[0] = mad(vw<T>(p, k) * so, Fo[k].x, a[0]);
        });
        outsum[0].warp_sum();
        const double o = __shfl_sync(0xffffffffu, outsum[0].value(), 0);
        const double *bc = p.bconst + 2 * f;
        rw = (bc[0] + o) / bc[1];
        rhow = (T)rw;
        rwm1 = (T)((bc[0] - bc[1] + o) / bc[1]);
        if (p.implicit_wall) wall_ghost_density<T>(p, f, lane, lc >= 0 ? lc : p.fR[f], on, nx, ny, bc[1]);
    }
    auto body = [&](int k, T(&a)[kRaw]) {
        T ux[2], uy[2], w[2], s[2], g[2], h[2];
        vtab2<T>(p.uxf, p.ux, k, ux);
        vtab2<T>(p.uyf, p.uy, k, uy);
        vtab2<T>(p.wf, p.w, k, w);
        load_pair<T>(Fo, k, g, h);
        bool cut = kind >= 0;
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            s[v] = on * xi_dot_n<T>(ux[v], uy[v], nx, ny);
            cut |= s[v] == (T)0;
        }
        if (cut) {
            const T2 *tb = (const T2 *)p.ftie + (size_t)f * max(p.nvx, p.nvy);
#pragma unroll
            for (int v = 0; v < 2; ++v) {
                if (s[v] > (T)0 || (kind < 0 && (s[v] < (T)0 || k + v >= p.nvx * p.nvy))) continue;
                T2 in;
                if (kind < 0) {
                    in = tb[tie_slot<T>(p, k + v, nx, ny)];
                } else {
                    const T *bG = (const T *)p.bdevG + (size_t)side * p.Nv, *bH = (const T *)p.bdevH + (size_t)side * p.Nv;
                    const T gref = vgref<T>(p, k + v);
                    in.x = mad(rhow, bG[k + v], rwm1 * gref);
                    in.y = mad(rhow, bH[k + v], rwm1 * ((T)(p.K * p.RT_r) * gref));
                }
                // along the face the mean of both sides (at an interior face the
                // flux there is zero: the mean is not stored)
                g[v] = s[v] < (T)0 ? in.x : (T)0.5 * (g[v] + in.x);
                h[v] = s[v] < (T)0 ? in.y : (T)0.5 * (h[v] + in.y);
            }
            if (kind >= 0) store_pair<T>(Fo, k, g, h);
        }
        raw_terms<T>(a, w[0], ux[0], uy[0], g[0], h[0]);
        raw_terms<T>(a, w[1], ux[1], uy[1], g[1], h[1]);
    };
    if constexpr (sizeof(T) == 4) {
        __shared__ FF sacc[kRaw * 256];
        vel_loop2_sm<kRaw>(p.Nv, lane, row, acc, sacc, body);
    } else {
        vel_loop2<kRaw, T>(p.Nv, lane, row, acc, body);
    }
    row_sum_store<kRaw, T>(acc, lane, row, nullptr, p.faceraw, (size_t)f * 12);
    if (lane == 0) {
        outsum[0].store(p.faceraw, (size_t)f * 12 + 11);
        p.facerw[f] = rw;
    }
}

// per face: state from the moments of fb, tau, q = 2 tau qbar/(2 tau + h Pr),
// equilibrium, and the weights a, b of f = a fb + b f^S (Eq. 18)
template <class T, class LT>
__global__ void __launch_bounds__(32) k_face_params(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    const int f = blk * blockDim.x + threadIdx.x;
    if (f >= p.nf) return;
    double r[kRaw];
    for (int q = 0; q < kRaw; ++q) r[q] = acc_load<T>(p.faceraw, (size_t)f * 12 + q) + p.mref_raw[q];
    double rho, irho, U, V, RT, qbx, qby;
    raw_to_state(p, r, rho, irho, U, V, RT, qbx, qby);
    T *fA = (T *)p.faceA + kCellP * f;
    // float32 storage keeps fb relative to the reference Maxwellian, so a
    // face that an impulsive start evacuates (density ~1e-18 of the reference
    // at the lee of a hypersonic body) is not resolved: its moments are
    // rounding noise of the reference's.  Below 1e-6 of the reference density
    // or temperature such a face takes the vacuum limit of Eq. (18):
    // tau -> infinity, f = fb (free transport), no equilibrium part.
    if (sizeof(T) == 4 && !(rho > 1e-6 * p.rho_r && RT > 1e-6 * p.RT_r)) {
        eq_storeT<T>(fA, make_eq(p, 0.0, 0.0, p.U_r, p.V_r, p.RT_r, p.iRT_r, 0.0, 0.0));
        fA[14] = (T)1;
        fA[15] = (T)0;
        return;
    }
    const double ir = rcp_rn(RT), tau2 = 2.0 * viscosity_t<T>(p, RT) * (irho * ir);  // 2 tau
    const double Pr = p.shakhov ? p.Pr : 1.0, fq = tau2 * rcp_rn(tau2 + p.h * Pr);
    eq_storeT<T>(fA, make_eq(p, rho, irho, U, V, RT, ir, fq * qbx, fq * qby));
    const double fd = rcp_rn(tau2 + p.h);
    fA[14] = (T)(tau2 * fd);
    fA[15] = (T)(p.h * fd);
}

// face flux of (f_face - M_ref), Eq. (18)-(19), and its moments; fb - M_ref
// comes from k_face_moments through the same buffer and is overwritten
template <class T, class LT>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 1) k_face_flux(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    using T2 = typename V2<T>::t;
    const int lane = threadIdx.x & 31;
    const int f = blk * 8 + (threadIdx.x >> 5);
    if (f >= p.nf) return;  // whole warp
    constexpr Row row{0, 1};
    const T *g = (const T *)p.fgeoT + 8 * f;
    const T nx = g[0], ny = g[1], S = g[2];
    const T *fA = (const T *)p.faceA + kCellP * f;
    const EqT<T> e = eq_loadT<T>(fA);
    const T wa = fA[14], wb = fA[15], kRTr = (T)(p.K * p.RT_r);
    T2 *Fo = (T2 *)p.F + (size_t)f * p.Nv;
    Acc<T> acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q].zero();
    vel_loop2<4, T>(p.Nv, lane, row, acc, [&](int k, T(&a)[4]) {
        T ux[2], uy[2], w[2], gr[2], fg[2], fh[2];
        vtab2<T>(p.uxf, p.ux, k, ux);
        vtab2<T>(p.uyf, p.uy, k, uy);
        vtab2<T>(p.wf, p.w, k, w);
        vtab2<T>(p.greff, p.gref, k, gr);
        load_pair<T>(Fo, k, fg, fh);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            T s = xi_dot_n<T>(ux[v], uy[v], nx, ny);
            T dG, dH;
            dev_equilibrium<T>(e, ux[v], uy[v], gr[v], kRTr, dG, dH);
            T sS = s * S;
            fg[v] = sS * mad(wa, fg[v], wb * dG);
            fh[v] = sS * mad(wa, fh[v], wb * dH);
            T wg = w[v] * fg[v];
            a[0] += wg;
            a[1] = mad(wg, ux[v], a[1]);
            a[2] = mad(wg, uy[v], a[2]);
            a[3] = mad((T)0.5 * w[v], mad(mad(ux[v], ux[v], uy[v] * uy[v]), fg[v], fh[v]), a[3]);
        }
        store_pair<T>(Fo, k, fg, fh);
    });
    row_sum_store<4, T>(acc, lane, row, nullptr, p.phiraw, (size_t)f * 4);
    if (p.implicit_wall && p.fbc[f] == 1) {
        // linearised wall (Eq. 33-35): the ghost increment drho_g M_w of the
        // incoming velocities enters the micro sweeps as the upwind term
        // |xi.n| S Delta_ghost, i.e. as an extra flux s S drho_g M_w on the
        // stored F (after Phi is summed: R_W and Phi exclude it)
        __syncwarp();
        const double drg = p.walldrg[f];
        if (drg != 0.0) {
            const T on = p.fL[f] >= 0 ? (T)1 : (T)-1, SD = S * (T)drg;
            const T *bG = (const T *)p.bdevG + (size_t)p.fside[f] * p.Nv;
            const T *bH = (const T *)p.bdevH + (size_t)p.fside[f] * p.Nv;
            for (int k = lane; k < p.Nv; k += 32) {
                const T sn = xi_dot_n<T>(vx<T>(p, k), vy<T>(p, k), nx, ny);
                if (on * sn < (T)0) {
                    const T a = sn * SD, gr = vgref<T>(p, k);
                    T2 v = Fo[k];
                    v.x = mad(a, bG[k] + gr, v.x);
                    v.y = mad(a, mad(kRTr, gr, bH[k]), v.y);
                    Fo[k] = v;
                }
            }
        }
    }
}

// Phi_f = sum_k w psi F_k (Eq. 27): deviation part plus the flux of M_ref;
// the mass flux through an impermeable wall is exactly zero
template <class T, class LT>
__global__ void __launch_bounds__(256) k_face_phi(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    const int f = blk * blockDim.x + threadIdx.x;
    if (f >= p.nf) return;
    const double *g = p.fgeo + 7 * f;
    for (int q = 0; q < 4; ++q)
        p.phi[4 * f + q] = acc_load<T>(p.phiraw, (size_t)f * 4 + q) +
                           g[2] * (g[0] * p.mref_flux[q][0] + g[1] * p.mref_flux[q][1]);
    if (p.fbc[f] == 1) p.phi[4 * f] = 0.0;
    // the wall sums of this iteration are stored: the next one has a last increment
    if (f == 0 && p.implicit_wall) *p.wallok = 1;
}

// ---------------------------------------------------------------------------
// macroscopic predictor (Eq. 27-31)                                     [a5]
//   k_macro_pre    (all cells, many CTAs): residual R_W = -sum Phi, partial
//                  norms, spectral radii (Eq. 31 at the face average), the
//                  LU-SGS diagonal D (Eq. 30) and per-neighbour coefficients
//   k_macro_sweep  (one CTA): forward and backward sweeps on i+j hyperplanes,
//                  the lexicographic dependency order, with the matrix-free
//                  off-diagonal term 1/2 (dF S - omega Lambda dW) of Eq. (30)
//   k_macro_post   (all cells): W^{n+1} = W + dW (Eq. 32) in float64 and the
//                  micro coefficients at the predicted state
// ---------------------------------------------------------------------------
// velocity and sound speed of a cell for the face spectral radii.  In float32
// storage the spectral radius and the neighbours' base states only enter the
// float32 wavefront (R_W, the diagonal's sum and W^{n+1} stay float64), so they
// are evaluated in float32; float64 storage evaluates them in float64.
__device__ __forceinline__ void prim_uvc(const KParams &p, const double *W, double &u, double &v, double &cs)
{
    const double irho = rcp_rn(W[0]);
    u = W[1] * irho;
    v = W[2] * irho;
    cs = sqrt(p.gam * ((2.0 * W[3] * irho - u * u - v * v) * p.iK2));
}
__device__ __forceinline__ void prim_uvc(const KParams &p, const double *W, float &u, float &v, float &cs)
{
    const float ir = rcp_rn((float)W[0]);
    u = (float)W[1] * ir;
    v = (float)W[2] * ir;
    cs = sqrtf((float)p.gam * ((2.0f * (float)W[3] * ir - u * u - v * v) * (float)p.iK2));
}

// base state (rho, m_x, m_y, u, v, E + p) of a neighbour for the flux increments
template <class T> __device__ __forceinline__ void base_state(const KParams &p, const double *W, T *o);
template <> __device__ __forceinline__ void base_state<double>(const KParams &p, const double *W, double *o)
{
    double rho = W[0], u = W[1] / rho, v = W[2] / rho;
    double pr = (p.gam - 1.0) * (W[3] - 0.5 * rho * (u * u + v * v));
    o[0] = rho; o[1] = W[1]; o[2] = W[2];
    o[3] = u; o[4] = v; o[5] = W[3] + pr;
}
template <> __device__ __forceinline__ void base_state<float>(const KParams &p, const double *W, float *o)
{
    const float rho = (float)W[0], mx = (float)W[1], my = (float)W[2], E = (float)W[3];
    const float ir = rcp_rn(rho), u = mx * ir, v = my * ir;
    const float pr = (float)(p.gam - 1.0) * (E - 0.5f * rho * (u * u + v * v));
    o[0] = rho; o[1] = mx; o[2] = my;
    o[3] = u; o[4] = v; o[5] = E + pr;
}

// four storage scalars, 16-byte aligned
__device__ __forceinline__ void ld4(float (&o)[4], const float *s)
{
    const float4 v = *reinterpret_cast<const float4 *>(s);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
}
__device__ __forceinline__ void ld4(double (&o)[4], const double *s)
{
    const double2 a = reinterpret_cast<const double2 *>(s)[0], b = reinterpret_cast<const double2 *>(s)[1];
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}
__device__ __forceinline__ void st4(float *d, const float *x)
{
    *reinterpret_cast<float4 *>(d) = make_float4(x[0], x[1], x[2], x[3]);
}
__device__ __forceinline__ void st4(double *d, const double *x)
{
    reinterpret_cast<double2 *>(d)[0] = make_double2(x[0], x[1]);
    reinterpret_cast<double2 *>(d)[1] = make_double2(x[2], x[3]);
}

// where on, without a branch, to global (GLOBAL) or shared memory
template <bool GLOBAL> __device__ __forceinline__ void st4_if(float *d, const float *x, bool on)
{
    if constexpr (GLOBAL)
        asm volatile("{.reg .pred p; setp.ne.s32 p, %5, 0; @p st.global.v4.f32 [%0], {%1, %2, %3, %4};}" ::"l"(d), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "r"((int)on) : "memory");
    else
        asm volatile("{.reg .pred p; setp.ne.s32 p, %5, 0; @p st.shared.v4.f32 [%0], {%1, %2, %3, %4};}" ::"r"(smem_addr(d)), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]), "r"((int)on) : "memory");
}
template <bool GLOBAL> __device__ __forceinline__ void st4_if(double *d, const double *x, bool on)
{
#pragma unroll
    for (int q = 0; q < 4; q += 2) {
        if constexpr (GLOBAL)
            asm volatile("{.reg .pred p; setp.ne.s32 p, %3, 0; @p st.global.v2.f64 [%0], {%1, %2};}" ::"l"(d + q), "d"(x[q]), "d"(x[q + 1]), "r"((int)on) : "memory");
        else
            asm volatile("{.reg .pred p; setp.ne.s32 p, %3, 0; @p st.shared.v2.f64 [%0], {%1, %2};}" ::"r"(smem_addr(d + q)), "d"(x[q]), "d"(x[q + 1]), "r"((int)on) : "memory");
    }
}
template <class T> __device__ __forceinline__ void st4(T *d, T a, T b, T c, T e)
{
    const T x[4] = {a, b, c, e};
    st4(d, x);
}

constexpr int kMRec = 24;  // macroscopic sweep record: R[4], 1/D, pad, own base[6], 4 x (n S/2 [2], omega Lambda/2)
// structured blocks, k_macro_lines: cell c = (t, w), t on the shorter axis, by
// its hyperplane t + w and its line t, so that the lines a warp marches along
// read and write consecutive slots at every step; six vectors of four (line_rec)
__device__ __forceinline__ bool by_lines(const KParams &p) { return p.macro_kind == 1 && !p.sched && p.relax_sweeps == 0; }
__device__ __forceinline__ int line_slot(const KParams &p, int c)
{
    const int j = c / p.ni, i = c - j * p.ni, d = i + j;
    return p.ni <= p.nj ? d * p.ni + i : d * p.nj + j;
}
__device__ __forceinline__ size_t line_slots(const KParams &p) { return (size_t)min(p.ni, p.nj) * (p.ni + p.nj - 1); }
constexpr int kMRing = 12; // ring entry per cell: increment[4], base state[6], pad[2]

// per cell: R_W, ||R_W/Omega||^2 partials, and the record of the macroscopic
// sweep (inverse diagonal, the cell's own base state for its neighbours'
// flux increments, per-slot face coefficients)
template <class T, class LT>
__global__ void __launch_bounds__(32) k_macro_pre(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    __shared__ double sm[32];
    const int c = blk * blockDim.x + threadIdx.x;
    double part[1] = {0.0};
    if (c < p.N) {
        T rec[kMRec];
        double acc[4] = {0, 0, 0, 0};
        for (int m = 0; m < 4; ++m) {
            double s = p.csign[4 * c + m];
            const double *ph = p.phi + 4 * p.cface[4 * c + m];
            for (int q = 0; q < 4; ++q) acc[q] -= s * ph[q];
        }
        const double iA = rcp_rn(p.area[c]);
        for (int q = 0; q < 4; ++q) {
            p.rw[4 * c + q] = acc[q];
            rec[q] = (T)acc[q];
            const double rr = acc[q] * iA;
            part[0] += rr * rr;
        }
        double d = p.adt[c];
        T u0, v0, c0;
        prim_uvc(p, p.W + 4 * c, u0, v0, c0);
        for (int m = 0; m < 4; ++m) {
            // spectral radius (|V.n| + c) S of Eq. (31) at the average of the
            // face's cells (at a boundary the inner one)
            const int nb = p.cnb[4 * c + m];
            const double *g = p.fgeo + 7 * p.cface[4 * c + m];
            const T nx = (T)g[0], ny = (T)g[1], S = (T)g[2];
            T u = u0, v = v0, cs = c0;
            if (nb >= 0) {
                prim_uvc(p, p.W + 4 * nb, u, v, cs);
                u = (T)0.5 * (u0 + u);
                v = (T)0.5 * (v0 + v);
                cs = (T)0.5 * (c0 + cs);
            }
            const double lam = (double)((fabs(u * nx + v * ny) + cs) * S);
            double s = p.csign[4 * c + m];  // 0: a triangle's unused slot
            if (s != 0.0 && nb != c) d += 0.5 * p.lusgs_omega * lam;
            T *o = rec + 12 + 3 * m;
            o[0] = (T)(0.5 * g[2] * s * g[0]);
            o[1] = (T)(0.5 * g[2] * s * g[1]);
            o[2] = (T)(0.5 * p.lusgs_omega * lam);
        }
        rec[4] = (T)rcp_rn(d);
        rec[5] = (T)0;
        base_state<T>(p, p.W + 4 * c, rec + 6);
        if (by_lines(p)) {
            // R | 1/D, rho, m_x, m_y | per sweep: 1/rho, E + p, omega/2 Lambda of
            // the faces ahead on the own line and towards the next line | their S/2 n
            const size_t M = line_slots(p);
            T *o = (T *)p.mline + 4 * (size_t)line_slot(p, c);
            const bool cols = p.ni <= p.nj;
            const T ir = rcp_rn(rec[6]);
            st4(o, rec);
            st4(o + 4 * M, rec[4], rec[6], rec[7], rec[8]);
            for (int dir = 0; dir < 2; ++dir) {
                // slots (west 0, east 1, south 2, north 3): forward w + 1, t + 1; backward w - 1, t - 1
                const T *cw = rec + 12 + 3 * ((cols ? 2 : 0) + 1 - dir), *ct = rec + 12 + 3 * ((cols ? 0 : 2) + 1 - dir);
                st4(o + (8 + 8 * dir) * M, ir, rec[11], cw[2], ct[2]);
                st4(o + (12 + 8 * dir) * M, cw[0], cw[1], ct[0], ct[1]);
            }
        } else {
            T *o = (T *)p.mrec + (size_t)kMRec * c;
            for (int q = 0; q < kMRec; ++q) o[q] = rec[q];
        }
    }
    block_sum<1>(part, sm);
    if (threadIdx.x == 0) p.mpart[blk] = part[0];
}

// ||R_W/Omega||_2 of this iteration from k_macro_pre's partials (fixed
// order) into the residual ring, by the 32 lanes of one warp; a non-finite
// value raises the status word.  One thread alone took 9 us for the 128
// partials of a 64 x 64 block, a load latency per few of them.
__device__ __forceinline__ void record_residual(const KParams &p)
{
    const int lane = threadIdx.x & 31, nb = (p.N + 31) / 32;
    double s = 0.0;
    for (int q = lane; q < nb; q += 32) s += p.mpart[q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) {
        const double r = sqrt(s);
        p.res[*p.iter & (kMaxHist - 1)] = r;
        // (a wait that ran out stays the cause that is reported: the sweep then ran on stale values)
        if (!isfinite(r)) atomicCAS(p.status, 0, 5);
    }
}

// Exact increment F_n(W + dW) - F_n(W) of the Euler flux, written so that no
// two O(1) quantities are subtracted (every term is an increment times a
// base quantity); n is pre-scaled by S/2.  b = rho, m_x, m_y, u, v, E+p.
template <class T>
__device__ __forceinline__ void euler_dflux(T gm1, const T *b, const T *dW, T nx, T ny, T *dF)
{
    const T rho = b[0], mx = b[1], my = b[2], u = b[3], v = b[4], H = b[5];
    const T ir1 = rcp_rn(rho + dW[0]);
    const T du = mad(-u, dW[0], dW[1]) * ir1, dv = mad(-v, dW[0], dW[2]) * ir1;
    const T dvn = mad(du, nx, dv * ny), vn1 = mad(u, nx, v * ny) + dvn;
    const T dmu = mad(dW[1], u + du, mad(dW[2], v + dv, mad(mx, du, my * dv)));
    const T dp = gm1 * mad((T)-0.5, dmu, dW[3]);
    dF[0] = mad(dW[0], vn1, rho * dvn);
    dF[1] = mad(dW[1], vn1, mad(mx, dvn, dp * nx));
    dF[2] = mad(dW[2], vn1, mad(my, dvn, dp * ny));
    dF[3] = mad(dW[3] + dp, vn1, H * dvn);
}

// One CTA: forward then backward sweep over the i+j hyperplanes (the
// lexicographic dependency order).  Two threads own one cell of the
// hyperplane: thread h handles the slot pair (west, east) for h = 0 and
// (south, north) for h = 1 -- of each pair at most one neighbour is on the
// already-swept side away from a periodic seam, so each thread usually
// evaluates one flux increment 1/2 (dF S - omega Lambda dW_nb).  The two
// partial sums meet in one pair shuffle and thread h writes components 2h and
// 2h+1 of the increment.  Neighbours are found from the cell's (i, j) and the
// periodic flags.  Records and (backward) the cell's own dW* are prefetched
// kStages-1 hyperplanes ahead with cp.async; the previous hyperplane's
// increments and base states sit in a shared-memory ring indexed by the slot
// in the hyperplane; neighbours across a periodic seam (earlier hyperplanes)
// come from global memory.
template <class T, int kStages>
__global__ void __launch_bounds__(512) k_macro_sweep(Launch L)
{
    IDG_LOCATE();
    extern __shared__ __align__(16) unsigned char smraw[];
    const int tid = threadIdx.x, ncs = blockDim.x >> 1;  // cell slots
    const int cs = tid >> 1, h = tid & 1;
    const int ni = p.ni, nj = p.nj, nh = ni + nj - 1;
    const bool per_i = p.per_i, per_j = p.per_j;
    T *srec = (T *)smraw;                               // [kStages][ncs][kMRec]
    T *sdw = srec + (size_t)kStages * ncs * kMRec;      // [kStages][ncs][4] own dW* (backward)
    T *ring = sdw + (size_t)kStages * ncs * 4;          // [2][ncs][kMRing]
    if (tid < 32) record_residual(p);
    const T gm1 = (T)(p.gam - 1.0);
    T *dWg = (T *)p.mdW;
    const T *mrec = (const T *)p.mrec;
    constexpr int RC = kMRec * sizeof(T) / 16;  // 16-byte chunks of one record
    constexpr int DC = 4 * sizeof(T) / 16;      // chunks of one dW
    for (int dir = 1; dir >= -1; dir -= 2) {
        auto step_d = [&](int s) { return dir > 0 ? s : nh - 1 - s; };
        auto issue = [&](int s) {
            if (s < nh) {
                const int d = step_d(s);
                const int i = max(0, d - (nj - 1)) + cs;
                if (i <= min(ni - 1, d)) {
                    const int c = (d - i) * ni + i;
                    const size_t e = (size_t)(s & (kStages - 1)) * ncs + cs;
                    const int nch = RC + (dir < 0 ? DC : 0);
                    for (int q = h; q < nch; q += 2) {
                        if (q < RC) cp_async16((char *)(srec + e * kMRec) + 16 * q, (const char *)(mrec + (size_t)kMRec * c) + 16 * q);
                        else cp_async16((char *)(sdw + e * 4) + 16 * (q - RC), (const char *)(dWg + 4 * (size_t)c) + 16 * (q - RC));
                    }
                }
            }
            cp_commit();
        };
        for (int s = 0; s < kStages - 1; ++s) issue(s);
        for (int s = 0; s < nh; ++s) {
            cp_wait<kStages - 2>();
            __syncthreads();
            issue(s + kStages - 1);
            const int d = step_d(s);
            const int ilo = max(0, d - (nj - 1)), ihi = min(ni - 1, d);
            const int i = ilo + cs, j = d - i;
            const bool valid = i <= ihi;
            const int c = j * ni + i;
            const size_t e = (size_t)(s & (kStages - 1)) * ncs + cs;
            const T *rec = srec + e * kMRec;
            T acc0 = 0, acc1 = 0, acc2 = 0, acc3 = 0;
            if (valid) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    // slot m = 2h + u: west, east (h = 0); south, north (h = 1)
                    const int m = 2 * h + u;
                    int nbi = i, nbj = j;
                    bool ex = true;
                    if (h == 0) {
                        nbi = u ? i + 1 : i - 1;
                        if (u ? i == ni - 1 : i == 0) { ex = per_i; nbi = u ? 0 : ni - 1; }
                    } else {
                        nbj = u ? j + 1 : j - 1;
                        if (u ? j == nj - 1 : j == 0) { ex = per_j; nbj = u ? 0 : nj - 1; }
                    }
                    const int nb = nbj * ni + nbi;
                    if (!ex || !(dir > 0 ? nb < c : nb > c)) continue;
                    T dn[4];
                    const T *base;
                    if (nbi + nbj == d - dir) {
                        const int ts = nbi - max(0, d - dir - (nj - 1));
                        const T *x = ring + ((size_t)((s + 1) & 1) * ncs + ts) * kMRing;
                        dn[0] = x[0]; dn[1] = x[1]; dn[2] = x[2]; dn[3] = x[3];
                        base = x + 4;
                    } else {
                        const T *x = dWg + 4 * (size_t)nb;
                        dn[0] = x[0]; dn[1] = x[1]; dn[2] = x[2]; dn[3] = x[3];
                        base = mrec + (size_t)kMRec * nb + 6;
                    }
                    const T *cf = rec + 12 + 3 * m;
                    T dF[4];
                    euler_dflux<T>(gm1, base, dn, cf[0], cf[1], dF);
                    acc0 += mad(-cf[2], dn[0], dF[0]);
                    acc1 += mad(-cf[2], dn[1], dF[1]);
                    acc2 += mad(-cf[2], dn[2], dF[2]);
                    acc3 += mad(-cf[2], dn[3], dF[3]);
                }
            }
            // sum over the two slot pairs of the cell
            acc0 += __shfl_xor_sync(0xffffffffu, acc0, 1);
            acc1 += __shfl_xor_sync(0xffffffffu, acc1, 1);
            acc2 += __shfl_xor_sync(0xffffffffu, acc2, 1);
            acc3 += __shfl_xor_sync(0xffffffffu, acc3, 1);
            if (valid) {
                // forward: dW*_c = (R_c - sum_lower) / D_c;  backward: dW_c = dW*_c - sum_upper / D_c
                const T iD = rec[4];
                const T a0 = h ? acc2 : acc0, a1 = h ? acc3 : acc1;
                const int q0 = 2 * h;
                T x0, x1;
                if (dir > 0) {
                    x0 = (rec[q0] - a0) * iD;
                    x1 = (rec[q0 + 1] - a1) * iD;
                } else {
                    x0 = mad(-a0, iD, sdw[e * 4 + q0]);
                    x1 = mad(-a1, iD, sdw[e * 4 + q0 + 1]);
                }
                T *r = ring + ((size_t)(s & 1) * ncs + cs) * kMRing;
                r[q0] = x0;
                r[q0 + 1] = x1;
                r[4 + 3 * h] = rec[6 + 3 * h];
                r[5 + 3 * h] = rec[7 + 3 * h];
                r[6 + 3 * h] = rec[8 + 3 * h];
                dWg[4 * (size_t)c + q0] = x0;
                dWg[4 * (size_t)c + q0 + 1] = x1;
            }
        }
        cp_wait<0>();
        __syncthreads();
    }
    if (tid == 0) *p.iter += 1;
}

// The same sweeps with one thread per line of cells.  The lines run along
// the longer axis (w), one thread per line of the shorter axis (t: columns,
// t = i, when ni <= nj, else rows, t = j); a thread marches along its line one
// step behind the line before it, so at every step the lines stand on an i+j
// hyperplane.  A cell's two already swept neighbours are the thread's own last
// cell and the last cell of the line before, and both enter a cell's equation
// only through the terms 1/2 (dF S - omega Lambda dW): each thread forms, from
// its new increment, the two terms that its own next cell and the next line's
// cell will need (half of their arithmetic is common) and passes the latter on
// by a warp shuffle -- four values and no base state.  Warps of 32 lines run as
// the strips of the micro sweeps do (see there): border terms in a ring, flags
// every kSweepBlock steps, no block barrier inside a sweep.  The cells' records
// and increments lie hyperplane by hyperplane (line_slot), so that the lines of
// a warp copy consecutive vectors, by cp.async kStages steps ahead into the
// thread's own slots (cell by cell each copy touched 32 cache lines, 670 cycles
// a step).  A line's first
// cell keeps its term across a seam along the lines in registers; the first
// line's terms across a seam to the last one lie in shared memory.
// Bound by the latency of a step, 140 instructions of one warp per scheduler.
// One barrier per step, base states passed along, both terms formed by the
// receiver and one thread adding up the residual took 62 us on 64 x 64 cells,
// 213 us on 128 x 128 and 39 us on 48 x 40; this 40, 85 and 30 us.
constexpr int kLRing = 32;        // border-ring entries (see sweep_shape)

template <class T> static size_t macro_lines_smem_bytes(int nlines, int stages, int nw, bool seam)
{
    return 64 + ((size_t)stages * nlines * 24 + (size_t)nlines / 32 * kLRing * 4 + (seam ? (size_t)nw * 4 : 0)) * sizeof(T);
}

// The part of the exact Euler-flux increment F_n(W + dW) - F_n(W) that does not
// depend on the normal, every term an increment times a base quantity:
// ir = 1 / (rho + drho), the pressure increment through
// d(|m|^2 / rho) = ((2 m + dm) . dm - (|m|^2 / rho) drho) ir.
template <class T> struct LineInc {
    T rho, mx, my, u, v, H, ir, dp;
    T dW[4];
};
// b: 1/D, rho, m_x, m_y; c: 1/rho, E + p
template <class T> __device__ __forceinline__ void line_inc(LineInc<T> &x, T gm1, const T (&b)[4], const T (&c)[4])
{
    x.rho = b[1]; x.mx = b[2]; x.my = b[3]; x.u = x.mx * c[0]; x.v = x.my * c[0]; x.H = c[1];
    x.ir = rcp_line(x.rho + x.dW[0]);
    const T k = mad(x.mx, x.u, x.my * x.v);
    const T q = mad(mad((T)2, x.mx, x.dW[1]), x.dW[1], mad(mad((T)2, x.my, x.dW[2]), x.dW[2], -k * x.dW[0]));
    x.dp = mad((T)-0.5 * gm1 * q, x.ir, gm1 * x.dW[3]);
}
// the term 1/2 (dF S - omega Lambda dW) of this cell's increment in the
// equation of the neighbour across the face with S/2 n out of this cell
// (ox, oy) and omega/2 Lambda = ol: the neighbour's normal is the opposite one
template <class T> __device__ __forceinline__ void line_term(const LineInc<T> &x, T ox, T oy, T ol, T (&o)[4])
{
    const T nx = -ox, ny = -oy;
    const T vn = mad(x.u, nx, x.v * ny);
    const T dm = mad(x.dW[1], nx, x.dW[2] * ny);
    const T dvn = mad(-vn, x.dW[0], dm) * x.ir, vn1 = vn + dvn;
    o[0] = mad(-ol, x.dW[0], dm);
    o[1] = mad(x.dW[1], vn1, mad(x.mx, dvn, mad(x.dp, nx, -ol * x.dW[1])));
    o[2] = mad(x.dW[2], vn1, mad(x.my, dvn, mad(x.dp, ny, -ol * x.dW[2])));
    o[3] = mad(x.dW[3] + x.dp, vn1, mad(x.H, dvn, -ol * x.dW[3]));
}

// what a sweep of k_macro_lines reads that does not change
template <class T> struct LineCtx {
    T *stage, *ring, *seam, *dWg;
    int *flags, *status;
    const T *rec;
    size_t M;  // slots
    T gm1;
    int nt, nw, nthr, lane, wid, strips, polls;
    bool per_t, per_w;
};

// one direction of k_macro_lines (SEAM: the block has a periodic seam); lines
// and cells are numbered from the corner the sweep starts at (tt, ww)
template <class T, int kStages, bool FWD, bool SEAM> __device__ __forceinline__ void line_sweep(const LineCtx<T> &x)
{
    constexpr int VC = 4 * sizeof(T) / 16;  // 16-byte chunks of a vector
    const int tt = x.wid * 32 + x.lane, tc = min(tt, x.nt - 1), t = FWD ? tc : x.nt - 1 - tc;
    // slot of (tt, ww): e0 + ww * es
    const int es = FWD ? x.nt : -x.nt, e0 = (FWD ? t : t + x.nw - 1) * x.nt + t;
    const unsigned nwl = tt < x.nt ? x.nw : 0;
    const int s_beg = x.wid * (32 + kSweepBlock);
    const int s_end = s_beg + x.nw + min(32, x.nt - x.wid * 32) - 1;
    const int start = tt + x.wid * kSweepBlock;
    // stage slots [kStages][6][nthr][4]: R or dW*, then the record's vectors (the
    // other sweep's faces, which a seam needs, last)
    T *stage = x.stage + 4 * (x.wid * 32 + x.lane);
    const size_t vec = (size_t)4 * x.nthr, slot = 6 * vec;
    const T *g0 = (FWD ? x.rec : x.dWg), *g1 = x.rec + 4 * x.M, *g2 = x.rec + (FWD ? 8 : 16) * x.M,
            *g3 = g2 + 4 * x.M, *g4 = x.rec + (FWD ? 16 : 8) * x.M, *g5 = g4 + 4 * x.M;
    auto issue = [&](int s) {
        const ptrdiff_t e = 4 * (ptrdiff_t)(e0 + min(max(s - start, 0), x.nw - 1) * es);
        T *dst = stage + (s & (kStages - 1)) * slot;
#pragma unroll
        for (int q = 0; q < VC; ++q) {
            constexpr int E = 16 / sizeof(T);
            cp_async16(dst + E * q, g0 + e + E * q);
            cp_async16(dst + vec + E * q, g1 + e + E * q);
            cp_async16(dst + 2 * vec + E * q, g2 + e + E * q);
            cp_async16(dst + 3 * vec + E * q, g3 + e + E * q);
            if (SEAM) {
                cp_async16(dst + 4 * vec + E * q, g4 + e + E * q);
                cp_async16(dst + 5 * vec + E * q, g5 + e + E * q);
            }
        }
        cp_commit();
    };
    for (int u = 0; u < kStages; ++u) issue(s_beg + u);
    const bool edge = x.lane == 0 && x.wid > 0, border = x.lane == 31 && x.wid + 1 < x.strips;
    T *xw = x.ring + (size_t)x.wid * kLRing * 4;
    const T *xr = x.wid > 0 ? xw - kLRing * 4 : xw;
    T to_w[4] = {0, 0, 0, 0}, to_t[4] = {0, 0, 0, 0}, first[4] = {0, 0, 0, 0};
    int seen_r = 0, seen_w = 0;
    for (int s0 = s_beg; s0 < s_end; s0 += kSweepBlock) {
        if (x.strips > 1) {
            if (x.wid > 0) flag_wait(x.flags + x.wid - 1, s0, seen_r, x.status, x.polls);
            if (x.wid + 1 < x.strips) flag_wait(x.flags + x.wid + 1, s0 + 2 * kSweepBlock + 1 - kLRing, seen_w, x.status, x.polls);
        }
#pragma unroll
        for (int b = 0; b < kSweepBlock; ++b) {
            const int s = s0 + b, ww = s - start;
            cp_wait<kStages - 1>();
            if (SEAM) __syncwarp();
            const T *rec = stage + (s & (kStages - 1)) * slot;
            T r[4], rb[4], rc[4], rd[4], e[4];
            ld4(r, rec);
            ld4(rb, rec + vec);
            ld4(rc, rec + 2 * vec);
            ld4(rd, rec + 3 * vec);
            ld4(e, xr + (ww & (kLRing - 1)) * 4);
            LineInc<T> inc;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const T sh = __shfl_up_sync(0xffffffffu, to_t[q], 1);
                const T adj = tt > 0 ? (edge ? e[q] : sh) : (T)0;
                T acc = adj + (ww > 0 ? to_w[q] : (T)0);
                if (SEAM && x.per_w && ww == x.nw - 1) acc += first[q];
                if (SEAM && x.per_t && tt == x.nt - 1 && (unsigned)ww < nwl) acc += x.seam[4 * ww + q];
                // forward: dW*_c = (R_c - sum_lower) / D_c;  backward: dW_c = dW*_c - sum_upper / D_c
                inc.dW[q] = FWD ? (r[q] - acc) * rb[0] : mad(-acc, rb[0], r[q]);
            }
            line_inc<T>(inc, x.gm1, rb, rc);
            line_term<T>(inc, rd[0], rd[1], rc[2], to_w);
            line_term<T>(inc, rd[2], rd[3], rc[3], to_t);
            const bool on = (unsigned)ww < nwl;
            st4_if<true>(x.dWg + 4 * (ptrdiff_t)(e0 + ww * es), inc.dW, on);
            st4_if<false>(xw + (ww & (kLRing - 1)) * 4, to_t, on && border);
            if (SEAM && on) {
                const T *oc = rec + 4 * vec, *od = rec + 5 * vec;  // the faces behind
                if (x.per_w && ww == 0) line_term<T>(inc, od[0], od[1], oc[2], first);
                if (x.per_t && tt == 0) {
                    T st[4];
                    line_term<T>(inc, od[2], od[3], oc[3], st);
                    st4(x.seam + 4 * ww, st);
                }
            }
            issue(s + kStages);
        }
        if (x.strips > 1) {
            __syncwarp();
            if (x.lane == 0) flag_store(x.flags + x.wid, s0 + kSweepBlock);
        }
    }
    cp_wait<0>();
    if (x.strips > 1) {
        __syncwarp();
        if (x.lane == 0) flag_store(x.flags + x.wid, 0x7fffffff);
    }
}

// 32 threads per strip and one more warp that records the residual meanwhile
template <class T, int kStages, bool SEAM>
__global__ void __launch_bounds__(288, 1) k_macro_lines(Launch L)
{
    IDG_LOCATE();
    (void)blk;
    extern __shared__ __align__(16) unsigned char smraw[];
    LineCtx<T> x;
    const bool cols = p.ni <= p.nj;
    x.nt = cols ? p.ni : p.nj;
    x.nw = cols ? p.nj : p.ni;
    x.strips = (x.nt + 31) / 32;
    x.lane = threadIdx.x & 31;
    x.wid = threadIdx.x >> 5;
    x.nthr = x.strips * 32;
    // periodic between the last and the first line / along the lines; a
    // direction one cell wide wraps onto the cell itself (no term)
    x.per_t = (cols ? p.per_i : p.per_j) && x.nt > 1;
    x.per_w = (cols ? p.per_j : p.per_i) && x.nw > 1;
    x.flags = (int *)smraw;                           // [8] steps done by each strip
    x.ring = (T *)(smraw + 64);                       // [strips][kLRing][4]
    x.stage = x.ring + (size_t)x.strips * kLRing * 4; // [kStages][6][nthr][4]
    x.seam = x.stage + (size_t)kStages * x.nthr * 24; // [nw][4] the first line's terms (per_t)
    x.status = p.status;
    x.polls = p.wait_polls;
    x.dWg = (T *)p.mdW;
    x.rec = (const T *)p.mline;
    x.M = line_slots(p);
    x.gm1 = (T)(p.gam - 1.0);
    const bool sweeps = x.wid < x.strips;
    auto arm = [&] {
        if (sweeps && x.lane == 0) x.flags[x.wid] = x.wid * (32 + kSweepBlock);
        __syncthreads();
    };
    arm();
    if (sweeps) line_sweep<T, kStages, true, SEAM>(x);
    else if (x.wid == x.strips) record_residual(p);
    __syncthreads();  // dW* of every line is written, the flags are free
    arm();
    if (sweeps) line_sweep<T, kStages, false, SEAM>(x);
    __syncthreads();  // the residual went to this iteration's slot
    if (threadIdx.x == 0) *p.iter += 1;
}

// The macroscopic LU-SGS sweeps on an unstructured mesh: one CTA walks the
// steps of the forward, then the backward schedule (the lower- and
// upper-neighbour levels of the cell numbering), a thread per cell of a step
// (a step holds at most blockDim.x cells); the same equations and cell order
// as k_macro_sweep.  Everything of a step that the sweep does not change -- the
// cell, its swept neighbours, its record, their base states -- is in registers
// before the barrier that opens the step, so that after it only the neighbours'
// increments are read.  The cell and its neighbours come from lists in schedule
// order two steps ahead, the records they name one step ahead: found through the
// mesh's tables when needed, the four loads of that chain (step, cell, neighbour,
// record) stood in each step's way, 0.8 us of it: 386 us on 8192 triangles, this
// 185 us.  SMEM: the increments of all cells live in shared memory for the two
// sweeps and go to global memory at the end; otherwise they are read from global
// memory.
template <class T> struct MacroCell {
    int c, nb[4];
    T r[4], iD, cf[12], base[4][6];
};

// base state (6 scalars at an even offset) by pairs
__device__ __forceinline__ void ld6(float (&o)[6], const float *s)
{
#pragma unroll
    for (int q = 0; q < 6; q += 2) {
        const float2 v = *reinterpret_cast<const float2 *>(s + q);
        o[q] = v.x;
        o[q + 1] = v.y;
    }
}
__device__ __forceinline__ void ld6(double (&o)[6], const double *s)
{
#pragma unroll
    for (int q = 0; q < 6; q += 2) {
        const double2 v = *reinterpret_cast<const double2 *>(s + q);
        o[q] = v.x;
        o[q + 1] = v.y;
    }
}

// the cell of this thread at step st and its already swept neighbours (-1: none)
struct SchedCell {
    int c;
    int4 nb;
};
__device__ __forceinline__ SchedCell sched_cell(const int *sc, const int4 *sn, const int *sp, int st, int ns)
{
    SchedCell x;
    x.c = -1;
    x.nb = make_int4(-1, -1, -1, -1);
    if (st < ns) {
        const int b = sp[st];
        if ((int)threadIdx.x < sp[st + 1] - b) {
            x.c = sc[b + threadIdx.x];
            x.nb = sn[b + threadIdx.x];
        }
    }
    return x;
}

template <class T> __device__ __forceinline__ void macro_cell_load(const KParams &p, const SchedCell &s, MacroCell<T> &x)
{
    x.c = s.c;
    if (s.c < 0) return;
    const T *mrec = (const T *)p.mrec, *rec = mrec + (size_t)kMRec * s.c;
    ld4(x.r, rec);
    x.iD = rec[4];
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        T v[4];
        ld4(v, rec + 12 + 4 * q);
#pragma unroll
        for (int u = 0; u < 4; ++u) x.cf[4 * q + u] = v[u];
    }
    x.nb[0] = s.nb.x; x.nb[1] = s.nb.y; x.nb[2] = s.nb.z; x.nb[3] = s.nb.w;
#pragma unroll
    for (int m = 0; m < 4; ++m)
        if (x.nb[m] >= 0) ld6(x.base[m], mrec + (size_t)kMRec * x.nb[m] + 6);
}

template <class T, bool SMEM>
__global__ void __launch_bounds__(256) k_macro_sweep_sched(Launch L)
{
    IDG_LOCATE();
    (void)blk;
    extern __shared__ __align__(16) unsigned char smraw[];
    if (threadIdx.x >= blockDim.x - 32) record_residual(p);
    const T gm1 = (T)(p.gam - 1.0);
    T *dWg = (T *)p.mdW;
    T *dw = SMEM ? (T *)smraw : dWg;  // [N][4]
    for (int dir = 1; dir >= -1; dir -= 2) {
        const int *sc = p.sched + (dir > 0 ? 0 : (size_t)p.N);
        const int4 *sn = (const int4 *)p.snb + (dir > 0 ? 0 : (size_t)p.N);
        const int *sp = p.sptr + (dir > 0 ? 0 : p.nsteps_f + 1);
        const int ns = dir > 0 ? p.nsteps_f : p.nsteps_b;
        SchedCell s1 = sched_cell(sc, sn, sp, 1, ns);
        MacroCell<T> cur;
        macro_cell_load<T>(p, sched_cell(sc, sn, sp, 0, ns), cur);
        for (int st = 0; st < ns; ++st) {
            const SchedCell s2 = sched_cell(sc, sn, sp, st + 2, ns);
            MacroCell<T> nxt;
            macro_cell_load<T>(p, s1, nxt);
            __syncthreads();
            if (cur.c >= 0) {
                T acc[4] = {0, 0, 0, 0};
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    if (cur.nb[m] < 0) continue;
                    T dn[4], dF[4];
                    ld4(dn, dw + 4 * (size_t)cur.nb[m]);
                    euler_dflux<T>(gm1, cur.base[m], dn, cur.cf[3 * m], cur.cf[3 * m + 1], dF);
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[q] += mad(-cur.cf[3 * m + 2], dn[q], dF[q]);
                }
                // forward: dW*_c = (R_c - sum_lower) / D_c;  backward: dW_c = dW*_c - sum_upper / D_c
                T *o = dw + 4 * (size_t)cur.c, v[4];
                if (dir < 0) ld4(v, o);
#pragma unroll
                for (int q = 0; q < 4; ++q) v[q] = dir > 0 ? (cur.r[q] - acc[q]) * cur.iD : mad(-acc[q], cur.iD, v[q]);
                st4(o, v);
            }
            cur = nxt;
            s1 = s2;
        }
        __syncthreads();
    }
    if (SMEM)
        for (int q = threadIdx.x; q < 4 * p.N; q += blockDim.x) dWg[q] = dw[q];
    if (threadIdx.x == 0) *p.iter += 1;
}

template <class T, class LT>
__global__ void __launch_bounds__(32) k_macro_post(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    const int c = blk * blockDim.x + threadIdx.x;
    if (c >= p.N) return;
    double *W = p.W + 4 * c;
    const T *dW = (const T *)p.mdW + 4 * (by_lines(p) ? line_slot(p, c) : c);
    for (int q = 0; q < 4; ++q) W[q] += (double)dW[q];
    const double rho = W[0], irho = rcp_rn(rho), U = W[1] * irho, V = W[2] * irho;
    const double RT = mad(-V, V, mad(-U, U, 2.0 * W[3] * irho)) * p.iK2, ir = rcp_rn(RT);
    const double tau2 = 2.0 * viscosity_t<T>(p, RT) * (irho * ir);  // 2 tau'
    T *ct = (T *)p.cellpT + kCellP * c;
    eq_storeT<T>(ct, make_eq(p, rho, irho, U, V, RT, ir, p.cellq[2 * c], p.cellq[2 * c + 1]));
    const double cq = 2.0 * p.area[c] * rcp_rn(tau2 + p.dt);
    const T D0 = (T)(p.adt[c] + cq);  // diagonal base of Eq. (26)
    ct[14] = (T)cq;
    ct[15] = D0;
    if (p.sgeo) {
        // where both line sweeps read it
        T *sg = (T *)p.sgeo + 8 * (size_t)c + 6;
        sg[0] = D0;
        sg[8 * (size_t)p.N] = D0;
    }
}

// Point relaxation of the predictor equations (the alternative to LU-SGS the
// conclusions name): D dW_c + sum_nb 1/2 (dF_nb S - omega Lambda dW_nb) = R_c
// solved by Jacobi sweeps from dW = 0, every cell at once from the previous
// sweep's increments of all its neighbours -- no wavefront, every SM busy.
// Sweep k of n (1-based) writes mdW when n - k is even, mdW2 when odd, so the
// last one leaves dW in mdW for k_macro_post; sweep 1 gives dW = R / D.  The
// record of k_macro_pre holds R, 1/D, the cell's base state and per slot
// (S/2) n_out and (omega/2) Lambda, as for the sweeps.
template <class T, class LT>
__global__ void __launch_bounds__(32) k_macro_relax(const __grid_constant__ LT L, int sweep, int nsweeps)
{
    IDG_LOCATE();
    const int c = blk * blockDim.x + threadIdx.x;
    if (c >= p.N) return;
    const bool odd = (nsweeps - sweep) & 1;
    T *dst = (T *)(odd ? p.mdW2 : p.mdW);
    const T *src = (const T *)(odd ? p.mdW : p.mdW2);
    const T *mrec = (const T *)p.mrec;
    const T *rec = mrec + (size_t)kMRec * c;
    const T gm1 = (T)(p.gam - 1.0);
    T acc[4] = {0, 0, 0, 0};
    if (sweep > 1) {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int nb = p.cnb[4 * c + m];
            if (nb < 0 || nb == c) continue;  // ghost, or a cell wrapped onto itself
            const T *x = src + 4 * (size_t)nb;
            const T dn[4] = {x[0], x[1], x[2], x[3]};
            const T *cf = rec + 12 + 3 * m;
            T dF[4];
            euler_dflux<T>(gm1, mrec + (size_t)kMRec * nb + 6, dn, cf[0], cf[1], dF);
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] += mad(-cf[2], dn[q], dF[q]);
        }
    }
    const T iD = rec[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) dst[4 * (size_t)c + q] = (rec[q] - acc[q]) * iD;
}

// ---------------------------------------------------------------------------
// explicit DUGKS (Eq. 10, 21): the cell and face kernels of the implicit
// iteration build the face fluxes with the physical step dt, then
//   k_explicit_update  per (cell, velocity):
//                      f~ <- (2tau-dt)/(2tau+dt) f~ + 2dt/(2tau+dt) f^S - dt/Omega sum F
//   k_cell_moments, k_explicit_w: W = moments of the new f~ (the collision
//                      conserves them, so f~ and f share them), which the
//                      next step's cell prep reads, and partial sums of
//                      ||(W^{n+1} - W^n)/dt||^2
//   k_record_residual  the step's residual ||(W^{n+1} - W^n)/dt||_2.
// At the fixed point of the march R_W = -sum Phi does not vanish: it balances
// the moments of the discrete collision term (the quadrature error of the
// discrete equilibrium), so the march is measured by its rate of change.
// ---------------------------------------------------------------------------

// one warp per instance: the residual of this iteration from the block
// partials of the kernel before it into the ring, and the iteration count
template <class T, class LT>
__global__ void __launch_bounds__(32) k_record_residual(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    (void)blk;
    record_residual(p);
    if (threadIdx.x == 0) *p.iter += 1;
}

template <class T, class LT>
__global__ void __launch_bounds__(128) k_explicit_update(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    int k;
    for_cells(p, blk, k, [&](int c) {
    const T *cA = (const T *)p.cellA + kCellP * c;
    const EqT<T> e = eq_loadT<T>(cA);
    // k_cell_params stores c2 = 3h/(2tau+dt) = (3/4) 2dt/(2tau+dt) (h = dt/2)
    const T b = cA[15] * (T)(4.0 / 3.0), a = (T)1 - b;
    const T dto = (T)(p.dt / p.area[c]), kRTr = (T)(p.K * p.RT_r);
    T ux[2], uy[2], gr[2];
    vtab2<T>(p.uxf, p.ux, k, ux);
    vtab2<T>(p.uyf, p.uy, k, uy);
    vtab2<T>(p.greff, p.gref, k, gr);
    T sg_[2] = {0, 0}, sh_[2] = {0, 0};
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        T fg[2], fh[2];
        load_pair<T>(p.F, (size_t)p.cface[4 * c + m] * p.Nv + k, fg, fh);
        const T sg = (T)p.csign[4 * c + m];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            sg_[v] = mad(sg, fg[v], sg_[v]);
            sh_[v] = mad(sg, fh[v], sh_[v]);
        }
    }
    const size_t ck = (size_t)c * p.Nv + k;
    T g[2], h[2];
    load_pair<T>(p.f, ck, g, h);
#pragma unroll
    for (int v = 0; v < 2; ++v) {
        T dG, dH;
        dev_equilibrium<T>(e, ux[v], uy[v], gr[v], kRTr, dG, dH);
        g[v] = mad(-dto, sg_[v], mad(a, g[v], b * dG));
        h[v] = mad(-dto, sh_[v], mad(a, h[v], b * dH));
    }
    store_pair<T>(p.f, ck, g, h);
    });
}

// W = (rho, rho U, rho V, rho E) of f~ from its raw moments (Eq. 4), and
// block partials of ||(W_new - W_old)/dt||^2 (fixed order)
template <class T, class LT>
__global__ void __launch_bounds__(32) k_explicit_w(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    __shared__ double sm[32];
    const int c = blk * blockDim.x + threadIdx.x;
    double part[1] = {0.0};
    if (c < p.N) {
        auto r = [&](int q) { return acc_load<T>(p.cellraw, (size_t)c * kRaw + q) + p.mref_raw[q]; };
        double *W = p.W + 4 * c;
        const double Wn[4] = {r(0), r(1), r(2), 0.5 * (r(3) + r(5) + r(8))};
        for (int q = 0; q < 4; ++q) {
            const double d = (Wn[q] - W[q]) / p.dt;
            part[0] += d * d;
            W[q] = Wn[q];
        }
    }
    block_sum<1>(part, sm);
    if (threadIdx.x == 0) p.mpart[blk] = part[0];
}

// ---------------------------------------------------------------------------
// micro LU-SGS (Eq. 22-26)                                            [a6-a7]
//   k_micro_residual  per (cell, velocity), fully parallel:
//                     R = -sum_faces F - (2 Omega/(2 tau' + dt)) (f~ - f^S(W^{n+1})),
//                     written into the increment buffer
//   forward sweep     Delta*_c = (R_c + sum_{lower inflow nb} |xi.n| S Delta*_nb) / D_c
//   backward sweep    Delta_c = Delta*_c + sum_{upper inflow nb} |xi.n| S Delta_nb / D_c,
//                     f~ += Delta (Eq. 32)
// with D = Omega/dt_imp + sum_{outflow} xi.n S + 2 Omega/(2 tau' + dt).
// A structured block's sweeps run lines of cells (k_sweep_lines), an
// unstructured mesh's the steps of its level schedule (k_sweep: one block per
// tile of sweep_tv velocities, a thread per (cell of the step, velocity),
// everything but the neighbours' increments copied kStages-1 steps ahead).
// ---------------------------------------------------------------------------
template <class T, class LT>
__global__ void __launch_bounds__(128) k_micro_residual(const __grid_constant__ LT L)
{
    IDG_LOCATE();
    int k;
    for_cells(p, blk, k, [&](int c) {
    const T *cp = (const T *)p.cellpT + kCellP * c;
    const EqT<T> e = eq_loadT<T>(cp);
    const T cq = cp[14], kRTr = (T)(p.K * p.RT_r);
    T ux[2], uy[2], gr[2];
    vtab2<T>(p.uxf, p.ux, k, ux);
    vtab2<T>(p.uyf, p.uy, k, uy);
    vtab2<T>(p.greff, p.gref, k, gr);
    const size_t ck = (size_t)c * p.Nv + k;
    T rg[2], rh[2];
    load_pair<T>(p.f, ck, rg, rh);
#pragma unroll
    for (int v = 0; v < 2; ++v) {
        T dG, dH;
        dev_equilibrium<T>(e, ux[v], uy[v], gr[v], kRTr, dG, dH);
        rg[v] = -cq * (rg[v] - dG);
        rh[v] = -cq * (rh[v] - dH);
    }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        T fg[2], fh[2];
        load_pair<T>(p.F, (size_t)p.cface[4 * c + m] * p.Nv + k, fg, fh);
        const T sg = (T)p.csign[4 * c + m];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            rg[v] = mad(-sg, fg[v], rg[v]);
            rh[v] = mad(-sg, fh[v], rh[v]);
        }
    }
    store_pair<T>(p.dst, ck, rg, rh);
    });
}

// Role of the neighbour across each slot of a cell in one scheduled micro sweep
// (computed on the host): <= kSeam the neighbour kSeam - code, already swept and
// read from global memory; otherwise a ghost or a neighbour not yet swept
// (outflow only adds to D).
constexpr int kSeam = -4;

// 8 storage scalars from 16-byte-aligned shared memory
template <class T> __device__ __forceinline__ void load8(T (&r)[8], const T *s);
template <> __device__ __forceinline__ void load8<float>(float (&r)[8], const float *s)
{
    const float4 a = ((const float4 *)s)[0], b = ((const float4 *)s)[1];
    r[0] = a.x; r[1] = a.y; r[2] = a.z; r[3] = a.w; r[4] = b.x; r[5] = b.y; r[6] = b.z; r[7] = b.w;
}
template <> __device__ __forceinline__ void load8<double>(double (&r)[8], const double *s)
{
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const double2 a = ((const double2 *)s)[u];
        r[2 * u] = a.x; r[2 * u + 1] = a.y;
    }
}

// shared-memory layout of the scheduled micro sweeps (VPT consecutive velocities per thread)
template <class T, int kStages, int VPT> struct SweepSmem {
    using T2 = typename V2<T>::t;
    T2 *R;      // [kStages][pc][tv*VPT]  R (forward) / Delta* (backward)
    T2 *F;      // [kStages][pc][tv*VPT]  f~ (backward only)
    T *geo;     // [kStages][pc][8]  per slot: sign*nx*S, sign*ny*S
    int *code;  // [kStages][pc][4]  per slot: the neighbour's role in this sweep
    T *D0;      // [kStages][pc]
    __device__ SweepSmem(unsigned char *base, int pc, int tv, bool withF)
    {
        size_t o = 0;
        const size_t w = (size_t)tv * VPT;
        R = (T2 *)(base + o); o += (size_t)kStages * pc * w * sizeof(T2);
        F = (T2 *)(base + o); if (withF) o += (size_t)kStages * pc * w * sizeof(T2);
        geo = (T *)(base + o); o += (size_t)kStages * pc * 8 * sizeof(T);
        code = (int *)(base + o); o += (size_t)kStages * pc * 4 * sizeof(int);
        D0 = (T *)(base + o);
    }
};

template <class T, int kStages, int VPT> static size_t sweep_smem_bytes(int pc, int tv, bool withF)
{
    using T2 = typename V2<T>::t;
    const size_t w = (size_t)tv * VPT;
    size_t o = (size_t)kStages * pc * w * sizeof(T2) * (withF ? 2 : 1);
    o += (size_t)kStages * pc * (9 * sizeof(T) + 4 * sizeof(int));
    return o;
}

// the parameters a scheduled sweep touches every step, held in registers
struct SweepArgs {
    int Nv, tv, pc;
    void *dst, *f;
    const void *cslotT, *cellpT;
    const int *codes;         // this sweep's [N][4] slot codes
    const int *sched, *sptr;  // this sweep's schedule
    int nsteps;               // steps of the sweep
};

// asynchronous copy of one step's data for the thread's cell: its VPT
// consecutive velocities of R (or Delta*, f~), and the cell's slot geometry
// and diagonal base spread over the cell's tv threads
template <class T, int kStages, int VPT>
__device__ __forceinline__ void sweep_issue(const SweepArgs &p, const SweepSmem<T, kStages, VPT> &sm, int s, int c,
                                            int slot, int t, int k0, bool act, bool withF)
{
    using T2 = typename V2<T>::t;
    const int tv = p.tv, pc = p.pc;
    {
        if (c >= 0) {
            int st = s & (kStages - 1);
            size_t e = ((size_t)st * pc + slot);
            if (act) {
                constexpr int B = VPT * sizeof(T2);
                constexpr int CH = B < 16 ? B : 16;
                size_t ck = (size_t)c * p.Nv + k0;
                char *sr = (char *)(sm.R + e * tv * VPT + (size_t)t * VPT);
                const char *gr = (const char *)((const T2 *)p.dst + ck);
#pragma unroll
                for (int b = 0; b < B; b += CH) cp_async_b<CH>(sr + b, gr + b);
                if (withF) {
                    char *sf = (char *)(sm.F + e * tv * VPT + (size_t)t * VPT);
                    const char *gf = (const char *)((const T2 *)p.f + ck);
#pragma unroll
                    for (int b = 0; b < B; b += CH) cp_async_b<CH>(sf + b, gf + b);
                }
            }
            constexpr int ng = 8 * sizeof(T) / 16;  // 16-byte chunks of the slot geometry
            for (int q = t; q < ng + 2; q += tv) {
                if (q < ng) cp_async16((char *)(sm.geo + e * 8) + 16 * q, (const char *)((const T *)p.cslotT + 8 * (size_t)c) + 16 * q);
                else if (q == ng) cp_async16(sm.code + e * 4, p.codes + 4 * (size_t)c);
                else cp_async_b<sizeof(T)>(sm.D0 + e, (const T *)p.cellpT + kCellP * (size_t)c + 15);
            }
        }
    }
    cp_commit();
}

// A step's coefficients at one cell, of its VPT velocities: |xi.n| S of the
// inflow slots from already-swept cells (bits of `in`; zero elsewhere), their
// cells, 1/D.
template <class T, int VPT> struct SweepCoef {
    T w[VPT][4], iD[VPT];
    int nb[4];
    unsigned in;  // a bit: in float64 a comparison costs the pipe as much as a sum
    __device__ __forceinline__ void load(const T *geo, const int *codes, T D0, const T (&ux)[VPT], const T (&uy)[VPT])
    {
        T g[8];
        load8<T>(g, geo);
        const int4 cd = *(const int4 *)codes;
        const int code[4] = {cd.x, cd.y, cd.z, cd.w};
#pragma unroll
        for (int m = 0; m < 4; ++m) nb[m] = kSeam - code[m];
        in = 0;
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            // outflow adds (xi.n) S to D
            T D = D0;
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                const T aS = add_rn(mul_rn(ux[v], g[2 * m]), mul_rn(uy[v], g[2 * m + 1]));
                D += aS > (T)0 ? aS : (T)0;
                const bool i = aS < (T)0 && nb[m] >= 0;
                w[v][m] = i ? -aS : (T)0;
                in |= i ? 1u << (4 * v + m) : 0u;
            }
            iD[v] = rcp_rn(D);
        }
    }
};

// Unstructured meshes: the sweeps walk the steps of the level schedule, a block
// barrier between them.  Bound by the latency of a step, whose chain is the
// barrier, the neighbours' increments from L2 and the update: the cells are
// read from the schedule a step before their copies are issued, and a step's
// coefficients are formed in the step before it, while that one's increments
// are on their way (float32 with one velocity per thread: more would take the
// registers of a second block, and float64 is bound by its arithmetic pipe).
// Forward + backward, float32, 64 x 64 squares of two triangles with 1024
// velocities: 178 + 159 us with the cells read and the coefficients formed
// behind the step's own barrier, 104 + 95 us this way; float64 488 + 488 and
// 500 + 500 us (48 x 48 with 576).
template <class T, bool FWD, int kStages, int VPT>
__global__ void __launch_bounds__(512) k_sweep(Launch L)
{
    static_assert(kStages >= 3, "the next step's records are read a step ahead");
    constexpr bool kAhead = VPT == 1 && sizeof(T) == 4;
    IDG_LOCATE();
    using T2 = typename V2<T>::t;
    extern __shared__ __align__(16) unsigned char smraw[];
    const SweepArgs a{p.Nv, p.sweep_tv, p.sweep_pc, p.dst, p.f, p.cslotT, p.cellpT,
                      p.scode + (FWD ? 0 : 4 * (size_t)p.N), p.sched + (FWD ? 0 : (size_t)p.N),
                      p.sptr + (FWD ? 0 : p.nsteps_f + 1), FWD ? p.nsteps_f : p.nsteps_b};
    const int tv = a.tv, pc = a.pc, Nv = a.Nv;
    const SweepSmem<T, kStages, VPT> sm(smraw, pc, tv, !FWD);
    const int t = threadIdx.x % tv, slot = threadIdx.x / tv;
    const int k0 = (blk * tv + t) * VPT;  // Nv is a multiple of VPT
    const bool act = k0 < Nv;
    T ux[VPT], uy[VPT];
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        const int kk = act ? k0 + v : 0;
        ux[v] = vx<T>(p, kk);
        uy[v] = vy<T>(p, kk);
    }
    T2 *ds = (T2 *)a.dst;
    T2 *f = (T2 *)a.f;
    const int nh = a.nsteps;
    // cells of the steps s .. s + kStages - 1 (-1: none), the bounds of the next one
    int cell[kStages];
    int b0 = a.sptr[0], b1 = a.sptr[min(1, nh)];
#pragma unroll
    for (int q = 0; q < kStages; ++q) {
        cell[q] = slot < b1 - b0 ? a.sched[b0 + slot] : -1;
        b0 = b1;
        b1 = a.sptr[min(q + 2, nh)];
    }
#pragma unroll
    for (int q = 0; q < kStages - 1; ++q) sweep_issue<T, kStages, VPT>(a, sm, q, cell[q], slot, t, k0, act, !FWD);
    SweepCoef<T, VPT> cf;
    cp_wait<kStages - 2>();
    __syncthreads();
    auto coef = [&](int s, int c) {
        const size_t e = (size_t)(s & (kStages - 1)) * pc + slot;
        if (c >= 0) cf.load(sm.geo + e * 8, sm.code + e * 4, sm.D0[e], ux, uy);
    };
    if (kAhead) coef(0, cell[0]);
    for (int s = 0; s < nh; ++s) {
        cp_wait<kStages - (kAhead ? 3 : 2)>();
        __syncthreads();
        const bool on = cell[0] >= 0 && act;
        if (!kAhead) coef(s, cell[0]);
        T w[4], dg[4], dh[4];
        auto neighbours = [&](int v) {
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                w[m] = cf.w[v][m];
                dg[m] = dh[m] = (T)0;
                if (on && (cf.in >> (4 * v + m) & 1)) {
                    const T2 x = ds[(size_t)cf.nb[m] * Nv + k0 + v];
                    dg[m] = x.x;
                    dh[m] = x.y;
                }
            }
        };
        neighbours(0);
        const int cnext = slot < b1 - b0 ? a.sched[b0 + slot] : -1;
        b0 = b1;
        b1 = a.sptr[min(s + kStages + 2, nh)];
        sweep_issue<T, kStages, VPT>(a, sm, s + kStages - 1, cell[kStages - 1], slot, t, k0, act, !FWD);
        T iD[VPT];
#pragma unroll
        for (int v = 0; v < VPT; ++v) iD[v] = cf.iD[v];
        if (kAhead) coef(s + 1, cell[1]);
        if (on) {
            const size_t ck = (size_t)cell[0] * Nv + k0;
            const size_t rbase = ((size_t)(s & (kStages - 1)) * pc + slot) * tv * VPT + (size_t)t * VPT;
#pragma unroll
            for (int v = 0; v < VPT; ++v) {
                if (v > 0) neighbours(v);
                T ag = 0, ah = 0;
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    ag = mad(w[m], dg[m], ag);
                    ah = mad(w[m], dh[m], ah);
                }
                const T2 r = sm.R[rbase + v];
                T2 o;
                if (FWD) {
                    o.x = (r.x + ag) * iD[v];
                    o.y = (r.y + ah) * iD[v];
                } else {
                    o.x = mad(ag, iD[v], r.x);
                    o.y = mad(ah, iD[v], r.y);
                    T2 fv = sm.F[rbase + v];
                    fv.x += o.x;
                    fv.y += o.y;
                    f[ck + v] = fv;
                }
                ds[ck + v] = o;
            }
        }
#pragma unroll
        for (int q = 0; q + 1 < kStages; ++q) cell[q] = cell[q + 1];
        cell[kStages - 1] = cnext;
    }
    cp_wait<0>();
}

// The micro sweeps of a structured block, a warp per bundle of lines: lines run
// along the longer axis (w), 32 / G neighbouring lines of the shorter axis (t)
// by G neighbouring groups of VPT velocities make up a warp, and lane (l, g)
// marches along line l one cell per step, one step behind line l - 1.  The two
// swept neighbours of a cell are then the thread's own result of the previous
// step (registers) and lane l - 1's (a shuffle): no barrier and no shared
// memory inside a bundle.  The bundles (strips) of a block pass their border
// line on through a shared-memory ring: every kSweepBlock steps a warp
// publishes how far it is and waits, if need be, for the strip before it (whose
// border it reads) and for the strip after it (whose unread entries it must not
// overwrite).  A strip runs kSweepBlock steps behind the one before on top of
// their distance in lines, so that a block of steps needs only finished blocks.
// Everything a step reads is copied PF steps ahead into shared memory
// (cp.async: the copies of a step are awaited by their group, while loads into
// registers share the warp's few scoreboards and would wait for one another).
// A cell's record holds only the normals that the march has not met yet: its next own
// face and the two faces towards the adjacent lines; the own face behind is the
// previous cell's, with the opposite sign.
// Seams: a line's first cell stays in registers for its last one; across a seam
// between the first and the last line the first line's increments are read from
// global memory, ordered by the same flags (in one warp by a __syncwarp).
// Bound by the latency of a step (issue a third of the cycles on 64 lines), on
// large states by the copies.  Measured against one barrier per hyperplane with
// all neighbours in shared memory, forward + backward, float32: 64 x 64 cells
// with 1024 velocities 79 + 84 -> 36 + 36 us, 128 x 128 with 784 234 + 326 ->
// 83 + 92 us, 121 x 81 with 7921 950 + 1436 -> 505 + 683 us; float64 64 x 64
// 462 + 467 -> 359 + 359 us.  Loads into registers instead of cp.async took
// 53 + 51 us on 64 x 64, a warp running through the steps before its first and
// after its last cell 57 + 61 us.
// VPT consecutive T2 / the 8-entry record, by the widest loads
template <int VPT> __device__ __forceinline__ void ld_vec(float2 (&o)[VPT], const float2 *s)
{
    if constexpr (VPT == 1) {
        o[0] = *s;
    } else {
#pragma unroll
        for (int v = 0; v < VPT; v += 2) {
            const float4 a = *reinterpret_cast<const float4 *>(s + v);
            o[v] = make_float2(a.x, a.y);
            o[v + 1] = make_float2(a.z, a.w);
        }
    }
}
template <int VPT> __device__ __forceinline__ void ld_vec(double2 (&o)[VPT], const double2 *s)
{
#pragma unroll
    for (int v = 0; v < VPT; ++v) o[v] = s[v];
}
// predicated stores to global (GLOBAL) or shared memory, without a branch
template <bool GLOBAL, int VPT> __device__ __forceinline__ void st_vec(float2 *d, const float2 (&x)[VPT], bool on)
{
    if constexpr (VPT == 1) {
        if constexpr (GLOBAL)
            asm volatile("{.reg .pred p; setp.ne.s32 p, %3, 0; @p st.global.v2.f32 [%0], {%1, %2};}" ::"l"(d), "f"(x[0].x), "f"(x[0].y), "r"((int)on) : "memory");
        else
            asm volatile("{.reg .pred p; setp.ne.s32 p, %3, 0; @p st.shared.v2.f32 [%0], {%1, %2};}" ::"r"(smem_addr(d)), "f"(x[0].x), "f"(x[0].y), "r"((int)on) : "memory");
    } else {
#pragma unroll
        for (int v = 0; v < VPT; v += 2) {
            if constexpr (GLOBAL)
                asm volatile("{.reg .pred p; setp.ne.s32 p, %5, 0; @p st.global.v4.f32 [%0], {%1, %2, %3, %4};}" ::"l"(d + v), "f"(x[v].x), "f"(x[v].y), "f"(x[v + 1].x), "f"(x[v + 1].y), "r"((int)on) : "memory");
            else
                asm volatile("{.reg .pred p; setp.ne.s32 p, %5, 0; @p st.shared.v4.f32 [%0], {%1, %2, %3, %4};}" ::"r"(smem_addr(d + v)), "f"(x[v].x), "f"(x[v].y), "f"(x[v + 1].x), "f"(x[v + 1].y), "r"((int)on) : "memory");
        }
    }
}
template <bool GLOBAL, int VPT> __device__ __forceinline__ void st_vec(double2 *d, const double2 (&x)[VPT], bool on)
{
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        if constexpr (GLOBAL)
            asm volatile("{.reg .pred p; setp.ne.s32 p, %3, 0; @p st.global.v2.f64 [%0], {%1, %2};}" ::"l"(d + v), "d"(x[v].x), "d"(x[v].y), "r"((int)on) : "memory");
        else
            asm volatile("{.reg .pred p; setp.ne.s32 p, %3, 0; @p st.shared.v2.f64 [%0], {%1, %2};}" ::"r"(smem_addr(d + v)), "d"(x[v].x), "d"(x[v].y), "r"((int)on) : "memory");
    }
}
// 16-byte cp.async where on
__device__ __forceinline__ void cp_async16_if(void *s, const void *g, bool on)
{
    asm volatile("{.reg .pred p; setp.ne.s32 p, %2, 0; @p cp.async.cg.shared.global [%0], [%1], 16;}" ::"r"(smem_addr(s)), "l"(g), "r"((int)on) : "memory");
}
__device__ __forceinline__ void ld_rec7(float (&o)[7], const float *s)
{
    const float4 a = reinterpret_cast<const float4 *>(s)[0], b = reinterpret_cast<const float4 *>(s)[1];
    o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w; o[4] = b.x; o[5] = b.y; o[6] = b.z;
}
__device__ __forceinline__ void ld_rec7(double (&o)[7], const double *s)
{
    const double2 *q = reinterpret_cast<const double2 *>(s);
    const double2 a = q[0], b = q[1], c = q[2];
    o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y; o[4] = c.x; o[5] = c.y; o[6] = s[6];
}

// (Four float64 velocities per thread spill in any case; without the bound of one
// block the compiler may give them 32 registers: a 64 x 64 block with a periodic
// seam and 576 velocities then took 1600 us backward, 1000 us with it.)
template <class T, bool FWD, int VPT, int PF, bool SEAM>
__global__ void __launch_bounds__(512, sizeof(T) == 8 && VPT == 4 ? 1 : 0) k_sweep_lines(Launch L)
{
    IDG_LOCATE();
    using T2 = typename V2<T>::t;
    extern __shared__ __align__(16) unsigned char smraw[];
    int *flags = (int *)smraw;  // [16] steps done by each warp
    const bool cols = p.ni <= p.nj;
    const int nt = cols ? p.ni : p.nj, nw = cols ? p.nj : p.ni, Nv = p.Nv;
    const int G = p.sweep_g, lw = 32 / G, strips = (nt + lw - 1) / lw, subs = p.sweep_ktv / G;
    const int wid = threadIdx.x >> 5, sub = wid / strips, strip = wid - sub * strips;
    // step s of the block's clock: the lane of line tt is at its cell
    // ww = s - tt - strip * kSweepBlock; a warp runs from its first line's first
    // cell to its last line's last one
    const int s_beg = (strip * (lw + kSweepBlock)) & ~(kSweepBlock - 1);
    const int s_end = strip * (lw + kSweepBlock) + nw + min(lw, nt - strip * lw) - 1;
    if ((threadIdx.x & 31) == 0) flags[wid] = s_beg;
    __syncthreads();
    if (sub >= subs) return;  // a smaller instance of a batch
    const int lane = threadIdx.x & 31, l = lane / G, g = lane - l * G;
    const int tt = strip * lw + l;  // line in sweep order
    const int tc = min(tt, nt - 1);
    const int k0 = ((blk * subs + sub) * G + g) * VPT;
    const bool line = tt < nt && k0 < Nv, has_adj = tt > 0;
    const int kk = k0 < Nv ? k0 : 0;
    T ux[VPT], uy[VPT];
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        ux[v] = vx<T>(p, kk + v);
        uy[v] = vy<T>(p, kk + v);
    }
    // cell of (tt, ww): c0 + ww * cs, ww counted from the end the sweep starts at
    const int t = FWD ? tc : nt - 1 - tc;
    const int cs = (FWD ? 1 : -1) * (cols ? p.ni : 1);
    const int c0 = (cols ? t : t * p.ni) + (FWD ? 0 : (nw - 1) * (cols ? p.ni : 1));
    const int sv = cs * Nv, sg = cs * 8;
    T2 *ds = (T2 *)p.dst + (ptrdiff_t)c0 * Nv + kk;
    T2 *fs = (T2 *)p.f + (ptrdiff_t)c0 * Nv + kk;
    const T *geo = (const T *)p.sgeo + (FWD ? 0 : (ptrdiff_t)p.N * 8) + (ptrdiff_t)c0 * 8;
    const unsigned nwl = line ? nw : 0;
    const int start = tt + strip * kSweepBlock;
    const bool seam_t = SEAM && (cols ? p.per_i : p.per_j) && nt > 1;
    const bool seam_w = SEAM && (cols ? p.per_j : p.per_i) && nw > 1;
    // shared memory: flags, border rings [warp][ring][G * VPT], stages
    // [warp][PF] of {R or Delta*, f~ (backward), cell records}
    const int ring = p.sweep_ring, xs = G * VPT, nwarp = subs * strips;
    T2 *xw = (T2 *)(smraw + 64) + (size_t)wid * ring * xs + g * VPT;
    const T2 *xr = strip > 0 ? xw - (size_t)ring * xs : xw;  // the strip before's
    const bool edge = l == 0 && strip > 0, border = l == lw - 1 && strip + 1 < strips;
    constexpr int RB = 32 * VPT * sizeof(T2), FB = FWD ? 0 : RB, CB = 8 * sizeof(T);
    const int SB = RB + FB + lw * CB;
    unsigned char *stage = smraw + 64 + (size_t)nwarp * ring * xs * sizeof(T2) + (size_t)wid * PF * SB;

    // every lane copies at every step (lanes without a cell their line's end
    // cells, or an existing line's): no branch in the step
    auto issue = [&](int s) {
        const int wc = min(max(s - start, 0), nw - 1);
        unsigned char *st = stage + (s & (PF - 1)) * SB;
        constexpr int B = VPT * sizeof(T2), CH = B < 16 ? B : 16;
        const char *gr = (const char *)(ds + (ptrdiff_t)wc * sv);
#pragma unroll
        for (int o = 0; o < B; o += CH) cp_async_b<CH>(st + lane * B + o, gr + o);
        if (!FWD) {
            const char *gf = (const char *)(fs + (ptrdiff_t)wc * sv);
#pragma unroll
            for (int o = 0; o < B; o += CH) cp_async_b<CH>(st + RB + lane * B + o, gf + o);
        }
        // the line's record, spread over its lanes
        const char *gg = (const char *)(geo + (ptrdiff_t)wc * sg);
#pragma unroll
        for (int q = 0; q < CB / 16; ++q)
            cp_async16_if(st + RB + FB + l * CB + 16 * (g + q * G), gg + 16 * (g + q * G), 16 * (g + q * G) < CB);
        cp_commit();
    };
    for (int u = 0; u < PF; ++u) issue(s_beg + u);
    // (xi.n) S of the line's end face, outward from its first cell (0 where
    // the cell is its own neighbour)
    T end[VPT];
    {
        const int wm = (cols ? 2 : 0) + (FWD ? 0 : 1);
        const bool self = nw == 1 && (cols ? p.per_j : p.per_i);
        const T *e = (const T *)p.cslotT + 8 * (ptrdiff_t)c0 + 2 * wm;
#pragma unroll
        for (int v = 0; v < VPT; ++v) end[v] = self ? (T)0 : xi_dot_n<T>(ux[v], uy[v], e[0], e[1]);
    }
    T2 prev[VPT], first[VPT];
    // a step's coefficients, formed one step ahead of their use so that only
    // the increments are left on the chain from step to step: (xi.n) S inflow
    // from the adjacent line and from the own one, 1 / D, and the two faces
    // that a seam can lie on
    T cl[VPT], co[VPT], iD[VPT], ca[VPT], cu[VPT], ahead[VPT];
    auto coef = [&](int s) {
        const int ww = s - start;
        T q[7];
        ld_rec7(q, (const T *)(stage + (s & (PF - 1)) * SB + RB + FB + l * CB));
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            const T own = ww > 0 ? -ahead[v] : end[v];  // the face ahead of the cell before
            ahead[v] = xi_dot_n<T>(ux[v], uy[v], q[0], q[1]);
            const T low = xi_dot_n<T>(ux[v], uy[v], q[2], q[3]);
            const T upp = xi_dot_n<T>(ux[v], uy[v], q[4], q[5]);
            // D = base + sum of the outflow (xi.n) S: half the sum of all
            // |xi.n| S, the cell's outward normals summing to zero; pair by pair
            // (opposite faces: on a uniform block the sum is exact) onto the
            // base, which differs from cell to cell: all four summed first are
            // rounded alike in every cell of a uniform block, an error that adds
            // up along the line (0.96e-9 instead of 0.42e-9 rms in G after 16
            // iterations on 90 x 70 cells, float32)
            const T D = mad((T)0.5, fabs(low) + fabs(upp), mad((T)0.5, fabs(own) + fabs(ahead[v]), q[6]));
            iD[v] = rcp_nr(D);
            cl[v] = low < (T)0 && has_adj ? -low : (T)0;
            co[v] = own < (T)0 && ww > 0 ? -own : (T)0;
            if (SEAM) {
                ca[v] = seam_w && ww == nw - 1 && ahead[v] < (T)0 ? -ahead[v] : (T)0;
                cu[v] = seam_t && tt == nt - 1 && upp < (T)0 ? -upp : (T)0;
            }
        }
    };
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        prev[v].x = prev[v].y = first[v].x = first[v].y = (T)0;
        ahead[v] = (T)0;
    }
    cp_wait<PF - 1>();
    __syncwarp();
    coef(s_beg);
    int seen_r = 0, seen_w = 0;

    for (int s0 = s_beg; s0 < s_end; s0 += kSweepBlock) {
        if (strips > 1) {
            // reads what the strip before wrote in steps < s0; overwrites what the
            // strip after reads in steps <= s0 + 2 kSweepBlock - ring
            if (strip > 0) flag_wait(flags + wid - 1, s0, seen_r, p.status, p.wait_polls);
            if (strip + 1 < strips) flag_wait(flags + wid + 1, s0 + 2 * kSweepBlock + 1 - ring, seen_w, p.status, p.wait_polls);
        }
#pragma unroll
        for (int b = 0; b < kSweepBlock; ++b) {
            const int s = s0 + b, ww = s - start;
            cp_wait<PF - 2>();  // the copies of this step and the next one's records
            __syncwarp();
            const bool on = (unsigned)ww < nwl;
            const unsigned char *st = stage + (s & (PF - 1)) * SB;
            T2 ev[VPT], out[VPT], r[VPT], f[VPT];
            ld_vec<VPT>(ev, xr + (ww & (ring - 1)) * xs);
            ld_vec<VPT>(r, (const T2 *)st + lane * VPT);
            if (!FWD) ld_vec<VPT>(f, (const T2 *)(st + RB) + lane * VPT);
#pragma unroll
            for (int v = 0; v < VPT; ++v) {
                T2 adj;
                adj.x = __shfl_up_sync(0xffffffffu, prev[v].x, G);
                adj.y = __shfl_up_sync(0xffffffffu, prev[v].y, G);
                adj.x = edge ? ev[v].x : adj.x;
                adj.y = edge ? ev[v].y : adj.y;
                // inflow from the swept side adds |xi.n| S Delta_nb
                T ag = co[v] * prev[v].x, ah = co[v] * prev[v].y;
                ag = mad(cl[v], adj.x, ag);
                ah = mad(cl[v], adj.y, ah);
                if (SEAM) {
                    if (ca[v] > (T)0) {
                        ag = mad(ca[v], first[v].x, ag);
                        ah = mad(ca[v], first[v].y, ah);
                    }
                    if (on && cu[v] > (T)0) {
                        const int nb = (FWD ? 0 : nt - 1) - t;  // lines to the first line of the sweep
                        const T2 dn = ds[(ptrdiff_t)ww * sv + (ptrdiff_t)nb * (cols ? 1 : p.ni) * Nv + v];
                        ag = mad(cu[v], dn.x, ag);
                        ah = mad(cu[v], dn.y, ah);
                    }
                }
                if (FWD) {
                    out[v].x = (r[v].x + ag) * iD[v];
                    out[v].y = (r[v].y + ah) * iD[v];
                } else {
                    out[v].x = mad(ag, iD[v], r[v].x);
                    out[v].y = mad(ah, iD[v], r[v].y);
                    f[v].x += out[v].x;
                    f[v].y += out[v].y;
                }
                prev[v] = out[v];
                if (SEAM && ww == 0) first[v] = out[v];
            }
            coef(s + 1);
            if (FWD || SEAM) st_vec<true, VPT>(ds + (ptrdiff_t)ww * sv, out, on && (FWD || (seam_t && tt == 0)));
            if (!FWD) st_vec<true, VPT>(fs + (ptrdiff_t)ww * sv, f, on);
            st_vec<false, VPT>(xw + (ww & (ring - 1)) * xs, out, on && border);
            issue(s + PF);
        }
        if (strips > 1) {
            __syncwarp();
            if (lane == 0) flag_store(flags + wid, s0 + kSweepBlock);
        }
    }
    cp_wait<0>();
    if (strips > 1) {
        __syncwarp();
        if (lane == 0) flag_store(flags + wid, 0x7fffffff);
    }
}

// ---------------------------------------------------------------------------
// state conversion and diagnostics
// ---------------------------------------------------------------------------
template <class T>
__global__ void k_to_dev(KParams p, const double *G, const double *H, int nvu, int deviation)
{
    using T2 = typename V2<T>::t;
    size_t n = (size_t)p.N * p.Nv;
    // deviation: G, H already hold f~ - M_ref (a checkpoint's stored form)
    const double ref = deviation ? 0.0 : 1.0;
    double kRTr = p.K * p.RT_r;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        const size_t c = i / p.Nv;
        const int k = (int)(i - c * p.Nv);
        T2 o;
        o.x = (T)0;
        o.y = (T)0;
        if (k < nvu) {
            const size_t j = c * nvu + k;
            o.x = (T)(G[j] - ref * p.gref[k]);
            o.y = (T)(H[j] - ref * kRTr * p.gref[k]);
        }
        ((T2 *)p.f)[i] = o;
    }
}

template <class T>
__global__ void k_from_dev(KParams p, double *G, double *H, int nvu, int deviation)
{
    using T2 = typename V2<T>::t;
    size_t n = (size_t)p.N * p.Nv;
    const double ref = deviation ? 0.0 : 1.0;
    double kRTr = p.K * p.RT_r;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        const size_t c = i / p.Nv;
        const int k = (int)(i - c * p.Nv);
        if (k >= nvu) continue;
        const size_t j = c * nvu + k;
        T2 v = ((const T2 *)p.f)[i];
        G[j] = ref * p.gref[k] + (double)v.x;
        H[j] = ref * kRTr * p.gref[k] + (double)v.y;
    }
}

// per cell: rho, u, v, T/T_ref from W; heat flux of f from f~ (cellraw)
template <class T>
__global__ void __launch_bounds__(256) k_moments_out(KParams p, double *out6)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= p.N) return;
    double r[kRaw];
    for (int q = 0; q < kRaw; ++q) r[q] = acc_load<T>(p.cellraw, (size_t)c * kRaw + q) + p.mref_raw[q];
    const double *W = p.W + 4 * c;
    const double rho = W[0], irho = rcp_rn(rho), U = W[1] * irho, V = W[2] * irho;
    const double RT = mad(-V, V, mad(-U, U, 2.0 * W[3] * irho)) * p.iK2;
    const double tau2 = 2.0 * viscosity_t<T>(p, RT) * (irho * rcp_rn(RT));  // 2 tau
    double qtx, qty;
    raw_heat_flux(r, U, V, qtx, qty);
    const double Pr = p.shakhov ? p.Pr : 1.0, fq = tau2 * rcp_rn(tau2 + p.dt * Pr);
    out6[6 * c + 0] = rho;
    out6[6 * c + 1] = U;
    out6[6 * c + 2] = V;
    out6[6 * c + 3] = RT * p.iRT_ref;
    out6[6 * c + 4] = fq * qtx;
    out6[6 * c + 5] = fq * qty;
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static inline int nblk(int n, int per) { return (n + per - 1) / per; }

static int macro_threads(const KParams &p) { return std::min(512, ((2 * std::min(p.ni, p.nj) + 31) / 32) * 32); }

template <class T> static size_t macro_smem_bytes(const KParams &p, int nt, int stages)
{
    return (size_t)stages * (nt / 2) * (kMRec + 4) * sizeof(T) + (size_t)2 * (nt / 2) * kMRing * sizeof(T);
}

// shared memory of the scheduled micro sweeps (a 4-step prefetch)
template <class T> static size_t sched_sweep_bytes(const KParams &p, bool withF)
{
    switch (p.sweep_vpt) {
    case 4: return sweep_smem_bytes<T, 4, 4>(p.sweep_pc, p.sweep_tv, withF);
    case 2: return sweep_smem_bytes<T, 4, 2>(p.sweep_pc, p.sweep_tv, withF);
    default: return sweep_smem_bytes<T, 4, 1>(p.sweep_pc, p.sweep_tv, withF);
    }
}

// warps of a line-sweep block, and its shared memory
static int sweep_line_warps(const KParams &p)
{
    const int lw = 32 / p.sweep_g;
    return p.sweep_ktv / p.sweep_g * ((p.sweep_pc + lw - 1) / lw);
}
static size_t sweep_line_bytes(const KParams &p, bool fp64, bool withF, int stages)
{
    const size_t T2 = fp64 ? 16 : 8, v = p.sweep_kvpt, g = p.sweep_g;
    return 64 + sweep_line_warps(p) * (p.sweep_ring * g * v * T2 + stages * (32 * v * T2 * (withF ? 2 : 1) + 32 / g * 4 * T2));
}

constexpr size_t kMaxSmem = 227 * 1024;  // dynamic shared memory of a block

// What a caller asks of the micro sweeps: the copies of sweep_stages steps of
// sweep_pc cells (backward: Delta* and f~ of the tile's velocities, a record of
// twelve scalars) and two steps' borders.  The line sweeps may need more, lines
// padded to whole warps and rings; they then take the next shallower depth
// (plan_shapes), which idg_get_tuning reads back: at two steps every tile fits
// that is accepted here.  (Where they need less, what they can run is taken too.)
bool sweep_request_fits(const KParams &p, bool fp64)
{
    const size_t T = fp64 ? 8 : 4, w = (size_t)p.sweep_tv * p.sweep_vpt * 2 * T, st = p.sweep_stages;
    return p.sweep_pc * (st * (2 * w + 9 * T + 16) + 2 * w) <= kMaxSmem;
}

void sweep_shape(KParams &p, bool fp64, int vpt)
{
    p.sweep_ktv = p.sweep_tv;
    p.sweep_kvpt = vpt ? vpt : p.sweep_vpt;
    if (p.sched) return;
    // at most eight velocity groups in a warp, so that it keeps at least four
    // lines in step, but none of its lanes goes to lines a narrow block lacks
    int lines = 1;
    while (lines < p.sweep_pc && lines < 32) lines *= 2;
    if (!(p.sweep_tuned & 1)) {
        // four groups (eight lines a warp) where the block has that many lines,
        // more on a narrow one
        p.sweep_ktv = std::max(4, 128 / lines > 32 ? 32 : 128 / lines);
        while (p.sweep_ktv * p.sweep_pc > 512) p.sweep_ktv /= 2;
    }
    if (!(p.sweep_tuned & 2) && !vpt) {
        // two velocities per thread (16-byte copies); one where that leaves
        // fewer than a warp for each scheduler; four where the warps are many
        // waves (float64 is bound by its arithmetic pipe: one)
        const int lw = 32 / std::min(p.sweep_ktv, std::max(8, 32 / lines));
        const int warps = (p.sweep_pc + lw - 1) / lw * (p.Nv / (2 * std::min(p.sweep_ktv, 32 / lw)));
        p.sweep_kvpt = fp64 || warps < 4 * kSMs ? 1 : warps > 32 * kSMs ? 4 : 2;
    }
    // 32 ring entries let neighbouring strips drift a few blocks of steps apart
    // (at least 2 blocks + 5 are needed: 16).  Where shared memory holds neither
    // that nor 16 -- the library's own tile at the shallowest prefetch, a caller's
    // at the one asked for, then the shallower ones -- a warp takes more lines:
    // fewer, longer strips with less border between them, as far as 512 threads
    // hold the padded lines
    const int g0 = std::min(p.sweep_ktv, std::max(8, 32 / lines));
    for (int st = p.sweep_tuned & 3 ? p.sweep_stages : 2; st >= 2; st /= 2)
        for (p.sweep_g = g0; p.sweep_g >= 1 && 16 * p.sweep_g >= p.sweep_ktv; p.sweep_g /= 2)
            for (p.sweep_ring = 32; p.sweep_ring >= 16; p.sweep_ring /= 2)
                if (sweep_line_bytes(p, fp64, true, st) <= kMaxSmem) return;
    p.sweep_g = g0;
    p.sweep_ring = 32;  // (does not fit: plan_shapes refuses it)
}

void blocks_per_instance(const KParams &p, int out[KT_COUNT])
{
    const int nvb = nblk(p.Nv, 256);
    out[KT_CELL_MOM] = nblk(p.N, 8 / p.row_warps);
    out[KT_CELL_PAR] = nblk(p.N, 32);
    out[KT_FBP] = nblk(p.N, p.cpb) * nvb;
    out[KT_FACE_MOM] = nblk(p.nf, 8);
    out[KT_FACE_PAR] = nblk(p.nf, 32);
    out[KT_FACE_FLUX] = nblk(p.nf, 8);
    out[KT_FACE_PHI] = nblk(p.nf, 64);
    out[KT_MACRO_PRE] = nblk(p.N, 32);
    out[KT_MACRO_SWEEP] = 1;
    out[KT_MACRO_POST] = nblk(p.N, 32);
    out[KT_MICRO_RES] = nblk(p.N, p.cpb) * nvb;
    out[KT_SWEEP] = nblk(p.Nv, p.sweep_ktv * p.sweep_kvpt);
}

// block shape, shared memory and prefetch depth common to all instances of
// a plan (the maxima of the instances; the deepest pipeline that fits all)
int plan_shapes(const KParams *hp, int n, bool fp64, Plan &pl)
{
    const size_t lim = kMaxSmem;
    pl.macro_threads = pl.sweep_threads = 0;
    pl.limiter_any = 0;
    pl.sweep_vpt = hp[0].sweep_kvpt;
    pl.relax_sweeps = hp[0].relax_sweeps;
    pl.sched = hp[0].sched != nullptr;
    pl.sched_smem = 0;
    for (int i = 0; i < n; ++i) {
        if ((hp[i].sched != nullptr) != (pl.sched != 0)) return (int)cudaErrorInvalidValue;
        pl.sched_smem = std::max(pl.sched_smem, (size_t)hp[i].N * 4 * (fp64 ? 8 : 4));
        if (hp[i].relax_sweeps != pl.relax_sweeps) return (int)cudaErrorInvalidValue;
        pl.macro_threads = std::max(pl.macro_threads, macro_threads(hp[i]));
        pl.sweep_threads = std::max(pl.sweep_threads, pl.sched ? hp[i].sweep_ktv * hp[i].sweep_pc : 32 * sweep_line_warps(hp[i]));
        pl.limiter_any |= hp[i].limiter;
        if (hp[i].sweep_vpt != hp[0].sweep_vpt || hp[i].sweep_kvpt != pl.sweep_vpt) return (int)cudaErrorInvalidValue;
    }
    if (!pl.sched || pl.sched_smem > 200 * 1024) pl.sched_smem = 0;
    pl.any_seam = 0;
    for (int i = 0; i < n; ++i) pl.any_seam |= hp[i].per_i | hp[i].per_j;
    pl.macro_kind = hp[0].macro_kind;
    for (int i = 0; i < n; ++i)
        if (hp[i].macro_kind != pl.macro_kind) return (int)cudaErrorInvalidValue;
    if (pl.macro_kind == 1 && !pl.sched) {
        // one thread per line of the shorter axis; the seam array holds the
        // walk axis' cells when the lines wrap around (a periodic shorter axis)
        int ntmax = 0;
        for (int i = 0; i < n; ++i) ntmax = std::max(ntmax, std::min(hp[i].ni, hp[i].nj));
        const int nlines = ((ntmax + 31) / 32) * 32;
        pl.macro_threads = nlines + 32;  // and the residual's warp
        for (int stages : {std::min(hp[0].macro_stages, 8), 4, 2}) {
            size_t m = 0;
            for (int i = 0; i < n; ++i) {
                const bool cols = hp[i].ni <= hp[i].nj;
                const bool seam = cols ? hp[i].per_i : hp[i].per_j;
                const int nw = std::max(hp[i].ni, hp[i].nj);
                m = std::max(m, fp64 ? macro_lines_smem_bytes<double>(nlines, stages, nw, seam)
                                     : macro_lines_smem_bytes<float>(nlines, stages, nw, seam));
            }
            pl.macro_stages = stages;
            pl.macro_smem = m;
            if (m <= lim) break;
        }
    } else {
    // a 2-stage prefetch is the fallback that fits a 256-cell hyperplane of
    // float64 records
    for (int stages : {std::min(hp[0].macro_stages, 8), 4, 2}) {
        size_t m = 0;
        for (int i = 0; i < n; ++i)
            m = std::max(m, fp64 ? macro_smem_bytes<double>(hp[i], pl.macro_threads, stages)
                                 : macro_smem_bytes<float>(hp[i], pl.macro_threads, stages));
        pl.macro_stages = stages;
        pl.macro_smem = m;
        if (m <= lim) break;
    }
    }
    for (int stages : {pl.sched ? 4 : std::min(hp[0].sweep_stages, 8), 4, 2}) {
        pl.sweep_stages = stages;
        pl.fwd_smem = pl.bwd_smem = 0;
        for (int i = 0; i < n; ++i) {
            auto bytes = [&](bool withF) {
                return !pl.sched ? sweep_line_bytes(hp[i], fp64, withF, stages)
                                 : fp64 ? sched_sweep_bytes<double>(hp[i], withF) : sched_sweep_bytes<float>(hp[i], withF);
            };
            pl.fwd_smem = std::max(pl.fwd_smem, bytes(false));
            pl.bwd_smem = std::max(pl.bwd_smem, bytes(true));
        }
        if (pl.bwd_smem <= lim || pl.sched) break;
    }
    if (pl.macro_smem > lim || pl.bwd_smem > lim) return (int)cudaErrorInvalidValue;
    return 0;
}

// every instantiation of the micro sweeps, by the plan's shape: visit(kernel)
template <class T, bool FWD, class F> static void sweep_kernel(const Plan &pl, F visit)
{
    const int v = pl.sweep_vpt;
    if (pl.sched) {
        if (v == 4) visit(k_sweep<T, FWD, 4, 4>);
        else if (v == 2) visit(k_sweep<T, FWD, 4, 2>);
        else visit(k_sweep<T, FWD, 4, 1>);
        return;
    }
    auto lines = [&](auto seam) {
        constexpr bool SEAM = decltype(seam)::value;
        auto depth = [&](auto stages) {
            constexpr int PF = decltype(stages)::value;
            if (v == 4) visit(k_sweep_lines<T, FWD, 4, PF, SEAM>);
            else if (v == 2) visit(k_sweep_lines<T, FWD, 2, PF, SEAM>);
            else visit(k_sweep_lines<T, FWD, 1, PF, SEAM>);
        };
        if (pl.sweep_stages == 8) depth(std::integral_constant<int, 8>{});
        else if (pl.sweep_stages == 4) depth(std::integral_constant<int, 4>{});
        else depth(std::integral_constant<int, 2>{});
    };
    if (pl.any_seam) lines(std::true_type{});
    else lines(std::false_type{});
}

template <class T, bool FWD> static void launch_sweep(const Plan &pl, cudaStream_t st, const Launch &L)
{
    const size_t sm = FWD ? pl.fwd_smem : pl.bwd_smem;
    sweep_kernel<T, FWD>(pl, [&](auto k) { k<<<pl.nblocks[KT_SWEEP], pl.sweep_threads, sm, st>>>(L); });
}

template <class T> static Launch launch_of(const Plan &pl, int kt)
{
    Launch L;
    L.params = pl.dparams;
    L.off = pl.doff ? pl.doff + (size_t)kt * (pl.ninst + 1) : nullptr;
    L.active = pl.dactive;
    L.ninst = pl.ninst;
    return L;
}

// run(launch, blocks) of kernel type kt, for one instance by value, for a batch
// through its tables
template <class F> static void run_plan(const Plan &pl, int kt, F launch)
{
    if (pl.hparams) launch(LaunchOne{*pl.hparams}, pl.nblocks[kt]);
    else launch(launch_of<void>(pl, kt), pl.nblocks[kt]);
}

// events (optional): kProfiled+1 cudaEvent_t recorded between the six groups
// cell prep | face moments+params | face flux+phi | macro | residual+fwd | bwd
template <class T>
static int iteration_t(const Plan &pl, cudaStream_t st, void **events)
{
    auto mark = [&](int q) {
        if (events) cudaEventRecord((cudaEvent_t)events[q], st);
    };
    auto L = [&](int kt) { return launch_of<T>(pl, kt); };
    auto run = [&](int kt, auto launch) { run_plan(pl, kt, launch); };
    const int *nb = pl.nblocks;
    if (pl.explicit_dugks) {
        // W^n and the raw moments of f~^n are left by the previous step (or
        // by launch_explicit_prologue)
        mark(0);
        run(KT_CELL_PAR, [&](const auto &l, int nb) { k_cell_params<T, std::decay_t<decltype(l)>><<<nb, 32, 0, st>>>(l); });
        run(KT_FBP, [&](const auto &l, int nb) { k_fbp<T, std::decay_t<decltype(l)>><<<nb, 128, 0, st>>>(l); });
        mark(1);
        if (pl.limiter_any) run(KT_FBP, [&](const auto &l, int nb) { k_cell_recon<T, true, std::decay_t<decltype(l)>><<<nb, 128, 0, st>>>(l); });
        else run(KT_FBP, [&](const auto &l, int nb) { k_cell_recon<T, false, std::decay_t<decltype(l)>><<<nb, 128, 0, st>>>(l); });
        run(KT_FACE_MOM, [&](const auto &l, int nb) { k_face_moments<T, std::decay_t<decltype(l)>><<<nb, 256, 0, st>>>(l); });
        run(KT_FACE_PAR, [&](const auto &l, int nb) { k_face_params<T, std::decay_t<decltype(l)>><<<nb, 32, 0, st>>>(l); });
        mark(2);
        run(KT_FACE_FLUX, [&](const auto &l, int nb) { k_face_flux<T, std::decay_t<decltype(l)>><<<nb, 256, 0, st>>>(l); });
        run(KT_FACE_PHI, [&](const auto &l, int nb) { k_face_phi<T, std::decay_t<decltype(l)>><<<nb, 64, 0, st>>>(l); });
        mark(3);
        mark(4);
        run(KT_MICRO_RES, [&](const auto &l, int nb) { k_explicit_update<T, std::decay_t<decltype(l)>><<<nb, 128, 0, st>>>(l); });
        run(KT_CELL_MOM, [&](const auto &l, int nb) { k_cell_moments<T, std::decay_t<decltype(l)>><<<nb, 256, 0, st>>>(l); });
        run(KT_CELL_PAR, [&](const auto &l, int nb) { k_explicit_w<T, std::decay_t<decltype(l)>><<<nb, 32, 0, st>>>(l); });
        run(KT_MACRO_SWEEP, [&](const auto &l, int nb) { k_record_residual<T, std::decay_t<decltype(l)>><<<nb, 32, 0, st>>>(l); });
        mark(5);
        mark(6);
        return (int)cudaGetLastError();
    }
    mark(0);
    run(KT_CELL_MOM, [&](const auto &l, int nb) { k_cell_moments<T, std::decay_t<decltype(l)>><<<nb, 256, 0, st>>>(l); });
    run(KT_CELL_PAR, [&](const auto &l, int nb) { k_cell_params<T, std::decay_t<decltype(l)>><<<nb, 32, 0, st>>>(l); });
    run(KT_FBP, [&](const auto &l, int nb) { k_fbp<T, std::decay_t<decltype(l)>><<<nb, 128, 0, st>>>(l); });
    mark(1);
    if (pl.limiter_any) run(KT_FBP, [&](const auto &l, int nb) { k_cell_recon<T, true, std::decay_t<decltype(l)>><<<nb, 128, 0, st>>>(l); });
    else run(KT_FBP, [&](const auto &l, int nb) { k_cell_recon<T, false, std::decay_t<decltype(l)>><<<nb, 128, 0, st>>>(l); });
    run(KT_FACE_MOM, [&](const auto &l, int nb) { k_face_moments<T, std::decay_t<decltype(l)>><<<nb, 256, 0, st>>>(l); });
    run(KT_FACE_PAR, [&](const auto &l, int nb) { k_face_params<T, std::decay_t<decltype(l)>><<<nb, 32, 0, st>>>(l); });
    mark(2);
    run(KT_FACE_FLUX, [&](const auto &l, int nb) { k_face_flux<T, std::decay_t<decltype(l)>><<<nb, 256, 0, st>>>(l); });
    run(KT_FACE_PHI, [&](const auto &l, int nb) { k_face_phi<T, std::decay_t<decltype(l)>><<<nb, 64, 0, st>>>(l); });
    mark(3);
    run(KT_MACRO_PRE, [&](const auto &l, int nb) { k_macro_pre<T, std::decay_t<decltype(l)>><<<nb, 32, 0, st>>>(l); });
    if (pl.relax_sweeps > 0) {
        run(KT_MACRO_SWEEP, [&](const auto &l, int nb) { k_record_residual<T, std::decay_t<decltype(l)>><<<nb, 32, 0, st>>>(l); });
        for (int k = 1; k <= pl.relax_sweeps; ++k)
            run(KT_MACRO_PRE, [&](const auto &l, int nb) { k_macro_relax<T, std::decay_t<decltype(l)>><<<nb, 32, 0, st>>>(l, k, pl.relax_sweeps); });
    } else if (pl.sched) {
        if (pl.sched_smem)
            k_macro_sweep_sched<T, true><<<nb[KT_MACRO_SWEEP], 256, pl.sched_smem, st>>>(L(KT_MACRO_SWEEP));
        else
            k_macro_sweep_sched<T, false><<<nb[KT_MACRO_SWEEP], 256, 0, st>>>(L(KT_MACRO_SWEEP));
    } else if (pl.macro_kind == 1) {
        const int nb1 = nb[KT_MACRO_SWEEP], nt1 = pl.macro_threads;
        const size_t sm1 = pl.macro_smem;
        const Launch L1 = L(KT_MACRO_SWEEP);
        if (pl.any_seam) {
            if (pl.macro_stages == 8) k_macro_lines<T, 8, true><<<nb1, nt1, sm1, st>>>(L1);
            else if (pl.macro_stages == 4) k_macro_lines<T, 4, true><<<nb1, nt1, sm1, st>>>(L1);
            else k_macro_lines<T, 2, true><<<nb1, nt1, sm1, st>>>(L1);
        } else {
            if (pl.macro_stages == 8) k_macro_lines<T, 8, false><<<nb1, nt1, sm1, st>>>(L1);
            else if (pl.macro_stages == 4) k_macro_lines<T, 4, false><<<nb1, nt1, sm1, st>>>(L1);
            else k_macro_lines<T, 2, false><<<nb1, nt1, sm1, st>>>(L1);
        }
    } else if (pl.macro_stages == 8)
        k_macro_sweep<T, 8><<<nb[KT_MACRO_SWEEP], pl.macro_threads, pl.macro_smem, st>>>(L(KT_MACRO_SWEEP));
    else if (pl.macro_stages == 4)
        k_macro_sweep<T, 4><<<nb[KT_MACRO_SWEEP], pl.macro_threads, pl.macro_smem, st>>>(L(KT_MACRO_SWEEP));
    else
        k_macro_sweep<T, 2><<<nb[KT_MACRO_SWEEP], pl.macro_threads, pl.macro_smem, st>>>(L(KT_MACRO_SWEEP));
    run(KT_MACRO_POST, [&](const auto &l, int nb) { k_macro_post<T, std::decay_t<decltype(l)>><<<nb, 32, 0, st>>>(l); });
    mark(4);
    run(KT_MICRO_RES, [&](const auto &l, int nb) { k_micro_residual<T, std::decay_t<decltype(l)>><<<nb, 128, 0, st>>>(l); });
    launch_sweep<T, true>(pl, st, L(KT_SWEEP));
    mark(5);
    launch_sweep<T, false>(pl, st, L(KT_SWEEP));
    mark(6);
    return (int)cudaGetLastError();
}

// opt the wavefront kernels in to the largest dynamic shared memory once
template <class T> static int configure_t()
{
    const int lim = (int)kMaxSmem;
    cudaError_t e = cudaSuccess;
    auto opt = [&](const void *fn) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    };
    opt((const void *)k_macro_sweep_sched<T, true>);
    opt((const void *)k_macro_lines<T, 8, false>);
    opt((const void *)k_macro_lines<T, 4, false>);
    opt((const void *)k_macro_lines<T, 2, false>);
    opt((const void *)k_macro_lines<T, 8, true>);
    opt((const void *)k_macro_lines<T, 4, true>);
    opt((const void *)k_macro_lines<T, 2, true>);
    opt((const void *)k_macro_sweep<T, 8>);
    opt((const void *)k_macro_sweep<T, 4>);
    opt((const void *)k_macro_sweep<T, 2>);
    return (int)e;
}

// the plan's two micro-sweep kernels likewise
template <class T> static int configure_sweeps_t(const Plan &pl)
{
    cudaError_t e = cudaSuccess;
    auto opt = [&](auto k) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute((const void *)k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
    };
    sweep_kernel<T, true>(pl, opt);
    sweep_kernel<T, false>(pl, opt);
    return (int)e;
}

int configure_sweeps(const Plan &pl, bool fp64)
{
    return fp64 ? configure_sweeps_t<double>(pl) : configure_sweeps_t<float>(pl);
}

int configure_kernels(bool fp64) { return fp64 ? configure_t<double>() : configure_t<float>(); }

int launch_iteration(const Plan &pl, bool fp64, void *stream, void **events)
{
    cudaStream_t st = (cudaStream_t)stream;
    return fp64 ? iteration_t<double>(pl, st, events) : iteration_t<float>(pl, st, events);
}

template <class T> static int explicit_prologue_t(const Plan &pl, cudaStream_t st)
{
    auto run = [&](int kt, auto launch) { run_plan(pl, kt, launch); };
    run(KT_CELL_MOM, [&](const auto &l, int nb) { k_cell_moments<T, std::decay_t<decltype(l)>><<<nb, 256, 0, st>>>(l); });
    run(KT_CELL_PAR, [&](const auto &l, int nb) { k_explicit_w<T, std::decay_t<decltype(l)>><<<nb, 32, 0, st>>>(l); });
    return (int)cudaGetLastError();
}

int launch_explicit_prologue(const Plan &pl, bool fp64, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    return fp64 ? explicit_prologue_t<double>(pl, st) : explicit_prologue_t<float>(pl, st);
}

int launch_cell_moments(const KParams &p, bool fp64, double *out6_dev, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (fp64) {
        k_cell_moments_v<double><<<nblk(p.N, 8 / p.row_warps), 256, 0, st>>>(p);
        k_moments_out<double><<<nblk(p.N, 256), 256, 0, st>>>(p, out6_dev);
    } else {
        k_cell_moments_v<float><<<nblk(p.N, 8 / p.row_warps), 256, 0, st>>>(p);
        k_moments_out<float><<<nblk(p.N, 256), 256, 0, st>>>(p, out6_dev);
    }
    return (int)cudaGetLastError();
}

// ---------------------------------------------------------------------------
// moments without a workspace scratch region
// ---------------------------------------------------------------------------
// Raw-moment scratch of idg_get_moments_noalloc: kNoAllocMaxCells cells x
// kRaw accumulators of 8 bytes (1.375 MiB), held by every GPU that loads the
// library until the process exits.  Every call overwrites all entries it
// reads, so nothing needs clearing; calls that overlap on the GPU race on it.
static __device__ __align__(256) unsigned char g_noalloc_raw[(size_t)kNoAllocMaxCells * kRaw * 8];

// Device address of the scratch, resolved once per device with that device
// current (a host-side use of the symbol's name is not a device address).
// The cache is guarded by a mutex: first calls from several host threads at
// once resolve it once.  It is keyed by device ordinal, so a cudaDeviceReset
// of that device (which unloads the module) leaves a stale address behind.
static void *noalloc_scratch(int device, int *err)
{
    static std::mutex mu;
    static void *addr[64] = {nullptr};
    *err = 0;
    if (device < 0 || device >= 64) {
        *err = (int)cudaErrorInvalidDevice;
        return nullptr;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[device]) {
        void *ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_raw);
        if (e != cudaSuccess) {
            *err = (int)e;
            return nullptr;
        }
        addr[device] = ptr;
    }
    return addr[device];
}

int launch_cell_moments_noalloc(const KParams &p0, bool fp64, int device, double *out6_dev, void *stream)
{
    if (p0.N > kNoAllocMaxCells) return (int)cudaErrorInvalidValue;
    int err = 0;
    void *scratch = noalloc_scratch(device, &err);
    if (!scratch) return err;
    KParams p = p0;
    p.cellraw = scratch;
    cudaStream_t st = (cudaStream_t)stream;
    if (fp64) {
        k_cell_moments_v<double><<<nblk(p.N, 8 / p.row_warps), 256, 0, st>>>(p);
        k_moments_out<double><<<nblk(p.N, 256), 256, 0, st>>>(p, out6_dev);
    } else {
        k_cell_moments_v<float><<<nblk(p.N, 8 / p.row_warps), 256, 0, st>>>(p);
        k_moments_out<float><<<nblk(p.N, 256), 256, 0, st>>>(p, out6_dev);
    }
    return (int)cudaGetLastError();
}

// residuals of the last `last` iterations and the status word of every
// instance of a batch (inactive instances repeat their last values)
__global__ void k_batch_gather(const KParams *ps, int n, int last, double *res, int *status)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const KParams &p = ps[i];
    const int it = *p.iter;
    for (int q = 0; q < last; ++q) res[(size_t)i * 16 + q] = p.res[(it - last + q) & (kMaxHist - 1)];
    status[i] = *p.status;
}

int launch_batch_gather(const KParams *dparams, int n, int last, double *dres, int *dstatus, void *stream)
{
    if (last > 16) return (int)cudaErrorInvalidValue;
    k_batch_gather<<<nblk(n, 64), 64, 0, (cudaStream_t)stream>>>(dparams, n, last, dres, dstatus);
    return (int)cudaGetLastError();
}

int launch_to_dev(const KParams &p, bool fp64, const double *G, const double *H, int nvu, void *stream,
                  bool deviation)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (fp64) k_to_dev<double><<<1024, 256, 0, st>>>(p, G, H, nvu, deviation ? 1 : 0);
    else k_to_dev<float><<<1024, 256, 0, st>>>(p, G, H, nvu, deviation ? 1 : 0);
    return (int)cudaGetLastError();
}

int launch_from_dev(const KParams &p, bool fp64, double *G, double *H, int nvu, void *stream, bool deviation)
{
    cudaStream_t st = (cudaStream_t)stream;
    if (fp64) k_from_dev<double><<<1024, 256, 0, st>>>(p, G, H, nvu, deviation ? 1 : 0);
    else k_from_dev<float><<<1024, 256, 0, st>>>(p, G, H, nvu, deviation ? 1 : 0);
    return (int)cudaGetLastError();
}

}  // namespace idg
