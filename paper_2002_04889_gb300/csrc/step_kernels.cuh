// Step kernels of the finite-volume shallow-water solver (Giles et al., Sec. 2),
// templated on the arithmetic type.  Included by step_f32.cu and step_f64.cu;
// the FP64 file is compiled with --fmad=false so that every expression rounds
// as written.
//
// One SSP-RK(2,2) step (Sec. 2.3) is two persistent kernels plus a one-CTA
// epilogue:
//   stage 1:  R0 = L(w^n) for every cell (written to scratch) and the running
//             minimum of the CFL bound |K| / (3 max_f l_f a_f)
//   stage 2:  w1 = w^n + dt R0 (dry-fixed), recomputed where needed;
//             w^{n+1} = w^n / 2 + (w1 + dt L(w1)) / 2, dry-fixed
//   epilogue: t += dt, gauges, reset of the CFL minimum (util_kernels.cu)
//
// Each CTA owns a block of B consecutive (renumbered) cells and stages the
// block plus a two-ring halo in shared memory (ring 1: face neighbours of the
// block; ring 2: face neighbours of ring 1), with local indices precomputed on
// the host so that no phase chases an index through global memory:
//   A  load the state of block + ring-1 + ring-2 cells (smem sW: packed
//      (W, Hu, Hv, z) slots) and queue the block's owned faces (a face is owned
//      by the lower local index, a block cell facing the halo, or a wall)
//   B  reconstruct face values of block + ring-1 cells (smem sF: three packed
//      face slots per cell)
//   C  one thread per owned face computes the interface flux once and writes
//      both sides' terms into the two face slots it read
//   D  one thread per block cell gathers its three faces in local order,
//      forms the residual and updates the cell.
// A block whose cells and ring 1 are exactly dry has zero fluxes: B and C are
// skipped for it (dry land).
// No float atomics: the gather order is fixed, and the CFL minimum uses an
// integer atomicMin on the bits of a non-negative value (exact, order-free).
//
// Two arithmetic forms of the same scheme:
//  * FP64: the state is (H, Hu, Hv).  Two builds of the same code: the literal
//    one (FAST = false, step_f64.cu, no multiply-add contraction) evaluates every
//    formula as written, in the same order as any plain implementation of the
//    scheme; the fast one (FAST = true, step_f64_fast.cu, contraction allowed)
//    multiplies by one reciprocal where the literal form forms several correctly
//    rounded quotients by the same value (face velocities, the HLL star flux, the
//    residual's 1/|K|) and forms a cell's increments with one precomputed matrix.
//  * FP32 ("deviation"): block_f32.cuh.
#pragma once

#include <cuda_runtime.h>
#include <math_constants.h>

#include <type_traits>

#include "exact_div.cuh"
#include "vg_internal.h"

namespace vg {

// FP64; the FP32 arguments and phases are in block_f32.cuh.
template <typename real>
struct KArgs {
    int64_t nc;
    int block, nblocks, max_halo, max_ring1, order;
    const real *geo;        // [GEO_ROWS][nc]
    const double *rarea;    // [nc] 1 / area (FP64)
    const double *M;        // [9][nc] M_fj = w_j . (x_f - x_K), contracted build only
    const real *z;          // [nc]
    const real *zf;         // [3][nc] face beds
    const uint16_t *nbrl;   // [3][nc]
    const int32_t *halo_ptr;  // [nblocks + 1]
    const int32_t *halo_n1;   // [nblocks] ring-1 count
    const int32_t *halo_ids;  // per block: ring 1 then ring 2
    const uint16_t *ring1_nbr;// [3 * ring cells] local neighbours of ring-1 cells
    const int32_t *fq_ptr;  // [nblocks + 1] into fq
    const uint16_t *fq;     // owned faces of each block: (local cell << 2) | face
    const real *w;          // w^n [3][nc]
    real *R0;               // [3][nc]
    real *wout;             // w^{n+1} [3][nc] (stage 2)
    uint8_t *mask2;         // optional: stage-2 dry-fix branch (0 none, 1 momentum cut, 2 emptied)
    real *fv_out;           // optional [3 vars][3 faces][nc]: face values of the block cells
    real *r1_out;           // optional [3][nc]: the stage-2 residual L(w1) (stage 2)
    uint8_t *rec_out;       // optional [nc]: 1 where the block cell reconstructed (FP64)
    double *bound_out;      // optional [nc]: the stage-1 CFL bound of each cell, +inf where nothing moves (FP64)
    DevScalars *sc;
    real g, half_g, hthr;
    double cfl, dt_fixed, dt_max;
    int cfl_min;            // stage 1: 1 adds the CFL bound to the step's minimum
};

// One cell's state in a state buffer: a double of a [3][nc] array, or a float4.
template <typename real> struct StateWord { using type = real; };
template <> struct StateWord<float> { using type = float4; };

template <typename real>
__host__ __device__ inline size_t stage_smem_bytes(int block, int max_halo, int max_ring1, int max_faces, bool gids = false);

__device__ __forceinline__ float vmin(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double vmin(double a, double b) { return fmin(a, b); }

// Compare and select.  GB300 runs FP64 compares and min/max on its FP64 units,
// which issue two lane-operations per SM and cycle, while its integer units are
// idle in the FP64 kernels; so the FP64 forms below work on the IEEE bit patterns
// with integer instructions.  For the non-NaN values of the step they decide and
// select exactly as the FP64 instructions do (a zero result may carry the other
// sign, which no later operation of the step distinguishes).
//   gt_nn(x, y): x > y for y >= +0;  is_zero(x): x == 0;  is_neg(x): x < 0;
//   is_pos(x): x > 0;  smax / smin: max / min;  max0(x): max(0, x).
__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ unsigned long long ubits(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ long long okey(double x)   // order-preserving for every non-NaN x
{
    const long long b = dbits(x);
    return b < 0 ? b ^ 0x7fffffffffffffffLL : b;
}
__device__ __forceinline__ bool gt_nn(double x, double y) { return dbits(x) > dbits(y); }
__device__ __forceinline__ bool is_zero(double x) { return (ubits(x) << 1) == 0; }
__device__ __forceinline__ bool is_neg(double x) { return dbits(x) < 0 && (ubits(x) << 1) != 0; }
__device__ __forceinline__ bool is_pos(double x) { return dbits(x) > 0; }
__device__ __forceinline__ double smax(double a, double b) { return okey(a) < okey(b) ? b : a; }
__device__ __forceinline__ float smin(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ double smin(double a, double b) { return okey(b) < okey(a) ? b : a; }
__device__ __forceinline__ double max0(double x) { return dbits(x) > 0 ? x : 0.0; }
// isfinite on the integer units.
__device__ __forceinline__ bool finite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// Programmatic dependent launch: a step's kernels are launched while their
// predecessor in the stream still runs (launch_after), wait in chain_wait for it to
// complete, and by chain_next, called by every CTA of a launch, let
// their successor do the same.  Nothing that another kernel writes is read before
// chain_wait.  A step on 20k triangles is three launches of a few microseconds:
// 15.6 -> 14.3 us.  Only the one-CTA epilogue is launched early (stage 2 calls
// chain_next, the epilogue once it runs): CTAs of a stage kernel that wait while the
// last stage still runs are placed where there happens to be room and stay there
// (literal FP64, 20k triangles: 55 -> 80 us a step; FP32, 1M: 68 -> 81).
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t s, const A &...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <typename real> __device__ __forceinline__ real real_inf();
template <> __device__ __forceinline__ float real_inf<float>() { return CUDART_INF_F; }
template <> __device__ __forceinline__ double real_inf<double>() { return CUDART_INF; }

// Order-preserving integer image of a non-negative real for atomicMin.
__device__ __forceinline__ unsigned long long min_bits(float v) { return (unsigned long long)__float_as_uint(v); }
__device__ __forceinline__ unsigned long long min_bits(double v) { return (unsigned long long)__double_as_longlong(v); }
template <typename real> __device__ __forceinline__ double decode_min(unsigned long long b);
template <> __device__ __forceinline__ double decode_min<float>(unsigned long long b) { return (double)__uint_as_float((unsigned int)b); }
template <> __device__ __forceinline__ double decode_min<double>(unsigned long long b) { return __longlong_as_double((long long)b); }

// Time step of the current step from the stage-1 CFL minimum (Sec. 2.3 CFL
// condition, read as dt = cfl * min_K |K| / (3 max_f l_f a_f)), then the
// dt_max and t_end clamps.
template <typename real>
__device__ __forceinline__ double step_dt(const DevScalars *sc, double cfl, double dt_fixed,
                                          double dt_max, double t_end)
{
    double dt;
    if (dt_fixed > 0.0) {
        dt = dt_fixed;
    } else {
        double mn = decode_min<real>(sc->dtmin_bits);
        dt = isinf(mn) ? (dt_max > 0.0 ? dt_max : 0.0) : cfl * mn;
    }
    if (dt_max > 0.0) dt = fmin(dt, dt_max);
    double t = sc->t;
    if (t_end > 0.0 && t + dt > t_end) dt = t_end - t;
    if (dt < 0.0) dt = 0.0;
    return dt;
}

// t_end > 0 and t >= t_end: the context has reached its end time (decided on the
// integer units: every thread of a launch asks, and on the FP64 units the two
// compares of an SM's 40 warps take about 1300 cycles).
__device__ __forceinline__ bool finished(double t_end, const DevScalars *sc)
{
    return is_pos(t_end) && okey(sc->t) >= okey(t_end);
}

// The step's dt for every thread of a CTA, formed by one of them: a dozen FP64
// instructions in each of the 48 warps that an SM then held were 10,700 cycles of its FP64 units
// (two lane-operations a cycle), 5 us a launch.  Every thread must call it.
template <typename real>
__device__ __forceinline__ real cta_step_dt(const DevScalars *sc, double cfl, double dt_fixed, double dt_max)
{
    __shared__ real s_dt;
    if (threadIdx.x == 0) s_dt = (real)step_dt<real>(sc, cfl, dt_fixed, dt_max, sc->t_end);
    __syncthreads();
    return s_dt;
}

// HLL flux in the face normal frame (Sec. 2.2) with the dry-bed speeds when one
// side is dry; each side is (H*, u_n, u_t).
template <typename real, bool FAST = false>
__device__ __forceinline__ void hll_normal(real g, real half_g, real HL, real unL, real utL,
                                           real HR, real unR, real utR, real F[3], real &amax)
{
    if (is_zero(HL) && is_zero(HR)) {
        F[0] = real(0); F[1] = real(0); F[2] = real(0);
        amax = real(0);
        return;
    }
    real cL = sqrt(g * HL);
    real cR = sqrt(g * HR);
    real sL, sR;
    if (is_zero(HL)) {
        sL = unR - real(2) * cR;
        sR = unR + cR;
    } else if (is_zero(HR)) {
        sL = unL - cL;
        sR = unL + real(2) * cL;
    } else {
        // u* = (u_L + u_R) / 2 + (c_L - c_R), c* = (c_L + c_R) / 2 - (u_R - u_L) / 4
        // (halving commutes with rounding: each difference is rounded once as written)
        real us = half_of(unL + unR) + (cL - cR);
        real cs = half_of((cL + cR) - half_of(unR - unL));
        sL = smin(unL - cL, us - cs);
        sR = smax(us + cs, unR + cR);
    }
    real qL = HL * unL, qR = HR * unR;
    real FL0 = qL, FL1 = qL * unL + half_g * HL * HL, FL2 = qL * utL;
    real FR0 = qR, FR1 = qR * unR + half_g * HR * HR, FR2 = qR * utR;
    if (!is_neg(sL)) {
        F[0] = FL0; F[1] = FL1; F[2] = FL2;
    } else if (!is_neg(sR)) {
        real den = sR - sL;
        real sLR = sL * sR;
        const Recip rd = recip(den);
        const real N0 = (sR * FL0 - sL * FR0) + sLR * (HR - HL);
        const real N1 = (sR * FL1 - sL * FR1) + sLR * (qR - qL);
        const real N2 = (sR * FL2 - sL * FR2) + sLR * (HR * utR - HL * utL);
        if constexpr (FAST) {
            const real r = inverse(rd);
            F[0] = N0 * r; F[1] = N1 * r; F[2] = N2 * r;
        } else {
            F[0] = quot(N0, rd); F[1] = quot(N1, rd); F[2] = quot(N2, rd);
        }
    } else {
        F[0] = FR0; F[1] = FR1; F[2] = FR2;
    }
    amax = smax(fabs(sL), fabs(sR));
}

// Flux through a face seen from its left cell: face velocities, hydrostatic
// interface depths z* = max(z_L, z_R), H*_s = max(0, H_{s,f} + z_s - z*) with z_s
// the bed under side s's face value (its face bed if it reconstructed), HLL,
// rotation back to (x, y), pressure corrections g (H_{s,f}^2 - H*_s^2) / 2.
// bnd: 0 interior; 1 wall, the ghost of Sec. 2.5 (u_n reversed, u_t kept, same
// depth); 2 open, the transmissive ghost (the face state itself); 3 absorbing,
// the characteristic ghost (u_n + 2c of the face state, u_n - 2c = -2 c_0 of the
// sea at rest with c_0 = sqrt(g max(0, -z)): depth c_g^2 / g, u_t kept).
template <typename real, bool FAST = false>
__device__ __forceinline__ void face_flux(real g, real half_g, real hthr,
                                          real HfL, real HufL, real HvfL, real zL,
                                          real HfR, real HufR, real HvfR, real zR,
                                          real nx, real ny, int bnd,
                                          real Phi[3], real &PL, real &PR, real &amax)
{
    real uL = real(0), vL = real(0);
    if (gt_nn(HfL, hthr)) {
        const Recip rH = recip(HfL);
        if constexpr (FAST) {
            const real r = inverse(rH);
            uL = HufL * r; vL = HvfL * r;
        } else {
            uL = quot(HufL, rH); vL = quot(HvfL, rH);
        }
    }
    real unL = uL * nx + vL * ny;
    real utL = -uL * ny + vL * nx;
    real HsL, HsR, unR, utR;
    if (bnd == 3) {
        // absorbing: the characteristic ghost of a sea at rest (eta = 0) beyond
        // the boundary, on the same bed (the oracle's order of operations)
        HsL = max0((HfL + zL) - zL);
        const real cL = sqrt(g * HsL), c0 = sqrt(g * max0(real(0) - zL));
        const real Rp = unL + real(2) * cL, Rm = real(0) - real(2) * c0;
        unR = real(0.5) * (Rp + Rm);
        const real cg = max0(real(0.25) * (Rp - Rm));
        HsR = cg * cg / g;
        utR = utL;
        HfR = HsR;
    } else if (bnd) {
        HsL = max0((HfL + zL) - zL);
        HsR = HsL;
        unR = bnd == 2 ? unL : -unL;
        utR = utL;
        HfR = HfL;
    } else {
        real uR = real(0), vR = real(0);
        if (gt_nn(HfR, hthr)) {
            const Recip rH = recip(HfR);
            if constexpr (FAST) {
                const real r = inverse(rH);
                uR = HufR * r; vR = HvfR * r;
            } else {
                uR = quot(HufR, rH); vR = quot(HvfR, rH);
            }
        }
        unR = uR * nx + vR * ny;
        utR = -uR * ny + vR * nx;
        real zs = smax(zL, zR);
        HsL = max0((HfL + zL) - zs);
        HsR = max0((HfR + zR) - zs);
    }
    real F[3];
    hll_normal<real, FAST>(g, half_g, HsL, unL, utL, HsR, unR, utR, F, amax);
    Phi[0] = F[0];
    Phi[1] = F[1] * nx - F[2] * ny;
    Phi[2] = F[1] * ny + F[2] * nx;
    PL = half_g * (HfL * HfL - HsL * HsL);
    PR = half_g * (HfR * HfR - HsR * HsR);
}

// Stored state of cell gid as seen by the stage (H, Hu, Hv):
// stage 1 reads w^n; stage 2 forms w1 = w^n + dt R0 and applies the dry fix
// (negative depth emptied; at or below the threshold, momentum zeroed).
// Returns true if a negative depth was met.
template <typename real, int STAGE>
__device__ __forceinline__ bool stage_state(const KArgs<real> &a, int gid, real dt, real &W, real &Hu, real &Hv)
{
    const int nc = (int)a.nc;
    W = a.w[gid];
    Hu = a.w[nc + gid];
    Hv = a.w[2 * nc + gid];
    if (STAGE == 1) return false;
    W = W + dt * a.R0[gid];
    Hu = Hu + dt * a.R0[nc + gid];
    Hv = Hv + dt * a.R0[2 * nc + gid];
    if (is_neg(W)) {
        W = real(0); Hu = real(0); Hv = real(0);
        return true;
    }
    if (!gt_nn(W, a.hthr)) { Hu = real(0); Hv = real(0); }
    return false;
}

// An exactly dry cell: no water and no momentum.
template <typename real>
__device__ __forceinline__ bool exactly_dry(real H, real Hu, real Hv)
{
    return is_zero(H) && is_zero(Hu) && is_zero(Hv);
}

// Stored state of cell gid as seen by the stage, and its bed.
template <typename real, int STAGE>
__device__ __forceinline__ bool stage_cell(const KArgs<real> &a, int gid, real dt, real &W, real &Hu, real &Hv,
                                           real &zc)
{
    zc = a.z[gid];
    return stage_state<real, STAGE>(a, gid, dt, W, Hu, Hv);
}

// Four reals in shared memory, moved as two 16-byte accesses.
__device__ __forceinline__ void ld4(const double *p, double &x, double &y, double &z, double &w)
{
    double2 a = reinterpret_cast<const double2 *>(p)[0], b = reinterpret_cast<const double2 *>(p)[1];
    x = a.x; y = a.y; z = b.x; w = b.y;
}
__device__ __forceinline__ void st4(double *p, double x, double y, double z, double w)
{
    reinterpret_cast<double2 *>(p)[0] = make_double2(x, y);
    reinterpret_cast<double2 *>(p)[1] = make_double2(z, w);
}

// SSP-RK(2,2) second stage (Sec. 2.3) of one cell: w^{n+1} = w^n / 2 + (w1 + dt R(w1)) / 2
// from w^n = x, w1 = (W1, Hu1, Hv1) and R(w1) = (RH, RHu, RHv), then the dry fix.
// Returns the fix's branch: 0 none, 1 momentum cut (depth at or below the
// threshold), 2 negative depth emptied.
// (FAST, the contracted build: half of the sum, which is the same number but at the
// ends of the range.)
template <typename real, bool FAST = false>
__device__ __forceinline__ uint8_t rk2_final(const real x[3], real W1, real Hu1, real Hv1, real RH, real RHu,
                                             real RHv, real dt, real hthr, real &W, real &Hu, real &Hv)
{
    const real yW = W1 + dt * RH, yHu = Hu1 + dt * RHu, yHv = Hv1 + dt * RHv;
    W = FAST ? half_of(x[0] + yW) : half_sum(x[0], yW);
    Hu = FAST ? half_of(x[1] + yHu) : half_sum(x[1], yHu);
    Hv = FAST ? half_of(x[2] + yHv) : half_sum(x[2], yHv);
    if (is_neg(W)) {
        W = real(0); Hu = real(0); Hv = real(0);
        return 2;
    }
    if (!gt_nn(W, hthr)) {
        Hu = real(0); Hv = real(0);
        return 1;
    }
    return 0;
}

// Phase D's end for block cell l (global gid), from the sums of its three face
// terms: R = -(aH, aHu, aHv) / |K|; stage 1 writes R0 and the CFL bound of
// am = max_f l_f a_f; stage 2 forms w^{n+1} = w^n / 2 + (w1 + dt R) / 2 with
// w^n = x, w1 from shared memory, and the dry fix.
template <typename real, int STAGE, bool FAST = false>
__device__ __forceinline__ void finish_cell(const KArgs<real> &a, int gid, const real *sWl, real aH, real aHu,
                                            real aHv, real am, const real x[3], real area, real rarea, real dt,
                                            real &my_min, long long &my_neg, bool &bad)
{
    const int nc = (int)a.nc;
    real RH, RHu, RHv;
    if constexpr (FAST) {
        RH = -aH * rarea; RHu = -aHu * rarea; RHv = -aHv * rarea;
    } else {
        const Recip ra = recip_given(area, rarea);
        RH = quot(-aH, ra); RHu = quot(-aHu, ra); RHv = quot(-aHv, ra);
    }
    if (STAGE == 1) {
        a.R0[gid] = RH;
        a.R0[nc + gid] = RHu;
        a.R0[2 * nc + gid] = RHv;
        real bnd = real_inf<real>();
        if (is_pos(am)) bnd = quot(area, recip(real(3) * am));
        my_min = smin(my_min, bnd);
        if (a.bound_out) a.bound_out[gid] = bnd;
    } else {
        if (a.r1_out) {
            a.r1_out[gid] = RH;
            a.r1_out[nc + gid] = RHu;
            a.r1_out[2 * nc + gid] = RHv;
        }
        real W1, Hu1, Hv1, z1;
        ld4(sWl, W1, Hu1, Hv1, z1);
        real W, Hu, Hv;
        const uint8_t branch = rk2_final<real, FAST>(x, W1, Hu1, Hv1, RH, RHu, RHv, dt, a.hthr, W, Hu, Hv);
        if (branch == 2) my_neg++;
        if (a.mask2) a.mask2[gid] = branch;
        if (!finite(W) || !finite(Hu) || !finite(Hv)) bad = true;
        a.wout[gid] = W;
        a.wout[nc + gid] = Hu;
        a.wout[2 * nc + gid] = Hv;
    }
}

// Shared memory of one CTA: cell states [L] x 4, face slots [3][L1] x 4 (L1 =
// block + ring 1), with gids the global ids of block and ring-1 cells [L1], face
// codes and owned-face queue [3B] each, one byte per block and ring-1 cell: whether it
// reconstructed (phase D adds its bed-slope source), and the cells' free surfaces [L]
// (formed once; four neighbours and the source read each).  Without gids phase
// B reads a ring-1 cell's global id again from the halo list.
template <>
__host__ __device__ inline size_t stage_smem_bytes<double>(int block, int max_halo, int max_ring1, int, bool gids)
{
    size_t L = (size_t)block + max_halo, L1 = (size_t)block + max_ring1;
    return sizeof(double) * (5 * L + 12 * L1) + (gids ? sizeof(int32_t) * L1 : 0) + sizeof(uint16_t) * 6 * (size_t)block + L1 + 16;
}

// One block of cells for one scenario: phases A-D (see the top of this file).
// my_min collects the thread's stage-1 CFL bound, my_neg its negative-depth
// events, bad a non-finite result.  Every thread of the CTA must call it;
// qcount is the CTA's shared count of queued faces.
//
// The queue of owned faces is copied from the list built with the partition
// (LISTED) or formed in phase A from the face codes by a warp-aggregated
// append; the list is faster in the stage-2 kernels and the batched kernels,
// the append in the single-scenario stage-1 kernels.
// Either way every face of the block is queued once, and the result does not
// depend on the queue order (each face writes its own two slots).
//
// There is no barrier after phase D: a thread's phase D reads only its own
// cell's state slot and face slots, the next block's phase A writes state
// slots of its own cells, codes, the face queue and its count only, and face
// slots are next written in phase B, behind the barrier that ends phase A.
// Consecutive blocks use the two queue counters alternately (an append's
// counter is reset in phase D, which may come after other warps have started
// the next block).
//
// Shared layout: sW[l] = (H, Hu, Hv, z) of local cell l; sF[f][l] = face values (W_f, Hu_f, Hv_f, z_f) of face f of cell l
// after phase B, z_f the bed the face value stands on, and after phase C the
// cell's own term (l_f Phi_0, l_f (Phi_1 + P n_x), l_f (Phi_2 + P n_y), l_f a_f).
// Stage 2's phase D reads w^n of its cell from global memory.
template <typename real, int STAGE, int DRY, bool LISTED, bool GIDS, bool FAST = false>
__device__ __forceinline__ void process_block(const KArgs<real> &a, const int b, const real dt,
                                              unsigned char *smem_raw, int &qcount, real &my_min,
                                              long long &my_neg, bool &bad)
{
    const int B = a.block;
    const int L = B + a.max_halo;
    const int L1 = B + a.max_ring1;
    const int nc = (int)a.nc;    // per-cell arrays hold < 2^31 entries (checked at upload)
    real *sW = reinterpret_cast<real *>(smem_raw);          // [L][4]
    real *sF = sW + 4 * L;                                   // [3][L1][4]
    real *sE = sF + 12 * L1;                                 // [L] H + z
    int32_t *sGid = reinterpret_cast<int32_t *>(sE + L);     // [L1] (GIDS)
    uint16_t *sCode = reinterpret_cast<uint16_t *>(GIDS ? sGid + L1 : sGid);   // [3][B]
    uint16_t *queue = sCode + 3 * B;                              // [3B]
    uint8_t *sRec = reinterpret_cast<uint8_t *>(queue + 3 * B);   // [L1]

    const int tid = threadIdx.x;
    const real g = a.g, half_g = a.half_g, hthr = a.hthr;
    const real *geo = a.geo;

    const int c0 = b * B;
    const int ncell = min(B, nc - c0);
    const int h0 = a.halo_ptr[b];
    const int nh = a.halo_ptr[b + 1] - h0;
    const int n1 = a.halo_n1[b];

    // A: block + ring-1 + ring-2 states into shared memory, and the block's
    // owned faces (a boundary face, a face to the halo, or a face to a block
    // cell of higher local index: every face once) into the queue.  Thread
    // tid < B takes block cell tid.  The threads also note whether the block
    // and its ring 1 are exactly dry (dry land): then every face of the block
    // has zero interface depths on both sides, hence zero flux and zero
    // pressure terms, and phases B and C reduce to zero face terms.
    bool dry = true;
    {
        int gh = -1;
        if (tid < nh) gh = a.halo_ids[h0 + tid];
        if constexpr (LISTED) {
            const int q0 = a.fq_ptr[b], nq = a.fq_ptr[b + 1] - q0;
            for (int q = tid; q < nq; q += blockDim.x) queue[q] = a.fq[q0 + q];
            if (tid == 0) qcount = nq;
        }
        int owned = 0;
        if (tid < ncell) {
            const int gid = c0 + tid;
#pragma unroll
            for (int f = 0; f < 3; f++) {
                const uint16_t code = a.nbrl[f * nc + gid];
                sCode[f * B + tid] = code;
                if (!LISTED && (code >= NBR_ABSORB || (code >> 2) >= B || (int)(code >> 2) > tid)) owned |= 1 << f;
            }
            real W, Hu, Hv, zc;
            bool neg = stage_cell<real, STAGE>(a, gid, dt, W, Hu, Hv, zc);
            if (neg) my_neg++;
            st4(sW + 4 * tid, W, Hu, Hv, zc);
            sE[tid] = W + zc;
            if constexpr (GIDS) sGid[tid] = gid;
            dry = exactly_dry(W, Hu, Hv);
        }
        if (gh >= 0) {
            real W, Hu, Hv, zc;
            stage_cell<real, STAGE>(a, gh, dt, W, Hu, Hv, zc);
            st4(sW + 4 * (B + tid), W, Hu, Hv, zc);
            sE[B + tid] = W + zc;
            if (tid < n1) {
                if constexpr (GIDS) sGid[B + tid] = gh;
                dry = dry && exactly_dry(W, Hu, Hv);
            }
        }
        for (int h = tid + blockDim.x; h < nh; h += blockDim.x) {
            const int gid = a.halo_ids[h0 + h];
            real W, Hu, Hv, zc;
            stage_cell<real, STAGE>(a, gid, dt, W, Hu, Hv, zc);
            st4(sW + 4 * (B + h), W, Hu, Hv, zc);
            sE[B + h] = W + zc;
            if (h < n1) {
                if constexpr (GIDS) sGid[B + h] = gid;
                dry = dry && exactly_dry(W, Hu, Hv);
            }
        }
        if constexpr (!LISTED) {
            // warp-aggregated queue append: n = popcount(owned) in 0..3
            const int n = __popc(owned);
            const unsigned lane = tid & 31;
            const unsigned lt = (1u << lane) - 1u;
            const unsigned b1 = __ballot_sync(0xffffffffu, n & 1), b2 = __ballot_sync(0xffffffffu, n & 2);
            const int total = __popc(b1) + 2 * __popc(b2);
            int base = 0;
            if (lane == 0 && total) base = atomicAdd(&qcount, total);
            base = __shfl_sync(0xffffffffu, base, 0);
            int pos = base + __popc(b1 & lt) + 2 * __popc(b2 & lt);
#pragma unroll
            for (int f = 0; f < 3; f++)
                if ((owned >> f) & 1) queue[pos++] = (uint16_t)((tid << 2) | f);
        }
    }
    // Dry land.  Mode 1 leaves the block here with a zero residual (phase D with
    // zero face terms; w^n from memory) and writes the adjoint's recordings as
    // the full phases would (a dry cell's face values are its own values); mode 2
    // has phase B write zero face terms for the block cells (and w^n for stage
    // 2) and phase C no faces, which costs a few instructions more but no
    // register spills where mode 1 would spill (runs with recordings take every
    // phase there).
    const bool skip = __syncthreads_and(dry) && (DRY == 1 || (!a.fv_out && !a.mask2 && !a.r1_out && !a.rec_out));
    if (DRY == 1 && skip) {
        if (!LISTED && tid == 0) qcount = 0;
        if (tid < ncell) {
            const int gid = c0 + tid;
            if (a.rec_out) a.rec_out[gid] = 0;
            if (a.fv_out) {
                real Wc, Huc, Hvc, zc;
                ld4(sW + 4 * tid, Wc, Huc, Hvc, zc);
#pragma unroll
                for (int f = 0; f < 3; f++) {
                    a.fv_out[(0 * 3 + f) * (size_t)nc + gid] = Wc;
                    a.fv_out[(1 * 3 + f) * (size_t)nc + gid] = Huc;
                    a.fv_out[(2 * 3 + f) * (size_t)nc + gid] = Hvc;
                }
            }
            real x[3] = {real(0), real(0), real(0)};
            if (STAGE == 2) { x[0] = a.w[gid]; x[1] = a.w[nc + gid]; x[2] = a.w[2 * nc + gid]; }
            // R = -0 / |K| = -0 for any area, so the area is not read
            finish_cell<real, STAGE, FAST>(a, gid, sW + 4 * tid, real(0), real(0), real(0), real(0), x, real(1), real(1),
                                           dt, my_min, my_neg, bad);
        }
        return;
    }
    const bool zero_terms = DRY == 2 && skip;

    // B: face values of block + ring-1 cells (Sec. 2.4, Eq. recon with the
    // Barth-Jespersen limiter); every neighbour is in shared memory
    for (int l = tid; l < (zero_terms ? ncell : B + n1); l += blockDim.x) {
        if (l < B && l >= ncell) continue;
        const int gid = GIDS ? sGid[l] : l < B ? c0 + l : a.halo_ids[h0 + (l - B)];
        if (zero_terms) {
#pragma unroll
            for (int f = 0; f < 3; f++) st4(sF + 4 * (f * L1 + l), real(0), real(0), real(0), real(0));
            sRec[l] = 0;
            continue;
        }
        real WK, HuK, HvK, zK;
        ld4(sW + 4 * l, WK, HuK, HvK, zK);
        const real HK = WK;
        real qK[3] = {sE[l], HuK, HvK};
        real qn[3][3];
        bool recon = (a.order == 2) && gt_nn(HK, hthr);
#pragma unroll
        for (int f = 0; f < 3; f++) {
            uint16_t code;
            int nl;
            if (l < B) {
                code = sCode[f * B + l];
                nl = code >> 2;
            } else {
                code = a.ring1_nbr[3 * (h0 + (l - B)) + f];
                nl = code;
            }
            if (code < NBR_ABSORB) {
                real Hj, Huj, Hvj, zj;
                ld4(sW + 4 * nl, Hj, Huj, Hvj, zj);
                qn[f][0] = sE[nl];
                qn[f][1] = Huj;
                qn[f][2] = Hvj;
                if (!gt_nn(Hj, hthr)) recon = false;
            } else if (code != NBR_WALL) {
                // open or absorbing face: the cell's own values (zero gradient)
                qn[f][0] = qK[0];
                qn[f][1] = HuK;
                qn[f][2] = HvK;
            } else {
                const real nxf = geo[(GEO_NX + f) * nc + gid], nyf = geo[(GEO_NY + f) * nc + gid];
                real mn = HuK * nxf + HvK * nyf;
                qn[f][0] = qK[0];
                qn[f][1] = HuK - real(2) * mn * nxf;
                qn[f][2] = HvK - real(2) * mn * nyf;
            }
        }
        real Hf[3], Huf[3], Hvf[3];
        real zfK[3] = {zK, zK, zK};       // the bed under each face value
        if (recon) {
            real face[3][3];
            real fx[3], fy[3], wx[3], wy[3];       // literal: gradient, then its dot products
            real Mf[3][3];                         // contracted: the increments' matrix, 9 instead of 12
#pragma unroll
            for (int f = 0; f < 3; f++) {
                if constexpr (FAST) {
#pragma unroll
                    for (int j = 0; j < 3; j++) Mf[f][j] = a.M[(3 * f + j) * (size_t)nc + gid];
                } else {
                    fx[f] = geo[(GEO_FX + f) * nc + gid];
                    fy[f] = geo[(GEO_FY + f) * nc + gid];
                    wx[f] = geo[(GEO_WX + f) * nc + gid];
                    wy[f] = geo[(GEO_WY + f) * nc + gid];
                }
            }
#pragma unroll
            for (int v = 0; v < 3; v++) {
                real d0 = qn[0][v] - qK[v], d1 = qn[1][v] - qK[v], d2 = qn[2][v] - qK[v];
                real D[3];
                if constexpr (FAST) {
#pragma unroll
                    for (int f = 0; f < 3; f++) D[f] = Mf[f][0] * d0 + Mf[f][1] * d1 + Mf[f][2] * d2;
                } else {
                    real gx = (wx[0] * d0 + wx[1] * d1) + wx[2] * d2;
                    real gy = (wy[0] * d0 + wy[1] * d1) + wy[2] * d2;
#pragma unroll
                    for (int f = 0; f < 3; f++) D[f] = gx * fx[f] + gy * fy[f];
                }
                real alpha = real(1);
                {
                    // alpha = min(1, min_f r_f / D_f), r_f = q_max - q_K or q_min - q_K by
                    // the sign of D_f.  Rounding is monotone, so q_max - q_K is the
                    // largest of the rounded differences d_j and 0, and the smallest
                    // quotient of a sign is that of its largest |D_f|: two candidates
                    // up / P and dn / M, compared by cross products (rounded products
                    // that differ order the quotients), and one division, none where
                    // neither limits.  Nine divisions per cell become at most three.
                    real up = max0(d0), dn = max0(-d0), P = max0(D[0]), M = max0(-D[0]);
                    if (gt_nn(d1, up)) up = d1;
                    if (gt_nn(d2, up)) up = d2;
                    if (gt_nn(-d1, dn)) dn = -d1;
                    if (gt_nn(-d2, dn)) dn = -d2;
                    if (gt_nn(D[1], P)) P = D[1];
                    if (gt_nn(D[2], P)) P = D[2];
                    if (gt_nn(-D[1], M)) M = -D[1];
                    if (gt_nn(-D[2], M)) M = -D[2];
                    const bool limP = gt_nn(P, up), limM = gt_nn(M, dn);
                    if (limP || limM) {
                        const real xP = up * M, xM = dn * P;
                        const bool takeM = limM && (!limP || gt_nn(xP, xM));
                        const real num = takeM ? dn : up, den = takeM ? M : P;
                        alpha = quot(num, recip(den));
                        if (limP && limM && dbits(xP) == dbits(xM)) alpha = smin(alpha, quot(dn, recip(M)));
                    }
                }
#pragma unroll
                for (int f = 0; f < 3; f++) face[f][v] = qK[v] + alpha * D[f];
            }
            // the face values stand on the face beds z_f (the linear bed at the
            // face midpoints); the face depths must stay above the threshold
#pragma unroll
            for (int f = 0; f < 3; f++) zfK[f] = a.zf[f * nc + gid];
#pragma unroll
            for (int f = 0; f < 3; f++) {
                Hf[f] = face[f][0] - zfK[f];
                if (!gt_nn(Hf[f], hthr)) recon = false;
                Huf[f] = face[f][1];
                Hvf[f] = face[f][2];
            }
        }
        if (!recon) {
#pragma unroll
            for (int f = 0; f < 3; f++) { Hf[f] = HK; Huf[f] = HuK; Hvf[f] = HvK; zfK[f] = zK; }
        }
        sRec[l] = recon ? 1 : 0;
        if (a.rec_out && l < B) a.rec_out[gid] = recon ? 1 : 0;
#pragma unroll
        for (int f = 0; f < 3; f++) st4(sF + 4 * (f * L1 + l), Hf[f], Huf[f], Hvf[f], zfK[f]);
        if (a.fv_out && l < B) {
#pragma unroll
            for (int f = 0; f < 3; f++) {
                a.fv_out[(0 * 3 + f) * (size_t)nc + gid] = Hf[f];
                a.fv_out[(1 * 3 + f) * (size_t)nc + gid] = Huf[f];
                a.fv_out[(2 * 3 + f) * (size_t)nc + gid] = Hvf[f];
            }
        }
    }
    __syncthreads();

    // C: owned faces, one flux each (Sec. 2.2).  The two face values a face
    // reads are used by no other face, so its thread overwrites them with the
    // two sides' terms l [Phi + P_s n_s] (the other side's flux and normal are
    // the exact negations, the face length the same).
    const int nq = zero_terms ? 0 : qcount;
    for (int q = tid; q < nq; q += blockDim.x) {
        const int item = queue[q];
        const int l = item >> 2, f = item & 3;
        const int gid = c0 + l;
        const uint16_t code = sCode[f * B + l];
        const bool wall = code >= NBR_ABSORB;         // wall, open or absorbing: no neighbour
        const int bnd = wall ? (code == NBR_WALL ? 1 : code == NBR_OPEN ? 2 : 3) : 0;
        const int nl = code >> 2, nf = code & 3;
        real *pL = sF + 4 * (f * L1 + l);
        real *pR = sF + 4 * (nf * L1 + nl);
        // zL, zR: the bed under each side's face value (its face bed where that
        // cell reconstructed, its cell bed otherwise), from the slots' 4th word
        real HfL, HufL, HvfL, zL;
        ld4(pL, HfL, HufL, HvfL, zL);
        real HfR = real(0), HufR = real(0), HvfR = real(0), zR = real(0);
        if (!wall) ld4(pR, HfR, HufR, HvfR, zR);
        real Phi[3], PL, PR, am;
        const real nx = geo[(GEO_NX + f) * nc + gid], ny = geo[(GEO_NY + f) * nc + gid];
        const real len = geo[(GEO_LEN + f) * nc + gid];
        face_flux<real, FAST>(g, half_g, hthr, HfL, HufL, HvfL, zL, HfR, HufR, HvfR, zR, nx, ny, bnd, Phi, PL, PR, am);
        const real t0 = len * Phi[0];
        const real la = len * am;
        st4(pL, t0, len * (Phi[1] + PL * nx), len * (Phi[2] + PL * ny), la);
        if (!wall) st4(pR, -t0, -(len * (Phi[1] + PR * nx)), -(len * (Phi[2] + PR * ny)), la);
    }
    __syncthreads();

    // D: residual R_K = -(1/|K|) sum_f l_f [Phi_f + (0, P_{K,f} n_f)], faces in local order
    if (!LISTED && tid == 0) qcount = 0;     // every thread read it before the barrier above
    if (tid < ncell) {
        const int l = tid;
        const int gid = c0 + l;
        real aH = real(0), aHu = real(0), aHv = real(0), am = real(0);
        real x[3];
        const real area = geo[GEO_AREA * nc + gid], rarea = a.rarea[gid];
#pragma unroll
        for (int f = 0; f < 3; f++) {
            real t0, t1, t2;
            ld4(sF + 4 * (f * L1 + l), t0, t1, t2, x[f]);
            aH = aH + t0;
            aHu = aHu + t1;
            aHv = aHv + t2;
            if (STAGE == 1) am = smax(am, x[f]);
        }
        {
            // centred bed-slope source of a cell standing on its face beds:
            // g sum_f l_f z_f (eta_K - z_f / 2) n_f, eta_K = H_K + z_K
            if (sRec[l]) {
                const real eK = sE[l];
#pragma unroll
                for (int f = 0; f < 3; f++) {
                    const real zff = a.zf[f * nc + gid];
                    const real sf = g * (geo[(GEO_LEN + f) * nc + gid] * (zff * (eK - half_of(zff))));
                    aHu = aHu + sf * geo[(GEO_NX + f) * nc + gid];
                    aHv = aHv + sf * geo[(GEO_NY + f) * nc + gid];
                }
            }
        }
        if (STAGE == 2) { x[0] = a.w[gid]; x[1] = a.w[nc + gid]; x[2] = a.w[2 * nc + gid]; }
        finish_cell<real, STAGE, FAST>(a, gid, sW + 4 * l, aH, aHu, aHv, am, x, area, rarea, dt, my_min, my_neg, bad);
    }
}

}  // namespace vg

#include "block_f32.cuh"

namespace vg {

// Resident CTAs per SM asked of the register allocator.  FP32 with one thread per
// cell: five of 256 threads at 48 registers (1M basin, us a step: 68 against 79 with
// six at 40 registers, which spill and leave less of the SM's memory to L1, and 73
// with four); two threads per cell are for meshes of one wave, which have registers
// to spare.  FP64 beyond 256 threads is left unbounded.
template <typename real, int MAXT> struct StageMinCtas { static constexpr int value = 1; };
template <> struct StageMinCtas<float, 256> { static constexpr int value = 5; };
template <> struct StageMinCtas<float, 384> { static constexpr int value = 3; };
template <> struct StageMinCtas<float, 512> { static constexpr int value = 2; };
// FP64 with one thread per cell: two CTAs per SM, so that one CTA's phases run
// while the other waits at a barrier (118-122 registers, no spills)
template <> struct StageMinCtas<double, 256> { static constexpr int value = 2; };
// The batched kernels' own budget (their extra scenario state needs the FP64
// registers of one CTA per SM).
template <typename real> struct BatchMinCtas { static constexpr int value = 1; };
template <> struct BatchMinCtas<float> { static constexpr int value = 4; };

// FP32 instances: the context's states, the caller's [3][nc] arrays (the no-allocation
// step), or the context's on a moving bed (block_f32.cuh has that form's arithmetic).
enum { OWN, CALLERS, ON_MOVING_BED };

// One block of a single-scenario stage (BATCH = false) or of a batch's scenario.
// FP64: the single-scenario kernels leave a dry block early, the batched ones let
// phase B write zero terms and keep the ids (see process_block).
template <int STAGE, bool FAST, bool BATCH, int STATE>
__device__ __forceinline__ void run_block(const KArgs<double> &a, int b, double dt, unsigned char *smem, int &qcount,
                                          double &my_min, long long &my_neg, bool &bad, bool &)
{
    process_block<double, STAGE, BATCH ? 2 : 1, BATCH || STAGE == 2, BATCH, FAST>(a, b, dt, smem, qcount, my_min, my_neg,
                                                                                  bad);
}
template <int STAGE, bool FAST, bool BATCH, int STATE>
__device__ __forceinline__ void run_block(const KArgs<float> &a, int b, float dt, unsigned char *smem, int &,
                                          float &my_min, long long &my_neg, bool &bad, bool &loaded)
{
    process_block<STAGE, STATE == CALLERS, BATCH ? KEEP_SCENARIOS : KEEP_NOTHING, STATE == ON_MOVING_BED>(a, b, dt, smem, my_min,
                                                                                                        my_neg, bad, loaded);
}

// w^{n+1} = w^n, bit for bit, by every thread of the launch.
template <bool SOA>
__device__ __forceinline__ void copy_state(const KArgs<double> &a, int64_t i0, int64_t stride)
{
    for (int64_t i = i0; i < 3 * a.nc; i += stride) a.wout[i] = a.w[i];
}
template <bool SOA>
__device__ __forceinline__ void copy_state(const KArgs<float> &a, int64_t i0, int64_t stride)
{
    if constexpr (SOA)
        for (int64_t i = i0; i < 3 * a.nc; i += stride) a.wout_soa[i] = a.w_soa[i];
    else
        for (int64_t i = i0; i < a.nc; i += stride) a.wout[i] = a.w[i];
}

template <typename real, int STAGE, int MAXT, bool FAST = false, int STATE = OWN>
__global__ void __launch_bounds__(MAXT, StageMinCtas<real, MAXT>::value) stage_kernel(const KArgs<real> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int qcount[2];
    __shared__ real red_min[32];
    __shared__ long long red_neg[32];
    const int tid = threadIdx.x;
    if (STAGE == 2) chain_next();
    chain_wait();

    // a context that has reached t_end takes steps of dt = 0 that leave its state
    // as it is: stage 1 does nothing (the CFL minimum stays empty) and stage 2
    // copies w^n to the output buffer, bit for bit (computing w/2 + (w + 0 R)/2
    // would flush the smallest FP32 values to zero), as the batched kernels do
    if (finished(a.sc->t_end, a.sc)) {
        if (STAGE == 2)
            copy_state<STATE == CALLERS>(a, blockIdx.x * (int64_t)blockDim.x + tid, (int64_t)gridDim.x * blockDim.x);
        return;
    }

    real dt = real(0);
    if (STAGE == 2) dt = cta_step_dt<real>(a.sc, a.cfl, a.dt_fixed, a.dt_max);

    real my_min = real_inf<real>();
    long long my_neg = 0;
    bool bad = false;
    if (tid < 2) qcount[tid] = 0;
    __syncthreads();

    int parity = 0;
    for (int b = blockIdx.x; b < a.nblocks; b += gridDim.x, parity ^= 1) {
        bool loaded = false;
        run_block<STAGE, FAST, false, STATE>(a, b, dt, smem_raw, qcount[parity], my_min, my_neg, bad, loaded);
    }

    // CTA-level reductions, then one atomic per CTA
    const int lane = tid & 31, warp = tid >> 5, nwarps = (blockDim.x + 31) >> 5;
    if (STAGE == 1) {
        for (int o = 16; o > 0; o >>= 1) my_min = smin(my_min, __shfl_xor_sync(0xffffffffu, my_min, o));
        if (lane == 0) red_min[warp] = my_min;
    }
    for (int o = 16; o > 0; o >>= 1) my_neg += __shfl_xor_sync(0xffffffffu, my_neg, o);
    if (lane == 0) red_neg[warp] = my_neg;
    bad = __syncthreads_or(bad);
    if (tid == 0) {
        long long neg = 0;
        real mn = real_inf<real>();
        for (int w = 0; w < nwarps; w++) {
            neg += red_neg[w];
            if (STAGE == 1) mn = smin(mn, red_min[w]);
        }
        if (STAGE == 1 && a.cfl_min && mn < real_inf<real>()) atomicMin(&a.sc->dtmin_bits, min_bits(mn));
        if (neg) atomicAdd((unsigned long long *)&a.sc->neg_count, (unsigned long long)neg);
        if (bad) atomicOr(&a.sc->flags, FLAG_NONFINITE_STATE);
    }
}

// ---------------------------------------------------------------------------
// Unfused SSP-RK(2,2) (Sec. 2.3; vg_params.rk_unfused): the two stage updates as
// kernels of their own, with w1 and R(w1) in global memory, to compare with the
// fused stage-2 kernel, which forms w1 = w^n + dt R0 as it loads a block and ends
// with the second update.  Update 1 writes w1 with the dry fix; the stage-1
// kernel, without its CFL bound, writes R(w1); update 2 writes w^{n+1}.  The
// arithmetic of each cell is the fused path's (stage_cell, rk2_final).
// 256 threads, grid-stride over the cells; one atomic per CTA for the counts.
template <typename real>
__device__ __forceinline__ void cta_counts(long long my_neg, bool bad, DevScalars *sc)
{
    __shared__ long long red[8];
    __shared__ int any_bad;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) any_bad = 0;
    for (int o = 16; o > 0; o >>= 1) my_neg += __shfl_xor_sync(0xffffffffu, my_neg, o);
    if (lane == 0) red[warp] = my_neg;
    __syncthreads();
    if (bad) any_bad = 1;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long n = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) n += red[w];
        if (n) atomicAdd((unsigned long long *)&sc->neg_count, (unsigned long long)n);
        if (any_bad) atomicOr(&sc->flags, FLAG_NONFINITE_STATE);
    }
}

__device__ __forceinline__ bool cell_update1(const KArgs<double> &a, int gid, double dt, double *w1)
{
    const int64_t nc = a.nc;
    double W, Hu, Hv, zc;
    const bool neg = stage_cell<double, 2>(a, gid, dt, W, Hu, Hv, zc);
    w1[gid] = W;
    w1[nc + gid] = Hu;
    w1[2 * nc + gid] = Hv;
    return neg;
}
__device__ __forceinline__ bool cell_update1(const KArgs<float> &a, int gid, float dt, float4 *w1)
{
    float4 q;
    const bool neg = stage_cell<2, false>(a, gid, dt, q);
    w1[gid] = q;
    return neg;
}
__device__ __forceinline__ bool cell_update2(const KArgs<double> &a, int gid, double dt, const double *w1,
                                             const double *R1, bool &bad)
{
    const int64_t nc = a.nc;
    const double x[3] = {a.w[gid], a.w[nc + gid], a.w[2 * nc + gid]};
    double W, Hu, Hv;
    const uint8_t branch = rk2_final(x, w1[gid], w1[nc + gid], w1[2 * nc + gid], R1[gid], R1[nc + gid], R1[2 * nc + gid],
                                     dt, a.hthr, W, Hu, Hv);
    if (!finite(W) || !finite(Hu) || !finite(Hv)) bad = true;
    a.wout[gid] = W;
    a.wout[nc + gid] = Hu;
    a.wout[2 * nc + gid] = Hv;
    return branch == 2;
}
__device__ __forceinline__ bool cell_update2(const KArgs<float> &a, int gid, float dt, const float4 *w1, const float4 *R1,
                                             bool &bad)
{
    const float4 r = R1[gid];
    float4 o;
    const bool neg = rk_second(a.w[gid], w1[gid], r.x, r.y, r.z, dt, a.hthr, o);
    if (!isfinite(o.x) || !isfinite(o.y) || !isfinite(o.z)) bad = true;
    a.wout[gid] = o;
    return neg;
}

template <typename real>
__global__ void __launch_bounds__(256) rk_update1_kernel(const KArgs<real> a, typename StateWord<real>::type *w1)
{
    if (finished(a.sc->t_end, a.sc)) return;                 // update 2 copies w^n
    const real dt = cta_step_dt<real>(a.sc, a.cfl, a.dt_fixed, a.dt_max);
    long long my_neg = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.nc; i += (int64_t)gridDim.x * blockDim.x)
        if (cell_update1(a, (int)i, dt, w1)) my_neg++;
    cta_counts<real>(my_neg, false, a.sc);
}

template <typename real>
__global__ void __launch_bounds__(256) rk_update2_kernel(const KArgs<real> a, const typename StateWord<real>::type *w1,
                                                         const typename StateWord<real>::type *R1)
{
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    if (finished(a.sc->t_end, a.sc)) {                       // as the fused kernel: w^n, bit for bit
        copy_state<false>(a, i0, stride);
        return;
    }
    const real dt = cta_step_dt<real>(a.sc, a.cfl, a.dt_fixed, a.dt_max);
    long long my_neg = 0;
    bool bad = false;
    for (int64_t i = i0; i < a.nc; i += stride)
        if (cell_update2(a, (int)i, dt, w1, R1, bad)) my_neg++;
    cta_counts<real>(my_neg, bad, a.sc);
}

// ---------------------------------------------------------------------------
// Batched ensembles: many scenarios on several meshes in one persistent launch
// per stage.  A work item is one block of one mesh and one of `groups` groups of its
// scenarios; the CTA runs that block for every scenario of the group in turn, so the
// block's mesh data stays in L1/L2 across scenarios.  Scenario e (meshes' scenarios numbered consecutively) has
// its own state slice, its own device scalars sc[e] and its own time step.
// ---------------------------------------------------------------------------

constexpr int kBatchMaxEntries = 512;

template <typename real>
struct BatchMesh {
    KArgs<real> a;         // mesh arrays; w, R0, wout, sc point at the mesh's first scenario
    int64_t stride;        // distance between scenario slices (FP64 3 nc values, FP32 nc float4)
    int n_scen;            // scenarios of this mesh
    int first_item;        // first work item (block) of this mesh in the launch
    int first_entry;       // index of its first scenario among all scenarios
    int n_gauges;          // gauges of this mesh (0: none)
    const int32_t *gauge_cells;  // [n_gauges] internal cell ids
    double *ring_t;        // [n_scen][ring_cap] record times
    double *ring_eta;      // [n_scen][ring_cap][n_gauges] eta at the gauges
    int ring_cap, pad;
};

__device__ __forceinline__ void copy_cell(const double *wi, double *wo, int c, int nc)
{
    wo[c] = wi[c];
    wo[nc + c] = wi[nc + c];
    wo[2 * nc + c] = wi[2 * nc + c];
}
__device__ __forceinline__ void copy_cell(const float4 *wi, float4 *wo, int c, int) { wo[c] = wi[c]; }

// The free surface of cell c.
__device__ __forceinline__ double surface(const double *w, const double *z, int c) { return w[c] + z[c]; }
__device__ __forceinline__ double surface(const float4 *w, const float *, int c) { return (double)w[c].x; }

// Order-preserving integer image of a non-negative value, as 32 bits (FP32) or
// 64 bits (FP64), kept in shared memory per scenario.
template <typename real>
__device__ __forceinline__ unsigned long long warp_min_bits(real v)
{
    for (int o = 16; o > 0; o >>= 1) v = vmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    return min_bits(v);
}

// Shared memory of a batched CTA beside the stage's: per scenario of the batch its
// CFL minimum, its dt and whether it has reached t_end.
template <typename real>
__host__ __device__ inline size_t batch_smem_offset(size_t stage) { return (stage + 15) / 16 * 16; }
template <typename real>
__host__ __device__ inline size_t batch_smem_bytes(size_t stage, int n_entries)
{
    return batch_smem_offset<real>(stage) + (8 + sizeof(real) + 1) * (size_t)n_entries;
}

// The block functions read a scenario's arguments from shared memory: from the
// mesh table in global memory each use was a load, and a copy in registers spilled
// (the arguments are two hundred bytes).  Three slots: while a CTA's slowest warp
// may still read the last scenario's and the others the current one's, thread 0
// fills the next one's.
template <typename real, int STAGE, bool FAST = false>
__global__ void __launch_bounds__(256, (BatchMinCtas<real>::value)) batch_stage_kernel(const BatchMesh<real> *meshes, int n_mesh,
                                                          int n_items, int groups, int n_entries, DevScalars *sc_all, int scen_at)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int qcount[2];
    __shared__ __align__(16) unsigned char s_args[3][sizeof(KArgs<real>)];
    __shared__ long long red_neg[32];
    unsigned long long *s_min = reinterpret_cast<unsigned long long *>(smem_raw + scen_at);
    real *s_dt = reinterpret_cast<real *>(s_min + n_entries);
    unsigned char *s_done = reinterpret_cast<unsigned char *>(s_dt + n_entries);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = (blockDim.x + 31) >> 5;
    const KArgs<real> &p0 = meshes[0].a;
    if (STAGE == 2) chain_next();
    chain_wait();
    const double t_end = sc_all[n_entries].t_end;
    for (int e = tid; e < n_entries; e += blockDim.x) {
        s_min[e] = min_bits(real_inf<real>());
        s_dt[e] = STAGE == 2 ? (real)step_dt<real>(sc_all + e, p0.cfl, p0.dt_fixed, p0.dt_max, t_end) : real(0);
        // a scenario that has reached t_end takes steps of dt = 0 that leave its
        // state as it is (as a single context's do): skip its work, copy its state
        s_done[e] = finished(t_end, sc_all + e) ? 1 : 0;
    }
    if (tid < 2) qcount[tid] = 0;
    long long my_neg = 0;
    int parity = 0, slot = 0, last_m = -1;
    bool bad = false;
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        const int blk = item / groups, group = item - blk * groups;
        int m = 0;
        while (m + 1 < n_mesh && blk >= meshes[m + 1].first_item) m++;
        const BatchMesh<real> &bm = meshes[m];
        const int b = blk - bm.first_item, e0 = bm.first_entry;
        const int per_group = (bm.n_scen + groups - 1) / groups;
        const int s0 = group * per_group, n_scen = min(s0 + per_group, bm.n_scen);
        const int64_t stride = bm.stride;
        __syncthreads();             // every thread has done with the last item's arguments
        if (m != last_m) {
            const int *src = reinterpret_cast<const int *>(&bm.a);
            for (int i = tid; i < 3 * (int)(sizeof(KArgs<real>) / 4); i += blockDim.x)
                reinterpret_cast<int *>(s_args[0])[i] = src[i % (int)(sizeof(KArgs<real>) / 4)];
            last_m = m;
            __syncthreads();
        }
        auto next = [&](int s) {     // the first scenario from s on that still advances
            while (s < n_scen && s_done[e0 + s]) s++;
            return s;
        };
        auto fill = [&](int s, int k) {
            KArgs<real> &a = *reinterpret_cast<KArgs<real> *>(s_args[k]);
            a.w = bm.a.w + s * stride;
            a.R0 = bm.a.R0 + s * stride;
            if (STAGE == 2) a.wout = bm.a.wout + s * stride;
        };
        if (STAGE == 2) {
            // a finished scenario's state carries over to the other buffer of the pair
            const int c = b * bm.a.block + tid;
            if (tid < bm.a.block && c < (int)bm.a.nc)
                for (int s = s0; s < n_scen; s++)
                    if (s_done[e0 + s]) copy_cell(bm.a.w + s * stride, bm.a.wout + s * stride, c, (int)bm.a.nc);
        }
        bool loaded = false;
        int s = next(s0);
        if (tid == 0 && s < n_scen) fill(s, slot);
        __syncthreads();
        while (s < n_scen) {
            const int after = next(s + 1), slot2 = slot == 2 ? 0 : slot + 1;
            if (tid == 0 && after < n_scen) fill(after, slot2);
            const KArgs<real> &a = *reinterpret_cast<const KArgs<real> *>(s_args[slot]);
            real mn = real_inf<real>();
            run_block<STAGE, FAST, true, OWN>(a, b, s_dt[e0 + s], smem_raw, qcount[parity], mn, my_neg, bad, loaded);
            parity ^= 1;
            if (STAGE == 1) {
                unsigned long long bits = warp_min_bits<real>(mn);
                if (lane == 0 && bits != min_bits(real_inf<real>())) atomicMin(&s_min[e0 + s], bits);
            }
            s = after;
            slot = slot2;
        }
    }
    for (int o = 16; o > 0; o >>= 1) my_neg += __shfl_xor_sync(0xffffffffu, my_neg, o);
    if (lane == 0) red_neg[warp] = my_neg;
    bad = __syncthreads_or(bad);
    if (STAGE == 1)
        for (int e = tid; e < n_entries; e += blockDim.x)
            if (s_min[e] != min_bits(real_inf<real>())) atomicMin(&sc_all[e].dtmin_bits, s_min[e]);
    if (tid == 0) {
        long long neg = 0;
        for (int w = 0; w < nwarps; w++) neg += red_neg[w];
        if (neg) atomicAdd((unsigned long long *)&sc_all[n_entries].neg_count, (unsigned long long)neg);
        if (bad) atomicOr(&sc_all[n_entries].flags, FLAG_NONFINITE_STATE);
    }
}

// Gauge records of one batched step (after the epilogue): a scenario that
// advanced records eta at its mesh's gauges every gauge_every of its steps, in
// the circular ring at index n_rec mod ring_cap (the host drains often enough
// that no unread record is overwritten).  One CTA per mesh.
template <typename real>
__global__ void batch_gauge_kernel(const BatchMesh<real> *meshes, DevScalars *sc_all, int gauge_every)
{
    __shared__ int slot[kBatchMaxEntries];
    const BatchMesh<real> &bm = meshes[blockIdx.x];
    const int G = bm.n_gauges;
    if (G == 0) return;
    for (int s = threadIdx.x; s < bm.n_scen; s += blockDim.x) {
        const DevScalars *sc = sc_all + bm.first_entry + s;
        slot[s] = (sc->dt > 0.0 && sc->steps % gauge_every == 0) ? (int)(sc->n_rec % bm.ring_cap) : -1;
    }
    __syncthreads();
    const real *z = bm.a.z;
    for (int k = threadIdx.x; k < bm.n_scen * G; k += blockDim.x) {
        const int s = k / G, g = k - s * G;
        if (slot[s] < 0) continue;
        const auto *w = bm.a.wout + s * bm.stride;
        const int32_t c = bm.gauge_cells[g];
        bm.ring_eta[((size_t)s * bm.ring_cap + slot[s]) * G + g] = surface(w, z, c);
    }
    __syncthreads();
    for (int s = threadIdx.x; s < bm.n_scen; s += blockDim.x) {
        if (slot[s] < 0) continue;
        DevScalars *sc = sc_all + bm.first_entry + s;
        bm.ring_t[(size_t)s * bm.ring_cap + slot[s]] = sc->t;
        sc->n_rec += 1;
    }
}

// Epilogue of one batched step: per scenario t += dt (dt = 0 once it reached
// t_end), and reset of its CFL minimum.
template <typename real>
__global__ void batch_post_kernel(int n_entries, DevScalars *sc_all, double cfl, double dt_fixed, double dt_max)
{
    chain_wait();
    chain_next();
    const double t_end = sc_all[n_entries].t_end;
    for (int e = threadIdx.x; e < n_entries; e += blockDim.x) {
        DevScalars *sc = sc_all + e;
        double dt = step_dt<real>(sc, cfl, dt_fixed, dt_max, t_end);
        sc->dt = dt;
        if (!isfinite(dt)) sc_all[n_entries].flags |= FLAG_NONFINITE_DT;
        if (dt > 0.0) {
            sc->t = sc->t + dt;
            sc->steps += 1;
        }
        sc->dtmin_bits = min_bits(real_inf<real>());
    }
}

// Kernel arguments; the fields that both precisions have.
template <typename real>
KArgs<real> common_args(const DevPtrs &d, const StepParams &p)
{
    KArgs<real> a{};
    a.nc = d.nc;
    a.block = d.block;
    a.nblocks = d.nblocks;
    a.max_halo = d.max_halo;
    a.max_ring1 = d.max_ring1;
    a.order = p.order;
    a.z = static_cast<const real *>(d.z);
    a.halo_ptr = d.halo_ptr;
    a.halo_n1 = d.halo_n1;
    a.halo_ids = d.halo_ids;
    a.sc = d.sc;
    a.g = (real)p.g;
    a.half_g = (real)(0.5 * p.g);
    a.hthr = (real)p.hthr;
    a.cfl = p.cfl;
    a.dt_fixed = p.dt_fixed;
    a.dt_max = p.dt_max;
    a.cfl_min = 1;
    return a;
}

template <typename real>
KArgs<real> make_args(const DevPtrs &d, const StepParams &p, const void *w_in, void *w_out, bool soa = false);

template <>
inline KArgs<double> make_args<double>(const DevPtrs &d, const StepParams &p, const void *w_in, void *w_out, bool)
{
    KArgs<double> a = common_args<double>(d, p);
    a.geo = static_cast<const double *>(d.geo);
    a.rarea = d.rarea;
    a.M = d.M64;
    a.zf = static_cast<const double *>(d.zf);
    a.nbrl = d.nbrl;
    a.ring1_nbr = d.ring1_nbr;
    a.fq_ptr = d.fq_ptr;
    a.fq = d.fq;
    a.w = static_cast<const double *>(w_in);
    a.R0 = static_cast<double *>(d.R0);
    a.wout = static_cast<double *>(w_out);
    a.mask2 = d.mask2;
    a.fv_out = static_cast<double *>(d.fv_out);
    a.r1_out = static_cast<double *>(d.r1_out);
    a.rec_out = d.rec_out;
    a.bound_out = d.bound_out;
    return a;
}

template <>
inline KArgs<float> make_args<float>(const DevPtrs &d, const StepParams &p, const void *w_in, void *w_out, bool soa)
{
    KArgs<float> a = common_args<float>(d, p);
    a.recA = static_cast<const float4 *>(d.geo);
    a.recB = static_cast<const float4 *>(d.geoB);
    a.area = d.area32;
    a.codes = static_cast<const uint2 *>(d.codes);
    a.ring_codes = static_cast<const uint2 *>(d.ring_codes);
    a.fr_ptr = d.fq_ptr;
    a.fr = static_cast<const float4 *>(d.fr);
    a.normals = static_cast<const float2 *>(d.normals);
    a.max_faces = d.max_faces;
    a.R0 = static_cast<float4 *>(d.R0);
    if (soa) {
        a.w_soa = static_cast<const float *>(w_in);
        a.wout_soa = static_cast<float *>(w_out);
    } else {
        a.w = static_cast<const float4 *>(w_in);
        a.wout = static_cast<float4 *>(w_out);
    }
    return a;
}

// Kernel instance for a launch: the register budget follows the thread count
// (launch bounds 256 or 512).
template <typename real, bool FAST = false, int STATE = OWN>
void *stage_kernel_ptr(int stage, int threads)
{
    if (threads <= 256)
        return stage == 1 ? (void *)stage_kernel<real, 1, 256, FAST, STATE> : (void *)stage_kernel<real, 2, 256, FAST, STATE>;
    if (threads <= 384)
        return stage == 1 ? (void *)stage_kernel<real, 1, 384, FAST, STATE> : (void *)stage_kernel<real, 2, 384, FAST, STATE>;
    return stage == 1 ? (void *)stage_kernel<real, 1, 512, FAST, STATE> : (void *)stage_kernel<real, 2, 512, FAST, STATE>;
}

// The dynamic shared memory limit is an attribute of the kernel function, shared
// by every context in the process: it is only ever raised, so that a context
// configured later with a smaller block never lowers it below what another
// context's launches need.
inline cudaError_t raise_smem_limit(const void *kern, size_t smem)
{
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    if ((size_t)fa.maxDynamicSharedSizeBytes >= smem) return cudaSuccess;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

template <typename real, bool FAST = false>
int stage_config(const DevPtrs &d, int stage, LaunchCfg &cfg)
{
    cfg.smem = stage_smem_bytes<real>(d.block, d.max_halo, d.max_ring1, d.max_faces);
    const void *kern = stage_kernel_ptr<real, FAST>(stage, d.threads);
    if constexpr (std::is_same<real, float>::value)
        if (d.moving) kern = stage_kernel_ptr<real, FAST, ON_MOVING_BED>(stage, d.threads);
    cudaError_t e = raise_smem_limit(kern, cfg.smem);
    if (e != cudaSuccess) return (int)e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, d.threads, cfg.smem);
    if (e != cudaSuccess) return (int)e;
    if (per_sm < 1) return (int)cudaErrorInvalidConfiguration;
    if constexpr (std::is_same<real, float>::value) {
        // the no-allocation step's kernels, loaded here so that the step loads nothing
        e = raise_smem_limit(stage_kernel_ptr<real, FAST, CALLERS>(stage, d.threads), cfg.smem);
        if (e != cudaSuccess) return (int)e;
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long grid = (long long)sms * per_sm;
    if (grid > d.nblocks) grid = d.nblocks;
    cfg.grid = (int)(grid < 1 ? 1 : grid);
    return 0;
}

template <typename real, bool FAST = false, int STATE = OWN>
int launch_stage_args(const KArgs<real> &a, int threads, int stage, const LaunchCfg &c, cudaStream_t s)
{
    void (*k)(const KArgs<real>);
    if (threads <= 256) k = stage == 1 ? stage_kernel<real, 1, 256, FAST, STATE> : stage_kernel<real, 2, 256, FAST, STATE>;
    else if (threads <= 384) k = stage == 1 ? stage_kernel<real, 1, 384, FAST, STATE> : stage_kernel<real, 2, 384, FAST, STATE>;
    else k = stage == 1 ? stage_kernel<real, 1, 512, FAST, STATE> : stage_kernel<real, 2, 512, FAST, STATE>;
    return (int)launch_after(k, c.grid, threads, c.smem, s, a);
}

// The unfused step's three launches after stage 1 (part 0: update 1; 1: the
// stage-1 kernel on w1 writing R(w1) to R1, without its CFL bound; 2: update 2).
// w1 and R1 are [3][nc] buffers of the context.
template <typename real, bool FAST = false>
int launch_rk_unfused(const DevPtrs &d, const StepParams &p, int part, const void *w_in, void *w_out, void *w1,
                      void *R1, const LaunchCfg &c1, void *stream)
{
    using word = typename StateWord<real>::type;
    KArgs<real> a = make_args<real>(d, p, w_in, w_out);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (part == 1) {
        a.w = static_cast<const word *>(w1);
        a.R0 = static_cast<word *>(R1);
        a.wout = nullptr;
        a.cfl_min = 0;
        if constexpr (std::is_same<real, float>::value)
            if (d.moving) return launch_stage_args<real, FAST, ON_MOVING_BED>(a, d.threads, 1, c1, s);
        return launch_stage_args<real, FAST>(a, d.threads, 1, c1, s);
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long want = (d.nc + 255) / 256, cap = 8LL * (sms > 0 ? sms : 1);
    const int grid = (int)(want < 1 ? 1 : want < cap ? want : cap);
    if (part == 0) rk_update1_kernel<real><<<grid, 256, 0, s>>>(a, static_cast<word *>(w1));
    else rk_update2_kernel<real><<<grid, 256, 0, s>>>(a, static_cast<const word *>(w1), static_cast<const word *>(R1));
    return (int)cudaGetLastError();
}

// soa: the states are [3][nc] arrays (always so in FP64).
template <typename real, bool FAST = false>
int launch_stage(const DevPtrs &d, const StepParams &p, int stage, const void *w_in, void *w_out,
                 const LaunchCfg &c, void *stream, bool soa = false)
{
    const KArgs<real> a = make_args<real>(d, p, w_in, w_out, soa);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if constexpr (std::is_same<real, float>::value) {
        if (soa) return launch_stage_args<real, FAST, CALLERS>(a, d.threads, stage, c, s);
        if (d.moving) return launch_stage_args<real, FAST, ON_MOVING_BED>(a, d.threads, stage, c, s);
    }
    return launch_stage_args<real, FAST>(a, d.threads, stage, c, s);
}

template <typename real, bool FAST = false>
int batch_config(int block, int max_halo, int max_ring1, int max_faces, int n_entries, int &grid, size_t &smem, int &scen_at)
{
    const size_t stage_bytes = stage_smem_bytes<real>(block, max_halo, max_ring1, max_faces, true);
    scen_at = (int)batch_smem_offset<real>(stage_bytes);
    smem = batch_smem_bytes<real>(stage_bytes, n_entries);
    int best = 1 << 30;
    for (int stage = 1; stage <= 2; stage++) {
        auto kern = stage == 1 ? batch_stage_kernel<real, 1, FAST> : batch_stage_kernel<real, 2, FAST>;
        cudaError_t e = raise_smem_limit((const void *)kern, smem);
        if (e != cudaSuccess) return (int)e;
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, block, smem);
        if (e != cudaSuccess) return (int)e;
        best = per_sm < best ? per_sm : best;
    }
    if (best < 1) return (int)cudaErrorInvalidConfiguration;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    grid = sms * best;
    return 0;
}

template <typename real, bool FAST = false>
int launch_batch_step(const void *table, int n_mesh, int n_items, int groups, int n_entries, DevScalars *sc_all, int block,
                      int grid, size_t smem, int scen_at, const StepParams &p, bool gauges, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const BatchMesh<real> *t = static_cast<const BatchMesh<real> *>(table);
    cudaError_t e = launch_after(batch_stage_kernel<real, 1, FAST>, grid, block, smem, s, t, n_mesh, n_items, groups, n_entries, sc_all, scen_at);
    if (e == cudaSuccess)
        e = launch_after(batch_stage_kernel<real, 2, FAST>, grid, block, smem, s, t, n_mesh, n_items, groups, n_entries, sc_all, scen_at);
    if (e == cudaSuccess)
        e = launch_after(batch_post_kernel<real>, 1, 256, 0, s, n_entries, sc_all, p.cfl, p.dt_fixed, p.dt_max);
    if (e != cudaSuccess) return (int)e;
    if (gauges) batch_gauge_kernel<real><<<n_mesh, 256, 0, s>>>(t, sc_all, p.gauge_every);
    return (int)cudaGetLastError();
}

template <typename real>
void fill_batch_mesh(void *dst, const DevPtrs &d, const StepParams &p, const void *w_in, void *w_out,
                     int n_scen, int first_item, int first_entry)
{
    BatchMesh<real> *bm = static_cast<BatchMesh<real> *>(dst);
    bm->a = make_args<real>(d, p, w_in, w_out);
    bm->stride = std::is_same<real, float>::value ? d.nc : 3 * d.nc;
    bm->n_scen = n_scen;
    bm->first_item = first_item;
    bm->first_entry = first_entry;
    bm->n_gauges = d.n_gauges;
    bm->gauge_cells = d.gauge_cells;
    bm->ring_t = d.ring_t;
    bm->ring_eta = d.ring_eta;
    bm->ring_cap = d.ring_cap;
    bm->pad = 0;
}

}  // namespace vg
