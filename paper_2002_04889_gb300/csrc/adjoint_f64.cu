// Hand-written discrete adjoint of the FP64 step (reverse mode), built with
// --fmad=false like the FP64 forward kernels.
//
// The reverse of one step is seven kernels, each thread owning what it writes (no
// atomics, fixed summation order):
//   adj_begin         per cell: the reverse of the second stage update, w1 again from
//                     w and R0, and parts of dt-bar and of the search for the cell
//                     that set the CFL step
//   adj_flux_vjp      per owned face: Phi-bar, P-bar from R-bar of both cells,
//                     reverse of the interface (hydrostatic depths, HLL with its
//                     branch and speed choices, velocities) -> FV-bar and the
//                     adjoint of the bed under each face value into the (cell,
//                     face) slots of both sides
//   adj_recon_vjp     per cell: reverse of the limited least-squares
//                     reconstruction and, for a cell standing on its face beds,
//                     of the centred bed-slope source -> the cell's own w-bar,
//                     cell-bed and face-bed adjoints, and what it sends to each
//                     face neighbour ((cell, face) slots)
//   adj_gather_mid    per cell: own part + the slots its neighbours sent to it, then
//                     the reverse of the first stage update, and more of dt-bar
//   adj_flux_vjp, adj_recon_vjp, adj_gather   the same for stage 1's residual (with
//                     CFL steps one more CTA of adj_flux_vjp finds the face that set
//                     dt and reverses its wave speed meanwhile)
// and the gauges'.  The face values, reconstruction flags, dry-fix branches and CFL
// bounds are the forward kernels' records.
// Branches are frozen where the forward run took them; min/max ties resolve to
// the first argument (the convention of the oracle's taping adjoint).
#include <cuda_runtime.h>

#include "step_kernels.cuh"

namespace vg {

namespace {

// Exact IEEE comparisons of FP64 values on the integer units (for every
// non-NaN input), beside the sign and threshold tests of step_kernels.cuh:
// the reverse kernels record which argument of a min / max or which side of a
// test carried the value, so a tie between +0 and -0 must decide as FP64 does.
__device__ __forceinline__ bool lt_x(double a, double b)      // a < b
{
    return okey(a) < okey(b) && ((ubits(a) | ubits(b)) << 1) != 0;
}
__device__ __forceinline__ bool lt_pos(double x, double y)    // x < y for y > 0
{
    return dbits(x) < dbits(y);
}
__device__ __forceinline__ bool gt_abs(double a, double b)    // |a| > |b|
{
    return (dbits(a) & 0x7fffffffffffffffLL) > (dbits(b) & 0x7fffffffffffffffLL);
}

// CTA reductions with a fixed order: a warp's shuffle tree, then the warps in turn;
// thread 0 has the result.
constexpr int kRedThreads = 256;
// The two heavy reverse kernels run 64-thread CTAs: what flows back from a few gauges
// fills a connected part of the mesh, and small CTAs spread it over the SMs (backward
// of 16 CFL steps, ms, with 128 / 64 / 32 threads: 49k triangles 10.4 / 9.4 / 9.3, 205k
// 22.9 / 22.6 / 23.2, 1M 92.5 / 86.1 / 87.9).
constexpr int kVjpThreads = 64;

__device__ __forceinline__ bool cfl_less(double b1, int o1, double b2, int o2)
{
    return b1 < b2 || (b1 == b2 && o1 < o2);
}

template <int NT>
__device__ __forceinline__ void cta_argmin(double &b, int &o, int &k)
{
    __shared__ double sb[NT / 32];
    __shared__ int so[NT / 32], sk[NT / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int s = 16; s > 0; s >>= 1) {
        const double b2 = __shfl_down_sync(0xffffffffu, b, s);
        const int o2 = __shfl_down_sync(0xffffffffu, o, s), k2 = __shfl_down_sync(0xffffffffu, k, s);
        if (cfl_less(b2, o2, b, o)) { b = b2; o = o2; k = k2; }
    }
    if (lane == 0) { sb[warp] = b; so[warp] = o; sk[warp] = k; }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < NT / 32; w++)
            if (cfl_less(sb[w], so[w], b, o)) { b = sb[w]; o = so[w]; k = sk[w]; }
}

template <int NT>
__device__ __forceinline__ double cta_sum(double s)
{
    __shared__ double sh[NT / 32];
    for (int k = 16; k > 0; k >>= 1) s += __shfl_down_sync(0xffffffffu, s, k);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < NT / 32; w++) s += sh[w];
    return s;
}

struct AdjMesh {
    int nc, order;
    const double *geo;       // [GEO_ROWS][nc]
    const double *rarea;     // [nc] 1 / area
    const double *z;         // [nc]
    const double *zf;        // [3][nc] face beds
    const uint8_t *rec;      // [nc] the stage's reconstruction flags (forward record)
    const int32_t *nbr;      // [3][nc]
    const uint16_t *nbrl;    // [3][nc]: low 2 bits = neighbour's face (not a wall)
    const int32_t *faces;    // every face once: (owning cell << 2) | face
    int nfaces;
    double g, half_g, hthr;
};

__device__ __forceinline__ double G(const AdjMesh &m, int row, int k) { return m.geo[row * m.nc + k]; }
__device__ __forceinline__ Recip by_area(const AdjMesh &m, int k) { return recip_given(G(m, GEO_AREA, k), m.rarea[k]); }

// The bed under face value f of cell K: its face bed where K reconstructed,
// its cell bed otherwise.
__device__ __forceinline__ double bed_under(const AdjMesh &m, int K, int f)
{
    return m.rec[K] ? m.zf[f * m.nc + K] : m.z[K];
}

// Forward reconstruction of cell K (the same evaluation order as the forward
// kernels), keeping what the reverse needs.
struct ReconFwd {
    double qK[3], qn[3][3];
    bool wall[3];            // boundary face (wall, open or absorbing)
    bool open[3];            // open or absorbing face: the ghost is the cell itself
    bool recon;
    double D[3][3];          // [v][f]
    double alpha[3];
    int fa[3];               // face whose phi is the active limiter (-1: alpha = 1)
    int imax[3], imin[3];    // stencil index of q_max / q_min (-1 = the cell)
    double r[3];             // q_max - q_K or q_min - q_K of the active face
};

__device__ __forceinline__ void recon_forward(const AdjMesh &m, const double *w, int K, ReconFwd &R, double Hf[3],
                              double Huf[3], double Hvf[3])
{
    const int nc = m.nc;
    const double *H = w, *Hu = w + nc, *Hv = w + 2 * (size_t)nc;
    double zK = m.z[K];
    double HK = H[K], HuK = Hu[K], HvK = Hv[K];
    R.qK[0] = HK + zK;
    R.qK[1] = HuK;
    R.qK[2] = HvK;
    bool recon = (m.order == 2) && (HK > m.hthr);
#pragma unroll
    for (int f = 0; f < 3; f++) {
        int j = m.nbr[f * nc + K];
        R.wall[f] = j < 0;
        R.open[f] = j == -2 || j == -3;
        if (j >= 0) {
            R.qn[f][0] = H[j] + m.z[j];
            R.qn[f][1] = Hu[j];
            R.qn[f][2] = Hv[j];
            if (!(H[j] > m.hthr)) recon = false;
        } else if (R.open[f]) {
            R.qn[f][0] = R.qK[0];
            R.qn[f][1] = HuK;
            R.qn[f][2] = HvK;
        } else {
            double nx = G(m, GEO_NX + f, K), ny = G(m, GEO_NY + f, K);
            double mn = HuK * nx + HvK * ny;
            R.qn[f][0] = R.qK[0];
            R.qn[f][1] = HuK - 2.0 * mn * nx;
            R.qn[f][2] = HvK - 2.0 * mn * ny;
        }
    }
    if (recon) {
        double face[3][3];
#pragma unroll
        for (int v = 0; v < 3; v++) {
            double d0 = R.qn[0][v] - R.qK[v], d1 = R.qn[1][v] - R.qK[v], d2 = R.qn[2][v] - R.qK[v];
            double gx = (G(m, GEO_WX, K) * d0 + G(m, GEO_WX + 1, K) * d1) + G(m, GEO_WX + 2, K) * d2;
            double gy = (G(m, GEO_WY, K) * d0 + G(m, GEO_WY + 1, K) * d1) + G(m, GEO_WY + 2, K) * d2;
            double qmax = R.qK[v], qmin = R.qK[v];
            int imax = -1, imin = -1;
#pragma unroll
            for (int f = 0; f < 3; f++) {
                if (lt_x(qmax, R.qn[f][v])) { qmax = R.qn[f][v]; imax = f; }
                if (lt_x(R.qn[f][v], qmin)) { qmin = R.qn[f][v]; imin = f; }
            }
            // The active limiter: the first face of smallest quotient r / D below 1.  The
            // smallest quotient is that of the largest D > 0 or of the largest -D > 0, so
            // two candidates and one division serve, as in the forward kernels; but a face
            // whose D is a few ulps smaller may have the same rounded quotient, and so may
            // the two candidates where their cross products differ in the last bits.  Where
            // the high words leave that open (or the quotient is near the subnormal
            // numbers) the quotients of all three faces are formed and compared.
            const double up = qmax - R.qK[v], dn = R.qK[v] - qmin;
            double P = 0.0, M = 0.0;
            int fP = -1, fM = -1;
#pragma unroll
            for (int f = 0; f < 3; f++) {
                const double D = gx * G(m, GEO_FX + f, K) + gy * G(m, GEO_FY + f, K);
                R.D[v][f] = D;
                if (is_pos(D) && gt_nn(D, P)) { P = D; fP = f; }
                if (is_neg(D) && gt_nn(-D, M)) { M = -D; fM = f; }
            }
            double alpha = 1.0, ra = 0.0;
            int fa = -1;
            const bool limP = gt_nn(P, up), limM = gt_nn(M, dn);
            if (limP || limM) {
                const double xP = up * M, xM = dn * P;
                const bool takeM = limM && (!limP || gt_nn(xP, xM));
                const double num = takeM ? dn : up, den = takeM ? M : P;
                alpha = quot(num, recip(den));
                fa = takeM ? fM : fP;
                ra = takeM ? -dn : up;
                // integer differences of high words: <= 1 for neighbours at most 2^32 steps apart
                const int hx = __double2hiint(xP) - __double2hiint(xM), hd = __double2hiint(den);
                bool open = (limP && limM && hx <= 1 && hx >= -1) || (__double2hiint(alpha) < (64 << 20) && !is_zero(num));
#pragma unroll
                for (int f = 2; f >= 0; f--) {
                    const int h = __double2hiint(R.D[v][f]) ^ (takeM ? (int)0x80000000 : 0);    // |D| if of the taken sign, else < 0
                    const bool same = h >= 0 && !is_zero(R.D[v][f]);
                    if (same && is_zero(num)) fa = f;                // every quotient of this sign is 0
                    open = open || (same && f < fa && hd - h <= 1 && !is_zero(num));
                }
                if (open) {
                    alpha = 1.0;
#pragma unroll
                    for (int f = 0; f < 3; f++) {
                        const double D = R.D[v][f];
                        if (is_zero(D)) continue;
                        const bool neg = is_neg(D);
                        const double t = quot(neg ? dn : up, recip(neg ? -D : D));
                        if (lt_pos(t, alpha)) { alpha = t; fa = f; ra = neg ? -dn : up; }
                    }
                }
            }
            R.alpha[v] = alpha;
            R.fa[v] = fa;
            R.r[v] = ra;
            R.imax[v] = imax;
            R.imin[v] = imin;
#pragma unroll
            for (int f = 0; f < 3; f++) face[f][v] = R.qK[v] + alpha * R.D[v][f];
        }
#pragma unroll
        for (int f = 0; f < 3; f++) {
            Hf[f] = face[f][0] - m.zf[f * nc + K];
            if (!(Hf[f] > m.hthr)) recon = false;
            Huf[f] = face[f][1];
            Hvf[f] = face[f][2];
        }
    }
    R.recon = recon;
    if (!recon) {
#pragma unroll
        for (int f = 0; f < 3; f++) { Hf[f] = HK; Huf[f] = HuK; Hvf[f] = HvK; }
    }
}

// The flux VJP skips a face where neither cell has a residual adjoint (the VJP of
// zero is zero).
__device__ __forceinline__ bool rb_nonzero(const double *Rb, int nc, int k)
{
    return !is_zero(Rb[k]) || !is_zero(Rb[nc + k]) || !is_zero(Rb[2 * (size_t)nc + k]);
}

// Reverse of the face flux seen from L (forward: face_flux / hll_normal).
// Inputs: the two face states, beds, normal, wall flag, and the adjoints of
// Phi[3], P_L, P_R and of the wave speed a = max(|s_L|, |s_R|) (amb: nonzero
// only for the face that sets the CFL time step); bnd, the kind of a boundary
// face: 1 wall, 2 open, 3 absorbing.  Outputs: adjoints of (H_f, Hu_f, Hv_f, z)
// on each side.  The absorbing ghost (characteristic ghost of a sea at rest at
// eta = 0 beyond the face) depends on the face state through the outgoing
// invariant u_n + 2c and on the bed under the face through c_0 = sqrt(g max(0, -z)).
__device__ __forceinline__ void flux_vjp(const AdjMesh &m, double HfL, double HufL, double HvfL, double zL, double HfR,
                         double HufR, double HvfR, double zR, double nx, double ny, bool wall,
                         const double Pb[3], double PLb, double PRb, double bL[4], double bR[4],
                         double amb = 0.0, int bnd = 1)
{
    const double g = m.g, hg = m.half_g, hthr = m.hthr;
    for (int k = 0; k < 4; k++) { bL[k] = 0.0; bR[k] = 0.0; }
    // ---- forward
    double uL = 0.0, vL = 0.0;
    bool velL = gt_nn(HfL, hthr);
    const Recip rL = recip(HfL), rR = recip(HfR);      // (used where the side has a velocity)
    if (velL) { uL = quot(HufL, rL); vL = quot(HvfL, rL); }
    double unL = uL * nx + vL * ny;
    double utL = -uL * ny + vL * nx;
    double HsL, HsR, unR, utR, uR = 0.0, vR = 0.0, zs = 0.0;
    bool velR = false, zR_max = false, actL, actR = false;
    double xL, xR = 0.0;
    double cgL = 0.0, c0 = 0.0, cg = 0.0;    // absorbing ghost: c of the face state, of the sea, of the ghost
    bool act0 = false, actg = false;
    if (wall && bnd == 3) {
        xL = (HfL + zL) - zL;
        actL = is_pos(xL);
        HsL = actL ? xL : 0.0;
        cgL = sqrt(g * HsL);
        const double x0 = 0.0 - zL;
        act0 = is_pos(x0);
        c0 = sqrt(g * (act0 ? x0 : 0.0));
        const double Rp = unL + 2.0 * cgL, Rm = 0.0 - 2.0 * c0;
        unR = 0.5 * (Rp + Rm);
        const double y = 0.25 * (Rp - Rm);
        actg = is_pos(y);
        cg = actg ? y : 0.0;
        HsR = cg * cg / g;
        utR = utL;
    } else if (wall) {
        xL = (HfL + zL) - zL;
        actL = is_pos(xL);
        HsL = actL ? xL : 0.0;
        HsR = HsL;
        unR = bnd == 2 ? unL : -unL;
        utR = utL;
    } else {
        velR = gt_nn(HfR, hthr);
        if (velR) { uR = quot(HufR, rR); vR = quot(HvfR, rR); }
        unR = uR * nx + vR * ny;
        utR = -uR * ny + vR * nx;
        zR_max = lt_x(zL, zR);
        zs = zR_max ? zR : zL;
        xL = (HfL + zL) - zs;
        xR = (HfR + zR) - zs;
        actL = is_pos(xL);
        actR = is_pos(xR);
        HsL = actL ? xL : 0.0;
        HsR = actR ? xR : 0.0;
    }
    // ---- reverse of the rotation and pressure terms
    double Fb0 = Pb[0];
    double Fb1 = Pb[1] * nx + Pb[2] * ny;
    double Fb2 = -Pb[1] * ny + Pb[2] * nx;
    double HfLb = PLb * hg * 2.0 * HfL, HsLb = -PLb * hg * 2.0 * HsL;
    double HfRb = 0.0, HsRb = 0.0;
    if (!wall) { HfRb = PRb * hg * 2.0 * HfR; HsRb = -PRb * hg * 2.0 * HsR; }
    double unLb = 0.0, utLb = 0.0, unRb = 0.0, utRb = 0.0;
    // ---- reverse of HLL
    if (!(is_zero(HsL) && is_zero(HsR))) {
        double cL = sqrt(g * HsL), cR = sqrt(g * HsR);
        double sL, sR, us = 0.0, cs = 0.0;
        int case_ = 0;    // 0 both wet, 1 L dry, 2 R dry
        bool sL_first = true, sR_first = true;
        if (is_zero(HsL)) {
            case_ = 1;
            sL = unR - 2.0 * cR;
            sR = unR + cR;
        } else if (is_zero(HsR)) {
            case_ = 2;
            sL = unL - cL;
            sR = unL + 2.0 * cL;
        } else {
            us = 0.5 * (unL + unR) + (cL - cR);
            cs = 0.5 * (cL + cR) - 0.25 * (unR - unL);
            double a1 = unL - cL, a2 = us - cs;
            sL_first = !lt_x(a2, a1);
            sL = sL_first ? a1 : a2;
            double b1 = us + cs, b2 = unR + cR;
            sR_first = !lt_x(b1, b2);
            sR = sR_first ? b1 : b2;
        }
        double qL = HsL * unL, qR = HsR * unR;
        double FL[3] = {qL, qL * unL + hg * HsL * HsL, qL * utL};
        double FR[3] = {qR, qR * unR + hg * HsR * HsR, qR * utR};
        double wL[3] = {HsL, qL, HsL * utL};
        double wR[3] = {HsR, qR, HsR * utR};
        double Fb[3] = {Fb0, Fb1, Fb2};
        double FLb[3] = {0, 0, 0}, FRb[3] = {0, 0, 0}, wLb[3] = {0, 0, 0}, wRb[3] = {0, 0, 0};
        double sLb = 0.0, sRb = 0.0;
        if (!is_neg(sL)) {
            for (int k = 0; k < 3; k++) FLb[k] = Fb[k];
        } else if (!is_neg(sR)) {
            double den = sR - sL, sLR = sL * sR, iden = inverse(recip(den));
            double denb = 0.0, sLRb = 0.0;
            for (int k = 0; k < 3; k++) {
                double N = (sR * FL[k] - sL * FR[k]) + sLR * (wR[k] - wL[k]);
                double F = N * iden;
                double Nb = Fb[k] * iden;
                denb -= Fb[k] * F * iden;
                FLb[k] += Nb * sR;
                FRb[k] -= Nb * sL;
                sRb += Nb * FL[k];
                sLb -= Nb * FR[k];
                sLRb += Nb * (wR[k] - wL[k]);
                wRb[k] += Nb * sLR;
                wLb[k] -= Nb * sLR;
            }
            sLb += sLRb * sR;
            sRb += sLRb * sL;
            sRb += denb;
            sLb -= denb;
        } else {
            for (int k = 0; k < 3; k++) FRb[k] = Fb[k];
        }
        // physical fluxes and conserved variables -> (Hs, q, un, ut)
        double qLb = FLb[0] + FLb[1] * unL + FLb[2] * utL + wLb[1];
        unLb += FLb[1] * qL;
        HsLb += FLb[1] * 2.0 * hg * HsL + wLb[0] + wLb[2] * utL;
        utLb += FLb[2] * qL + wLb[2] * HsL;
        HsLb += qLb * unL;
        unLb += qLb * HsL;
        double qRb = FRb[0] + FRb[1] * unR + FRb[2] * utR + wRb[1];
        unRb += FRb[1] * qR;
        HsRb += FRb[1] * 2.0 * hg * HsR + wRb[0] + wRb[2] * utR;
        utRb += FRb[2] * qR + wRb[2] * HsR;
        HsRb += qRb * unR;
        unRb += qRb * HsR;
        // the wave speed a = max(|s_L|, |s_R|) (a tie takes |s_L|; |s| at s = 0 takes +s)
        if (!is_zero(amb)) {
            if (gt_abs(sR, sL)) sRb += is_neg(sR) ? -amb : amb;
            else sLb += is_neg(sL) ? -amb : amb;
        }
        // speeds
        double cLb = 0.0, cRb = 0.0;
        if (case_ == 1) {
            unRb += sLb + sRb;
            cRb += -2.0 * sLb + sRb;
        } else if (case_ == 2) {
            unLb += sLb + sRb;
            cLb += -sLb + 2.0 * sRb;
        } else {
            double usb = 0.0, csb = 0.0;
            if (sL_first) { unLb += sLb; cLb -= sLb; } else { usb += sLb; csb -= sLb; }
            if (sR_first) { usb += sRb; csb += sRb; } else { unRb += sRb; cRb += sRb; }
            unLb += 0.5 * usb;
            unRb += 0.5 * usb;
            cLb += usb;
            cRb -= usb;
            cLb += 0.5 * csb;
            cRb += 0.5 * csb;
            unRb -= 0.25 * csb;
            unLb += 0.25 * csb;
        }
        if (is_pos(cL)) HsLb += cLb * quot(0.5, recip(cL)) * g;
        if (is_pos(cR)) HsRb += cRb * quot(0.5, recip(cR)) * g;
    }
    // ---- reverse of the interface depths and velocities
    if (wall && bnd == 3) {
        // HsR = c_g^2 / g, c_g = max(0, (R+ - R-)/4), u_n,R = (R+ + R-)/2,
        // R+ = u_n,L + 2 c_L, R- = -2 c_0
        const double yb = actg ? HsRb * (2.0 * cg / g) : 0.0;
        const double Rpb = 0.5 * unRb + 0.25 * yb, Rmb = 0.5 * unRb - 0.25 * yb;
        unLb += Rpb;
        if (is_pos(cgL)) HsLb += (2.0 * Rpb) * (0.5 / cgL) * g;
        if (is_pos(c0) && act0) bL[3] -= (-2.0 * Rmb) * (0.5 / c0) * g;
        utLb += utRb;
        if (actL) { HfLb += HsLb; bL[3] += HsLb; bL[3] -= HsLb; }
    } else if (wall) {
        unLb += bnd == 2 ? unRb : -unRb;
        utLb += utRb;
        HsLb += HsRb;
        if (actL) { HfLb += HsLb; bL[3] += HsLb; bL[3] -= HsLb; }
    } else {
        double zsb = 0.0;
        if (actL) { HfLb += HsLb; bL[3] += HsLb; zsb -= HsLb; }
        if (actR) { HfRb += HsRb; bR[3] += HsRb; zsb -= HsRb; }
        if (zR_max) bR[3] += zsb; else bL[3] += zsb;
        double uRb = unRb * nx - utRb * ny, vRb = unRb * ny + utRb * nx;
        if (velR) {
            double inv = inverse(rR);
            bR[1] += uRb * inv;
            bR[2] += vRb * inv;
            HfRb -= (uRb * uR + vRb * vR) * inv;
        }
    }
    double uLb = unLb * nx - utLb * ny, vLb = unLb * ny + utLb * nx;
    if (velL) {
        double inv = inverse(rL);
        bL[1] += uLb * inv;
        bL[2] += vLb * inv;
        HfLb -= (uLb * uL + vLb * vL) * inv;
    }
    bL[0] += HfLb;
    bR[0] += HfRb;
}

// Per cell: reverse of the reconstruction.  own[7][nc] = (H, Hu, Hv, z_K)-bar of
// the cell itself, then the adjoints of its three face beds; send[(f*4+k)*nc + K]
// = the (H, Hu, Hv, z)-bar that cell K passes to its face-f neighbour.  The
// flux slots' bed adjoint (zfb) belongs to the bed under the face value: the
// face bed where the cell reconstructed, its cell bed otherwise.  A cell that
// reconstructed also carries the centred source g sum_f l_f z_f (eta_K - z_f/2)
// n_f of its momentum residual R = -(1/|K|)(... + source): with
// q_f = -(g/|K|) l_f (n_f . (R-bar_Hu, R-bar_Hv)), eta-bar_K += sum_f q_f z_f and
// z_f-bar += q_f (eta_K - z_f).
__global__ void __launch_bounds__(kVjpThreads) adj_recon_vjp_kernel(AdjMesh m, const double *w, const double *Rb, const double *FVb,
                                     const double *zfb, double *own, double *send, const AdjCflFace *cf)
{
    const int nc = m.nc;
    for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < nc; K += gridDim.x * blockDim.x) {
        double fb[3][3];   // [v][f]
        bool any = m.rec[K] && (!is_zero(Rb[nc + K]) || !is_zero(Rb[2 * (size_t)nc + K]));
#pragma unroll
        for (int v = 0; v < 3; v++)
#pragma unroll
            for (int f = 0; f < 3; f++) fb[v][f] = FVb[(v * 3 + f) * (size_t)nc + K];
        double zsl[3];
#pragma unroll
        for (int f = 0; f < 3; f++) zsl[f] = zfb[f * (size_t)nc + K];
        if (cf && (cf->cell[0] == K || cf->cell[1] == K)) {
            // the face that set the CFL step: its wave speed's adjoint on this side
            const int side = cf->cell[0] == K ? 0 : 1;
#pragma unroll
            for (int f = 0; f < 3; f++)
                if (f == cf->face[side]) {
#pragma unroll
                    for (int v = 0; v < 3; v++) fb[v][f] += cf->bar[side][v];
                    zsl[f] += cf->bar[side][3];
                }
        }
#pragma unroll
        for (int v = 0; v < 3; v++)
#pragma unroll
            for (int f = 0; f < 3; f++) any = any || !is_zero(fb[v][f]);
        if (!any) {                      // nothing flows back through the reconstruction
            own[K] = 0.0;
            own[nc + K] = 0.0;
            own[2 * (size_t)nc + K] = 0.0;
            const bool rk = m.rec[K];
            own[3 * (size_t)nc + K] = rk ? 0.0 : (zsl[0] + zsl[1]) + zsl[2];
#pragma unroll
            for (int f = 0; f < 3; f++) own[(4 + f) * (size_t)nc + K] = rk ? zsl[f] : 0.0;
#pragma unroll
            for (int q = 0; q < 12; q++) send[q * (size_t)nc + K] = 0.0;
            continue;
        }
        ReconFwd R;
        double Hf[3], Huf[3], Hvf[3];
        recon_forward(m, w, K, R, Hf, Huf, Hvf);
        double Hb = 0.0, Hub = 0.0, Hvb = 0.0, zb = 0.0, zfbK[3] = {0.0, 0.0, 0.0};
        double qnb[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};   // [f][v]
        if (!R.recon) {
            zb = (zsl[0] + zsl[1]) + zsl[2];
#pragma unroll
            for (int f = 0; f < 3; f++) { Hb += fb[0][f]; Hub += fb[1][f]; Hvb += fb[2][f]; }
        } else {
            double qKb[3] = {0, 0, 0};
#pragma unroll
            for (int f = 0; f < 3; f++) zfbK[f] = zsl[f] - fb[0][f];      // H_f = eta_f - z_f
            {
                // the centred source
                const double c = quot(-m.g, by_area(m, K));
                const double rbu = Rb[nc + K], rbv = Rb[2 * (size_t)nc + K];
                const double eK = w[K] + m.z[K];
                double eb = 0.0;
#pragma unroll
                for (int f = 0; f < 3; f++) {
                    const double zff = m.zf[f * nc + K];
                    const double q = c * (G(m, GEO_LEN + f, K) * (G(m, GEO_NX + f, K) * rbu + G(m, GEO_NY + f, K) * rbv));
                    eb += q * zff;
                    zfbK[f] += q * (eK - zff);
                }
                Hb += eb;
                zb += eb;
            }
#pragma unroll
            for (int v = 0; v < 3; v++) {
                double ab = 0.0, Db[3];
#pragma unroll
                for (int f = 0; f < 3; f++) {
                    qKb[v] += fb[v][f];
                    ab += fb[v][f] * R.D[v][f];
                    Db[f] = fb[v][f] * R.alpha[v];
                }
                const int fa = R.fa[v];
                if (fa >= 0) {
                    // (faces picked by compare and select, not by index: indexed
                    // arrays would live in local memory)
                    const double D = fa == 0 ? R.D[v][0] : fa == 1 ? R.D[v][1] : R.D[v][2];
                    double iD = inverse(recip(D));
                    double rb = ab * iD;
#pragma unroll
                    for (int f = 0; f < 3; f++)
                        if (f == fa) Db[f] -= rb * R.r[v] * iD;
                    int idx = is_pos(D) ? R.imax[v] : R.imin[v];
                    if (idx < 0) qKb[v] += rb;
#pragma unroll
                    for (int f = 0; f < 3; f++)
                        if (f == idx) qnb[f][v] += rb;
                    qKb[v] -= rb;
                }
                double gxb = 0.0, gyb = 0.0;
#pragma unroll
                for (int f = 0; f < 3; f++) {
                    gxb += Db[f] * G(m, GEO_FX + f, K);
                    gyb += Db[f] * G(m, GEO_FY + f, K);
                }
#pragma unroll
                for (int f = 0; f < 3; f++) {
                    double db = gxb * G(m, GEO_WX + f, K) + gyb * G(m, GEO_WY + f, K);
                    qnb[f][v] += db;
                    qKb[v] -= db;
                }
            }
#pragma unroll
            for (int f = 0; f < 3; f++) {
                if (!R.wall[f]) continue;
                if (R.open[f]) {                 // ghost = the cell's own values
                    qKb[0] += qnb[f][0];
                    Hub += qnb[f][1];
                    Hvb += qnb[f][2];
                    qnb[f][0] = qnb[f][1] = qnb[f][2] = 0.0;
                    continue;
                }
                double nx = G(m, GEO_NX + f, K), ny = G(m, GEO_NY + f, K);
                qKb[0] += qnb[f][0];
                double mnb = -2.0 * nx * qnb[f][1] - 2.0 * ny * qnb[f][2];
                Hub += qnb[f][1] + mnb * nx;
                Hvb += qnb[f][2] + mnb * ny;
                qnb[f][0] = qnb[f][1] = qnb[f][2] = 0.0;
            }
            Hb += qKb[0];
            zb += qKb[0];
            Hub += qKb[1];
            Hvb += qKb[2];
        }
        own[K] = Hb;
        own[nc + K] = Hub;
        own[2 * (size_t)nc + K] = Hvb;
        own[3 * (size_t)nc + K] = zb;
#pragma unroll
        for (int f = 0; f < 3; f++) own[(4 + f) * (size_t)nc + K] = zfbK[f];
#pragma unroll
        for (int f = 0; f < 3; f++) {
            send[(f * 4 + 0) * (size_t)nc + K] = qnb[f][0];     // eta-bar -> H-bar and z-bar
            send[(f * 4 + 1) * (size_t)nc + K] = qnb[f][1];
            send[(f * 4 + 2) * (size_t)nc + K] = qnb[f][2];
            send[(f * 4 + 3) * (size_t)nc + K] = qnb[f][0];
        }
    }
}

// Own part + what the face neighbours sent: a = the adjoints of (H, Hu, Hv, z_K) of
// cell K; zb[nc] (cell beds) and rows 1..3 (face beds) +=.
__device__ __forceinline__ void gathered(const AdjMesh &m, int K, const double *own, const double *send, double *zb, double a[3])
{
    const int nc = m.nc;
    double s[4] = {own[K], own[nc + K], own[2 * (size_t)nc + K], own[3 * (size_t)nc + K]};
    for (int f = 0; f < 3; f++) {
        const int j = m.nbr[f * nc + K];
        if (j < 0) continue;
        const int fj = m.nbrl[f * nc + K] & 3;
        for (int k = 0; k < 4; k++) s[k] += send[(fj * 4 + k) * (size_t)nc + j];
    }
    zb[K] += s[3];
    for (int f = 0; f < 3; f++) zb[(1 + f) * (size_t)nc + K] += own[(4 + f) * (size_t)nc + K];
    a[0] = s[0]; a[1] = s[1]; a[2] = s[2];
}

// wb[3][nc] += the gathered adjoints.
__global__ void adj_gather_kernel(AdjMesh m, const double *own, const double *send, double *wb, double *zb)
{
    const int nc = m.nc;
    for (int K = blockIdx.x * blockDim.x + threadIdx.x; K < nc; K += gridDim.x * blockDim.x) {
        double a[3];
        gathered(m, K, own, send, zb, a);
        for (int k = 0; k < 3; k++) wb[k * (size_t)nc + K] += a[k];
    }
}

// Dry fix after a stage (forward: H < 0 empties the cell; H <= H_threshold zeroes
// the momentum): its adjoint masks the incoming adjoint.
__device__ __forceinline__ void dry_fix_mask(double Hpre, double hthr, double &Hb, double &Hub, double &Hvb)
{
    if (is_neg(Hpre)) { Hb = 0.0; Hub = 0.0; Hvb = 0.0; }
    else if (!gt_nn(Hpre, hthr)) { Hub = 0.0; Hvb = 0.0; }
}

// The beginning of a step's reverse, per cell:
//  * w1 = fix(w + dt R0), keeping the pre-fix depth for the mask;
//  * the reverse of stage 2, w^{n+1} = fix(w/2 + (w1 + dt R1)/2), with the dry-fix
//    branch recorded by the forward stage-2 kernel (0 none, 1 momentum cut, 2
//    emptied): from wb (adjoint of w^{n+1}), wb_n = wb_1 = 1/2 wbpre, Rb = dt/2 wbpre;
//  * with CFL steps the CTA's part of sum Rb . R1 (dt-bar) and of the search for the
//    cell of smallest CFL bound.
// (Three elementwise kernels and a reduction of their own moved these arrays through
// memory twice, 18 us of launches and passes at 49k triangles.)
__global__ void __launch_bounds__(kRedThreads) adj_begin_kernel(int nc, double dt, double hthr, const double *w, const double *R0,
                                                                double *w1, double *H1pre, const uint8_t *mask2, const double *wb,
                                                                double *wbn, double *wb1, double *Rb, const AdjCfl cfl)
{
    double sum = 0.0, bb = INFINITY;
    int bo = 0x7fffffff, bk = -1;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nc; k += gridDim.x * blockDim.x) {
        double q[3];
        for (int c = 0; c < 3; c++) q[c] = w[c * (size_t)nc + k] + dt * R0[c * (size_t)nc + k];
        H1pre[k] = q[0];
        if (is_neg(q[0])) { q[0] = 0.0; q[1] = 0.0; q[2] = 0.0; }
        else if (!gt_nn(q[0], hthr)) { q[1] = 0.0; q[2] = 0.0; }
        const uint8_t br = mask2[k];
        double b[3] = {wb[k], wb[nc + k], wb[2 * (size_t)nc + k]};
        if (br == 2) { b[0] = 0.0; b[1] = 0.0; b[2] = 0.0; }
        else if (br == 1) { b[1] = 0.0; b[2] = 0.0; }
        for (int c = 0; c < 3; c++) {
            const size_t i = c * (size_t)nc + k;
            w1[i] = q[c];
            const double h = half_of(b[c]), r = 0.5 * dt * b[c];
            wbn[i] = h;
            wb1[i] = h;
            Rb[i] = r;
            if (cfl.dt) sum += r * cfl.R1[i];
        }
        if (cfl.dt) {
            const double bd = cfl.bound[k];              // +inf where nothing moves
            if (bd <= bb && bd < INFINITY && cfl_less(bd, cfl.orig[k], bb, bo)) { bb = bd; bo = cfl.orig[k]; bk = k; }
        }
    }
    if (!cfl.dt) return;
    sum = cta_sum<kRedThreads>(sum);
    cta_argmin<kRedThreads>(bb, bo, bk);
    if (threadIdx.x == 0) {
        cfl.part_s1[blockIdx.x] = sum;
        cfl.part_b[blockIdx.x] = bb;
        cfl.part_o[blockIdx.x] = bo;
        cfl.part_k[blockIdx.x] = bk;
    }
}

// Between the two residuals, per cell: wb1 += what stage 2's residual gathered, then
// the reverse of stage 1, w1 = fix(w + dt R0): wbn += wb1pre, Rb = dt wb1pre, and
// with CFL steps the CTA's part of sum Rb . R0.
__global__ void __launch_bounds__(kRedThreads) adj_gather_mid_kernel(AdjMesh m, const double *own, const double *send, double *zb,
                                                                     double dt, double hthr, const double *H1pre, const double *wb1,
                                                                     double *wbn, double *Rb, const AdjCfl cfl)
{
    const int nc = m.nc;
    double sum = 0.0;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nc; k += gridDim.x * blockDim.x) {
        double b[3];
        gathered(m, k, own, send, zb, b);
        for (int c = 0; c < 3; c++) b[c] = wb1[c * (size_t)nc + k] + b[c];
        dry_fix_mask(H1pre[k], hthr, b[0], b[1], b[2]);
        for (int c = 0; c < 3; c++) {
            const size_t i = c * (size_t)nc + k;
            const double r = dt * b[c];
            wbn[i] += b[c];
            Rb[i] = r;
            if (cfl.dt) sum += r * cfl.R0[i];
        }
    }
    if (!cfl.dt) return;
    sum = cta_sum<kRedThreads>(sum);
    if (threadIdx.x == 0) cfl.part_s0[blockIdx.x] = sum;
}

// Gauge functional J = sum weights * (H + z) at the gauge cells: its adjoint.
// Two gauges may share a cell: the first gauge of a cell adds all of that cell's
// weights, in gauge order (one thread per gauge; one thread walking all gauges
// was a chain of dependent loads, 18 us for 16 gauges).
__global__ void adj_gauge_kernel(int n_gauges, const int32_t *cells, const double *weights, double *wb, double *zb)
{
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < n_gauges; g += gridDim.x * blockDim.x) {
        const int c = cells[g];
        bool first = true;
        for (int h = 0; h < g && first; h++) first = cells[h] != c;
        if (!first) continue;
        double bw = wb[c], bz = zb[c];
        for (int h = g; h < n_gauges; h++)
            if (cells[h] == c) { bw += weights[h]; bz += weights[h]; }
        wb[c] = bw;
        zb[c] = bz;
    }
}

// ---------------------------------------------------------------------------
// Adjoint through the CFL time step (Sec. 2.3 rule, vg_adj_forward with dt = 0):
// dt = cfl |K*| / (3 l_f* a_f*) for the cell K* of smallest bound and its face
// f* of largest l_f a_f, so dt-bar reaches the state only through the wave
// speed of that one face: a-bar = -dt-bar dt / a.  dt-bar itself is
// sum (w1-bar . R0) + sum (w-bar^{n+1}_pre . R1 / 2), the two stages' use of dt.
// ---------------------------------------------------------------------------

// Forward wave speed of one face, the forward kernels' arithmetic.
__device__ double face_speed(const AdjMesh &m, double HfL, double HufL, double HvfL, double zL, double HfR,
                             double HufR, double HvfR, double zR, double nx, double ny, bool wall, int bnd)
{
    const double g = m.g, hthr = m.hthr;
    double uL = 0.0, vL = 0.0;
    if (gt_nn(HfL, hthr)) { uL = HufL / HfL; vL = HvfL / HfL; }
    double unL = uL * nx + vL * ny;
    double HsL, HsR, unR;
    if (wall && bnd == 3) {
        HsL = max0((HfL + zL) - zL);
        const double cL = sqrt(g * HsL), c0 = sqrt(g * max0(0.0 - zL));
        const double Rp = unL + 2.0 * cL, Rm = 0.0 - 2.0 * c0;
        unR = 0.5 * (Rp + Rm);
        const double cg = max0(0.25 * (Rp - Rm));
        HsR = cg * cg / g;
    } else if (wall) {
        HsL = max0((HfL + zL) - zL);
        HsR = HsL;
        unR = bnd == 2 ? unL : -unL;
    } else {
        double uR = 0.0, vR = 0.0;
        if (gt_nn(HfR, hthr)) { uR = HufR / HfR; vR = HvfR / HfR; }
        unR = uR * nx + vR * ny;
        double zs = smax(zL, zR);
        HsL = max0((HfL + zL) - zs);
        HsR = max0((HfR + zR) - zs);
    }
    if (is_zero(HsL) && is_zero(HsR)) return 0.0;
    double cL = sqrt(g * HsL), cR = sqrt(g * HsR), sL, sR;
    if (is_zero(HsL)) {
        sL = unR - 2.0 * cR;
        sR = unR + cR;
    } else if (is_zero(HsR)) {
        sL = unL - cL;
        sR = unL + 2.0 * cL;
    } else {
        double us = 0.5 * (unL + unR) + (cL - cR);
        double cs = 0.5 * (cL + cR) - 0.25 * (unR - unL);
        sL = smin(unL - cL, us - cs);
        sR = smax(us + cs, unR + cR);
    }
    return smax(fabs(sL), fabs(sR));
}

// The face states of face f of cell K (and its neighbour across it) from FV.
struct FaceIn {
    double HfL, HufL, HvfL, zL, HfR, HufR, HvfR, zR, nx, ny, l;
    int j, fj;
    bool wall;
    int bnd;                 // boundary kind: 1 wall, 2 open, 3 absorbing (0: interior)
};
__device__ FaceIn face_in(const AdjMesh &m, const double *FV, int K, int f)
{
    const int nc = m.nc;
    FaceIn r;
    r.j = m.nbr[f * nc + K];
    r.wall = r.j < 0;
    r.bnd = r.wall ? -r.j : 0;
    r.fj = r.wall ? 0 : (m.nbrl[f * nc + K] & 3);
    r.HfL = FV[(0 * 3 + f) * (size_t)nc + K];
    r.HufL = FV[(1 * 3 + f) * (size_t)nc + K];
    r.HvfL = FV[(2 * 3 + f) * (size_t)nc + K];
    r.zL = bed_under(m, K, f);
    r.HfR = r.HufR = r.HvfR = r.zR = 0.0;
    if (!r.wall) {
        r.HfR = FV[(0 * 3 + r.fj) * (size_t)nc + r.j];
        r.HufR = FV[(1 * 3 + r.fj) * (size_t)nc + r.j];
        r.HvfR = FV[(2 * 3 + r.fj) * (size_t)nc + r.j];
        r.zR = bed_under(m, r.j, r.fj);
    }
    r.nx = G(m, GEO_NX + f, K);
    r.ny = G(m, GEO_NY + f, K);
    r.l = G(m, GEO_LEN + f, K);
    return r;
}


// dt-bar's face (one CTA): sums the parts of dt-bar, reduces the parts of the search,
// forms the speeds of the chosen cell's faces, finds f* (the first of largest l_f a_f)
// and writes its wave speed's adjoint on both sides to *cfl.out, from where the
// reconstruction VJP adds it.  (A kernel of its own between the flux and the
// reconstruction VJP was 28 us of latency at any size.)
__device__ __noinline__ void cfl_face_vjp(const AdjMesh &m, const double *FV, const AdjCfl &cfl)
{
    __shared__ double s_a[3], s_la[3];
    __shared__ int s_k;
    AdjCflFace *out = cfl.out;
    double s1 = 0.0, s0 = 0.0, bb = INFINITY;
    int bo = 0x7fffffff, K = -1;
    for (int q = threadIdx.x; q < cfl.nparts; q += blockDim.x) {
        s1 += cfl.part_s1[q];
        s0 += cfl.part_s0[q];
        if (cfl.part_k[q] >= 0 && cfl_less(cfl.part_b[q], cfl.part_o[q], bb, bo)) {
            bb = cfl.part_b[q]; bo = cfl.part_o[q]; K = cfl.part_k[q];
        }
    }
    s1 = cta_sum<kVjpThreads>(s1);
    __syncthreads();
    s0 = cta_sum<kVjpThreads>(s0);
    cta_argmin<kVjpThreads>(bb, bo, K);
    if (threadIdx.x == 0) {
        s_k = K;
        out->cell[0] = out->cell[1] = -1;
    }
    __syncthreads();
    K = s_k;
    if (K < 0) return;                                   // nothing moves: dt = dt_max or 0
    if (threadIdx.x < 3) {
        const FaceIn q = face_in(m, FV, K, threadIdx.x);
        const double a = face_speed(m, q.HfL, q.HufL, q.HvfL, q.zL, q.HfR, q.HufR, q.HvfR, q.zR, q.nx, q.ny, q.wall,
                                    q.bnd);
        s_a[threadIdx.x] = a;
        s_la[threadIdx.x] = q.l * a;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    const double dtc = cfl.cfl * bb;
    if (cfl.dt_max > 0.0 && cfl.dt_max < dtc) return;    // clamped by dt_max: no dependence
    int f = 0;
    for (int k = 1; k < 3; k++)
        if (gt_nn(s_la[k], s_la[f])) f = k;
    const FaceIn q = face_in(m, FV, K, f);
    // dt-bar: sum w-bar_pre . R1 / 2 + sum w1-bar_pre . R0 (each Rb . R / dt), and with
    // a moving bed every later bed through the time
    double dtbar = (s1 + s0) / cfl.dt;
    if (cfl.tsum) dtbar += *cfl.tsum;
    const double ab = -dtbar * dtc / s_a[f];
    const double P0[3] = {0.0, 0.0, 0.0};
    double bL[4], bR[4];
    flux_vjp(m, q.HfL, q.HufL, q.HvfL, q.zL, q.HfR, q.HufR, q.HvfR, q.zR, q.nx, q.ny, q.wall, P0, 0.0, 0.0, bL, bR, ab,
             q.bnd);
    for (int k = 0; k < 4; k++) { out->bar[0][k] = bL[k]; out->bar[1][k] = bR[k]; }
    out->face[0] = f;
    out->cell[0] = K;
    if (!q.wall) { out->face[1] = q.fj; out->cell[1] = q.j; }
}

// One thread per face (the face list: the lower-numbered cell owns an interior
// face, the cell a boundary face): R-bar of both cells -> Phi-bar, P-bar ->
// face-state adjoints.  FVb[(v*3+f)*nc + K] and zfb[f*nc + K] are the (cell,
// face) slots; each is written exactly once per residual.
// With CFL steps the launch has one more CTA, which reverses the time step meanwhile.
__global__ void __launch_bounds__(kVjpThreads) adj_flux_vjp_kernel(AdjMesh m, const double *FV, const double *Rb, double *FVb,
                                                                   double *zfb, const AdjCfl cfl)
{
    const int nc = m.nc, ctas = gridDim.x - (cfl.dt ? 1 : 0);
    if ((int)blockIdx.x == ctas) {
        cfl_face_vjp(m, FV, cfl);
        return;
    }
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < m.nfaces; q += ctas * blockDim.x) {
        {
            const int K = m.faces[q] >> 2, f = m.faces[q] & 3;
            int j = m.nbr[f * nc + K];
            bool wall = j < 0;
            int fj = wall ? 0 : (m.nbrl[f * nc + K] & 3);
            if (!rb_nonzero(Rb, nc, K) && (wall || !rb_nonzero(Rb, nc, j))) {
                for (int v = 0; v < 3; v++) FVb[(v * 3 + f) * (size_t)nc + K] = 0.0;
                zfb[f * (size_t)nc + K] = 0.0;
                if (!wall) {
                    for (int v = 0; v < 3; v++) FVb[(v * 3 + fj) * (size_t)nc + j] = 0.0;
                    zfb[fj * (size_t)nc + j] = 0.0;
                }
                continue;
            }
            double nx = G(m, GEO_NX + f, K), ny = G(m, GEO_NY + f, K), l = G(m, GEO_LEN + f, K);
            double cLf = quot(-l, by_area(m, K));
            double Pb[3], PLb, PRb = 0.0;
            double RLH = Rb[K], RLU = Rb[nc + K], RLV = Rb[2 * (size_t)nc + K];
            Pb[0] = cLf * RLH;
            Pb[1] = cLf * RLU;
            Pb[2] = cLf * RLV;
            PLb = cLf * (RLU * nx + RLV * ny);
            double HfR = 0.0, HufR = 0.0, HvfR = 0.0, zR = 0.0;
            if (!wall) {
                double cRf = quot(l, by_area(m, j));
                double RRH = Rb[j], RRU = Rb[nc + j], RRV = Rb[2 * (size_t)nc + j];
                Pb[0] += cRf * RRH;
                Pb[1] += cRf * RRU;
                Pb[2] += cRf * RRV;
                PRb = cRf * (RRU * nx + RRV * ny);
                HfR = FV[(0 * 3 + fj) * (size_t)nc + j];
                HufR = FV[(1 * 3 + fj) * (size_t)nc + j];
                HvfR = FV[(2 * 3 + fj) * (size_t)nc + j];
                zR = bed_under(m, j, fj);
            }
            double bL[4], bR[4];
            flux_vjp(m, FV[(0 * 3 + f) * (size_t)nc + K], FV[(1 * 3 + f) * (size_t)nc + K],
                     FV[(2 * 3 + f) * (size_t)nc + K], bed_under(m, K, f), HfR, HufR, HvfR, zR, nx, ny, wall, Pb, PLb,
                     PRb, bL, bR, 0.0, wall ? -j : 0);
            for (int v = 0; v < 3; v++) FVb[(v * 3 + f) * (size_t)nc + K] = bL[v];
            zfb[f * (size_t)nc + K] = bL[3];
            if (!wall) {
                for (int v = 0; v < 3; v++) FVb[(v * 3 + fj) * (size_t)nc + j] = bR[v];
                zfb[fj * (size_t)nc + j] = bR[3];
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Moving bed: the beds of step n are z_K(t_n) = -(1/3) sum_{v in K} d_v(t_n) and
// z_f(t_n) = -(1/2) sum_{v on f} d_v(t_n), d_v(t) = depth0_v - uplift_v R((t -
// onset_v) / rise).  With zs the adjoints of that step's beds (its residuals
// and gauge record; row 0 cell beds, rows 1..3 face beds), per vertex
// s_v = sum over the cells K around v of zs_K / 3 + (zs of K's two faces at v) / 2,
// in a fixed order, and
//   uplift-bar_v += s_v R,   onset-bar_v += -s_v uplift_v R',
//   t-bar_n = sum_v s_v uplift_v R'      (R' = dR/dt = 1 / rise inside the ramp),
// the last summed per CTA into part (adaptive steps carry it to every earlier dt).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kRedThreads) adj_bed_vertex_kernel(int nv, int ncs, const int32_t *vptr, const int32_t *vcell, const double *zs,
                                      const double *uplift, const double *onset, double rise, double t, double *gU,
                                      double *gOn, double *part)
{
    double tb = 0.0;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < nv; v += gridDim.x * blockDim.x) {
        double sv = 0.0;
        for (int k = vptr[v]; k < vptr[v + 1]; k++) {
            const int K = vcell[k] >> 2, j = vcell[k] & 3;
            // faces j (vertices j, j+1) and j+2 (vertices j+2, j) of K touch vertex j
            sv += zs[K] / 3.0 + (zs[(size_t)(1 + j) * ncs + K] + zs[(size_t)(1 + (j + 2) % 3) * ncs + K]) / 2.0;
        }
        double R, Rp = 0.0;
        if (rise > 0.0) {
            const double x = __dsub_rn(t, onset[v]) / rise;
            R = fmin(1.0, fmax(0.0, x));
            if (x > 0.0 && x < 1.0) Rp = 1.0 / rise;
        } else {
            R = t >= onset[v] ? 1.0 : 0.0;
        }
        gU[v] += sv * R;
        const double q = sv * uplift[v] * Rp;
        gOn[v] -= q;
        tb += q;
    }
    tb = cta_sum<kRedThreads>(tb);
    if (threadIdx.x == 0) part[blockIdx.x] = tb;
}

// *acc += the sum of nparts partial sums.
__global__ void __launch_bounds__(kRedThreads) adj_sum_parts_kernel(int nparts, const double *part, double *acc)
{
    double s = 0.0;
    for (int q = threadIdx.x; q < nparts; q += blockDim.x) s += part[q];
    s = cta_sum<kRedThreads>(s);
    if (threadIdx.x == 0) *acc += s;
}

__global__ void adj_axpy_kernel(int64_t n, const double *x, double *y)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] += x[i];
}

// CTAs of a reduction over n values: at least four values a thread, at most
// kAdjCflParts parts.
int grid_red(int64_t n)
{
    const int64_t g = (n + 4 * kRedThreads - 1) / (4 * kRedThreads);
    return (int)(g < 1 ? 1 : g < kAdjCflParts ? g : kAdjCflParts);
}
int grid_of(int n) { return (n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096; }
int grid_vjp(int n) { return (n + kVjpThreads - 1) / kVjpThreads < 8192 ? (n + kVjpThreads - 1) / kVjpThreads : 8192; }

AdjMesh adj_mesh(const DevPtrs &d, const StepParams &p)
{
    AdjMesh m;
    m.nc = (int)d.nc;
    m.order = p.order;
    m.geo = static_cast<const double *>(d.geo);
    m.rarea = d.rarea;
    m.z = static_cast<const double *>(d.z);
    m.zf = static_cast<const double *>(d.zf);
    m.rec = nullptr;
    m.nbr = d.nbr;
    m.nbrl = d.nbrl;
    m.faces = d.adj_faces;
    m.nfaces = (int)d.n_adj_faces;
    m.g = p.g;
    m.half_g = 0.5 * p.g;
    m.hthr = p.hthr;
    return m;
}

}  // namespace

// CTAs of the per-cell kernels that also reduce.
static int grid_cells(int nc) { const int g = (nc + kRedThreads - 1) / kRedThreads; return g < kAdjCflParts ? g : kAdjCflParts; }

// The reverse of one step (see the top of this file).
int adjoint_step(const DevPtrs &d, const StepParams &p, const AdjStep &a, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    AdjMesh m = adj_mesh(d, p);
    if (!m.faces) return (int)cudaErrorInvalidValue;     // the face list is built by vg_adj_backward
    const int nc = m.nc, cells = grid_cells(nc), vjp_cells = grid_vjp(nc), vjp_faces = grid_vjp(m.nfaces);
    AdjCfl cfl = a.cfl, none{};
    cfl.nparts = cells;
    adj_begin_kernel<<<cells, kRedThreads, 0, s>>>(nc, a.dt, p.hthr, a.w, a.R0, a.w1, a.H1pre, a.mask2, a.wb, a.wbn, a.wb1, a.Rb,
                                                   cfl);
    m.rec = a.rec1;
    adj_flux_vjp_kernel<<<vjp_faces, kVjpThreads, 0, s>>>(m, a.FV1, a.Rb, a.FVb, a.zfb, none);
    adj_recon_vjp_kernel<<<vjp_cells, kVjpThreads, 0, s>>>(m, a.w1, a.Rb, a.FVb, a.zfb, a.own, a.send, nullptr);
    adj_gather_mid_kernel<<<cells, kRedThreads, 0, s>>>(m, a.own, a.send, a.zb, a.dt, p.hthr, a.H1pre, a.wb1, a.wbn, a.Rb, cfl);
    m.rec = a.rec0;
    adj_flux_vjp_kernel<<<vjp_faces + (cfl.dt ? 1 : 0), kVjpThreads, 0, s>>>(m, a.FV0, a.Rb, a.FVb, a.zfb, cfl);
    adj_recon_vjp_kernel<<<vjp_cells, kVjpThreads, 0, s>>>(m, a.w, a.Rb, a.FVb, a.zfb, a.own, a.send, cfl.dt ? cfl.out : nullptr);
    adj_gather_kernel<<<grid_of(nc), 256, 0, s>>>(m, a.own, a.send, a.wbn, a.zb);
    return (int)cudaGetLastError();
}

int adjoint_bed_flush(int nc, int nv, const int32_t *vptr, const int32_t *vcell, double *zs, const double *uplift,
                      const double *onset, double rise, double t, double *gU, double *gOn, double *zb_total,
                      double *tsum, double *part, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int parts = grid_red(nv);
    adj_bed_vertex_kernel<<<parts, kRedThreads, 0, s>>>(nv, nc, vptr, vcell, zs, uplift, onset, rise, t, gU, gOn, part);
    adj_sum_parts_kernel<<<1, kRedThreads, 0, s>>>(parts, part, tsum);
    adj_axpy_kernel<<<grid_of(4 * nc), 256, 0, s>>>(4 * (int64_t)nc, zs, zb_total);
    return (int)cudaGetLastError();
}

int adjoint_gauge(int n_gauges, const int32_t *cells, const double *weights, double *wb, double *zb, void *stream)
{
    adj_gauge_kernel<<<(n_gauges + 63) / 64, 64, 0, static_cast<cudaStream_t>(stream)>>>(n_gauges, cells, weights, wb, zb);
    return (int)cudaGetLastError();
}

}  // namespace vg
