// One block of cells of a stage in FP32 (deviation form).  Included by
// step_kernels.cuh, which describes the step, the blocks with their two-ring
// halos and the phases A-D; this file holds the FP32 layout and phases.
//
// The state is (eta, Hu, Hv) with eta = H + z, and the momentum flux through each
// face is carried relative to the hydrostatic pressure g (eta_K - z_{K,f})^2 / 2 of
// the cell's own free surface over the bed z_{K,f} under its face value.  Summed
// over a closed triangle these references give exactly the centred bed-slope
// source of a cell standing on its face beds (and zero for a cell on its flat cell
// bed), so the scheme is unchanged; but the large terms g H^2 / 2 (1e8 in a 4000 m
// ocean) never appear, only products of small differences (eta_f - eta_K, z* - z_K),
// so still water stays still in FP32 and eta keeps full FP32 resolution.
//
// What bounds it: latency.  4M triangles: 50 % of issue slots busy at 37 resident warps
// per SM, DRAM at 44 %; warps wait for halo states and records (7.5 cycles an issue) and
// at the barriers between the phases (4.6).  The layout is the one with the fewest
// instructions and shared or global accesses per cell (the former one, separate arrays,
// was at 58-60 % of the issue slots with 40 % more instructions):
//   state   float4 per cell (eta, Hu, Hv, z): one 16-byte load per block or halo
//           cell and one 16-byte shared slot, where separate arrays took four loads
//           with an address each and touched four sectors per halo cell
//   R0      float4 per cell (the fourth word unused)
//   recA    8 floats per cell, one 32-byte sector: M00 M01 M02 M10 M11 M12 dz0 dz1,
//           all that a reconstruction reads (ring-1 cells included)
//   recB    float4 per cell: N0x N0y N1x N1y, the outward normals of faces 0 and 1
//           times their lengths (face 2: minus their sum, the triangle is closed)
//   codes   four uint16 per cell: the three neighbours' local slots (a boundary face:
//           the cell's own slot, whose values are the open ghost's) and one bit per
//           wall face
//   fr      float4 per owned face of a block: unit normal, length, and the face's two
//           shared-memory slots; the face's left cell is the one of lower internal
//           id whatever block computes it, so results do not depend on the partition
//           (on a moving bed, face_terms_by_side, they do)
// with M_fj = w_j . (x_f - x_K) in FP64 on the host: D_f = sum_j M_fj (q_j - q_K) is
// grad q . (x_f - x_K) for the least-squares gradient, and since the face midpoints
// average to the centroid D_2 = -(D_0 + D_1), dz_2 = -(dz_0 + dz_1).
#pragma once

namespace vg {

template <>
struct KArgs<float> {
    int64_t nc;
    int block, nblocks, max_halo, max_ring1, order;
    const float4 *recA;     // [nc][2]
    const float4 *recB;     // [nc]
    const float *area;      // [nc]
    const uint2 *codes;     // [nc]
    const int32_t *halo_ptr;  // [nblocks + 1]
    const int32_t *halo_n1;   // [nblocks] ring-1 count
    const int32_t *halo_ids;  // per block: ring 1 then ring 2
    const uint2 *ring_codes;  // beside halo_ids: codes of the ring-1 cells
    const int32_t *fr_ptr;  // [nblocks + 1] into fr
    const float4 *fr;       // owned faces of each block, interior faces first
    const float2 *normals;  // moving bed: [3][nc] unit normals of every cell's faces
    int max_faces;          // owned faces of a block at most
    const float *w_soa;     // SOA kernels: w^n [3][nc] and w^{n+1} [3][nc] of the caller, the bed [nc]
    float *wout_soa;
    const float *z;
    const float4 *w;        // w^n [nc]
    float4 *R0;             // [nc]
    float4 *wout;           // w^{n+1} [nc] (stage 2)
    DevScalars *sc;
    float g, half_g, hthr;
    double cfl, dt_fixed, dt_max;
    int cfl_min;            // stage 1: 1 adds the CFL bound to the step's minimum
};

// Approximate reciprocal (PTX rcp.approx.ftz.f32, max error 1 ulp); rcp(0) = +inf.
__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The roundings are written out (fused where fma is written, never elsewhere), so
// that every kernel these functions are inlined into -- single-scenario, batched,
// unfused, no-allocation -- gives the same bits.
__device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float sub_(float a, float b) { return __fsub_rn(a, b); }

// L1 prefetch (a hint: nothing waits for it and it holds no register).
__device__ __forceinline__ void prefetch_l1(const void *ptr)
{
    asm volatile("prefetch.global.L1 [%0];" :: "l"(ptr));
}

// Stored state (eta, Hu, Hv, z) of cell gid.
template <bool SOA>
__device__ __forceinline__ float4 load_w(const KArgs<float> &a, int gid)
{
    if constexpr (SOA) {
        const int nc = (int)a.nc;
        return make_float4(a.w_soa[gid], a.w_soa[nc + gid], a.w_soa[2 * nc + gid], a.z[gid]);
    } else {
        return a.w[gid];
    }
}

// w1 = w + dt R0 of one cell with the dry fix (negative depth emptied; at or below
// the threshold, momentum zeroed).  Returns true if a negative depth was met.
__device__ __forceinline__ bool rk_first(float4 &q, float4 r, float dt, float hthr)
{
    q.x = fma_(dt, r.x, q.x);
    q.y = fma_(dt, r.y, q.y);
    q.z = fma_(dt, r.z, q.z);
    const float H = sub_(q.x, q.w);
    if (H < 0.f) {
        q.x = q.w; q.y = 0.f; q.z = 0.f;
        return true;
    }
    if (!(H > hthr)) { q.y = 0.f; q.z = 0.f; }
    return false;
}

// SSP-RK(2,2) second stage (Sec. 2.3) of one cell: w^{n+1} = w^n / 2 + (w1 + dt R(w1)) / 2
// and the dry fix.  Returns true if a negative depth was met.
__device__ __forceinline__ bool rk_second(float4 x, float4 w1, float RH, float RHu, float RHv, float dt, float hthr,
                                          float4 &o)
{
    o.x = fma_(0.5f, fma_(dt, RH, w1.x), mul_(0.5f, x.x));
    o.y = fma_(0.5f, fma_(dt, RHu, w1.y), mul_(0.5f, x.y));
    o.z = fma_(0.5f, fma_(dt, RHv, w1.z), mul_(0.5f, x.z));
    o.w = w1.w;
    const float H = sub_(o.x, o.w);
    if (H < 0.f) {
        o.x = o.w; o.y = 0.f; o.z = 0.f;
        return true;
    }
    if (!(H > hthr)) { o.y = 0.f; o.z = 0.f; }
    return false;
}

// Cell gid as seen by the stage: w^n, or w1.
template <int STAGE, bool SOA>
__device__ __forceinline__ bool stage_cell(const KArgs<float> &a, int gid, float dt, float4 &q)
{
    q = load_w<SOA>(a, gid);
    if (STAGE == 1) return false;
    return rk_first(q, a.R0[gid], dt, a.hthr);
}

__device__ __forceinline__ bool exactly_dry(float4 q) { return q.x == q.w && q.y == 0.f && q.z == 0.f; }

// Phase D's end for cell gid: R = (RH, RHu, RHv); stage 1 writes R0 and the CFL
// bound of am = max_f l_f a_f, stage 2 w^{n+1} (w1 from shared memory).
template <int STAGE, bool SOA>
__device__ __forceinline__ void finish_cell(const KArgs<float> &a, int gid, const float4 *sWl, float RH, float RHu,
                                            float RHv, float am, float area, float dt, float &my_min,
                                            long long &my_neg, bool &bad)
{
    if (STAGE == 1) {
        a.R0[gid] = make_float4(RH, RHu, RHv, 0.f);
        if (am > 0.f) my_min = fminf(my_min, area / mul_(3.f, am));
    } else {
        float4 o;
        if (rk_second(load_w<SOA>(a, gid), *sWl, RH, RHu, RHv, dt, a.hthr, o)) my_neg++;
        if (!isfinite(o.x) || !isfinite(o.y) || !isfinite(o.z)) bad = true;
        if constexpr (SOA) {
            const int nc = (int)a.nc;
            a.wout_soa[gid] = o.x;
            a.wout_soa[nc + gid] = o.y;
            a.wout_soa[2 * nc + gid] = o.z;
        } else {
            a.wout[gid] = o;
        }
    }
}

// Flux through one face in the deviation form, between the face values L and R
// (eta_f, z under the face value, Hu_f, Hv_f) with unit normal (nx, ny) from L to R
// and length len, and each side's term of the residual's sum:
//   d* = H*_L - H*_R          (eta_fL - eta_fR when both sides are wet)
//   F1 - C_e for C_e = g H*_L H*_R / 2:  L: q_L u_nL + p_L, R: q_R u_nR - p_R with
//   p_s = g H*_s d* / 2       (HLL is affine in F with weights summing to one, so F*
//                              shifts by -C_e)
//   L:  l [F0, (F1 - p_L) n_x - F2 n_y, ...],  R: minus l [F0, (F1 + p_R) n_x - F2 n_y, ...]
// The part of the pressure correction that holds one cell's own values only,
// g/2 (eta_f - eta_K)(H_f + H_K), is summed by that cell in phase B.
// bnd: 0 interior; 1 wall, the ghost of Sec. 2.5; 2 open, the transmissive ghost;
// 3 absorbing, the characteristic ghost of a sea at rest (R is then not read).
// HLL runs with the speeds clamped to a <= 0 <= b, which also gives F_L when
// s_L >= 0 and F_R when s_R <= 0 (b - a > 0 unless both sides are dry).
__device__ __forceinline__ void face_terms(float g, float half_g, float hthr, float4 L, float4 R, float nx, float ny,
                                           float len, int bnd, float4 &tL, float4 &tR)
{
    const float HfL = sub_(L.x, L.y);
    const float rL = HfL > hthr ? rcp_approx(HfL) : 0.f;
    const float unL = mul_(fma_(L.w, ny, mul_(L.z, nx)), rL);
    const float utL = mul_(fma_(L.w, nx, -mul_(L.z, ny)), rL);
    float HsL, HsR, unR, utR, ds;
    if (bnd == 0) {
        const float HfR = sub_(R.x, R.y);
        const float rR = HfR > hthr ? rcp_approx(HfR) : 0.f;
        unR = mul_(fma_(R.w, ny, mul_(R.z, nx)), rR);
        utR = mul_(fma_(R.w, nx, -mul_(R.z, ny)), rR);
        const float zs = fmaxf(L.y, R.y);
        HsL = fmaxf(0.f, sub_(L.x, zs));
        HsR = fmaxf(0.f, sub_(R.x, zs));
        ds = (HsL > 0.f && HsR > 0.f) ? sub_(L.x, R.x) : sub_(HsL, HsR);
    } else {
        HsL = fmaxf(0.f, HfL);
        utR = utL;
        if (bnd == 3) {
            // the outgoing invariant u_n + 2c of the face state and the incoming
            // u_n - 2c of the sea at rest (eta = 0) beyond the boundary
            const float cL = sqrtf(mul_(g, HsL)), c0 = sqrtf(mul_(g, fmaxf(0.f, -L.y)));
            const float Rp = fma_(2.f, cL, unL), Rm = -2.f * c0;
            const float cg = fmaxf(0.f, mul_(0.25f, sub_(Rp, Rm)));
            unR = mul_(0.5f, add_(Rp, Rm));
            HsR = mul_(cg, cg) / g;
            ds = sub_(HsL, HsR);
        } else {
            HsR = HsL;
            unR = bnd == 2 ? unL : -unL;
            ds = 0.f;
        }
    }
    if (HsL == 0.f && HsR == 0.f) {
        tL = tR = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const float cL = sqrtf(mul_(g, HsL)), cR = sqrtf(mul_(g, HsR));
    float sL, sR;
    if (HsL == 0.f) {
        sL = fma_(-2.f, cR, unR);
        sR = add_(unR, cR);
    } else if (HsR == 0.f) {
        sL = sub_(unL, cL);
        sR = fma_(2.f, cL, unL);
    } else {
        const float us = fma_(0.5f, add_(unL, unR), sub_(cL, cR));
        const float cs = fma_(0.5f, add_(cL, cR), mul_(-0.25f, sub_(unR, unL)));
        sL = fminf(sub_(unL, cL), sub_(us, cs));
        sR = fmaxf(add_(us, cs), add_(unR, cR));
    }
    const float qL = mul_(HsL, unL), qR = mul_(HsR, unR);
    const float hd = mul_(half_g, ds), pL = mul_(HsL, hd), pR = mul_(HsR, hd);
    const float FL1 = fma_(qL, unL, pL), FR1 = fma_(qR, unR, -pR);
    const float a = fminf(sL, 0.f), b = fmaxf(sR, 0.f);
    const float rden = rcp_approx(sub_(b, a)), ab = mul_(a, b);
    const float vL = mul_(HsL, utL), vR = mul_(HsR, utR);
    const float F0 = mul_(fma_(-ab, ds, fma_(b, qL, -mul_(a, qR))), rden);
    const float F1 = mul_(fma_(ab, sub_(qR, qL), fma_(b, FL1, -mul_(a, FR1))), rden);
    const float F2 = mul_(fma_(ab, sub_(vR, vL), fma_(b, mul_(vL, unL), -mul_(a, mul_(vR, unR)))), rden);
    const float lx = mul_(len, nx), ly = mul_(len, ny);
    const float mL = sub_(F1, pL), mR = add_(F1, pR), vx = mul_(F2, ly), vy = mul_(F2, lx);
    const float t0 = mul_(len, F0), la = mul_(len, fmaxf(fabsf(sL), fabsf(sR)));
    tL = make_float4(t0, fma_(mL, lx, -vx), fma_(mL, ly, vy), la);
    tR = make_float4(-t0, fma_(-mR, lx, vx), -fma_(mR, ly, vy), la);
}

// Limited face values of one variable, q + alpha D_f, from the cell's value q and the
// neighbours' values: differences d, increments D_f, and
// alpha = min(1, min_f r_f / |D_f|) with r_f = max(0, d_j) or max(0, -d_j) by the sign
// of D_f (Barth-Jespersen).  The smallest ratio of a sign is that of its largest
// |D_f|, so two reciprocals serve the three faces; the D_f sum to zero, so both
// maxima are >= 0, and rcp(0) = +inf gives +inf or NaN, which fminf ignores.
__device__ __forceinline__ void limited(const float4 m0, const float4 m1, float q, float q0, float q1, float q2, float D[3])
{
    const float d0 = sub_(q0, q), d1 = sub_(q1, q), d2 = sub_(q2, q);
    D[0] = fma_(m0.x, d0, fma_(m0.y, d1, mul_(m0.z, d2)));
    D[1] = fma_(m0.w, d0, fma_(m1.x, d1, mul_(m1.y, d2)));
    D[2] = -add_(D[0], D[1]);
    const float up = fmaxf(fmaxf(d0, d1), fmaxf(d2, 0.f)), dn = -fminf(fminf(d0, d1), fminf(d2, 0.f));
    const float P = fabsf(fmaxf(fmaxf(D[0], D[1]), D[2])), M = fabsf(fminf(fminf(D[0], D[1]), D[2]));   // never -0
    const float alpha = fminf(fminf(1.f, mul_(up, rcp_approx(P))), mul_(dn, rcp_approx(M)));
    D[0] = fma_(alpha, D[0], q);
    D[1] = fma_(alpha, D[1], q);
    D[2] = fma_(alpha, D[2], q);
}

// ---------------------------------------------------------------------------
// The form of a moving bed: pressure terms per face side, the limiter's ratios one by
// one, a face's left cell the one whose block computes it.  The same scheme; only the
// roundings differ.  A moving bed keeps them because its update is no continuous
// function of the state: the free surface of a moving cell is rounded to the bed's grid
// (2.4e-4 m over 4000 m of water) in every step, so that one ulp of dt, which another
// order of these sums changes now and then, decides many of those roundings: momenta
// off by 3e-5 of their norm and 2e-3 at most (298k cells, 40 steps; 2 of 24 sources).
// With this form a run repeats those of the kernels before the 16-byte states bit for
// bit, as static beds, which have no such switch, need not.  The expressions are left
// to the compiler's contraction, as they were there.  Not slower: 298k cells, 40 steps
// 1.76 ms, 1.79 to 1.81 with the form of a static bed (its two kernels spill a little,
// these do not).
// ---------------------------------------------------------------------------

// Limited face values of one variable from the cell's value q and the neighbours' qn.
__device__ __forceinline__ void limited_by_face(const float4 m0, const float4 m1, float q, float qn0, float qn1, float qn2,
                                                float face[3])
{
    const float d0 = qn0 - q, d1 = qn1 - q, d2 = qn2 - q;
    float D[3];
    D[0] = m0.x * d0 + m0.y * d1 + m0.z * d2;
    D[1] = m0.w * d0 + m1.x * d1 + m1.y * d2;
    D[2] = -(D[0] + D[1]);
    const float up = fmaxf(fmaxf(fmaxf(q, qn0), qn1), qn2) - q, dn = q - fminf(fminf(fminf(q, qn0), qn1), qn2);
    float alpha = 1.f;
#pragma unroll
    for (int f = 0; f < 3; f++) alpha = fminf(alpha, (D[f] > 0.f ? up : dn) * rcp_approx(fabsf(D[f])));
#pragma unroll
    for (int f = 0; f < 3; f++) face[f] = q + alpha * D[f];
}

// Flux and side terms of one face, arguments as face_terms and the cells' own eta:
//   Q_L = g/2 [(eta_fL - eta_L)(H_fL + H_L) - H*_L d*],
//   Q_R = g/2 [(eta_fR - eta_R)(H_fR + H_R) + H*_R d*].
__device__ __forceinline__ void face_terms_by_side(float g, float half_g, float hthr, float4 L, float eL, float4 R, float eR,
                                                   float nx, float ny, float len, int bnd, float4 &tL, float4 &tR)
{
    const float efL = L.x, zL = L.y, HufL = L.z, HvfL = L.w;
    float efR = R.x, zR = R.y;
    const float HufR = R.z, HvfR = R.w;
    float HfL = efL - zL;
    float uL = 0.f, vL = 0.f;
    if (HfL > hthr) { const float r = rcp_approx(HfL); uL = HufL * r; vL = HvfL * r; }
    float unL = uL * nx + vL * ny;
    float utL = -uL * ny + vL * nx;
    float HsL, HsR, unR, utR, ds, HfR;
    if (bnd == 3) {
        HsL = fmaxf(0.f, HfL);
        const float cL = sqrtf(g * HsL), c0 = sqrtf(g * fmaxf(0.f, -zL));
        const float Rp = unL + 2.f * cL, Rm = -2.f * c0;
        const float cg = fmaxf(0.f, 0.25f * (Rp - Rm));
        unR = 0.5f * (Rp + Rm);
        HsR = cg * cg / g;
        utR = utL;
        ds = HsL - HsR;
        HfR = HsR; efR = zL + HsR; eR = efR; zR = zL;
    } else if (bnd) {
        HsL = fmaxf(0.f, HfL);
        HsR = HsL;
        unR = bnd == 2 ? unL : -unL;
        utR = utL;
        ds = 0.f;
        HfR = HfL; efR = efL; eR = eL; zR = zL;
    } else {
        HfR = efR - zR;
        float uR = 0.f, vR = 0.f;
        if (HfR > hthr) { const float r = rcp_approx(HfR); uR = HufR * r; vR = HvfR * r; }
        unR = uR * nx + vR * ny;
        utR = -uR * ny + vR * nx;
        float zs = fmaxf(zL, zR);
        HsL = fmaxf(0.f, efL - zs);
        HsR = fmaxf(0.f, efR - zs);
        ds = (HsL > 0.f && HsR > 0.f) ? efL - efR : HsL - HsR;
    }
    float F[3], amax;
    if (HsL == 0.f && HsR == 0.f) {
        F[0] = 0.f; F[1] = 0.f; F[2] = 0.f;
        amax = 0.f;
    } else {
        float cL = sqrtf(g * HsL), cR = sqrtf(g * HsR);
        float sL, sR;
        if (HsL == 0.f) {
            sL = unR - 2.f * cR;
            sR = unR + cR;
        } else if (HsR == 0.f) {
            sL = unL - cL;
            sR = unL + 2.f * cL;
        } else {
            float us = 0.5f * (unL + unR) + (cL - cR);
            float cs = 0.5f * (cL + cR) - 0.25f * (unR - unL);
            sL = fminf(unL - cL, us - cs);
            sR = fmaxf(us + cs, unR + cR);
        }
        float qL = HsL * unL, qR = HsR * unR;
        float FL0 = qL, FL1 = qL * unL + half_g * HsL * ds, FL2 = qL * utL;
        float FR0 = qR, FR1 = qR * unR - half_g * HsR * ds, FR2 = qR * utR;
        const float a = fminf(sL, 0.f), b = fmaxf(sR, 0.f);
        const float rden = rcp_approx(b - a), ab = a * b;
        F[0] = ((b * FL0 - a * FR0) - ab * ds) * rden;
        F[1] = ((b * FL1 - a * FR1) + ab * (qR - qL)) * rden;
        F[2] = ((b * FL2 - a * FR2) + ab * (HsR * utR - HsL * utL)) * rden;
        amax = fmaxf(fabsf(sL), fabsf(sR));
    }
    const float P0 = F[0], P1 = F[1] * nx - F[2] * ny, P2 = F[1] * ny + F[2] * nx;
    float HL = eL - zL, HR = eR - zR;
    const float QL = half_g * ((efL - eL) * (HfL + HL) - HsL * ds);
    const float QR = half_g * ((efR - eR) * (HfR + HR) + HsR * ds);
    const float t0 = len * P0, la = len * amax;
    tL = make_float4(t0, len * (P1 + QL * nx), len * (P2 + QL * ny), la);
    tR = make_float4(-t0, -(len * (P1 + QR * nx)), -(len * (P2 + QR * ny)), la);
}

// The wall ghost's momentum for a wall face of normal N (any length): m - 2 (m.n) n.
__device__ __forceinline__ void wall_ghost(float4 &q, float Nx, float Ny)
{
    const float s = mul_(2.f, fma_(q.y, Nx, mul_(q.z, Ny))) / fma_(Nx, Nx, mul_(Ny, Ny));
    q.y = fma_(-s, Nx, q.y);
    q.z = fma_(-s, Ny, q.z);
}

template <>
__host__ __device__ inline size_t stage_smem_bytes<float>(int block, int max_halo, int max_ring1, int max_faces, bool)
{
    const size_t L = (size_t)block + max_halo, L1 = (size_t)block + max_ring1;
    return 16 * (L + 3 * L1 + max_faces) + 12 * (size_t)block + 4 * (size_t)max_halo + 32;
}

// What phase B reads from global memory for a wet cell, on its way into L1.
__device__ __forceinline__ void prefetch_block_cell(const KArgs<float> &a, int gid)
{
    prefetch_l1(a.recA + 2 * gid);
    prefetch_l1(a.recB + gid);
    prefetch_l1(a.codes + gid);
}
__device__ __forceinline__ void prefetch_ring_cell(const KArgs<float> &a, int gid, int at)
{
    prefetch_l1(a.recA + 2 * gid);
    prefetch_l1(a.ring_codes + at);
}

// 16 bytes global -> shared without a register, completed by cp_wait (and, for other
// threads, a barrier behind it).
__device__ __forceinline__ void cp16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                 :: "r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Shared memory of one CTA, all but the last four of 16 bytes: cell states [L], face
// slots [3][L1] (L = block + halo, L1 = block + ring 1), the block's face records,
// phase B's own sums (8 bytes) and areas (4 bytes) of the block cells, the halo's ids
// and the block's counts (kept for a next time, KEEP).
struct Smem {
    float4 *sW, *sF, *sFr;
    float2 *sS;
    float *sArea;
    int32_t *sHid;
    int *sMeta;
    int L1;
};
__device__ __forceinline__ Smem smem_of(const KArgs<float> &a, unsigned char *raw)
{
    Smem m;
    m.L1 = a.block + a.max_ring1;
    m.sW = reinterpret_cast<float4 *>(raw);
    m.sF = m.sW + (a.block + a.max_halo);
    m.sFr = m.sF + 3 * m.L1;
    m.sS = reinterpret_cast<float2 *>(m.sFr + a.max_faces);
    m.sArea = reinterpret_cast<float *>(m.sS + a.block);
    m.sHid = reinterpret_cast<int32_t *>(m.sArea + a.block);
    m.sMeta = m.sHid + a.max_halo;
    return m;
}
// One block for one scenario: phases A-D.  my_min collects the thread's stage-1 CFL
// bound, my_neg its negative-depth events, bad a non-finite result.  Every thread of
// the CTA must call it.  There is no barrier after phase D: its thread reads only its
// own cell's slots, the next block's phase A writes slots of its own cells only, and
// face slots and records are next written behind the barrier that ends phase A.
//
// sW[l] = state of local cell l as the stage sees it; sF[f L1 + l] = (eta_f, z_f,
// Hu_f, Hv_f) of face f of cell l after phase B, z_f the bed the face value stands on,
// and after phase C the cell's own term (three sums, l_f a_f); sS[l] = phase B's own
// part of the momentum sums.
//
// loaded: the block's areas and face records are in shared memory already, and with
// KEEP its counts and halo ids: a batch's later scenarios of the same block (their
// records of cells come from L1), or the later steps of a CTA with one block (behind a
// grid barrier, which empties L1).  The halo's states then wait for one load, not for
// three in a row (8.7k cells 9.8 -> 9.0 us a step, 99k 14.5 -> 13.5; 32 coast
// scenarios 215 -> 210).
enum { KEEP_NOTHING, KEEP_SCENARIOS, KEEP_STEPS };
template <int STAGE, bool SOA, int KEEP, bool MOVING = false>
__device__ __forceinline__ void process_block(const KArgs<float> &a, const int b, const float dt,
                                              unsigned char *smem_raw, float &my_min, long long &my_neg, bool &bad,
                                              bool &loaded)
{
    const int B = a.block, tid = threadIdx.x;
    const Smem m = smem_of(a, smem_raw);
    const int c0 = b * B;
    const int ncell = min(B, (int)a.nc - c0);
    int h0, nh, n1, q0, nq;
    if (KEEP && loaded) {
        h0 = m.sMeta[0];
        nh = m.sMeta[1];
        n1 = m.sMeta[2];
        nq = m.sMeta[3];
        q0 = 0;
    } else {
        h0 = a.halo_ptr[b];
        nh = a.halo_ptr[b + 1] - h0;
        n1 = a.halo_n1[b];
        q0 = a.fr_ptr[b];
        nq = a.fr_ptr[b + 1] - q0;
        if (KEEP && tid == 0) {
            m.sMeta[0] = h0;
            m.sMeta[1] = nh;
            m.sMeta[2] = n1;
            m.sMeta[3] = nq;
        }
    }
    auto halo_id = [&](int h) {
        if (KEEP && loaded) return m.sHid[h];
        const int32_t id = a.halo_ids[h0 + h];
        if (KEEP) m.sHid[h] = id;
        return id;
    };

    // A: states of the block and its halo, and the areas that phase D divides by
    bool dry = true;
    {
        int gh = -1;
        if (tid < nh) gh = halo_id(tid);
        if (tid < ncell) {
            const int gid = c0 + tid;
            float area = 0.f;
            if (!loaded) area = a.area[gid];
            float4 q = load_w<SOA>(a, gid);
            if (STAGE == 2 && rk_first(q, a.R0[gid], dt, a.hthr)) my_neg++;
            if ((!loaded || KEEP == KEEP_STEPS) && q.x - q.w > a.hthr) prefetch_block_cell(a, gid);
            if (!loaded) m.sArea[tid] = area;
            m.sW[tid] = q;
            dry = exactly_dry(q);
        }
        for (int h = tid; h < nh; h += blockDim.x) {
            if (h != tid) gh = halo_id(h);
            float4 q = load_w<SOA>(a, gh);
            if (STAGE == 2) rk_first(q, a.R0[gh], dt, a.hthr);
            if (h < n1) {
                if ((!loaded || KEEP == KEEP_STEPS) && q.x - q.w > a.hthr) prefetch_ring_cell(a, gh, h0 + h);
                dry = dry && exactly_dry(q);
            }
            m.sW[B + h] = q;
        }
    }
    // Dry land: when the block's cells and its ring 1 are exactly dry, every face of
    // the block has two dry sides, hence no flux and no pressure term.
    if (__syncthreads_and(dry)) {
        if (tid < ncell)
            finish_cell<STAGE, SOA>(a, c0 + tid, m.sW + tid, -0.f, -0.f, -0.f, 0.f, 1.f, dt, my_min, my_neg, bad);
        return;
    }
    // phase C's face records, on their way into shared memory during phase B
    if (!loaded)
        for (int q = tid; q < nq; q += blockDim.x) cp16(m.sFr + q, a.fr + q0 + q);
    loaded = true;

    // B: face values of block + ring-1 cells (Sec. 2.4, Eq. recon with the
    // Barth-Jespersen limiter); every neighbour is in shared memory
    for (int l = tid; l < B + n1; l += blockDim.x) {
        if (l < B && l >= ncell) continue;
        const float4 q = m.sW[l];
        // the slots' first and second halves, stored as they come: (eta_f, z_f), (Hu_f, Hv_f)
        float2 *f0 = reinterpret_cast<float2 *>(m.sF + l), *f1 = f0 + 2 * m.L1, *f2 = f1 + 2 * m.L1;
        bool recon = false;
        if (MOVING && a.order == 2 && q.x - q.w > a.hthr) {
            const int gid = l < B ? c0 + l : a.halo_ids[h0 + (l - B)];
            const uint2 c = l < B ? a.codes[gid] : a.ring_codes[h0 + (l - B)];
            const float4 m0 = a.recA[2 * gid], m1 = a.recA[2 * gid + 1];
            const float4 qn[3] = {m.sW[c.x & 0xffffu], m.sW[c.x >> 16], m.sW[c.y & 0xffffu]};
            recon = qn[0].x - qn[0].w > a.hthr && qn[1].x - qn[1].w > a.hthr && qn[2].x - qn[2].w > a.hthr;
            if (recon) {
                float un[3], vn[3], e[3], u[3], v[3];
#pragma unroll
                for (int f = 0; f < 3; f++) {
                    un[f] = qn[f].y;
                    vn[f] = qn[f].z;
                    if ((c.y >> (16 + f)) & 1) {
                        const float2 n = a.normals[f * (size_t)a.nc + gid];
                        const float mn = q.y * n.x + q.z * n.y;
                        un[f] = q.y - 2.f * mn * n.x;
                        vn[f] = q.z - 2.f * mn * n.y;
                    }
                }
                limited_by_face(m0, m1, q.x, qn[0].x, qn[1].x, qn[2].x, e);
                limited_by_face(m0, m1, q.y, un[0], un[1], un[2], u);
                limited_by_face(m0, m1, q.z, vn[0], vn[1], vn[2], v);
                const float z0 = q.w + m1.z, z1 = q.w + m1.w, z2 = q.w - (m1.z + m1.w);
                recon = e[0] - z0 > a.hthr && e[1] - z1 > a.hthr && e[2] - z2 > a.hthr;
                if (recon) {
                    f0[0] = make_float2(e[0], z0); f0[1] = make_float2(u[0], v[0]);
                    f1[0] = make_float2(e[1], z1); f1[1] = make_float2(u[1], v[1]);
                    f2[0] = make_float2(e[2], z2); f2[1] = make_float2(u[2], v[2]);
                }
            }
        }
        if (!MOVING && a.order == 2 && q.x - q.w > a.hthr) {
            const int gid = l < B ? c0 + l : KEEP ? m.sHid[l - B] : a.halo_ids[h0 + (l - B)];
            const uint2 c = l < B ? a.codes[gid] : a.ring_codes[h0 + (l - B)];
            // the records in flight together, before the neighbours' states decide on them
            // (4M triangles 226.5 -> 222.5 us a step; all wet, 1M: 86.8 -> 85.5)
            const float4 m0 = a.recA[2 * gid], m1 = a.recA[2 * gid + 1];
            float4 N = make_float4(0.f, 0.f, 0.f, 0.f);
            if (l < B || c.y >> 16) N = a.recB[gid];
            float4 q0 = m.sW[c.x & 0xffffu], q1 = m.sW[c.x >> 16], q2 = m.sW[c.y & 0xffffu];
            if (q0.x - q0.w > a.hthr && q1.x - q1.w > a.hthr && q2.x - q2.w > a.hthr) {
                float D[3];
                limited(m0, m1, q.x, q0.x, q1.x, q2.x, D);
                // the face values stand on the face beds (the linear bed at the face
                // midpoints); the face depths must stay above the threshold
                const float e0 = D[0], e1 = D[1], e2 = D[2];
                const float z0 = add_(q.w, m1.z), z1 = add_(q.w, m1.w), z2 = sub_(q.w, add_(m1.z, m1.w));
                const float h0f = sub_(e0, z0), h1f = sub_(e1, z1), h2f = sub_(e2, z2);
                recon = h0f > a.hthr && h1f > a.hthr && h2f > a.hthr;
                if (recon) {
                    f0[0] = make_float2(e0, z0);
                    f1[0] = make_float2(e1, z1);
                    f2[0] = make_float2(e2, z2);
                    if (l < B) {
                        // the cell's own part of the pressure corrections over a closed triangle
                        const float p2 = mul_(sub_(e2, q.x), add_(h2f, sub_(q.x, z2)));
                        const float p0 = fma_(sub_(e0, q.x), add_(h0f, sub_(q.x, z0)), -p2);
                        const float p1 = fma_(sub_(e1, q.x), add_(h1f, sub_(q.x, z1)), -p2);
                        m.sS[l] = make_float2(mul_(a.half_g, fma_(p0, N.x, mul_(p1, N.z))),
                                              mul_(a.half_g, fma_(p0, N.y, mul_(p1, N.w))));
                    }
                    if (c.y >> 16) {             // some wall face: its ghost mirrors the momentum
                        if (c.y & 0x10000u) wall_ghost(q0, N.x, N.y);
                        if (c.y & 0x20000u) wall_ghost(q1, N.z, N.w);
                        if (c.y & 0x40000u) wall_ghost(q2, N.x + N.z, N.y + N.w);
                    }
                    limited(m0, m1, q.y, q0.y, q1.y, q2.y, D);
                    const float u0 = D[0], u1 = D[1], u2 = D[2];
                    limited(m0, m1, q.z, q0.z, q1.z, q2.z, D);
                    f0[1] = make_float2(u0, D[0]);
                    f1[1] = make_float2(u1, D[1]);
                    f2[1] = make_float2(u2, D[2]);
                }
            }
        }
        if (!recon) {
            const float4 v = make_float4(q.x, q.w, q.y, q.z);
            m.sF[l] = v;
            m.sF[m.L1 + l] = v;
            m.sF[2 * m.L1 + l] = v;
            if (!MOVING && l < B) m.sS[l] = make_float2(0.f, 0.f);
        }
    }
    cp_wait();
    __syncthreads();

    // C: owned faces, one flux each (Sec. 2.2).  The two face values a face reads are
    // used by no other face, so its thread overwrites them with the two sides' terms.
    for (int q = tid; q < nq; q += blockDim.x) {
        const float4 r = m.sFr[q];
        const unsigned u = __float_as_uint(r.w);
        const unsigned sl = u & 0xffffu, sr = u >> 16;
        const int bnd = sr < NBR_ABSORB ? 0 : (int)(NBR_WALL - sr) + 1;
        const float4 L = m.sF[sl];
        const float4 R = bnd ? L : m.sF[sr];
        float4 tL, tR;
        if constexpr (MOVING) {
            auto own_eta = [&](unsigned slot) { return m.sW[slot >= 2 * m.L1 ? slot - 2 * m.L1 : slot >= m.L1 ? slot - m.L1 : slot].x; };
            const float eL = own_eta(sl), eR = bnd ? eL : own_eta(sr);
            face_terms_by_side(a.g, a.half_g, a.hthr, L, eL, R, eR, r.x, r.y, r.z, bnd, tL, tR);
        } else
            face_terms(a.g, a.half_g, a.hthr, L, R, r.x, r.y, r.z, bnd, tL, tR);
        m.sF[sl] = tL;
        if (!bnd) m.sF[sr] = tR;
    }
    __syncthreads();

    // D: residual R_K = -(1/|K|) sum_f (side terms), faces in local order
    if (tid < ncell) {
        const float4 t0 = m.sF[tid], t1 = m.sF[m.L1 + tid], t2 = m.sF[2 * m.L1 + tid];
        const float area = m.sArea[tid];
        if constexpr (MOVING) {
            const float aH = t0.x + t1.x + t2.x, aHu = t0.y + t1.y + t2.y, aHv = t0.z + t1.z + t2.z;
            const float am = STAGE == 1 ? fmaxf(fmaxf(t0.w, t1.w), t2.w) : 0.f;
            finish_cell<STAGE, SOA>(a, c0 + tid, m.sW + tid, -aH / area, -aHu / area, -aHv / area, am, area, dt, my_min, my_neg,
                                    bad);
            return;
        }
        const float2 own = m.sS[tid];
        const float aH = add_(add_(t0.x, t1.x), t2.x);
        const float aHu = add_(add_(add_(own.x, t0.y), t1.y), t2.y);
        const float aHv = add_(add_(add_(own.y, t0.z), t1.z), t2.z);
        const float am = STAGE == 1 ? fmaxf(fmaxf(t0.w, t1.w), t2.w) : 0.f;
        const float ra = -rcp_approx(area);
        finish_cell<STAGE, SOA>(a, c0 + tid, m.sW + tid, mul_(aH, ra), mul_(aHu, ra), mul_(aHv, ra), am, area, dt,
                                my_min, my_neg, bad);
    }
}

}  // namespace vg
