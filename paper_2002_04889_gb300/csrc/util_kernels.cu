// Small kernels around the step: the per-step epilogue (time, gauges, reset of
// the CFL minimum), state import/export with the cell permutation, and the
// diagnostics reduction.
#include "step_kernels.cuh"

namespace vg {

namespace {

template <typename real> using word = typename StateWord<real>::type;    // of a state buffer

template <typename real>
__device__ __forceinline__ unsigned long long inf_bits();
template <> __device__ __forceinline__ unsigned long long inf_bits<float>() { return (unsigned long long)__float_as_uint(CUDART_INF_F); }
template <> __device__ __forceinline__ unsigned long long inf_bits<double>() { return (unsigned long long)__double_as_longlong(CUDART_INF); }

// Epilogue of one step: t += dt (Sec. 2.3), gauge record (Sec. 3 virtual gauges:
// eta = H + z of each gauge cell), reset of the CFL minimum for the next step.  One
// CTA on the critical path of every step: the scalars are read in one go and the
// first gauges' values before it is known whether the step records (a chain of
// dependent loads and stores otherwise, 2.5 of 15 us a step at 20k triangles).
template <typename real>
__global__ void post_step_kernel(DevPtrs d, StepParams p, const word<real> *w)
{
    __shared__ long long rec;
    DevScalars *sc = d.sc;
    chain_wait();
    chain_next();
    const real *z = static_cast<const real *>(d.z);
    const bool mine = (int)threadIdx.x < d.n_gauges;
    double eta = 0.0;
    if (mine) eta = surface(w, z, d.gauge_cells[threadIdx.x]);
    if (threadIdx.x == 0) {
        const DevScalars v = *sc;
        const double dt = step_dt<real>(&v, p.cfl, p.dt_fixed, p.dt_max, v.t_end);
        sc->dt = dt;
        long long r = -1;
        if (!isfinite(dt)) sc->flags = v.flags | FLAG_NONFINITE_DT;
        if (dt > 0.0) {
            const double t = v.t + dt;
            const long long steps = v.steps + 1;
            sc->t = t;
            sc->steps = steps;
            if (d.n_gauges > 0 && (p.gauge_every == 1 || steps % p.gauge_every == 0)) {
                if (v.n_rec < d.ring_cap) {
                    r = v.n_rec;
                    sc->n_rec = r + 1;
                    d.ring_t[r] = t;
                } else {
                    sc->flags = v.flags | FLAG_RING_FULL | (isfinite(dt) ? 0u : FLAG_NONFINITE_DT);
                }
            }
        }
        sc->dtmin_bits = inf_bits<real>();
        rec = r;
    }
    __syncthreads();
    if (rec >= 0) {
        if (mine) d.ring_eta[rec * d.n_gauges + threadIdx.x] = eta;
        for (int g = threadIdx.x + blockDim.x; g < d.n_gauges; g += blockDim.x)
            d.ring_eta[rec * d.n_gauges + g] = surface(w, z, d.gauge_cells[g]);
    }
}

template <typename real>
__global__ void record_gauges_kernel(DevPtrs d, const word<real> *w)
{
    DevScalars *sc = d.sc;
    long long rec = sc->n_rec;
    if (rec >= d.ring_cap) {
        if (threadIdx.x == 0) sc->flags |= FLAG_RING_FULL;
        return;
    }
    const real *z = static_cast<const real *>(d.z);
    for (int g = threadIdx.x; g < d.n_gauges; g += blockDim.x) {
        int32_t c = d.gauge_cells[g];
        d.ring_eta[rec * d.n_gauges + g] = surface(w, z, c);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        d.ring_t[rec] = sc->t;
        sc->n_rec = rec + 1;
    }
}

// Moving bed (time-dependent depth of Sec. 2.1, read as a kinematic rupture):
// depth_v(t) = depth0_v - uplift_v R((t - onset_v) / rise), R(s) = min(1, max(0, s))
// (rise = 0: a step at onset), cell bed z_K = -(mean of its vertices' depths) and face
// beds z_f = -(mean of the face's two vertex depths),
// applied with H unchanged.  The products and sums are rounded one by one
// (__dmul_rn / __dadd_rn are never contracted), as written.
//
// The kernel was bound by FP64 divisions (three ramps and one mean per cell: 45 us
// of an 84 us FP32 step on 298k triangles).  A vertex before its onset or after its
// rise needs none, found by integer compares; the others divide by rise and by 3
// through their reciprocals; and a cell whose vertices are all at rest over the
// step keeps its bed untouched, so a step costs the cells above the moving part of
// the rupture plus one look at the onsets of the others.

// Where a vertex stands: 0 before its onset (R = 0), 2 after its rise (R = 1), 1 between.
// (RN(x / rise) >= 1 exactly where x >= rise.)
__device__ __forceinline__ int ramp_phase(double t, double onset, double rise)
{
    if (!(rise > 0.0)) return t >= onset ? 2 : 0;
    if (okey(t) <= okey(onset)) return 0;
    return okey(__dsub_rn(t, onset)) >= okey(rise) ? 2 : 1;
}

template <typename real>
__global__ void bed_update_kernel(DevPtrs d, StepParams p, word<real> *w, int at_step_end, double t_set)
{
    __shared__ double s_t[2];        // the stored bed's time and the new one's, formed once per CTA
    if (threadIdx.x == 0) {
        s_t[0] = d.sc->t;
        s_t[1] = at_step_end ? d.sc->t + step_dt<real>(d.sc, p.cfl, p.dt_fixed, p.dt_max, d.sc->t_end) : t_set;
    }
    __syncthreads();
    const double t0 = s_t[0], t = s_t[1];
    const Recip by_rise = recip_given(d.bed_rise, d.bed_rrise), by_3 = recip_given(3.0, 1.0 / 3.0);
    real *z = static_cast<real *>(const_cast<void *>(d.z));
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < d.nc; k += (int64_t)gridDim.x * blockDim.x) {
        int32_t v[3];
        double onset[3];
        int phase[3];
        bool moves = !at_step_end;   // set outright: the stored bed may be of any time
#pragma unroll
        for (int j = 0; j < 3; j++) {
            v[j] = d.bed_vtx[j * d.nc + k];
            onset[j] = d.bed_onset[v[j]];
            phase[j] = ramp_phase(t, onset[j], d.bed_rise);
            // at rest over the step: before the onset still, or after the rise already
            moves = moves || phase[j] == 1 || (phase[j] == 2 && ramp_phase(t0, onset[j], d.bed_rise) != 2);
        }
        if (!moves) continue;
        double dv[3];
#pragma unroll
        for (int j = 0; j < 3; j++) {
            double r = phase[j] == 2 ? 1.0 : 0.0;
            if (phase[j] == 1) r = quot(__dsub_rn(t, onset[j]), by_rise);
            dv[j] = __dsub_rn(d.bed_depth0[v[j]], __dmul_rn(d.bed_uplift[v[j]], r));
        }
        const double zn = -quot(__dadd_rn(__dadd_rn(dv[0], dv[1]), dv[2]), by_3);
        // face beds: -(mean of the face's two vertex depths); FP32 keeps z_f - z_K
        // of faces 0 and 1, beside its reconstruction matrix
        double zfn[3];
#pragma unroll
        for (int f = 0; f < 3; f++) zfn[f] = -half_of(__dadd_rn(dv[f], dv[(f + 1) % 3]));
        if constexpr (std::is_same<real, float>::value) {
            float *recA = static_cast<float *>(const_cast<void *>(d.geo));
            *reinterpret_cast<float2 *>(recA + 8 * k + 6) = make_float2((float)(zfn[0] - zn), (float)(zfn[1] - zn));
            // keep H = eta - z; a dry cell (eta == z) stays exactly dry
            const float zr = (float)zn;
            if (w) {
                float4 q = w[k];
                if (zr != q.w) {
                    q.x = q.x - q.w <= 0.f ? zr : (q.x - q.w) + zr;
                    q.w = zr;
                    w[k] = q;
                }
            }
            z[k] = zr;
            const_cast<double *>(d.z64)[k] = zn;
        } else {
            double *zf = static_cast<double *>(const_cast<void *>(d.zf));
            for (int f = 0; f < 3; f++) zf[f * d.nc + k] = zfn[f];
            z[k] = zn;
        }
    }
}

// FP32: the bed of every cell of a state buffer, eta kept.
__global__ void state_bed_kernel(int64_t nc, const float *z, float4 *w)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nc; k += (int64_t)gridDim.x * blockDim.x)
        w[k].w = z[k];
}

// One cell's state (H, Hu, Hv) in a state buffer; zk the FP64 bed (FP32: eta = H + z
// formed with it before rounding, so still water at a common level gets exactly
// the same eta everywhere).
template <typename src_t>
__device__ __forceinline__ void store_cell(double *w, int64_t nc, int64_t k, src_t h, src_t hu, src_t hv, double)
{
    w[k] = (double)h;
    w[nc + k] = (double)hu;
    w[2 * nc + k] = (double)hv;
}
template <typename src_t>
__device__ __forceinline__ void store_cell(float4 *w, int64_t, int64_t k, src_t h, src_t hu, src_t hv, double zk)
{
    w[k] = make_float4((float)((double)h + zk), (float)hu, (float)hv, (float)zk);
}

// The inverse.  FP32: a cell is dry when eta <= z in the kernels' own (rounded)
// bed, and then H is exactly 0.
template <typename dst_t>
__device__ __forceinline__ void fetch_cell(const double *w, int64_t nc, int64_t k, double, dst_t &h, dst_t &hu, dst_t &hv)
{
    h = (dst_t)w[k];
    hu = (dst_t)w[nc + k];
    hv = (dst_t)w[2 * nc + k];
}
template <typename dst_t>
__device__ __forceinline__ void fetch_cell(const float4 *w, int64_t, int64_t k, double zk, dst_t &h, dst_t &hu, dst_t &hv)
{
    const float4 q = w[k];
    h = (dst_t)((q.x - q.w <= 0.f) ? 0.0 : fmax(0.0, (double)q.x - zk));
    hu = (dst_t)q.y;
    hv = (dst_t)q.z;
}

// State in (original order, H) -> internal order, stored form.
template <typename real, typename src_t>
__global__ void import_state_kernel(int64_t nc, const int32_t *old_of_new, const src_t *H,
                                    const src_t *Hu, const src_t *Hv, const double *z, word<real> *w, DevScalars *sc)
{
    bool bad = false;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nc; k += (int64_t)gridDim.x * blockDim.x) {
        int64_t o = old_of_new[k];
        src_t h = H[o], hu = Hu[o], hv = Hv[o];
        if (!(h >= src_t(0)) || !isfinite(h) || !isfinite(hu) || !isfinite(hv)) bad = true;
        store_cell(w, nc, k, h, hu, hv, std::is_same<real, float>::value ? z[k] : 0.0);
    }
    if (bad) atomicOr(&sc->flags, FLAG_BAD_INPUT);
}

// Internal order, stored form -> original order, H.
template <typename real, typename dst_t>
__global__ void export_state_kernel(int64_t nc, const int32_t *old_of_new, const word<real> *w, const double *z, dst_t *H,
                                    dst_t *Hu, dst_t *Hv)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nc; k += (int64_t)gridDim.x * blockDim.x) {
        int64_t o = old_of_new[k];
        dst_t h, hu, hv;
        fetch_cell(w, nc, k, std::is_same<real, float>::value ? z[k] : 0.0, h, hu, hv);
        H[o] = h;
        Hu[o] = hu;
        Hv[o] = hv;
    }
}

// The same two conversions with one thread per V consecutive ORIGINAL cells o
// (k = new_of_old[o]): the host-order arrays are read or written contiguously,
// 16 bytes per thread and array (V = 4 floats or 2 doubles), so they can be
// pinned host memory that the kernel reads or writes in place over the CPU-GPU
// link (the internal-order side is scattered in HBM instead).  vec = false (a
// host array not 16-byte aligned) takes every cell one at a time.
template <typename T> struct Vec16;
template <> struct Vec16<float> { using type = float4; };
template <> struct Vec16<double> { using type = double2; };

template <typename real, typename src_t>
__device__ __forceinline__ void import_one(int64_t nc, int64_t k, src_t h, src_t hu, src_t hv, double zk,
                                           word<real> *w, bool &bad)
{
    if (!(h >= src_t(0)) || !isfinite(h) || !isfinite(hu) || !isfinite(hv)) bad = true;
    store_cell(w, nc, k, h, hu, hv, zk);
}

// zo: the FP64 bed in the original order (contiguous reads), or null (z[k]).
template <typename real, typename src_t>
__global__ void import_state_orig_kernel(int64_t nc, const int32_t *new_of_old, const src_t *H, const src_t *Hu,
                                         const src_t *Hv, const double *z, const double *zo, word<real> *w,
                                         DevScalars *sc, bool vec)
{
    constexpr int V = 16 / sizeof(src_t);
    using vt = typename Vec16<src_t>::type;
    bool bad = false;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t ng = vec ? nc / V : 0;
    for (int64_t gi = tid; gi < ng; gi += stride) {
        const vt h = reinterpret_cast<const vt *>(H)[gi], hu = reinterpret_cast<const vt *>(Hu)[gi],
                 hv = reinterpret_cast<const vt *>(Hv)[gi];
        const src_t *ph = reinterpret_cast<const src_t *>(&h), *phu = reinterpret_cast<const src_t *>(&hu),
                    *phv = reinterpret_cast<const src_t *>(&hv);
#pragma unroll
        for (int j = 0; j < V; j++) {
            const int64_t o = gi * V + j, k = new_of_old[o];
            import_one<real, src_t>(nc, k, ph[j], phu[j], phv[j],
                                    std::is_same<real, float>::value ? (zo ? zo[o] : z[k]) : 0.0, w, bad);
        }
    }
    for (int64_t o = ng * V + tid; o < nc; o += stride) {
        const int64_t k = new_of_old[o];
        import_one<real, src_t>(nc, k, H[o], Hu[o], Hv[o], std::is_same<real, float>::value ? (zo ? zo[o] : z[k]) : 0.0, w,
                                bad);
    }
    if (bad) atomicOr(&sc->flags, FLAG_BAD_INPUT);
}

// zo: the FP64 bed in the original order, or null (z[k]).
template <typename real, typename dst_t>
__global__ void export_state_orig_kernel(int64_t nc, const int32_t *new_of_old, const word<real> *w, const double *z,
                                         const double *zo, dst_t *H, dst_t *Hu, dst_t *Hv, bool vec)
{
    constexpr int V = 16 / sizeof(dst_t);
    using vt = typename Vec16<dst_t>::type;
    const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t ng = vec ? nc / V : 0;
    for (int64_t gi = tid; gi < ng; gi += stride) {
        vt h, hu, hv;
        dst_t *ph = reinterpret_cast<dst_t *>(&h), *phu = reinterpret_cast<dst_t *>(&hu),
              *phv = reinterpret_cast<dst_t *>(&hv);
#pragma unroll
        for (int j = 0; j < V; j++) {
            const int64_t o = gi * V + j, k = new_of_old[o];
            fetch_cell(w, nc, k, std::is_same<real, float>::value ? (zo ? zo[o] : z[k]) : 0.0, ph[j], phu[j], phv[j]);
        }
        reinterpret_cast<vt *>(H)[gi] = h;
        reinterpret_cast<vt *>(Hu)[gi] = hu;
        reinterpret_cast<vt *>(Hv)[gi] = hv;
    }
    for (int64_t o = ng * V + tid; o < nc; o += stride) {
        const int64_t k = new_of_old[o];
        fetch_cell(w, nc, k, std::is_same<real, float>::value ? (zo ? zo[o] : z[k]) : 0.0, H[o], Hu[o], Hv[o]);
    }
}

constexpr int DIAG_BLOCKS = 1024;

// Fixed grid, fixed reduction tree: the sums do not depend on timing.
template <typename real>
__global__ void diag_partial_kernel(int64_t nc, const word<real> *w, const double *z, const real *areas, double hthr,
                                    double *part)
{
    __shared__ double s_mass[256], s_min[256], s_dry[256];
    double mass = 0.0, mn = CUDART_INF, dry = 0.0;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nc; k += (int64_t)gridDim.x * blockDim.x) {
        double h;
        if constexpr (std::is_same<real, float>::value) h = (double)w[k].x - z[k];
        else h = w[k];
        const double area = (double)areas[k];
        mass += area * h;
        mn = fmin(mn, h);
        dry += h <= hthr ? 1.0 : 0.0;
    }
    s_mass[threadIdx.x] = mass; s_min[threadIdx.x] = mn; s_dry[threadIdx.x] = dry;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            s_mass[threadIdx.x] += s_mass[threadIdx.x + o];
            s_min[threadIdx.x] = fmin(s_min[threadIdx.x], s_min[threadIdx.x + o]);
            s_dry[threadIdx.x] += s_dry[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[3 * blockIdx.x] = s_mass[0];
        part[3 * blockIdx.x + 1] = s_min[0];
        part[3 * blockIdx.x + 2] = s_dry[0];
    }
}

__global__ void diag_final_kernel(const double *part, int n, double *out)
{
    if (threadIdx.x == 0) {
        double mass = 0.0, mn = CUDART_INF, dry = 0.0;
        for (int i = 0; i < n; i++) {
            mass += part[3 * i];
            mn = fmin(mn, part[3 * i + 1]);
            dry += part[3 * i + 2];
        }
        out[0] = mass; out[1] = mn; out[2] = dry;
    }
}

int grid_for(int64_t n) { return (int)std::min<int64_t>(std::max<int64_t>((n + 255) / 256, 1), 4096); }

}  // namespace

int launch_post_step(const DevPtrs &d, const StepParams &p, const void *w, int precision, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (precision == 64) return (int)launch_after(post_step_kernel<double>, 1, 128, 0, s, d, p, static_cast<const double *>(w));
    return (int)launch_after(post_step_kernel<float>, 1, 128, 0, s, d, p, static_cast<const float4 *>(w));
}

int launch_bed_update(const DevPtrs &d, const StepParams &p, void *w, int precision, bool at_step_end,
                      double t_set, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int blocks = grid_for(d.nc);
    if (precision == 64)
        bed_update_kernel<double><<<blocks, 256, 0, s>>>(d, p, static_cast<double *>(w), at_step_end, t_set);
    else
        bed_update_kernel<float><<<blocks, 256, 0, s>>>(d, p, static_cast<float4 *>(w), at_step_end, t_set);
    return (int)cudaGetLastError();
}

int launch_state_bed(const DevPtrs &d, void *w, void *stream)
{
    state_bed_kernel<<<grid_for(d.nc), 256, 0, static_cast<cudaStream_t>(stream)>>>(d.nc, static_cast<const float *>(d.z),
                                                                                    static_cast<float4 *>(w));
    return (int)cudaGetLastError();
}

int util_preload()
{
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, (const void *)post_step_kernel<double>);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, (const void *)post_step_kernel<float>);
    return (int)e;
}

int launch_record_gauges(const DevPtrs &d, const void *w, int precision, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (precision == 64) record_gauges_kernel<double><<<1, 128, 0, s>>>(d, static_cast<const double *>(w));
    else record_gauges_kernel<float><<<1, 128, 0, s>>>(d, static_cast<const float4 *>(w));
    return (int)cudaGetLastError();
}

int launch_import_state(const DevPtrs &d, const int32_t *old_of_new, const void *H, const void *Hu,
                        const void *Hv, int src_is_double, void *w, int precision, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int grid = grid_for(d.nc);
    if (precision == 64) {
        const double *z = d.z64;
        if (src_is_double)
            import_state_kernel<double, double><<<grid, 256, 0, s>>>(d.nc, old_of_new, (const double *)H, (const double *)Hu, (const double *)Hv, z, (double *)w, d.sc);
        else
            import_state_kernel<double, float><<<grid, 256, 0, s>>>(d.nc, old_of_new, (const float *)H, (const float *)Hu, (const float *)Hv, z, (double *)w, d.sc);
    } else {
        const double *z = d.z64;
        if (src_is_double)
            import_state_kernel<float, double><<<grid, 256, 0, s>>>(d.nc, old_of_new, (const double *)H, (const double *)Hu, (const double *)Hv, z, (float4 *)w, d.sc);
        else
            import_state_kernel<float, float><<<grid, 256, 0, s>>>(d.nc, old_of_new, (const float *)H, (const float *)Hu, (const float *)Hv, z, (float4 *)w, d.sc);
    }
    return (int)cudaGetLastError();
}

static bool aligned16(const void *a, const void *b, const void *c)
{
    return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(c)) & 15) == 0;
}

int launch_import_state_orig(const DevPtrs &d, const int32_t *new_of_old, const void *H, const void *Hu,
                             const void *Hv, int src_is_double, void *w, int precision, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int grid = grid_for(d.nc);
    const double *z = d.z64, *zo = d.z64_orig;
    const bool vec = aligned16(H, Hu, Hv);
    if (precision == 64) {
        if (src_is_double)
            import_state_orig_kernel<double, double><<<grid, 256, 0, s>>>(d.nc, new_of_old, (const double *)H, (const double *)Hu, (const double *)Hv, z, zo, (double *)w, d.sc, vec);
        else
            import_state_orig_kernel<double, float><<<grid, 256, 0, s>>>(d.nc, new_of_old, (const float *)H, (const float *)Hu, (const float *)Hv, z, zo, (double *)w, d.sc, vec);
    } else {
        if (src_is_double)
            import_state_orig_kernel<float, double><<<grid, 256, 0, s>>>(d.nc, new_of_old, (const double *)H, (const double *)Hu, (const double *)Hv, z, zo, (float4 *)w, d.sc, vec);
        else
            import_state_orig_kernel<float, float><<<grid, 256, 0, s>>>(d.nc, new_of_old, (const float *)H, (const float *)Hu, (const float *)Hv, z, zo, (float4 *)w, d.sc, vec);
    }
    return (int)cudaGetLastError();
}

int launch_export_state_orig(const DevPtrs &d, const int32_t *new_of_old, const void *w, int precision, void *H,
                             void *Hu, void *Hv, int dst_is_double, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int grid = grid_for(d.nc);
    const bool vec = aligned16(H, Hu, Hv);
    const double *zo = d.z64_orig;
    if (precision == 64) {
        if (dst_is_double)
            export_state_orig_kernel<double, double><<<grid, 256, 0, s>>>(d.nc, new_of_old, (const double *)w, d.z64, zo, (double *)H, (double *)Hu, (double *)Hv, vec);
        else
            export_state_orig_kernel<double, float><<<grid, 256, 0, s>>>(d.nc, new_of_old, (const double *)w, d.z64, zo, (float *)H, (float *)Hu, (float *)Hv, vec);
    } else {
        if (dst_is_double)
            export_state_orig_kernel<float, double><<<grid, 256, 0, s>>>(d.nc, new_of_old, (const float4 *)w, d.z64, zo, (double *)H, (double *)Hu, (double *)Hv, vec);
        else
            export_state_orig_kernel<float, float><<<grid, 256, 0, s>>>(d.nc, new_of_old, (const float4 *)w, d.z64, zo, (float *)H, (float *)Hu, (float *)Hv, vec);
    }
    return (int)cudaGetLastError();
}

int launch_export_state(const DevPtrs &d, const int32_t *old_of_new, const void *w, int precision,
                        void *H, void *Hu, void *Hv, int dst_is_double, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int grid = grid_for(d.nc);
    if (precision == 64) {
        const double *z = d.z64;
        if (dst_is_double)
            export_state_kernel<double, double><<<grid, 256, 0, s>>>(d.nc, old_of_new, (const double *)w, z, (double *)H, (double *)Hu, (double *)Hv);
        else
            export_state_kernel<double, float><<<grid, 256, 0, s>>>(d.nc, old_of_new, (const double *)w, z, (float *)H, (float *)Hu, (float *)Hv);
    } else {
        const double *z = d.z64;
        if (dst_is_double)
            export_state_kernel<float, double><<<grid, 256, 0, s>>>(d.nc, old_of_new, (const float4 *)w, z, (double *)H, (double *)Hu, (double *)Hv);
        else
            export_state_kernel<float, float><<<grid, 256, 0, s>>>(d.nc, old_of_new, (const float4 *)w, z, (float *)H, (float *)Hu, (float *)Hv);
    }
    return (int)cudaGetLastError();
}

int launch_diagnostics(const DevPtrs &d, const void *w, int precision, double hthr, double *part,
                       double *out, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (precision == 64)
        diag_partial_kernel<double><<<DIAG_BLOCKS, 256, 0, s>>>(d.nc, (const double *)w, d.z64, (const double *)d.geo + GEO_AREA * d.nc, hthr, part);
    else
        diag_partial_kernel<float><<<DIAG_BLOCKS, 256, 0, s>>>(d.nc, (const float4 *)w, d.z64, d.area32, hthr, part);
    diag_final_kernel<<<1, 32, 0, s>>>(part, DIAG_BLOCKS, out);
    return (int)cudaGetLastError();
}

}  // namespace vg
