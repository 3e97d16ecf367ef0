// FP32 instantiation of the step kernels (multiply-add contraction allowed).
#include <algorithm>

#include "step_kernels.cuh"

namespace vg {
// ---------------------------------------------------------------------------
// Many steps in one cooperative launch: the stage kernels' blocks, the same ones for a
// CTA in every stage, with a grid barrier where one kernel ends and the next begins.
//
// A step of three kernels from a graph pays for two ends of a kernel and starts of the
// next, and for the one-CTA epilogue: 12.4 us on 20k triangles, of which the blocks'
// chains of phases take about 7.  The barriers cost about 1.3 us each: 9.9 us, and 9.3
// where a CTA keeps its one block's mesh data in shared memory (steps_config_f32 has the
// other sizes).  A barrier is bound by the arrivals at one address (2400 CTAs of 64
// threads: 10 us), so the waiting CTAs poll with pauses (99k: 14.8 -> 14.5); arrivals
// spread over eight addresses, all of which every CTA then polls, and a flag written by
// the last to arrive were both slower (14.7, 16.5).
//
// Every CTA keeps the time and forms dt for itself, from the same bits.  The last CTA
// (it has no more blocks than another) also keeps the counts and records the gauges,
// while the others begin the next step: the state that it reads is next written behind
// two more barriers.  dtmin3[i % 3] is step i's CFL minimum; the last CTA empties the
// next step's between the two barriers of a step, when nobody uses it.  The last CTA to
// leave empties all three and the barrier's counts, also when CTAs have given up (the
// others may then still be in stage 1): a launch leaves nothing behind for the next.
// ---------------------------------------------------------------------------

// What a CTA wrote before it every CTA sees behind it.  Every thread must call it.
// False when the others have not arrived after about a second: the launch is
// cooperative, all its CTAs are resident, so this says that one of them has stopped.
__device__ __forceinline__ bool grid_barrier(StepsBarrier *bar, unsigned &target, unsigned max_polls)
{
    __shared__ int arrived;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&bar->arrived, 1u);
        target += gridDim.x;
        int ok = 0;
        for (unsigned polls = 0; polls < max_polls; polls++) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&bar->arrived) : "memory");
            if ((ok = (int)(v - target) >= 0)) break;
            __nanosleep(64);
        }
        __threadfence();
        arrived = ok;
    }
    __syncthreads();
    return arrived != 0;
}

// The step's epilogue: a gauge record every gauge_every steps into the device ring.
struct Gauges {
    int n, ring_cap, every;
    const int32_t *cells;
    double *ring_t, *ring_eta;
};

// SOA: one step of the caller's states from its time (CallerStep); the context's own
// scalars keep their values, and the last CTA writes the outcome to host memory.
struct CallerStep {
    double t, t_end;
    StepOutcome *out;
};

template <int MAXT, int MINCTAS, bool SOA>
__global__ void __launch_bounds__(MAXT, MINCTAS) steps_kernel(const KArgs<float> args, StepsBarrier *bar, const Gauges gauges,
                                                             int n_steps, const CallerStep caller, unsigned max_polls)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float red_min[32], s_dt;
    __shared__ long long red_neg[32], s_rec;
    __shared__ double s_t;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = (blockDim.x + 31) >> 5;
    const bool scribe = blockIdx.x == gridDim.x - 1;
    KArgs<float> a = args;
    DevScalars *sc = args.sc;
    const double t_end = SOA ? caller.t_end : sc->t_end;
    double dt_last = 0.0;                    // dt_last ... target: thread 0 only
    long long steps = 0, n_rec = 0;
    unsigned flags = 0, target = 0;
    if (tid == 0) {
        s_t = SOA ? caller.t : sc->t;
        steps = SOA ? 0 : sc->steps;
        n_rec = SOA ? 0 : sc->n_rec;
    }
    __syncthreads();
    long long my_neg = 0;
    bool bad = false, ok = true;
    const bool one_block = a.nblocks <= (int)gridDim.x;       // its mesh data stay in shared memory
    bool loaded = false;
    int i = 0;
    for (; i < n_steps; i++) {
        if (is_pos(t_end) && okey(s_t) >= okey(t_end)) break;      // the same in every CTA
        // stage 1 and the CTA's CFL bound
        float my_min = real_inf<float>();
        for (int b = blockIdx.x; b < a.nblocks; b += gridDim.x) {
            if (!one_block) loaded = false;
            process_block<1, SOA, KEEP_STEPS>(a, b, 0.f, smem_raw, my_min, my_neg, bad, loaded);
        }
        for (int o = 16; o > 0; o >>= 1) my_min = smin(my_min, __shfl_xor_sync(0xffffffffu, my_min, o));
        if (lane == 0) red_min[warp] = my_min;
        __syncthreads();
        if (tid == 0) {
            float mn = real_inf<float>();
            for (int w = 0; w < nwarps; w++) mn = smin(mn, red_min[w]);
            if (mn < real_inf<float>()) atomicMin(&sc->dtmin3[i % 3], min_bits(mn));
        }
        if (!(ok = grid_barrier(bar, target, max_polls))) break;
        if (tid == 0) {
            DevScalars v;
            v.t = s_t;
            v.dtmin_bits = __ldcg(&sc->dtmin3[i % 3]);
            dt_last = step_dt<float>(&v, a.cfl, a.dt_fixed, a.dt_max, t_end);
            s_dt = (float)dt_last;
            if (scribe) sc->dtmin3[(i + 1) % 3] = min_bits(real_inf<float>());
        }
        __syncthreads();
        const float dt = s_dt;
        for (int b = blockIdx.x; b < a.nblocks; b += gridDim.x) {
            if (!one_block) loaded = false;
            process_block<2, SOA, KEEP_STEPS>(a, b, dt, smem_raw, my_min, my_neg, bad, loaded);
        }
        if (!(ok = grid_barrier(bar, target, max_polls))) break;
        if (tid == 0) {
            if (!isfinite(dt_last)) flags |= FLAG_NONFINITE_DT;
            long long rec = -1;
            if (dt_last > 0.0) {
                s_t = s_t + dt_last;
                steps++;
                if (scribe && gauges.n > 0 && (gauges.every == 1 || steps % gauges.every == 0)) {
                    if (n_rec < gauges.ring_cap) {
                        rec = n_rec++;
                        gauges.ring_t[rec] = s_t;
                    } else {
                        flags |= FLAG_RING_FULL;
                    }
                }
            }
            s_rec = rec;
        }
        __syncthreads();
        if constexpr (!SOA) {
            if (scribe && s_rec >= 0)
                for (int g = tid; g < gauges.n; g += blockDim.x)
                    gauges.ring_eta[s_rec * gauges.n + g] = surface(a.wout, a.z, gauges.cells[g]);
            float4 *w_new = a.wout;            // the state buffers change roles
            a.wout = const_cast<float4 *>(a.w);
            a.w = w_new;
        }
    }
    // steps past t_end leave the state as it is; an odd number of them leaves it in
    // the other buffer
    if (ok && ((n_steps - i) & 1))
        copy_state<SOA>(a, blockIdx.x * (int64_t)blockDim.x + tid, (int64_t)gridDim.x * blockDim.x);
    for (int o = 16; o > 0; o >>= 1) my_neg += __shfl_xor_sync(0xffffffffu, my_neg, o);
    if (lane == 0) red_neg[warp] = my_neg;
    bad = __syncthreads_or(bad);
    if (tid == 0) {
        long long neg = 0;
        for (int w = 0; w < nwarps; w++) neg += red_neg[w];
        if (!ok) flags |= FLAG_TIMEOUT;
        if (bad) flags |= FLAG_NONFINITE_STATE;
        if (neg) atomicAdd((unsigned long long *)(SOA ? &bar->neg_count : &sc->neg_count), (unsigned long long)neg);
        if (flags) atomicOr(SOA ? &bar->flags : &sc->flags, flags);
        if (!SOA && scribe) {
            sc->t = s_t;
            sc->dt = i < n_steps ? 0.0 : dt_last;
            sc->steps = steps;
            sc->n_rec = n_rec;
        }
        __threadfence();
        if (atomicAdd(&bar->left, 1u) == gridDim.x - 1) {    // the last CTA to leave
            __threadfence();
            for (int k = 0; k < 3; k++) sc->dtmin3[k] = min_bits(real_inf<float>());
            if constexpr (SOA) {
                StepOutcome o;
                o.dt = i < n_steps ? 0.0 : dt_last;
                o.neg_count = (long long)atomicExch((unsigned long long *)&bar->neg_count, 0ull);
                o.flags = atomicExch(&bar->flags, 0u);
                *caller.out = o;
            }
            bar->left = 0;
            bar->arrived = 0;
        }
    }
}

// The kernel for a thread count with `ctas` CTAs of 256 threads per SM (null: none).
template <bool SOA>
static const void *steps_kernel_ptr(int threads, int ctas)
{
    if (threads <= 256) return ctas > 4 ? (const void *)steps_kernel<256, 5, SOA> : (const void *)steps_kernel<256, 4, SOA>;
    return threads > 384 ? (const void *)steps_kernel<512, 2, SOA> : nullptr;
}

// Rounds of blocks that a launch of `kern` takes (grid: its resident CTAs, at most one
// per block).
static cudaError_t steps_rounds(const void *kern, const DevPtrs &d, size_t smem, int &grid, int &rounds)
{
    int per_sm = 0, dev = 0, sms = 0;
    cudaError_t e = raise_smem_limit(kern, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, d.threads, smem);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    grid = (int)std::min<long long>((long long)sms * per_sm, d.nblocks);
    rounds = grid > 0 ? (d.nblocks + grid - 1) / grid : 0;
    return cudaSuccess;
}

// Four CTAs of 256 threads per SM have registers enough; five spill a little and are
// taken where they save a round of blocks.  Figures: us a step, four / five CTAs / the
// three kernels in a graph (basin, 256 cells; before a CTA with one block kept its mesh
// data, which took another us off one round):
//   99,458 (389 blocks): 14.5 / 15.7 / 17.6;  151,250 (591): 16.3 / 17.3 / 18.9
//   186,050 (727): 21.6 / 19.1 / 19.6;  245,000 (958): 23.2 / 24.8 / 25.8
//   320,000 (1250): 25.0 / 26.3 / 28.8;  500,000 (1954): 34.5 / 35.7 / 36.9
//   605,000 (2364): 41.7 / 39.2 / 39.4;  845,000: 59.6 / 57.4 / 57.7
// Beyond three rounds the graph is as fast and hands the blocks out evenly (1M: 65.4
// against 68.4; 4M: 225 against 249).
int steps_config_f32(const DevPtrs &d, LaunchCfg &cfg)
{
    cfg.grid = 0;
    cfg.smem = stage_smem_bytes<float>(d.block, d.max_halo, d.max_ring1, d.max_faces);
    const void *k4 = steps_kernel_ptr<false>(d.threads, 4), *k5 = steps_kernel_ptr<false>(d.threads, 5);
    if (!k4) return 0;
    int g4 = 0, r4 = 0, g5 = 0, r5 = 0;
    cudaError_t e = steps_rounds(k4, d, cfg.smem, g4, r4);
    if (e == cudaSuccess) e = steps_rounds(k5, d, cfg.smem, g5, r5);
    if (e != cudaSuccess) return (int)e;
    cfg.ctas = r5 < r4 ? 5 : 4;
    if (std::min(r4, r5) > 3) return 0;
    // the same grid has to fit with the caller's states
    int g = 0, r = 0;
    e = steps_rounds(steps_kernel_ptr<true>(d.threads, cfg.ctas), d, cfg.smem, g, r);
    if (e == cudaSuccess) cfg.grid = std::min(g, cfg.ctas == 5 ? g5 : g4);
    return (int)e;
}

static int launch_steps(const void *kern, const DevPtrs &d, KArgs<float> a, Gauges gauges, int n, CallerStep caller,
                        LaunchCfg c, void *stream)
{
    StepsBarrier *bar = reinterpret_cast<StepsBarrier *>(reinterpret_cast<char *>(d.sc) + kBarrierAt);
    void *args[] = {&a, &bar, &gauges, &n, &caller, &c.max_polls};
    return (int)cudaLaunchCooperativeKernel(kern, dim3(c.grid), dim3(d.threads), args, c.smem, static_cast<cudaStream_t>(stream));
}

int launch_steps_f32(const DevPtrs &d, const StepParams &p, const void *w_in, void *w_out, int n, const LaunchCfg &c, void *stream)
{
    return launch_steps(steps_kernel_ptr<false>(d.threads, c.ctas), d, make_args<float>(d, p, w_in, w_out),
                        {d.n_gauges, d.ring_cap, p.gauge_every, d.gauge_cells, d.ring_t, d.ring_eta}, n, {}, c, stream);
}

int launch_caller_step_f32(const DevPtrs &d, const StepParams &p, const void *w_in, void *w_out, double t, double t_end,
                           StepOutcome *out, const LaunchCfg &c, void *stream)
{
    return launch_steps(steps_kernel_ptr<true>(d.threads, c.ctas), d, make_args<float>(d, p, w_in, w_out, true), {}, 1,
                        {t, t_end, out}, c, stream);
}

size_t stage_smem_f32(int block, int max_halo, int max_ring1, int max_faces)
{
    return stage_smem_bytes<float>(block, max_halo, max_ring1, max_faces);
}
int stage_config_f32(const DevPtrs &d, int stage, LaunchCfg &cfg) { return stage_config<float>(d, stage, cfg); }
int launch_stage1_f32(const DevPtrs &d, const StepParams &p, const void *w_in, const LaunchCfg &c, void *stream)
{
    return launch_stage<float>(d, p, 1, w_in, nullptr, c, stream);
}
int launch_stage2_f32(const DevPtrs &d, const StepParams &p, const void *w_in, void *w_out, const LaunchCfg &c, void *stream)
{
    return launch_stage<float>(d, p, 2, w_in, w_out, c, stream);
}
int launch_stage_soa_f32(const DevPtrs &d, const StepParams &p, int stage, const void *w_in, void *w_out, const LaunchCfg &c,
                         void *stream)
{
    return launch_stage<float>(d, p, stage, w_in, w_out, c, stream, true);
}
int launch_rk_unfused_f32(const DevPtrs &d, const StepParams &p, int part, const void *w_in, void *w_out, void *w1,
                          void *R1, const LaunchCfg &c1, void *stream)
{
    return launch_rk_unfused<float>(d, p, part, w_in, w_out, w1, R1, c1, stream);
}
size_t batch_mesh_bytes_f32() { return sizeof(BatchMesh<float>); }
void fill_batch_mesh_f32(void *dst, const DevPtrs &d, const StepParams &p, const void *w_in, void *w_out, int n_scen,
                         int first_item, int first_entry)
{
    fill_batch_mesh<float>(dst, d, p, w_in, w_out, n_scen, first_item, first_entry);
}
int batch_config_f32(int block, int max_halo, int max_ring1, int max_faces, int n_entries, int &grid, size_t &smem, int &scen_at)
{
    return batch_config<float>(block, max_halo, max_ring1, max_faces, n_entries, grid, smem, scen_at);
}
int launch_batch_step_f32(const void *table, int n_mesh, int n_items, int groups, int n_entries, DevScalars *sc_all, int block,
                          int grid, size_t smem, int scen_at, const StepParams &p, bool gauges, void *stream)
{
    return launch_batch_step<float>(table, n_mesh, n_items, groups, n_entries, sc_all, block, grid, smem, scen_at, p, gauges, stream);
}
}  // namespace vg
