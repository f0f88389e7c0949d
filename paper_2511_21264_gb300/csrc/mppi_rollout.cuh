// The rollout kernel (sampling + H-step contact rollout + stage cost of K
// samples, Alg. 1) and its launch: template over the arm size NA, the lanes
// per sample LPS (32, 16 or 8 -- one, two or four samples per warp), the
// control source MODE (0 explicit, 1 Philox with the diagonal sigma, 2
// Philox through the covariance factors when they are given: the draw's
// covariance branch stays out of the plain kernel), the ball-task cost suite and
// the placement of the lone ball contact's solve.  Each arm size is
// instantiated in a translation unit of its own (mppi_rollout_dh7.cu,
// mppi_rollout_planar3.cu) so that they compile in parallel.
#pragma once
#include <cuda_runtime.h>

#include "../../include/mppi.h"
#include "mppi_device.cuh"
#include "mppi_internal.h"
#include "mppi_kernels.cuh"
#include "mppi_task.cuh"

namespace mppi {

// Byte stride between the workspaces of consecutive samples of a CTA.  With
// several samples per warp the workspaces of a warp's samples start
// 128 / (samples per warp) bytes apart modulo 128, so that the groups'
// lane-indexed shared-memory accesses fall in different banks.
template <int NA, int LPS>
__host__ __device__ constexpr size_t ws_stride(size_t at_least = 0) {
    size_t s = sizeof(WarpWS<NA>);
    if (s < at_least) s = at_least;
    s = (s + 31) / 32 * 32;
    if (LPS == 32) return s;
    const size_t want = 128 / (32 / LPS);
    while (s % 128 != want) s += 32;
    return s;
}
// The ball-task suite keeps the previous state's points behind the workspace.
template <int NA, int LPS, bool TASK>
__host__ __device__ constexpr size_t ctl_stride() {
    return ws_stride<NA, LPS>(TASK ? sizeof(WarpWS<NA>) + sizeof(TaskPrev<NA>) : 0);
}

inline size_t unom_bytes(int unom_floats) { return ((size_t)unom_floats * sizeof(float) + 15) / 16 * 16; }

template <int NA, int LPS, bool TASK>
size_t rollout_smem(int spc, int unom_floats) {
    return sizeof(DevModel) + (TASK ? sizeof(DevTask) : 0) + unom_bytes(unom_floats) +
           (size_t)spc * ctl_stride<NA, LPS, TASK>();
}

// The samples per CTA that a launch accepts do not follow a smaller workspace (what
// the entry points refused stays refused): spc workspaces of at least 7.3 KB (5.6 KB
// for 3-link arms) fit max_sm bytes.
template <int NA, int LPS, bool TASK>
bool shape_fits(int spc, int unom_floats, int max_sm) {
    constexpr size_t least = ws_stride<NA, LPS>(NA == 7 ? 7328 : 5600);
    constexpr size_t stride = ctl_stride<NA, LPS, TASK>() > least ? ctl_stride<NA, LPS, TASK>() : least;
    return sizeof(DevModel) + (TASK ? sizeof(DevTask) : 0) + unom_bytes(unom_floats) + spc * stride <= (size_t)max_sm;
}

template <int NA, int LPS, int MODE, bool TASK, int PLACE>
__global__ void __launch_bounds__(512) rollout_kernel(RolloutArgs args) {
    using d = Dims<NA>;
    // launched as a programmatic dependent: wait for the previous kernel's
    // results (u_nom, the counter), then let the next kernel launch early
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
    extern __shared__ __align__(16) unsigned char smem[];
    DevModel& M = *reinterpret_cast<DevModel*>(smem);
    constexpr size_t task_b = TASK ? sizeof(DevTask) : 0;
    DevTask* task_s = reinterpret_cast<DevTask*>(smem + sizeof(DevModel));
    float* unom_s = reinterpret_cast<float*>(smem + sizeof(DevModel) + task_b);
    const int unom_n = (MODE >= 1 && args.stage_unom) ? args.H * d::NU : 0;
    const size_t ws_off = sizeof(DevModel) + task_b + ((size_t)unom_n * sizeof(float) + 15) / 16 * 16;
    stage_model(smem, args.model, unom_s, args.u_nom, unom_n);
    if constexpr (TASK) {
        const float4* src = reinterpret_cast<const float4*>(args.task);
        float4* dst = reinterpret_cast<float4*>(task_s);
        for (int t = threadIdx.x; t < (int)(sizeof(DevTask) / 16); t += blockDim.x) dst[t] = src[t];
    }
    __syncthreads();

    const int spc = blockDim.x / LPS, gi = threadIdx.x / LPS;
    const Lanes<LPS> g(threadIdx.x & 31);
    const int k = blockIdx.x * spc + gi;
    if (k >= args.n) return;
    WarpWS<NA>& w = *reinterpret_cast<WarpWS<NA>*>(smem + ws_off + (size_t)gi * ctl_stride<NA, LPS, TASK>());
    SampleIO io{};
    io.x = args.states + (size_t)k * args.state_stride;
    io.k = k;
    io.H = args.H;
    io.err = args.err;
    io.stats = args.stats;
    io.task = TASK ? task_s : nullptr;
    io.x_out = args.states_out ? args.states_out + (size_t)k * d::NX : nullptr;
    io.U_store = MODE >= 1 ? args.U_store : nullptr;
    io.Kn = args.n;
    io.Lfac = MODE == 2 ? args.Lfac : nullptr;
    if (MODE >= 1) {
        io.unom = unom_n ? unom_s : args.u_nom;
        io.iter = (uint32_t)(args.iter_ptr ? *args.iter_ptr : args.iter_val);
        io.key = make_uint2((uint32_t)args.seed, (uint32_t)(args.seed >> 32));
        if (g.sl < d::NU) {
            io.sig = ld_checked(args.sigma, g.sl, d::NU);
            io.lo = M.link[g.sl / NA][g.sl % NA].u_lo;
            io.hi = M.link[g.sl / NA][g.sl % NA].u_hi;
        }
    } else {
        const long long total = (long long)args.n * args.H * d::NU;
        if (args.U_hmajor) {
            io.U = args.U + (size_t)k * d::NU;
            io.u_stride = (long long)args.n * d::NU;
            io.u_ext = total - (long long)k * d::NU;
        } else {
            io.U = args.U + (size_t)k * args.H * d::NU;
            io.u_stride = d::NU;
            io.u_ext = total - (long long)k * args.H * d::NU;
        }
    }
    const float cost = rollout_sample<NA, LPS, MODE, TASK, PLACE>(M, w, g, io);
    if (g.sl == 0 && MPPI_IN_RANGE(k, args.n)) args.costs[k] = cost;
}

namespace rollout_launch {

inline int cuda_fail(cudaError_t e) {
    if (e == cudaSuccess) return MPPI_OK;
    if (e == cudaErrorMemoryAllocation) return MPPI_ERR_OOM;
    return MPPI_ERR_CUDA;
}

template <int NA, int LPS, int MODE, bool TASK, int PLACE>
int launch_t(const RolloutArgs& a, int spc, cudaStream_t s) {
    const int unom = (MODE >= 1 && a.stage_unom) ? a.H * Dims<NA>::NU : 0;
    const size_t sm = rollout_smem<NA, LPS, TASK>(spc, unom);
    auto fn = rollout_kernel<NA, LPS, MODE, TASK, PLACE>;
    int dev = 0, max_sm = 0;
    cudaError_t q = cudaGetDevice(&dev);
    if (q == cudaSuccess) q = cudaDeviceGetAttribute(&max_sm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (q != cudaSuccess) return cuda_fail(q);
    if (!shape_fits<NA, LPS, TASK>(spc, unom, max_sm)) return MPPI_ERR_INVALID_ARG;  // too many samples per CTA
    if (sm > 48 * 1024) {
        cudaError_t e = open_shared_memory(fn);
        if (e != cudaSuccess) return cuda_fail(e);
    }
    const int grid = (a.n + spc - 1) / spc;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(spc * LPS);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = a.pdl ? at : nullptr;
    cfg.numAttrs = a.pdl ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, fn, a);
    return cuda_fail(e != cudaSuccess ? e : cudaGetLastError());
}

template <int NA, int LPS>
int launch_lps(int mode, const RolloutArgs& a, int spc, cudaStream_t s) {
    if (mode == 0) return launch_t<NA, LPS, 0, false, 0>(a, spc, s);
    if (a.Lfac) return a.place ? launch_t<NA, LPS, 2, false, 1>(a, spc, s) : launch_t<NA, LPS, 2, false, 0>(a, spc, s);
    return a.place ? launch_t<NA, LPS, 1, false, 1>(a, spc, s) : launch_t<NA, LPS, 1, false, 0>(a, spc, s);
}

template <int NA, int LPS>
int launch_task(int mode, const RolloutArgs& a, int spc, cudaStream_t s) {
    if (mode == 0) return launch_t<NA, LPS, 0, true, 0>(a, spc, s);
    return a.Lfac ? launch_t<NA, LPS, 2, true, 0>(a, spc, s) : launch_t<NA, LPS, 1, true, 0>(a, spc, s);
}

}  // namespace rollout_launch

// Launch for one arm size.  a.lps (0 = 32) and a.place select the layout;
// spc is rounded up to whole warps.  The ball-task suite runs on 32 or 16
// lanes per sample with the fused placement only.  A shape that shape_fits turns
// down is refused with MPPI_ERR_INVALID_ARG.
template <int NA>
int dispatch_rollout(int mode, const RolloutArgs& a, int spc, cudaStream_t s) {
    using namespace rollout_launch;
    const int lps = a.lps ? a.lps : 32;
    if (lps != 8 && lps != 16 && lps != 32) return MPPI_ERR_INVALID_ARG;
    if (a.place < 0 || a.place > 1) return MPPI_ERR_INVALID_ARG;
    const int spw = 32 / lps;
    spc = (spc + spw - 1) / spw * spw;
    if (spc * lps > 512) return MPPI_ERR_INVALID_ARG;
    if (a.task) {
        if (lps == 8 || a.place != 0) return MPPI_ERR_UNSUPPORTED;
        return lps == 32 ? launch_task<NA, 32>(mode, a, spc, s) : launch_task<NA, 16>(mode, a, spc, s);
    }
    if (lps == 32) return launch_lps<NA, 32>(mode, a, spc, s);
    if (lps == 16) return launch_lps<NA, 16>(mode, a, spc, s);
    if constexpr (Lanes<8>::SEG > NA) return launch_lps<NA, 8>(mode, a, spc, s);
    return MPPI_ERR_UNSUPPORTED;
}

// Samples per CTA for K samples in layout LPS (sampling rollout, fused
// placement).  One wave matters most: every sample runs the same H steps, so
// a partial second wave doubles the time of the samples in it.  So: the
// fewest waves of CTAs over the SMs; within one wave the fewest samples on
// the busiest SM, then the larger CTA (fewer model copies to stage; on
// GB300 a 28-sample CTA per SM beat two 14-sample CTAs by 5%); past one wave
// the most samples resident per SM, then the smaller CTA.  A load of
// five warps of 7-link arms counts as six: a scheduler has two of them either
// way, and in iterations whose launches overlap two five-warp CTAs come to share
// SMs while others idle.  One GB300, us, 10 / 12 samples per CTA on 16 lanes:
// K = 1217 transfer samples x 64 steps 249 / 208 per iteration (199 / 199 for the
// rollout alone), K = 1500 lift x 32 120 / 100; 5 / 6 on 32 lanes: K = 650 transfer
// 213 / 171, lift 106 / 86.
template <int NA, int LPS, bool TASK>
bool spc_occupancy(int spc, int unom_floats, int max_sm, int* per_sm) {
    const auto fn = rollout_kernel<NA, LPS, 1, TASK, 0>;
    const size_t sm = rollout_smem<NA, LPS, TASK>(spc, unom_floats);
    *per_sm = 0;
    return shape_fits<NA, LPS, TASK>(spc, unom_floats, max_sm) &&
           open_shared_memory(fn) == cudaSuccess &&
           cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, fn, spc * LPS, sm) == cudaSuccess && *per_sm > 0;
}

template <int NA>
int choose_spc(int lps, int K, int unom_floats, bool task) {
    int dev = 0, nsm = 0, max_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&max_sm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || nsm <= 0)
        return 4;
    const int spw = 32 / lps;
    long best_w = 1L << 40, best_key = 1L << 40;
    int best = spw;
    for (int spc = spw; spc * lps <= 512; spc += spw) {
        int per_sm = 0;
        bool ok = false;
        if (lps == 32) {
            ok = task ? spc_occupancy<NA, 32, true>(spc, unom_floats, max_sm, &per_sm)
                      : spc_occupancy<NA, 32, false>(spc, unom_floats, max_sm, &per_sm);
        } else if (lps == 16) {
            ok = task ? spc_occupancy<NA, 16, true>(spc, unom_floats, max_sm, &per_sm)
                      : spc_occupancy<NA, 16, false>(spc, unom_floats, max_sm, &per_sm);
        } else if constexpr (Lanes<8>::SEG > NA) {
            ok = !task && spc_occupancy<NA, 8, false>(spc, unom_floats, max_sm, &per_sm);
        }
        if (!ok) continue;
        const long blocks = (K + spc - 1) / spc;
        const long cap = (long)per_sm * nsm;
        const long waves = (blocks + cap - 1) / cap;
        // lower is better: one wave -> load on the busiest SM (ties to the
        // larger CTA below); more -> minus the samples resident per SM
        long key = waves == 1 ? (blocks + nsm - 1) / nsm * spc : -(long)per_sm * spc;
        if (NA == 7 && key == 5 * spw) key = 6 * spw;
        const bool tie_larger = waves == 1;
        if (waves < best_w || (waves == best_w && (key < best_key || (key == best_key && tie_larger)))) {
            best_w = waves;
            best_key = key;
            best = spc;
        }
    }
    return best;
}

// Whether a launch of spc samples per CTA fits one CTA's shared memory.
template <int NA>
bool task_fits(int spc, int unom_floats) {
    int dev = 0, max_sm = 0;
    return cudaGetDevice(&dev) == cudaSuccess &&
           cudaDeviceGetAttribute(&max_sm, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
           shape_fits<NA, 16, true>((spc + 1) / 2 * 2, unom_floats, max_sm);
}

// SMs of the current device, 0 if unknown.
inline int sm_count() {
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    return nsm;
}

// Default layout for K samples: 16 lanes per sample once 32-lane groups would
// take more than 8 warps per SM (7-link arms; 16 for the shorter 3-link steps,
// where 32-lane groups can no longer hold all samples at once), else 32 (the
// shorter per-step chain of one sample per warp).  One GB300, us per iteration
// on 32 / 16 lanes: transfer H = 64, K = 1216 180 / 193, K = 1217 215 / 208,
// K = 1824 224 / 210, K = 2432 260 / 227; lift H = 32, K = 1216 91 / 88, K = 1217
// 108 / 99, K = 2048 129 / 100; planar H = 20, K = 2048 138 / 135, K = 2500
// 220 / 144, K = 4096 277 / 167.
// The ball-task suite forms every pair's distance on 32 lanes but screens the
// pairs on 16, which costs more per step: 16 lanes from 12 samples per SM on
// (H = 32, us on 32 / 16 lanes: transfer K = 1217 172 / 192, K = 1824 181 / 196, K =
// 2048 198 / 195, K = 2500 299 / 222; lift 161 / 176, 171 / 180, 187 / 180, 280 / 205).
inline int default_lps(int na, long long K, bool task = false) {
    const int nsm = sm_count();
    return nsm > 0 && K > (na == 7 ? (task ? 12LL : 8LL) : 16LL) * nsm ? 16 : 32;
}

int launch_rollout_na7(int mode, const RolloutArgs& a, int spc, cudaStream_t s);
int launch_rollout_na3(int mode, const RolloutArgs& a, int spc, cudaStream_t s);
int choose_spc_na7(int lps, int K, int unom_floats, bool task);
int choose_spc_na3(int lps, int K, int unom_floats, bool task);

}  // namespace mppi
