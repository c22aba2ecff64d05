// launch.cuh -- batched kernels over the per-system state machines and the
// host-side launcher they share.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"
#include "kernels.cuh"
#include "team.cuh"

namespace bode {

// Registered right-hand side (host copy).
struct RhsEntry {
    int32_t kind;
    int32_t neq;
    int32_t n_params;
    MassActionNet net;
    double bruss_A, bruss_B, bruss_ubc, bruss_vbc;
    double coupling;
    double masses[kMaxBodies];
    KinDevice kin;          // device mechanism (ODE_RHS_KINETICS), freed at release
    void* kin_alloc;        // the one device allocation behind kin
};

// Launch configuration resolved by the API layer.
struct LaunchCfg {
    int mapping;     // ODE_MAP_THREAD or ODE_MAP_QUEUE
    int block;       // threads per block
    int team;        // requested lanes per system (0 = family default; 32 keeps grids at a warp per system)
    int sm_count;
    cudaStream_t stream;
    // the block size is neither the caller's nor timed: a one-launch kernel of
    // the plain form then takes a warp per block.  Its warps share nothing,
    // the FP64 pipe is what they wait for, a warp alone on its SM issues an
    // FP64 instruction every 64 cycles where four take 76 each, and four-warp
    // blocks leave a batch of a few warps per SM unevenly spread.  Measured,
    // 128 / 32 threads: kinetics, 1,000 systems 94.9 / 83.2 ms; 32-point
    // grids, 2,500 systems 26.0 / 18.6; van der Pol, 30,000 systems 7.04 /
    // 6.11; 8,192 grids and 16,384 n-body systems the same.
    bool any_block = false;
};

// What the calling thread's last launch took (bode_last_launch).
struct LaunchInfo {
    int32_t ordered = 0;  // systems read through an order or a plan's index
    int32_t lanes = 0, block = 0, mapping = 0;
};
inline thread_local LaunchInfo g_last_launch;

template <class T>
struct is_double {
    static constexpr bool value = false;
};
template <>
struct is_double<double> {
    static constexpr bool value = true;
};

template <class Method, class Ctx>
cudaError_t launch_method(const BatchArgs& a, const Ctx& ctx, const LaunchCfg& c) {
    constexpr int W = Method::W;
    const int block = c.any_block && c.mapping == ODE_MAP_THREAD && is_double<typename Method::R>::value ? 32 : c.block;
    const size_t smem = sizeof(float) * Method::SMEM_FLOATS * (size_t)block;
    const int64_t threads = a.nsys * W;
    g_last_launch = LaunchInfo{a.index != nullptr, W, block, c.mapping};
    if (smem > 48 * 1024) {  // above the default dynamic shared-memory limit: opt in
        cudaError_t e = cudaFuncSetAttribute(k_static<Method, Ctx>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_queue<Method, Ctx>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    if (c.mapping == ODE_MAP_QUEUE) {
        int per_sm = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_queue<Method, Ctx>, block, smem);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) per_sm = 1;
        int64_t grid = (int64_t)per_sm * c.sm_count;
        const int64_t need = (threads + block - 1) / block;
        if (grid > need) grid = need;
        BatchArgs q = a;
        q.warp_sched = 1;
        k_queue<Method, Ctx><<<(unsigned)grid, block, smem, c.stream>>>(q, ctx);
    } else {
        const int64_t grid = (threads + block - 1) / block;
        k_static<Method, Ctx><<<(unsigned)grid, block, smem, c.stream>>>(a, ctx);
    }
    return cudaGetLastError();
}

enum { kMethodRkck = 0, kMethodRkc = 1 };

// Lanes per system of the plain form's grid families (Brusselator grids,
// oscillator chains).  The FP64 pipe bounds them, and a warp pays for an
// FP64 instruction whatever its active lanes: the per-system part of a step
// (controller, logarithm and powers, the norm's sequential sum) costs a warp
// with four systems in it as much as a warp with one.  So where the batch
// fills the GPU a system takes as few lanes as hold it at four points each
// (more points a lane spill), and where it does not, a whole warp, which
// has the shortest step.  Time is taken as rounds of warps over the SMs'
// four sub-partitions times a step's FP64 work, in units of one point's:
// G points a lane plus kOwn + kSum npts for the system (from the FP64
// instruction counts of an RKC step: 150 a point, 110 a system and two per
// point in the norm).  Measured on 32 points: 8,192 systems 68.3 ms wide,
// 52.5 narrow; 608 systems wide 6.3 ms, where a round of the narrow kernel
// takes 15.4.
inline int grid_team_f64(int npts, int64_t nsys, int sm_count) {
    constexpr double kOwn = 0.75, kSum = 0.0133;
    int w = 1;
    while (w < 32 && 4 * w < npts) w *= 2;
    const int64_t slots = 4 * (int64_t)sm_count;
    auto rounds = [&](int lanes) { return (double)(((nsys * lanes + 31) / 32 + slots - 1) / slots); };
    const double system = kOwn + kSum * npts;
    const double narrow = rounds(w) * (4.0 + system), wide = rounds(32) * ((npts + 31) / 32 + system);
    return narrow < wide ? w : 32;
}

// Per-family dispatch (defined in k_*.cu).  Each sets *ok = false when the
// family / size / precision / mapping combination is not built.
cudaError_t launch_vdp(int method, int prec, const RhsEntry& r, const BatchArgs& a, const LaunchCfg& c, bool* ok);
cudaError_t launch_mass(int method, int prec, const RhsEntry& r, const BatchArgs& a, const LaunchCfg& c, bool* ok);
cudaError_t launch_bruss(int method, int prec, const RhsEntry& r, const BatchArgs& a, const LaunchCfg& c, bool* ok);
cudaError_t launch_chain(int method, int prec, const RhsEntry& r, const BatchArgs& a, const LaunchCfg& c, bool* ok);
cudaError_t launch_nbody(int method, int prec, const RhsEntry& r, const BatchArgs& a, const LaunchCfg& c, bool* ok);
cudaError_t launch_kinetics(int method, int prec, const RhsEntry& r, const BatchArgs& a, const LaunchCfg& c, bool* ok);

// Builds the RKC stage-coefficient tables on the current device.
cudaError_t build_rkc_tables(double* tab64, float4* tab32, int mmax, cudaStream_t s);

}  // namespace bode
