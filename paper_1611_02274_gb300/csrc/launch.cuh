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
    // 6.11; 8,192 grids and 16,384 n-body systems the same; kinetics, 5,000
    // systems of 12 species (more warps than an SM holds blocks) 115.7 / 106.1.
    bool any_block = false;
};

constexpr size_t kSmemPerBlock = 227 * 1024;

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
    const int64_t threads = a.nsys * W;
    const int block = c.any_block && c.mapping == ODE_MAP_THREAD && is_double<typename Method::R>::value ? 32 : c.block;
    const size_t smem = sizeof(float) * Method::SMEM_FLOATS * (size_t)block;
    g_last_launch = LaunchInfo{a.index != nullptr, W, block, c.mapping};
    if (smem > 48 * 1024) {
        // Above the default dynamic shared-memory limit: opt in, always to what
        // the largest block takes (the attribute is the kernel's, and another
        // entry point's thread may launch it with a smaller block in between).
        constexpr size_t kMost = sizeof(float) * Method::SMEM_FLOATS * BODE_MAX_THREADS;
        const size_t limit = smem > kSmemPerBlock ? smem : kMost < kSmemPerBlock ? kMost : kSmemPerBlock;
        cudaError_t e = cudaFuncSetAttribute(k_static<Method, Ctx>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_queue<Method, Ctx>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit);
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
// has the shortest step.  How much filling that takes depends on what a warp
// loses to its longest system: little for grids by RKC, a third to a half of
// the time for RKCK and for chains (whose mu spans more than a grid's
// diffusion), unless the systems of a warp are alike (a batch read through an
// order).  Measured, narrow / wide, by systems (608 sub-partitions):
//   grids by RKC, 1-32 points   1,500: 0.97-1.28   2,500: 0.47-0.75   10,000: 0.18-0.66
//     48, 64 points             1,000: 1.10        2,500: 0.91-1.03   10,000: 0.81
//   grids by RKCK, <= 16        1,500: 0.94-1.59   2,500: 0.53-1.01   10,000: 0.15-0.66
//     24-64, in order / not     5,000: 0.84-0.89 / 1.08-1.23
//   chains by RKC, <= 16        2,500: 1.0-1.34    5,000: 0.70-0.88   10,000: 0.42-0.68
//     24-64, in order / not     5,000: 0.80-0.87 / 1.06-1.12
//   chains by RKCK, <= 8        5,000: 1.0-1.06    7,000: 0.79-0.87
//     in order, 12-32 / 48, 64  5,000: 1.2 / 0.9   7,000: 0.98 / 0.8  10,000: 0.73-0.91 / 0.8
inline int grid_team_f64(int npts, int64_t nsys, int sm_count, bool chain, int method, bool ordered) {
    int w = 1;
    while (w < 32 && 4 * w < npts) w *= 2;
    const double wide = (double)nsys / (4 * sm_count), narrow = wide * w / 32;  // rounds of warps
    const bool rkck = method == kMethodRkck;
    bool take;
    if (!chain && !rkck)
        take = wide >= 4;
    else if (ordered && narrow >= 2)
        take = !(chain && rkck) || narrow >= 2.8 || wide >= 11;
    else if (!chain)
        take = w <= 4 && wide >= 4;
    else
        take = rkck ? w <= 2 && wide >= 11 : w <= 4 && wide >= 8;
    return take ? w : 32;
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
