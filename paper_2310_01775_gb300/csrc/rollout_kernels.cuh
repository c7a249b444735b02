// Rollout kernels (single problem, batched class) and their
// launchers, templated on the block count NB and the lanes QL per block
// (block_team.cuh).
#pragma once

#include "block_team.cuh"
#include "rollout.cuh"

namespace stamp {
namespace rollout {

// A launch gives each particle `lanes` lanes; a block team takes at most four
// per block.  Where more were asked for, the other teams of the particle
// shadow it: they compute the same and store nothing but its shared memory.
template <int NB, int QL>
__device__ __forceinline__ bool real_team(int gtid, int lanes) {
    return (gtid & (lanes - 1)) < team_lanes(NB, QL);
}

template <int NB, int QL, bool kRows>
__global__ void __launch_bounds__(128) rollout_fwd_kernel(const SimConst sc, const RolloutArgs a) {
    after_previous();
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x;
    int i = gtid / a.lanes;
    const bool on = i < a.N && real_team<NB, QL>(gtid, a.lanes);
    if (i >= a.N) i = a.N - 1;   // surplus teams shadow the last particle, store nothing
    fwd_block_team<NB, QL, kRows>(sc, a, i, on);
}

// Batched launch: team t -> (instance, particle) through the instances' first
// teams (warp aligned, so a warp never mixes instances); the instance's
// horizon, scene and buffers replace the class-wide constants.  Teams of
// stopped instances return at once.
template <int NB>
__device__ __forceinline__ bool batch_team(const SimConst& sc0, const BatchArgs& b, int t,
                                           SimConst& sc, RolloutArgs& a, int& i, bool& on) {
    if (t >= b.n_teams) return false;
    int lo = 0, hi = b.n_inst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&b.inst[mid].team0) <= t) lo = mid; else hi = mid - 1;
    }
    const BatchInst* in = b.inst + lo;
    if (!__ldg(&b.active[in->gid])) return false;
    sc = sc0;
    sc.H = in->H;
    sc.D = in->D;
    sc.n_ckpt = in->n_ckpt;
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            sc.init[q][c] = in->init[q][c];
            sc.goal[q][c] = in->goal[q][c];
        }
    a = RolloutArgs{};
    a.theta = in->theta;
    a.N = in->N;
    a.seed = in->seed;
    a.iter = b.iter_dev ? *b.iter_dev : b.iter;
    a.hard = b.hard;
    a.tape = in->tape;
    a.cost = in->cost;
    a.grad = in->grad;
    a.dropped = b.dropped;
    i = t - in->team0;
    on = i < in->N;
    if (!on) i = in->N - 1;
    return true;
}

template <int NB, int QL>
__global__ void __launch_bounds__(128) rollout_fwd_batch_kernel(const SimConst sc0, const BatchArgs b) {
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x;
    SimConst sc;
    RolloutArgs a;
    int i;
    bool on;
    if (!batch_team<NB>(sc0, b, gtid / b.lanes, sc, a, i, on)) return;
    on = on && real_team<NB, QL>(gtid, b.lanes);
    fwd_block_team<NB, QL>(sc, a, i, on);
}

template <int NB, int QL>
__global__ void __launch_bounds__(128) rollout_adj_kernel(const SimConst sc, const RolloutArgs a) {
    after_previous();
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x;
    int i = gtid / a.lanes;
    const bool on = i < a.N && real_team<NB, QL>(gtid, a.lanes);
    if (i >= a.N) i = a.N - 1;
    extern __shared__ float2 seg_smem[];
    adj_block_team<NB, QL>(sc, a, i, on,
                           seg_smem + (size_t)(threadIdx.x / a.lanes) * seg_stride<NB>(sc.C));
}

template <int NB, int QL>
__global__ void __launch_bounds__(128) rollout_adj_batch_kernel(const SimConst sc0, const BatchArgs b) {
    const int gtid = blockIdx.x * blockDim.x + threadIdx.x;
    SimConst sc;
    RolloutArgs a;
    int i;
    bool on;
    if (!batch_team<NB>(sc0, b, gtid / b.lanes, sc, a, i, on)) return;
    on = on && real_team<NB, QL>(gtid, b.lanes);
    extern __shared__ float2 seg_smem[];
    adj_block_team<NB, QL>(sc, a, i, on,
                           seg_smem + (size_t)(threadIdx.x / b.lanes) * seg_stride<NB>(sc.C));
}

// ------------------------------ launch --------------------------------------
constexpr size_t kMaxSmem = 227 * 1024;   // of a CTA

template <int NB, int QL>
cudaError_t launch(const SimConst& sc, const RolloutArgs& a, bool adjoint, cudaStream_t st) {
    const long long threads_total = (long long)a.N * a.lanes;
    // spread over the SMs: small CTAs when there are few particles
    const int sms = sm_count();
    int cta = 32;
    while (cta < 128 && threads_total / (cta * 2) >= sms) cta *= 2;
    if (!adjoint) {
        const dim3 grid((unsigned)((threads_total + cta - 1) / cta));
        // one block on two lanes (N = 16384) is the other way round: 123 us, 128 without stores
        if constexpr (NB > 1 || QL == 4)
            if (sc.C > 1 && !a.full)
                return launch_after(rollout_fwd_kernel<NB, QL, false>, grid, cta, 0, st, sc, a);
        return launch_after(rollout_fwd_kernel<NB, QL, true>, grid, cta, 0, st, sc, a);
    }
    // narrow teams with long segments: fewer of them per CTA, so that theirs fit
    const size_t seg = seg_stride<NB>(sc.C) * sizeof(float2);
    while (cta > 32 && cta / a.lanes * seg > kMaxSmem) cta /= 2;
    const int grid = (int)((threads_total + cta - 1) / cta);
    const size_t smem = cta / a.lanes * seg;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(rollout_adj_kernel<NB, QL>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    return launch_after(rollout_adj_kernel<NB, QL>, dim3(grid), cta, smem, st, sc, a);
}

// Batched launch of one block-count class: b.n_teams teams of b.lanes lanes (as
// the kernels number them, shadow teams included) in CTAs of `cta` threads (a
// multiple of 32).
template <int NB, int QL>
cudaError_t launch_batch(const SimConst& sc, const BatchArgs& b, int cta, bool adjoint, cudaStream_t st) {
    const long long threads_total = (long long)b.n_teams * b.lanes;
    const int grid = (int)((threads_total + cta - 1) / cta);
    if (grid < 1) return cudaSuccess;
    if (!adjoint) {
        rollout_fwd_batch_kernel<NB, QL><<<grid, cta, 0, st>>>(sc, b);
    } else {
        const size_t smem = (size_t)(cta / b.lanes) * seg_stride<NB>(sc.C) * sizeof(float2);
        if (smem > 48 * 1024) {
            cudaError_t e = cudaFuncSetAttribute(rollout_adj_batch_kernel<NB, QL>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)smem);
            if (e != cudaSuccess) return e;
        }
        rollout_adj_batch_kernel<NB, QL><<<grid, cta, smem, st>>>(sc, b);
    }
    return cudaGetLastError();
}

// By lanes per particle: 1, 2 or 4 per block.  Four blocks never run on one
// (lanes_supported, default_lanes), and three do only alone, from some count on.
constexpr int lanes_per_block(int nb, int lanes) {
    const int q = lanes / team_groups(nb);
    return q < 4 ? q : 4;
}
template <int NB>
cudaError_t launch_lanes(const SimConst& sc, RolloutArgs a, int lanes, bool adjoint, cudaStream_t st) {
    a.lanes = lanes;
    switch (lanes_per_block(NB, lanes)) {
        case 1:
            if constexpr (NB < 4) return launch<NB, 1>(sc, a, adjoint, st);
            break;
        case 2: return launch<NB, 2>(sc, a, adjoint, st);
        case 4: return launch<NB, 4>(sc, a, adjoint, st);
    }
    return cudaErrorInvalidValue;
}
template <int NB>
cudaError_t launch_batch_lanes(const SimConst& sc, BatchArgs b, int lanes, int cta, bool adjoint,
                               cudaStream_t st) {
    b.lanes = lanes;
    switch (lanes_per_block(NB, lanes)) {
        case 1:
            if constexpr (NB < 3) return launch_batch<NB, 1>(sc, b, cta, adjoint, st);
            break;
        case 2: return launch_batch<NB, 2>(sc, b, cta, adjoint, st);
        case 4: return launch_batch<NB, 4>(sc, b, cta, adjoint, st);
    }
    return cudaErrorInvalidValue;
}
}  // namespace rollout
}  // namespace stamp
