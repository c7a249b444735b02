// The surrogate's rollout in one launch each way: every push of a plan needs
// only that plan's poses, so a CTA takes a 128-row tile through all of them.
//
// Forward, per push: layer 0 reads the push's features (BF16, written straight
// into its K-major operand), the layers run as in mlp_fwd_kernel, and the
// head's epilogue moves the poses it holds in registers and writes the next
// push's pose features.  The action's features (softmax, tanh, sigmoid) do
// not depend on the poses: four warps compute the next push's beside the
// layer-1 MMA.  What it replaces, per push at 131072 rows on GB300: features
// 40 us, packing 13.5, MLP 88, unpacking 6; at 2048 rows 8 + 3 + 18 + 3, and
// the launches between them; six pushes of 131072 rows take 548 us here, of 2048
// rows 95 (and 97 in reverse, where the 12 launches took 155).
// Reverse, per push: the pose adjoints (in registers) are the head's dy; the
// input-gradient chain of mlp_bwd_kernel; the features' reverse on the row.
//
// The arithmetic of every stage is that of the kernels it replaces.
#include "mlp_tc.cuh"
#include "rollout.cuh"
#include "stamp_internal.cuh"
#include "surrogate_mlp.cuh"

namespace stamp {
namespace mlp {
namespace {

struct SurSmem {
    alignas(128) unsigned char act[kActBytes];
    alignas(128) unsigned char w[kWBytes];
    alignas(128) unsigned char x[kInBytes];   // a push's features: layer 0's A operand
    uint64_t tma_bar, mma_bar;
    unsigned tmem_slot;
};

__device__ __forceinline__ void put_bf16(unsigned char* tile, int row, int col, float v) {
    *reinterpret_cast<__nv_bfloat16*>(tile + tile_off(row, col, kIn)) = __float2bfloat16_rn(v);
}

// Push k's action features of plan i into row `row` of the tile (zero for a
// row past the plans), and what the cost and the reverse sweep need of them.
template <int NB>
__device__ __forceinline__ void action_features(const SimConst& sc, const SurArgs& a, int i, bool on,
                                                int k, uint64_t gkey, unsigned char* tile, int row) {
    constexpr int M = rollout::Dims<NB>::M, P = M + 2;
    float f[P];
#pragma unroll
    for (int c = 0; c < P; ++c) f[c] = 0.f;
    if (on) {
        float z[M], uu, vv;
        rollout::relax_action<NB>(sc, a.theta + (size_t)i * sc.D, k, i, gkey, a.iter >= 0, false, z, uu, vv);
#pragma unroll
        for (int c = 0; c < M; ++c) f[c] = z[c];
        f[M] = tanhf(uu);
        f[M + 1] = rollout::sigmoidf_(vv);
        float* r = a.relax + ((size_t)i * sc.H + k) * P;
        if (a.zsave) {
#pragma unroll
            for (int c = 0; c < P; ++c) r[c] = f[c];
        } else {
            r[M + 1] = f[M + 1];   // the cost's push lengths
        }
    }
#pragma unroll
    for (int c = 0; c < P; ++c) put_bf16(tile, row, 4 * NB + c, f[c]);
}

template <int NB>
__device__ __forceinline__ void pose_features(const float (&q)[3 * NB], bool on, unsigned char* tile,
                                              int row) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        float sn, cs;
        sincosf(q[3 * b + 2], &sn, &cs);
        put_bf16(tile, row, 4 * b, on ? q[3 * b] : 0.f);
        put_bf16(tile, row, 4 * b + 1, on ? q[3 * b + 1] : 0.f);
        put_bf16(tile, row, 4 * b + 2, on ? cs : 0.f);
        put_bf16(tile, row, 4 * b + 3, on ? sn : 0.f);
    }
}

template <int NB>
__global__ void __launch_bounds__(kThreads, 1) sur_fwd_kernel(const SimConst sc, const SurArgs a) {
    constexpr int S3 = 3 * NB;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    SurSmem& sm = *reinterpret_cast<SurSmem*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        mbar_init(&sm.tma_bar, 1);
        mbar_init(&sm.mma_bar, 1);
        fence_async_shared();
    }
    if (warp == 0) tmem_alloc(&sm.tmem_slot, kTmemCols);
    for (int t = tid * 16; t < (int)kInBytes; t += kThreads * 16)   // the unused columns stay zero
        *reinterpret_cast<uint4*>(sm.x + t) = make_uint4(0, 0, 0, 0);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = sm.tmem_slot;
    // warp w: TMEM lane quarter w % 4, column part w / 4; part 0 holds the rows' poses
    const int quarter = warp & 3, part = warp >> 2, row = quarter * 32 + lane;
    const unsigned lane_base = tmem + ((unsigned)(quarter * 32) << 16);
    const uint64_t gkey = a.iter >= 0 ? sm64(sm64(a.seed, kStreamGumbel), (uint64_t)a.iter) : 0ull;
    unsigned tma_phase = 0, mma_phase = 0;
    bool failed = false, tma_pending = false, mma_pending = false;
    auto issue_load = [&](int l) {   // layer l's weights into shared memory
        const unsigned wbytes = (unsigned)(layer_n(l) * layer_k(l) * 2);
        mbar_expect_tx(&sm.tma_bar, wbytes);
        tma_load_1d(sm.w, a.w_tiled + layer_w_offset(l), wbytes, &sm.tma_bar);
    };
    if (blockIdx.x < a.n_tiles) {
        if (tid == 0) issue_load(0);
        tma_pending = true;
    }
    for (int tile = blockIdx.x; tile < a.n_tiles && !failed; tile += gridDim.x) {
        const int i = tile * kRows + row;
        const bool on = i < a.N;
        float q[S3];
#pragma unroll
        for (int t = 0; t < S3; ++t) q[t] = sc.init[t / 3][t % 3];
        if (part == 0) {
            pose_features<NB>(q, on, sm.x, row);
            if (on && (a.zsave || sc.H == 1))
#pragma unroll
                for (int t = 0; t < S3; ++t) a.pose[(size_t)i * S3 + t] = q[t];
        } else if (part == 1) {
            action_features<NB>(sc, a, i, on, 0, gkey, sm.x, row);
        }
        fence_async_shared();
        __syncthreads();
        for (int k = 0; k < sc.H && !failed; ++k)
            for (int l = 0; l < 4 && !failed; ++l) {
                const int K = layer_k(l), N = layer_n(l);
                const size_t slot = (size_t)k * a.n_tiles + tile;
                unsigned spins = 0;
                bool ok = true;
                while (!(ok = mbar_try_wait(&sm.tma_bar, tma_phase)) && ++spins < kWaitLimit) {
                }
                if (__syncthreads_or(!ok)) { failed = true; break; }   // the copy stays pending
                tma_phase ^= 1u;
                tma_pending = false;
                if (tid == 0) {
                    tc_fence_after();
                    const uint32_t idesc = idesc_bf16(kRows, N);
                    const unsigned char* A = l == 0 ? sm.x : sm.act;
                    for (int kk = 0; kk < K / 16; ++kk)
                        mma_bf16(tmem, smem_desc(A + kk * 256, 128, (K / 8) * 128),
                                 smem_desc(sm.w + kk * 256, 128, (K / 8) * 128), idesc, kk > 0);
                    mma_commit(&sm.mma_bar);
                }
                mma_pending = true;
                // layer 0 has read the push's features: the next push's, beside this MMA
                if (l == 1 && part == 1 && k + 1 < sc.H)
                    action_features<NB>(sc, a, i, on, k + 1, gkey, sm.x, row);
                spins = 0;
                while (!(ok = mbar_try_wait(&sm.mma_bar, mma_phase)) && ++spins < kWaitLimit) {
                }
                if (__syncthreads_or(!ok)) { failed = true; break; }   // the MMA stays pending
                mma_phase ^= 1u;
                mma_pending = false;
                tc_fence_after();
                // the weight buffer is free: the next layer's copy runs beside this epilogue
                if (l < 3 || k + 1 < sc.H || tile + (int)gridDim.x < a.n_tiles) {
                    if (tid == 0) {
                        fence_async_shared();
                        issue_load(l < 3 ? l + 1 : 0);
                    }
                    tma_pending = true;
                }
                const float* bl = a.bias + l * kHidden;
                if (l < 3) {
                    for (int c0 = part * (N / kParts); c0 < (part + 1) * (N / kParts); c0 += 32) {
                        float v[32];
                        tmem_ld32(lane_base + c0, v);
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            uint4 pk, pz;
                            unsigned* pw = reinterpret_cast<unsigned*>(&pk);
                            unsigned* pzw = reinterpret_cast<unsigned*>(&pz);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const int c = c0 + g * 8 + 2 * e;
                                const float z0 = v[g * 8 + 2 * e] + __ldg(bl + c);
                                const float z1 = v[g * 8 + 2 * e + 1] + __ldg(bl + c + 1);
                                pw[e] = pack_bf16(silu(z0), silu(z1));
                                pzw[e] = pack_bf16(z0, z1);
                            }
                            const unsigned off = tile_off(row, c0 + g * 8, kHidden);
                            *reinterpret_cast<uint4*>(sm.act + off) = pk;
                            if (a.zsave)   // pre-activation of layer l, for the reverse sweep
                                *reinterpret_cast<uint4*>(
                                    a.zsave + ((size_t)l * a.tile_cap + slot) * kActBytes + off) = pz;
                        }
                    }
                } else if (part == 0) {
                    float v[16];
                    tmem_ld16(lane_base, v);
                    float d[S3];
#pragma unroll
                    for (int t = 0; t < S3; ++t) d[t] = v[t] + __ldg(bl + t);
                    if (k + 1 == sc.H) {   // the cost adds the last pose change itself
                        if (on)
#pragma unroll
                            for (int t = 0; t < S3; ++t) a.y[(size_t)i * S3 + t] = d[t];
                    } else {
#pragma unroll
                        for (int t = 0; t < S3; ++t) q[t] += d[t];
                        if (on && (a.zsave || k + 2 == sc.H))
#pragma unroll
                            for (int t = 0; t < S3; ++t)
                                a.pose[((size_t)(k + 1) * a.N + i) * S3 + t] = q[t];
                        pose_features<NB>(q, on, sm.x, row);
                    }
                }
                // the next MMA reads act / x (written here) and overwrites TMEM (read here)
                fence_async_shared();
                tc_fence_before();
                __syncthreads();
            }
    }
    if (failed && tid == 0) {
        atomicOr(a.err, 2);
        // a last bounded wait for what is still in flight before the tensor memory is released
        if (tma_pending)
            for (unsigned w = 0; w < kWaitLimit && !mbar_try_wait(&sm.tma_bar, tma_phase); ++w) {
            }
        if (mma_pending)
            for (unsigned w = 0; w < kWaitLimit && !mbar_try_wait(&sm.mma_bar, mma_phase); ++w) {
            }
    }
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

// Reverse of one push's features on row i: di = dC/df, the pose adjoint is
// advanced from q_{k+1} to q_k, and grad log rho of the push's parameters
// written (with the push-length term).
template <int NB>
__device__ __forceinline__ void features_reverse(const SimConst& sc, const SurArgs& a, int i, int k,
                                                 const float* di, float (&ai)[3 * NB]) {
    constexpr int M = rollout::Dims<NB>::M, P = M + 2;
    const float* pi = a.pose + ((size_t)k * a.N + i) * 3 * NB;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        float sn, cs;
        sincosf(pi[3 * b + 2], &sn, &cs);
        ai[3 * b] += di[4 * b];
        ai[3 * b + 1] += di[4 * b + 1];
        ai[3 * b + 2] += cs * di[4 * b + 3] - sn * di[4 * b + 2];
    }
    const float* ri = a.relax + ((size_t)i * sc.H + k) * P;
    float r[P], zg = 0.f;
#pragma unroll
    for (int c = 0; c < P; ++c) r[c] = ri[c];
#pragma unroll
    for (int c = 0; c < M; ++c) zg += r[c] * di[4 * NB + c];
    float* gi = a.grad + (size_t)i * sc.D + k * P;
    // softmax((a+g)/tau): dC/da_j = z_j (dC/dz_j - sum_c z_c dC/dz_c) / tau
#pragma unroll
    for (int c = 0; c < M; ++c) gi[c] = -(r[c] * (di[4 * NB + c] - zg) * sc.inv_tau);
    const float tu = r[M], sv = r[M + 1];
    gi[M] = -(di[4 * NB + M] * (1.f - tu * tu));
    const float dist = sc.dist_max * sv;
    gi[M + 1] = -((di[4 * NB + M + 1] + 2.f * sc.w_push * dist * sc.dist_max) * sv * (1.f - sv));
}

template <int NB>
__global__ void __launch_bounds__(kThreads, 1) sur_bwd_kernel(const SimConst sc, const SurArgs a) {
    constexpr int S3 = 3 * NB;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    FwdSmem& sm = *reinterpret_cast<FwdSmem*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        mbar_init(&sm.tma_bar, 1);
        mbar_init(&sm.mma_bar, 1);
        fence_async_shared();
    }
    if (warp == 0) tmem_alloc(&sm.tmem_slot, kTmemCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = sm.tmem_slot;
    const int quarter = warp & 3, part = warp >> 2, row = quarter * 32 + lane;
    const unsigned lane_base = tmem + ((unsigned)(quarter * 32) << 16);
    unsigned tma_phase = 0, mma_phase = 0;
    bool failed = false, tma_pending = false, mma_pending = false;
    auto issue_load = [&](int m) {   // W_m^T into shared memory
        const unsigned wbytes = (unsigned)(layer_k(m) * layer_n(m) * 2);
        mbar_expect_tx(&sm.tma_bar, wbytes);
        tma_load_1d(sm.w, a.wt_tiled + layer_w_offset(m), wbytes, &sm.tma_bar);
    };
    if (blockIdx.x < a.n_tiles) {
        if (tid == 0) issue_load(3);
        tma_pending = true;
    }
    for (int tile = blockIdx.x; tile < a.n_tiles && !failed; tile += gridDim.x) {
        const int i = tile * kRows + row;
        const bool on = i < a.N;
        float ap[S3];   // dC/dq_{k+1} (part 0)
#pragma unroll
        for (int t = 0; t < S3; ++t) ap[t] = part == 0 && on ? a.apose[(size_t)i * S3 + t] : 0.f;
        for (int k = sc.H - 1; k >= 0 && !failed; --k) {
            const size_t slot = (size_t)k * a.n_tiles + tile;
            if (part == 0) {   // dz_3 = dy = dC/dq_{k+1}: a BF16 K-major tile of 16 columns
                float d[kOut];
#pragma unroll
                for (int c = 0; c < kOut; ++c) d[c] = c < S3 ? ap[c < S3 ? c : 0] : 0.f;
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    uint4 pk;
                    unsigned* pw = reinterpret_cast<unsigned*>(&pk);
#pragma unroll
                    for (int e = 0; e < 4; ++e) pw[e] = pack_bf16(d[g * 8 + 2 * e], d[g * 8 + 2 * e + 1]);
                    *reinterpret_cast<uint4*>(sm.act + tile_off(row, g * 8, kOut)) = pk;
                }
            }
            fence_async_shared();
            __syncthreads();
            for (int m = 3; m >= 0 && !failed; --m) {
                const int Kb = layer_n(m), Nb = layer_k(m);   // da_m = dz_m (., Kb) W_m (Kb, Nb)
                unsigned spins = 0;
                bool ok = true;
                while (!(ok = mbar_try_wait(&sm.tma_bar, tma_phase)) && ++spins < kWaitLimit) {
                }
                if (__syncthreads_or(!ok)) { failed = true; break; }
                tma_phase ^= 1u;
                tma_pending = false;
                if (tid == 0) {
                    tc_fence_after();
                    const uint32_t idesc = idesc_bf16(kRows, Nb);
                    for (int kk = 0; kk < Kb / 16; ++kk)
                        mma_bf16(tmem, smem_desc(sm.act + kk * 256, 128, (Kb / 8) * 128),
                                 smem_desc(sm.w + kk * 256, 128, (Kb / 8) * 128), idesc, kk > 0);
                    mma_commit(&sm.mma_bar);
                }
                mma_pending = true;
                spins = 0;
                while (!(ok = mbar_try_wait(&sm.mma_bar, mma_phase)) && ++spins < kWaitLimit) {
                }
                if (__syncthreads_or(!ok)) { failed = true; break; }
                mma_phase ^= 1u;
                mma_pending = false;
                tc_fence_after();
                if (m > 0 || k > 0 || tile + (int)gridDim.x < a.n_tiles) {
                    if (tid == 0) {
                        fence_async_shared();
                        issue_load(m > 0 ? m - 1 : 3);
                    }
                    tma_pending = true;
                }
                if (m > 0) {
                    const unsigned char* zt = a.zsave + ((size_t)(m - 1) * a.tile_cap + slot) * kActBytes;
                    for (int c0 = part * (kHidden / kParts); c0 < (part + 1) * (kHidden / kParts); c0 += 32) {
                        float v[32];
                        tmem_ld32(lane_base + c0, v);
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            const unsigned off = tile_off(row, c0 + g * 8, kHidden);
                            const uint4 zq = *reinterpret_cast<const uint4*>(zt + off);
                            const unsigned zw[4] = {zq.x, zq.y, zq.z, zq.w};
                            uint4 pk;
                            unsigned* pw = reinterpret_cast<unsigned*>(&pk);
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                pw[e] = pack_bf16(v[g * 8 + 2 * e] * silu_grad(bf_lo(zw[e])),
                                                  v[g * 8 + 2 * e + 1] * silu_grad(bf_hi(zw[e])));
                            *reinterpret_cast<uint4*>(sm.act + off) = pk;
                        }
                    }
                } else if (part == 0) {
                    float v[32];
                    tmem_ld32(lane_base, v);
                    if (on) features_reverse<NB>(sc, a, i, k, v, ap);
                }
                fence_async_shared();
                tc_fence_before();
                __syncthreads();
            }
        }
    }
    if (failed && tid == 0) {
        atomicOr(a.err, 2);
        if (tma_pending)
            for (unsigned w = 0; w < kWaitLimit && !mbar_try_wait(&sm.tma_bar, tma_phase); ++w) {
            }
        if (mma_pending)
            for (unsigned w = 0; w < kWaitLimit && !mbar_try_wait(&sm.mma_bar, mma_phase); ++w) {
            }
    }
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

template <int NB>
cudaError_t launch(const SimConst& sc, const SurArgs& a, bool reverse, int sms, cudaStream_t st) {
    const size_t smem = (reverse ? sizeof(FwdSmem) : sizeof(SurSmem)) + 1024;
    auto* kernel = reverse ? sur_bwd_kernel<NB> : sur_fwd_kernel<NB>;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<a.n_tiles < sms ? a.n_tiles : sms, kThreads, smem, st>>>(sc, a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t surrogate_pass(const SimConst& sc, const SurArgs& a, bool reverse, int sms, cudaStream_t st) {
    switch (sc.nb) {
        case 1: return launch<1>(sc, a, reverse, sms, st);
        case 2: return launch<2>(sc, a, reverse, sms, st);
        case 3: return launch<3>(sc, a, reverse, sms, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace mlp
}  // namespace stamp
