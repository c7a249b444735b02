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
// the launches between them; six pushes of 131072 rows take 530 us here.  Few
// plans would leave most SMs idle (2048 rows: 16 tiles, 95 us, and 97 in reverse):
// they go to the cluster kernels below (36 and 37 us).
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

// All pushes' action features of plans i0 ... i0 + rows - 1 to a.relax, by all
// threads of a cluster: (push, plan) pairs n0, n0 + step, ...
template <int NB>
__device__ __forceinline__ void all_action_features(const SimConst& sc, const SurArgs& a, int i0, int rows,
                                                    uint64_t gkey, int n0, int step) {
    constexpr int M = rollout::Dims<NB>::M, P = M + 2;
    for (int n = n0; n < sc.H * rows; n += step) {
        const int k = n / rows, i = i0 + n % rows;
        if (i >= a.N) continue;
        float z[M], uu, vv;
        rollout::relax_action<NB>(sc, a.theta + (size_t)i * sc.D, k, i, gkey, a.iter >= 0, false, z, uu, vv);
        float* r = a.relax + ((size_t)i * sc.H + k) * P;
#pragma unroll
        for (int c = 0; c < M; ++c) r[c] = z[c];
        r[M] = tanhf(uu);
        r[M + 1] = rollout::sigmoidf_(vv);
    }
}
// Push k's, from there, into row `row` of the tile.
template <int NB>
__device__ __forceinline__ void stored_features(const SimConst& sc, const SurArgs& a, int i, bool on, int k,
                                                unsigned char* tile, int row) {
    constexpr int P = rollout::Dims<NB>::M + 2;
    const float* r = a.relax + ((size_t)i * sc.H + k) * P;
#pragma unroll
    for (int c = 0; c < P; ++c) put_bf16(tile, row, 4 * NB + c, on ? r[c] : 0.f);
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
                    mma_tile(tmem, l == 0 ? sm.x : sm.act, sm.w, K, N);
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
// written (with the push-length term).  load() reads what it needs, beside an MMA.
template <int NB>
struct FeaturesReverse {
    static constexpr int M = rollout::Dims<NB>::M, P = M + 2;
    float sn[NB], cs[NB], r[P];
    __device__ __forceinline__ void load(const SimConst& sc, const SurArgs& a, int i, int k) {
        const float* pi = a.pose + ((size_t)k * a.N + i) * 3 * NB;
        const float* ri = a.relax + ((size_t)i * sc.H + k) * P;
#pragma unroll
        for (int c = 0; c < P; ++c) r[c] = ri[c];
#pragma unroll
        for (int b = 0; b < NB; ++b) sincosf(pi[3 * b + 2], &sn[b], &cs[b]);
    }
    __device__ __forceinline__ void apply(const SimConst& sc, const SurArgs& a, int i, int k, const float* di,
                                          float (&ai)[3 * NB], bool store) const {
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            ai[3 * b] += di[4 * b];
            ai[3 * b + 1] += di[4 * b + 1];
            ai[3 * b + 2] += cs[b] * di[4 * b + 3] - sn[b] * di[4 * b + 2];
        }
        if (!store) return;
        float zg = 0.f;
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
};

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
                    mma_tile(tmem, sm.act, sm.w, Kb, Nb);
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
                    if (on) {
                        FeaturesReverse<NB> f;
                        f.load(sc, a, i, k);
                        f.apply(sc, a, i, k, v, ap, true);
                    }
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

// Few plans: two CTAs of a cluster take TR (32 or 64) rows, so that 2048 rows use
// 128 SMs where 128-row tiles use 16, and the weights stay in shared memory.
// The roles of the operands are swapped: M = 128 of a hidden layer's units per
// CTA, N = the rows, so a narrow N costs less and nothing is computed for
// padding.  A hidden output is stored as the N-major operand it comes out as
// (TMEM lane = unit, column = row: a thread holds 8 rows of a unit, 16 bytes of
// an 8 x 8 core matrix; row groups 128 B apart, unit groups TR * 16 B): the CTA's
// 128 units are contiguous and go to the peer by bulk copies between the shared
// memories that complete on the receiver's barrier.  The head (and the reverse's
// input gradient) takes the rows as M instead, a thread per row; both CTAs
// compute it, the poses and the features, so nothing else is exchanged.  Two
// output buffers in turn: who has the peer's half of an output knows that the
// peer has read the one before, which is what the next write replaces.
template <int TR>
struct SurClSmem {
    alignas(128) unsigned char act[2][kHidden * TR * 2];
    alignas(128) unsigned char x[TR * kIn * 2];             // features, or dz_3: K-major
    alignas(128) unsigned char w_in[kIn * kHidden * 2];     // forward: half of layer 0; reverse: W_0^T
    alignas(128) unsigned char w_out[kOut * kHidden * 2];   // forward: the head; reverse: half of W_3^T
    alignas(128) unsigned char w_mid[2][kHidden / 2 * kHidden * 2];
    uint64_t w_bar, mma_bar, in_bar[2];
    unsigned tmem_slot;
};
constexpr int kUnits = kHidden / 2;   // of a CTA
constexpr unsigned kClCols = 64;

// One CTA's side of the cluster.
template <int TR>
struct ClusterSide {
    static constexpr int kGroups = TR / 8 / kParts;          // row groups of a thread
    static constexpr unsigned kUnitGroup = TR / 8 * 128;     // bytes of 8 units
    static constexpr unsigned kHalf = kUnits / 8 * kUnitGroup;
    SurClSmem<TR>& sm;
    const unsigned rank = async::cluster_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // hidden layers: unit `unit` of this CTA, row groups part * kGroups ...
    const int quarter = warp & 3, part = warp >> 2, unit = quarter * 32 + lane;
    unsigned tmem = 0, out = 0, mma_phase = 0;   // out: hidden outputs so far
    bool w_ready = false, in_pending = false, mma_pending = false;

    __device__ explicit ClusterSide(SurClSmem<TR>& s) : sm(s) {
        if (tid == 0) {
            mbar_init(&sm.w_bar, 1);
            mbar_init(&sm.mma_bar, 1);
            mbar_init(&sm.in_bar[0], 1);
            mbar_init(&sm.in_bar[1], 1);
            async::fence_mbar_init();
            fence_async_shared();
        }
        if (warp == 0) tmem_alloc(&sm.tmem_slot, kClCols);
        // the features' unused columns stay zero, and so do the rows past TR that the
        // row-major products read (their results are not used)
        for (int t = tid * 16; t < (int)(sizeof sm.act + sizeof sm.x); t += kThreads * 16)
            *reinterpret_cast<uint4*>(sm.act[0] + t) = make_uint4(0, 0, 0, 0);
        tc_fence_before();
        async::cluster_sync();
        tc_fence_after();
        tmem = sm.tmem_slot;
    }
    __device__ unsigned lane_base() const { return tmem + ((unsigned)(quarter * 32) << 16); }
    __device__ static bool wait(uint64_t* bar, unsigned parity) {
        for (unsigned w = 0; w < kWaitLimit; ++w)
            if (mbar_try_wait(bar, parity)) return true;
        return false;
    }
    // units x rows: W (128 units, K-major) times x (K columns) or the last output.
    // rows x N: the last output times W (N units, K-major), when rows_first.
    // False (in every thread): a wait gave up.
    __device__ bool multiply(const unsigned char* W, int from_x_columns, int rows_first_units) {
        bool ok = w_ready || wait(&sm.w_bar, 0);
        if (!from_x_columns) ok = ok && wait(&sm.in_bar[(out - 1) & 1], ((out - 1) >> 1) & 1);
        if (__syncthreads_or(!ok)) return false;   // the copies stay pending
        w_ready = true;
        in_pending = false;
        if (tid == 0) {
            tc_fence_after();
            if (from_x_columns) {
                mma_tile(tmem, W, sm.x, from_x_columns, TR);
            } else {
                const uint64_t dw = smem_desc(W, 128, (kHidden / 8) * 128);
                const uint64_t da = smem_desc(sm.act[(out - 1) & 1], kUnitGroup, 128);
                if (rows_first_units) {
                    const uint32_t idesc = idesc_bf16(kRows, rows_first_units) | (1u << 15);   // A: M-major
#pragma unroll
                    for (int kk = 0; kk < kHidden / 16; ++kk)
                        mma_bf16(tmem, da + kk * (2 * kUnitGroup >> 4), dw + kk * 16, idesc, kk > 0);
                } else {
                    const uint32_t idesc = idesc_bf16(kRows, TR) | (1u << 16);   // B: N-major
#pragma unroll
                    for (int kk = 0; kk < kHidden / 16; ++kk)
                        mma_bf16(tmem, dw + kk * 16, da + kk * (2 * kUnitGroup >> 4), idesc, kk > 0);
                }
            }
            mma_commit(&sm.mma_bar);
        }
        mma_pending = true;
        return true;
    }
    __device__ bool product_done() {
        const bool ok = wait(&sm.mma_bar, mma_phase);
        if (__syncthreads_or(!ok)) return false;   // the MMA stays pending
        mma_phase ^= 1u;
        mma_pending = false;
        tc_fence_after();
        return true;
    }
    // this thread's rows of its unit, from the product
    __device__ void read(float (&v)[8 * kGroups]) const {
        if constexpr (kGroups == 1) tmem_ld8(lane_base() + part * 8, v);
        else tmem_ld16(lane_base() + part * 16, v);
    }
    // before this layer's epilogue: the bytes that the peer will send; where this thread writes
    __device__ unsigned char* begin_output() {
        if (tid == 0) mbar_expect_tx(&sm.in_bar[out & 1], kHalf);
        in_pending = true;
        return sm.act[out & 1] + rank * kHalf + (unit >> 3) * kUnitGroup + part * kGroups * 128 + (unit & 7) * 16;
    }
    // after it: the four warps of 32 units are done, and one thread sends these to the peer
    __device__ void send_output() {
        fence_async_shared();
        tc_fence_before();
        asm volatile("bar.sync %0, 128;" ::"r"(1 + quarter) : "memory");
        if (part == 0 && lane == 0)
            async::bulk_to_peer(sm.act[out & 1] + rank * kHalf + quarter * 4 * kUnitGroup, 4 * kUnitGroup,
                                &sm.in_bar[out & 1], rank ^ 1u);
        ++out;
    }
    // pre-activations of layer l, push k: 16 bytes for 8 rows of a unit
    __device__ unsigned char* z_slot(const SurArgs& a, int l, int k, int tile) const {
        return a.zsave + ((size_t)l * a.tile_cap + (size_t)k * a.n_tiles) * kActBytes +
               (size_t)tile * (kHidden * TR * 2) + ((size_t)(part * kGroups) * kHidden + rank * kUnits + unit) * 16;
    }
    __device__ void finish(bool failed, int* err) {
        if (failed && tid == 0) {
            atomicOr(err, 2);
            // a last bounded wait for what is still in flight before the memory is given up
            if (!w_ready) wait(&sm.w_bar, 0);
            if (in_pending) wait(&sm.in_bar[(out - 1) & 1], ((out - 1) >> 1) & 1);
            if (mma_pending) wait(&sm.mma_bar, mma_phase);
        }
        async::cluster_sync();   // no CTA leaves while the peer's copy reads or writes its memory
        if (warp == 0) tmem_dealloc(tmem, kClCols);
    }
};

template <int NB, int TR>
__global__ void __launch_bounds__(kThreads, 1) sur_fwd_cluster_kernel(const SimConst sc, const SurArgs a) {
    constexpr int S3 = 3 * NB, kG = ClusterSide<TR>::kGroups;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    SurClSmem<TR>& sm = *reinterpret_cast<SurClSmem<TR>*>(smem_raw);
    ClusterSide<TR> s(sm);
    after_previous();
    const int tile = blockIdx.x / 2;
    // a thread per row: warps 0 .. hold the poses, warps 4 .. fetch the action's features
    const int row = s.tid % 128, i = tile * TR + row;
    const bool posed = s.tid < TR, acted = s.tid >= 128 && s.tid < 128 + TR;
    const bool on = i < a.N, first = s.rank == 0;
    const uint64_t gkey = a.iter >= 0 ? sm64(sm64(a.seed, kStreamGumbel), (uint64_t)a.iter) : 0ull;
    if (s.tid == 0) {   // this CTA's units of the weights (K-major: contiguous), the whole head
        constexpr unsigned w0 = kUnits * kIn * 2, w1 = kUnits * kHidden * 2, w3 = kOut * kHidden * 2;
        mbar_expect_tx(&sm.w_bar, w0 + 2 * w1 + w3);
        fence_async_shared();
        tma_load_1d(sm.w_in, a.w_tiled + layer_w_offset(0) + s.rank * w0, w0, &sm.w_bar);
        tma_load_1d(sm.w_mid[0], a.w_tiled + layer_w_offset(1) + s.rank * w1, w1, &sm.w_bar);
        tma_load_1d(sm.w_mid[1], a.w_tiled + layer_w_offset(2) + s.rank * w1, w1, &sm.w_bar);
        tma_load_1d(sm.w_out, a.w_tiled + layer_w_offset(3), w3, &sm.w_bar);
    }
    float bias[3];
#pragma unroll
    for (int l = 0; l < 3; ++l) bias[l] = a.bias[l * kHidden + s.rank * kUnits + s.unit];
    float q[S3];
#pragma unroll
    for (int t = 0; t < S3; ++t) q[t] = sc.init[t / 3][t % 3];
    if (posed) {
        pose_features<NB>(q, on, sm.x, row);
        if (on && first && (a.zsave || sc.H == 1))
#pragma unroll
            for (int t = 0; t < S3; ++t) a.pose[(size_t)i * S3 + t] = q[t];
    }
    all_action_features<NB>(sc, a, tile * TR, TR, gkey, s.tid * 2 + s.rank, 2 * kThreads);
    async::cluster_sync();   // the cluster's stores to a.relax are there
    if (acted) stored_features<NB>(sc, a, i, on, 0, sm.x, row);
    fence_async_shared();
    bool failed = false;
    for (int k = 0; k < sc.H && !failed; ++k) {
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            if (!s.multiply(l == 0 ? sm.w_in : sm.w_mid[l ? l - 1 : 0], l == 0 ? kIn : 0, 0)) { failed = true; break; }
            // layer 0 has read the push's features: the next push's, beside this MMA
            if (l == 1 && acted && k + 1 < sc.H) stored_features<NB>(sc, a, i, on, k + 1, sm.x, row);
            if (!s.product_done()) { failed = true; break; }
            unsigned char* dst = s.begin_output();
            float v[8 * kG];
            s.read(v);
#pragma unroll
            for (int g = 0; g < kG; ++g) {
                uint4 pk, pz;
                unsigned* pw = reinterpret_cast<unsigned*>(&pk);
                unsigned* pzw = reinterpret_cast<unsigned*>(&pz);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float z0 = v[g * 8 + 2 * e] + bias[l], z1 = v[g * 8 + 2 * e + 1] + bias[l];
                    pw[e] = pack_bf16(silu(z0), silu(z1));
                    pzw[e] = pack_bf16(z0, z1);
                }
                *reinterpret_cast<uint4*>(dst + g * 128) = pk;
                if (a.zsave)   // pre-activation of layer l, for the reverse sweep
                    *reinterpret_cast<uint4*>(s.z_slot(a, l, k, tile) + g * kHidden * 16) = pz;
            }
            s.send_output();
        }
        if (failed || !s.multiply(sm.w_out, 0, kOut) || !s.product_done()) { failed = true; break; }
        if (posed) {
            float v[16];
            tmem_ld16(s.lane_base(), v);
            const float* bl = a.bias + 3 * kHidden;
            float d[S3];
#pragma unroll
            for (int t = 0; t < S3; ++t) d[t] = v[t] + bl[t];
            if (k + 1 == sc.H) {   // the cost adds the last pose change itself
                if (on && first)
#pragma unroll
                    for (int t = 0; t < S3; ++t) a.y[(size_t)i * S3 + t] = d[t];
            } else {
#pragma unroll
                for (int t = 0; t < S3; ++t) q[t] += d[t];
                if (on && first && (a.zsave || k + 2 == sc.H))
#pragma unroll
                    for (int t = 0; t < S3; ++t) a.pose[((size_t)(k + 1) * a.N + i) * S3 + t] = q[t];
                pose_features<NB>(q, on, sm.x, row);
            }
        }
        fence_async_shared();
        tc_fence_before();
    }
    s.finish(failed, a.err);
}

template <int NB, int TR>
__global__ void __launch_bounds__(kThreads, 1) sur_bwd_cluster_kernel(const SimConst sc, const SurArgs a) {
    constexpr int S3 = 3 * NB, kG = ClusterSide<TR>::kGroups;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    SurClSmem<TR>& sm = *reinterpret_cast<SurClSmem<TR>*>(smem_raw);
    ClusterSide<TR> s(sm);
    after_previous();
    const int tile = blockIdx.x / 2, row = s.tid % 128, i = tile * TR + row;
    const bool posed = s.tid < TR, on = posed && i < a.N;   // a thread per row
    if (s.tid == 0) {   // this CTA's rows of the transposed weights, all of W_0^T
        constexpr unsigned w0 = kIn * kHidden * 2, w1 = kUnits * kHidden * 2, w3 = kOut * kUnits * 2;
        mbar_expect_tx(&sm.w_bar, w0 + 2 * w1 + w3);
        fence_async_shared();
        tma_load_1d(sm.w_out, a.wt_tiled + layer_w_offset(3) + s.rank * w3, w3, &sm.w_bar);
        tma_load_1d(sm.w_mid[1], a.wt_tiled + layer_w_offset(2) + s.rank * w1, w1, &sm.w_bar);
        tma_load_1d(sm.w_mid[0], a.wt_tiled + layer_w_offset(1) + s.rank * w1, w1, &sm.w_bar);
        tma_load_1d(sm.w_in, a.wt_tiled + layer_w_offset(0), w0, &sm.w_bar);
    }
    float ap[S3];   // dC/dq_{k+1}
#pragma unroll
    for (int t = 0; t < S3; ++t) ap[t] = on ? a.apose[(size_t)i * S3 + t] : 0.f;
    bool failed = false;
    for (int k = sc.H - 1; k >= 0 && !failed; --k) {
        if (posed) {   // dz_3 = dy = dC/dq_{k+1}: a BF16 K-major tile of 16 columns
            float d[kOut];
#pragma unroll
            for (int c = 0; c < kOut; ++c) d[c] = c < S3 ? ap[c < S3 ? c : 0] : 0.f;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                uint4 pk;
                unsigned* pw = reinterpret_cast<unsigned*>(&pk);
#pragma unroll
                for (int e = 0; e < 4; ++e) pw[e] = pack_bf16(d[g * 8 + 2 * e], d[g * 8 + 2 * e + 1]);
                *reinterpret_cast<uint4*>(sm.x + tile_off(row, g * 8, kOut)) = pk;
            }
        }
        fence_async_shared();
        FeaturesReverse<NB> f;
#pragma unroll
        for (int m = 3; m > 0; --m) {   // da_m = dz_m W_m
            if (!s.multiply(m == 3 ? sm.w_out : sm.w_mid[m < 3 ? m - 1 : 0], m == 3 ? kOut : 0, 0)) {
                failed = true;
                break;
            }
            uint4 z[kG];   // beside the MMA
#pragma unroll
            for (int g = 0; g < kG; ++g)
                z[g] = *reinterpret_cast<const uint4*>(s.z_slot(a, m - 1, k, tile) + g * kHidden * 16);
            if (m == 2 && on) f.load(sc, a, i, k);
            if (!s.product_done()) { failed = true; break; }
            unsigned char* dst = s.begin_output();
            float v[8 * kG];
            s.read(v);
#pragma unroll
            for (int g = 0; g < kG; ++g) {
                const unsigned zw[4] = {z[g].x, z[g].y, z[g].z, z[g].w};
                uint4 pk;
                unsigned* pw = reinterpret_cast<unsigned*>(&pk);
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    pw[e] = pack_bf16(v[g * 8 + 2 * e] * silu_grad(bf_lo(zw[e])),
                                      v[g * 8 + 2 * e + 1] * silu_grad(bf_hi(zw[e])));
                *reinterpret_cast<uint4*>(dst + g * 128) = pk;
            }
            s.send_output();
        }
        if (failed || !s.multiply(sm.w_in, 0, kIn) || !s.product_done()) { failed = true; break; }
        if (posed) {
            float v[32];
            tmem_ld32(s.lane_base(), v);
            if (on) f.apply(sc, a, i, k, v, ap, s.rank == 0);
        }
        tc_fence_before();
    }
    s.finish(failed, a.err);
}

template <int NB, int TR>
cudaError_t launch_cluster(const SimConst& sc, const SurArgs& a, bool reverse, cudaStream_t st) {
    auto* kernel = reverse ? sur_bwd_cluster_kernel<NB, TR> : sur_fwd_cluster_kernel<NB, TR>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.N + TR - 1) / TR * 2);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = sizeof(SurClSmem<TR>);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // as launch_after
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)cfg.dynamicSmemBytes);
    if (e != cudaSuccess) return e;
    return cudaLaunchKernelEx(&cfg, kernel, sc, a);
}

template <int NB>
cudaError_t launch(const SimConst& sc, const SurArgs& a, bool reverse, int sms, cudaStream_t st) {
    // The narrowest tile whose clusters all run at once: its time does not depend on
    // N (GB300, 6 pushes with the gradient, launches one after the other: 78 us on 32
    // rows, 96 on 64, 181 on 128-row tiles; a second wave would double it).  The
    // outputs' bits are the same.
    if (a.N <= sms / 2 * 32) return launch_cluster<NB, 32>(sc, a, reverse, st);
    if (a.N <= sms / 2 * 64) return launch_cluster<NB, 64>(sc, a, reverse, st);
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
