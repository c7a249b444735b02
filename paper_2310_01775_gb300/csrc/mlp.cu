// BF16 tensor-core MLP for the pose-dynamics surrogate (tcgen05 + TMEM + TMA).
//
// Network: in (<= 32, zero-padded to 32) -> 256 -> 256 -> 256 -> out (<= 16,
// padded to 16), SiLU between layers, linear head; BF16 weights and
// activations, FP32 accumulation in tensor memory.
//
// Operand layout (tcgen05 K-major, no swizzle): a tile of R rows x K columns
// of BF16 is stored as 8x8 "core matrices" of 128 contiguous bytes (8 rows of
// 16 bytes); core matrix (i, j) -- rows 8i..8i+7, columns 8j..8j+7 -- sits at
// byte i*SBO + j*128 with SBO = (K/8)*128.  The matrix descriptor of a 16-wide
// K slice then has leading-dimension offset 128 B (next core matrix along K)
// and stride-dimension offset SBO (next 8-row group).  Weights are packed once
// into this layout in HBM and streamed per layer with 1-D TMA bulk copies;
// each layer's epilogue writes the next layer's A operand straight into it.
#include <cstdint>
#include <cstring>
#include <vector>

#include "mlp.cuh"
#include "mlp_tc.cuh"
#include "stamp.h"
#include "stamp_internal.cuh"
#include "surrogate_mlp.cuh"

namespace stamp {
namespace mlp {
namespace {

// Forward of all four layers for 128-row tiles: x (rows x in_dim FP32) becomes
// layer 0's operand, rounded to BF16 and zero-padded, on the way in, and the
// head writes the out_dim columns of y (row stride ldy).  Optionally stores,
// for the backward pass, the input tile a_0 (x_tiled), the input activations
// a_1..a_3 and the pre-activations z_0..z_2 (BF16 tiles): slot (l, tile_base +
// tile) of buffers holding tile_cap tiles per layer.  Packing the input and
// unpacking a padded output in launches of their own cost 3.8 + 3.0 us at 16384
// rows beside the 18.2 of this kernel (GB300).
__global__ void __launch_bounds__(kThreads, 1)
mlp_fwd_kernel(const float* __restrict__ x, int in_dim, unsigned char* __restrict__ x_tiled, int n_tiles,
               const unsigned char* __restrict__ w_tiled, const float* __restrict__ bias,
               float* __restrict__ y, int ldy, int out_dim, int rows,
               unsigned char* __restrict__ saved, unsigned char* __restrict__ zsave, int tile_base,
               int tile_cap, int* __restrict__ err) {
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
    unsigned tma_phase = 0, mma_phase = 0;
    bool failed = false, tma_pending = false, mma_pending = false;
    auto issue_load = [&](int l) {   // layer l's weights into shared memory
        const unsigned wbytes = (unsigned)(layer_n(l) * layer_k(l) * 2);
        mbar_expect_tx(&sm.tma_bar, wbytes);
        tma_load_1d(sm.w, w_tiled + layer_w_offset(l), wbytes, &sm.tma_bar);
    };
    // a tile's input: thread -> row tid % 128, columns 8 (tid / 128) ...
    const int xr = tid % kRows, xc = tid / kRows * 8;
    float xv[8];
    auto read_x = [&](int tile) {
        const int r = tile * kRows + xr;
#pragma unroll
        for (int c = 0; c < 8; ++c)
            xv[c] = r < rows && xc + c < in_dim ? __ldg(x + (size_t)r * in_dim + xc + c) : 0.f;
    };
    auto put_x = [&](int tile) {
        const uint4 pk = make_uint4(pack_bf16(xv[0], xv[1]), pack_bf16(xv[2], xv[3]),
                                    pack_bf16(xv[4], xv[5]), pack_bf16(xv[6], xv[7]));
        const unsigned off = tile_off(xr, xc, kIn);
        *reinterpret_cast<uint4*>(sm.act + off) = pk;
        if (saved) *reinterpret_cast<uint4*>(x_tiled + (size_t)(tile_base + tile) * kInBytes + off) = pk;
    };
    if (blockIdx.x < n_tiles) {
        if (tid == 0) issue_load(0);
        tma_pending = true;
        read_x(blockIdx.x);
        put_x(blockIdx.x);
        fence_async_shared();
    }
    for (int tile = blockIdx.x; tile < n_tiles && !failed; tile += gridDim.x) {
        for (int l = 0; l < 4 && !failed; ++l) {
            const int K = layer_k(l), N = layer_n(l);
            unsigned spins = 0;
            bool ok = true;
            while (!(ok = mbar_try_wait(&sm.tma_bar, tma_phase)) && ++spins < kWaitLimit) {
            }
            if (__syncthreads_or(!ok)) { failed = true; break; }   // the copy stays pending
            tma_phase ^= 1u;
            tma_pending = false;
            if (tid == 0) {
                tc_fence_after();
                mma_tile(tmem, sm.act, sm.w, K, N);
                mma_commit(&sm.mma_bar);
            }
            mma_pending = true;
            if (l == 3 && tile + (int)gridDim.x < n_tiles) read_x(tile + gridDim.x);
            if (saved && l > 0) {   // this layer's input activation, for the backward pass
                // (read beside the MMA, which only reads it too)
                unsigned char* dst = saved + ((size_t)l * tile_cap + tile_base + tile) * kActBytes;
                for (int b = tid * 16; b < (int)kActBytes; b += kThreads * 16)
                    *reinterpret_cast<uint4*>(dst + b) = *reinterpret_cast<const uint4*>(sm.act + b);
            }
            spins = 0;
            while (!(ok = mbar_try_wait(&sm.mma_bar, mma_phase)) && ++spins < kWaitLimit) {
            }
            if (__syncthreads_or(!ok)) { failed = true; break; }   // the MMA stays pending
            mma_phase ^= 1u;
            mma_pending = false;
            tc_fence_after();
            // the weight buffer is free: start the next layer's (or next tile's)
            // copy now, so it runs beside this epilogue
            if (l < 3 || tile + (int)gridDim.x < n_tiles) {
                if (tid == 0) {
                    fence_async_shared();
                    issue_load(l < 3 ? l + 1 : 0);
                }
                tma_pending = true;
            }
            // epilogue: this warp's 32 rows, its part of the N columns
            const int quarter = warp & 3, half = warp >> 2;
            const int row = quarter * 32 + lane;
            const unsigned lane_base = tmem + ((unsigned)(quarter * 32) << 16);
            const float* bl = bias + l * kHidden;
            if (l < 3) {
                for (int c0 = half * (N / kParts); c0 < (half + 1) * (N / kParts); c0 += 32) {
                    float v[32];
                    tmem_ld32(lane_base + c0, v);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        uint4 pk;
                        unsigned* pw = reinterpret_cast<unsigned*>(&pk);
                        uint4 pz;
                        unsigned* pzw = reinterpret_cast<unsigned*>(&pz);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int c = c0 + q * 8 + 2 * e;
                            const float z0 = v[q * 8 + 2 * e] + __ldg(bl + c);
                            const float z1 = v[q * 8 + 2 * e + 1] + __ldg(bl + c + 1);
                            pw[e] = pack_bf16(silu(z0), silu(z1));
                            pzw[e] = pack_bf16(z0, z1);
                        }
                        const unsigned off = tile_off(row, c0 + q * 8, kHidden);
                        *reinterpret_cast<uint4*>(sm.act + off) = pk;
                        if (zsave)   // pre-activation of layer l, for the backward pass
                            *reinterpret_cast<uint4*>(
                                zsave + ((size_t)l * tile_cap + tile_base + tile) * kActBytes + off) = pz;
                    }
                }
            } else {
                if (tile + (int)gridDim.x < n_tiles) put_x(tile + gridDim.x);   // act is free too
                if (half == 0) {
                    float v[16];
                    tmem_ld16(lane_base, v);
                    const int r = tile * kRows + row;
                    if (r < rows) {
                        float* dst = y + (size_t)r * ldy;
#pragma unroll
                        for (int c = 0; c < kOut; ++c)
                            if (c < out_dim) dst[c] = v[c] + __ldg(bl + c);
                    }
                }
            }
            // the next MMA reads act (written here) and overwrites TMEM (read here)
            fence_async_shared();
            tc_fence_before();
            __syncthreads();
        }
    }
    if (failed && tid == 0) {
        atomicOr(err, 2);
        // a last bounded wait for the copy / MMA still in flight before the
        // tensor memory is released
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

// Master FP32 parameters (W_l as (n_l, k_l) real sizes, then b_l) -> packed BF16
// K-major weight tiles (zero-padded to the kernel's sizes) and FP32 biases.
__global__ void pack_weights_kernel(const float* __restrict__ params, int in_dim, int out_dim,
                                    unsigned char* __restrict__ w_tiled,
                                    unsigned char* __restrict__ wt_tiled, float* __restrict__ bias) {
    const int l = blockIdx.y;
    const int K = layer_k(l), N = layer_n(l);
    const int kr = l == 0 ? in_dim : kHidden, nr = l == 3 ? out_dim : kHidden;
    const float* W = params + param_offset(l, in_dim, out_dim);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < N * K; t += gridDim.x * blockDim.x) {
        const int n = t / K, k = t % K;
        const __nv_bfloat16 v = __float2bfloat16_rn((n < nr && k < kr) ? W[n * kr + k] : 0.f);
        // forward operand: (N = out, K = in); backward operand W^T: (N = in, K = out)
        *reinterpret_cast<__nv_bfloat16*>(w_tiled + layer_w_offset(l) + tile_off(n, k, K)) = v;
        *reinterpret_cast<__nv_bfloat16*>(wt_tiled + layer_w_offset(l) + tile_off(k, n, N)) = v;
    }
    if (blockIdx.x == 0)
        for (int n = threadIdx.x; n < kHidden; n += blockDim.x)
            bias[l * kHidden + n] = (n < nr) ? W[nr * kr + n] : 0.f;
}

__global__ void unpack_output_kernel(const float* __restrict__ ypad, int rows, int out_dim,
                                     float* __restrict__ y) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < rows * out_dim) y[t] = ypad[(size_t)(t / out_dim) * kOut + t % out_dim];
}

// Reverse sweep through the four layers for 128-row tiles:
//   dz_3 = dy;  da_m = dz_m W_m (MMA, B = W_m^T tiles);  dz_{m-1} = da_m * SiLU'(z_{m-1});
//   dx = da_0.
// dz_m (BF16 tiles) go to dzsave slot (m, tile_base + tile) for the weight
// gradients; zsave holds the forward's pre-activations.
__global__ void __launch_bounds__(kThreads, 1)
mlp_bwd_kernel(const float* dy, int rows, int out_dim, int n_tiles,
               const unsigned char* wt_tiled, const unsigned char* zsave,
               unsigned char* __restrict__ dzsave, int tile_base, int tile_cap,
               float* __restrict__ dx, int in_dim, int* __restrict__ err) {
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
    const int quarter = warp & 3, half = warp >> 2;
    const int row = quarter * 32 + lane;
    unsigned tma_phase = 0, mma_phase = 0;
    bool failed = false, tma_pending = false, mma_pending = false;
    after_previous();
    auto issue_load = [&](int m) {   // W_m^T into shared memory
        const unsigned wbytes = (unsigned)(layer_k(m) * layer_n(m) * 2);
        mbar_expect_tx(&sm.tma_bar, wbytes);
        tma_load_1d(sm.w, wt_tiled + layer_w_offset(m), wbytes, &sm.tma_bar);
    };
    if (blockIdx.x < n_tiles) {
        if (tid == 0) issue_load(3);
        tma_pending = true;
    }
    for (int tile = blockIdx.x; tile < n_tiles && !failed; tile += gridDim.x) {
        const int r = tile * kRows + row;
        const size_t slot = (size_t)tile_base + tile;
        if (half == 0) {   // dz_3 = dy as a BF16 K-major tile of 16 columns
            float d[kOut];
            const float* dr = dy + (size_t)min(r, rows - 1) * out_dim;
#pragma unroll
            for (int c = 0; c < kOut; ++c) d[c] = dr[c < out_dim ? c : 0];   // no branch: all in flight
#pragma unroll
            for (int c = 0; c < kOut; ++c) d[c] = (r < rows && c < out_dim) ? d[c] : 0.f;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                uint4 pk;
                unsigned* pw = reinterpret_cast<unsigned*>(&pk);
#pragma unroll
                for (int e = 0; e < 4; ++e) pw[e] = pack_bf16(d[q * 8 + 2 * e], d[q * 8 + 2 * e + 1]);
                const unsigned off = tile_off(row, q * 8, kOut);
                *reinterpret_cast<uint4*>(sm.act + off) = pk;
                *reinterpret_cast<uint4*>(dzsave + ((size_t)3 * tile_cap + slot) * kActBytes + off) = pk;
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
            // the weight buffer is free: the next layer's (or next tile's first)
            // weights load beside this epilogue
            if (m > 0 || tile + (int)gridDim.x < n_tiles) {
                if (tid == 0) {
                    fence_async_shared();
                    issue_load(m > 0 ? m - 1 : 3);
                }
                tma_pending = true;
            }
            const unsigned lane_base = tmem + ((unsigned)(quarter * 32) << 16);
            if (m > 0) {
                const unsigned char* zt = zsave + ((size_t)(m - 1) * tile_cap + slot) * kActBytes;
                unsigned char* dzt = dzsave + ((size_t)(m - 1) * tile_cap + slot) * kActBytes;
                for (int c0 = half * (kHidden / kParts); c0 < (half + 1) * (kHidden / kParts); c0 += 32) {
                    uint4 zq[4];   // before the read of tensor memory, which they may not pass
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        zq[q] = *reinterpret_cast<const uint4*>(zt + tile_off(row, c0 + q * 8, kHidden));
                    float v[32];
                    tmem_ld32(lane_base + c0, v);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const unsigned off = tile_off(row, c0 + q * 8, kHidden);
                        const uint4 zv = zq[q];
                        const unsigned zw[4] = {zv.x, zv.y, zv.z, zv.w};
                        uint4 pk;
                        unsigned* pw = reinterpret_cast<unsigned*>(&pk);
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            pw[e] = pack_bf16(v[q * 8 + 2 * e] * silu_grad(bf_lo(zw[e])),
                                              v[q * 8 + 2 * e + 1] * silu_grad(bf_hi(zw[e])));
                        *reinterpret_cast<uint4*>(sm.act + off) = pk;
                        *reinterpret_cast<uint4*>(dzt + off) = pk;
                    }
                }
            } else if (dx && half == 0) {
                float v[32];
                tmem_ld32(lane_base, v);
                if (r < rows)
                    for (int c = 0; c < in_dim; ++c) dx[(size_t)r * in_dim + c] = v[c];
            }
            fence_async_shared();
            tc_fence_before();
            __syncthreads();
        }
    }
    if (failed && tid == 0) {
        atomicOr(err, 2);
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

// Weight gradients of all four layers in one launch: the sum over rows of
// outer products is an MMA whose reduction dimension K is the rows.  The saved
// activations and dz tiles hold, per 8 x 8 core matrix, 8 rows of 8 units:
// units contiguous, so as operands over rows they are M/N-major as they lie
// (descriptor: unit groups 128 B apart, row groups (units / 8) * 128 B apart;
// the transpose bits of the instruction descriptor), and their tiles go to
// shared memory by TMA as they are:
//   D (M = 128 units of P, half mb) x (N = NQ units of Q)
//     += P^T (M x 128 rows) . Q (128 rows x N)      per 128-row tile,
// accumulated in TMEM over the tiles of the CTA's row split, two tiles in
// flight; then stored as the split's partial, which a second launch sums in
// split order (deterministic: no atomics).  The bias gradient of the dz
// operand's units is summed beside the MMA, in a fixed order, per split.  The
// splits give each SM one CTA with about the same bytes (the hidden layers'
// 96 KB a tile, the outer ones' 40 and 36).  GB300, 16384 rows, cold caches: 19.5
// us (52 MB from DRAM) and 10 us for the reduction; a launch per layer that
// transposed every core matrix through registers (movmatrix), and its
// reduction, took 80 + 44.
constexpr int kDwMaxSplits = 32;     // of a layer
constexpr unsigned kDwStage = 96 * 1024;   // P half (32 KB) and Q (up to 64 KB) of a tile
struct DwSmem {
    alignas(128) unsigned char stage[2][kDwStage];
    uint64_t full[2], mma_bar;
    unsigned tmem_slot;
};
struct DwLayer {
    const unsigned char *P, *Q;   // first tile; P: 256 units, Q: NQ units
    size_t p_stride, q_stride;    // bytes per tile
    int NQ, dz_is_P, splits, per; // per: tiles per split
    size_t part, bias;            // first float of the splits' partials
    int out_r, in_r;              // real sizes of W
    size_t w;                     // offset of W in the packed gradient
    int cta0;                     // first CTA: (split, half) pairs, split-major
    int e0;                       // first element of the reduction
};
struct DwArgs {
    DwLayer l[kLayers];   // in order of their CTAs and elements
    int n_tiles;
    float *part, *grad;
    int* err;
};

__device__ __forceinline__ uint32_t idesc_bf16_mn(int M, int N) {   // both operands M/N-major
    return idesc_bf16(M, N) | (1u << 15) | (1u << 16);
}

__global__ void __launch_bounds__(kThreads, 1) mlp_dw_kernel(const DwArgs a) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    DwSmem& sm = *reinterpret_cast<DwSmem*>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int li = 0;
#pragma unroll
    for (int q = 1; q < kLayers; ++q)
        if ((int)blockIdx.x >= a.l[q].cta0) li = q;
    const DwLayer& L = a.l[li];
    const int NQ = L.NQ, c = blockIdx.x - L.cta0, mb = c & 1, split = c >> 1;
    const unsigned cols = NQ <= 32 ? 32u : 256u;
    if (tid == 0) {
        mbar_init(&sm.full[0], 1);
        mbar_init(&sm.full[1], 1);
        mbar_init(&sm.mma_bar, 1);
        fence_async_shared();
    }
    if (warp == 0) tmem_alloc(&sm.tmem_slot, cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = sm.tmem_slot;
    after_previous();
    const int t0 = split * L.per, t1 = min(a.n_tiles, t0 + L.per);
    constexpr unsigned kPHalf = kRows * kRows * 2;   // 32 KB: 16 row groups of 2 KB
    auto issue = [&](int t) {
        unsigned char* st = sm.stage[(t - t0) & 1];
        uint64_t* bar = &sm.full[(t - t0) & 1];
        const unsigned q_bytes = (unsigned)(kRows * NQ * 2);
        mbar_expect_tx(bar, kPHalf + q_bytes);
        const unsigned char* p = L.P + (size_t)t * L.p_stride + mb * 2048;
        for (int g = 0; g < kRows / 8; ++g) tma_load_1d(st + g * 2048, p + g * 4096, 2048, bar);
        tma_load_1d(st + kPHalf, L.Q + (size_t)t * L.q_stride, q_bytes, bar);
    };
    if (tid == 0)
        for (int t = t0; t < t1 && t < t0 + 2; ++t) issue(t);
    // the dz operand's units whose bias gradient this CTA sums: warp g takes unit
    // group g, a lane every 32nd row (16 bytes of it: no bank conflicts)
    const int n_bias = L.dz_is_P ? kRows : (mb == 0 ? NQ : 0);
    const bool biased = warp < n_bias / 8;
    const unsigned bias_at = (L.dz_is_P ? 0u : kPHalf) + warp * 128 + (lane & 7) * 16;
    const unsigned bias_rg = L.dz_is_P ? 2048u : (unsigned)(NQ / 8) * 128u;
    float bsum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    unsigned full_phase = 0, mma_phase = 0;   // bit s: parity of stage s
    bool failed = false, mma_pending = false;
    int t = t0;
    for (; t < t1 && !failed; ++t) {
        const int s = (t - t0) & 1;
        unsigned char* st = sm.stage[s];
        unsigned spins = 0;
        bool ok = true;
        while (!(ok = mbar_try_wait(&sm.full[s], (full_phase >> s) & 1u)) && ++spins < kWaitLimit) {
        }
        if (__syncthreads_or(!ok)) { failed = true; break; }   // the copies stay pending
        full_phase ^= 1u << s;
        if (tid == 0) {
            const uint32_t idesc = idesc_bf16_mn(kRows, NQ);
            const unsigned q_rg = (unsigned)(NQ / 8) * 128u;   // bytes per row group of Q
            for (int kk = 0; kk < kRows / 16; ++kk)
                mma_bf16(tmem, smem_desc(st + kk * 4096, 2048, 128),
                         smem_desc(st + kPHalf + kk * 2 * q_rg, q_rg, 128), idesc, (t > t0 || kk > 0) ? 1u : 0u);
            mma_commit(&sm.mma_bar);
        }
        mma_pending = true;
        if (biased) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint4 w = *reinterpret_cast<const uint4*>(st + bias_at + (4 * q + (lane >> 3)) * bias_rg);
                const unsigned e[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    bsum[2 * u] += bf_lo(e[u]);
                    bsum[2 * u + 1] += bf_hi(e[u]);
                }
            }
        }
        spins = 0;
        while (!(ok = mbar_try_wait(&sm.mma_bar, mma_phase)) && ++spins < kWaitLimit) {
        }
        if (__syncthreads_or(!ok)) { failed = true; break; }   // the MMA stays pending
        mma_phase ^= 1u;
        mma_pending = false;
        if (tid == 0 && t + 2 < t1) {
            fence_async_shared();
            issue(t + 2);
        }
    }
    tc_fence_after();
    if (!failed) {
        // epilogue: TMEM lane = unit of P (row of D), column = unit of Q
        const int quarter = warp & 3, cpart = warp >> 2, row = quarter * 32 + lane;
        const unsigned lane_base = tmem + ((unsigned)(quarter * 32) << 16);
        float* out = a.part + L.part + ((size_t)(split * 2 + mb) * kRows + row) * NQ;
        if (NQ == kHidden) {
            for (int c0 = cpart * (kHidden / 4); c0 < (cpart + 1) * (kHidden / 4); c0 += 32) {
                float v[32];
                tmem_ld32(lane_base + c0, v);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    reinterpret_cast<float4*>(out + c0)[q] =
                        make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            }
        } else if (cpart == 0 && NQ == kIn) {
            float v[32];
            tmem_ld32(lane_base, v);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                reinterpret_cast<float4*>(out)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        } else if (cpart == 0) {   // NQ == kOut
            float v[16];
            tmem_ld16(lane_base, v);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                reinterpret_cast<float4*>(out)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        }
        if (biased) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) bsum[u] += __shfl_xor_sync(~0u, bsum[u], o);
                if (lane == 0)
                    a.part[L.bias + (size_t)split * kHidden + (L.dz_is_P ? mb * kRows : 0) + warp * 8 + u] = bsum[u];
            }
        }
    }
    if (failed && tid == 0) {
        atomicOr(a.err, 2);
        // a last bounded wait for the copies and the MMA still in flight
        for (int q = 0; q < 2; ++q)
            if (t + q < t1) {
                const int s = (t + q - t0) & 1;
                const bool waited = q == 0 && mma_pending;   // this tile's copies have landed
                if (!waited)
                    for (unsigned w = 0; w < kWaitLimit && !mbar_try_wait(&sm.full[s], (full_phase >> s) & 1u); ++w) {
                    }
            }
        if (mma_pending)
            for (unsigned w = 0; w < kWaitLimit && !mbar_try_wait(&sm.mma_bar, mma_phase); ++w) {
            }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, cols);
}

// dW and db of every layer from the splits' partials, summed in split order.
// part: [split][256 units of P][NQ]; where P holds the layer's inputs, D = dW^T.
__global__ void __launch_bounds__(256) mlp_dw_reduce_kernel(const DwArgs a) {
    after_previous();
    const int e = blockIdx.x * 256 + threadIdx.x;
    int li = 0;
#pragma unroll
    for (int q = 1; q < kLayers; ++q)
        if (e >= a.l[q].e0) li = q;
    const DwLayer& L = a.l[li];
    const int r = e - L.e0, n = kHidden * L.NQ;
    if (r < n) {
        const float* p = a.part + L.part + r;
        float s = 0.f;
#pragma unroll 8
        for (int q = 0; q < L.splits; ++q) s += p[(size_t)q * n];
        const int m = r / L.NQ, u = r % L.NQ;
        const int o = L.dz_is_P ? m : u, i = L.dz_is_P ? u : m;
        if (o < L.out_r && i < L.in_r) a.grad[L.w + (size_t)o * L.in_r + i] = s;
    }
    if (r < L.out_r) {
        float s = 0.f;
        for (int q = 0; q < L.splits; ++q) s += a.part[L.bias + (size_t)q * kHidden + r];
        a.grad[L.w + (size_t)L.out_r * L.in_r + r] = s;
    }
}

// Mean squared error over rows x out_dim: dy = 2 (y - t) / n, loss += sum (y-t)^2 / n.
__global__ void mse_kernel(const float* __restrict__ y, const float* __restrict__ t, int n,
                           float* __restrict__ dy, float* __restrict__ loss) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    float e2 = 0.f;
    if (i < n) {
        const float e = y[i] - t[i];
        dy[i] = 2.f * e / (float)n;
        e2 = e * e / (float)n;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, o);
    if ((threadIdx.x & 31) == 0 && e2 != 0.f) atomicAdd(loss, e2);
}

// Adam (Kingma & Ba 2015) minimising along g.
__global__ void param_adam_kernel(float* __restrict__ p, const float* __restrict__ g,
                                  float* __restrict__ m, float* __restrict__ v, int n, float lr,
                                  float bc1, float bc2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float mt = 0.9f * m[i] + 0.1f * g[i];
    const float vt = 0.999f * v[i] + 0.001f * g[i] * g[i];
    m[i] = mt;
    v[i] = vt;
    p[i] -= lr * (mt / bc1) / (sqrtf(vt / bc2) + 1e-8f);
}

}  // namespace

size_t fwd_smem_bytes() { return sizeof(FwdSmem) + 1024; }

cudaError_t pack_weights(const float* params, int in_dim, int out_dim, unsigned char* w_tiled,
                         unsigned char* wt_tiled, float* bias, cudaStream_t st) {
    pack_weights_kernel<<<dim3(64, 4), 256, 0, st>>>(params, in_dim, out_dim, w_tiled, wt_tiled,
                                                     bias);
    return cudaGetLastError();
}

cudaError_t forward(const float* x, int rows, int in_dim, int out_dim, const unsigned char* w_tiled,
                    const float* bias, unsigned char* x_tiled, float* ypad, float* y,
                    unsigned char* saved, unsigned char* zsave, int tile_base, int tile_cap,
                    int* err, int sm_count, cudaStream_t st) {
    const int n_tiles = (rows + kRows - 1) / kRows;
    const size_t smem = fwd_smem_bytes();
    cudaError_t e = cudaFuncSetAttribute(mlp_fwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    const int grid = n_tiles < sm_count ? n_tiles : sm_count;
    // a y that shares storage with x is written after every row of x has been read
    const bool overlap = x < y + (size_t)rows * out_dim && y < x + (size_t)rows * in_dim;
    mlp_fwd_kernel<<<grid, kThreads, smem, st>>>(x, in_dim, x_tiled, n_tiles, w_tiled, bias,
                                                 overlap ? ypad : y, overlap ? kOut : out_dim, out_dim,
                                                 rows, saved, zsave, tile_base, tile_cap, err);
    e = cudaGetLastError();
    if (e != cudaSuccess || !overlap) return e;
    unpack_output_kernel<<<(rows * out_dim + 255) / 256, 256, 0, st>>>(ypad, rows, out_dim, y);
    return cudaGetLastError();
}

cudaError_t backward(const float* dy, int rows, int in_dim, int out_dim,
                     const unsigned char* wt_tiled, const unsigned char* zsave,
                     unsigned char* dzsave, int tile_base, int tile_cap, float* dx, int* err,
                     int sm_count, cudaStream_t st) {
    const int n_tiles = (rows + kRows - 1) / kRows;
    const size_t smem = fwd_smem_bytes();
    cudaError_t e = cudaFuncSetAttribute(mlp_bwd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    const int grid = n_tiles < sm_count ? n_tiles : sm_count;
    return launch_after(mlp_bwd_kernel, dim3(grid), kThreads, smem, st, dy, rows, out_dim, n_tiles, wt_tiled, zsave,
                        dzsave, tile_base, tile_cap, dx, in_dim, err);
}

size_t dw_part_floats() {   // a layer: 256 x NQ and 256 bias sums per split
    return (size_t)kDwMaxSplits * kHidden * (2 * kHidden + kIn + kOut + kLayers);
}

cudaError_t weight_grads(const unsigned char* x_tiled, const unsigned char* saved,
                         const unsigned char* dzsave, int tile_base, int tile_cap, int rows,
                         int in_dim, int out_dim, float* grad, float* part, int* err, int sm_count,
                         cudaStream_t st) {
    const int n_tiles = (rows + kRows - 1) / kRows;
    const size_t smem = sizeof(DwSmem) + 1024;
    cudaError_t e = cudaFuncSetAttribute(mlp_dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    DwArgs a{};
    a.n_tiles = n_tiles;
    a.part = part;
    a.grad = grad;
    a.err = err;
    // one CTA per SM in all, the splits by a tile's bytes: 27 and 11 of the
    // hidden and the outer layers on 152 SMs (two halves of P each)
    const int order[kLayers] = {1, 2, 0, 3};   // the longest CTAs first
    size_t at = 0;
    int cta = 0, elem = 0;
    for (int q = 0; q < kLayers; ++q) {
        const int l = order[q];
        DwLayer& L = a.l[q];
        const unsigned char* act = l == 0 ? x_tiled + (size_t)tile_base * kInBytes
                                          : saved + ((size_t)l * tile_cap + tile_base) * kActBytes;
        const size_t act_stride = l == 0 ? kInBytes : kActBytes;
        const unsigned char* dz = dzsave + ((size_t)l * tile_cap + tile_base) * kActBytes;
        // P: the operand of 256 units; Q: the other one
        const bool dz_is_P = layer_n(l) == kHidden;
        L.P = dz_is_P ? dz : act;
        L.Q = dz_is_P ? act : dz;
        L.p_stride = dz_is_P ? kActBytes : act_stride;
        L.q_stride = dz_is_P ? act_stride : kActBytes;
        L.NQ = dz_is_P ? layer_k(l) : layer_n(l);
        L.dz_is_P = dz_is_P ? 1 : 0;
        int splits = L.NQ == kHidden ? sm_count * 27 / 152 : sm_count * 11 / 152;
        splits = splits < 1 ? 1 : splits > kDwMaxSplits ? kDwMaxSplits : splits;
        splits = splits > n_tiles ? n_tiles : splits;
        L.per = (n_tiles + splits - 1) / splits;
        L.splits = (n_tiles + L.per - 1) / L.per;
        L.part = at;
        at += (size_t)L.splits * kHidden * L.NQ;
        L.bias = at;
        at += (size_t)L.splits * kHidden;
        L.in_r = l == 0 ? in_dim : kHidden;
        L.out_r = l == 3 ? out_dim : kHidden;
        L.w = param_offset(l, in_dim, out_dim);
        L.cta0 = cta;
        cta += 2 * L.splits;
        L.e0 = elem;
        elem += kHidden * L.NQ;
    }
    e = launch_after(mlp_dw_kernel, dim3(cta), kThreads, smem, st, a);
    if (e != cudaSuccess) return e;
    return launch_after(mlp_dw_reduce_kernel, dim3((elem + 255) / 256), 256, 0, st, a);
}

cudaError_t mse(const float* y, const float* t, int n, float* dy, float* loss, cudaStream_t st) {
    mse_kernel<<<(n + 255) / 256, 256, 0, st>>>(y, t, n, dy, loss);
    return cudaGetLastError();
}

cudaError_t adam(float* p, const float* g, float* m, float* v, int n, int step, float lr,
                 cudaStream_t st) {
    const float bc1 = 1.f - powf(0.9f, (float)step), bc2 = 1.f - powf(0.999f, (float)step);
    param_adam_kernel<<<(n + 255) / 256, 256, 0, st>>>(p, g, m, v, n, lr, bc1, bc2);
    return cudaGetLastError();
}

}  // namespace mlp
}  // namespace stamp

// ----------------------------- C ABI ----------------------------------------
struct stamp_mlp {
    int in_dim = 0, out_dim = 0, max_rows = 0, train_rows = 0, tile_cap = 0, sm_count = 0;
    size_t n_params = 0;
    cudaStream_t stream = nullptr;
    char* arena = nullptr;
    unsigned char *w_tiled = nullptr, *wt_tiled = nullptr, *x_tiled = nullptr;
    unsigned char *saved = nullptr, *zsave = nullptr, *dzsave = nullptr;
    float *bias = nullptr, *ypad = nullptr, *ytrain = nullptr, *dy = nullptr;
    float *grad = nullptr, *adam_m = nullptr, *adam_v = nullptr, *loss = nullptr;
    float* dw_part = nullptr;   // per-split partial weight gradients (deterministic reduction)
    int* err = nullptr;
    int step = 0;
};

namespace stamp {
namespace mlp {
View view(const stamp_mlp* m) {
    return View{m->w_tiled, m->wt_tiled, m->bias, m->zsave, m->tile_cap, m->sm_count, m->err};
}
}  // namespace mlp
}  // namespace stamp

namespace {
stamp_status mlp_fail(stamp_status s, const char* msg, cudaError_t e = cudaSuccess) {
    char buf[256];
    std::strncpy(buf, msg, sizeof buf - 1);
    buf[sizeof buf - 1] = 0;
    if (e != cudaSuccess) {
        cudaGetLastError();
        std::strncat(buf, ": ", sizeof buf - std::strlen(buf) - 1);
        std::strncat(buf, cudaGetErrorString(e), sizeof buf - std::strlen(buf) - 1);
    }
    stamp::set_last_error(buf);
    return s;
}
bool on_device(const void* p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}
#define MLP_TRY(call, what)                                          \
    do {                                                             \
        cudaError_t e_ = (call);                                     \
        if (e_ != cudaSuccess) return mlp_fail(STAMP_ECUDA, what, e_); \
    } while (0)
}  // namespace

extern "C" stamp_status stamp_mlp_create(int in_dim, int out_dim, int max_rows, int train_rows,
                                         void* cuda_stream, stamp_mlp** out) {
    using namespace stamp::mlp;
    if (!out) return mlp_fail(STAMP_EINVAL, "out is NULL");
    *out = nullptr;
    if (in_dim < 1 || in_dim > kIn || out_dim < 1 || out_dim > kOut || max_rows < 1 || train_rows < 0)
        return mlp_fail(STAMP_EINVAL,
                        "need 1 <= in_dim <= 32, 1 <= out_dim <= 16, max_rows >= 1, train_rows >= 0");
    stamp_mlp* m = new stamp_mlp();
    m->in_dim = in_dim; m->out_dim = out_dim; m->max_rows = max_rows; m->train_rows = train_rows;
    m->tile_cap = (train_rows + 127) / 128;
    m->n_params = param_count(in_dim, out_dim);
    m->stream = static_cast<cudaStream_t>(cuda_stream);
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&m->sm_count, cudaDevAttrMultiProcessorCount, dev);
    const size_t xt = (size_t)((max_rows > train_rows ? max_rows : train_rows) + 127) / 128;
    const size_t cap = (size_t)m->tile_cap, np = m->n_params;
    void** dst[] = {(void**)&m->w_tiled, (void**)&m->wt_tiled, (void**)&m->x_tiled, (void**)&m->bias,
                    (void**)&m->ypad,    (void**)&m->saved,    (void**)&m->zsave,   (void**)&m->dzsave,
                    (void**)&m->ytrain,  (void**)&m->dy,       (void**)&m->grad,    (void**)&m->adam_m,
                    (void**)&m->adam_v,  (void**)&m->loss,     (void**)&m->err,     (void**)&m->dw_part};
    const size_t bytes[] = {kWeightBytes, kWeightBytes, xt * 128 * kIn * 2, (size_t)kLayers * kHidden * 4,
                            (size_t)max_rows * kOut * 4, 4 * cap * kRows * kHidden * 2,
                            3 * cap * kRows * kHidden * 2, 4 * cap * kRows * kHidden * 2,
                            (size_t)train_rows * out_dim * 4, (size_t)train_rows * out_dim * 4,
                            np * 4, np * 4, np * 4, 4, 4,
                            train_rows > 0 ? dw_part_floats() * 4 : 0};
    size_t total = 0;
    for (size_t b : bytes) total += (b + 255) / 256 * 256;
    cudaError_t e = cudaMalloc(&m->arena, total);
    if (e != cudaSuccess) { delete m; return mlp_fail(STAMP_ENOMEM, "cudaMalloc failed", e); }
    char* p = m->arena;
    for (size_t q = 0; q < sizeof bytes / sizeof bytes[0]; ++q) {
        *dst[q] = p;
        p += (bytes[q] + 255) / 256 * 256;
    }
    e = cudaMemset(m->arena, 0, total);
    if (e != cudaSuccess) { cudaFree(m->arena); delete m; return mlp_fail(STAMP_ECUDA, "memset failed", e); }
    *out = m;
    return STAMP_OK;
}

extern "C" void stamp_mlp_destroy(stamp_mlp* m) {
    if (!m) return;
    cudaStreamSynchronize(m->stream);
    cudaFree(m->arena);
    delete m;
}

extern "C" size_t stamp_mlp_param_count(int in_dim, int out_dim) {
    return stamp::mlp::param_count(in_dim, out_dim);
}

extern "C" stamp_status stamp_mlp_set_params(stamp_mlp* m, const float* params) {
    if (!m || !params || !on_device(params)) return mlp_fail(STAMP_EINVAL, "NULL mlp or non-device params");
    MLP_TRY(stamp::mlp::pack_weights(params, m->in_dim, m->out_dim, m->w_tiled, m->wt_tiled, m->bias,
                                     m->stream), "weight packing failed");
    return STAMP_OK;
}

extern "C" stamp_status stamp_mlp_forward(stamp_mlp* m, const float* x, int rows, float* y) {
    if (!m || !x || !y || !on_device(x) || !on_device(y)) return mlp_fail(STAMP_EINVAL, "NULL or non-device argument");
    if (rows < 1 || rows > m->max_rows) return mlp_fail(STAMP_EINVAL, "rows outside [1, max_rows]");
    MLP_TRY(stamp::mlp::forward(x, rows, m->in_dim, m->out_dim, m->w_tiled, m->bias, m->x_tiled,
                                m->ypad, y, nullptr, nullptr, 0, 0, m->err, m->sm_count, m->stream),
            "MLP forward launch failed");
    return STAMP_OK;
}

extern "C" stamp_status stamp_mlp_forward_saved(stamp_mlp* m, const float* x, int rows, float* y,
                                                int tile_base) {
    if (!m || !x || !y || !on_device(x) || !on_device(y)) return mlp_fail(STAMP_EINVAL, "NULL or non-device argument");
    const int tiles = (rows + 127) / 128;
    if (rows < 1 || rows > m->max_rows || tile_base < 0 || tile_base + tiles > m->tile_cap)
        return mlp_fail(STAMP_EINVAL, "rows / tile_base outside the saved-activation capacity");
    MLP_TRY(stamp::mlp::forward(x, rows, m->in_dim, m->out_dim, m->w_tiled, m->bias, m->x_tiled,
                                m->ypad, y, m->saved, m->zsave, tile_base, m->tile_cap, m->err,
                                m->sm_count, m->stream),
            "MLP forward launch failed");
    return STAMP_OK;
}

extern "C" stamp_status stamp_mlp_backward(stamp_mlp* m, const float* dy, int rows, int tile_base,
                                           float* dx, float* dparams) {
    if (!m || !dy || !on_device(dy) || (dx && !on_device(dx)) || (dparams && !on_device(dparams)))
        return mlp_fail(STAMP_EINVAL, "NULL or non-device argument");
    const int tiles = (rows + 127) / 128;
    if (rows < 1 || tile_base < 0 || tile_base + tiles > m->tile_cap)
        return mlp_fail(STAMP_EINVAL, "rows / tile_base outside the saved-activation capacity");
    MLP_TRY(stamp::mlp::backward(dy, rows, m->in_dim, m->out_dim, m->wt_tiled, m->zsave, m->dzsave,
                                 tile_base, m->tile_cap, dx, m->err, m->sm_count, m->stream),
            "MLP backward launch failed");
    if (dparams) {
        MLP_TRY(stamp::mlp::weight_grads(m->x_tiled, m->saved, m->dzsave, tile_base, m->tile_cap,
                                         rows, m->in_dim, m->out_dim, dparams, m->dw_part, m->err,
                                         m->sm_count, m->stream),
                "weight-gradient launch failed");
    }
    return STAMP_OK;
}

extern "C" stamp_status stamp_mlp_train(stamp_mlp* m, float* params, const float* x,
                                        const float* target, int rows, int epochs, int batch,
                                        float lr, float* loss_out) {
    if (!m || !params || !x || !target || !on_device(params) || !on_device(x) || !on_device(target))
        return mlp_fail(STAMP_EINVAL, "NULL or non-device argument");
    if (batch < 1 || batch > m->train_rows || batch > m->max_rows || rows < batch || epochs < 1)
        return mlp_fail(STAMP_EINVAL, "need 1 <= batch <= train_rows, rows >= batch, epochs >= 1");
    const int nb = rows / batch, n = batch * m->out_dim;
    std::vector<float> losses(epochs);
    for (int ep = 0; ep < epochs; ++ep) {
        MLP_TRY(cudaMemsetAsync(m->loss, 0, 4, m->stream), "memset failed");
        for (int b = 0; b < nb; ++b) {
            MLP_TRY(stamp::mlp::pack_weights(params, m->in_dim, m->out_dim, m->w_tiled, m->wt_tiled,
                                             m->bias, m->stream), "weight packing failed");
            MLP_TRY(stamp::mlp::forward(x + (size_t)b * batch * m->in_dim, batch, m->in_dim, m->out_dim,
                                        m->w_tiled, m->bias, m->x_tiled, m->ypad, m->ytrain, m->saved,
                                        m->zsave, 0, m->tile_cap, m->err, m->sm_count, m->stream),
                    "MLP forward launch failed");
            MLP_TRY(stamp::mlp::mse(m->ytrain, target + (size_t)b * n, n, m->dy, m->loss, m->stream),
                    "loss launch failed");
            MLP_TRY(stamp::mlp::backward(m->dy, batch, m->in_dim, m->out_dim, m->wt_tiled, m->zsave,
                                         m->dzsave, 0, m->tile_cap, nullptr, m->err, m->sm_count,
                                         m->stream), "MLP backward launch failed");
            MLP_TRY(stamp::mlp::weight_grads(m->x_tiled, m->saved, m->dzsave, 0, m->tile_cap, batch,
                                             m->in_dim, m->out_dim, m->grad, m->dw_part, m->err,
                                             m->sm_count, m->stream),
                    "weight-gradient launch failed");
            MLP_TRY(stamp::mlp::adam(params, m->grad, m->adam_m, m->adam_v, (int)m->n_params,
                                     ++m->step, lr, m->stream), "Adam launch failed");
        }
        float l = 0.f;
        MLP_TRY(cudaMemcpyAsync(&l, m->loss, 4, cudaMemcpyDeviceToHost, m->stream), "copy failed");
        MLP_TRY(cudaStreamSynchronize(m->stream), "synchronisation failed");
        losses[ep] = l / nb;
    }
    if (loss_out) std::memcpy(loss_out, losses.data(), epochs * sizeof(float));
    int f = 0;
    MLP_TRY(cudaMemcpy(&f, m->err, sizeof f, cudaMemcpyDeviceToHost), "flag read failed");
    if (f) {
        cudaMemset(m->err, 0, sizeof(int));
        return mlp_fail(STAMP_ETIMEOUT, "a bounded device wait of the MLP kernels gave up");
    }
    return STAMP_OK;
}

extern "C" stamp_status stamp_mlp_sync(stamp_mlp* m) {
    if (!m) return mlp_fail(STAMP_EINVAL, "NULL mlp");
    MLP_TRY(cudaStreamSynchronize(m->stream), "stream synchronisation failed");
    int f = 0;
    MLP_TRY(cudaMemcpy(&f, m->err, sizeof f, cudaMemcpyDeviceToHost), "flag read failed");
    if (f) {
        cudaMemset(m->err, 0, sizeof(int));
        return mlp_fail(STAMP_ETIMEOUT, "a bounded device wait of the MLP kernels gave up");
    }
    return STAMP_OK;
}
