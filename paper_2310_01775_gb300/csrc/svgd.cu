// Stein update of Algorithm 1 (Eq. svgd with unit weights), its median
// bandwidth, Adam, the initial particles and the final distinct-plan top-k.
//
// Bandwidth: h = med/ln(N+1), med the lower median (rank floor((M-1)/2)) of
// the M = N(N-1)/2 squared distances d2_ij, i<j -- the median heuristic the
// paper uses for its RBF kernels (App. C.3).  It is selected exactly by a
// three-digit radix select on the float bits (11 + 11 + 10 bits; the bits of
// non-negative floats order like the floats) over the d2 matrix, which stays
// in L2 (4 MB at N = 1024).  Each pass histograms one digit; the last CTA of
// the pass to finish (a device-scope counter, no waiting) picks the digit for
// the next pass, and the last pass writes h.
#include <climits>

#include "svgd_bodies.cuh"

namespace stamp {
namespace {

// d2 and the first median digit over 64 x 64 tile pairs: each thread owns 4 x 4
// pairs and walks the columns in chunks of 32, both tiles held column-major in
// shared memory (two 16-byte loads for 16 pairs, so the subtraction and the
// multiply-add per pair and column are the bound; one pair row and four pairs
// a thread, five 4-byte loads, was bound by the loads).  16-byte groups of
// rows are swizzled by the column so that storing a tile (4 rows x 8 columns
// a warp) meets no bank twice.  Two pairs per instruction (f32x2).  The sums
// over the columns run in column order.  GB300: 57 -> 26 us at N = 2048, D = 84,
// 454 -> 179 us at N = 6001, D = 108; 10 us at N = 1024, D = 16, as before.
constexpr int kPT = 64, kPC = 32;   // tile edge, columns per chunk
__device__ __forceinline__ int pw_at(int d, int row) {   // float index in a chunk
    return d * kPT + ((((row >> 2) ^ (d & 7)) << 2) | (row & 3));
}
// blockIdx.y: the matrix, of one or two side by side (the structured kernel's two
// bandwidths: too few CTAs each to fill the chip.  GB300, N = 1024: distances and
// the median's two passes 52 us one after the other, 29 side by side).
struct Matrix {
    const float* x;   // N x D
    int D;
    float* d2;
    unsigned *hist, *sel, *counter;
    float *h, *h_out;
};
struct Matrices { Matrix m[2]; };
__global__ void __launch_bounds__(256) pairwise_kernel(const __grid_constant__ Matrices ms, int N, int nt) {
    const Matrix& m = ms.m[blockIdx.y];
    const float* __restrict__ theta = m.x;
    float* __restrict__ d2 = m.d2;
    unsigned* __restrict__ hist = m.hist;
    const int D = m.D;
    // A and B chunks; the finished tile takes their place
    __shared__ __align__(16) float buf[kPT * (kPT + 1) > 2 * kPC * kPT ? kPT * (kPT + 1) : 2 * kPC * kPT];
    __shared__ unsigned h0[kBins0];
    float* A = buf;
    float* B = buf + kPC * kPT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // tile pair (bi <= bj) number blockIdx.x of the nt (nt + 1) / 2, row by row
    int bi = 0, left = blockIdx.x;
    while (left >= nt - bi) left -= nt - bi++;
    const int bj = bi + left, i0 = bi * kPT, j0 = bj * kPT;
    for (int t = tid; t < kBins0; t += 256) h0[t] = 0u;
    const int tx = tid & 15, ty = tid >> 4;
    f32x2 acc[4][2];
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[r][0] = acc[r][1] = 0ull;
    // this thread's elements of a chunk: column lane & 7 (+ 8 v), row (lane >> 3) + 4 warp (+ 32 u)
    const int lr = (lane >> 3) + 4 * warp, ld = lane & 7;
    for (int c0 = 0; c0 < D; c0 += kPC) {
        float va[2][4], vb[2][4];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const int d = c0 + ld + 8 * v, ra = i0 + lr + 32 * u, rb = j0 + lr + 32 * u;
                va[u][v] = d < D && ra < N ? theta[(size_t)ra * D + d] : 0.f;
                vb[u][v] = d < D && rb < N ? theta[(size_t)rb * D + d] : 0.f;
            }
        __syncthreads();   // the previous chunk is read
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                A[pw_at(ld + 8 * v, lr + 32 * u)] = va[u][v];
                B[pw_at(ld + 8 * v, lr + 32 * u)] = -vb[u][v];   // a - b as a + (-b)
            }
        __syncthreads();
        const int nd = min(kPC, D - c0);
#pragma unroll 8
        for (int d = 0; d < nd; ++d) {
            const float4 a = *reinterpret_cast<const float4*>(A + pw_at(d, 4 * ty));
            const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(B + pw_at(d, 4 * tx));
            const f32x2 av[4] = {pack2(a.x, a.x), pack2(a.y, a.y), pack2(a.z, a.z), pack2(a.w, a.w)};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const f32x2 e0 = add2(av[r], b.x), e1 = add2(av[r], b.y);
                acc[r][0] = fma2(e0, e0, acc[r][0]);
                acc[r][1] = fma2(e1, e1, acc[r][1]);
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            float lo, hi;
            unpack2(acc[r][q], lo, hi);
            float* p = buf + (4 * ty + r) * (kPT + 1) + 4 * tx + 2 * q;
            p[0] = lo;
            p[1] = hi;
        }
    __syncthreads();
    // coalesced rows of the tile and of its mirror; the pairs i < j counted by
    // digit, equal digits of a warp's 32 pairs at once (the distances of a set
    // share a few exponents: one atomic a pair would queue on a few counters)
    for (int t = tid; t < kPT * kPT; t += 256) {
        const int r = t / kPT, c = t % kPT, i = i0 + r, j = j0 + c;
        const float v = buf[r * (kPT + 1) + c];
        if (i < N && j < N) d2[(size_t)i * N + j] = v;
        const unsigned bin = i < j && j < N ? digit_of(__float_as_uint(v), 0) : 0xffffffffu;
        const unsigned same = __match_any_sync(0xffffffffu, bin);
        if (bin != 0xffffffffu && lane == __ffs(same) - 1) atomicAdd(&h0[bin], (unsigned)__popc(same));
        if (bi != bj) {   // r indexes j, c indexes i
            const int jm = j0 + r, im = i0 + c;
            if (jm < N && im < N) d2[(size_t)jm * N + im] = buf[c * (kPT + 1) + r];
        }
    }
    __syncthreads();
    for (int t = tid; t < kBins0; t += 256)
        if (h0[t]) atomicAdd(&hist[t], h0[t]);
    if (last_block(m.counter, gridDim.x)) {
        if (N < 2) {
            if (tid == 0) *m.h = 1.f;
            return;
        }
        unsigned b0, r0;
        find_bin<kBins0, 256>(hist, median_rank(N), b0, r0);
        if (tid == 0) { m.sel[0] = b0; m.sel[1] = r0; }
    }
}

// Batched: one CTA per work item (instance, tile row bi, tile column bj >= bi).
__global__ void __launch_bounds__(256) pairwise_batch_kernel(const SvgdInst* __restrict__ inst,
                                                             const int4* __restrict__ items,
                                                             const int* __restrict__ active) {
    const int4 it = items[blockIdx.x];
    const SvgdInst& g = inst[it.x];
    if (!active[g.gid]) return;
    pairwise_body(g.theta, g.N, g.D, g.d2, g.hist, g.sel, g.counter, g.h, it.y, it.z, g.nt);
}


__global__ void __launch_bounds__(256) median_digit_kernel(const __grid_constant__ Matrices ms, int N, int dg) {
    after_previous();
    const Matrix& m = ms.m[blockIdx.y];
    median_digit_body(N, dg, m.d2, m.hist, m.sel, m.counter + dg, m.h, m.h_out, blockIdx.x, gridDim.x);
}

// Batched: work item (instance, CTA index) of the instance's med_ctas CTAs.
__global__ void __launch_bounds__(256) median_digit_batch_kernel(const SvgdInst* __restrict__ inst,
                                                                 const int2* __restrict__ items,
                                                                 const int* __restrict__ active,
                                                                 int dg) {
    const int2 it = items[blockIdx.x];
    const SvgdInst& g = inst[it.x];
    if (!active[g.gid] || g.N < 2) return;
    median_digit_body(g.N, dg, g.d2, g.hist, g.sel, g.counter + dg, g.h, nullptr, it.y, g.med_ctas);
}


// CTAs per SM that the registers are kept to (GB300, N = 3000, D = 60: 92 -> 87 us with
// the bound, N = 4096, D = 144: 392 -> 383).
constexpr int phi_resident(int DP) { return DP <= 3 ? 4 : DP <= 4 ? 3 : 2; }
template <int DP>
__global__ void __launch_bounds__(kW * 32, phi_resident(DP)) phi_kernel(const float* theta, const float* grad,
                                                      int N, int D, const float* d2, const float* h_dev,
                                                      float* __restrict__ part, int shares,
                                                      int* err, const float* wn,
                                                      unsigned wait_limit, int skip_first, int row0,
                                                      int rows) {
    after_previous();
    phi_body<DP, kW, 8>(theta, grad, N, D, d2, h_dev, part, shares, err, blockIdx.x, blockIdx.y, wn,
                           wait_limit, skip_first != 0, row0, rows);
}

// Batched: work item (instance, row block, j-share); DP covers the batch's largest D.
template <int DP>
__global__ void __launch_bounds__(kW * 32) phi_batch_kernel(const SvgdInst* __restrict__ inst,
                                                            const int4* __restrict__ items,
                                                            const int* __restrict__ active,
                                                            int* err) {
    const int4 it = items[blockIdx.x];
    const SvgdInst& g = inst[it.x];
    if (!active[g.gid]) return;
    phi_body<DP>(g.theta, g.grad, g.N, g.D, g.d2, g.h, g.part, g.shares, err, it.y, it.z, nullptr,
                 kWaitLimit, false, 0, g.N);
}

// Adam (Kingma & Ba 2015) with gradient -phi, phi the in-order sum of the
// `shares` partial directions (stride n); optionally stores phi.  Flags
// non-finite inputs/results.
__global__ void adam_kernel(float* __restrict__ theta, const float* part, int shares,
                            float* __restrict__ phi_out, float* __restrict__ m,
                            float* __restrict__ v, int n, float lr, float bc1, float bc2,
                            int* flag) {
    after_previous();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    float phi = part[t];
    for (int q = 1; q < shares; ++q) phi += part[(size_t)q * n + t];
    if (phi_out) phi_out[t] = phi;
    float mt = m[t], vt = v[t], th = theta[t];
    if (!adam_update(-phi, lr, bc1, bc2, mt, vt, th)) atomicOr(flag, 1);
    m[t] = mt;
    v[t] = vt;
    theta[t] = th;
}

// Batched Adam over the concatenated particles of all instances: element t
// belongs to the last instance whose first element is <= t; its phi is the
// in-order sum of that instance's shares.  step is read on the device.
__global__ void adam_batch_kernel(float* __restrict__ theta, float* __restrict__ m,
                                  float* __restrict__ v, long long n, const SvgdInst* __restrict__ inst,
                                  int n_inst, const int* __restrict__ active,
                                  const int* __restrict__ step_dev, const float2* __restrict__ bc,
                                  float lr, int* flag) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    int lo = 0, hi = n_inst - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&inst[mid].elem0) <= t) lo = mid; else hi = mid - 1;
    }
    const SvgdInst& g = inst[lo];
    const long long loc = t - g.elem0, ne = (long long)g.N * g.D;
    if (loc >= ne || !active[g.gid]) return;
    const float* part = g.part;
    float phi = part[loc];
    for (int q = 1; q < g.shares; ++q) phi += part[(size_t)q * ne + loc];
    const float2 b12 = bc[*step_dev + 1];
    float mt = m[t], vt = v[t], th = theta[t];
    if (!adam_update(-phi, lr, b12.x, b12.y, mt, vt, th)) atomicOr(flag, 1);
    m[t] = mt;
    v[t] = vt;
    theta[t] = th;
}

// A whole Stein step of at most kSmallN particles in one CTA: distances, their
// exact lower median (bisection on the float bits), direction and Adam.  The
// six launches it replaces cost more than their work (N = 32, D = 12: 30 us
// against 9).
// Every sum has the terms and the order of the kernels above and of phi_body, 32
// particles a share, so an instance of a batch moves as one solved alone does.
template <int E>   // N <= E (32 or 64)
__global__ void __launch_bounds__(1024) small_step_kernel(
    float* __restrict__ theta, const float* __restrict__ grad, int N, int D, float* __restrict__ m,
    float* __restrict__ v, const float* __restrict__ wn, float lr, float bc1, float bc2,
    float* __restrict__ h_dev, float* __restrict__ h_out, float* __restrict__ phi_out, int* flag) {
    extern __shared__ float ssm[];
    const int ld = D | 1;   // odd row stride: rows fall in different banks
    float* T = ssm;
    float* G = T + E * ld;
    __shared__ float K[E][E + 1];   // d2, then the kernel values
    const int tid = threadIdx.x;
    for (int t = tid; t < N * D; t += 1024) {
        T[(t / D) * ld + t % D] = theta[t];
        G[(t / D) * ld + t % D] = grad[t];
    }
    __syncthreads();
    for (int t = tid; t < N * N; t += 1024) {
        const int i = t / N, j = t % N;
        if (i <= j) {
            float a = 0.f;
            for (int d = 0; d < D; ++d) {
                const float e = T[i * ld + d] - T[j * ld + d];
                a = fmaf(e, e, a);
            }
            K[i][j] = K[j][i] = a;
        }
    }
    __syncthreads();
    // the lower median of the pairs: the smallest value with more than `rank` values <= it
    const int pairs = N * (N - 1) / 2;
    constexpr int V = E * E / 1024;
    unsigned val[V];
#pragma unroll
    for (int q = 0; q < V; ++q) {
        const int t = tid + q * 1024, i = t / E, j = t % E;
        val[q] = i < j && j < N ? __float_as_uint(K[i][j]) : 0xffffffffu;
    }
    float h = 1.f;
    if (N >= 2) {
        const int rank = (pairs - 1) / 2;
        unsigned lo = 0u, hi = 0xffffffffu;   // the answer lies in [lo, hi]
        while (lo < hi) {
            const unsigned mid = lo + (hi - lo) / 2;
            int c = 0;
#pragma unroll
            for (int q = 0; q < V; ++q) c += __syncthreads_count(val[q] <= mid);
            if (c > rank) hi = mid; else lo = mid + 1;
        }
        h = __uint_as_float(lo) / logf((float)N + 1.f);
        h = (h >= 1e-12f) ? h : 1.f;
    }
    if (tid == 0) {
        *h_dev = h;
        if (h_out) *h_out = h;
    }
    const float inv_h = 1.f / h, m2h = -2.f * inv_h;
    for (int t = tid; t < N * N; t += 1024) {
        const int i = t / N, j = t % N;
        float k = 0.f;
        if (i != j) {
            k = expf(-K[i][j] * inv_h);
            if (wn) k *= wn[j];
        }
        K[i][j] = k;
    }
    __syncthreads();
    const float inv_n = wn ? 1.f : 1.f / (float)N;
    for (int t = tid; t < N * D; t += 1024) {
        const int i = t / D, d = t % D;
        const float ti = T[i * ld + d], self = wn ? wn[i] : 1.f;
        float phi = 0.f;
        for (int j0 = 0; j0 < N; j0 += kTJ) {
            float a = 0.f;
            for (int j = j0; j < min(N, j0 + kTJ); ++j)
                a = fmaf(K[i][j], fmaf(m2h, T[j * ld + d] - ti, G[j * ld + d]), a);
            if (self != 0.f && i / kTJ == j0 / kTJ) a = fmaf(self, G[i * ld + d], a);
            const float share = __fmul_rn(a, inv_n);
            phi = j0 ? __fadd_rn(phi, share) : share;
        }
        if (phi_out) phi_out[t] = phi;
        float mt = m[t], vt = v[t], th = ti;
        if (!adam_update(-phi, lr, bc1, bc2, mt, vt, th)) atomicOr(flag, 1);
        m[t] = mt;
        v[t] = vt;
        theta[t] = th;
    }
}

// Eq. dsvgd weights, normalised: w_j = exp(C_j - C~_j - max) / sum, C the hard
// and C~ the relaxed cost of particle j; a non-finite difference weighs 0.
// One CTA; fixed per-thread strides and a fixed tree: deterministic.
__global__ void __launch_bounds__(1024) dsvgd_weights_kernel(const float* __restrict__ c_relaxed,
                                                            const float* __restrict__ c_hard, int N,
                                                            float* __restrict__ wn) {
    __shared__ float red[1024];
    float mx = -INFINITY;
    for (int j = threadIdx.x; j < N; j += 1024) {
        const float d = c_hard[j] - c_relaxed[j];
        if (isfinite(d)) mx = fmaxf(mx, d);
    }
    red[threadIdx.x] = mx;
    __syncthreads();
    for (int o = 512; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] = fmaxf(red[threadIdx.x], red[threadIdx.x + o]);
        __syncthreads();
    }
    mx = red[0];
    __syncthreads();
    float sum = 0.f;
    for (int j = threadIdx.x; j < N; j += 1024) {
        const float d = c_hard[j] - c_relaxed[j];
        const float e = isfinite(d) ? expf(d - mx) : 0.f;
        wn[j] = e;
        sum += e;
    }
    red[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 512; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    const float inv = red[0] > 0.f ? 1.f / red[0] : 0.f;
    for (int j = threadIdx.x; j < N; j += 1024) wn[j] *= inv;
}

__global__ void init_theta_kernel(float* theta, int n, uint64_t key) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) theta[t] = 2.f * u23(sm64(key, (uint64_t)t)) - 1.f;
}

// Distinct-plan top-k: sort (cost bits, index) ascending, then keep the first
// k distinct argmax sequences (Gamma, Eq. gamma_map; ties to the lowest index).
__device__ __forceinline__ void topk_body(const float* __restrict__ theta,
                                          const float* __restrict__ cost, int N, int H, int M, int P,
                                          int k, int* out) {
    extern __shared__ unsigned long long sk[];
    int n2 = 1;
    while (n2 < N) n2 <<= 1;
    unsigned long long* key = sk;
    unsigned long long* code = sk + n2;
    for (int t = threadIdx.x; t < n2; t += blockDim.x) {
        if (t < N) {
            unsigned cb = __float_as_uint(cost[t]);
            if (cb & 0x80000000u) cb = 0xFFFFFFFFu;   // costs are >= 0; anything else last
            key[t] = ((unsigned long long)cb << 32) | (unsigned)t;
            unsigned long long cd = 0;
            for (int a = 0; a < H; ++a) {
                const float* lg = theta + (size_t)t * H * P + a * P;
                int best = 0;
                float bv = lg[0];
                for (int c = 1; c < M; ++c)
                    if (lg[c] > bv) { bv = lg[c]; best = c; }
                cd |= (unsigned long long)best << (4 * a);
            }
            code[t] = cd;
        } else {
            key[t] = ~0ull;
        }
    }
    __syncthreads();
    for (int size = 2; size <= n2; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int t = threadIdx.x; t < n2; t += blockDim.x) {
                const int p = t ^ stride;
                if (p > t) {
                    const bool up = (t & size) == 0;
                    const unsigned long long a = key[t], b = key[p];
                    if ((a > b) == up) { key[t] = b; key[p] = a; }
                }
            }
            __syncthreads();
        }
    if (threadIdx.x == 0) {
        int got = 0;
        for (int r = 0; r < N && got < k; ++r) {
            const int idx = (int)(key[r] & 0xFFFFFFFFu);
            const unsigned long long cd = code[idx];
            bool dup = false;
            for (int q = 0; q < got; ++q) dup |= code[out[q]] == cd;
            if (!dup) out[got++] = idx;
        }
        for (int q = got; q < k; ++q) out[q] = -1;
    }
}

__global__ void __launch_bounds__(1024) topk_kernel(const float* __restrict__ theta,
                                                    const float* __restrict__ cost, int N, int H,
                                                    int M, int P, int k, int* out) {
    topk_body(theta, cost, N, H, M, P, k, out);
}
// One CTA per instance (64 launches of one CTA each took 1.9 ms, one of 64 CTAs 0.05).
__global__ void __launch_bounds__(1024) topk_batch_kernel(const InstItem* __restrict__ items) {
    const InstItem& it = items[blockIdx.x];
    topk_body(it.theta, it.cost, it.N, it.H, it.M, it.M + 2, it.k, it.topk);
}

__global__ void init_theta_batch_kernel(const InstItem* __restrict__ items, int n, long long n_elem) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_elem) return;
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&items[mid].elem0) <= t) lo = mid; else hi = mid - 1;
    }
    const InstItem& it = items[lo];
    const long long loc = t - it.elem0;
    if (loc < (long long)it.N * it.H * (it.M + 2)) it.theta[loc] = 2.f * u23(sm64(it.key, (uint64_t)loc)) - 1.f;
}

template <int DP>
cudaError_t phi_launch(const float* theta, const float* grad, int N, int D, const float* d2,
                       const float* h_dev, float* part, int shares, int* err, const float* wn,
                       unsigned wait_limit, int skip_first, int row0, int rows, bool chained,
                       cudaStream_t st) {
    const size_t smem = phi_smem(D, DP, kW);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(phi_kernel<DP>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const int per_cta = kW * kR;
    const dim3 grid((rows + per_cta - 1) / per_cta, shares);
    if (chained)
        return launch_after(phi_kernel<DP>, grid, kW * 32, smem, st, theta, grad, N, D, d2, h_dev, part, shares,
                            err, wn, wait_limit, skip_first, row0, rows);
    phi_kernel<DP><<<grid, kW * 32, smem, st>>>(theta, grad, N, D, d2, h_dev, part, shares, err, wn, wait_limit,
                                                   skip_first, row0, rows);
    return cudaGetLastError();
}
// Shares of the Stein sum of N particles: the tiles of the busiest SM, CTAs times
// tiles of the longest share, are the time (GB300, D = 108, N = 6001: 2.3 to 2.5 us a tile
// at any split, 561 us at 4 shares, 618 at 5); among equal ones the more CTAs, which
// hide more latency.  A function of N alone, so that a shard of the rows sums as
// all do; at most max_shares.
int phi_plan(int N, int max_shares) {
    const int sms = sm_count(), rows = (N + kR * kW - 1) / (kR * kW), tiles = (N + kTJ - 1) / kTJ;
    int best = 1;
    long long least = LLONG_MAX;
    for (int s = 1; s <= max_shares && s <= tiles; ++s) {
        const long long t = (long long)((rows * s + sms - 1) / sms) * ((tiles + s - 1) / s);
        if (t <= least) {
            least = t;
            best = s;
        }
    }
    return best;
}

}  // namespace

static Matrix matrix(const float* x, int D, const SvgdScratch& s, float* h_out) {
    return Matrix{x, D, s.d2, s.hist, s.sel, s.counter, s.h, h_out};
}
static cudaError_t pairwise(const Matrices& ms, int n, int N, cudaStream_t st) {
    const int nt = (N + kPT - 1) / kPT;
    pairwise_kernel<<<dim3(nt * (nt + 1) / 2, n), 256, 0, st>>>(ms, N, nt);
    return cudaGetLastError();
}
static cudaError_t median_digit(const Matrices& ms, int n, int N, int digit, cudaStream_t st) {
    // a CTA flushes its bins once: few CTAs for a small matrix (two a SM: 13 us
    // a digit at N = 2048, 18 with six), more loads in flight for a large one
    // (N = 6001: 42 + 34 us for the two digits with two, 27 + 21 with six)
    const int cap = (N >= 4096 ? 6 : 2) * sm_count();
    int grid = N - 1 < cap ? N - 1 : cap;
    if (grid < 1) grid = 1;
    return launch_after(median_digit_kernel, dim3(grid, n), 256, 0, st, ms, N, digit);
}
cudaError_t launch_pairwise(const float* theta, int N, int D, const SvgdScratch& s,
                            cudaStream_t st) {
    return pairwise(Matrices{{matrix(theta, D, s, nullptr)}}, 1, N, st);
}
cudaError_t launch_median_digit(int N, int digit, const SvgdScratch& s, float* h_out,
                                cudaStream_t st) {
    return median_digit(Matrices{{matrix(nullptr, 0, s, h_out)}}, 1, N, digit, st);
}
cudaError_t launch_pairwise2(const float* x0, int D0, const SvgdScratch& s0, const float* x1, int D1,
                             const SvgdScratch& s1, int N, cudaStream_t st) {
    return pairwise(Matrices{{matrix(x0, D0, s0, nullptr), matrix(x1, D1, s1, nullptr)}}, 2, N, st);
}
cudaError_t launch_median_digit2(int N, int digit, const SvgdScratch& s0, const SvgdScratch& s1,
                                 cudaStream_t st) {
    return median_digit(Matrices{{matrix(nullptr, 0, s0, nullptr), matrix(nullptr, 0, s1, nullptr)}}, 2, N,
                        digit, st);
}

cudaError_t launch_phi_rows(const float* theta, const float* grad, int N, int D, int row0,
                            int rows, const SvgdScratch& s, float* part, int max_shares, int* shares,
                            cudaStream_t st, const float* wn) {
    // TMA bulk copies need 16-byte aligned sources
    if ((reinterpret_cast<uintptr_t>(theta) | reinterpret_cast<uintptr_t>(grad)) & 15u)
        return cudaErrorMisalignedAddress;
    *shares = phi_plan(N, max_shares);
    const unsigned limit = s.wait_limit ? s.wait_limit : kWaitLimit;
    const int dp = (D + 31) / 32;
    switch (dp) {
        case 1: return phi_launch<1>(theta, grad, N, D, s.d2, s.h, part, *shares, s.err, wn, limit, s.skip_first_copy, row0, rows, s.chained, st);
        case 2: return phi_launch<2>(theta, grad, N, D, s.d2, s.h, part, *shares, s.err, wn, limit, s.skip_first_copy, row0, rows, s.chained, st);
        case 3: return phi_launch<3>(theta, grad, N, D, s.d2, s.h, part, *shares, s.err, wn, limit, s.skip_first_copy, row0, rows, s.chained, st);
        case 4: return phi_launch<4>(theta, grad, N, D, s.d2, s.h, part, *shares, s.err, wn, limit, s.skip_first_copy, row0, rows, s.chained, st);
        case 5: case 6:
            return phi_launch<6>(theta, grad, N, D, s.d2, s.h, part, *shares, s.err, wn, limit, s.skip_first_copy, row0, rows, s.chained, st);
        case 7: case 8: case 9:
            return phi_launch<9>(theta, grad, N, D, s.d2, s.h, part, *shares, s.err, wn, limit, s.skip_first_copy, row0, rows, s.chained, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_phi(const float* theta, const float* grad, int N, int D, const SvgdScratch& s,
                       float* part, int max_shares, int* shares, cudaStream_t st, const float* wn) {
    return launch_phi_rows(theta, grad, N, D, 0, N, s, part, max_shares, shares, st, wn);
}

cudaError_t launch_adam(float* theta, const float* part, int shares, float* phi_out, float* m,
                        float* v, int n, int step, float lr, int* flag, cudaStream_t st) {
    const float bc1 = 1.f - powf(0.9f, (float)step);
    const float bc2 = 1.f - powf(0.999f, (float)step);
    return launch_after(adam_kernel, dim3((n + 255) / 256), 256, 0, st, theta, part, shares, phi_out, m, v,
                        n, lr, bc1, bc2, flag);
}

cudaError_t launch_small_step(float* theta, const float* grad, int N, int D, float* m, float* v,
                              const float* wn, int step, float lr, const SvgdScratch& s, float* h_out,
                              float* phi_out, cudaStream_t st) {
    const int edge = N <= 32 ? 32 : kSmallN;
    const size_t smem = (size_t)2 * edge * (D | 1) * sizeof(float);   // up to 148 KB
    auto* kernel = N <= 32 ? small_step_kernel<32> : small_step_kernel<kSmallN>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const float bc1 = 1.f - powf(0.9f, (float)step);
    const float bc2 = 1.f - powf(0.999f, (float)step);
    kernel<<<1, 1024, smem, st>>>(theta, grad, N, D, m, v, wn, lr, bc1, bc2, s.h, h_out, phi_out, s.err);
    return cudaGetLastError();
}

cudaError_t launch_pairwise_batch(const SvgdInst* inst, const int4* items, int n_items, int max_D,
                                  const int* active, cudaStream_t st) {
    const size_t smem = 2 * kTile * (max_D + 1) * sizeof(float);
    if (smem + kPairwiseStatic > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(pairwise_batch_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    pairwise_batch_kernel<<<n_items, 256, smem, st>>>(inst, items, active);
    return cudaGetLastError();
}

cudaError_t launch_median_digit_batch(const SvgdInst* inst, const int2* items, int n_items,
                                      const int* active, int digit, cudaStream_t st) {
    median_digit_batch_kernel<<<n_items, 256, 0, st>>>(inst, items, active, digit);
    return cudaGetLastError();
}

int phi_batch_shares(int N) { return phi_plan(N, kMaxShares); }
int phi_rows_per_block() { return kW * kR; }

template <int DP>
cudaError_t phi_batch_launch(const SvgdInst* inst, const int4* items, int n_items, int max_D,
                             const int* active, int* err, cudaStream_t st) {
    const size_t smem = phi_smem(max_D, DP, kW);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(phi_batch_kernel<DP>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    phi_batch_kernel<DP><<<n_items, kW * 32, smem, st>>>(inst, items, active, err);
    return cudaGetLastError();
}

cudaError_t launch_phi_batch(const SvgdInst* inst, const int4* items, int n_items, int max_D,
                             const int* active, int* err, cudaStream_t st) {
    switch ((max_D + 31) / 32) {
        case 1: return phi_batch_launch<1>(inst, items, n_items, max_D, active, err, st);
        case 2: return phi_batch_launch<2>(inst, items, n_items, max_D, active, err, st);
        case 3: return phi_batch_launch<3>(inst, items, n_items, max_D, active, err, st);
        case 4: return phi_batch_launch<4>(inst, items, n_items, max_D, active, err, st);
        case 5: case 6: return phi_batch_launch<6>(inst, items, n_items, max_D, active, err, st);
        case 7: case 8: case 9: return phi_batch_launch<9>(inst, items, n_items, max_D, active, err, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_adam_batch(float* theta, float* m, float* v, long long n, const SvgdInst* inst,
                              int n_inst, const int* active, const int* step_dev, const float2* bc,
                              float lr, int* flag, cudaStream_t st) {
    adam_batch_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(theta, m, v, n, inst, n_inst, active,
                                                                   step_dev, bc, lr, flag);
    return cudaGetLastError();
}

cudaError_t launch_dsvgd_weights(const float* c_relaxed, const float* c_hard, int N, float* wn,
                                 cudaStream_t st) {
    dsvgd_weights_kernel<<<1, 1024, 0, st>>>(c_relaxed, c_hard, N, wn);
    return cudaGetLastError();
}

cudaError_t launch_init_theta(float* theta, int N, int D, uint64_t seed, cudaStream_t st) {
    const int n = N * D;
    init_theta_kernel<<<(n + 255) / 256, 256, 0, st>>>(theta, n, sm64(seed, kStreamInit));
    return cudaGetLastError();
}

cudaError_t launch_topk(const float* theta, const float* cost, int N, const SimConst& sc, int k,
                        int* topk_out, cudaStream_t st) {
    int n2 = 1;
    while (n2 < N) n2 <<= 1;
    const size_t smem = (size_t)2 * n2 * sizeof(unsigned long long);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(topk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
    }
    topk_kernel<<<1, 1024, smem, st>>>(theta, cost, N, sc.H, sc.M, sc.P, k, topk_out);
    return cudaGetLastError();
}

cudaError_t launch_topk_batch(const InstItem* items, int n, int max_n, cudaStream_t st) {
    int n2 = 1;
    while (n2 < max_n) n2 <<= 1;
    const size_t smem = (size_t)2 * n2 * sizeof(unsigned long long);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(topk_batch_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    topk_batch_kernel<<<n, 1024, smem, st>>>(items);
    return cudaGetLastError();
}

cudaError_t launch_init_theta_batch(const InstItem* items, int n, long long n_elem, cudaStream_t st) {
    init_theta_batch_kernel<<<(unsigned)((n_elem + 255) / 256), 256, 0, st>>>(items, n, n_elem);
    return cudaGetLastError();
}

}  // namespace stamp
