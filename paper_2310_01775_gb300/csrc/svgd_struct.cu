// Stein direction with the structured kernel of App. D.3, restated for plans
// of [logits a_k, offset parameter u_k, distance parameter v_k] per action:
//   K(a, b) = (1/2H) sum_k [ exp(-|c_k(a) - c_k(b)|^2 / h_c)
//                            + exp(-|softmax(a_k) - softmax(b_k)|^2 / h_z) ],
// c_k = (u_k, v_k), K(a, a) = 1.  (The paper's kernel is defined on DMP goal
// poses: RBF on goal positions, RBF on softmax(a_k), von Mises on goal yaws;
// these plans have push parameters where it has goal positions and no angle.)
// phi_i = sum_j wn_j [K_ji grad log rho_j + grad_{theta_j} K_ji], wn_j = 1/N or
// the normalised weights of Eq. dsvgd, with
//   grad_{u,v of action k} K_ji = (1/2H)(2/h_c) e^c_ijk (c_ik - c_jk),
//   grad_{a_jk} K_ji          = (1/2H)(2/h_z) e^z_ijk J(a_jk)^T (s_ik - s_jk),
//   J^T x = s (x - s.x)  (softmax Jacobian, symmetric).
// h_c, h_z: the median heuristic on the concatenated component (pairwise
// distances and radix-select median of svgd.cu) divided by H.
#include <cstdint>

#include "stamp_internal.cuh"

namespace stamp {
namespace {

constexpr int kTJ = 32;         // j per tile
constexpr int kMaxHs = 16;      // actions per plan

// C (N x 2H): (u_k, v_k); S (N x M H): softmax(a_k).
__global__ void struct_prep_kernel(const float* __restrict__ theta, int N, int H, int M,
                                   float* __restrict__ C, float* __restrict__ S) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= N * H) return;
    const int i = t / H, k = t % H, P = M + 2;
    const float* a = theta + (size_t)i * H * P + k * P;
    float mx = a[0];
    for (int c = 1; c < M; ++c) mx = fmaxf(mx, a[c]);
    float sum = 0.f;
    float* s = S + (size_t)i * M * H + k * M;
    for (int c = 0; c < M; ++c) {
        const float e = expf(a[c] - mx);
        s[c] = e;
        sum += e;
    }
    const float inv = 1.f / sum;
    for (int c = 0; c < M; ++c) s[c] *= inv;
    C[(size_t)i * 2 * H + 2 * k] = a[M];
    C[(size_t)i * 2 * H + 2 * k + 1] = a[M + 1];
}

// HP lanes (H rounded up to a power of two) own kRows rows of the plan, a lane an
// action of each: its softmax row, its (u, v) and the accumulators of its M + 2
// columns stay in registers, a pair's exponentials are computed once, and K is
// their sum over the lanes.  Tiles of theta's, the softmax's and grad's columns
// are staged in shared memory, where the lanes of an action read the same
// address.  What bounds it is arithmetic, about 10 + 7 (M + 2) operations per
// pair and action; kSplit warps share the rows of a tile's j to keep enough of
// them in flight, and are summed in order at the end.  GB300, N = 1024, H = 4, M =
// 4: 68 -> 19.8 us (a lane per column read the pair's exponentials, computed by
// other threads, from shared memory: five reads per pair and column).
constexpr int kRows = 2, kSplit = 4, kWarps = 8;
template <int HP>
constexpr int kCtaRows = kWarps / kSplit * (32 / HP) * kRows;

template <int M, int HP>
__global__ void __launch_bounds__(kWarps * 32)
struct_phi_kernel(const float* theta, const float* grad, const float* S, int N, int H,
                  const float* hc_dev, const float* hz_dev, const float* wn, float* __restrict__ phi,
                  int j_chunk) {
    extern __shared__ float ssm[];
    constexpr int P = M + 2, kGroups = 32 / HP;
    const int D = H * P;
    float* Xj = ssm;               // kTJ x D: softmax(a_k) on the logits, theta on (u_k, v_k)
    float* Gj = Xj + kTJ * D;      // kTJ x D
    float* Wj = Gj + kTJ * D;      // kTJ
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int split = warp % kSplit, k = lane % HP, ks = k < H ? k : 0;
    const int row0 = (warp / kSplit * kGroups + lane / HP) * kRows, i0 = blockIdx.x * kCtaRows<HP>;
    after_previous();
    const float Hf = (float)H;
    const float inv_hc = Hf / *hc_dev, inv_hz = Hf / *hz_dev;   // h = h_plain / H
    const float alpha = 0.5f / Hf, ac = alpha * (2.f * inv_hc), az = alpha * (2.f * inv_hz);
    float xi[kRows][P], acc[kRows][P];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const int i = i0 + row0 + r;
#pragma unroll
        for (int c = 0; c < P; ++c) {
            xi[r][c] = i >= N ? 0.f
                       : c < M ? S[(size_t)i * M * H + ks * M + c] : theta[(size_t)i * D + ks * P + c];
            acc[r][c] = 0.f;
        }
    }
    // this CTA's share of the sum over j; partial directions go to share blockIdx.y
    const int jb = blockIdx.y * j_chunk, je = min(N, jb + j_chunk);
    phi += (size_t)blockIdx.y * N * D;
    for (int j0 = jb; j0 < je; j0 += kTJ) {
        const int nj = min(kTJ, je - j0);
        for (int t = tid; t < nj * H; t += kWarps * 32) {
            const int jj = t / H, q = t - jj * H;
            const float* s = S + (size_t)(j0 + jj) * M * H + q * M;
            const float* th = theta + (size_t)(j0 + jj) * D + q * P;
            float* x = Xj + t * P;
#pragma unroll
            for (int c = 0; c < P; ++c) x[c] = c < M ? s[c] : th[c];
        }
        for (int t = tid; t < nj * D; t += kWarps * 32) Gj[t] = grad[(size_t)j0 * D + t];
        if (tid < nj) Wj[tid] = wn ? wn[j0 + tid] : 1.f;
        __syncthreads();
#pragma unroll 2
        for (int jj = split; jj < nj; jj += kSplit) {
            const float2* xp = reinterpret_cast<const float2*>(Xj + jj * D + ks * P);
            const float2* gp = reinterpret_cast<const float2*>(Gj + jj * D + ks * P);
            const float w = Wj[jj];
            float x[P], g[P];
#pragma unroll
            for (int c = 0; c < P / 2; ++c) {
                const float2 xv = xp[c], gv = gp[c];
                x[2 * c] = xv.x; x[2 * c + 1] = xv.y;
                g[2 * c] = gv.x; g[2 * c + 1] = gv.y;
            }
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
                float dz = 0.f, q = 0.f, df[P];
#pragma unroll
                for (int c = 0; c < P; ++c) df[c] = xi[r][c] - x[c];
#pragma unroll
                for (int c = 0; c < M; ++c) {
                    dz = fmaf(df[c], df[c], dz);
                    q = fmaf(x[c], df[c], q);
                }
                const float ec = expf(-(df[M] * df[M] + df[M + 1] * df[M + 1]) * inv_hc);
                const float ez = expf(-dz * inv_hz);
                float sum = k < H ? ec + ez : 0.f;
#pragma unroll
                for (int o = 1; o < HP; o <<= 1) sum += __shfl_xor_sync(~0u, sum, o);
                const float K = alpha * sum * w, Az = az * w * ez, Ac = ac * w * ec;
                // logits: A^z s_j ((s_i - s_j) - q); offset, distance: A^c (c_i - c_j)
#pragma unroll
                for (int c = 0; c < P; ++c) {
                    const float rep = c < M ? Az * (x[c] * (df[c] - q)) : Ac * df[c];
                    acc[r][c] = fmaf(K, g[c], acc[r][c] + rep);
                }
            }
        }
        __syncthreads();
    }
    // the splits' sums, in order: split x row x column
    float* sums = ssm;
    if (k < H)
#pragma unroll
        for (int r = 0; r < kRows; ++r)
#pragma unroll
            for (int c = 0; c < P; ++c)
                sums[((size_t)split * kCtaRows<HP> + row0 + r) * D + k * P + c] = acc[r][c];
    __syncthreads();
    const float scale = wn ? 1.f : 1.f / (float)N;
    const int n = min(kCtaRows<HP>, N - i0) * D;
    for (int t = tid; t < n; t += kWarps * 32) {
        float v = sums[t];
#pragma unroll
        for (int q = 1; q < kSplit; ++q) v += sums[q * kCtaRows<HP> * D + t];
        phi[(size_t)i0 * D + t] = v * scale;
    }
}

template <int M, int HP>
cudaError_t struct_launch(const float* theta, const float* grad, const float* S, int N, int H,
                          const float* hc, const float* hz, const float* wn, float* phi, int max_shares,
                          int* shares, cudaStream_t st) {
    const int D = H * (M + 2), rows = (N + kCtaRows<HP> - 1) / kCtaRows<HP>;
    // split the sum over j so that about two CTAs (16 warps) per SM are in flight
    int want = (2 * sm_count() + rows - 1) / rows;
    want = want < 1 ? 1 : (want > max_shares ? max_shares : want);
    const int j_chunk = ((N + want - 1) / want + kTJ - 1) / kTJ * kTJ;
    *shares = (N + j_chunk - 1) / j_chunk;
    const size_t tile = (2 * (size_t)kTJ * D + kTJ) * sizeof(float);
    const size_t sums = (size_t)kSplit * kCtaRows<HP> * D * sizeof(float);
    const size_t smem = tile > sums ? tile : sums;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(struct_phi_kernel<M, HP>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    return launch_after(struct_phi_kernel<M, HP>, dim3(rows, *shares), kWarps * 32, smem, st, theta, grad, S, N,
                        H, hc, hz, wn, phi, j_chunk);
}

__global__ void scale_scalar_kernel(const float* src, float s, float* dst) { *dst = *src * s; }

}  // namespace

cudaError_t launch_scale_scalar(const float* src, float s, float* dst, cudaStream_t st) {
    scale_scalar_kernel<<<1, 1, 0, st>>>(src, s, dst);
    return cudaGetLastError();
}

cudaError_t launch_struct_prep(const float* theta, int N, int H, int M, float* C, float* S,
                               cudaStream_t st) {
    struct_prep_kernel<<<(N * H + 127) / 128, 128, 0, st>>>(theta, N, H, M, C, S);
    return cudaGetLastError();
}

cudaError_t launch_struct_phi(const float* theta, const float* grad, const float* S,
                              int N, int H, int M, const float* hc_dev, const float* hz_dev,
                              const float* wn, float* phi, int max_shares, int* shares,
                              cudaStream_t st) {
    if (H < 1 || H > kMaxHs) return cudaErrorInvalidValue;
#define STRUCT_HP(M_, HP_) \
    return struct_launch<M_, HP_>(theta, grad, S, N, H, hc_dev, hz_dev, wn, phi, max_shares, shares, st)
#define STRUCT_M(M_)                    \
    if (H == 1) STRUCT_HP(M_, 1);       \
    if (H == 2) STRUCT_HP(M_, 2);       \
    if (H <= 4) STRUCT_HP(M_, 4);       \
    if (H <= 8) STRUCT_HP(M_, 8);       \
    STRUCT_HP(M_, 16)
    switch (M) {
        case 4: STRUCT_M(4);
        case 8: STRUCT_M(8);
        case 12: STRUCT_M(12);
        case 16: STRUCT_M(16);
    }
#undef STRUCT_M
#undef STRUCT_HP
    return cudaErrorInvalidValue;
}

}  // namespace stamp
