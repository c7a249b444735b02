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

constexpr int kTJ = 16;         // j per tile
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

// A warp owns kRowsPerWarp rows; lane l owns columns l, l + 32, ... of each.  A
// tile's grad, theta (its offsets and distances) and softmax rows are staged in
// shared memory once per CTA; each pair and action costs two exponentials and
// M multiply-adds there, spread over the CTA's threads, and each pair and
// column four multiply-adds per lane.  The exponentials' weights (w_j, alpha,
// 2/h) are folded into what is stored: A_ijk = alpha w_j (2/h) e_ijk.  GB300, N =
// 1024, H = 4, M = 4: 184 -> 68 us (every lane used to read its j's values from
// global memory, one row per warp).
constexpr int kRowsPerWarp = 2, kWarps = 8, kRows = kRowsPerWarp * kWarps;
__host__ __device__ constexpr size_t struct_smem(int D, int H) {
    return ((size_t)(2 * kTJ + kRows) * D + (size_t)kRows * kTJ * (3 * H + 1)) * sizeof(float);
}
template <int DP>
__global__ void __launch_bounds__(kWarps * 32)
struct_phi_kernel(const float* __restrict__ theta, const float* __restrict__ grad,
                  const float* __restrict__ S, int N, int H, int M,
                  const float* __restrict__ hc_dev, const float* __restrict__ hz_dev,
                  const float* __restrict__ wn, float* __restrict__ phi, int j_chunk) {
    extern __shared__ float ssm[];
    const int P = M + 2, D = H * P;
    // per column: softmax(a_k) on the logits, theta on (u_k, v_k)
    float* Xi = ssm;                   // kRows x D
    float* Xj = Xi + kRows * D;        // kTJ x D
    float* Gj = Xj + kTJ * D;          // kTJ x D
    float* Ac = Gj + kTJ * D;          // kRows x kTJ x H: alpha w_j (2/h_c) e^c
    float* Az = Ac + kRows * kTJ * H;  // alpha w_j (2/h_z) e^z
    float* Q = Az + kRows * kTJ * H;   // s_j . (s_i - s_j)
    float* Ks = Q + kRows * kTJ * H;   // kRows x kTJ: w_j K_ij
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int i0 = blockIdx.x * kRows;
    const float Hf = (float)H;
    const float inv_hc = Hf / __ldg(hc_dev), inv_hz = Hf / __ldg(hz_dev);   // h = h_plain / H
    const float alpha = 0.5f / Hf, ac = alpha * (2.f * inv_hc), az = alpha * (2.f * inv_hz);
    auto column = [&](int i, int d) {   // X of particle i
        const int k = d / P, c = d - k * P;
        return c < M ? S[(size_t)i * M * H + k * M + c] : theta[(size_t)i * D + d];
    };
    for (int t = tid; t < kRows * D; t += kWarps * 32) {
        const int r = t / D, d = t % D;
        Xi[t] = i0 + r < N ? column(i0 + r, d) : 0.f;
    }
    float xi[kRowsPerWarp][DP], acc[kRowsPerWarp][DP];
    int kd[DP];
    bool logit[DP];
#pragma unroll
    for (int q = 0; q < DP; ++q) {
        const int d = lane + 32 * q;
        kd[q] = d < D ? d / P : 0;
        logit[q] = d < D && d % P < M;
#pragma unroll
        for (int r = 0; r < kRowsPerWarp; ++r) {
            const int i = i0 + warp * kRowsPerWarp + r;
            xi[r][q] = i < N && d < D ? column(i, d) : 0.f;
            acc[r][q] = 0.f;
        }
    }
    // this CTA's share of the sum over j; partial directions go to share blockIdx.y
    const int jb = blockIdx.y * j_chunk, je = min(N, jb + j_chunk);
    phi += (size_t)blockIdx.y * N * D;
    for (int j0 = jb; j0 < je; j0 += kTJ) {
        const int nj = min(kTJ, je - j0);
        for (int t = tid; t < kTJ * D; t += kWarps * 32) {
            const int jj = t / D, d = t % D;
            Xj[t] = jj < nj ? column(j0 + jj, d) : 0.f;
            Gj[t] = jj < nj ? grad[(size_t)j0 * D + t] : 0.f;
        }
        __syncthreads();
        // one (row, j) pair per thread: every action's kernels, and their sum K
        for (int e = tid; e < kRows * kTJ; e += kWarps * 32) {
            const int r = e / kTJ, jj = e % kTJ;
            const float w = jj < nj ? (wn ? wn[j0 + jj] : 1.f) : 0.f;
            float ksum = 0.f;
            for (int k = 0; k < H; ++k) {
                const float* a = Xi + r * D + k * P;
                const float* b = Xj + jj * D + k * P;
                float dz = 0.f, q = 0.f;
                for (int c = 0; c < M; ++c) {
                    const float bc = b[c], x = a[c] - bc;
                    dz = fmaf(x, x, dz);
                    q = fmaf(bc, x, q);
                }
                const float du = a[M] - b[M], dv = a[M + 1] - b[M + 1];
                const float ec = expf(-(du * du + dv * dv) * inv_hc);
                const float ez = expf(-dz * inv_hz);
                ksum += ec + ez;
                const int o = (r * kTJ + jj) * H + k;
                Ac[o] = ac * w * ec;
                Az[o] = az * w * ez;
                Q[o] = q;
            }
            Ks[e] = alpha * ksum * w;
        }
        __syncthreads();
        for (int jj = 0; jj < nj; ++jj) {
#pragma unroll
            for (int q = 0; q < DP; ++q) {
                const int d = lane + 32 * q;
                if (d >= D) continue;
                const float g = Gj[jj * D + d], x = Xj[jj * D + d];
#pragma unroll
                for (int r = 0; r < kRowsPerWarp; ++r) {
                    const int rj = (warp * kRowsPerWarp + r) * kTJ + jj, o = rj * H + kd[q];
                    // logits: A^z s_j ((s_i - s_j) - q); offset, distance: A^c (c_i - c_j)
                    const float rep = logit[q] ? Az[o] * (x * ((xi[r][q] - x) - Q[o]))
                                               : Ac[o] * (xi[r][q] - x);
                    acc[r][q] = fmaf(Ks[rj], g, acc[r][q] + rep);
                }
            }
        }
        __syncthreads();
    }
    const float scale = wn ? 1.f : 1.f / (float)N;
#pragma unroll
    for (int r = 0; r < kRowsPerWarp; ++r) {
        const int i = i0 + warp * kRowsPerWarp + r;
        if (i < N)
#pragma unroll
            for (int q = 0; q < DP; ++q) {
                const int d = lane + 32 * q;
                if (d < D) phi[(size_t)i * D + d] = acc[r][q] * scale;
            }
    }
}

template <int DP>
cudaError_t struct_launch(dim3 grid, const float* theta, const float* grad, const float* S, int N, int H,
                          int M, const float* hc, const float* hz, const float* wn, float* phi,
                          int j_chunk, cudaStream_t st) {
    const size_t smem = struct_smem(H * (M + 2), H);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(struct_phi_kernel<DP>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    struct_phi_kernel<DP><<<grid, kWarps * 32, smem, st>>>(theta, grad, S, N, H, M, hc, hz, wn, phi, j_chunk);
    return cudaGetLastError();
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
    if (H > kMaxHs) return cudaErrorInvalidValue;
    const int D = H * (M + 2), rows = (N + kRows - 1) / kRows;
    // split the sum over j so that about four CTAs per SM are in flight
    int want = (4 * sm_count() + rows - 1) / rows;
    want = want < 1 ? 1 : (want > max_shares ? max_shares : want);
    const int j_chunk = ((N + want - 1) / want + kTJ - 1) / kTJ * kTJ;
    *shares = (N + j_chunk - 1) / j_chunk;
    const dim3 grid(rows, *shares);
    switch ((D + 31) / 32) {
        case 1: return struct_launch<1>(grid, theta, grad, S, N, H, M, hc_dev, hz_dev, wn, phi, j_chunk, st);
        case 2: return struct_launch<2>(grid, theta, grad, S, N, H, M, hc_dev, hz_dev, wn, phi, j_chunk, st);
        case 3: return struct_launch<3>(grid, theta, grad, S, N, H, M, hc_dev, hz_dev, wn, phi, j_chunk, st);
        case 4: return struct_launch<4>(grid, theta, grad, S, N, H, M, hc_dev, hz_dev, wn, phi, j_chunk, st);
        case 5: case 6: return struct_launch<6>(grid, theta, grad, S, N, H, M, hc_dev, hz_dev, wn, phi, j_chunk, st);
        case 7: case 8: case 9: return struct_launch<9>(grid, theta, grad, S, N, H, M, hc_dev, hz_dev, wn, phi, j_chunk, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace stamp
