// Backward pass of the truncated SVD with U absent from the forward pass (Eq. 13-15 and
// the appendix that derives them):
//   dL/dH = U [ diag(dS) + 2 Sigma sym(F o (Vbar^T V)) ] V^T,   U = H V Sigma^-1,
//   F_ij = 1 / (sigma_i^2 - sigma_j^2)  (Eq. 14), zero on the diagonal.
// The Hadamard factor is Vbar^T V: the appendix expands Tr((V^T Vbar)^T Omega_V) with the
// indices of V^T Vbar transposed, which flips the sign of the off-diagonal term; this is
// the form that agrees with finite differences of the forward pass.
//
// Because U = H V Sigma^-1, the gradient is one right-multiplication of the history,
//   dH_b = H_b K_b,   K_b = V W V^T  (d x d),   W = Sigma^-1 [ diag(dS) + Sigma (X + X^T) ],
//   X = F o (Vbar^T V),
// so the backward pass streams H once more (the same kernel that forms U Sigma = H V)
// instead of materialising U.  This file holds the per-user kernel that forms K_b.
//
// Stabilisation (the paper gives none): F_ij = D / (D^2 + eps^2) with
// D = sigma_i^2 - sigma_j^2 and eps = eps_rel * max sigma^2; eps_rel = 0 is Eq. 14 itself,
// with F_ij = 0 where D = 0.  A direction with sigma_i = 0 has no U column and gets no
// gradient (row i of W is zero).
#include "solar_internal.cuh"

namespace solar {

namespace {

constexpr int kGradThreads = 256;
// CTAs per user: each forms W and a share of K's rows.  As many as stay within one per SM: every further one
// forms W again (64 users, d = r = 64, with dH over 100 rows: 37.2, 31.7 and 37.1 us on one, two and four; 128
// users 43.3, 47.4, 61.7; 16 users 37.2, 31.0, 29.0).
inline int grad_parts(int B) { return 4 * B <= kNumSMs ? 4 : 2 * B <= kNumSMs ? 2 : 1; }

// out(i, j) = sum_k a(i, k) b(k, j) for i < rows, j < cols, in tiles of 2 x 2 (four reads for four FMAs).
template <typename FA, typename FB, typename FS>
__device__ __forceinline__ void gemm22(int rows, int cols, int K, FA a, FB b, FS store, int tid) {
  const int ct = (cols + 1) / 2, tiles = ((rows + 1) / 2) * ct;
  for (int t = tid; t < tiles; t += kGradThreads) {
    const int i = 2 * (t / ct), j = 2 * (t % ct);
    float c00 = 0.f, c01 = 0.f, c10 = 0.f, c11 = 0.f;
#pragma unroll 8
    for (int k = 0; k < K; ++k) {
      const float a0 = a(i, k), a1 = a(i + 1, k), b0 = b(k, j), b1 = b(k, j + 1);
      c00 = fmaf(a0, b0, c00); c01 = fmaf(a0, b1, c01); c10 = fmaf(a1, b0, c10); c11 = fmaf(a1, b1, c11);
    }
    store(i, j, c00);
    if (j + 1 < cols) store(i, j + 1, c01);
    if (i + 1 < rows) {
      store(i + 1, j, c10);
      if (j + 1 < cols) store(i + 1, j + 1, c11);
    }
  }
}

// Bound by latency: one round of loads and four products with a barrier each.  16 users, d = 64, r = 32:
// 14.7 us on one CTA of 1024 threads per user, 8.2 on four of 256.
template <int D>
__global__ void __launch_bounds__(kGradThreads)
svd_grad_kernel(const float* __restrict__ S, const float* __restrict__ V, const float* __restrict__ dS,
                const float* __restrict__ dV, float eps_rel, int r, float* __restrict__ K) {
  extern __shared__ __align__(16) float sm[];
  const int lw = (r | 1) + 2;           // odd pitch (every matrix here is read along rows and along columns), room for a tile's edge
  float* Vs = sm;                       // [D][lw]
  float* dVs = Vs + D * lw;             // [D][lw]  Vbar
  float* Pt = dVs + D * lw;             // [r+1][lw]  Vbar^T V
  float* W = Pt + (r + 1) * lw;         // [r+1][lw]
  const int KR = D / (int)gridDim.y;    // rows of K of a CTA
  float* T1 = W + (r + 1) * lw;         // [KR][lw]  a share of V W
  float* ss = T1 + KR * lw;             // [r] sigma
  float* ds = ss + r;                   // [r] dL/dsigma
  const int b = blockIdx.x, tid = threadIdx.x;
  const int k0 = blockIdx.y * KR;       // this CTA's rows of K

  pdl_wait();          // the first kernel of its entry point: everything below reads the caller's buffers
#pragma unroll 4
  for (int e = tid; e < D * r; e += kGradThreads) {
    const int k = e / r, i = e - k * r;
    Vs[k * lw + i] = ld_dep(V + (size_t)b * D * r + e);
    dVs[k * lw + i] = ld_dep(dV + (size_t)b * D * r + e);
  }
  for (int e = tid; e < r; e += kGradThreads) { ss[e] = ld_dep(S + (size_t)b * r + e); ds[e] = ld_dep(dS + (size_t)b * r + e); }
  __syncthreads();

  // Pt[i][j] = sum_k Vbar[k][i] V[k][j]
  gemm22(r, r, D, [&](int i, int k) { return dVs[k * lw + i]; }, [&](int k, int j) { return Vs[k * lw + j]; },
         [&](int i, int j, float v) { Pt[i * lw + j] = v; }, tid);
  float smax = 0.f;
  for (int i = 0; i < r; ++i) smax = fmaxf(smax, ss[i]);
  const float eps = eps_rel * smax * smax;
  __syncthreads();

  // W = Sigma^-1 diag(dS) + (X + X^T) on the rows with sigma_i > 0
  for (int e = tid; e < r * r; e += kGradThreads) {
    const int i = e / r, j = e - i * r;
    const float si = ss[i], sj = ss[j];
    float w = 0.f;
    if (si > 0.f) {
      if (i == j) {
        w = ds[i] / si;
      } else {
        const float dd = (si - sj) * (si + sj);               // sigma_i^2 - sigma_j^2 without cancellation
        const float den = fmaf(dd, dd, eps * eps);
        const float f = den > 0.f ? dd / den : 0.f;
        w = f * (Pt[i * lw + j] - Pt[j * lw + i]);            // F_ij P_ij + F_ji P_ji, F skew-symmetric
      }
    }
    W[i * lw + j] = w;
  }
  __syncthreads();
  pdl_trigger();

  // T1 = V W, rows k0 ..
  gemm22(KR, r, r, [&](int k, int i) { return Vs[(k0 + k) * lw + i]; }, [&](int i, int j) { return W[i * lw + j]; },
         [&](int k, int j, float v) { T1[k * lw + j] = v; }, tid);
  __syncthreads();

  // K = T1 V^T, rows k0 ..
  float* Kb = K + (size_t)b * D * D;
  gemm22(KR, D, r, [&](int k, int j) { return T1[k * lw + j]; }, [&](int j, int l) { return Vs[l * lw + j]; },
         [&](int k, int l, float v) { Kb[(k0 + k) * D + l] = v; }, tid);
}

template <int D>
cudaError_t launch_d(int B, int r, const float* S, const float* V, const float* dS, const float* dV,
                     float eps_rel, float* K, cudaStream_t st) {
  const int parts = grad_parts(B);
  auto smem = [](int rank, int shares) {
    const int lw = (rank | 1) + 2;
    return (size_t)(2 * D * lw + 2 * (rank + 1) * lw + D / shares * lw + 2 * rank) * sizeof(float);
  };
  static bool limits_set[kMaxDevicesCached] = {};
  const cudaError_t e = set_kernel_limits(reinterpret_cast<const void*>(&svd_grad_kernel<D>), smem(D < 64 ? D : 64, 1), limits_set);
  if (e != cudaSuccess) return e;
  return launch_pdl(svd_grad_kernel<D>, dim3(B, parts), dim3(kGradThreads), smem(r, parts), st, S, V, dS, dV, eps_rel, r, K);
}

}  // namespace

cudaError_t launch_svd_grad(int B, int d, int r, const float* S, const float* V, const float* dS,
                            const float* dV, float eps_rel, float* K, cudaStream_t st) {
  switch (d) {
    case 32: return launch_d<32>(B, r, S, V, dS, dV, eps_rel, K, st);
    case 64: return launch_d<64>(B, r, S, V, dS, dV, eps_rel, K, st);
    case 128: return launch_d<128>(B, r, S, V, dS, dV, eps_rel, K, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace solar
