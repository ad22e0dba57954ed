// SVD-Attention over the r factor tokens (Eq. 12), FFMA version (fp32 storage, and bf16 at d = 32).
// One candidate row per thread: its scores stay in registers (R = r rounded up to the template's
// token count), so the softmax needs no shuffles, and the operands T and Value_r are read from shared
// memory as 16-byte broadcasts, four FMAs each.  The candidate tile comes in and the output tile goes
// out coalesced through one shared buffer of odd 16-byte pitch.  Bound by shared-memory reads and
// FMAs alike (2 d r of each row's lanes), then by HBM.  16 x 1000 candidates, d = 64, r = 24, fp32:
// 33 us with a warp per row over 64 padded tokens, 15 now.
#include <math.h>

#include "solar_internal.cuh"

namespace solar {

namespace {

constexpr int kRows = 128;     // candidate rows per CTA = threads

template <int D, int R> struct SimtAttn {
  static constexpr int LC = D + 4;                                        // row pitch of the candidate tile
  static constexpr size_t SMEM = (size_t)(2 * D * R + kRows * LC) * sizeof(float);
};

template <typename T, int D, int R>
__global__ void __launch_bounds__(kRows)
attn_simt_kernel(const T* __restrict__ C, T* __restrict__ O, const char* __restrict__ ws,
                 AttnWs lay, int M, int r, unsigned flags, int early_c) {
  using L = SimtAttn<D, R>;
  constexpr int LC = L::LC, VE = Vec16<T>::kElems, VPR = D / VE;
  extern __shared__ __align__(16) float sm[];
  float* Ts = sm;                       // [D][R]
  float* Vs = Ts + D * R;               // [R][D]
  float* Cs = Vs + R * D;               // [kRows][LC]

  const int b = blockIdx.y, m0 = blockIdx.x * kRows, tid = threadIdx.x;
  const int rows = min(kRows, M - m0);
  const char* wsb = ws + (size_t)b * lay.per_user;
  const float* Tf = reinterpret_cast<const float*>(wsb + lay.tf_off);
  const float* Vr = reinterpret_cast<const float*>(wsb + lay.vr_off);
  // The candidates are the caller's: ahead of the wait only when an earlier kernel of the same
  // library call has already waited for whatever ran before the call (early_c).
  if (!early_c) pdl_wait();
  const T* Cb = C + ((size_t)b * M + m0) * D;
#pragma unroll 4
  for (int v = tid; v < rows * VPR; v += kRows) {
    float x[VE];
    Vec16<T>::load(Cb + (size_t)v * VE, x);
    float* dst = Cs + (v / VPR) * LC + (v % VPR) * VE;
#pragma unroll
    for (int e = 0; e < VE; e += 4) *reinterpret_cast<float4*>(dst + e) = make_float4(x[e], x[e + 1], x[e + 2], x[e + 3]);
  }
  if (early_c) pdl_wait();
#pragma unroll 4
  for (int e = tid; e < D * R; e += kRows) {
    const int k = e / R, i = e % R;
    Ts[e] = i < r ? ld_dep(Tf + k * r + i) : 0.f;
  }
#pragma unroll 4
  for (int e = tid; e < R * D / 4; e += kRows)
    reinterpret_cast<float4*>(Vs)[e] = e / (D / 4) < r ? ld_dep(reinterpret_cast<const float4*>(Vr) + e) : make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  pdl_trigger();

  if (tid < rows) {
    float* row = Cs + tid * LC;
    float p[R];
#pragma unroll
    for (int i = 0; i < R; ++i) p[i] = 0.f;
#pragma unroll 1
    for (int k = 0; k < D; k += 4) {
      const float4 c4 = *reinterpret_cast<const float4*>(row + k);
      const float c[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int i = 0; i < R; i += 4) {
          const float4 t = *reinterpret_cast<const float4*>(Ts + (k + u) * R + i);
          p[i] = fmaf(c[u], t.x, p[i]);         p[i + 1] = fmaf(c[u], t.y, p[i + 1]);
          p[i + 2] = fmaf(c[u], t.z, p[i + 2]); p[i + 3] = fmaf(c[u], t.w, p[i + 3]);
        }
    }
    if (!(flags & SOLAR_FLAG_NO_SOFTMAX)) {
      float mx = -INFINITY;
#pragma unroll
      for (int i = 0; i < R; ++i) mx = fmaxf(mx, i < r ? p[i] : -INFINITY);
      float sum = 0.f;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        p[i] = i < r ? expf(p[i] - mx) : 0.f;
        sum += p[i];
      }
      const float inv = 1.f / sum;
#pragma unroll
      for (int i = 0; i < R; ++i) p[i] *= inv;
    }                                     // without it: padded tokens have zero scores and zero Value_r rows
#pragma unroll 1
    for (int j = 0; j < D; j += 8) {
      float o[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) o[u] = 0.f;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(Vs + i * D + j), w = *reinterpret_cast<const float4*>(Vs + i * D + j + 4);
        o[0] = fmaf(p[i], v.x, o[0]); o[1] = fmaf(p[i], v.y, o[1]); o[2] = fmaf(p[i], v.z, o[2]); o[3] = fmaf(p[i], v.w, o[3]);
        o[4] = fmaf(p[i], w.x, o[4]); o[5] = fmaf(p[i], w.y, o[5]); o[6] = fmaf(p[i], w.z, o[6]); o[7] = fmaf(p[i], w.w, o[7]);
      }
      *reinterpret_cast<float4*>(row + j) = make_float4(o[0], o[1], o[2], o[3]);
      *reinterpret_cast<float4*>(row + j + 4) = make_float4(o[4], o[5], o[6], o[7]);
    }
  }
  __syncthreads();
  T* Ob = O + ((size_t)b * M + m0) * D;
#pragma unroll 4
  for (int v = tid; v < rows * VPR; v += kRows) {
    const float* src = Cs + (v / VPR) * LC + (v % VPR) * VE;
    T out[VE];
#pragma unroll
    for (int e = 0; e < VE; ++e) out[e] = from_f32<T>(src[e]);
    *reinterpret_cast<uint4*>(Ob + (size_t)v * VE) = *reinterpret_cast<const uint4*>(out);
  }
}

template <typename T, int D, int R>
cudaError_t launch_tdr(int B, int M, int r, const void* C, unsigned flags, void* O, const char* ws, const AttnWs& lay,
                       bool early_c, cudaStream_t st) {
  constexpr size_t smem = SimtAttn<D, R>::SMEM;
  static bool limits_set[kMaxDevicesCached] = {};
  const cudaError_t e = set_kernel_limits(reinterpret_cast<const void*>(&attn_simt_kernel<T, D, R>), smem, limits_set);
  if (e != cudaSuccess) return e;
  return launch_pdl(attn_simt_kernel<T, D, R>, dim3((M + kRows - 1) / kRows, B), dim3(kRows), smem, st,
                    static_cast<const T*>(C), static_cast<T*>(O), ws, lay, M, r, flags, (int)early_c);
}

// Token counts: multiples of 8 to 32, of 16 above -- the work is proportional to them.
template <typename T, int D>
cudaError_t launch_td(int B, int M, int r, const void* C, unsigned flags, void* O, const char* ws, const AttnWs& lay,
                      bool early_c, cudaStream_t st) {
  if (r <= 8) return launch_tdr<T, D, 8>(B, M, r, C, flags, O, ws, lay, early_c, st);
  if (r <= 16) return launch_tdr<T, D, 16>(B, M, r, C, flags, O, ws, lay, early_c, st);
  if (r <= 24) return launch_tdr<T, D, 24>(B, M, r, C, flags, O, ws, lay, early_c, st);
  if (r <= 32) return launch_tdr<T, D, 32>(B, M, r, C, flags, O, ws, lay, early_c, st);
  if constexpr (D > 32) {
    if (r <= 48) return launch_tdr<T, D, 48>(B, M, r, C, flags, O, ws, lay, early_c, st);
    return launch_tdr<T, D, 64>(B, M, r, C, flags, O, ws, lay, early_c, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_attn_simt(int B, int M, int d, int r, solar_dtype_t dt, const void* C,
                             unsigned flags, void* O, const char* ws, const AttnWs& lay, bool early_c,
                             cudaStream_t st) {
  if (dt == SOLAR_BF16)                  // d = 64 and 128 take the tensor-core kernel
    return d == 32 ? launch_td<__nv_bfloat16, 32>(B, M, r, C, flags, O, ws, lay, early_c, st) : cudaErrorInvalidValue;
  switch (d) {
    case 32: return launch_td<float, 32>(B, M, r, C, flags, O, ws, lay, early_c, st);
    case 64: return launch_td<float, 64>(B, M, r, C, flags, O, ws, lay, early_c, st);
    case 128: return launch_td<float, 128>(B, M, r, C, flags, O, ws, lay, early_c, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace solar
