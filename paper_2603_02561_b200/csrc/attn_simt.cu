// SVD-Attention over the r factor tokens (Eq. 12), FFMA version (fp32 storage, and bf16 at d = 32).
// Two neighbouring lanes have two candidate rows: each the scores of half of the tokens (R = r rounded up
// to the template's token count) and, once the probabilities are exchanged, half of the output columns.
// The operands T and Value_r are read from shared memory as 16-byte broadcasts, eight FMAs each: such a
// read takes four cycles a warp, so with a row per lane and four FMAs the reads were the bound.  The
// candidate tile comes in and the output tile goes out coalesced through one shared buffer of odd 16-byte
// pitch.  16 x 1000 candidates, d = 64, r = 24, fp32: 33 us with a warp per row over 64 padded tokens, 15
// with a row per lane; two rows and longer Gram stages: 71.8 -> 69.8 us per pass over 5000 x 64 histories.
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
    const uint4 raw = ld_dep(reinterpret_cast<const uint4*>(Cb) + v);
    float x[VE];
    Vec16<T>::load(reinterpret_cast<const T*>(&raw), x);
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
  // A large grid releases the next kernel only behind its work: the next call's first kernel would be packed
  // onto the SMs that are free (two of its CTAs on one: 16 x 5000 x 64 in fp32 70 -> 81 us per pass).  A small
  // one leaves most SMs free, and an early release hides the launch (one user: 22.5 -> 22.0 us).
  const bool few = gridDim.x * gridDim.y <= kNumSMs / 2;
  if (few) pdl_trigger();

  if ((tid & ~31) < rows) {              // (rows past the end compute on what lies there and are not stored)
    constexpr int RH = R / 2, DH = D / 2;
    const int half = tid & 1, i0 = half * RH;
    float* const row = Cs + (tid & ~1) * LC;           // rows tid & ~1 and the next
    float p[2][R];                                      // p[.][i]: this lane's tokens i0 + i first, the partner's behind
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int i = 0; i < RH; ++i) p[q][i] = 0.f;
#pragma unroll 1
    for (int k = 0; k < D; k += 4) {
      const float4 a4 = *reinterpret_cast<const float4*>(row + k), b4 = *reinterpret_cast<const float4*>(row + LC + k);
      const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int i = 0; i < RH; i += 4) {
          const float4 t4 = *reinterpret_cast<const float4*>(Ts + (k + u) * R + i0 + i);
          const float t[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            p[0][i + c] = fmaf(a[u], t[c], p[0][i + c]);
            p[1][i + c] = fmaf(b[u], t[c], p[1][i + c]);
          }
        }
    }
    if (!(flags & SOLAR_FLAG_NO_SOFTMAX)) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float mx = -INFINITY;
#pragma unroll
        for (int i = 0; i < RH; ++i) mx = fmaxf(mx, i0 + i < r ? p[q][i] : -INFINITY);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        float sum = 0.f;
#pragma unroll
        for (int i = 0; i < RH; ++i) {
          p[q][i] = i0 + i < r ? expf(p[q][i] - mx) : 0.f;
          sum += p[q][i];
        }
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        const float inv = 1.f / sum;
#pragma unroll
        for (int i = 0; i < RH; ++i) p[q][i] *= inv;
      }
    } else {                              // an infinite candidate times the zeros of a padded token is a NaN
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int i = 0; i < RH; ++i) p[q][i] = i0 + i < r ? p[q][i] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int i = 0; i < RH; ++i) p[q][RH + i] = __shfl_xor_sync(0xffffffffu, p[q][i], 1);
    __syncwarp();                         // the rows have been read: they take the output
    const float* const mine = Vs + i0 * D + half * DH, * const theirs = Vs + (RH - i0) * D + half * DH;
#pragma unroll 1
    for (int j4 = 0; j4 < DH; j4 += 4) {
      const int j = (j4 + 4 * half) & (DH - 1);        // the partner's 16 bytes lie in other banks
      float o[2][4];
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int u = 0; u < 4; ++u) o[q][u] = 0.f;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const float4 v = *reinterpret_cast<const float4*>((i < RH ? mine + i * D : theirs + (i - RH) * D) + j);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          o[q][0] = fmaf(p[q][i], v.x, o[q][0]); o[q][1] = fmaf(p[q][i], v.y, o[q][1]);
          o[q][2] = fmaf(p[q][i], v.z, o[q][2]); o[q][3] = fmaf(p[q][i], v.w, o[q][3]);
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q)
        *reinterpret_cast<float4*>(row + q * LC + half * DH + j) = make_float4(o[q][0], o[q][1], o[q][2], o[q][3]);
    }
  }
  __syncthreads();
  if (!few) pdl_trigger();
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

// Token counts: multiples of 8 to 48, then 64 -- the work is proportional to them (16 candidates of one user,
// d = 128, r = 33: 57.0 us as 48 tokens, 51.5 as 40).
template <typename T, int D>
cudaError_t launch_td(int B, int M, int r, const void* C, unsigned flags, void* O, const char* ws, const AttnWs& lay,
                      bool early_c, cudaStream_t st) {
  if (r <= 8) return launch_tdr<T, D, 8>(B, M, r, C, flags, O, ws, lay, early_c, st);
  if (r <= 16) return launch_tdr<T, D, 16>(B, M, r, C, flags, O, ws, lay, early_c, st);
  if (r <= 24) return launch_tdr<T, D, 24>(B, M, r, C, flags, O, ws, lay, early_c, st);
  if (r <= 32) return launch_tdr<T, D, 32>(B, M, r, C, flags, O, ws, lay, early_c, st);
  if constexpr (D > 32) {
    if (r <= 40) return launch_tdr<T, D, 40>(B, M, r, C, flags, O, ws, lay, early_c, st);
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
