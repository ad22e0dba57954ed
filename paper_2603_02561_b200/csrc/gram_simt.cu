// Streaming Gram pass, FFMA version: P[b,s] = sum_{n in slice s} h_n h_n^T.
// Used for fp32 storage (bf16 products would break the 1e-4 tolerance of that mode),
// for d = 32 and for N < 128 (shapes the tensor-core kernel does not take);
// G_b = H_b^T H_b is the matrix whose eigenvectors are V of Eq. 9.
//
// Bound by the FMA pipes: d^2/2 FMAs a row, the matrix being symmetric.  A thread owns one 8 x 8 tile
// on or above the diagonal (36 of 64 at d = 64) for every KG-th row, so 64 FMAs follow four 16-byte
// shared-memory reads, most of them broadcasts; KG groups of such threads fill the CTA and their
// tiles are added up in group order at the end.  Rows arrive by cp.async in a ring of three stages,
// in the storage type.  16 x 5000 x 64 fp32: 54 us with 4 x 4 tiles of the full matrix and one
// synchronous stage, 19.6 with stages of 56 rows, 18.8 now (112 rows, the last stage only as long as it has
// rows; 8 of them FMA time).  The next kernel is not released early: its few
// CTAs would be packed onto the SMs that are free first and slow each other down.
#include "solar_internal.cuh"

namespace solar {

namespace {

template <int D> struct SimtGram {
  static constexpr int NB = D / 8, TILES = NB * (NB + 1) / 2;            // 8 x 8 tiles on and above the diagonal
  static constexpr int NT = D == 128 ? 288 : 256;                         // threads: KG groups of TILES, a few idle
  static constexpr int KG = NT / TILES;                                   // 25, 7, 2
  static constexpr int IT = D == 32 ? 4 : 16;                             // rows of a group per stage
  static constexpr int TR = KG * IT;                                      // rows per stage: 100, 112, 32
  static constexpr int STAGES = 3;
  template <typename T> static constexpr size_t smem() {
    const size_t ring = (size_t)STAGES * TR * D * sizeof(T), red = (size_t)KG * TILES * 64 * sizeof(float);
    return ring > red ? ring : red;
  }
};

__device__ __forceinline__ void load8(const float* p, float (&x)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&x)[8]) { Vec16<__nv_bfloat16>::load(p, x); }

template <typename T, int D>
__global__ void __launch_bounds__(SimtGram<D>::NT)
gram_simt_kernel(const T* __restrict__ H, float* __restrict__ gpart, int* __restrict__ status,
                 int N, int chunk_rows, int splits) {
  using C = SimtGram<D>;
  constexpr int NT = C::NT, TR = C::TR, KG = C::KG;
  constexpr int VE = 16 / (int)sizeof(T), VPR = D / VE;                   // 16-byte pieces of a row
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* ring = reinterpret_cast<T*>(smem_raw);

  const int b = blockIdx.y, s = blockIdx.x, tid = threadIdx.x;
  const int row0 = s * chunk_rows, rows = min(N, row0 + chunk_rows) - row0;
  const T* Hb = H + ((size_t)b * N + row0) * D;
  const int nst = (rows + TR - 1) / TR;

  // the thread's tile (ti <= tj) and group; the threads left over repeat the last tile and drop it
  const int grp = min(tid / C::TILES, KG - 1), t = tid - (tid / C::TILES) * C::TILES;
  const bool mine = tid < KG * C::TILES;
  int ti = 0, first = 0;
  while (t >= first + C::NB - ti) { first += C::NB - ti; ++ti; }
  const int tj = ti + t - first;

  pdl_wait();            // H is the caller's: whatever wrote it earlier on the stream has completed
  auto fetch = [&](int st) {
    T* dst = ring + (size_t)(st % C::STAGES) * TR * D;
    const int want = min(TR, (rows - st * TR + KG - 1) / KG * KG);        // whole rounds of the groups
    for (int v = tid; v < want * VPR; v += NT) {
      const int rr = st * TR + v / VPR;
      const int bytes = rr < rows ? 16 : 0;                               // rows past the end arrive as zeros
      const T* src = Hb + (size_t)min(rr, rows - 1) * D + (v % VPR) * VE;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                   ::"r"((uint32_t)__cvta_generic_to_shared(dst + v * VE)), "l"(src), "r"(bytes) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(0);
  if (nst > 1) fetch(1); else asm volatile("cp.async.commit_group;" ::: "memory");

  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
  for (int st = 0; st < nst; ++st) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();                       // stage st is there; everybody is done with stage st - 1
    if (st + 2 < nst) fetch(st + 2); else asm volatile("cp.async.commit_group;" ::: "memory");
    const T* rowp = ring + (size_t)(st % C::STAGES) * TR * D + (size_t)grp * D;
    const int rounds = min(C::IT, (rows - st * TR + KG - 1) / KG);
#pragma unroll 2
    for (int it = 0; it < rounds; ++it) {
      float a[8], c[8];
      load8(rowp + (size_t)it * KG * D + 8 * ti, a);
      load8(rowp + (size_t)it * KG * D + 8 * tj, c);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], c[j], acc[i][j]);
    }
  }
  __syncthreads();
  // the groups' tiles, entry-major so that neither the stores nor the sums conflict
  float* red = reinterpret_cast<float*>(smem_raw);
  if (mine) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) red[(size_t)(grp * 64 + 8 * i + j) * C::TILES + t] = acc[i][j];
  }
  __syncthreads();
  pdl_wait();            // (a no-op by now) nothing is written before the previous kernel has read this workspace
  float* out = gpart + ((size_t)b * splits + s) * D * D;
  for (int e = tid; e < D * D; e += NT) {
    const int row = e / D, col = e % D, i = min(row, col), j = max(row, col);   // the entry on or above the diagonal
    const int bi = i / 8, bj = j / 8, tt = bi * C::NB - bi * (bi - 1) / 2 + bj - bi;
    const float* src = red + (size_t)(8 * (i % 8) + j % 8) * C::TILES + tt;
    float sum = 0.f;
#pragma unroll
    for (int q = 0; q < KG; ++q) sum += src[(size_t)q * 64 * C::TILES];
    out[e] = sum;
  }
  if (tid == 0) status[b * splits + s] = kGramStatusOk;   // this kernel has no waits to lose
}

template <typename T, int D>
cudaError_t launch_td(int B, int N, const void* H, float* gpart, int* status, const GramPlan& plan, cudaStream_t st) {
  using C = SimtGram<D>;
  static bool limits_set[kMaxDevicesCached] = {};
  const cudaError_t e = set_kernel_limits(reinterpret_cast<const void*>(&gram_simt_kernel<T, D>), C::template smem<T>(), limits_set);
  if (e != cudaSuccess) return e;
  return launch_pdl(gram_simt_kernel<T, D>, dim3(plan.splits, B), dim3(C::NT), C::template smem<T>(), st,
                    static_cast<const T*>(H), gpart, status, N, plan.chunk_tiles * kGramTileRows, plan.splits);
}

template <typename T>
cudaError_t launch_t(int B, int N, int d, const void* H, float* gpart, int* status, const GramPlan& plan, cudaStream_t st) {
  switch (d) {
    case 32: return launch_td<T, 32>(B, N, H, gpart, status, plan, st);
    case 64: return launch_td<T, 64>(B, N, H, gpart, status, plan, st);
    case 128: return launch_td<T, 128>(B, N, H, gpart, status, plan, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_gram_simt(int B, int N, int d, solar_dtype_t dt, const void* H, float* gpart,
                             int* status, const GramPlan& plan, cudaStream_t st) {
  return dt == SOLAR_BF16 ? launch_t<__nv_bfloat16>(B, N, d, H, gpart, status, plan, st)
                          : launch_t<float>(B, N, d, H, gpart, status, plan, st);
}

}  // namespace solar
