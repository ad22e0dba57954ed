// Batched symmetric eigensolver, tridiagonal route: the top-r eigenpairs of every Gram matrix
// G_b = H_b^T H_b (Eq. 9 without U: s_i = sqrt(lambda_i), V = eigenvectors) by the classical
// dense-symmetric chain, one CTA per user (128 threads; 256 at d = 128):
//
//   1. G = sum of the slices' partial Grams (fixed order), scaled by a power of two.
//   2. Householder tridiagonalisation T = Q^T G Q (only as far as the kept vectors reach) with the matrix in REGISTERS, in tiles of d/32
//      rows x 16 columns per thread (rows 32 apart, so that finished ones leave the later stages for all
//      threads: at d = 64 43.9 thousand cycles for the 62 steps with adjacent rows, 37.6 now; at d = 128
//      165 and 138, in fp64 319 and 297, 260 with the reciprocals and A x as below); the vectors of a step live in registers too, at the thread's
//      columns and at its rows, so the norm, the inner product and a row of A x are each complete
//      after the two (three) shuffles over the threads of a row.  The product is taken with the
//      column x itself and corrected to the reflector v = x - alpha e_1 afterwards, so that the
//      square root runs beside it; the next column comes from row k+1 (by symmetry) of the matrix
//      before the update.  What crosses warps is A x and that row, at ONE barrier per step.
//   3. The r largest eigenvalues of T by multisection on Sturm counts: the points of an eigenvalue
//      are lanes of one warp (a ballot instead of a barrier), the counts come from the three-term
//      recurrence of the leading principal minors -- one FMA per row on the dependency chain.
//   4. One eigenvector per eigenvalue from the twisted factorisation of T - lambda I: inverse
//      iteration from the best unit vector, O(d) per vector, no pivoting.  Leading and trailing
//      minors run on two warps; gamma_k = det / (p_k t_{k+1}), so the twist is where the product
//      of the two minors is largest and their logarithms are all that has to be compared.
//   5. V = Q Z.  fp32, d <= 64: Q is accumulated during step 2 (each thread's tile of Q beside its
//      tile of A, in the shadow of the step's shuffles) and this is one small product; otherwise
//      the reflectors are applied one by one (no registers left for Q).
//   6. Gram-Schmidt passes in matrix form, V <- V (I - strict_upper(V^T V - I)) D^-1, repeated
//      while V^T V - I is above the rounding level (vectors of close eigenvalues come out of
//      step 4 with a mutual error of order eps |T| / gap); a column is only ever corrected by
//      the columns of larger eigenvalues.
//   7. Rayleigh quotients theta_i = v_i^T G v_i and residuals G v_i - theta_i v_i against the
//      ORIGINAL G: the result is accepted only if every residual is small against its gap (or
//      at the rounding floor), V^T V = I to rounding, trace(T) and the trace of the rows left out add up to
//      trace(G), and those rows cannot hold an eigenvalue above the last kept one.
//
// The chain runs in fp32 first.  A reduction to tridiagonal form is backward stable in the norm of
// G only: it fixes a kept vector to an angle of a few eps |T| / gap, whatever the size of its
// eigenvalue.  Where a gap among the kept eigenvalues is too small for that (sigma_i = i^-1 over 128
// directions), or the certificate fails, the CTA runs the same chain with steps 2-4 in fp64, where
// the angle is eps_64 |T| / gap; the fp32 eigenvalues are its starting brackets.  Only what that
// cannot certify either (vectors of equal eigenvalues) goes to the parallel Jacobi solve on the
// whole matrix, which is valid for any spectrum.  Where SMs are idle (r > 32, few users) the user has two
// CTAs, a cluster: one runs the fp32 chain, the other starts the fp64 chain at once; when the fp32
// eigenvalues are there, the first either sends them across and leaves the user to the second, or sends
// the second home.  Forward pass of 8 users, d = 128, r = 64 of a power
// law (every user takes the fp64 chain): 3075 us with Jacobi in its place, 374 with the fp64 chain behind
// the fp32 one, 239 beside it; 64 users, d = r = 64, one or none of them: 440, 148 and 109 us.
//
// What bounds it: the dependency chain (d steps of a matrix-vector product, an inner product and a
// barrier, then the recurrences over the rows of T), not work or bandwidth: 16 users keep 16 of
// 148 SMs busy.  A warp that is alone on its scheduler pays the full latency of every dependent
// instruction and shared-memory load, and tens of cycles for every branch, taken or not; the code
// below is therefore straight-line over static ranges (the Householder loop is cut into stages
// with fixed live columns; conditions are predicates of single instructions), fetches ahead, and
// keeps divisions off the dependency chains.
#include "eig_jacobi.cuh"
#include "eig_rest.cuh"
#include "project_mma.cuh"

namespace solar {

namespace {

constexpr unsigned kFull = 0xffffffffu;

template <int D> struct TriCfg {
  static constexpr int GX = (D == 128) ? 8 : 4;       // threads across a row; 32 groups of them
  // rows of a thread: group, group + 32, ..: they are finished for all threads at once, and the later stages
  // leave them out
  static constexpr int RT = D / 32;
  static constexpr int NT = 32 * GX;                  // threads of the CTA
  static constexpr int NW = NT / 32;
  static constexpr int CW = 4 * GX;                   // columns of a chunk: thread g of a group has 4 g .. 4 g + 3
  static constexpr int NCH = D / CW;                  // chunks of a row
  static constexpr int WG = 32 / NW;                  // groups of a warp
  __device__ static constexpr int first_row(int m) { return CW * m / 32; }                 // a thread's first unfinished row in chunk m's stage
  __device__ static constexpr int last_next(int m) { return CW * (m + 1) / 32 < RT && RT > 2 ? CW * (m + 1) / 32 : RT - 1; }   // row k+1 is among the rows to this one (of two, both are tried: not slower)
  __device__ static constexpr int rows_end(int warp) { return WG * (warp + 1) + 32 * (RT - 1); }   // behind a warp's last row
  // Resident CTAs that the register count has to allow.  d = 64: three (168 registers) for r <= 32 -- with 255 or
  // 128 the schedule is worse (16 x 10240 x 64 47.8 us per pass; 51.3, 50.2); above, shared memory allows two
  // anyway (64 users, d = r = 64: 1.4 % faster than with three).
  static constexpr int ctas(int rp) { return D == 128 ? 1 : rp > 32 ? 2 : 3; }
  static constexpr int LD = D + 4;                    // pitch of Q^T and of the row-major G
  // of a thread's tile: the entry at(m, c) on the diagonal in row row0 + 32 rr, where its columns have it
  template <typename F> __device__ static __forceinline__ auto diagonal(F at, int rr, int row0) {
    const bool up = CW < 32 && (row0 & 16);
    auto four = [&](int c) { return up ? at((32 * rr + 16) / CW, c) : at(32 * rr / CW, c); };
    const auto a = (row0 & 1) ? four(1) : four(0), b = (row0 & 1) ? four(3) : four(2);
    return (row0 & 2) ? b : a;
  }
};

// Shared-memory layout (floats) for subspace width RP = 32 * ceil(r / 32).
template <int D, int RP> struct TriSmem {
  using C = TriCfg<D>;
  static constexpr int R0 = 0;                                   // Q^T [D][LD] or the reflectors [D][D]; later G [D][D]
  static constexpr int A1 = R0 + (D == 128 ? D * D : D * C::LD); // [D][RP] upward multipliers; V
  static constexpr int A2 = A1 + D * RP;                         // [D][RP] downward multipliers; V'
  static constexpr int A3 = A2 + D * RP;                         // [D][RP] log2 of the leading minors; Z
  static constexpr int A4 = A3 + D * RP;                         // [D][RP] log2 of the trailing minors; V^T V - I [RP][RP]
  static constexpr int DG = A4 + D * RP;                         // diagonal of T (this and the next five with room for fp64)
  static constexpr int EO = DG + 2 * D;                          // off-diagonal: e[k] couples k, k+1
  static constexpr int E2 = EO + 2 * D;                          // e2s[i] = e[i-1]^2 (floored), e2s[0] = 0
  static constexpr int YV = E2 + 2 * D;                          // [2][D] A x
  static constexpr int XP = YV + 4 * D;                          // [2][D] row k+1 of the matrix before step k's update
  static constexpr int LAM = XP + 4 * D;                         // [RP] eigenvalues of T
  static constexpr int BE = LAM + 2 * RP;                        // [D] beta of reflector k
  static constexpr int TH = BE + D;                              // [RP] Rayleigh quotients
  static constexpr int L32 = TH + RP;                            // [RP] eigenvalues of the fp32 chain
  static constexpr int PART = L32 + RP;                          // [3][NW][RP] per-warp partial results
  static constexpr int TRI_FLOATS = PART + 3 * C::NW * RP;
  // the projection epilogue: V Sigma, Key_r^T, two weights (FFMA form) or the tensor-core form's staging
  static constexpr int EPI_FFMA = 2 * D * RP + 2 * D * D;
  static constexpr int EPI_MMA = (D >= 64) ? pmma::Lay<(D >= 64 ? D : 64)>::bytes(RP) / 4 : 0;
  static constexpr int EPI_FLOATS = EPI_FFMA > EPI_MMA ? EPI_FFMA : EPI_MMA;
  static constexpr int M1 = TRI_FLOATS > full_jacobi_floats<D>() ? TRI_FLOATS : full_jacobi_floats<D>();
  static constexpr int FLOATS = M1 > EPI_FLOATS ? M1 : EPI_FLOATS;
  static constexpr size_t BYTES = (size_t)FLOATS * sizeof(float);
  static_assert(A1 % 4 == 0 && DG % 4 == 0 && YV % 4 == 0 && LAM % 4 == 0 && BE % 4 == 0 && TH % 4 == 0 && PART % 4 == 0,
                "16-byte alignment of the regions");
  static_assert(RP <= D && BYTES <= 226 * 1024, "V^T V - I fits; one CTA fits an SM");
};

// ---- arithmetic in fp32 and fp64 -------------------------------------------------------------
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o));
  return v;
}
// sum over the GX threads of a row (every thread gets the same bits)
template <int GX, typename T> __device__ __forceinline__ T row_sum(T v) {
#pragma unroll
  for (int o = 1; o < GX; o <<= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ float fma_t(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float abs_t(float x) { return fabsf(x); }
__device__ __forceinline__ double abs_t(double x) { return fabs(x); }
__device__ __forceinline__ float rcp_fast(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// 1 / sqrt(x) and 1 / x to the accuracy of the type for normal x (the hardware's approximation plus one
// Newton step in fp32, two in fp64; without the library functions' branches for special values):
// the reflector I - beta v v^T is orthogonal only as far as beta v^T v = 2 holds.
__device__ __forceinline__ float rsqrt_t(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y * fmaf(-0.5f * x * y, y, 1.5f);
}
__device__ __forceinline__ double rsqrt_t(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
#pragma unroll
  for (int i = 0; i < 2; ++i) y = fma(0.5 * y, fma(-x * y, y, 1.0), y);
  return y;
}
__device__ __forceinline__ float rcp_t(float x) {
  const float y = rcp_fast(x);
  return y * fmaf(-x, y, 2.f);
}
__device__ __forceinline__ double rcp_t(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
#pragma unroll
  for (int i = 0; i < 2; ++i) y = fma(y, fma(-x, y, 1.0), y);
  return y;
}
// the word that holds the sign and the exponent
__device__ __forceinline__ unsigned top_word(float x) { return __float_as_uint(x); }
__device__ __forceinline__ unsigned top_word(double x) { return (unsigned)__double2hiint(x); }
// a power of two that brings max(|p|, |q|) into [1, 2)
__device__ __forceinline__ float pow2_scale(float p, float q) {
  return __uint_as_float(0x7f000000u - (__float_as_uint(fmaxf(fabsf(p), fabsf(q))) & 0x7f800000u));
}
__device__ __forceinline__ double pow2_scale(double p, double q) {
  const int m = max(__double2hiint(p) & 0x7ff00000, __double2hiint(q) & 0x7ff00000);
  return __hiloint2double(0x7fe00000 - m, 0);
}
__device__ __forceinline__ int log2_int(float x) { return (int)(__float_as_uint(x) >> 23) - 127; }       // of x >= 0, rounded down; denormals -127
__device__ __forceinline__ int exponent(float pow2) { return (int)(__float_as_uint(pow2) >> 23) - 127; }
__device__ __forceinline__ int exponent(double pow2) { return (__double2hiint(pow2) >> 20) - 1023; }
__device__ __forceinline__ void ld4(const float* p, float (&o)[4]) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
}
__device__ __forceinline__ void ld4(const double* p, double (&o)[4]) {
  const double2 t = *reinterpret_cast<const double2*>(p), u = *reinterpret_cast<const double2*>(p + 2);
  o[0] = t.x; o[1] = t.y; o[2] = u.x; o[3] = u.y;
}
// N consecutive floats
template <int N> __device__ __forceinline__ void ldn(const float* p, float (&o)[N]) {
  if constexpr (N == 2) {
    const float2 t = *reinterpret_cast<const float2*>(p);
    o[0] = t.x; o[1] = t.y;
  } else {
#pragma unroll
    for (int q = 0; q < N; q += 4) {
      const float4 t = *reinterpret_cast<const float4*>(p + q);
      o[q] = t.x; o[q + 1] = t.y; o[q + 2] = t.z; o[q + 3] = t.w;
    }
  }
}
__device__ __forceinline__ void st4(float* p, const float (&v)[4]) { *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]); }
__device__ __forceinline__ void st4(double* p, const double (&v)[4]) {
  *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  *reinterpret_cast<double2*>(p + 2) = make_double2(v[2], v[3]);
}
// Stores to shared memory under a predicate, without a branch.
__device__ __forceinline__ void st4_if(float* p, const float (&v)[4], bool pred) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %5, 0;\n\t@p st.shared.v4.f32 [%0], {%1, %2, %3, %4};\n\t}"
               ::"r"((uint32_t)__cvta_generic_to_shared(p)), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "r"((int)pred)
               : "memory");
}
__device__ __forceinline__ void st4_if(double* p, const double (&v)[4], bool pred) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %5, 0;\n\t@p st.shared.v2.f64 [%0], {%1, %2};\n\t"
               "@p st.shared.v2.f64 [%0+16], {%3, %4};\n\t}"
               ::"r"((uint32_t)__cvta_generic_to_shared(p)), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3]), "r"((int)pred)
               : "memory");
}
__device__ __forceinline__ void st_if(float* p, float v, bool pred) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p st.shared.f32 [%0], %1;\n\t}"
               ::"r"((uint32_t)__cvta_generic_to_shared(p)), "f"(v), "r"((int)pred) : "memory");
}
__device__ __forceinline__ void st_if(double* p, double v, bool pred) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p st.shared.f64 [%0], %1;\n\t}"
               ::"r"((uint32_t)__cvta_generic_to_shared(p)), "d"(v), "r"((int)pred) : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Two CTAs for one user: which chain a CTA runs, and what the fp32 one tells the other.
constexpr int kAlone = 0, kFp32Half = 1, kFp64Half = 2;
constexpr int kNotNeeded = 1, kCarryOn = 2;
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Store to the same place in the other CTA's shared memory.
__device__ __forceinline__ void st_peer(void* local, uint32_t v, uint32_t rank) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(rank));
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote), "r"(v) : "memory");
}

// log2 of the residual that an early end of T may leave, the largest diagonal entry being in [1, 2): 2^-4 of what
// rounding does anyway
constexpr float kTailBits = -28.f;

// What a thread carries through the Householder steps.
template <typename T, int D, bool KEEP> struct TriState {
  using C = TriCfg<D>;
  T a[C::RT][C::NCH][4];        // its tile of the current matrix
  float q[KEEP ? C::RT : 1][KEEP ? C::NCH : 1][4];   // its tile of Q
  T x[C::NCH][4], xr[C::RT];    // column k below the diagonal at its columns and rows, zero elsewhere
  T y[C::RT];                   // A x at its rows
  T s2, x1, dk;                 // |x|^2, the subdiagonal entry, the diagonal entry
  float tr_rest, tr_comp, stop_tr, stop_x2;   // trace not yet reduced, compensated; the stop
  int k_stop;                   // step at which the reduction stopped early (uniform), or -1
  // for the lane's shift x (fp32): 2 log2(x / 2), e^2 over the last pivot of x - T, its negative pivots so far, and
  // 2 log2 of the bound on what a vector of an eigenvalue above x leaves behind the last row
  float sx, lx, cpl, left;
  int above;
};
// Where the steps exchange and leave their results.
template <typename T> struct TriOut {
  T *dg, *eo, *yv, *xp;
  float *betas, *hv;
  float* stop;                  // [2] (0 or 1) for warps without unfinished rows: the reduction ended in the step before
  const volatile int* verdict;  // fp64 beside an fp32 partner: what it says, looked at every eight steps; else nullptr
  int r;
};

// From the new column k (s.x, s.xr: not yet masked) to the state before step k: A x and row k+1
// into shared memory.  M: the chunk that holds column k.
template <int M, typename T, int D, bool KEEP>
__device__ __forceinline__ void tri_prepare(TriState<T, D, KEEP>& s, const TriOut<T>& o, int k, int tid) {
  using C = TriCfg<D>;
  constexpr int GX = C::GX, RT = C::RT, NCH = C::NCH, CW = C::CW, M2 = M + 1 < NCH ? M + 1 : M, R0 = C::first_row(M);
  const int lane = tid & 31, g = lane & (GX - 1), row0 = tid / GX;
  const int k1 = k + 1, par = k & 1, kc = k1 - CW * M;      // column k+1 within the chunk (CW: it opens the next one)
  // the entries k and k+1 of the column
  const T dkl = (k & 2) ? ((k & 1) ? s.x[M][3] : s.x[M][2]) : ((k & 1) ? s.x[M][1] : s.x[M][0]);
  const T x1l = (k1 & 2) ? ((k1 & 1) ? s.x[M][3] : s.x[M][2]) : ((k1 & 1) ? s.x[M][1] : (kc == CW ? s.x[M2][0] : s.x[M][0]));
  s.dk = __shfl_sync(kFull, dkl, (k & (CW - 1)) >> 2);
  s.x1 = __shfl_sync(kFull, x1l, (k1 & (CW - 1)) >> 2);
#pragma unroll
  for (int c = 0; c < 4; ++c) s.x[M][c] = (4 * g + c >= kc) ? s.x[M][c] : T(0);
#pragma unroll
  for (int rr = R0; rr < RT; ++rr) s.xr[rr] = (row0 + 32 * rr >= k1) ? s.xr[rr] : T(0);
  // row k+1 of the matrix (predicated stores: no index into the registers may depend on k)
#pragma unroll
  for (int rr = R0; rr <= C::last_next(M); ++rr)
#pragma unroll
    for (int m = M; m < NCH; ++m) st4_if(o.xp + par * D + CW * m + 4 * g, s.a[rr][m], row0 + 32 * rr == k1);
  T n0 = 0, n1 = 0;
#pragma unroll
  for (int rr = R0; rr < RT; ++rr) {
    T t0 = 0, t1 = 0;
#pragma unroll
    for (int m = M; m < NCH; ++m) {
      t0 = fma_t(s.a[rr][m][0], s.x[m][0], t0); t1 = fma_t(s.a[rr][m][1], s.x[m][1], t1);
      t0 = fma_t(s.a[rr][m][2], s.x[m][2], t0); t1 = fma_t(s.a[rr][m][3], s.x[m][3], t1);
    }
    s.y[rr] = row_sum<GX>(t0 + t1);
  }
#pragma unroll
  for (int m = M; m < NCH; ++m) {
    n0 = fma_t(s.x[m][0], s.x[m][0], n0); n1 = fma_t(s.x[m][1], s.x[m][1], n1);
    n0 = fma_t(s.x[m][2], s.x[m][2], n0); n1 = fma_t(s.x[m][3], s.x[m][3], n1);
  }
  s.s2 = row_sum<GX>(n0 + n1);
#pragma unroll
  for (int rr = R0; rr < RT; ++rr) st_if(o.yv + par * D + row0 + 32 * rr, s.y[rr], g == 0);
}

// ---- Householder steps k whose column k+1 lies in chunk M ---------------------------------------
// A <- H A H with H = I - beta v v^T: w = u - kappa v, u = A v, kappa = beta v^T u / 2,
// A <- A - beta (v w^T + w v^T); Q <- Q H.
template <int M, int RP, typename T, int D, bool KEEP>
__device__ __forceinline__ void tri_stage(TriState<T, D, KEEP>& s, const TriOut<T>& o, int tid) {
  using C = TriCfg<D>;
  constexpr int GX = C::GX, RT = C::RT, NCH = C::NCH, CW = C::CW, NW = C::NW;
  constexpr int R0 = C::first_row(M);
  constexpr int K0 = CW * M > 0 ? CW * M - 1 : 0, K1 = CW * (M + 1) - 1 < D - 2 ? CW * (M + 1) - 1 : D - 2;
  constexpr bool F64 = sizeof(T) == 8;
  const int lane = tid & 31, warp = tid >> 5, g = lane & (GX - 1), row0 = tid / GX;
  if (s.k_stop >= 0) return;
  int kend = K1;
#pragma unroll 1
  for (int k = K0; k < kend; ++k) {
    const int k1 = k + 1, par = k & 1, kc = k1 - CW * M;
    const T* const yv = o.yv + par * D;
    const T* const xp = o.xp + par * D;
    if (F64 && o.verdict != nullptr && (k & 7) == 7 && __syncthreads_or(*o.verdict == kNotNeeded)) { s.k_stop = D; return; }
    __syncthreads();
    if (!KEEP && C::rows_end(warp) <= k1) {                    // only finished rows
      if (!F64 && *(volatile float*)(o.stop + par) != 0.f) { s.k_stop = k - 1; return; }
      continue;
    }
    // Whether T may end at row k.  The vote, and what the answer goes into, come behind the update: before it they held it up
    // (8 power-law users, r = 8: d = 32 30.8 -> 29.9 us per pass, d = 64 51.3 -> 50.8, d = 128 147.3 -> 146.6; without
    // the tail 30.5, 51.9 and 146.4).  The scalars for it are known already at this point.  They are worked out where a schedule
    // measured best: at d = 128 here, beside the reads; at d = 64 for r > 32 between the reflector's scalars and the
    // update (all 64 directions 100.9 -> 100.3); else behind the update (elsewhere registers spill at d = 64).
    bool stop = false;
    auto look = [&] {
      if (F64) return;
      // Rank-revealing stop: once the rows below k carry a negligible trace (G is positive
      // semi-definite, so that bounds every entry of the block) and row k hardly couples to them,
      // T ends at row k.  A history of low rank -- the premise of the method -- then costs its rank
      // in Householder steps, and every later phase works on the shorter T.
      const float d = -(float)s.dk - s.tr_comp, t = s.tr_rest + d;   // compensated: the trace is ~10^7 stop thresholds
      s.tr_comp = (t - s.tr_rest) - d;
      s.tr_rest = t;
      stop = (int)(k1 >= o.r) & (int)(t <= s.stop_tr) & (int)((float)s.s2 <= s.stop_x2);   // no branches
      // Or the kept vectors do not reach the rows below k.  Those behind row j have trace t_j, so no eigenvalue of
      // theirs, reduced or not, is above that, and the pivots of x - T_{j+1..k} are above x - t_j for a shift
      // x >= 2 t_j.  Entry k of a vector of an eigenvalue above x is then at most prod_{j <= i < k} |e_i| / (x / 2)^(k-j),
      // and times |e_k| that is the residual (for a norm of 1) that ending T at row k adds.  So T may end there once
      // it has r eigenvalues above some x for which that is below the rounding level.  Every lane watches an x.
      // A history of rank r plus noise, whose other rows never become negligible, so ends after about r + 5 steps
      // instead of d - 2: 32 x 1024 x 64 with r = 16 50.4 -> 33.2 us per pass, 8 x 4096 x 128 with r = 32 149 -> 82.
      const float pv = (s.sx - (float)s.dk) - s.cpl, s2 = (float)s.s2;
      s.above += (int)(__float_as_uint(pv) >> 31);
      s.cpl = s2 * rcp_fast(pv);
      s.left = t + t <= s.sx ? s.left + (lg2(s2) - s.lx) : s.lx;
    };
    if (D == 128) look();
    // x^T A x; meanwhile the reflector's scalars
    const T yk1 = yv[k1], xpk1 = xp[k1];
    // A x at the thread's columns; kept for the update where there are registers for it (d = 128: a
    // read of 16 bytes takes the SM's shared memory four cycles a warp)
    T d0 = 0, d1 = 0, d2 = 0, d3 = 0, yc[D == 128 ? NCH : 1][4];
#pragma unroll
    for (int m = M; m < NCH; ++m) {
      T (&t)[4] = yc[D == 128 ? m : 0];
      ld4(yv + CW * m + 4 * g, t);
      d0 = fma_t(s.x[m][0], t[0], d0); d1 = fma_t(s.x[m][1], t[1], d1);
      d2 = fma_t(s.x[m][2], t[2], d2); d3 = fma_t(s.x[m][3], t[3], d3);
    }
    const T xax = row_sum<GX>((d0 + d1) + (d2 + d3));
    // A column of zeros has beta = 0: w and the update vanish, and the step still hands on column k+1.
    const T tiny = T(F64 ? 1e-290 : 1e-35);
    const bool reflect = s.s2 > tiny;
    const T nrm = s.s2 * rsqrt_t(reflect ? s.s2 : tiny);
    const T alpha = reflect ? (s.x1 < 0 ? nrm : -nrm) : s.x1;
    const T vk1 = reflect ? s.x1 - alpha : T(0);
    const T beta = reflect ? rcp_t(nrm * abs_t(vk1)) : T(0);
    if (D != 128 && RP > 32) look();
    // x becomes v
#pragma unroll
    for (int c = 0; c < 4; ++c) s.x[M][c] = (4 * g + c == kc) ? vk1 : s.x[M][c];
    if (!KEEP) {                                             // reflector k (zero at rows <= k)
#pragma unroll
      for (int m = M; m < NCH; ++m) {
        const float f[4] = {(float)s.x[m][0], (float)s.x[m][1], (float)s.x[m][2], (float)s.x[m][3]};
        st4_if(o.hv + k * D + CW * m + 4 * g, f, (int)(warp == NW - 1) & (int)(lane < GX));
      }
    }
    float qs[KEEP ? RT : 1];
    if (KEEP) {
#pragma unroll
      for (int rr = 0; rr < RT; ++rr) {
        float q0 = 0.f, q1 = 0.f;
#pragma unroll
        for (int m = M; m < NCH; ++m)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            if (c & 1) q1 = fmaf(s.q[KEEP ? rr : 0][KEEP ? m : 0][c], (float)s.x[m][c], q1);
            else q0 = fmaf(s.q[KEEP ? rr : 0][KEEP ? m : 0][c], (float)s.x[m][c], q0);
          }
        qs[KEEP ? rr : 0] = (float)beta * row_sum<GX>(q0 + q1);
      }
    }
    // v^T A v = x^T A x - 2 alpha (A x)_{k+1} + alpha^2 a_{k+1,k+1}
    const T kap = T(0.5) * beta * fma_t(alpha, fma_t(alpha, xpk1, T(-2) * yk1), xax);
    const T wk1 = fma_t(-kap, vk1, fma_t(-alpha, xpk1, yk1));
    const T bv1 = beta * vk1, bw1 = beta * wk1;
    T bv[RT], bw[RT];
#pragma unroll
    for (int rr = R0; rr < RT; ++rr) {
      const int row = row0 + 32 * rr;
      const T xpi = xp[row], v = row == k1 ? vk1 : s.xr[rr];
      T w = fma_t(-kap, v, fma_t(-alpha, xpi, s.y[rr]));
      w = row >= k1 ? w : T(0);
      bv[rr] = beta * v; bw[rr] = beta * w;
      s.xr[rr] = fma_t(-bw1, v, fma_t(-bv1, w, xpi));
    }
#pragma unroll
    for (int m = M; m < NCH; ++m) {
      T pp[4];
      T (&yy)[4] = yc[D == 128 ? m : 0];
      if (D != 128) ld4(yv + CW * m + 4 * g, yy);
      ld4(xp + CW * m + 4 * g, pp);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const T v = s.x[m][c];
        T w = fma_t(-kap, v, fma_t(-alpha, pp[c], yy[c]));
        if (m == M) w = (4 * g + c >= kc) ? w : T(0);        // finished columns stay as they are
#pragma unroll
        for (int rr = R0; rr < RT; ++rr) s.a[rr][m][c] = fma_t(-bw[rr], v, fma_t(-bv[rr], w, s.a[rr][m][c]));
        if (KEEP) {
#pragma unroll
          for (int rr = 0; rr < RT; ++rr)
            s.q[KEEP ? rr : 0][KEEP ? m : 0][c] = fmaf(-qs[KEEP ? rr : 0], (float)v, s.q[KEEP ? rr : 0][KEEP ? m : 0][c]);
        }
        s.x[m][c] = fma_t(-bw1, v, fma_t(-bv1, w, pp[c]));   // column k+1 of the updated matrix
      }
    }
    if (D != 128 && RP <= 32) look();
    if (!F64) stop = (int)stop | __any_sync(kFull, (int)(s.above >= o.r) & (int)(s.left <= 2.f * kTailBits));
    const bool last = tid == C::NT - 1;
    st_if(o.dg + k, s.dk, last);
    st_if(o.eo + k, stop ? T(0) : alpha, last);
    if (!KEEP) st_if(o.betas + k, (float)beta, last);
    if (!KEEP && !F64) st_if(o.stop + (par ^ 1), stop ? 1.f : 0.f, last);
    kend = stop ? k1 : kend;
    s.k_stop = stop ? k : -1;              // this step is still made: it touches nothing left of column k+1
    tri_prepare<M, T, D, KEEP>(s, o, k1, tid);
  }
}

// Number of eigenvalues of T below x.  p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1} is the leading
// principal minor of order i+1 of T - x I; the sign changes along p_0 = 1, p_1, ... count the
// eigenvalues below x.  The off-diagonal squares are floored above zero, so an exact zero never
// persists, and an isolated zero gives one change whichever sign the hardware gives it.  The
// signs are shifted into a word (one instruction per row) and their changes counted by blocks of
// eight rows.  The pair (p, q) is brought back near 1 by a power of two taken two rows before it is
// applied, off the dependency chain: |d - x| and e^2 are bounded by the scaling of G, and rows
// shrink by 2^-23 (fp64: 2^-52) at most, so in fp32 every four rows keep it in range, in fp64 every
// eight.  The next block's rows are fetched while this one is counted.  CH points at once: one
// chain alone leaves more than half of a scheduler's slots empty.  Two blocks an iteration in fp64 (8 x 16384
// x 128: 239.9 -> 234.3 us per pass), one in fp32 (two: 16 x 10240 x 64 48.2 -> 48.6).
template <typename T, int CH>
__device__ __forceinline__ void sturm(const T* __restrict__ dg, const T* __restrict__ e2s, const T (&x)[CH], int (&n)[CH], int nb8) {
  T p[CH], q[CH], sc[CH];
  unsigned bits[CH];
#pragma unroll
  for (int h = 0; h < CH; ++h) { p[h] = 1; q[h] = 0; bits[h] = 0; n[h] = 0; }
  T dd[8], ee[8];
  auto fetch = [&](int at, T (&d)[8], T (&e)[8]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      T t[4], u[4];
      ld4(dg + at + 4 * h, t); ld4(e2s + at + 4 * h, u);
#pragma unroll
      for (int c = 0; c < 4; ++c) { d[4 * h + c] = t[c]; e[4 * h + c] = u[c]; }
    }
  };
  fetch(0, dd, ee);
#pragma unroll (sizeof(T) == 8 ? 2 : 1)
  for (int ib = 0; ib < nb8; ++ib) {
    T dn[8], en[8];
    fetch(8 * min(ib + 1, nb8 - 1), dn, en);
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int h = 0; h < CH; ++h) {
        const T rr = fma_t(dd[u] - x[h], p[h], -(ee[u] * q[h]));
        bits[h] = __funnelshift_l(top_word(rr), bits[h], 1);
        q[h] = p[h]; p[h] = rr;
        constexpr int P = sizeof(T) == 4 ? 4 : 8;
        if (u % P == P - 3) sc[h] = pow2_scale(p[h], q[h]);
        if (u % P == P - 1) { p[h] *= sc[h]; q[h] *= sc[h]; }
      }
#pragma unroll
    for (int h = 0; h < CH; ++h) n[h] += __popc((bits[h] ^ (bits[h] >> 1)) & 0xffu);
#pragma unroll
    for (int u = 0; u < 8; ++u) { dd[u] = dn[u]; ee[u] = en[u]; }
  }
}

// One of the two minor sequences of T - lambda I for one eigenvalue, and the multipliers of z:
//   DOWN = false: leading minors p_i;   z_i = mul_i z_{i+1},  mul_i = -e_i p_i / p_{i+1}
//   DOWN = true:  trailing minors t_i;  z_i = mul_i z_{i-1},  mul_i = -e_{i-1} t_{i+1} / t_i
// mn[i] = log2 of the minor before row i (p_i, t_{i+1}).  A minor below pfl times the one before is
// replaced by that much (a perturbation of d_i by pfl).  Four rows are fetched ahead.
template <bool DOWN, typename T, int RP>
__device__ __forceinline__ void minors(const T* __restrict__ dg, const T* __restrict__ eo, const T* __restrict__ e2s, int de,
                                       T lam, T pfl, float* __restrict__ mul, float* __restrict__ mn) {
  T p = 1, po = 0;
  int ex = 0;
  auto fetch = [&](int t0, T (&d)[4], T (&e2)[4], T (&e1)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = min(t0 + u, de - 1), n = DOWN ? de - 1 - t : t;
      d[u] = dg[n];
      if (DOWN) {                       // e2s[0] = 0 stands for the coupling past the last row
        e2[u] = e2s[t > 0 ? n + 1 : 0];
        e1[u] = eo[max(n - 1, 0)];      // unused at n = 0
      } else {
        e2[u] = e2s[n];
        e1[u] = eo[n];
      }
    }
  };
  T d[4], e2[4], e1[4];
  fetch(0, d, e2, e1);
#pragma unroll 1
  for (int t0 = 0; t0 < de; t0 += 4) {
    T dn[4], e2n[4], e1n[4];
    fetch(t0 + 4, dn, e2n, e1n);
    float mu[4], lg[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if constexpr (sizeof(T) == 4) lg[u] = lg2(fabsf(p)) + (float)ex;
      T np = fma_t(d[u] - lam, p, -(e2[u] * po));
      const T fl = pfl * abs_t(p);
      np = abs_t(np) >= fl ? np : -fl;
      if constexpr (sizeof(T) == 4) {
        mu[u] = -e1[u] * (p * rcp_fast(np));
      } else {
        // The fp64 minors of four rows can shrink past the range of fp32, which takes their ratio and logarithm:
        // both are brought near 1 by their exponents (they differ by 2^61 at most).
        const int m = max(__double2hiint(p) & 0x7ff00000, __double2hiint(np) & 0x7ff00000) - 0x3ff00000;
        const float pf = (float)__hiloint2double(__double2hiint(p) - m, __double2loint(p));
        lg[u] = lg2(fabsf(pf)) + (float)(ex + (m >> 20));
        mu[u] = -(float)e1[u] * (pf * rcp_fast((float)__hiloint2double(__double2hiint(np) - m, __double2loint(np))));
      }
      po = p; p = np;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int n = DOWN ? de - 1 - (t0 + u) : t0 + u;
      st_if(mul + n * RP, mu[u], t0 + u < de);
      st_if(mn + n * RP, lg[u], t0 + u < de);
    }
    const T sc = pow2_scale(p, po);
    p *= sc; po *= sc; ex -= exponent(sc);
#pragma unroll
    for (int u = 0; u < 4; ++u) { d[u] = dn[u]; e2[u] = e2n[u]; e1[u] = e1n[u]; }
  }
}

// Acceptance thresholds (chosen by the storage type).
struct TriTol {
  float eps_vec;     // bound on sin(angle) of a kept vector implied by its residual and gap
  float floor_rel;   // residuals below floor_rel * theta_1 are at the rounding level of fp32
  float ortho;       // largest |V^T V - I| entry that needs no further orthogonalisation
  float gap_min;     // smallest gap between kept eigenvalues, relative to the largest, the route is trusted with
  float stop_trace;  // the reduction stops once the remaining rows' trace is below this fraction of trace(G) ...
  float stop_couple; // ... and the current row couples to them by less than this fraction of it
  float sweep_stop;  // of the Jacobi fallback
};

struct TriShared {
  double trace;
  float tr_t, rest;  // traces of T and of the rows left out
  int rows;          // of T
  float stop[2];
  int flags[4];
  int why;
  int verdict;       // written by the other CTA of the user's pair
};

// Steps 2-7 in T for the user of this CTA; acc: the thread's tile of G in fp32.  Returns whether the
// result is certified; Vc: where the vectors are ([D][RP]).  theta[] holds the eigenvalues of sc * G,
// part[NW ..] the largest component of every vector per warp.  Without force, nothing is finished
// that cannot be certified any more.  With two CTAs for the user (half) `not_mine` comes back true where
// the other one has the result.
template <typename T, int D, int RP>
__device__ __forceinline__ bool tri_chain(const float (&acc)[TriCfg<D>::RT][TriCfg<D>::NCH][4], float* __restrict__ smem,
                                          TriShared& sh, const float* __restrict__ gout, float sc, int r, bool force,
                                          const TriTol& tol, bool trigger_early, int half, bool& not_mine, float*& Vc_out, int& passes, int tid) {
  using C = TriCfg<D>;
  using L = TriSmem<D, RP>;
  constexpr int GX = C::GX, RT = C::RT, NT = C::NT, NW = C::NW, NCH = C::NCH, CW = C::CW, LD = C::LD;
  constexpr bool F64 = sizeof(T) == 8, KEEP = !F64 && D <= 64;
  constexpr int NE = RP / 32;                 // groups of 32 eigenvalues (columns)
  const int lane = tid & 31, warp = tid >> 5, g = lane & (GX - 1), row0 = tid / GX;
  T* const dg = reinterpret_cast<T*>(smem + L::DG);
  T* const eo = reinterpret_cast<T*>(smem + L::EO);
  T* const e2s = reinterpret_cast<T*>(smem + L::E2);
  T* const lamv = reinterpret_cast<T*>(smem + L::LAM);
  float* const theta = smem + L::TH;
  float* const lam32 = smem + L::L32;
  float* const part = smem + L::PART;
  bool ok = true;
  passes = 0;
  not_mine = false;

  // ---- 2. Householder tridiagonalisation, the matrix in registers ------------------------------
  int k_stop;
  {
    TriOut<T> o;
    o.dg = dg; o.eo = eo;
    o.yv = reinterpret_cast<T*>(smem + L::YV);
    o.xp = reinterpret_cast<T*>(smem + L::XP);
    o.betas = smem + L::BE; o.hv = smem + L::R0;
    o.stop = sh.stop; o.r = r;
    o.verdict = F64 && half == kFp64Half ? &sh.verdict : nullptr;
    TriState<T, D, KEEP> s;
    const float trs = (float)((double)sc * sh.trace);
    s.tr_rest = trs; s.tr_comp = 0.f;
    s.stop_tr = trs * tol.stop_trace;
    s.stop_x2 = (trs * tol.stop_couple) * (trs * tol.stop_couple);
    s.k_stop = -1;
    s.sx = trs * ex2(-1.f - 0.5f * (float)lane); s.lx = 2.f * lg2(s.sx) - 2.f;     // trace / 2 .. trace / 2^16.5
    s.cpl = 0.f; s.left = s.lx; s.above = 0;
#pragma unroll
    for (int rr = 0; rr < RT; ++rr)
#pragma unroll
      for (int m = 0; m < NCH; ++m)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          s.a[rr][m][c] = (T)(acc[rr][m][c] * sc);
          if (KEEP) s.q[KEEP ? rr : 0][KEEP ? m : 0][c] = (CW * m + 4 * g + c == row0 + 32 * rr) ? 1.f : 0.f;
        }
    // column 0 (= row 0), by way of the buffer that step 1 writes
#pragma unroll
    for (int m = 0; m < NCH; ++m) st4_if(o.xp + D + CW * m + 4 * g, s.a[0][m], row0 == 0);
    if (!KEEP)
      for (int e = tid; e < D * D / 4; e += NT) reinterpret_cast<float4*>(o.hv)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
#pragma unroll
    for (int m = 0; m < NCH; ++m) ld4(o.xp + D + CW * m + 4 * g, s.x[m]);
#pragma unroll
    for (int rr = 0; rr < RT; ++rr) s.xr[rr] = o.xp[D + row0 + 32 * rr];
    tri_prepare<0, T, D, KEEP>(s, o, 0, tid);
    tri_stage<0, RP, T, D, KEEP>(s, o, tid);
    tri_stage<1, RP, T, D, KEEP>(s, o, tid);
    if constexpr (NCH > 2) {
      tri_stage<2, RP, T, D, KEEP>(s, o, tid);
      tri_stage<3, RP, T, D, KEEP>(s, o, tid);
    }
    // Finished warps learn of a stop one barrier later.  Those that did in the loop have passed that
    // barrier there; for all others (no stop, or one in the very last step) it is this one.
    if (!KEEP && !F64 && (s.k_stop < 0 || C::rows_end(warp) > s.k_stop + 1)) {
      __syncthreads();
      if (s.k_stop < 0 && *(volatile float*)(sh.stop + (D & 1)) != 0.f) s.k_stop = D - 3;
    }
    // the diagonal of the rows left out by an early end, for the certificate
    if (!F64 && s.k_stop >= 0) {
#pragma unroll
      for (int rr = 0; rr < RT; ++rr) {
        const int row = row0 + 32 * rr;
        const float v = (float)C::diagonal([&](int m, int c) { return s.a[rr][m][c]; }, rr, row0);
        st_if(part + row, v, (int)(row > s.k_stop) & (int)(((row & (CW - 1)) >> 2) == g));
      }
    }
    // the last 2 x 2 block
    if (s.k_stop < 0 && tid == NT - 1) {
      dg[D - 2] = s.dk; eo[D - 2] = s.x1; eo[D - 1] = 0;
      dg[D - 1] = s.a[RT - 1][NCH - 1][3];
    }
    if (KEEP) {
      float* Qt = smem + L::R0;
#pragma unroll
      for (int rr = 0; rr < RT; ++rr)
#pragma unroll
        for (int m = 0; m < NCH; ++m)
#pragma unroll
          for (int c = 0; c < 4; ++c) Qt[(CW * m + 4 * g + c) * LD + row0 + 32 * rr] = s.q[KEEP ? rr : 0][KEEP ? m : 0][c];
    }
    k_stop = s.k_stop;
  }
  if (F64 && half == kFp64Half) {            // the fp32 chain is long past its eigenvalues; they lie in lam32[]
    cluster_arrive();
    cluster_wait();
    if (sh.verdict == kNotNeeded) { not_mine = true; return false; }
  }
  // T has `de` rows (all D unless the reduction stopped early), padded with zero rows to a multiple of 8
  const int de = k_stop >= 0 ? k_stop + 1 : D, de8 = (de + 7) & ~7;
  const int kb = k_stop >= 0 ? k_stop : D - 2;            // reflectors 0 .. kb-1 exist
  if (tid < de8 - de) { dg[de + tid] = 0; eo[de + tid] = 0; }
  __syncthreads();

  // ---- 3. Gershgorin interval, floored squares, trace (every warp for itself); multisection ------
  T lo, hi, tnorm;
  {
    T l = T(3.0e38), h = T(-3.0e38), tr = 0;
    float rest = 0.f;
#pragma unroll
    for (int q = 0; q < D / 32; ++q) {
      const int n = lane + 32 * q;
      const bool in = n < de;
      const T el0 = eo[max(n - 1, 0)], er0 = eo[n], dd0 = dg[n];
      const T el = ((int)in & (int)(n > 0)) ? el0 : T(0), er = in ? er0 : T(0), dd = in ? dd0 : T(0);   // eo[de-1] = 0
      const T rad = abs_t(er) + abs_t(el);
      l = ((int)in & (int)(dd - rad < l)) ? dd - rad : l;
      h = ((int)in & (int)(dd + rad > h)) ? dd + rad : h;
      tr += dd;
      if (!F64 && n >= de) rest += part[n];
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const T l2 = __shfl_xor_sync(kFull, l, o), h2 = __shfl_xor_sync(kFull, h, o);
      l = l2 < l ? l2 : l; h = h2 > h ? h2 : h;
      tr += __shfl_xor_sync(kFull, tr, o);
      if (!F64) rest += __shfl_xor_sync(kFull, rest, o);
    }
    const T span = h - l;
    lo = l - T(1e-6) * span - T(1e-30); hi = h + T(1e-6) * span + T(1e-30);
    tnorm = -lo > hi ? -lo : hi;
    const T fl = tnorm * T(F64 ? 2.7755575615628914e-17 : 1.4901161e-08);           // 2^-55, 2^-26 of |T|
    if (warp == 0) {
      for (int n = lane; n < de8; n += 32) {
        const T e = n > 0 ? eo[n - 1] : T(0);
        e2s[n] = n > 0 ? (e * e > fl * fl ? e * e : fl * fl) : T(0);
      }
      if (lane == 0) { sh.tr_t = (float)tr; sh.rest = rest; sh.rows = de; }
    }
  }
  __syncthreads();
  {
    constexpr int PT = NT / RP < 8 ? NT / RP : 8;               // lanes per eigenvalue
    constexpr int CH = NW == 4 ? 2 : 1, NPT = PT * CH;          // points per lane (one warp per scheduler: two)
    constexpr int NP0 = 256, PRB = 16 / PT;                     // points of the first step, all threads together
    constexpr int STEPS = (NPT == 8 ? 6 : 9);                   // (NP0 + 1) (NPT + 1)^STEPS >= 2^27
    constexpr int STEPS64 = (NPT == 8 ? 14 : 19);               // fp64: (NPT + 1)^STEPS64 >= 2^44 from the Gershgorin interval
    constexpr int STEPS_B = (NPT == 8 ? 9 : 12);                // >= 2^27.9, from a bracket of 2^-14 |T|: to 2^-42 |T|
    static_assert(PT * RP == NT && (NPT == 8 || NPT == 4) && CH * NT == NP0 && NP0 <= 3 * NW * RP, "every lane has points");
    const int j = tid / PT, pt = tid % PT, jj = j < r ? j : r - 1;     // surplus lanes shadow column r-1
    const int target = de8 - 1 - jj;    // lambda_(jj-th largest) >= x  <=>  #(eigenvalues < x) <= target
    int steps = STEPS;
    if (!F64) {
      // The first step starts from one interval for all eigenvalues, so they share its points: 256 instead
      // of NPT; every eigenvalue finds its place among their counts by two 16-ary searches.
      const T w = (hi - lo) * T(1.0 / (NP0 + 1));
      T x[CH];
      int n[CH];
#pragma unroll
      for (int h = 0; h < CH; ++h) x[h] = fma_t(T(tid + h * NT + 1), w, lo);
      sturm<T, CH>(dg, e2s, x, n, de8 >> 3);
      int* const cnt = reinterpret_cast<int*>(part);
#pragma unroll
      for (int h = 0; h < CH; ++h) cnt[tid + h * NT] = n[h];
      __syncthreads();
      int a = 0, c = 0;
#pragma unroll
      for (int q = 0; q < PRB; ++q)
        a += __popc((__ballot_sync(kFull, cnt[16 * (PT * q + pt) + 15] <= target) >> (lane & ~(PT - 1))) & ((1u << PT) - 1));
      const int a0 = min(a, NP0 / 16 - 1) * 16;
#pragma unroll
      for (int q = 0; q < PRB; ++q)
        c += __popc((__ballot_sync(kFull, cnt[a0 + PT * q + pt] <= target) >> (lane & ~(PT - 1))) & ((1u << PT) - 1));
      const int idx = a0 + c;                                   // points at or below the eigenvalue
      const T nlo = fma_t(T(idx), w, lo), nhi = fma_t(T(idx + 1), w, lo);
      lo = idx == 0 ? lo : nlo;
      hi = idx == NP0 ? hi : nhi;
    } else {
      // bracket: the fp32 chain's eigenvalue +- 2^-15 |T| where the counts confirm it
      const T c0 = (T)lam32[j], dl = tnorm * T(3.0517578125e-05);
      T x[CH];
      int n[CH];
      if (CH == 2) { x[0] = c0 - dl; x[CH - 1] = c0 + dl; }
      else x[0] = (pt & 1) ? c0 + dl : c0 - dl;
      sturm<T, CH>(dg, e2s, x, n, de8 >> 3);
      const bool in = CH == 2 ? (int)(n[0] <= target) & (int)(n[CH - 1] > target) : ((pt & 1) ? n[0] > target : n[0] <= target);
      const unsigned all = __ballot_sync(kFull, in);
      const bool mine = ((~all >> (lane & ~(PT - 1))) & ((1u << PT) - 1)) == 0;
      lo = mine ? c0 - dl : lo; hi = mine ? c0 + dl : hi;
      steps = all == kFull ? STEPS_B : STEPS64;
    }
#pragma unroll 1
    for (int step = 0; step < steps; ++step) {
      const T w = (hi - lo) * T(1.0 / (NPT + 1));
      T x[CH];
      int n[CH], idx = 0;                                        // points at or below the eigenvalue
#pragma unroll
      for (int h = 0; h < CH; ++h) x[h] = fma_t(T(pt + h * PT + 1), w, lo);
      sturm<T, CH>(dg, e2s, x, n, de8 >> 3);
#pragma unroll
      for (int h = 0; h < CH; ++h)
        idx += __popc((__ballot_sync(kFull, n[h] <= target) >> (lane & ~(PT - 1))) & ((1u << PT) - 1));
      const T nlo = fma_t(T(idx), w, lo), nhi = fma_t(T(idx + 1), w, lo);
      lo = idx == 0 ? lo : nlo;
      hi = idx == NPT ? hi : nhi;
    }
    if (pt == 0) lamv[j] = T(0.5) * (lo + hi);
    if (!F64 && pt == 0) lam32[j] = (float)(T(0.5) * (lo + hi));
  }
  __syncthreads();
  if (!F64) {                            // gaps too small for the angle the storage type needs
    const int tight = tid < r - 1 && (float)(lamv[tid] - lamv[tid + 1]) < tol.gap_min * (float)lamv[0];
    const bool gap = __syncthreads_or(tight);
    if (half == kFp32Half) {
      if (gap && tid < RP) st_peer(lam32 + tid, __float_as_uint(lam32[tid]), 1);
      if (tid == 0) st_peer(&sh.verdict, gap ? kCarryOn : kNotNeeded, 1);
      __syncwarp();
      cluster_arrive();
      not_mine = gap;
    }
    if (gap) {
      ok = false;
      if (tid == 0) sh.why |= kWhyGap;
      if (!force) return false;
    }
  }

  // ---- 4. twisted factorisation -----------------------------------------------------------------
  float* const up = smem + L::A1;
  float* const dn = smem + L::A2;
  float* const lp = smem + L::A3;
  float* const lt = smem + L::A4;
  {
    const T pfl = tnorm * T(F64 ? 1.734723475976807e-18 : 9.3132257e-10);            // pivot floor 2^-59, 2^-30 of |T|
    if (warp < NE) minors<false, T, RP>(dg, eo, e2s, de, lamv[32 * warp + lane], pfl, up + 32 * warp + lane, lp + 32 * warp + lane);
    else if (warp < 2 * NE)
      minors<true, T, RP>(dg, eo, e2s, de, lamv[32 * (warp - NE) + lane], pfl, dn + 32 * (warp - NE) + lane, lt + 32 * (warp - NE) + lane);
  }
  __syncthreads();
  constexpr int NS = NT / RP;                                    // threads per eigenvalue here
  {
    const int j = tid % RP, sl = tid / RP;
    float best = -3.0e38f;
    int kbest = 0;
#pragma unroll 4
    for (int n = sl; n < de; n += NS) {
      const float v = lp[n * RP + j] + lt[n * RP + j];
      kbest = v > best ? n : kbest;
      best = fmaxf(v, best);
    }
    part[sl * RP + j] = best;
    reinterpret_cast<int*>(part)[(NW + sl) * RP + j] = kbest;
  }
  __syncthreads();
  // z_kt = 1, upwards and downwards from there on two warps (no branches: a lane that has not
  // reached its twist index yet keeps z = 1)
  float* const Z = lp;
  if (warp < 2 * NE) {
    const bool dwn = warp >= NE;
    const int j = 32 * (dwn ? warp - NE : warp) + lane;
    float best = -3.4e38f;
    int kt = 0;
#pragma unroll
    for (int sl = 0; sl < NS; ++sl) {
      const float v = part[sl * RP + j];
      const int kk = reinterpret_cast<const int*>(part)[(NW + sl) * RP + j];
      const bool take = (int)(v > best) | ((int)(v == best) & (int)(kk < kt));
      best = take ? v : best;
      kt = take ? kk : kt;
    }
    const float* const mul = (dwn ? dn : up) + j;
    const int n0 = dwn ? 0 : de - 1, sg = dwn ? 1 : -1, tk = dwn ? kt : de - 1 - kt;   // the twist is met at t = tk
    float z = 1.f, ss = 0.f;
#pragma unroll 1
    for (int t0 = 0; t0 < de; t0 += 8) {
      float mu[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) mu[u] = mul[(n0 + sg * min(t0 + u, de - 1)) * RP];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int t = t0 + u;
        z = t > tk ? z * mu[u] : 1.f;
        const float zi = ((int)(t > tk) & (int)(t < de)) ? z : 0.f;
        ss = fmaf(zi, zi, ss);
        st_if(Z + (n0 + sg * t) * RP + j, z, (int)(t >= tk) & (int)(t < de));
      }
    }
    // behind the entries that the other half may still be reading
    part[(2 * NW + (dwn ? 1 : 0)) * RP + j] = ss;
  }
  __syncthreads();

  // ---- 5. V = Q Z -------------------------------------------------------------------------------
  float* Vc = smem + L::A1;      // current vectors
  float* Vn = smem + L::A2;      // next
  const float* const zs = part + 2 * NW * RP;
  if constexpr (KEEP) {
    const float* Qt = smem + L::R0;
    constexpr int CG = RP / 4, RS = NT / CG, NP = (D / 4 + RS - 1) / RS;      // 4 x 4 tiles of V, NP per thread
    const int cg = tid % CG, rq = tid / CG;
    if (RS * NP == D / 4 || rq < D / 4) {
      float v[NP][4][4];
#pragma unroll
      for (int n = 0; n < NP; ++n)
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int c = 0; c < 4; ++c) v[n][x][c] = 0.f;
#pragma unroll 4
      for (int t = 0; t < de; ++t) {
        float z[4];
        ld4(Z + t * RP + 4 * cg, z);
#pragma unroll
        for (int n = 0; n < NP; ++n) {
          float q[4];
          ld4(Qt + t * LD + 4 * (rq + n * RS), q);
#pragma unroll
          for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int c = 0; c < 4; ++c) v[n][x][c] = fmaf(q[x], z[c], v[n][x][c]);
        }
      }
      float zn[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) zn[c] = rsqrtf(1.f + zs[4 * cg + c] + zs[RP + 4 * cg + c]);   // 1 / |z|
#pragma unroll
      for (int n = 0; n < NP; ++n)
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const float t[4] = {v[n][x][0] * zn[0], v[n][x][1] * zn[1], v[n][x][2] * zn[2], v[n][x][3] * zn[3]};
          st4(Vc + (4 * (rq + n * RS) + x) * RP + 4 * cg, t);
        }
    }
  } else {
    // v = H_0 H_1 ... H_{kb-1} z: TPV threads per vector, RB rows each (16-byte pieces dealt round
    // robin: conflict-free), the reflector's inner product completed by shuffles
    constexpr int TPV = NT / RP, RB = D / TPV;
    const int j = tid / TPV, qt = tid % TPV;
    const float zn = rsqrtf(1.f + zs[j] + zs[RP + j]);
    const float* hv = smem + L::R0 + 4 * qt;
    const float* betas = smem + L::BE;
    float z[RB];
#pragma unroll
    for (int u = 0; u < RB; ++u) {
      const int n = ((u >> 2) * TPV + qt) * 4 + (u & 3);
      z[u] = n < de ? Z[n * RP + j] * zn : 0.f;
    }
#pragma unroll 2
    for (int k = kb - 1; k >= 0; --k) {
      float h[RB], d0 = 0.f, d1 = 0.f;
#pragma unroll
      for (int u = 0; u < RB; u += 4) {
        float t[4];
        ld4(hv + k * D + (u >> 2) * TPV * 4, t);
        h[u] = t[0]; h[u + 1] = t[1]; h[u + 2] = t[2]; h[u + 3] = t[3];
        d0 = fmaf(t[0], z[u], d0);     d1 = fmaf(t[1], z[u + 1], d1);
        d0 = fmaf(t[2], z[u + 2], d0); d1 = fmaf(t[3], z[u + 3], d1);
      }
      const float c = -betas[k] * row_sum<TPV>(d0 + d1);
#pragma unroll
      for (int u = 0; u < RB; ++u) z[u] = fmaf(c, h[u], z[u]);
    }
#pragma unroll
    for (int u = 0; u < RB; ++u) Vc[(((u >> 2) * TPV + qt) * 4 + (u & 3)) * RP + j] = z[u];
  }
  __syncthreads();
  // The long serial part is over: the next kernel may start launching -- unless the process runs
  // many requests at once, where its parked CTAs are better kept out a little longer (after the
  // certificate).
  if (trigger_early) pdl_trigger();

  // G for the residuals, over Q or the reflectors; it arrives behind step 6
  float* const Gsm = smem + L::R0;
  for (int e = tid; e < D * D / 4; e += NT) cp_async16(Gsm + 4 * e, gout + 4 * e);

  // The products of steps 6 and 7 are bound by shared-memory reads (16 bytes a lane take four cycles a warp,
  // whatever the lanes share), so every thread has a tile of at least 4 x 4 outputs (2 x 4 at d = 32): column
  // group fastest, so that the eight lanes of a read's phase share the other operand.  A column per lane and
  // 16 rows per thread: 25.7 thousand cycles for both steps at d = 64, r = 64, 20.2 so; 9.3 and 7.3 at r = 32.
  constexpr int CG = RP / 4, TR = D * RP / (4 * NT);        // tile of V: TR rows, 4 columns
  constexpr int UN = RP == 32 ? 8 : 4;                      // rows fetched ahead of their FMAs, as far as registers go
  const int r0 = (tid / CG) * TR, c0 = (tid % CG) * 4;

  // ---- 6. orthogonalisation passes while V^T V - I is above the rounding level ---------------------
  constexpr int TA = RP == 64 ? 8 : 4, SPL = NT / (RP / TA * CG), LPS = 32 / SPL;      // tile of E: TA x 4, SPL lanes share its sum
  static_assert(SPL >= 1 && LPS >= 8, "a read's phase has one row of V");
  float* const Em = smem + L::A4;                            // strict upper triangle of E
  float* const diag = part + RP;
  float* const scol = part + 2 * RP;
  for (;;) {
    const int sp = lane / LPS, tile = warp * LPS + lane % LPS, xa = tile / CG * TA, xc = tile % CG * 4;
    float ev[TA][4];
#pragma unroll
    for (int u = 0; u < TA; ++u)
#pragma unroll
      for (int c = 0; c < 4; ++c) ev[u][c] = 0.f;
#pragma unroll UN
    for (int n = sp * (D / SPL); n < (sp + 1) * (D / SPL); ++n) {
      float va[TA], vc[4];
      ldn(Vc + n * RP + xa, va);
      ld4(Vc + n * RP + xc, vc);
#pragma unroll
      for (int u = 0; u < TA; ++u)
#pragma unroll
        for (int c = 0; c < 4; ++c) ev[u][c] = fmaf(va[u], vc[c], ev[u][c]);
    }
    float emax = 0.f;
#pragma unroll
    for (int u = 0; u < TA; ++u) {
      float up[4];
      const int x = xa + u;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
#pragma unroll
        for (int o = LPS; o < 32; o <<= 1) ev[u][c] += __shfl_xor_sync(kFull, ev[u][c], o);
        float e = ev[u][c] - (x == xc + c ? 1.f : 0.f);
        e = ((int)(x >= r) | (int)(xc + c >= r)) ? 0.f : e;  // surplus columns are copies of column r-1
        up[c] = x < xc + c ? e : 0.f;
        st_if(diag + x, e, x == xc + c);
        emax = (fabsf(e) <= emax) ? emax : fabsf(e);         // a NaN stays
      }
      st4_if(Em + x * RP + xc, up, sp == 0);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const float e2 = __shfl_xor_sync(kFull, emax, o);
      emax = (e2 <= emax) ? emax : e2;
    }
    if (lane == 0) part[warp] = emax;
    __syncthreads();
    float em = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) { const float e = part[w]; em = (e <= em) ? em : e; }
    if (em <= tol.ortho) break;                       // orthonormal to rounding
    if (passes == 6 || !(em <= 0.98f)) { ok = false; if (tid == 0) sh.why |= kWhyOrtho; break; }
    ++passes;
    // One pass of Gram-Schmidt against the ORIGINAL earlier columns (larger eigenvalues, the
    // better determined vectors): v_c <- (v_c - sum_{a<c} E_ac v_a) / |.|.  A later column never
    // changes an earlier one, so a poorly separated pair cannot damage its neighbours; for
    // two vectors the pass is exact, for more it converges quadratically like the symmetric
    // form.
    if (tid < RP) {
      float n0 = 1.f + diag[tid], n1 = 0.f;
#pragma unroll 8
      for (int x = 0; x < RP; x += 2) {
        const float e0 = Em[x * RP + tid], e1 = Em[(x + 1) * RP + tid];
        n0 = fmaf(-e0, e0, n0);
        n1 = fmaf(-e1, e1, n1);
      }
      scol[tid] = rsqrtf(fmaxf(n0 + n1, 1e-6f));
    }
    __syncthreads();
    {
      float o[TR][4];
#pragma unroll
      for (int u = 0; u < TR; ++u)
#pragma unroll
        for (int c = 0; c < 4; ++c) o[u][c] = 0.f;
#pragma unroll 2
      for (int x = 0; x < RP; x += 4) {
        float e[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) ld4(Em + (x + q) * RP + c0, e[q]);
#pragma unroll
        for (int u = 0; u < TR; ++u) {
          float v[4];
          ld4(Vc + (r0 + u) * RP + x, v);
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int c = 0; c < 4; ++c) o[u][c] = fmaf(v[q], e[q][c], o[u][c]);
        }
      }
      float sc4[4];
      ld4(scol + c0, sc4);
#pragma unroll
      for (int u = 0; u < TR; ++u) {
        float v[4];
        ld4(Vc + (r0 + u) * RP + c0, v);
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = (v[c] - o[u][c]) * sc4[c];
        st4(Vn + (r0 + u) * RP + c0, v);
      }
    }
    __syncthreads();
    float* t = Vc; Vc = Vn; Vn = t;
    // With E = L + diag + L^T the pass leaves (I - L)(I + E)(I - L^T) = I + diag - L L^T - L^2 -
    // (L^T)^2 + O(E^3), and the scaling removes the diagonal: what remains off the diagonal is
    // below 3 r max|E|^2.  Where that is a quarter of the bound, V^T V is not formed again.
    if (3.f * (float)r * em * em <= 0.25f * tol.ortho) break;
  }
  Vc_out = Vc;
  cp_async_wait_all();
  __syncthreads();      // G is staged; the vectors are settled; the warps' maxima are read
  if (!ok && !force) return false;

  // ---- 7. Rayleigh quotients and residuals against G; certification; the largest components -------
  {
    // Y = G V (row k of G in the place of column k)
    float y[TR][4], v[TR][4], t[4];
#pragma unroll
    for (int u = 0; u < TR; ++u)
#pragma unroll
      for (int c = 0; c < 4; ++c) y[u][c] = 0.f;
#pragma unroll UN
    for (int k = 0; k < D; ++k) {
      float gg[TR], vk[4];
      ldn(Gsm + k * D + r0, gg);
      ld4(Vc + k * RP + c0, vk);
#pragma unroll
      for (int u = 0; u < TR; ++u)
#pragma unroll
        for (int c = 0; c < 4; ++c) y[u][c] = fmaf(gg[u], vk[c], y[u][c]);
    }
    // sum over the rows of the warp; every column group's first lane stores
    auto column_sums = [&](float* dst) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int o = CG; o < 32; o <<= 1) t[c] += __shfl_xor_sync(kFull, t[c], o);
      st4_if(dst + warp * RP + c0, t, lane < CG);
    };
#pragma unroll
    for (int c = 0; c < 4; ++c) t[c] = 0.f;
#pragma unroll
    for (int u = 0; u < TR; ++u) {
      ld4(Vc + (r0 + u) * RP + c0, v[u]);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        y[u][c] *= sc;
        t[c] = fmaf(v[u][c], y[u][c], t[c]);
      }
    }
    column_sums(part);
    {
      constexpr int RW = D / NW;                       // the largest component of the warp's rows, a column per lane
      float* const lead = part + NW * RP;              // [NW][RP]
#pragma unroll
      for (int h = 0; h < NE; ++h) {
        float best = -1.f, lv = 1.f;
#pragma unroll 8
        for (int u = 0; u < RW; ++u) {
          const float x = Vc[(warp * RW + u) * RP + 32 * h + lane];
          lv = fabsf(x) > best ? x : lv;               // strict: lowest index wins a tie
          best = fmaxf(fabsf(x), best);
        }
        lead[warp * RP + 32 * h + lane] = lv;
      }
    }
    __syncthreads();
    float th[4] = {0.f, 0.f, 0.f, 0.f};
    if (F64) {
#pragma unroll
      for (int c = 0; c < 4; ++c) th[c] = (float)lamv[c0 + c];   // accurate relative to the eigenvalue itself, unlike an fp32 quotient
    } else {
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        float q[4];
        ld4(part + w * RP + c0, q);
#pragma unroll
        for (int c = 0; c < 4; ++c) th[c] += q[c];
      }
    }
    st4_if(theta + c0, th, tid < CG);
#pragma unroll
    for (int c = 0; c < 4; ++c) t[c] = 0.f;
#pragma unroll
    for (int u = 0; u < TR; ++u)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float d = fmaf(-th[c], v[u][c], y[u][c]);
        t[c] = fmaf(d, d, t[c]);
      }
    column_sums(part + 2 * NW * RP);
    __syncthreads();
    int good = 1;
    if (tid < r) {
      const float th1 = theta[0], thi = theta[tid];
      float gap = 3.0e38f, rho2 = 0.f;
#pragma unroll
      for (int w = 0; w < NW; ++w) rho2 += part[(2 * NW + w) * RP + tid];
      if (tid > 0) gap = fminf(gap, theta[tid - 1] - thi);
      if (tid < r - 1) gap = fminf(gap, thi - theta[tid + 1]);
      const float most = fmaxf(tol.eps_vec * gap, tol.floor_rel * th1);
      const bool res_ok = (int)(most >= 0.f) & (int)(rho2 <= most * most);
      // T and the rows left out are similar to sc * G: the traces agree to rounding; and nothing kept is among those rows
      const float trG = (float)((double)sc * sh.trace);
      const bool tr_ok = fabsf(sh.tr_t + sh.rest - trG) <= 1e-4f * fabsf(trG) && rest_keeps_result(sh.rest, trG, theta[r - 1]) &&
                         isfinite(thi) && isfinite(rho2);
      if (!res_ok) atomicOr(&sh.why, kWhyResidual);
      if (!tr_ok) atomicOr(&sh.why, kWhyTrace);
      good = res_ok && tr_ok;
    }
    ok = __syncthreads_and(good) && ok;
  }
  return ok;
}

// The eigensolve of user b; every thread of the CTA calls it and all leave together.
// With want_vs, a certified tridiagonal result also leaves V Sigma at the start of the dynamic
// shared memory ([D][rp], rp = r rounded up to 4, zero in the padding).
enum EigEnd { kEnded, kEndedVs, kOtherHalf };      // S and V written; V Sigma in shared memory too; the pair's other CTA does it
template <int D, int RP>
__device__ __forceinline__ EigEnd eig_user(int b, int half, bool& joined, const float* __restrict__ gpart, const int* gram_status,
                                         int parts, int splits, float* __restrict__ gsum, int r, int route, int sweep_cap,
                                         const TriTol& tol, bool want_vs, bool late_trigger, float* __restrict__ S,
                                         float* __restrict__ V, int* __restrict__ info,
                                         int* __restrict__ route_taken) {
  using C = TriCfg<D>;
  using L = TriSmem<D, RP>;
  constexpr int GX = C::GX, RT = C::RT, NT = C::NT, NW = C::NW, NCH = C::NCH, CW = C::CW, LD = C::LD, NE = RP / 32;
  extern __shared__ __align__(16) float smem[];
  __shared__ TriShared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane & (GX - 1), row0 = tid / GX;
  float* const theta = smem + L::TH;
  float* const part = smem + L::PART;
  joined = false;
  if (half != kAlone) {
    if (tid == 0) sh.verdict = 0;
    __syncwarp();
    cluster_arrive();
    cluster_wait();
  }
  pdl_wait();          // everything below reads what the Gram kernel wrote

  // ---- 1. G = sum of the slices' partial Grams, in a fixed order, in the registers' layout ---------
  // the summed matrix in global memory: a user's only partial as it is, else written below
  const float* gout = parts == 1 ? gpart + (size_t)b * D * D : gsum + (size_t)b * D * D;
  float acc[RT][NCH][4];
  {
    const float4* gp = reinterpret_cast<const float4*>(gpart + (size_t)b * parts * D * D);
    int lost = 0;                        // (gram_status is no __restrict__ pointer: its loads stay behind the wait)
    for (int s = tid; s < splits; s += NT) lost |= (gram_status[b * splits + s] != kGramStatusOk);
    // fp32 sums in slice order; the loads of SCN slices are issued before the first add: the
    // phase is bound by their latency
    constexpr int SCN = RT * NCH >= 16 ? 2 : RT * NCH >= 8 ? 3 : 8;
#pragma unroll
    for (int rr = 0; rr < RT; ++rr)
#pragma unroll
      for (int m = 0; m < NCH; ++m)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[rr][m][c] = 0.f;
    for (int s0 = 0; s0 < parts; s0 += SCN) {
      float4 v[SCN][RT][NCH];
#pragma unroll
      for (int s = 0; s < SCN; ++s)
#pragma unroll
        for (int rr = 0; rr < RT; ++rr)
#pragma unroll
          for (int m = 0; m < NCH; ++m)
            v[s][rr][m] = (s0 + s < parts) ? ld_dep(gp + (size_t)(s0 + s) * (D * D / 4) + (row0 + 32 * rr) * (D / 4) + GX * m + g)
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int s = 0; s < SCN; ++s)
#pragma unroll
        for (int rr = 0; rr < RT; ++rr)
#pragma unroll
          for (int m = 0; m < NCH; ++m) {
            acc[rr][m][0] += v[s][rr][m].x; acc[rr][m][1] += v[s][rr][m].y;
            acc[rr][m][2] += v[s][rr][m].z; acc[rr][m][3] += v[s][rr][m].w;
          }
    }
    float zero = 0.f;
#pragma unroll
    for (int rr = 0; rr < RT; ++rr)
#pragma unroll
      for (int m = 0; m < NCH; ++m) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          zero = fmaf(acc[rr][m][c], 0.f, zero);             // NaN where an entry is not finite
          if (D == 128) st_if(part + row0 + 32 * rr, acc[rr][m][c], CW * m + 4 * g + c == row0 + 32 * rr);
        }
        if (parts > 1)                                        // read back by the residual check and the fallback
          reinterpret_cast<float4*>(gsum + (size_t)b * D * D)[(row0 + 32 * rr) * (D / 4) + GX * m + g] =
              make_float4(acc[rr][m][0], acc[rr][m][1], acc[rr][m][2], acc[rr][m][3]);
      }
    // (d = 128: one store of these per row makes the steps' schedule worse, 149.8 -> 153.7 us for 8 x 4096 x 128.)
#pragma unroll
    for (int rr = 0; rr < (D == 128 ? 0 : RT); ++rr)
      st_if(part + row0 + 32 * rr, C::diagonal([&](int m, int c) { return acc[rr][m][c]; }, rr, row0), ((row0 & (CW - 1)) >> 2) == g);
    if (tid < 4) sh.flags[tid] = 0;
    if (tid == 0) sh.why = 0;
    if (__syncthreads_or(lost | (int)!(zero == 0.f))) {
      lost = __syncthreads_or(lost);
      const float qnan = __int_as_float(0x7fc00000);
      for (int e = tid; e < D * r; e += NT) V[(size_t)b * D * r + e] = qnan;
      for (int e = tid; e < r; e += NT) S[(size_t)b * r + e] = qnan;
      if (tid == 0 && info) info[b] = lost ? SOLAR_INFO_DEVICE_WAIT : SOLAR_INFO_NONFINITE;
      if (tid == 0 && route_taken) route_taken[b] = 0;
      return half == kFp64Half ? kOtherHalf : kEnded;
    }
  }
  float gmax = 0.f;
  {
    double tr = 0.0;
#pragma unroll
    for (int q = 0; q < D / 32; ++q) {
      const float d = part[lane + 32 * q];
      gmax = fmaxf(gmax, fabsf(d));
      tr += (double)d;
    }
    gmax = warp_max(gmax);
#pragma unroll
    for (int o = 16; o; o >>= 1) tr += __shfl_xor_sync(kFull, tr, o);
    if (tid == 0) sh.trace = tr;
  }
  // Power-of-two scale that brings the largest diagonal entry into [1, 2): everything below works
  // on sc * G (exact), and the eigenvalues are divided by sc at the end.  The thresholds of the chain are absolute and
  // the Sturm recurrence relies on the range, so it has to hold for every normal entry (the scale and 1 / scale are normal
  // to 2^+-126; with a limit of 2^+-100 entries from 2^116 on, or below 2^-113, sent every user through the fp64 chain).
  const float sc = gmax > 0.f ? __uint_as_float((unsigned)(127 - max(-126, min(126, log2_int(gmax)))) << 23) : 1.f;
  __syncthreads();

  if (route != kRouteFull && gmax > 0.f) {
    float* Vc = nullptr;
    int passes = 0, wide = 0;            // wide: the fp64 chain gave the result
    bool ok = false, not_mine = false;
    if (half != kFp64Half) {
      ok = tri_chain<float, D, RP>(acc, smem, sh, gout, sc, r, route == kRouteTridiag, tol, !late_trigger, half, not_mine, Vc, passes, tid);
      joined = half != kAlone;
      if (not_mine) return kOtherHalf;
    } else if (tid == 0) {
      sh.why = kWhyGap;
    }
    if (!ok && route != kRouteTridiag) {
      __syncthreads();
#pragma unroll
      for (int rr = 0; rr < RT; ++rr)
#pragma unroll
        for (int m = 0; m < NCH; ++m) ld4(gout + (row0 + 32 * rr) * D + CW * m + 4 * g, acc[rr][m]);
      wide = 1;
      ok = tri_chain<double, D, RP>(acc, smem, sh, gout, sc, r, false, tol, false, half, not_mine, Vc, passes, tid);
      if (not_mine) return kOtherHalf;
    }
    if (ok || route == kRouteTridiag) {
      if (late_trigger || wide) pdl_trigger();
      // singular values (non-increasing: a Rayleigh quotient may pass its neighbour by a rounding
      // error), sign gauge, output
      const int rp = (r + 3) & ~3;
      float sv[NE], sg[NE], carry = 3.0e38f;
#pragma unroll
      for (int h = 0; h < NE; ++h) {
        const int c = 32 * h + lane, j = c < r ? c : r - 1;
        float m = theta[j];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const float t = __shfl_up_sync(kFull, m, o);
          m = lane >= o ? fminf(m, t) : m;
        }
        m = fminf(m, carry);
        carry = __shfl_sync(kFull, m, 31);
        float best = -1.f, lv = 1.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
          const float v = part[(NW + w) * RP + c];
          lv = fabsf(v) > best ? v : lv;
          best = fmaxf(fabsf(v), best);
        }
        sg[h] = lv < 0.f ? -1.f : 1.f;
        sv[h] = sqrtf(fmaxf(m, 0.f) * pow2_scale(sc, 0.f));          // 1 / sc, exactly
        if (warp == 0 && c < r) S[(size_t)b * r + c] = sv[h];
      }
      float* vsig = smem;                            // over G: the residuals are done
      // Code that runs once costs some three cycles an instruction (fetch), so addresses run along by additions: with
      // the divisions of the projections' index arithmetic gone too, 32 x 1024 x 64, r = 16 34.8 -> 33.9 us per pass.
      constexpr int RB = 8 / NE;                     // rows read ahead of their stores, which are not reordered with loads
      float* to = V + ((size_t)b * D + warp) * r + lane;
      float* vs = vsig + warp * rp + lane;
#pragma unroll 1
      for (int n0 = warp; n0 < D; n0 += RB * NW) {
        const float* from = Vc + n0 * RP + lane;
        float v[RB][NE];
#pragma unroll
        for (int u = 0; u < RB; ++u)
#pragma unroll
          for (int h = 0; h < NE; ++h) v[u][h] = from[u * NW * RP + 32 * h] * sg[h];
#pragma unroll
        for (int u = 0; u < RB; ++u, to += NW * r, vs += NW * rp)
#pragma unroll
          for (int h = 0; h < NE; ++h) {
            const int c = 32 * h + lane;
            if (c < r) to[32 * h] = v[u][h];
            st_if(vs + 32 * h, c < r ? v[u][h] * sv[h] : 0.f, (int)want_vs & (int)(c < rp));
          }
      }
      if (tid == 0) {
        if (info) info[b] = ok ? 0 : SOLAR_INFO_NOT_CERTIFIED;
        if (route_taken) route_taken[b] = (wide ? kRouteFull | (kDetailWide << 8) : kRouteTridiag | (sh.rows << 8)) | (passes << 16) | (sh.why << 24);
      }
      return want_vs ? kEndedVs : kEnded;
    }
    __syncthreads();
  }
  if (half == kFp64Half && !(gmax > 0.f)) return kOtherHalf;

  // ---- last resort (or the caller's choice): Jacobi on the whole matrix ----------------------------
  for (int e = tid; e < D * D / 4; e += NT) {
    float4 t = reinterpret_cast<const float4*>(gout)[e];
    t.x *= sc; t.y *= sc; t.z *= sc; t.w *= sc;
    *reinterpret_cast<float4*>(smem + (e / (D / 4)) * LD + (e % (D / 4)) * 4) = t;
  }
  __syncthreads();
  const float thr_abs2 = (kTolAbs * gmax * sc) * (kTolAbs * gmax * sc);
  full_jacobi_route<D, NT>(smem, sh.flags, b, tid, r, sc, thr_abs2, tol.sweep_stop * tol.sweep_stop, sh.why,
                           sweep_cap, S, V, info, route_taken);
  return kEnded;
}

// ---- optional epilogue: the factor-token projections of Eq. 11 for this user ---------------
// Key_r = (V Sigma)^T W_K, Value_r = (V Sigma)^T W_V and the folded score operand
// T = scale * W_Q Key_r^T, written to the attention workspace in the layout and with the
// summation order of the stand-alone projection kernel, so that a forward pass which ends its
// eigensolver CTAs with this epilogue needs one launch less and gives the same bits.
struct FuseArgs {
  const void* Wq; const void* Wk; const void* Wv;
  float scale;
  char* ws;            // attention workspace (all users)
  AttnWs lay;
  int mode;            // 0: no epilogue; 1: weights are bf16; 2: weights are fp32
  int late_trigger;    // release the next kernel after the certificate instead of before the residuals
};

// Four consecutive elements of a weight matrix as fp32.
__device__ __forceinline__ float4 weight4(const void* __restrict__ W, int mode, int e4) {
  if (mode != 1) return ld_dep(static_cast<const float4*>(W) + e4);
  const uint2 u = ld_dep(static_cast<const uint2*>(W) + e4);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xffff0000u));
}

// vs_ready: V Sigma of this user already lies at sm[0 .. D * rp) (pitch rp = r rounded up to 4,
// zero in the padding), left there by the eigensolver; otherwise it is read back from S and V.
template <int D, int NT>
__device__ __forceinline__ void prepare_epilogue(float* __restrict__ sm, int b, int r, const float* __restrict__ S,
                                                 const float* __restrict__ V, const FuseArgs& fa, bool vs_ready,
                                                 int tid) {
  const int rp = (r + 3) & ~3;          // token pitch: rows of VS / KrT are read 4 at a time
  float* VS = sm;                       // [D][rp]  V Sigma (zero in the padding)
  float* KrT = VS + D * rp;             // [D][rp]  Key_r^T
  float* W0 = KrT + D * rp;             // [D][D]   W_K; later W_Q with row pitch D + 4
  float* W1 = W0 + D * D;               // [D][D]   W_V
  char* wsb = fa.ws + (size_t)b * fa.lay.per_user;
  const bool mma = D >= 64 && fa.mode == 1;
  if (!mma && fa.mode == 2) {
#pragma unroll 4
    for (int e = tid; e < D * D / 4; e += NT) {
      cp_async16(W0 + 4 * e, static_cast<const float*>(fa.Wk) + 4 * e);
      cp_async16(W1 + 4 * e, static_cast<const float*>(fa.Wv) + 4 * e);
    }
  }
  if (!vs_ready) {
    for (int e = tid; e < D * rp; e += NT) {
      const int k = e / rp, i = e % rp;
      // written earlier by this CTA: read through the L2, not the non-coherent path
      VS[e] = i < r ? __ldcg(V + ((size_t)b * D + k) * r + i) * __ldcg(S + (size_t)b * r + i) : 0.f;
    }
    if (mma) __syncthreads();
  }
  if constexpr (D >= 64) {
    if (mma) {
      // bf16 weights: the three products on the tensor cores
      pmma::Weights<D, NT, 3> w;
      w.load(fa.Wq, fa.Wk, fa.Wv, tid);
      pmma::project<D, NT, 3>(reinterpret_cast<unsigned char*>(sm), r, w, fa.scale,
                              pmma::Out{reinterpret_cast<__nv_bfloat16*>(wsb + fa.lay.tpk_off),
                                        reinterpret_cast<__nv_bfloat16*>(wsb + fa.lay.vpk_off), nullptr, nullptr, nullptr, nullptr}, tid);
      return;
    }
  }
  // FFMA form (fp32 weights, d = 32): the fp32 operands of the FFMA attention kernel, T [D][r] and
  // Value_r [r][D].  Bound by latency and issue of the CTA's four (eight) warps: Key_r and Value_r in one
  // loop over the rows of V Sigma, W_Q on its way meanwhile and read by rows, not transposed, results
  // straight from registers.  A pass over 16 x 5000 x 64 with r = 24 took 82.2 us with one product after the
  // other and the packed operands (which only the tensor-core kernels read) written beside the fp32 ones,
  // 76.9 now; one user of 256 x 32 with r = 8: 23.8 and 22.1.
  float* Tf = reinterpret_cast<float*>(wsb + fa.lay.tf_off);
  float* Vr = reinterpret_cast<float*>(wsb + fa.lay.vr_off);
  const int nt4 = rp / 4;               // groups of four tokens
  constexpr int CT = D == 32 ? 1 : 4;   // columns (rows of T) of a thread's tile: a small user still has work for the threads
  constexpr int NV = D * D / 4 / NT, LQ = D + 4;
  if (fa.mode == 1) {
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      reinterpret_cast<float4*>(W0)[tid + n * NT] = weight4(fa.Wk, 1, tid + n * NT);
      reinterpret_cast<float4*>(W1)[tid + n * NT] = weight4(fa.Wv, 1, tid + n * NT);
    }
  }
  float4 wq[NV];
#pragma unroll
  for (int n = 0; n < NV; ++n) wq[n] = weight4(fa.Wq, fa.mode, tid + n * NT);
  cp_async_wait_all();
  __syncthreads();
  // Key_r and Value_r: every output summed over k in ascending order
  for (int t = tid; t < nt4 * (D / CT); t += NT) {
    const int j0 = (t % (D / CT)) * CT, i0 = (t / (D / CT)) * 4;
    float ka[4][CT], va[4][CT];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < CT; ++c) ka[a][c] = va[a][c] = 0.f;
#pragma unroll 4
    for (int k = 0; k < D; ++k) {
      float v[4], wk[CT], wv[CT];
      ld4(VS + k * rp + i0, v);
      if constexpr (CT == 4) {
        ld4(W0 + k * D + j0, wk);
        ld4(W1 + k * D + j0, wv);
      } else {
        wk[0] = W0[k * D + j0];
        wv[0] = W1[k * D + j0];
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < CT; ++c) {
          ka[a][c] = fmaf(v[a], wk[c], ka[a][c]);
          va[a][c] = fmaf(v[a], wv[c], va[a][c]);
        }
    }
#pragma unroll
    for (int c = 0; c < CT; ++c)
      *reinterpret_cast<float4*>(KrT + (j0 + c) * rp + i0) = make_float4(ka[0][c], ka[1][c], ka[2][c], ka[3][c]);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      if (i0 + a >= r) continue;
      if constexpr (CT == 4) *reinterpret_cast<float4*>(Vr + (size_t)(i0 + a) * D + j0) = make_float4(va[a][0], va[a][1], va[a][2], va[a][3]);
      else Vr[(size_t)(i0 + a) * D + j0] = va[a][0];
    }
  }
  __syncthreads();
#pragma unroll
  for (int n = 0; n < NV; ++n) {
    const int e = tid + n * NT;
    *reinterpret_cast<float4*>(W0 + (e / (D / 4)) * LQ + (e % (D / 4)) * 4) = wq[n];
  }
  __syncthreads();
  // T[k][i] = scale * sum_j Wq[k][j] Key_r[i][j]: rows k0 + (D / CT) x, four tokens i
  for (int t = tid; t < nt4 * (D / CT); t += NT) {
    const int i0 = (t % nt4) * 4, k0 = t / nt4;
    float acc[CT][4];
#pragma unroll
    for (int x = 0; x < CT; ++x)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[x][c] = 0.f;
#pragma unroll 2
    for (int j = 0; j < D; j += 4) {
      float w[CT][4], kr[4][4];
#pragma unroll
      for (int x = 0; x < CT; ++x) ld4(W0 + (k0 + x * (D / CT)) * LQ + j, w[x]);
#pragma unroll
      for (int u = 0; u < 4; ++u) ld4(KrT + (j + u) * rp + i0, kr[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int x = 0; x < CT; ++x)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[x][c] = fmaf(w[x][u], kr[u][c], acc[x][c]);
    }
#pragma unroll
    for (int x = 0; x < CT; ++x)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (i0 + c < r) Tf[(size_t)(k0 + x * (D / CT)) * r + i0 + c] = acc[x][c] * fa.scale;
  }
}

template <int D, int RP>
__global__ void __launch_bounds__(TriCfg<D>::NT, TriCfg<D>::ctas(RP))
eig_tridiag_kernel(const float* __restrict__ gpart, const int* gram_status, int parts, int splits,
                   float* __restrict__ gsum, int r, int route, int sweep_cap, TriTol tol,
                   float* __restrict__ S, float* __restrict__ V, int* __restrict__ info,
                   int* __restrict__ route_taken, FuseArgs fa, int pairs) {
  const bool two = RP > 32 && pairs;
  const int b = two ? blockIdx.x >> 1 : blockIdx.x, half = !two ? kAlone : (blockIdx.x & 1) ? kFp64Half : kFp32Half;
  bool joined;                          // this CTA has arrived at the pair's second barrier and not yet waited
  const EigEnd end = eig_user<D, RP>(b, half, joined, gpart, gram_status, parts, splits, gsum, r, route, sweep_cap, tol, fa.mode != 0,
                                     fa.late_trigger != 0, S, V, info, route_taken);
  if (fa.mode != 0 && end != kOtherHalf) {
    extern __shared__ __align__(16) float smem[];
    __syncthreads();                    // S and V of this user are written (and visible to the CTA)
    prepare_epilogue<D, TriCfg<D>::NT>(smem, b, r, S, V, fa, end == kEndedVs, threadIdx.x);
  }
  __syncwarp();
  if (RP > 32 && joined) cluster_wait();
}

template <int D, int RP>
cudaError_t launch_tri(int B, int r, int route, int sweep_cap, TriTol tol, const float* gpart,
                       const int* gram_status, int parts, int splits, float* gsum, float* S, float* V, int* info,
                       int* route_taken, const FuseArgs& fa, bool pairs, cudaStream_t st) {
  using L = TriSmem<D, RP>;
  static bool limits_set[kMaxDevicesCached] = {};
  const cudaError_t e = set_kernel_limits(reinterpret_cast<const void*>(&eig_tridiag_kernel<D, RP>), L::BYTES,
                                          limits_set);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(pairs ? 2 * B : B); cfg.blockDim = dim3(TriCfg<D>::NT); cfg.dynamicSmemBytes = L::BYTES; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = pairs ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, eig_tridiag_kernel<D, RP>, gpart, gram_status, parts, splits, gsum, r, route, sweep_cap, tol, S, V,
                            info, route_taken, fa, (int)pairs);
}

}  // namespace

cudaError_t launch_eig_tridiag(int B, int d, int r, solar_dtype_t dt, int route, int sweep_cap,
                               const float* gpart, const int* gram_status, int parts, int splits, float* gsum,
                               float* S, float* V, int* info, int* route_taken, const EigFuse* fuse,
                               cudaStream_t st) {
  FuseArgs fa = {};
  if (fuse != nullptr) {
    fa.Wq = fuse->Wq; fa.Wk = fuse->Wk; fa.Wv = fuse->Wv; fa.scale = fuse->scale;
    fa.ws = fuse->attn_ws; fa.lay = attn_ws_layout(d, r);
    fa.mode = (dt == SOLAR_BF16) ? 1 : 2;
    fa.late_trigger = slice_limit() > 0;
  }
  TriTol tol;
  if (dt == SOLAR_BF16) {
    tol.eps_vec = 1e-3f; tol.floor_rel = 64.f * kUnit; tol.ortho = 4e-6f; tol.sweep_stop = 1e-3f;
    tol.gap_min = 4.f * kUnit / 1e-2f;      // angle 1e-2: outputs are rounded to bf16 (2^-9)
    tol.stop_trace = 1.9073486e-06f; tol.stop_couple = 2.3841858e-07f;     // 2^-19, 2^-22
  } else {
    tol.eps_vec = 1e-5f; tol.floor_rel = 32.f * kUnit; tol.ortho = 2e-6f; tol.sweep_stop = 1e-5f;
    tol.gap_min = 4.f * kUnit / 1e-3f;
    tol.stop_trace = 1.1920929e-07f; tol.stop_couple = 2.9802322e-08f;     // 2^-23, 2^-25
  }
  const bool wide = r > 32;
  // Two CTAs per user where the fp64 chain is likely (gaps among 33 and more kept eigenvalues), half of the
  // SMs would stay idle anyway and no slice limit says that other requests use them.  For smaller ranks
  // the second chain is hardly ever needed, and it costs: 16 x 10240 x 64 with r = 32 51.8 -> 52.8 us per
  // pass, one user of 256 x 32 with r = 8 22.1 -> 24.6.
  const bool pairs = route == SOLAR_ROUTE_AUTO && wide && B <= kNumSMs / 2 && slice_limit() == 0;
  switch (d) {
    case 32:
      return launch_tri<32, 32>(B, r, route, sweep_cap, tol, gpart, gram_status, parts, splits, gsum, S, V, info, route_taken, fa, pairs, st);
    case 64:
      return wide ? launch_tri<64, 64>(B, r, route, sweep_cap, tol, gpart, gram_status, parts, splits, gsum, S, V, info, route_taken, fa, pairs, st)
                  : launch_tri<64, 32>(B, r, route, sweep_cap, tol, gpart, gram_status, parts, splits, gsum, S, V, info, route_taken, fa, pairs, st);
    case 128:
      return wide ? launch_tri<128, 64>(B, r, route, sweep_cap, tol, gpart, gram_status, parts, splits, gsum, S, V, info, route_taken, fa, pairs, st)
                  : launch_tri<128, 32>(B, r, route, sweep_cap, tol, gpart, gram_status, parts, splits, gsum, S, V, info, route_taken, fa, pairs, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace solar
