// Softmax attention over the N history positions evaluated through the rank-r factors
// (bf16 storage, d = 64 or 128, r = 16, 32 or 64):
//   O = softmax_N( scale * (C W_Q W_K^T V) (U Sigma)^T ) (U Sigma) (V^T W_V)
// On a history of rank <= r this IS the softmax attention of Eq. 6-7 (H = U Sigma V^T makes
// Key = U Sigma V^T W_K and Value = U Sigma V^T W_V), at O(N M r) instead of O(N M d); it
// is not the paper's SVD-Attention operator, which removes U (Eq. 10) and takes the softmax
// over the r factor tokens.
//
// One CTA per 128 candidates of one user, flash-attention style, everything on chip.  Warps 0-3 own a
// candidate row per thread, warp 4 issues the GEMMs, warp 5 streams U Sigma through a ring of TMA stages:
//   Q' [128 x r] = C A1 (A1 = scale log2(e) W_Q W_K^T V, hi + lo bf16 halves), tcgen05.mma
//   for each tile of 128 positions:
//     S [128 x 128] = Q' US_tile^T      tcgen05.mma, US tile as a K-major operand; issued as soon as the
//                                       row warps hold the tile before in registers
//     p = 2^(s - m), l += sum p         registers; P as bf16 pairs back to tensor memory
//     Y [128 x r] += P US_tile          tcgen05.mma, P as the A operand from tensor memory, the SAME tile as an
//                                       MN-major operand; accumulates in tensor memory and overlaps the
//                                       next tile's exponentials
//   O [128 x d] = (Y / l) B1  (B1 = V^T W_V, hi/lo halves), tcgen05.mma, TMA store.
// Where the candidates do not fill the GPU, the positions are split as well (flash_split): a CTA then leaves
// Y, l and m of its range, and the one that arrives last adds up the ranges in their order.  128 candidates,
// 32768 positions, d = 64, r = 32: 281 us a call with one CTA, 35 now; 8 x 512 candidates,
// 10240 positions: 98 and 44 in the three ranges that solar_workspace_bytes has room for.
// The reference m of a row is the maximum of its first tile and is raised (Y and l rescaled) only when a
// score passes it by more than 2^8: any m gives the same quotient, and bf16 keeps its relative accuracy
// at every magnitude.  The N x M score matrix never exists outside tensor memory.  Every wait is bounded;
// if one runs out the tile's output rows are written as NaN.
//
// Bound by the row warps: 128 exponentials a tile and thread (the special-function units give 16 per
// clock and SM: 72 us for 16 x 2048 x 10240) and as many issue slots for the rest, with two warps per
// scheduler.  So additions go in pairs, nothing of Y passes through registers, and no wait stands between
// the scores and their exponentials (the one for the P before comes after them).
// Measured at that size: 164 us with one chain per CTA (GEMM, softmax, GEMM, rescale of Y in registers,
// a CTA barrier each), 133 us now.  Evaluating every 8th / 4th / 2nd exponential by a polynomial on the
// FMA pipes was slower (+5 / +12 / +45 us): the issue slots are as scarce as the special-function units.
#include "sm100_ptx.cuh"
#include "solar_internal.cuh"

namespace solar {

namespace {

constexpr int kRows = 128;                 // candidates per CTA = accumulator lanes
constexpr int kPos = 128;                  // history positions per tile
constexpr int kBox = kRows * 128;          // bytes of a [128 rows][128 B] swizzled box
constexpr int kMmaWarp = 4, kTmaWarp = 5, kThreads = 192, kRowThreads = 128, kRowWarps = 4;
constexpr int kStages = 3;                 // U Sigma tiles in flight: one being read by Y, one by the next S, one on its way
constexpr float kRaise = 8.f;              // log2 by which a score may pass the row's reference
constexpr int kErrLoad = 0x31, kErrQ = 0x32, kErrTile = 0x33, kErrS = 0x34, kErrY = 0x35, kErrO = 0x36, kErrP = 0x37;

template <int D, int R> struct FlashCfg {
  static constexpr int KB = D / 64;                   // 64-wide K boxes of C
  static constexpr int RB = R * 2;                    // bytes of one US row = swizzle span of its tile
  static constexpr uint32_t US_LAYOUT = (R == 64) ? 2u : (R == 32) ? 4u : 6u;   // descriptor swizzle code
  static constexpr int C_BYTES = KB * kBox;           // candidate tile; later the output tile
  static constexpr int T_BYTES = 2 * KB * R * 128;    // A1^T hi/lo: [2][KB][R rows][128 B]
  static constexpr int V_BYTES = 2 * D * 128;         // B1^T hi/lo: [2][D rows][128 B] (K = token)
  static constexpr int QH = kRows * RB;               // one half of Q'
  static constexpr int Q_BYTES = 2 * QH;              // Q' hi/lo, later y hi/lo: [2][128][RB]
  static constexpr int US_TILE = kPos * RB;           // one tile of U Sigma
  static constexpr size_t SMEM = (size_t)T_BYTES + V_BYTES + Q_BYTES + C_BYTES + kStages * US_TILE + 1024;
  // tensor-memory columns: Y; S, which also takes Q' before the first scores and O after the last; P as
  // bf16 pairs
  static constexpr int COL_Y = 0, COL_S = 64, COL_P = 192, TMEM_COLS = 256;
};

// Offset of 16-byte chunk c of a row in a K-major tile whose rows are one swizzle span of R bf16.
template <int R> __device__ __forceinline__ uint32_t swz_span(int row, int c) {
  return R == 64 ? ptx::swz128(row, c) : R == 32 ? ptx::swz64(row, c) : ptx::swz32(row, c);
}

// Writes R fp32 values of this thread's row as bf16 high and low halves into two swizzled
// K-major tiles of R-wide rows (hi at `dst`, lo behind it).
template <int R>
__device__ __forceinline__ void store_hi_lo(uint8_t* dst, int row, const float (&x)[R]) {
#pragma unroll
  for (int c = 0; c < R / 8; ++c) {
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float a = x[8 * c + 2 * q], b = x[8 * c + 2 * q + 1];
      const float ha = __bfloat162float(__float2bfloat16_rn(a)), hb = __bfloat162float(__float2bfloat16_rn(b));
      hi[q] = ptx::pack_bf16(ha, hb);
      lo[q] = ptx::pack_bf16(a - ha, b - hb);
    }
    *reinterpret_cast<uint4*>(dst + swz_span<R>(row, c)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(dst + kRows * R * 2 + swz_span<R>(row, c)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

// Loads this thread's row of a tensor-memory block of R (<= 64) fp32 columns.
template <int R>
__device__ __forceinline__ void tmem_row(uint32_t taddr, float (&x)[R]) {
  uint32_t v[32];
  ptx::tmem_ld_32x32(taddr, v);
  ptx::tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < (R < 32 ? R : 32); ++i) x[i] = __uint_as_float(v[i]);
  if constexpr (R > 32) {
    ptx::tmem_ld_32x32(taddr + 32, v);
    ptx::tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < R - 32; ++i) x[32 + i] = __uint_as_float(v[i]);
  }
}

template <int D, int R>
__global__ void __launch_bounds__(kThreads, 2)
flash_factored_kernel(const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmO,
                      const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmV,
                      const __grid_constant__ CUtensorMap tmUS, int N, int M, __nv_bfloat16* __restrict__ O,
                      int tiles_per_range, float* __restrict__ part, int* __restrict__ counters) {
  using Cfg = FlashCfg<D, R>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sT = base;                         // [2][KB][R][128 B]
  uint8_t* sV = sT + Cfg::T_BYTES;            // [2][D][128 B]
  uint8_t* sQ = sV + Cfg::V_BYTES;            // [2][128][RB]
  uint8_t* sC = sQ + Cfg::Q_BYTES;            // [KB][128][128 B]  candidate tile first, output tile last
  uint8_t* sUS = sC + Cfg::C_BYTES;           // [kStages][128][RB]
  __shared__ __align__(8) uint64_t bar_load, bar_q, bar_qs, bar_s, bar_sf, bar_p, bar_y, bar_o, us_full[kStages], us_free[kStages];
  __shared__ uint32_t s_tmem;
  __shared__ int s_err, s_last;

  const int b = blockIdx.y, m0 = blockIdx.x * kRows;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ranges = gridDim.z, t0 = blockIdx.z * tiles_per_range;     // this CTA's tiles: t0 ..
  const int ntiles = min((N + kPos - 1) / kPos - t0, tiles_per_range), p0 = t0 * kPos;

  if (tid == 0) {
    s_err = 0; s_last = 1;
    ptx::mbar_init(&bar_load, 1); ptx::mbar_init(&bar_q, 1); ptx::mbar_init(&bar_qs, kRowWarps);
    ptx::mbar_init(&bar_s, 1); ptx::mbar_init(&bar_sf, kRowWarps); ptx::mbar_init(&bar_p, kRowWarps);
    ptx::mbar_init(&bar_y, 1); ptx::mbar_init(&bar_o, 1);
    for (int i = 0; i < kStages; ++i) { ptx::mbar_init(&us_full[i], 1); ptx::mbar_init(&us_free[i], 1); }
    ptx::fence_mbar_init();
    ptx::prefetch_tensormap(&tmC); ptx::prefetch_tensormap(&tmT); ptx::prefetch_tensormap(&tmV);
    ptx::prefetch_tensormap(&tmUS); ptx::prefetch_tensormap(&tmO);
  }
  if (warp == kMmaWarp) ptx::tmem_alloc(&s_tmem, Cfg::TMEM_COLS);
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
  const uint32_t tm_y = s_tmem + Cfg::COL_Y, tm_s = s_tmem + Cfg::COL_S, tm_p = s_tmem + Cfg::COL_P;
  volatile int* err = &s_err;

  if (warp == kTmaWarp) {
    if (lane == 0) {
      ptx::mbar_arrive_expect_tx(&bar_load, Cfg::C_BYTES + Cfg::T_BYTES + Cfg::V_BYTES);
#pragma unroll
      for (int x = 0; x < Cfg::KB; ++x) ptx::tma_load_3d(sC + x * kBox, &tmC, &bar_load, x * 64, m0, b);
      pdl_wait();        // the packed operands and U Sigma come from earlier kernels on the stream
#pragma unroll
      for (int x = 0; x < Cfg::KB; ++x)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          ptx::tma_load_3d(sT + (h * Cfg::KB + x) * (R * 128), &tmT, &bar_load, x * 64, h * kTokenSlots, b);
#pragma unroll
      for (int h = 0; h < 2; ++h) ptx::tma_load_3d(sV + h * (D * 128), &tmV, &bar_load, 0, h * D, b);
      int issued = 0;
      for (int t = 0; t < ntiles; ++t) {
        const int st = t % kStages;
        if (t >= kStages && !ptx::mbar_wait(&us_free[st], (t / kStages - 1) & 1, err, kErrTile)) break;
        ptx::mbar_arrive_expect_tx(&us_full[st], Cfg::US_TILE);
        ptx::tma_load_3d(sUS + st * Cfg::US_TILE, &tmUS, &us_full[st], 0, p0 + t * kPos, b);
        issued = t + 1;
      }
      // the copies still in flight land before the CTA leaves, whatever happened
      int dummy = 0;
      ptx::mbar_wait(&bar_load, 0, &dummy, 0);
      for (int t = max(0, issued - kStages); t < issued; ++t) {
        int d2 = 0;
        ptx::mbar_wait(&us_full[t % kStages], (t / kStages) & 1, &d2, 0);
      }
    }
  } else if (warp == kMmaWarp) {
    if (lane == 0) {
      // ---- Q' = C A1_hi + C A1_lo : M = 128, N = R, K = D (over the scores' columns) -------------
      bool ok = ptx::mbar_wait(&bar_load, 0, err, kErrLoad);
      if (ok) {
        ptx::tc_fence_after_sync();
        const uint32_t idesc = ptx::umma_idesc_bf16(kRows, R, false, false);
        bool acc = false;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint32_t a = ptx::smem_u32(sC) + (kk / 4) * kBox + (kk % 4) * 32;
            const uint32_t t = ptx::smem_u32(sT) + (h * Cfg::KB + kk / 4) * (R * 128) + (kk % 4) * 32;
            ptx::umma_bf16_ss(tm_s, ptx::umma_smem_desc(a, 0, 1024), ptx::umma_smem_desc(t, 0, 1024), idesc, acc);
            acc = true;
          }
      }
      ptx::umma_commit(&bar_q);
      ok = ok && ptx::mbar_wait(&bar_qs, 0, err, kErrQ);

      const uint32_t idesc_s = ptx::umma_idesc_bf16(kRows, kPos, false, false);   // S = Q' US^T
      const uint32_t idesc_y = ptx::umma_idesc_bf16(kRows, R, false, true);       // Y += P US (US MN-major)
      auto scores = [&](int t) {
        const uint32_t us = ptx::smem_u32(sUS + (t % kStages) * Cfg::US_TILE);
        if (!ptx::mbar_wait(&us_full[t % kStages], (t / kStages) & 1, err, kErrTile)) return false;
        ptx::tc_fence_after_sync();
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int kk = 0; kk < R / 16; ++kk) {
            // A: Q' half h.  B: the tile's rows are the K-major operand rows.  Both have rows of RB bytes
            // (one candidate, one position), swizzle span RB, 8-row atoms of 8*RB bytes.
            const uint64_t a = ptx::umma_smem_desc_sw(ptx::smem_u32(sQ) + h * Cfg::QH + kk * 32, 0, 8 * Cfg::RB, Cfg::US_LAYOUT);
            const uint64_t bd = ptx::umma_smem_desc_sw(us + kk * 32, 0, 8 * Cfg::RB, Cfg::US_LAYOUT);
            ptx::umma_bf16_ss(tm_s, a, bd, idesc_s, (h | kk) != 0);
          }
        ptx::umma_commit(&bar_s);
        return true;
      };
      ok = ok && scores(0);
      for (int t = 0; ok && t < ntiles; ++t) {
        if (t + 1 < ntiles) {
          ok = ptx::mbar_wait(&bar_sf, t & 1, err, kErrS);       // the row warps hold tile t's scores
          ok = ok && scores(t + 1);
        }
        ok = ok && ptx::mbar_wait(&bar_p, t & 1, err, kErrP);
        if (!ok) break;
        ptx::tc_fence_after_sync();
        const uint32_t us = ptx::smem_u32(sUS + (t % kStages) * Cfg::US_TILE);
#pragma unroll
        for (int kk = 0; kk < kPos / 16; ++kk) {
          // A: P from tensor memory, 16 positions = 8 columns of pairs.  B: the same U Sigma tile read
          // MN-major: 16 positions = two groups of 8 rows (8*RB bytes apart); its R columns are one MN block.
          const uint64_t bd = ptx::umma_smem_desc_sw(us + kk * 16 * Cfg::RB, 0, 8 * Cfg::RB, Cfg::US_LAYOUT);
          ptx::umma_bf16_ts(tm_y, tm_p + kk * 8, bd, idesc_y, (t | kk) != 0);
        }
        ptx::umma_commit(&us_free[t % kStages]);
        ptx::umma_commit(&bar_y);
      }
      // ---- O = (y / l) B1 : M = 128, N = D, K = R, hi*hi + hi*lo + lo*hi ---------------------
      ok = ok && ptx::mbar_wait(&bar_p, ntiles & 1, err, kErrP);
      if (ok && *(volatile int*)&s_last) {
        ptx::tc_fence_after_sync();
        const uint32_t idesc = ptx::umma_idesc_bf16(kRows, D, false, false);
        bool acc = false;
#pragma unroll
        for (int term = 0; term < 3; ++term) {
          const uint32_t ya = ptx::smem_u32(sQ) + (term == 2 ? Cfg::QH : 0);
          const uint32_t vb = ptx::smem_u32(sV) + (term == 1 ? D * 128 : 0);
#pragma unroll
          for (int kk = 0; kk < R / 16; ++kk) {
            ptx::umma_bf16_ss(tm_s, ptx::umma_smem_desc_sw(ya + kk * 32, 0, 8 * Cfg::RB, Cfg::US_LAYOUT),
                              ptx::umma_smem_desc(vb + kk * 32, 0, 1024), idesc, acc);
            acc = true;
          }
        }
      }
      ptx::umma_commit(&bar_o);                      // everything issued so far has completed when it arrives
    }
  } else {
    // ---- row warps -------------------------------------------------------------------------
    ptx::mbar_wait(&bar_q, 0, err, kErrQ);
    __syncwarp();
    ptx::tc_fence_after_sync();
    {
      float q[R];
      tmem_row<R>(tm_s + lane_base, q);
      store_hi_lo<R>(sQ, tid, q);
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before_sync();
    ptx::mbar_arrive_warp(&bar_qs, lane);

    // (after a lost wait every thread still walks through all the tiles, but the waits return at once)
    float m_ref = 0.f, l_run = 0.f;
    for (int t = 0; t < ntiles; ++t) {
      ptx::mbar_wait(&bar_s, t & 1, err, kErrS);
      __syncwarp();
      ptx::tc_fence_after_sync();
      float s[kPos];                                 // this thread's 128 scores, already in log2 units
      {
        uint32_t v0[32], v1[32], v2[32], v3[32];
        ptx::tmem_ld_32x32(tm_s + lane_base, v0);
        ptx::tmem_ld_32x32(tm_s + lane_base + 32, v1);
        ptx::tmem_ld_32x32(tm_s + lane_base + 64, v2);
        ptx::tmem_ld_32x32(tm_s + lane_base + 96, v3);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          s[i] = __uint_as_float(v0[i]);      s[32 + i] = __uint_as_float(v1[i]);
          s[64 + i] = __uint_as_float(v2[i]); s[96 + i] = __uint_as_float(v3[i]);
        }
      }
      ptx::tc_fence_before_sync();
      ptx::mbar_arrive_warp(&bar_sf, lane);          // the next tile's scores may be formed
      const int valid = N - p0 - t * kPos;           // positions past N hold zero-filled rows
      if (valid < kPos) {
#pragma unroll
        for (int j = 0; j < kPos; ++j) s[j] = (j < valid) ? s[j] : -INFINITY;
      }
      float mx[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) mx[q] = s[q];
#pragma unroll
      for (int j = 8; j < kPos; j += 16)
#pragma unroll
        for (int q = 0; q < 8; ++q) mx[q] = (j + 8 < kPos) ? fmaxf(fmaxf(mx[q], s[j + q]), s[j + 8 + q]) : fmaxf(mx[q], s[j + q]);
      const float m_tile = fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])),
                                 fmaxf(fmaxf(mx[4], mx[5]), fmaxf(mx[6], mx[7])));
      if (t == 0) m_ref = m_tile;
      if (__any_sync(0xffffffffu, m_tile > m_ref + kRaise)) {
        // rare: raise the reference of the rows that need it; once Y is up to date nobody else touches this
        // thread's row of it
        ptx::mbar_wait(&bar_y, (t - 1) & 1, err, kErrY);
        const float m_new = fmaxf(m_ref, m_tile), alpha = ptx::fast_exp2(m_ref - m_new);
        m_ref = m_new;
        l_run *= alpha;
        __syncwarp();
        ptx::tc_fence_after_sync();
#pragma unroll
        for (int c0 = 0; c0 < R; c0 += 16) {
          uint32_t v[16];
          ptx::tmem_ld_32x16(tm_y + lane_base + c0, v);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) * alpha);
          ptx::tmem_st_32x16(tm_y + lane_base + c0, v);
        }
        ptx::tmem_st_wait();
      }
      // 2^(s - m) in pairs, packed to bf16 as they come; masked positions: 2^-inf = 0
      float2 sum2[4];
      const float2 nm2 = make_float2(-m_ref, -m_ref);
#pragma unroll
      for (int q = 0; q < 4; ++q) sum2[q] = make_float2(0.f, 0.f);
      uint32_t w[kPos / 2];
#pragma unroll
      for (int j = 0; j < kPos; j += 2) {
        const float2 x = ptx::add2(make_float2(s[j], s[j + 1]), nm2);
        const float2 e = make_float2(ptx::fast_exp2(x.x), ptx::fast_exp2(x.y));
        sum2[(j / 2) % 4] = ptx::add2(sum2[(j / 2) % 4], e);
        w[j / 2] = ptx::pack_bf16(e.x, e.y);
      }
      l_run += ((sum2[0].x + sum2[0].y) + (sum2[1].x + sum2[1].y)) + ((sum2[2].x + sum2[2].y) + (sum2[3].x + sum2[3].y));
      if (t > 0) ptx::mbar_wait(&bar_y, (t - 1) & 1, err, kErrY);      // the P before has been read
      __syncwarp();
      ptx::tc_fence_after_sync();
#pragma unroll
      for (int c = 0; c < kPos / 2; c += 16) {
        uint32_t v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = w[c + i];
        ptx::tmem_st_32x16(tm_p + lane_base + c, v);
      }
      ptx::tmem_st_wait();
      ptx::tc_fence_before_sync();
      ptx::mbar_arrive_warp(&bar_p, lane);
    }
    pdl_trigger();

    ptx::mbar_wait(&bar_y, (ntiles - 1) & 1, err, kErrY);
    __syncwarp();
    ptx::tc_fence_after_sync();
    {
      float y[R];
      tmem_row<R>(tm_y + lane_base, y);
      if (ranges > 1) {
        // ---- the ranges' sums: whoever comes last adds them up, in their order ----------------------
        pdl_wait();                                  // the counters were set by the kernel before
        const size_t item = (size_t)b * gridDim.x + blockIdx.x;
        float* mine = part + (item * ranges + blockIdx.z) * (R + 2) * kRows + tid;
        const float bad = *err != 0 ? __int_as_float(0x7fc00000) : 0.f;
#pragma unroll
        for (int i = 0; i < R; ++i) mine[i * kRows] = y[i];
        mine[R * kRows] = l_run + bad;               // after a lost wait the rows come out as NaN
        mine[(R + 1) * kRows] = m_ref;
        __threadfence();
        asm volatile("bar.sync 1, %0;" ::"n"(kRowThreads) : "memory");
        if (tid == 0) s_last = atomicAdd(counters + item, 1) == ranges - 1;
        asm volatile("bar.sync 1, %0;" ::"n"(kRowThreads) : "memory");
        if (s_last) {
          __threadfence();
          const float* all = part + item * ranges * (R + 2) * kRows + tid;
          float m = -INFINITY;
#pragma unroll 8
          for (int z = 0; z < ranges; ++z) m = fmaxf(m, __ldcg(all + ((size_t)z * (R + 2) + R + 1) * kRows));
          l_run = 0.f;
#pragma unroll
          for (int i = 0; i < R; ++i) y[i] = 0.f;
#pragma unroll 1
          for (int z = 0; z < ranges; ++z) {
            const float* from = all + (size_t)z * (R + 2) * kRows;
            const float f = ptx::fast_exp2(__ldcg(from + (R + 1) * kRows) - m);
            l_run = fmaf(f, __ldcg(from + R * kRows), l_run);
#pragma unroll
            for (int i = 0; i < R; ++i) y[i] = fmaf(f, __ldcg(from + i * kRows), y[i]);
          }
        }
      }
      const float inv = 1.f / l_run;
#pragma unroll
      for (int i = 0; i < R; ++i) y[i] *= inv;
      store_hi_lo<R>(sQ, tid, y);
    }
    ptx::fence_proxy_async_smem();
    ptx::tc_fence_before_sync();
    ptx::mbar_arrive_warp(&bar_p, lane);
    ptx::mbar_wait(&bar_o, 0, err, kErrO);
    __syncwarp();
    ptx::tc_fence_after_sync();
#pragma unroll
    for (int c0 = 0; c0 < D; c0 += 32) {
      uint32_t v[32];
      ptx::tmem_ld_32x32(tm_s + lane_base + c0, v);
      ptx::tmem_ld_wait();
      uint8_t* box = sC + (c0 / 64) * kBox;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint4 w = make_uint4(ptx::pack_bf16(__uint_as_float(v[8 * c + 0]), __uint_as_float(v[8 * c + 1])),
                                   ptx::pack_bf16(__uint_as_float(v[8 * c + 2]), __uint_as_float(v[8 * c + 3])),
                                   ptx::pack_bf16(__uint_as_float(v[8 * c + 4]), __uint_as_float(v[8 * c + 5])),
                                   ptx::pack_bf16(__uint_as_float(v[8 * c + 6]), __uint_as_float(v[8 * c + 7])));
        *reinterpret_cast<uint4*>(box + ptx::swz128(tid, (c0 % 64) / 8 + c)) = w;
      }
    }
    ptx::fence_proxy_async_smem();
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (!s_last) {
  } else if (s_err == 0) {
    if (tid == 0) {
#pragma unroll
      for (int x = 0; x < Cfg::KB; ++x) ptx::tma_store_3d(&tmO, sC + x * kBox, x * 64, m0, b);
      ptx::tma_store_commit();
      ptx::tma_store_wait_read();
    }
  } else if (tid < kRowThreads && m0 + tid < M) {
    uint4* dst = reinterpret_cast<uint4*>(O + ((size_t)b * M + m0 + tid) * D);
    const uint4 qnan = make_uint4(0x7fc07fc0u, 0x7fc07fc0u, 0x7fc07fc0u, 0x7fc07fc0u);
#pragma unroll
    for (int c = 0; c < D / 8; ++c) dst[c] = qnan;
  }
  if (warp == kMmaWarp) {
    if (s_err != 0) {                                // a wait ran out: the GEMMs in flight end first (bounded)
      int dummy = 0;
      ptx::mbar_wait(&bar_o, 0, &dummy, 0);
      __syncwarp();
    }
    ptx::tmem_dealloc(s_tmem, Cfg::TMEM_COLS);
  }
}

template <int D, int R>
cudaError_t launch_dr(int B, int M, int N, const void* C, const void* US, void* O, char* ws,
                      const AttnWs& lay, const FlashSplit& split, cudaStream_t st) {
  using Cfg = FlashCfg<D, R>;
  CUtensorMap tmC, tmO, tmT, tmV, tmUS;
  const uint64_t pu = lay.per_user;
  bool ok = encode_tmap_bf16_3d(&tmC, C, D, (uint64_t)M, (uint64_t)B, (uint64_t)D * 2, (uint64_t)M * D * 2, 64, kRows);
  ok = ok && encode_tmap_bf16_3d(&tmO, O, D, (uint64_t)M, (uint64_t)B, (uint64_t)D * 2, (uint64_t)M * D * 2, 64, kRows);
  ok = ok && encode_tmap_bf16_3d(&tmT, ws + lay.tpk_off, D, 2 * kTokenSlots, (uint64_t)B, (uint64_t)D * 2, pu, 64, R);
  ok = ok && encode_tmap_bf16_3d(&tmV, ws + lay.vpk_off, kTokenSlots, 2 * D, (uint64_t)B, kTokenSlots * 2, pu,
                                 kTokenSlots, D);
  ok = ok && encode_tmap_bf16_3d_sw(&tmUS, US, R, (uint64_t)N, (uint64_t)B, (uint64_t)R * 2, (uint64_t)N * R * 2, R,
                                    kPos, Cfg::RB);
  if (!ok) return cudaErrorInvalidValue;
  static bool limits_set[kMaxDevicesCached] = {};
  const cudaError_t e = set_kernel_limits(reinterpret_cast<const void*>(&flash_factored_kernel<D, R>), Cfg::SMEM,
                                          limits_set);
  if (e != cudaSuccess) return e;
  const dim3 grid((M + kRows - 1) / kRows, B, split.ranges), block(kThreads);
  return launch_pdl(flash_factored_kernel<D, R>, grid, block, Cfg::SMEM, st, tmC, tmO, tmT, tmV, tmUS, N, M,
                    static_cast<__nv_bfloat16*>(O), split.tiles_per_range, reinterpret_cast<float*>(ws + split.part_off),
                    reinterpret_cast<int*>(ws + split.counter_off));
}

}  // namespace

bool flash_factored_supported(int d, int r, solar_dtype_t dt) {
  return dt == SOLAR_BF16 && (d == 64 || d == 128) && (r == 16 || r == 32 || r == 64);
}

// Few candidates: the positions of 128 candidates are split into ranges, a CTA each, so that the CTAs fill the
// SMs once (twice where two fit).  Ranges of at least four tiles (a CTA's start costs about two), and no more
// than 3 sqrt(tiles) of them: the last CTA reads every range's sums, about a sixth of a tile's time each, so
// the sum of both is smallest near sqrt(6 tiles).  The ranges' sums lie behind the operands, as many as the
// workspace holds: it is sized for the factorization and the operands (solar_workspace_bytes), which often is fewer
// than are wanted (8 x 512 candidates, 10240 positions, d = 64, r = 32: three of nine; 1 x 512, 32768: fourteen of
// 48).  A larger workspace has more of them, and rounds differently.
FlashSplit flash_split(int B, int M, int N, int d, int r, size_t workspace_bytes) {
  FlashSplit s = {};
  const int tiles = (N + kPos - 1) / kPos;
  s.items_per_user = (M + kRows - 1) / kRows;
  const size_t items = (size_t)B * s.items_per_user, part = (size_t)(r + 2) * kRows * sizeof(float);
  s.counter_off = align_up(attn_ws_bytes(B, d, r), 256);
  s.part_off = s.counter_off + align_up(items * sizeof(int), 256);
  const int per_sm = (d == 64 && r <= 32) || r == 16 ? 2 : 1;                    // by shared memory
  size_t k = (size_t)(kNumSMs * per_sm) / items;
  if (k > (size_t)tiles / 4) k = (size_t)tiles / 4;
  while (k > 1 && k * k > (size_t)9 * tiles) --k;
  const size_t room = workspace_bytes > s.part_off ? (workspace_bytes - s.part_off) / (items * part) : 0;
  if (k > room) k = room;
  if (k < 1) k = 1;
  s.tiles_per_range = (int)((tiles + k - 1) / k);
  s.ranges = (tiles + s.tiles_per_range - 1) / s.tiles_per_range;
  return s;
}

cudaError_t launch_flash_factored(int B, int M, int N, int d, int r, const void* C, const void* US, void* O,
                                  char* ws, const AttnWs& lay, const FlashSplit& split, cudaStream_t st) {
#define SOLAR_FF(DD, RR) \
  if (d == DD && r == RR) return launch_dr<DD, RR>(B, M, N, C, US, O, ws, lay, split, st);
  SOLAR_FF(64, 16) SOLAR_FF(64, 32) SOLAR_FF(64, 64) SOLAR_FF(128, 16) SOLAR_FF(128, 32) SOLAR_FF(128, 64)
#undef SOLAR_FF
  return cudaErrorInvalidValue;
}

}  // namespace solar
