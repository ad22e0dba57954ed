// Factor-token projections of Eq. 11 on the tensor cores, for bf16 weights and d = 64 or 128:
//   Key_r   = (V Sigma)^T W_K   [r,d]
//   Value_r = (V Sigma)^T W_V   [r,d]
//   T       = scale * W_Q Key_r^T  [d,r]   (so that the scores of Eq. 12 are C T)
// written as the attention kernels' packed operands (T^T and Value_r^T, each as a high and a
// low bf16 half; token rows up to the next multiple of 16, which is what those kernels read) and, on
// request, as fp32 copies and as the backward kernel's operands.  Three small GEMMs per user -- far too small
// for tcgen05 (M would be 16 or 32) -- so they run as warp-level mma.sync.m16n8k16 with fp32
// accumulation: the fp32 factor V Sigma enters as a high and a low bf16 half (two MMAs per
// product, ~16 mantissa bits), the weights are bf16 already, and Key_r never leaves the
// registers: the accumulator fragment of the first GEMM has the layout of the second GEMM's A
// fragment.  One job = (16 tokens) x (Key -> T | Value); the CTA's warps share the jobs.
// Included by the eigensolver (as the epilogue of a user's CTA) and by the stand-alone
// projection kernel, so both produce the same bits.
#pragma once

#include <cuda_bf16.h>

#include <type_traits>

#include "sm100_ptx.cuh"
#include "solar_internal.cuh"

namespace solar {
namespace pmma {

// Shared-memory layout in bytes for rp16 = 16 ceil(r / 16) token rows.  The fp32 factor
// [D][rp] (rp = r rounded up to 4) is expected at offset 0.
template <int D> struct Lay {
  static constexpr int P = (D + 8) * 2;                 // row pitch of the k-contiguous bf16 arrays: conflict-free
  __host__ __device__ static constexpr int vsh(int rp16) { return D * rp16 * 4; }          // [rp16][D+8] high halves of (V Sigma)^T
  __host__ __device__ static constexpr int vsl(int rp16) { return vsh(rp16) + rp16 * P; }  // low halves
  __host__ __device__ static constexpr int wk(int rp16) { return vsl(rp16) + rp16 * P; }   // [D][D+8] W_K as stored
  __host__ __device__ static constexpr int wq(int rp16) { return wk(rp16) + D * P; }
  __host__ __device__ static constexpr int wv(int rp16) { return wq(rp16) + D * P; }
  __host__ __device__ static constexpr int vout(int rp16) { return wv(rp16) + D * P; }     // [2][D][rp16+8] Value_r^T halves
  __host__ __device__ static constexpr int bytes(int rp16) { return vout(rp16) + 2 * D * (rp16 + 8) * 2; }
};

__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// (a, b) as a pair of high halves and the pair of what they leave over
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
  const float ah = __bfloat162float(__float2bfloat16_rn(a)), bh = __bfloat162float(__float2bfloat16_rn(b));
  hi = pack2(ah, bh);
  lo = pack2(a - ah, b - bh);
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Four 8x8 bf16 blocks, transposed on the way: B fragments (pairs along k) from a matrix stored
// with k along the rows.
__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&x)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}

// The weights of the products wanted (KINDS: bit 0 Key_r and T, bit 1 Value_r) as a thread's 16-byte
// pieces; loaded ahead of project() so that their latency runs beside whatever comes between.
template <int D, int NT, int KINDS> struct Weights {
  static constexpr int NV = D * D / 8 / NT;
  static_assert(NV * NT * 8 == D * D, "whole pieces");
  uint4 k[(KINDS & 1) ? NV : 1], q[(KINDS & 1) ? NV : 1], v[(KINDS & 2) ? NV : 1];
  __device__ __forceinline__ void load(const void* Wq, const void* Wk, const void* Wv, int tid) {
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      if (KINDS & 1) {
        k[n] = ld_dep(static_cast<const uint4*>(Wk) + tid + n * NT);
        q[n] = ld_dep(static_cast<const uint4*>(Wq) + tid + n * NT);
      }
      if (KINDS & 2) v[n] = ld_dep(static_cast<const uint4*>(Wv) + tid + n * NT);
    }
  }
};

// Where the results go.  Tpk, Vpk: the attention kernels' operands T^T [2][64][D] and Value_r^T
// [2][D][64].  Tf, Vr: fp32 copies T [D][r] and Value_r [r][D], or nullptr.  Tkm, Vkm: the backward
// kernel's further operands T [2][D][64] (zero past r) and Value_r [2][64][D], or nullptr (Tkm only
// where a CTA makes one kind).
struct Out {
  __nv_bfloat16 *Tpk, *Vpk, *Tkm, *Vkm;
  float *Tf, *Vr;
};
// Or, in the kernel that uses them (d = 64), straight to the tiles that its MMAs read: T^T [2][rp16 rows][128 B] and
// Value_r^T [2][64 rows][128 B], 128-byte swizzle.
struct Tiles { unsigned char *T, *V; };

// Every thread of the CTA (NT threads) calls this after a barrier behind the writes of the fp32
// factor at sm[0 ..).  The MMAs of a job run as four independent accumulator chains; where the CTA has
// more warps than jobs, two warps share the columns of T or Value_r.
template <int D, int NT, int KINDS, typename DST = Out>
__device__ __forceinline__ void project(unsigned char* __restrict__ sm, int r, const Weights<D, NT, KINDS>& w, float scale,
                                        const DST& o, int tid) {
  constexpr bool TILES = std::is_same<DST, Tiles>::value;
  static_assert(!TILES || (D == 64 && KINDS == 3), "both operands, one 64-wide box");
  using L = Lay<D>;
  constexpr int P = L::P, NW = NT / 32, KS = D / 16, NTL = D / 8, NV = Weights<D, NT, KINDS>::NV;
  constexpr int NK = KINDS == 3 ? 2 : 1;
  const int rp = (r + 3) & ~3, rp16 = (r + 15) & ~15, mt_n = rp16 / 16;
  const float* VS = reinterpret_cast<const float*>(sm);
  unsigned char* vsh = sm + L::vsh(rp16);
  unsigned char* vsl = sm + L::vsl(rp16);
  unsigned char* wks = sm + L::wk(rp16);
  unsigned char* wqs = sm + L::wq(rp16);
  unsigned char* wvs = sm + L::wv(rp16);
  unsigned char* stage = sm + L::vout(rp16);             // [2][D][rp16+8] Value_r^T (or T) halves
  const int lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;

#pragma unroll
  for (int n = 0; n < NV; ++n) {
    const int v = tid + n * NT, row = v / (D / 8), c = v % (D / 8);
    if (KINDS & 1) {
      *reinterpret_cast<uint4*>(wks + row * P + c * 16) = w.k[n];
      *reinterpret_cast<uint4*>(wqs + row * P + c * 16) = w.q[n];
    }
    if (KINDS & 2) *reinterpret_cast<uint4*>(wvs + row * P + c * 16) = w.v[n];
  }
  // (V Sigma)^T as bf16 halves, token-major; token rows >= rp are zero rows
  // (no division by rp16, which is known at run time only)
  for (int i = tid & 15; i < rp16; i += 16) {
    const int ic = min(i, rp - 1);
    const float* col = VS + ic;
#pragma unroll 4
    for (int kp = tid >> 4; kp < D / 2; kp += NT / 16) {
      const float a0 = col[(2 * kp) * rp], c0 = col[(2 * kp + 1) * rp];
      uint32_t hi, lo;
      split2(i < rp ? a0 : 0.f, i < rp ? c0 : 0.f, hi, lo);
      *reinterpret_cast<uint32_t*>(vsh + i * P + kp * 4) = hi;
      *reinterpret_cast<uint32_t*>(vsl + i * P + kp * 4) = lo;
    }
  }
  __syncthreads();

  const int slices = (NK * mt_n * 2 <= NW) ? 2 : 1, per = NTL / slices;   // columns (blocks of 8) of a warp
  for (int job = warp; job < NK * mt_n * slices; job += NW) {
    const int sl = job % slices, mt = (job / slices) % mt_n;
    const int kind = KINDS == 3 ? job / (slices * mt_n) : KINDS - 1;        // 0: Key_r, then T; 1: Value_r
    const int i0 = 16 * mt + g;                            // this lane's token rows: i0 and i0 + 8
    // A fragments of (V Sigma)^T for all k
    uint32_t ah[KS][4], al[KS][4];
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      const int o0 = i0 * P + (16 * ks + 2 * t) * 2, o1 = o0 + 8 * P;
      ah[ks][0] = *reinterpret_cast<const uint32_t*>(vsh + o0);
      ah[ks][1] = *reinterpret_cast<const uint32_t*>(vsh + o1);
      ah[ks][2] = *reinterpret_cast<const uint32_t*>(vsh + o0 + 16);
      ah[ks][3] = *reinterpret_cast<const uint32_t*>(vsh + o1 + 16);
      al[ks][0] = *reinterpret_cast<const uint32_t*>(vsl + o0);
      al[ks][1] = *reinterpret_cast<const uint32_t*>(vsl + o1);
      al[ks][2] = *reinterpret_cast<const uint32_t*>(vsl + o0 + 16);
      al[ks][3] = *reinterpret_cast<const uint32_t*>(vsl + o1 + 16);
    }
    // acc[c] = columns 8 (nt0 + c) .. of X[i][j] = sum_k (V Sigma)[k][i] W[k][j], four blocks at a time
    auto four = [&](float (&acc)[4][4], const unsigned char* wsrc, int nt0) {
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[c][0] = acc[c][1] = acc[c][2] = acc[c][3] = 0.f;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        uint32_t b0[4], b1[4];       // b0, b1 of a column block; b0, b1 of the next
        const unsigned char* wr = wsrc + (16 * ks + 8 * ((lane >> 3) & 1) + (lane & 7)) * P + (8 * (nt0 + (lane >> 4))) * 2;
        ldsm_x4_trans(b0, wr);
        ldsm_x4_trans(b1, wr + 32);
        mma16816(acc[0], ah[ks], b0[0], b0[1]); mma16816(acc[1], ah[ks], b0[2], b0[3]);
        mma16816(acc[2], ah[ks], b1[0], b1[1]); mma16816(acc[3], ah[ks], b1[2], b1[3]);
        mma16816(acc[0], al[ks], b0[0], b0[1]); mma16816(acc[1], al[ks], b0[2], b0[3]);
        mma16816(acc[2], al[ks], b1[0], b1[1]); mma16816(acc[3], al[ks], b1[2], b1[3]);
      }
    };
    // a 2 x 2 piece (tokens i, i + 8; columns j, j + 1) into the staging tile [h][j][token]
    auto put = [&](const float (&x)[4], int j) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const __nv_bfloat16 hi = __float2bfloat16_rn(x[q]);
        if constexpr (TILES) {
          const int tok = i0 + 8 * (q >> 1);
          unsigned char* at = o.V + ptx::swz128(j + (q & 1), tok >> 3) + 2 * (tok & 7);
          *reinterpret_cast<__nv_bfloat16*>(at) = hi;
          *reinterpret_cast<__nv_bfloat16*>(at + D * 128) = __float2bfloat16_rn(x[q] - __bfloat162float(hi));
          continue;
        }
        __nv_bfloat16* row = reinterpret_cast<__nv_bfloat16*>(stage) + (size_t)(j + (q & 1)) * (rp16 + 8) + i0 + 8 * (q >> 1);
        row[0] = hi;
        row[(size_t)D * (rp16 + 8)] = __float2bfloat16_rn(x[q] - __bfloat162float(hi));
      }
    };
    if ((KINDS & 2) && kind == 1) {
#pragma unroll 1
      for (int nt0 = sl * per; nt0 < (sl + 1) * per; nt0 += 4) {
        float acc[4][4];
        four(acc, wvs, nt0);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int j = 8 * (nt0 + c) + 2 * t;
          put(acc[c], j);
          if constexpr (!TILES) {
            if (o.Vr != nullptr) {
              if (i0 < r) *reinterpret_cast<float2*>(o.Vr + (size_t)i0 * D + j) = make_float2(acc[c][0], acc[c][1]);
              if (i0 + 8 < r) *reinterpret_cast<float2*>(o.Vr + (size_t)(i0 + 8) * D + j) = make_float2(acc[c][2], acc[c][3]);
            }
            if (o.Vkm != nullptr) {                             // zero rows come out of zero rows of V Sigma
              uint32_t hi, lo;
              split2(acc[c][0], acc[c][1], hi, lo);
              *reinterpret_cast<uint32_t*>(o.Vkm + (size_t)i0 * D + j) = hi;
              *reinterpret_cast<uint32_t*>(o.Vkm + (size_t)(kTokenSlots + i0) * D + j) = lo;
              split2(acc[c][2], acc[c][3], hi, lo);
              *reinterpret_cast<uint32_t*>(o.Vkm + (size_t)(i0 + 8) * D + j) = hi;
              *reinterpret_cast<uint32_t*>(o.Vkm + (size_t)(kTokenSlots + i0 + 8) * D + j) = lo;
            }
          }
        }
      }
    }
    if ((KINDS & 1) && kind == 0) {
      // Key_r, all D columns, as the A operand of T^T[i][k] = scale * sum_j Key_r[i][j] W_Q[k][j]
      uint32_t kh[KS][4], kl[KS][4];
#pragma unroll
      for (int nt0 = 0; nt0 < NTL; nt0 += 4) {
        float acc[4][4];
        four(acc, wks, nt0);
#pragma unroll
        for (int c = 0; c < 4; c += 2) {
          const int ks = (nt0 + c) / 2;
          split2(acc[c][0], acc[c][1], kh[ks][0], kl[ks][0]);
          split2(acc[c][2], acc[c][3], kh[ks][1], kl[ks][1]);
          split2(acc[c + 1][0], acc[c + 1][1], kh[ks][2], kl[ks][2]);
          split2(acc[c + 1][2], acc[c + 1][3], kh[ks][3], kl[ks][3]);
        }
      }
#pragma unroll 1
      for (int nt0 = sl * per; nt0 < (sl + 1) * per; nt0 += 4) {
        float tc[4][4];
#pragma unroll
        for (int c = 0; c < 4; ++c) tc[c][0] = tc[c][1] = tc[c][2] = tc[c][3] = 0.f;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          uint32_t b0[4], b1[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const unsigned char* wrow = wqs + (8 * (nt0 + c) + g) * P + (16 * ks + 2 * t) * 2;     // W_Q[k = 8 nt + g][j ..]
            b0[c] = *reinterpret_cast<const uint32_t*>(wrow); b1[c] = *reinterpret_cast<const uint32_t*>(wrow + 16);
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) mma16816(tc[c], kh[ks], b0[c], b1[c]);
#pragma unroll
          for (int c = 0; c < 4; ++c) mma16816(tc[c], kl[ks], b0[c], b1[c]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
#pragma unroll
          for (int q = 0; q < 4; ++q) tc[c][q] *= scale;
          const int k0 = 8 * (nt0 + c) + 2 * t;
          uint32_t hi, lo;
          if constexpr (TILES) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {                        // token rows i0, i0 + 8
              split2(tc[c][2 * h], tc[c][2 * h + 1], hi, lo);
              unsigned char* at = o.T + ptx::swz128(i0 + 8 * h, k0 >> 3) + 2 * (k0 & 7);
              *reinterpret_cast<uint32_t*>(at) = hi;
              *reinterpret_cast<uint32_t*>(at + rp16 * 128) = lo;
            }
          } else {
            split2(tc[c][0], tc[c][1], hi, lo);
            *reinterpret_cast<uint32_t*>(o.Tpk + (size_t)i0 * D + k0) = hi;
            *reinterpret_cast<uint32_t*>(o.Tpk + ((size_t)kTokenSlots + i0) * D + k0) = lo;
            split2(tc[c][2], tc[c][3], hi, lo);
            *reinterpret_cast<uint32_t*>(o.Tpk + (size_t)(i0 + 8) * D + k0) = hi;
            *reinterpret_cast<uint32_t*>(o.Tpk + ((size_t)kTokenSlots + i0 + 8) * D + k0) = lo;
            if (KINDS == 1 && o.Tkm != nullptr) put(tc[c], k0);
            if (o.Tf != nullptr) {
              if (i0 < r) { o.Tf[(size_t)k0 * r + i0] = tc[c][0]; o.Tf[(size_t)(k0 + 1) * r + i0] = tc[c][1]; }
              if (i0 + 8 < r) { o.Tf[(size_t)k0 * r + i0 + 8] = tc[c][2]; o.Tf[(size_t)(k0 + 1) * r + i0 + 8] = tc[c][3]; }
            }
          }
        }
      }
    }
  }
  if constexpr (!TILES) {
    // what was staged, as 16-byte pieces of the rows [h][j][0 .. rp16); Tkm is read to its 64th column
    __nv_bfloat16* dst = (KINDS & 2) ? o.Vpk : o.Tkm;
    if ((KINDS & 2) || dst != nullptr) {
      __syncthreads();
      const int pc = (KINDS & 2) ? rp16 / 8 : kTokenSlots / 8;
      const unsigned inv = pc == 2 ? 32768u : pc == 4 ? 16384u : pc == 6 ? 10923u : 8192u;    // 2^16 / pc, up: exact for e < 2048
#pragma unroll 4
      for (int e = tid; e < 2 * D * pc; e += NT) {
        const int row = (int)((unsigned)e * inv >> 16), c = e - row * pc;                    // row runs over [2][D]
        reinterpret_cast<uint4*>(dst + (size_t)row * kTokenSlots)[c] =
            c < rp16 / 8 ? *reinterpret_cast<const uint4*>(stage + ((size_t)row * (rp16 + 8) + 8 * c) * 2) : make_uint4(0u, 0u, 0u, 0u);
      }
    }
  }
}

}  // namespace pmma
}  // namespace solar
