// Device-side parameters, tile order and element-wise epilogue shared by the GEMM kernels (gemm.cu: CTA pairs on large
// outputs; gemm_small.cu: single-CTA tiles with the contraction split inside a cluster).
#pragma once
#include "common.cuh"
#include "gemm.h"

namespace il {

constexpr int BK = 64;                           // contraction elements per k-slab

struct GemmDev {
  int M, N, K;
  int tiles_m, tiles_n;
  int group_m;                   // row blocks per group of the tile order
  int split_k, kb_per_split;     // work unit = (tile, k-range); split_k > 1 adds into C with red.add
  void* C;
  int ldc;
  void* C2;
  const float* bias;
  const float* resid;
  const bf16* aux;
  int ld_aux, aux_rows;
  float* colsum;                 // EPI_BF16_DGELU: += column sums of the output over rows < aux_rows (or NULL)
  int accumulate;
  const int* targets;
  float* part_max;
  float* part_sum;
  int part_ld;
  float* tgt_logit;
  const float* lse;
  float scale;
  int col0;
  const float* rowscale;
  int store_exp;
  unsigned* err;
};

// Tile order: groups of group_m row blocks are swept across all column blocks before the next group starts, so
// that the pairs running at the same time share a small set of A rows and the whole of B in L2.  B is read from
// DRAM once per group, A once in total: the host makes the group as tall as the matrix when all of A fits in
// L2 beside the streams passing through it (the heads' [Ntok, V, d] projection: W would otherwise be read four
// times), and 8 row blocks otherwise.
__device__ __forceinline__ void tile_coords(int t, int tiles_m, int tiles_n, int group_m, int& m_blk, int& n_blk) {
  const int per_group = group_m * tiles_n;
  const int g = t / per_group;
  const int within = t - g * per_group;
  const int gm = min(group_m, tiles_m - g * group_m);
  m_blk = g * group_m + within % gm;
  n_blk = within / gm;
}

// Element-wise part of the epilogue, after the 32 x 32 chunk has been transposed through shared memory: a
// lane now holds 4 consecutive columns (gcol..gcol+3) of row grow, 8 lanes cover 128 contiguous bytes of
// fp32 output (64 of bf16), so every global access is coalesced.  The loads of the second operand
// (residual, saved pre-activation, or C itself when accumulating) are split from the stores so that all of
// a chunk's loads are in flight before the first store (C may alias the residual).
template <int EPI>
__device__ __forceinline__ float4 epilogue_load4(const GemmDev& p, int grow, int arow, int gcol) {
  float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
  const bool vec = (gcol + 4 <= p.N);
  if constexpr (EPI == EPI_F32_RESID || EPI == EPI_F32) {
    const float* add = nullptr;
    if constexpr (EPI == EPI_F32_RESID) add = p.resid + (size_t)grow * p.ldc + gcol;
    else if (p.accumulate) add = reinterpret_cast<const float*>(p.C) + (size_t)grow * p.ldc + gcol;
    if (add) {
      if (vec) {
        e = *reinterpret_cast<const float4*>(add);
      } else {
        e.x = add[0];
        if (gcol + 1 < p.N) e.y = add[1];
        if (gcol + 2 < p.N) e.z = add[2];
      }
    }
  } else if constexpr (EPI == EPI_BF16_DGELU) {
    const bf16* h = p.aux + (size_t)arow * p.ld_aux + gcol;   // arow = grow % aux_rows
    if (vec) {
      const uint2 hv = *reinterpret_cast<const uint2*>(h);
      const float2 h0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hv.x));
      const float2 h1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&hv.y));
      e = make_float4(h0.x, h0.y, h1.x, h1.y);
    } else {
      e.x = __bfloat162float(h[0]);
      if (gcol + 1 < p.N) e.y = __bfloat162float(h[1]);
      if (gcol + 2 < p.N) e.z = __bfloat162float(h[2]);
    }
  }
  return e;
}

// COLSUM: with p.colsum, the column sums of EPI_BF16_DGELU are added here (otherwise the caller does it).
template <int EPI, bool COLSUM = true>
__device__ __forceinline__ void epilogue_store4(const GemmDev& p, int grow, int gcol, float4 a, float4 e) {
  const bool vec = (gcol + 4 <= p.N);
  float v[4] = {a.x, a.y, a.z, a.w};
  if constexpr (EPI == EPI_BF16 || EPI == EPI_BF16_GELU || EPI == EPI_F32_RESID) {
    if (p.bias) {
      if (vec) {
        const float4 b = __ldg(reinterpret_cast<const float4*>(p.bias + gcol));
        v[0] += b.x; v[1] += b.y; v[2] += b.z; v[3] += b.w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (gcol + j < p.N) v[j] += __ldg(p.bias + gcol + j);
      }
    }
  }
  if constexpr (EPI == EPI_BF16 || EPI == EPI_BF16_GELU || EPI == EPI_DZ || EPI == EPI_BF16_DGELU || EPI == EPI_LSE) {
    bf16* c = reinterpret_cast<bf16*>(p.C) + (size_t)grow * p.ldc + gcol;
    if constexpr (EPI == EPI_BF16_DGELU) {
      v[0] *= e.x; v[1] *= e.y; v[2] *= e.z; v[3] *= e.w;
      if (COLSUM && p.colsum && grow < p.aux_rows) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (gcol + j < p.N) atomicAdd(p.colsum + gcol + j, v[j]);
      }
    }
    float y[4] = {0.f, 0.f, 0.f, 0.f};
    if constexpr (EPI == EPI_BF16_GELU) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float d;
        gelu_tanh_both(v[j], y[j], d);
        v[j] = d;                                   // C receives gelu'(pre), C2 gelu(pre)
      }
    }
    if (vec) {
      uint2 o;
      o.x = pack_bf16x2(v[0], v[1]);
      o.y = pack_bf16x2(v[2], v[3]);
      *reinterpret_cast<uint2*>(c) = o;
      if constexpr (EPI == EPI_BF16_GELU) {
        uint2 g;
        g.x = pack_bf16x2(y[0], y[1]);
        g.y = pack_bf16x2(y[2], y[3]);
        *reinterpret_cast<uint2*>(reinterpret_cast<bf16*>(p.C2) + (size_t)grow * p.ldc + gcol) = g;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (gcol + j < p.N) {
          c[j] = __float2bfloat16(v[j]);
          if constexpr (EPI == EPI_BF16_GELU)
            (reinterpret_cast<bf16*>(p.C2) + (size_t)grow * p.ldc + gcol)[j] = __float2bfloat16(y[j]);
        }
    }
  } else if constexpr (EPI == EPI_F32_RESID || EPI == EPI_F32) {
    float* c = reinterpret_cast<float*>(p.C) + (size_t)grow * p.ldc + gcol;
    v[0] += e.x; v[1] += e.y; v[2] += e.z; v[3] += e.w;
    if (EPI == EPI_F32 && p.split_k > 1) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (gcol + j < p.N) atomicAdd(c + j, v[j]);
    } else if (vec) {
      *reinterpret_cast<float4*>(c) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (gcol + j < p.N) c[j] = v[j];
    }
  }
}

// gemm_small.cu: 128 x tn tiles (tn 128 or 64), the contraction split over `split` (1, 2, 4 or 8) CTAs of a cluster.
bool gemm_small_supported(int a_mn, int b_mn, int epi);
cudaError_t gemm_small_init();
cudaError_t gemm_small_launch(const GemmArgs& a, GemmDev p, int tn, int split, int num_sms, cudaStream_t stream);

// Tensor map of one operand: rows = extent of its own index (M or N), kdim = contraction extent, box_rows = tile rows.
bool encode_gemm_operand(CUtensorMap* tm, const GemmOperand& op, int rows, int kdim, int box_rows);

}  // namespace il
