// tcgen05 GEMM for outputs that do not fill the GPU with 256-row tiles of CTA pairs: C[M,N] = A[M,K] * B[N,K]^T with
// one CTA per 128 x 128 or 128 x 64 tile and, when even those tiles are few, the contraction split over a cluster of
// 2, 4 or 8 CTAs.
//
// Every CTA of a cluster accumulates its k-range of the same tile in its own tensor memory (M128 K16 MMAs from a
// TMA-fed ring), writes the fp32 partial tile to its shared memory and meets the others at the cluster barrier.
// Each then owns 128 / S rows of the tile: it reads those rows from all S partial tiles over distributed shared
// memory, adds them in rank order (a fixed order: the result does not depend on scheduling) and applies the fused
// epilogue, 16 bytes per thread and row.  No workspace, no atomics, no zeroing pass.
// All eight warps run the epilogue; before it one thread of warp 0 feeds the ring and one thread of warp 1 issues the
// MMAs.  Every wait is bounded; on expiry the CTA sets the error word, skips its stores and still meets its cluster.
//
// What bounds it: with one CTA per SM a slab costs 0.26 us (the ring's load latency: 6 stages of 32 KB, 9 of 24 KB),
// so the contraction's length per CTA decides, and a launch costs 3.5 us around it.  Measured (back to back in a
// graph, us; paired 256 x 256 tiles / this kernel): 256 x 768 x 3072 with residual 22.4 (256 x 512 tiles: 41.1) /
// 8.2; 256 x 768 x 50257 228 (450) / 36; 256 x 512 x 128 with GELU 7.6 / 4.4; 2505 x 512 x 2048 14.9 (25.5) / 13.2.
#include "common.cuh"
#include "gemm.h"
#include "gemm_dev.cuh"

namespace il {

namespace {

constexpr int TM = 128;                          // tile rows; the tile has TN = 128 or 64 columns
constexpr int A_BYTES = TM * BK * 2;             // 16 KB per slab
constexpr int THREADS = 256;
constexpr int GROUP = 8;                         // float4 items of a thread whose second operands are in flight together
template <int TN> struct SmallCfg {
  static constexpr int STAGE_BYTES = A_BYTES + TN * BK * 2;
  static constexpr int MAX_STAGES = TN == 128 ? 6 : 9;
  static constexpr int SHARED_STAGES = TN == 128 ? 3 : 4;  // ring depth when two CTAs share an SM
  static constexpr int PART_BYTES = TM * TN * 4;           // fp32 partial tile, over the ring once its last MMA has retired
  static constexpr int SLOTS = TN / 4;                     // 16-byte slots of a tile row
  static constexpr int ROWS_IT = THREADS / SLOTS;          // rows the CTA covers per item
  static constexpr int ITEMS = TM / ROWS_IT;               // items of a thread (one CTA per tile)
  __host__ __device__ static constexpr int ring_bytes(int stages) {
    return stages * STAGE_BYTES > PART_BYTES ? stages * STAGE_BYTES : PART_BYTES;
  }
  __host__ __device__ static constexpr int smem_bytes(int stages) {
    return ring_bytes(stages) + 1024 + 256 + THREADS * 16 /* column sums */;
  }
};

__device__ __forceinline__ float4 ld_cluster_f32x4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

template <bool A_MN, bool B_MN, int EPI, int TN>
__global__ void __launch_bounds__(THREADS, 2)
gemm_small_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmDev p,
                  const int stages, const int S) {
  using C = SmallCfg<TN>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_smem;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  const int ring = C::ring_bytes(stages);
  const uint32_t bars = base + ring;
  const uint32_t acc_bar = bars + 16u * stages;
  float4* s_cs = reinterpret_cast<float4*>(gen + ring + 256);
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (stages + s); };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = S > 1 ? cluster_ctarank() : 0u;
  int m_blk, n_blk;
  tile_coords(blockIdx.x / S, p.tiles_m, p.tiles_n, p.group_m, m_blk, n_blk);
  const int m0 = m_blk * TM, n0 = n_blk * TN;
  const int num_kb = (p.K + BK - 1) / BK;
  const int kb0 = (int)rank * p.kb_per_split, kb1 = min(num_kb, kb0 + p.kb_per_split);

  if (tid == 0) {
    abort_flag = 0;
    for (int s = 0; s < stages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(acc_bar, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmA);
    tma_prefetch_desc(&tmB);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_base_smem), TN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dep_wait();          // tensor memory is held, nothing in global memory has been touched yet
  const uint32_t tmem_base = tmem_base_smem;
  volatile int* abortp = &abort_flag;

  // This thread's part of the epilogue: four columns of rows row_first + ROWS_IT i.
  const int items = C::ITEMS / S;
  const int slot = tid % C::SLOTS;
  const int row_first = (int)rank * (TM / S) + tid / C::SLOTS;
  const int gcol = n0 + 4 * slot;
  const bool vec = gcol + 4 <= p.N;
  constexpr bool HAS_EXTRA = (EPI == EPI_F32_RESID || EPI == EPI_BF16_DGELU || EPI == EPI_F32);
  float4 extra[GROUP], b4 = make_float4(0.f, 0.f, 0.f, 0.f);
  float rs[GROUP];
#pragma unroll
  for (int i = 0; i < GROUP; ++i) { extra[i] = make_float4(0.f, 0.f, 0.f, 0.f); rs[i] = 1.0f; }
  auto load_extra = [&](int g) {
    if constexpr (HAS_EXTRA) {
      int arow = 0;
      if constexpr (EPI == EPI_BF16_DGELU) arow = (m0 + row_first + C::ROWS_IT * g * GROUP) % p.aux_rows;
#pragma unroll
      for (int i = 0; i < GROUP; ++i) {
        const int grow = m0 + row_first + C::ROWS_IT * (g * GROUP + i);
        if (g * GROUP + i < items && grow < p.M && gcol < p.N) {
          if (EPI != EPI_F32 || p.accumulate) extra[i] = epilogue_load4<EPI>(p, grow, arow, gcol);
          if (EPI == EPI_F32 && p.rowscale) rs[i] = __ldg(p.rowscale + grow);
        }
        if constexpr (EPI == EPI_BF16_DGELU) {
          arow += C::ROWS_IT;
          while (arow >= p.aux_rows) arow -= p.aux_rows;
        }
      }
    }
    if constexpr (EPI == EPI_BF16 || EPI == EPI_BF16_GELU || EPI == EPI_F32_RESID)
      if (g == 0 && p.bias && vec) b4 = __ldg(reinterpret_cast<const float4*>(p.bias + gcol));
  };

  if (warp == 0) {
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait(empty_bar(stage), phase ^ 1u, abortp)) {
          atomicExch(p.err, DEV_TIMEOUT_PRODUCER);
          abort_flag = 1;
          break;
        }
        const uint32_t sa = base + stage * C::STAGE_BYTES, sb = sa + A_BYTES, fb = full_bar(stage);
        mbar_expect_tx(fb, C::STAGE_BYTES);
        const int k0 = kb * BK;
        if constexpr (!A_MN) {
          tma_load_2d(sa, &tmA, k0, m0, fb);
        } else {
          tma_load_2d(sa, &tmA, m0, k0, fb);
          tma_load_2d(sa + 8192, &tmA, m0 + 64, k0, fb);
        }
        if constexpr (!B_MN) {
          tma_load_2d(sb, &tmB, k0, n0, fb);
        } else {
#pragma unroll
          for (int i = 0; i < TN / 64; ++i) tma_load_2d(sb + i * 8192, &tmB, n0 + 64 * i, k0, fb);
        }
        if (++stage == stages) { stage = 0; phase ^= 1u; }
      }
      grid_dep_launch();
    }
    __syncwarp();
    load_extra(0);
  } else {
    load_extra(0);
    if (warp == 1) {
      if (lane == 0) {
        constexpr uint32_t idesc = make_idesc_bf16(TM, TN, A_MN ? 1 : 0, B_MN ? 1 : 0);
        int stage = 0;
        uint32_t phase = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(full_bar(stage), phase, abortp)) {
            atomicExch(p.err, DEV_TIMEOUT_MMA);
            abort_flag = 1;
            break;
          }
          tc_fence_after();
          const uint32_t sa = base + stage * C::STAGE_BYTES, sb = sa + A_BYTES;
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            const uint64_t ad = A_MN ? make_smem_desc(sa + k * 2048, 8192, 1024) : make_smem_desc(sa + k * 32, 16, 1024);
            const uint64_t bd = B_MN ? make_smem_desc(sb + k * 2048, 8192, 1024) : make_smem_desc(sb + k * 32, 16, 1024);
            umma_bf16(tmem_base, ad, bd, idesc, (kb > kb0 || k != 0) ? 1u : 0u);
          }
          umma_commit(empty_bar(stage));
          if (++stage == stages) { stage = 0; phase ^= 1u; }
        }
        umma_commit(acc_bar);
      }
      __syncwarp();
    }
  }

  {   // the accumulator is complete (one lane per warp polls)
    int got = 1;
    if (lane == 0) got = mbar_wait(acc_bar, 0, abortp) ? 1 : 0;
    if (!__shfl_sync(0xffffffffu, got, 0) && lane == 0) {
      atomicExch(p.err, DEV_TIMEOUT_EPILOGUE);
      abort_flag = 1;
    }
    tc_fence_after();
  }
  // Partial tile to shared memory: row r, 16-byte slot c at r * 4 TN + (c ^ (r & 7)) * 16.  A CTA whose k-range is
  // empty (the split does not divide the slabs) contributes zeros.
  {
    const int q = warp & 3, half = warp >> 2, r = q * 32 + lane;
#pragma unroll
    for (int c = 0; c < TN / 64; ++c) {
      uint32_t v[32];
      tmem_ld_32x32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * (TN / 2) + c * 32), v);
      tmem_ld_wait();
      if (kb0 >= kb1) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = 0u;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
        *reinterpret_cast<uint4*>(gen + r * (TN * 4) + (((half * (TN / 8) + c * 8 + j) ^ (r & 7)) << 4)) =
            make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
    }
  }
  tc_fence_before();
  if (S > 1) cluster_sync_all();
  else __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, TN);
  }

  float4 cs = make_float4(0.f, 0.f, 0.f, 0.f);
  if (!*abortp && gcol < p.N) {
#pragma unroll 1
    for (int g = 0; g * GROUP < items; ++g) {
      float4 a[GROUP];
#pragma unroll
      for (int i = 0; i < GROUP; ++i) {
        if (g * GROUP + i >= items) break;
        const int r = row_first + C::ROWS_IT * (g * GROUP + i);
        const uint32_t off = (uint32_t)(r * (TN * 4) + ((slot ^ (r & 7)) << 4));
        if (S == 1) {
          a[i] = *reinterpret_cast<const float4*>(gen + off);
        } else {
          float4 t[8];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (k < S) t[k] = ld_cluster_f32x4(mapa_cluster(base + off, k));
          a[i] = t[0];
#pragma unroll
          for (int k = 1; k < 8; ++k)
            if (k < S) { a[i].x += t[k].x; a[i].y += t[k].y; a[i].z += t[k].z; a[i].w += t[k].w; }
        }
      }
#pragma unroll
      for (int i = 0; i < GROUP; ++i) {
        if (g * GROUP + i >= items) break;
        const int grow = m0 + row_first + C::ROWS_IT * (g * GROUP + i);
        if (grow >= p.M) break;
        if constexpr (EPI == EPI_F32) { a[i].x *= rs[i]; a[i].y *= rs[i]; a[i].z *= rs[i]; a[i].w *= rs[i]; }
        if constexpr (EPI == EPI_BF16_DGELU) {
          if (grow < p.aux_rows) {
            cs.x += a[i].x * extra[i].x; cs.y += a[i].y * extra[i].y; cs.z += a[i].z * extra[i].z; cs.w += a[i].w * extra[i].w;
          }
        }
        if (!vec) {                      // ragged last columns
          epilogue_store4<EPI, false>(p, grow, gcol, a[i], extra[i]);
          continue;
        }
        const float x0 = a[i].x + b4.x, x1 = a[i].y + b4.y, x2 = a[i].z + b4.z, x3 = a[i].w + b4.w;
        const size_t at = (size_t)grow * p.ldc + gcol;
        if constexpr (EPI == EPI_F32_RESID || EPI == EPI_F32) {
          *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.C) + at) =
              make_float4(x0 + extra[i].x, x1 + extra[i].y, x2 + extra[i].z, x3 + extra[i].w);
        } else if constexpr (EPI == EPI_BF16_GELU) {
          float y0, y1, y2, y3, d0, d1, d2, d3;
          gelu_tanh_both(x0, y0, d0); gelu_tanh_both(x1, y1, d1);
          gelu_tanh_both(x2, y2, d2); gelu_tanh_both(x3, y3, d3);
          *reinterpret_cast<uint2*>(reinterpret_cast<bf16*>(p.C) + at) = make_uint2(pack_bf16x2(d0, d1), pack_bf16x2(d2, d3));
          *reinterpret_cast<uint2*>(reinterpret_cast<bf16*>(p.C2) + at) = make_uint2(pack_bf16x2(y0, y1), pack_bf16x2(y2, y3));
        } else {
          float4 x = make_float4(x0, x1, x2, x3);
          if constexpr (EPI == EPI_BF16_DGELU) { x.x *= extra[i].x; x.y *= extra[i].y; x.z *= extra[i].z; x.w *= extra[i].w; }
          *reinterpret_cast<uint2*>(reinterpret_cast<bf16*>(p.C) + at) = make_uint2(pack_bf16x2(x.x, x.y), pack_bf16x2(x.z, x.w));
        }
      }
      if ((g + 1) * GROUP < items) load_extra(g + 1);
    }
  }
  if constexpr (EPI == EPI_BF16_DGELU) {
    if (p.colsum) {           // uniform
      s_cs[tid] = cs;
      __syncthreads();
      if (tid < C::SLOTS && gcol < p.N && !*abortp) {
        float4 t = s_cs[tid];
#pragma unroll
        for (int w = 1; w < C::ROWS_IT; ++w) {
          const float4 u = s_cs[w * C::SLOTS + tid];
          t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
        }
        if (vec) {
          red_add_f32x4(p.colsum + gcol, t);
        } else {
          const float e[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (gcol + j < p.N) atomicAdd(p.colsum + gcol + j, e[j]);
        }
      }
    }
  }
  if (S > 1) cluster_sync_all();       // nobody leaves while a peer may still read its partial tile
}

typedef void (*SmallFn)(const CUtensorMap, const CUtensorMap, const GemmDev, const int, const int);

template <bool A_MN, bool B_MN, int TN>
SmallFn pick_small(int epi) {
  if constexpr (!A_MN && !B_MN) {
    switch (epi) {
      case EPI_BF16: return gemm_small_kernel<false, false, EPI_BF16, TN>;
      case EPI_BF16_GELU: return gemm_small_kernel<false, false, EPI_BF16_GELU, TN>;
      case EPI_F32_RESID: return gemm_small_kernel<false, false, EPI_F32_RESID, TN>;
    }
  } else if constexpr (!A_MN && B_MN) {
    switch (epi) {
      case EPI_BF16: return gemm_small_kernel<false, true, EPI_BF16, TN>;
      case EPI_BF16_DGELU: return gemm_small_kernel<false, true, EPI_BF16_DGELU, TN>;
      case EPI_F32: return gemm_small_kernel<false, true, EPI_F32, TN>;
    }
  } else if constexpr (A_MN && B_MN) {
    if (epi == EPI_F32) return gemm_small_kernel<true, true, EPI_F32, TN>;
  }
  return nullptr;
}

template <int TN>
SmallFn pick_small_tn(int a_mn, int b_mn, int epi) {
  if (!a_mn && !b_mn) return pick_small<false, false, TN>(epi);
  if (!a_mn && b_mn) return pick_small<false, true, TN>(epi);
  if (a_mn && b_mn) return pick_small<true, true, TN>(epi);
  return nullptr;
}
SmallFn pick_small_kernel(int a_mn, int b_mn, int epi, int tn) {
  return tn == 64 ? pick_small_tn<64>(a_mn, b_mn, epi) : pick_small_tn<128>(a_mn, b_mn, epi);
}

}  // namespace

bool gemm_small_supported(int a_mn, int b_mn, int epi) { return pick_small_kernel(a_mn, b_mn, epi, 128) != nullptr; }

cudaError_t gemm_small_init() {
  for (int l = 0; l < 4; ++l)
    for (int epi = 0; epi < EPI_COUNT; ++epi)
      for (int tn = 64; tn <= 128; tn += 64) {
        SmallFn k = pick_small_kernel(l & 1, l >> 1, epi, tn);
        if (!k) continue;
        const int bytes = tn == 64 ? SmallCfg<64>::smem_bytes(SmallCfg<64>::MAX_STAGES) : SmallCfg<128>::smem_bytes(SmallCfg<128>::MAX_STAGES);
        cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void*>(k), cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
      }
  return cudaSuccess;
}

cudaError_t gemm_small_launch(const GemmArgs& a, GemmDev p, int tn, int split, int num_sms, cudaStream_t stream) {
  SmallFn kern = pick_small_kernel(a.A.mn_major, a.B.mn_major, a.epilogue, tn);
  if (!kern) return cudaErrorInvalidValue;
  CUtensorMap tmA, tmB;
  if (!encode_gemm_operand(&tmA, a.A, a.M, a.K, TM) || !encode_gemm_operand(&tmB, a.B, a.N, a.K, tn)) return cudaErrorInvalidValue;
  p.tiles_m = (a.M + TM - 1) / TM;
  p.tiles_n = (a.N + tn - 1) / tn;
  p.group_m = p.tiles_m < 16 ? p.tiles_m : 16;
  const int num_kb = (a.K + BK - 1) / BK;
  p.split_k = 1;                                 // (the atomic form of the paired kernel)
  p.kb_per_split = (num_kb + split - 1) / split;
  const int ctas = p.tiles_m * p.tiles_n * split;
  // A deep ring while every CTA has an SM to itself (clusters of four and eight do not pack every SM), a shallow one
  // (two CTAs per SM) beyond that; never deeper than the contraction is long.
  int stages = tn == 64 ? SmallCfg<64>::MAX_STAGES : SmallCfg<128>::MAX_STAGES;
  if (ctas > (split == 8 ? num_sms * 2 / 3 : split == 4 ? num_sms * 5 / 6 : num_sms))
    stages = tn == 64 ? SmallCfg<64>::SHARED_STAGES : SmallCfg<128>::SHARED_STAGES;
  if (stages > p.kb_per_split) stages = p.kb_per_split;
  const size_t smem = tn == 64 ? SmallCfg<64>::smem_bytes(stages) : SmallCfg<128>::smem_bytes(stages);
  return launch_dep_cluster(kern, dim3(ctas), dim3(THREADS), smem, stream, split, tmA, tmB, p, stages, split);
}

}  // namespace il
