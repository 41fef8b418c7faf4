// Causal self-attention backward for sequences of at most 128 positions (sm_100a): one kernel, one work item per
// (gradient sequence, head).
//
// The whole score matrix of an item is one 128 x 128 tile, so nothing is swept and nothing is summed across CTAs: the
// row sums delta_i = sum_j P_ij dP_ij are formed from the tile itself (equal to sum_c dO_ic O_ic, so O is not read), and
// dQ, dK and dV are complete when their one product is.  Rows of a tile are queries throughout:
//   S = Q K^T, dP = dO V^T          M128 N=T (rounded up to 16), operands K-major, into tensor memory
//   P = exp(scale S - lse), dS = P (dP - delta)     two threads per row, rounded to bf16, to shared memory in 128-byte
//                                   swizzled rows of 64 keys, which the next products read either way round:
//   dV = P^T dO, dK = dS^T Q        A MN-major (M = keys), contraction over the queries
//   dQ = dS K                       A K-major (M = queries)
// The contractions run over T rounded up to 16 only.  Each result is converted into the shared memory of an operand that
// is no longer needed (dV over dO, dK over Q, dQ over K) and leaves by TMA, rows past the sequence dropped by the map.
// Warps 0-7 do the row work and the conversions; one thread of warp 8 issues every load, MMA and store.
//
// Tensor memory is reused within an item: up to dh 80 the three results lie over S and dP (256 columns, so two CTAs per
// SM up to dh 64); dh 256 puts dV beside them, dK over them and dQ where dV was.  Shared memory at dh 256: Q, K and dO
// stay (192 KB), V comes through two 16 KB chunks, whose place P and then dS take.
//
// What bounds it: a CTA's chain of loads, products, row work and stores, half of it under the bytes (Q, K, V, dO in, dQ, dK,
// dV out) that have to move; small batches: the chain alone.  Measured against the sweeps of attention.cu, which take three
// or four launches with their delta and conversion passes (gradient sequences x heads x T, dh; floor of the bytes):
//   128 x 4 x 128, dh 256   60 us, was 182 (29)        64 x 16 x 128, dh 64   39 us, one sweep 69, two kernels 85 (18)
//   64 x 8 x 100, dh 128    29 us, was 77 (14)         32 x 32 x 128, dh 80   56 us, was 140 (23)
//   128 x 12 x 64, dh 64    42 us, 73 and 70 (14)      4 x 4 x 64, dh 32      7.6 us, 14.9 and 14.2
// So there is no length up to 128 at which the sweeps are kept.  A step of the paper's shape 156.2 -> 147.9 ms.
#include "common.cuh"
#include "kernels.h"
#include "tma.h"

namespace il {

namespace {

constexpr int SHORT_ROWS = 128;
constexpr int SHORT_THREADS = 288;
constexpr int SHORT_CHUNK = SHORT_ROWS * 128;                   // 128 rows x 64 bf16

template <int DH>
struct ShortCfg {
  static constexpr int NCH = (DH + 63) / 64;
  static constexpr int OP = NCH * SHORT_CHUNK;                  // one operand
  static constexpr bool RING = DH > 128;                        // V through two chunks that P / dS take over
  static constexpr bool SHARED = RING || DH <= 64;              // dS takes P's place (else a buffer of its own)
  static constexpr int P_BYTES = 2 * SHORT_CHUNK;
  static constexpr int O_Q = 0, O_K = OP, O_DO = 2 * OP, O_V = 3 * OP;
  static constexpr int O_P = RING ? O_V : 4 * OP;
  static constexpr int O_DS = SHARED ? O_P : O_P + P_BYTES;
  static constexpr int O_END = O_DS + P_BYTES;
  static constexpr int SMEM = 1024 + O_END + 256 + 2 * SHORT_ROWS * 4;   // (barriers, row sums)
  static constexpr int C_S = 0, C_DP = 128;
  static constexpr int C_DV = RING ? 256 : 0, C_DK = RING ? 0 : DH, C_DQ = RING ? 256 : 2 * DH;
  static constexpr int TCOLS = 3 * DH <= 256 ? 256 : 512;
  static constexpr int CTAS = DH <= 64 ? 2 : 1;                 // resident per SM
  static constexpr int UNIT = DH % 64 == 0 ? 32 : 16;           // columns a thread converts at a time
};

__device__ __forceinline__ void tma_store_4d(const void* tmap, uint32_t src_smem, int c0, int c1, int c2, int c3) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
               ::"l"(tmap), "r"(src_smem), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
               : "memory");
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

template <int DH>
__global__ void __launch_bounds__(SHORT_THREADS, ShortCfg<DH>::CTAS)
attn_bwd_short_kernel(const __grid_constant__ CUtensorMap tm_qkv, const __grid_constant__ CUtensorMap tm_do,
                      const __grid_constant__ CUtensorMap tm_out, const float* __restrict__ lse, int NB, int B, int T, int H,
                      float scale, unsigned* err) {
  using C = ShortCfg<DH>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_smem;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bars = base + C::O_END;
  enum { B_Q, B_K, B_DO, B_V0, B_V1, B_VF0, B_VF1, B_S, B_DP, B_P, B_DS, B_DV, B_DK, B_DQ, B_O0, B_O1, B_O2, B_X, B_DRAIN = B_X + 4, B_COUNT };
  auto bar = [&](int i) { return bars + 8 * i; };
  float* s_part = reinterpret_cast<float*>(smem_raw + (base - smem_u32(smem_raw)) + C::O_END + 256);   // [2][128]

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nk = (T + 15) >> 4, R = nk << 4;                    // contraction steps and padded length
  const int nitems = NB * H;
  volatile int* abortp = &abort_flag;

  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < B_COUNT; ++i) mbar_init(bar(i), i == B_P || i == B_DS || (i >= B_O0 && i <= B_O2) ? 8 : i >= B_X && i < B_X + 4 ? 2 : 1);
    fence_mbar_init();
    tma_prefetch_desc(&tm_qkv);
    tma_prefetch_desc(&tm_do);
    tma_prefetch_desc(&tm_out);
  }
  if (warp == 8) {
    tmem_alloc(smem_u32(&tmem_base_smem), C::TCOLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dep_wait();
  const uint32_t tmem = tmem_base_smem;
  int fail = 0;

  if (warp == 8) {
    if (lane == 0) {
      const uint32_t bytes = (uint32_t)R * 128u;                // of one chunk of a box
      const uint32_t idesc_s = make_idesc_bf16(SHORT_ROWS, R, 0, 0);
      constexpr uint32_t idesc_mn = make_idesc_bf16(SHORT_ROWS, DH, 1, 1), idesc_k = make_idesc_bf16(SHORT_ROWS, DH, 0, 1);
      const uint32_t sQ = base + C::O_Q, sK = base + C::O_K, sDO = base + C::O_DO, sV = base + C::O_V, sP = base + C::O_P,
                     sDS = base + C::O_DS;
      auto load = [&](uint32_t dst, const CUtensorMap* tm, int slot, int seq, int b) {
        mbar_expect_tx(bar(b), C::NCH * bytes);
#pragma unroll
        for (int c = 0; c < C::NCH; ++c) tma_load_4d(dst + c * SHORT_CHUNK, tm, c * 64, slot, 0, seq, bar(b));
      };
      auto load_v = [&](int c, int h, int bs) {                 // one chunk of V into its place of the ring
        mbar_expect_tx(bar(B_V0 + (c & 1)), bytes);
        tma_load_4d(sV + (c & 1) * SHORT_CHUNK, &tm_qkv, c * 64, 2 * H + h, 0, bs, bar(B_V0 + (c & 1)));
      };
      auto store = [&](uint32_t src, int slot, int nb) {
#pragma unroll
        for (int c = 0; c < C::NCH; ++c) tma_store_4d(&tm_out, src + c * SHORT_CHUNK, c * 64, slot, 0, nb);
        bulk_commit_group();
      };
      auto wait = [&](int b, uint32_t parity) -> bool {
        if (mbar_wait(bar(b), parity, abortp)) return true;
        fail = 1;
        abort_flag = 1;
        return false;
      };
      if (blockIdx.x < nitems) {
        const int nb = blockIdx.x / H, h = blockIdx.x - nb * H, bs = nb % B;
        load(sQ, &tm_qkv, h, bs, B_Q);
        load(sK, &tm_qkv, H + h, bs, B_K);
        load(sDO, &tm_do, h, nb, B_DO);
        if (C::RING) { load_v(0, h, bs); load_v(1, h, bs); }
        else load(sV, &tm_qkv, 2 * H + h, bs, B_V0);
      }
      const SmemDescBase dq_k = make_smem_desc_base(sQ, 16, 1024), dk_k = make_smem_desc_base(sK, 16, 1024);
      const SmemDescBase ddo_k = make_smem_desc_base(sDO, 16, 1024), dv_k = make_smem_desc_base(sV, 16, 1024);
      const SmemDescBase dq_mn = make_smem_desc_base(sQ, SHORT_CHUNK, 1024), dk_mn = make_smem_desc_base(sK, SHORT_CHUNK, 1024);
      const SmemDescBase ddo_mn = make_smem_desc_base(sDO, SHORT_CHUNK, 1024), dp_mn = make_smem_desc_base(sP, SHORT_CHUNK, 1024);
      const SmemDescBase dds_mn = make_smem_desc_base(sDS, SHORT_CHUNK, 1024), dds_k = make_smem_desc_base(sDS, 16, 1024);
      uint32_t ph = 0;
      for (int item = blockIdx.x; item < nitems; item += gridDim.x, ph ^= 1u) {
        const int nb = item / H, h = item - nb * H, bs = nb % B;
        const int item1 = item + gridDim.x;
        const bool more = item1 < nitems;
        const int nb1 = item1 / H, h1 = item1 - nb1 * H, bs1 = nb1 % B;
        if (!more) grid_dep_launch();                           // this CTA's last loads have been issued
        if (!wait(B_Q, ph) || !wait(B_K, ph)) break;
        tc_fence_after();
#pragma unroll
        for (int ks = 0; ks < DH / 16; ++ks) {
          const uint32_t off = (ks >> 2) * SHORT_CHUNK + (ks & 3) * 32;
          umma_bf16(tmem + C::C_S, desc_at(dq_k, off), desc_at(dk_k, off), idesc_s, ks ? 1u : 0u);
        }
        umma_commit(bar(B_S));
        if (!wait(B_DO, ph)) break;
        if (!C::RING) {
          if (!wait(B_V0, ph)) break;
          tc_fence_after();
#pragma unroll
          for (int ks = 0; ks < DH / 16; ++ks) {
            const uint32_t off = (ks >> 2) * SHORT_CHUNK + (ks & 3) * 32;
            umma_bf16(tmem + C::C_DP, desc_at(ddo_k, off), desc_at(dv_k, off), idesc_s, ks ? 1u : 0u);
          }
        } else {
          for (int c = 0; c < C::NCH && !fail; ++c) {           // a chunk's barrier completes twice an item
            if (!wait(B_V0 + (c & 1), (uint32_t)(c >> 1) & 1u)) break;
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              umma_bf16(tmem + C::C_DP, desc_at(ddo_k, c * SHORT_CHUNK + ks * 32), desc_at(dv_k, (c & 1) * SHORT_CHUNK + ks * 32),
                        idesc_s, (c | ks) ? 1u : 0u);
            if (c < 2) umma_commit(bar(B_VF0 + c));
            if (c == 1)
              for (int q = 0; q < 2; ++q) {
                if (!wait(B_VF0 + q, ph)) break;
                load_v(2 + q, h, bs);
              }
          }
          if (fail) break;
        }
        umma_commit(bar(B_DP));
        if (!wait(B_P, ph)) break;
        tc_fence_after();
        for (int ks = 0; ks < nk; ++ks)
          umma_bf16(tmem + C::C_DV, desc_at(dp_mn, ks * 2048), desc_at(ddo_mn, ks * 2048), idesc_mn, ks ? 1u : 0u);
        umma_commit(bar(B_DV));
        if (!wait(B_DS, ph)) break;
        tc_fence_after();
        for (int ks = 0; ks < nk; ++ks)
          umma_bf16(tmem + C::C_DK, desc_at(dds_mn, ks * 2048), desc_at(dq_mn, ks * 2048), idesc_mn, ks ? 1u : 0u);
        umma_commit(bar(B_DK));
        auto issue_dq = [&]() {
          for (int ks = 0; ks < nk; ++ks)
            umma_bf16(tmem + C::C_DQ, desc_at(dds_k, (ks >> 2) * SHORT_CHUNK + (ks & 3) * 32), desc_at(dk_mn, ks * 2048), idesc_k,
                      ks ? 1u : 0u);
          umma_commit(bar(B_DQ));
        };
        if (!C::RING) issue_dq();
        if (more && !C::RING) load(sV, &tm_qkv, 2 * H + h1, bs1, B_V0);     // (dP is complete: P came from it)
        if (!wait(B_O0, ph)) break;
        if (C::RING) { tc_fence_after(); issue_dq(); }           // dV's columns are free
        store(sDO, 2 * H + h, nb);
        if (more) { bulk_wait_group_read0(); load(sDO, &tm_do, h1, nb1, B_DO); }
        if (!wait(B_O1, ph)) break;
        store(sQ, H + h, nb);
        if (more) { bulk_wait_group_read0(); load(sQ, &tm_qkv, h1, bs1, B_Q); }
        if (!wait(B_O2, ph)) break;
        if (C::RING && more) { load_v(0, h1, bs1); load_v(1, h1, bs1); }
        store(sK, h, nb);
        if (more) { bulk_wait_group_read0(); load(sK, &tm_qkv, H + h1, bs1, B_K); }
      }
      bulk_wait_group_read0();                                   // the stores have read this CTA's shared memory
      umma_commit(bar(B_DRAIN));                                 // every MMA issued has retired before TMEM goes
      int never = 0;
      mbar_wait(bar(B_DRAIN), 0, &never);
    }
  } else {
    const int hf = warp >> 2, row = (warp & 3) * 32 + lane;      // keys 64 hf .. 64 hf + 63 of query `row`
    const uint32_t t_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t swz = (uint32_t)(row & 7);
    const float c2 = scale * 1.4426950408889634f;
    const bool some = hf == 0 || (warp & 3) >= 2;                // (warp-uniform) any key of this half before any of these queries
    auto wait = [&](int b, uint32_t parity) -> bool { return __all_sync(0xffffffffu, mbar_wait(bar(b), parity, abortp)); };
    auto arrive = [&](int b) {
      fence_proxy_async();                                       // what was written to shared memory is read by MMA / TMA
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(b));
    };
    // 8 keys of this row, from key 64 hf + 8 u on, into chunk hf of a buffer
    auto put8 = [&](uint32_t buf, int u, const float (&x)[8]) {
      st_shared_v4(buf + hf * SHORT_CHUNK + row * 128 + (((uint32_t)u ^ swz) << 4), pack_bf16x2(x[0], x[1]), pack_bf16x2(x[2], x[3]),
                   pack_bf16x2(x[4], x[5]), pack_bf16x2(x[6], x[7]));
    };
    // meeting of the two warps that share these rows (a phase for "written", one for "read")
    auto meet = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(B_X + (warp & 3)));
    };
    // result columns (fp32 accumulator at tensor-memory column col) times f, as bf16, into the buffer of an operand
    auto put_result = [&](uint32_t col, uint32_t buf, float f) {
      constexpr int U = C::UNIT;
#pragma unroll 1
      for (int u = hf; u < DH / U; u += 2) {
        const int c0 = u * U;
        uint32_t v[U], w[U / 2];
        if constexpr (U == 32) tmem_ld_32x32(t_lane + col + c0, v);
        else tmem_ld_32x16(t_lane + col + c0, v);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < U / 2; ++i) w[i] = pack_bf16x2(__uint_as_float(v[2 * i]) * f, __uint_as_float(v[2 * i + 1]) * f);
        const uint32_t a = buf + (c0 >> 6) * SHORT_CHUNK + row * 128;
        const uint32_t u0 = (uint32_t)(c0 & 63) >> 3;
#pragma unroll
        for (int i = 0; i < U / 8; ++i) st_shared_v4(a + (((u0 + i) ^ swz) << 4), w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
      }
    };
    uint32_t ph = 0;
    for (int item = blockIdx.x; item < nitems; item += gridDim.x, ph ^= 1u) {
      const int nb = item / H, h = item - nb * H, bs = nb % B;
      const float lse2 = row < T ? lse[((size_t)bs * H + h) * T + row] * 1.4426950408889634f : 0.f;
      const int last = row < T ? row : -1;                       // last key this row sees
      float p[64];
      if (!wait(B_S, ph)) { fail = 1; break; }
      tc_fence_after();
      if (some) {
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          uint32_t v[16];
          tmem_ld_32x16(t_lane + C::C_S + 64 * hf + 16 * g, v);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float e = ex2_fast(fmaf(__uint_as_float(v[i]), c2, -lse2));
            p[16 * g + i] = 64 * hf + 16 * g + i <= last ? e : 0.f;
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < 64; ++i) p[i] = 0.f;
      }
      if (C::RING && !wait(B_DP, ph)) { fail = 1; break; }       // V has been read: P takes its place
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        float x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = p[8 * u + i];
        put8(base + C::O_P, u, x);
      }
      arrive(B_P);
      if (!C::RING && !wait(B_DP, ph)) { fail = 1; break; }
      tc_fence_after();
      // delta: the row's sum over both halves (tensor memory is read a second time below: 64 more values a thread would
      // not fit its registers).  Masked entries may hold anything, not-a-numbers included: selected, not multiplied, away.
      float part[4] = {0.f, 0.f, 0.f, 0.f};
      if (some) {
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          uint32_t v[16];
          tmem_ld_32x16(t_lane + C::C_DP + 64 * hf + 16 * g, v);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) part[i & 3] += 64 * hf + 16 * g + i <= last ? p[16 * g + i] * __uint_as_float(v[i]) : 0.f;
        }
      }
      if (item != (int)blockIdx.x && !wait(B_X + (warp & 3), 1u)) { fail = 1; break; }   // the last item's sums have been read
      s_part[hf * SHORT_ROWS + row] = (part[0] + part[1]) + (part[2] + part[3]);
      meet();
      if (!wait(B_X + (warp & 3), 0u)) { fail = 1; break; }
      const float delta = s_part[row] + s_part[SHORT_ROWS + row];
      meet();
      if (C::SHARED && !wait(B_DV, ph)) { fail = 1; break; }     // P has been read: dS takes its place
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        uint32_t v[16];
        if (some) {
          tmem_ld_32x16(t_lane + C::C_DP + 64 * hf + 16 * g, v);
          tmem_ld_wait();
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          float x[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int c = 16 * g + 8 * u + i;
            x[i] = some && 64 * hf + c <= last ? p[c] * (__uint_as_float(v[8 * u + i]) - delta) : 0.f;
          }
          put8(base + C::O_DS, 2 * g + u, x);
        }
      }
      arrive(B_DS);
      if (!C::SHARED && !wait(B_DV, ph)) { fail = 1; break; }
      tc_fence_after();
      put_result(C::C_DV, base + C::O_DO, 1.0f);
      arrive(B_O0);
      if (!wait(B_DK, ph)) { fail = 1; break; }
      tc_fence_after();
      put_result(C::C_DK, base + C::O_Q, scale);
      arrive(B_O1);
      if (!wait(B_DQ, ph)) { fail = 1; break; }
      tc_fence_after();
      put_result(C::C_DQ, base + C::O_K, scale);
      arrive(B_O2);
    }
    if (fail) abort_flag = 1;
  }
  fail = __syncthreads_or(fail);
  if (tid == 0 && fail && err) atomicExch(err, DEV_TIMEOUT_MMA);
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem, C::TCOLS);
  }
}

template <int DH>
cudaError_t launch(const bf16* qkv, const float* lse, const bf16* dout, bf16* dqkv, int NB, int B, int T, int H, unsigned* err,
                   cudaStream_t s) {
  using C = ShortCfg<DH>;
  const unsigned long long d3 = 3ull * H * DH, d1 = (unsigned long long)H * DH;
  const unsigned long long dims[4] = {(unsigned long long)DH, 3ull * H, (unsigned long long)T, (unsigned long long)B};
  const unsigned long long odims[4] = {(unsigned long long)DH, 3ull * H, (unsigned long long)T, (unsigned long long)NB};
  const unsigned long long strides[3] = {(unsigned long long)DH * 2, d3 * 2, (unsigned long long)T * d3 * 2};
  const unsigned long long ddims[4] = {(unsigned long long)DH, (unsigned long long)H, (unsigned long long)T, (unsigned long long)NB};
  const unsigned long long dstrides[3] = {(unsigned long long)DH * 2, d1 * 2, (unsigned long long)T * d1 * 2};
  const unsigned box[4] = {64, 1, (unsigned)((T + 15) / 16 * 16), 1};
  CUtensorMap tm_qkv, tm_do, tm_out;
  if (!tma_encode_bf16(&tm_qkv, qkv, 4, dims, strides, box) || !tma_encode_bf16(&tm_do, dout, 4, ddims, dstrides, box) ||
      !tma_encode_bf16(&tm_out, dqkv, 4, odims, strides, box))
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(attn_bwd_short_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const long long items = (long long)NB * H, slots = (long long)sms * C::CTAS;
  launch_dep(attn_bwd_short_kernel<DH>, dim3((unsigned)(items < slots ? items : slots)), dim3(SHORT_THREADS), C::SMEM, s, tm_qkv,
             tm_do, tm_out, lse, NB, B, T, H, rsqrtf((float)DH), err);
  return cudaGetLastError();
}

}  // namespace

cudaError_t attention_bwd_short(const bf16* qkv, const float* lse, const bf16* dout, bf16* dqkv, int NB, int B, int T, int H,
                                int dh, unsigned* err, cudaStream_t s) {
  if (T > ATTN_BWD_SHORT_T) return cudaErrorInvalidValue;
  switch (dh) {
    case 32: return launch<32>(qkv, lse, dout, dqkv, NB, B, T, H, err, s);
    case 64: return launch<64>(qkv, lse, dout, dqkv, NB, B, T, H, err, s);
    case 80: return launch<80>(qkv, lse, dout, dqkv, NB, B, T, H, err, s);
    case 128: return launch<128>(qkv, lse, dout, dqkv, NB, B, T, H, err, s);
    case 256: return launch<256>(qkv, lse, dout, dqkv, NB, B, T, H, err, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace il
