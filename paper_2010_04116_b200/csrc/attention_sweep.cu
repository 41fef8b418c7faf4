// Causal self-attention backward with sums of fixed order (sm_100a), head dimensions up to 128: one kernel for dV and dK, one for
// dQ, both instances of the same sweep.
//
// A CTA owns 128 rows (keys for dV / dK, queries for dQ) of one (gradient sequence, head) and sweeps the other index in blocks of
// 64.  Row operands R1, R2 (K, V / Q, dO) stay in shared memory; the swept tiles W1, W2 (Q, dO / K, V) come through a ring of four
// TMA stages.  Per step j
//   S = R1 W1^T, dP = R2 W2^T      M128 N64, both operands K-major, into score buffer j % 2 of tensor memory
//   P = exp(scale S - lse), dS = P (dP - delta)     two threads per row, 32 columns each; rounded to bf16 and stored, packed, over
//                                  the score columns the thread has read
//   dV += P W2, dK += dS W1  /  dQ += dS W1         A from those columns, B MN-major; accumulated in tensor memory over the sweep
// Warps 0-15 do the row work, a thread each of warps 16 and 17 issues MMAs, warp 18 loads (and, for dV / dK, puts the swept queries' lse
// and delta into shared memory).  With two score buffers the scores of step j + 1 are ready when the row work of step j ends, and
// the tensor pipe runs step j's products and the scores of step j + 2 meanwhile.  Tensor memory: 2 x 128 score columns and one or
// two accumulators of dh: one CTA per SM.  Items are numbered so that the longest sweeps start first.
//
// What bounds it: the issuing threads.  A thread issues an MMA of this size no faster than every 60 cycles wherever A comes
// from, a commit costs it 120, a look at a barrier 150 beside the busy pipe; a step of dQ at dh 128
// takes 1440 cycles (one issuing thread: 1810), of which a row-work warp is busy 880.  Short sweeps pay 5 us an item for set-up,
// first loads and output.
// Measured, delta included (gradient sequences x heads x T, dh), us; the synchronous two-kernel form before it / this one:
//   1 x 8 x 4096, dh 128  333 / 126      2 x 32 x 2048, dh 80  490 / 262      8 x 16 x 1024, dh 64  180 / 165
//   16 x 16 x 1024, dh 64  323 / 323     1 x 12 x 256, dh 64  20.8 / 17.0     2 x 4 x 129, dh 64  17.7 / 16.3
#include "common.cuh"
#include "kernels.h"
#include "tma.h"

namespace il {

namespace {

constexpr int SW_ROWS = 128;           // rows of a CTA
constexpr int SW_COLS = 64;            // positions per step
constexpr int SW_WARPS = 16;           // row-work warps
constexpr int SW_THREADS = 32 * (SW_WARPS + 3);
constexpr int SW_STAGES = 4;

template <int DH>
struct SweepCfg {
  static constexpr int NCH = (DH + 63) / 64;
  static constexpr int ROW_BYTES = NCH * SW_ROWS * 128;
  static constexpr int BLK_BYTES = NCH * SW_COLS * 128;
  static constexpr int VEC_BYTES = 2 * SW_COLS * 4;             // lse (log2 units), delta of a step's queries
  static constexpr int O_RING = 2 * ROW_BYTES, O_VEC = O_RING + SW_STAGES * 2 * BLK_BYTES, O_BARS = O_VEC + SW_STAGES * VEC_BYTES;
  static constexpr int SMEM = 1024 + O_BARS + 256;
  static constexpr int C_ACC = 256;                             // score buffer b: S at 128 b, dP at 128 b + 64
};

// KV: rows are keys, results dV and dK; otherwise rows are queries, result dQ.
template <int DH, bool KV>
__global__ void __launch_bounds__(SW_THREADS, 1)
attn_bwd_sweep_kernel(const __grid_constant__ CUtensorMap tm_row, const __grid_constant__ CUtensorMap tm_blk,
                      const __grid_constant__ CUtensorMap tm_do, const float* __restrict__ lse, const float* __restrict__ delta,
                      bf16* __restrict__ dqkv, int NB, int B, int T, int H, float scale, unsigned* err) {
  using C = SweepCfg<DH>;
  // The row operands as the score products' A operand from tensor memory, where the columns suffice.  With two issuing threads
  // the shared-memory reads of the operands begin to show (us, cold cache, from tensor / from shared memory: 8 x 16 x 1024,
  // dh 64 174.1 / 177.2; 16 x 16 x 1024 330.8 / 338.9; 2 x 32 x 2048, dh 80 271.4 / 272.4; 1 x 8 x 4096, dh 128 133.8 / 134.2); with
  // one it was the other way round.
  constexpr uint32_t C_ROW = C::C_ACC + (KV ? 2 : 1) * DH;
  constexpr bool ROWS_IN_TMEM = C_ROW + DH <= 512;
  extern __shared__ uint8_t smem_raw[];
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_smem;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sR1 = base, sR2 = base + C::ROW_BYTES, sRing = base + C::O_RING, bars = base + C::O_BARS;
  float* s_vec = reinterpret_cast<float*>(smem_raw + (base - smem_u32(smem_raw)) + C::O_VEC);     // [stage][lse, delta][64]
  const uint32_t bar_row = bars, bar_acc = bars + 8, bar_copied = bars + 16;
  auto bar_drain = [&](int x) { return bars + 24 + 8 * x; };
  auto bar_full = [&](int st) { return bars + 40 + 8 * st; };
  auto bar_empty = [&](int st) { return bars + 40 + 8 * (SW_STAGES + st); };
  auto bar_vec = [&](int st) { return bars + 40 + 8 * (2 * SW_STAGES + st); };
  auto bar_s = [&](int b) { return bars + 40 + 8 * (3 * SW_STAGES + b); };        // scores in buffer b
  auto bar_p = [&](int b) { return bars + 40 + 8 * (3 * SW_STAGES + 2 + b); };    // ... turned into P / dS

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nbh = NB * H, tiles = (T + SW_ROWS - 1) / SW_ROWS, blocks = (T + SW_COLS - 1) / SW_COLS;
  const int rank = blockIdx.x / nbh, which = blockIdx.x - rank * nbh;
  const int tile = KV ? rank : tiles - 1 - rank;                // (the sweeps over many blocks come first)
  const int nb = which / H, h = which - nb * H, bs = nb % B;
  const int j0 = KV ? 2 * tile : 0;                             // blocks j0 .. j0 + n - 1 see these rows
  const int n = KV ? blocks - j0 : min(2 * tile + 2, blocks);
  volatile int* abortp = &abort_flag;

  if (tid == 0) {
    abort_flag = 0;
    mbar_init(bar_row, 1);
    mbar_init(bar_acc, 2);               // the two issuing threads
    mbar_init(bar_drain(0), 1);
    mbar_init(bar_drain(1), 1);
    mbar_init(bar_copied, SW_WARPS);
    for (int st = 0; st < SW_STAGES; ++st) { mbar_init(bar_full(st), 1); mbar_init(bar_empty(st), 2); mbar_init(bar_vec(st), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(bar_s(b), 2); mbar_init(bar_p(b), SW_WARPS / 2); }
    fence_mbar_init();
    tma_prefetch_desc(&tm_row);
    tma_prefetch_desc(&tm_blk);
    tma_prefetch_desc(&tm_do);
  }
  if (warp == SW_WARPS) {
    tmem_alloc(smem_u32(&tmem_base_smem), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dep_wait();
  const uint32_t tmem = tmem_base_smem;
  int fail = 0;

  if (warp == SW_WARPS + 2) {
    // ---------------------------------------------------------------- loads
    if (lane == 0) {
      mbar_expect_tx(bar_row, 2 * C::ROW_BYTES);
#pragma unroll
      for (int c = 0; c < C::NCH; ++c) {
        tma_load_4d(sR1 + c * (SW_ROWS * 128), &tm_row, c * 64, KV ? H + h : h, tile * SW_ROWS, bs, bar_row);
        if (KV) tma_load_4d(sR2 + c * (SW_ROWS * 128), &tm_row, c * 64, 2 * H + h, tile * SW_ROWS, bs, bar_row);
        else tma_load_4d(sR2 + c * (SW_ROWS * 128), &tm_do, c * 64, h, tile * SW_ROWS, nb, bar_row);
      }
    }
    const float* lse_b = lse + ((size_t)bs * H + h) * T;
    const float* del_b = delta + ((size_t)nb * H + h) * T;
    for (int j = 0; j < n; ++j) {
      const int st = j % SW_STAGES, at = (j0 + j) * SW_COLS;
      if (j >= SW_STAGES && !__all_sync(0xffffffffu, mbar_wait(bar_empty(st), (uint32_t)(j / SW_STAGES - 1) & 1u, abortp))) { fail = 1; break; }
      if (lane == 0) {
        const uint32_t w1 = sRing + st * 2 * C::BLK_BYTES, w2 = w1 + C::BLK_BYTES;
        mbar_expect_tx(bar_full(st), 2 * C::BLK_BYTES);
#pragma unroll
        for (int c = 0; c < C::NCH; ++c) {
          tma_load_4d(w1 + c * (SW_COLS * 128), &tm_blk, c * 64, KV ? h : H + h, at, bs, bar_full(st));
          if (KV) tma_load_4d(w2 + c * (SW_COLS * 128), &tm_do, c * 64, h, at, nb, bar_full(st));
          else tma_load_4d(w2 + c * (SW_COLS * 128), &tm_blk, c * 64, 2 * H + h, at, bs, bar_full(st));
        }
      }
      if (KV) {
        float* v = s_vec + st * 2 * SW_COLS;
#pragma unroll
        for (int i = lane; i < SW_COLS; i += 32) {
          const bool in = at + i < T;
          const float a = in ? lse_b[at + i] * 1.4426950408889634f : 0.f, b = in ? del_b[at + i] : 0.f;
          v[i] = a;
          v[SW_COLS + i] = b;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_vec(st));
      }
    }
    grid_dep_launch();
    if (fail) abort_flag = 1;
  } else if (warp >= SW_WARPS) {
    // ---------------------------------------------------------------- MMA issue
    // One thread takes S and dV, another dP and dK / dQ.  Each accumulator belongs to one thread, so its sums keep their order.
    if (lane == 0) {
      constexpr uint32_t idesc_s = make_idesc_bf16(SW_ROWS, SW_COLS, 0, 0), idesc_g = make_idesc_bf16(SW_ROWS, DH, 0, 1);
      const int x = warp - SW_WARPS;                            // 0: S, dV from P; 1: dP, dK or dQ from dS
      const SmemDescBase rows = make_smem_desc_base(x ? sR2 : sR1, 16, 1024);
      const SmemDescBase cols = make_smem_desc_base(sRing + (x ? C::BLK_BYTES : 0), 16, 1024);
      const SmemDescBase other = make_smem_desc_base(sRing + (x ? 0 : C::BLK_BYTES), SW_COLS * 128, 1024);     // W1 for dS, W2 for P
      const uint32_t t_rows = tmem + C_ROW + (uint32_t)x * (DH / 2), t_acc = tmem + C::C_ACC + (KV ? (uint32_t)x * DH : 0u);
      const bool sums = KV || x == 1;
      auto loaded = [&](int j) -> bool { return mbar_wait(bar_full(j % SW_STAGES), (uint32_t)(j / SW_STAGES) & 1u, abortp); };
      auto scores = [&](int j) {
        const uint32_t so = (uint32_t)(j % SW_STAGES) * 2 * C::BLK_BYTES, t_s = tmem + 128 * (j & 1) + 64 * x;
#pragma unroll
        for (int ks = 0; ks < DH / 16; ++ks) {
          const uint32_t off_w = so + (ks >> 2) * (SW_COLS * 128) + (ks & 3) * 32;
          if constexpr (ROWS_IN_TMEM) umma_bf16_ts(t_s, t_rows + 8 * ks, desc_at(cols, off_w), idesc_s, ks ? 1u : 0u);
          else umma_bf16(t_s, desc_at(rows, (ks >> 2) * (SW_ROWS * 128) + (ks & 3) * 32), desc_at(cols, off_w), idesc_s, ks ? 1u : 0u);
        }
        umma_commit(bar_s(j & 1));
      };
      bool ok = mbar_wait(ROWS_IN_TMEM ? bar_copied : bar_row, 0, abortp) && loaded(0);
      tc_fence_after();
      if (ok) scores(0);
      if (ok && n > 1) { ok = loaded(1); if (ok) scores(1); }
      for (int j = 0; j < n && ok; ++j) {
        const int st = j % SW_STAGES;
        if (j + 2 < n && !loaded(j + 2)) { ok = false; break; }
        if (!mbar_wait(bar_p(j & 1), (uint32_t)(j >> 1) & 1u, abortp)) { ok = false; break; }
        tc_fence_after();
        if (sums) {
          const uint32_t so = (uint32_t)st * 2 * C::BLK_BYTES, t_s = tmem + 128 * (j & 1) + 64 * x;
#pragma unroll
          for (int ks = 0; ks < SW_COLS / 16; ++ks)             // packed K-step ks: 8 columns of a 32-column half
            umma_bf16_ts(t_acc, t_s + (uint32_t)((ks >> 1) * 32 + (ks & 1) * 8), desc_at(other, so + ks * 2048), idesc_g, (j | ks) ? 1u : 0u);
        }
        umma_commit(bar_empty(st));
        if (j + 2 < n) scores(j + 2);                           // behind the products that read these columns, in pipe order
      }
      umma_commit(bar_acc);
      if (!ok) { fail = 1; abort_flag = 1; }
      umma_commit(bar_drain(x));                                // every MMA issued has retired before TMEM goes
      int never = 0;
      mbar_wait(bar_drain(x), 0, &never);
    }
  } else {
    // ---------------------------------------------------------------- row work: thread = row r, columns 32 hf .. 32 hf + 31
    // Warps 0-7 take the even steps, 8-15 the odd ones: two steps are in hand at a time.
    const int g = warp >> 2, hf = g & 1, r = (warp & 3) * 32 + lane;
    const uint32_t t_lane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const float c2 = scale * 1.4426950408889634f;
    const int row = tile * SW_ROWS + r;
    auto wait = [&](uint32_t bar, uint32_t parity) -> bool { return __all_sync(0xffffffffu, mbar_wait(bar, parity, abortp)); };
    float lse2 = 0.f, del = 0.f;
    if (!KV && row < T) {
      lse2 = lse[((size_t)bs * H + h) * T + row] * 1.4426950408889634f;
      del = delta[((size_t)nb * H + h) * T + row];
    }
    if constexpr (ROWS_IN_TMEM) {
      // this row of R1 (threads of hf 0) and of R2 (hf 1), groups of 16 columns in turn between the two warps of a half
      if (!wait(bar_row, 0)) fail = 1;
      const uint32_t src = (hf ? sR2 : sR1) + r * 128, dst = t_lane + C_ROW + hf * (DH / 2);
#pragma unroll
      for (int c = 0; c < DH / 16; ++c) {
        if ((c & 1) != (g >> 1)) continue;
        uint32_t v[8];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const uint32_t at = src + (c >> 2) * (SW_ROWS * 128) + (((uint32_t)((c & 3) * 2 + u) ^ (uint32_t)(r & 7)) << 4);
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[4 * u]), "=r"(v[4 * u + 1]), "=r"(v[4 * u + 2]), "=r"(v[4 * u + 3]) : "r"(at));
        }
        tmem_st_32x8(dst + 8 * c, v);
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_copied);
    }
    const int b = g >> 1;
    const uint32_t t_s = t_lane + 128 * b + 32 * hf;
    for (int j = b; j < n; j += 2) {
      const int st = j % SW_STAGES;
      if (KV && !wait(bar_vec(st), (uint32_t)(j / SW_STAGES) & 1u)) { fail = 1; break; }
      if (!wait(bar_s(b), (uint32_t)(j >> 1) & 1u)) { fail = 1; break; }
      tc_fence_after();
      uint32_t s[32], dp[32];
      tmem_ld_32x32(t_s, s);
      tmem_ld_32x32(t_s + 64, dp);
      tmem_ld_wait();
      const float4* lv = reinterpret_cast<const float4*>(s_vec + st * 2 * SW_COLS + 32 * hf);
      const float4* dv = reinterpret_cast<const float4*>(s_vec + st * 2 * SW_COLS + SW_COLS + 32 * hf);
      const int at = (j0 + j) * SW_COLS + 32 * hf;
      float p[32];
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        float4 l = make_float4(lse2, lse2, lse2, lse2);
        if (KV) l = lv[i / 4];
        p[i] = ex2_fast(fmaf(__uint_as_float(s[i]), c2, -l.x));
        p[i + 1] = ex2_fast(fmaf(__uint_as_float(s[i + 1]), c2, -l.y));
        p[i + 2] = ex2_fast(fmaf(__uint_as_float(s[i + 2]), c2, -l.z));
        p[i + 3] = ex2_fast(fmaf(__uint_as_float(s[i + 3]), c2, -l.w));
      }
      // (uniform) blocks on the diagonal, and for swept queries the one past the sequence's end
      if (KV ? (j < 2 || (j0 + j + 1) * SW_COLS > T) : (j0 + j + 1) * SW_COLS > tile * SW_ROWS) {
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (KV ? (at + i < row || at + i >= T) : at + i > row) p[i] = 0.f;
      }
      uint32_t w[16];
      if (KV) {
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = pack_bf16x2(p[2 * i], p[2 * i + 1]);
        tmem_st_32x16(t_s, w);                     // P over the first half of the columns this thread has read
      }
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        float4 e = make_float4(del, del, del, del);
        if (KV) e = dv[i / 4];
        w[i / 2] = pack_bf16x2(p[i] * (__uint_as_float(dp[i]) - e.x), p[i + 1] * (__uint_as_float(dp[i + 1]) - e.y));
        w[i / 2 + 1] = pack_bf16x2(p[i + 2] * (__uint_as_float(dp[i + 2]) - e.z), p[i + 3] * (__uint_as_float(dp[i + 3]) - e.w));
      }
      tmem_st_32x16(t_s + 64, w);                  // dS likewise
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_p(b));
    }
    if (!fail && !wait(bar_acc, 0)) fail = 1;
    tc_fence_after();
    if (fail) {
      abort_flag = 1;
    } else {
      const int d = H * DH;
      bf16* out = dqkv + ((size_t)nb * T + row) * (3 * d) + h * DH;
      constexpr int PER = DH / 16, UNITS = (KV ? 2 : 1) * PER;  // 16-column units, shared out among the row's four threads
#pragma unroll
      for (int u0 = 0; u0 < UNITS; u0 += 4) {
        const int u = u0 + g;
        if (u >= UNITS) break;                                  // uniform across the warp
        uint32_t v[16];
        tmem_ld_32x16(t_lane + C::C_ACC + 16 * u, v);
        tmem_ld_wait();
        const float f = KV && u < PER ? 1.0f : scale;
        bf16* dst = out + (KV ? (u < PER ? 2 * d + 16 * u : d + 16 * (u - PER)) : 16 * u);
        if (row < T) {
#pragma unroll
          for (int i = 0; i < 16; i += 8) {
            uint4 pk;
            pk.x = pack_bf16x2(__uint_as_float(v[i]) * f, __uint_as_float(v[i + 1]) * f);
            pk.y = pack_bf16x2(__uint_as_float(v[i + 2]) * f, __uint_as_float(v[i + 3]) * f);
            pk.z = pack_bf16x2(__uint_as_float(v[i + 4]) * f, __uint_as_float(v[i + 5]) * f);
            pk.w = pack_bf16x2(__uint_as_float(v[i + 6]) * f, __uint_as_float(v[i + 7]) * f);
            *reinterpret_cast<uint4*>(dst + i) = pk;
          }
        }
      }
    }
  }
  fail = __syncthreads_or(fail);
  if (tid == 0 && fail && err) atomicExch(err, DEV_TIMEOUT_MMA);
  tc_fence_before();
  __syncthreads();
  if (warp == SW_WARPS) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

template <int DH>
cudaError_t launch(const bf16* qkv, const float* lse, const bf16* dout, bf16* dqkv, const float* delta, int NB, int B, int T, int H,
                   unsigned* err, cudaStream_t s) {
  using C = SweepCfg<DH>;
  const unsigned long long d3 = 3ull * H * DH, d1 = (unsigned long long)H * DH;
  const unsigned long long dims[4] = {(unsigned long long)DH, 3ull * H, (unsigned long long)T, (unsigned long long)B};
  const unsigned long long strides[3] = {(unsigned long long)DH * 2, d3 * 2, (unsigned long long)T * d3 * 2};
  const unsigned long long ddims[4] = {(unsigned long long)DH, (unsigned long long)H, (unsigned long long)T, (unsigned long long)NB};
  const unsigned long long dstrides[3] = {(unsigned long long)DH * 2, d1 * 2, (unsigned long long)T * d1 * 2};
  const unsigned box_row[4] = {64, 1, SW_ROWS, 1}, box_blk[4] = {64, 1, SW_COLS, 1};
  CUtensorMap tm_row, tm_blk, tm_do_row, tm_do_blk;
  if (!tma_encode_bf16(&tm_row, qkv, 4, dims, strides, box_row) || !tma_encode_bf16(&tm_blk, qkv, 4, dims, strides, box_blk) ||
      !tma_encode_bf16(&tm_do_row, dout, 4, ddims, dstrides, box_row) || !tma_encode_bf16(&tm_do_blk, dout, 4, ddims, dstrides, box_blk))
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(attn_bwd_sweep_kernel<DH, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(attn_bwd_sweep_kernel<DH, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  const long long items = (long long)((T + SW_ROWS - 1) / SW_ROWS) * NB * H;
  if (items > 0x7fffffff) return cudaErrorInvalidValue;
  const float scale = rsqrtf((float)DH);
  launch_dep(attn_bwd_sweep_kernel<DH, true>, dim3((unsigned)items), dim3(SW_THREADS), C::SMEM, s, tm_row, tm_blk, tm_do_blk, lse, delta,
             dqkv, NB, B, T, H, scale, err);
  launch_dep(attn_bwd_sweep_kernel<DH, false>, dim3((unsigned)items), dim3(SW_THREADS), C::SMEM, s, tm_row, tm_blk, tm_do_row, lse, delta,
             dqkv, NB, B, T, H, scale, err);
  return cudaGetLastError();
}

}  // namespace

cudaError_t attention_bwd_sweep(const bf16* qkv, const float* lse, const bf16* dout, bf16* dqkv, const float* delta, int NB, int B,
                                int T, int H, int dh, unsigned* err, cudaStream_t s) {
  switch (dh) {
    case 32: return launch<32>(qkv, lse, dout, dqkv, delta, NB, B, T, H, err, s);
    case 64: return launch<64>(qkv, lse, dout, dqkv, delta, NB, B, T, H, err, s);
    case 80: return launch<80>(qkv, lse, dout, dqkv, delta, NB, B, T, H, err, s);
    case 128: return launch<128>(qkv, lse, dout, dqkv, delta, NB, B, T, H, err, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace il
