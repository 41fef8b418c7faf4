// Causal self-attention forward on the tcgen05 tensor cores (sm_100a).
//
// One CTA owns 128 query rows of one (sequence, head) and sweeps the keys in blocks of 64.  Q, K and V
// tiles come in by TMA from the packed qkv tensor viewed as a 4-D tensor (column within head, head slot,
// position, sequence) so that head selection, the ragged last rows of a sequence and head dimensions
// that are not a multiple of 64 are all handled by the tensor map's bounds (zero fill).  Per key block:
//   S = Q K^T        tcgen05.mma (M128 N64, both operands K-major in shared memory) -> TMEM columns [0, 64)
//   softmax          thread r owns query row r: tcgen05.ld its 64 scores, running max / sum in registers
//                    (no cross-lane reduction), P = exp2(...) rounded to bf16, packed in pairs and stored back
//                    over the first 32 of the score columns (tcgen05.st)
//   O += P V         tcgen05.mma (M128 N=dh, A = P read from TMEM, B = V MN-major), accumulated in TMEM columns
//                    [64, 64+dh).  The reference maximum of a row is raised only when a block exceeds it by a
//                    factor 2^8, so the accumulator is rescaled (tcgen05.ld / st) rarely.
// A CTA runs these phases one after the other; several CTAs are resident per SM (128 threads, 64-144 KB of
// shared memory, 128-256 TMEM columns each), which is what overlaps one CTA's softmax with another's MMAs.
// K and V come through a ring of TMA stages filled two or more sweep steps ahead.
// The T x T score matrix is never stored.  Every wait is bounded.
#include "common.cuh"
#include "kernels.h"
#include "tma.h"

namespace il {

namespace {

constexpr int TQ = 128;     // query rows per CTA
constexpr int TK = 64;      // keys per sweep step
#define IL_LOG2E 1.4426950408889634f

template <int DH>
struct FwdCfg {
  static constexpr int NCH = (DH + 63) / 64;            // 64-column chunks of the head dimension
  static constexpr int Q_BYTES = NCH * TQ * 128;
  static constexpr int KV_BYTES = NCH * TK * 128;
  static constexpr int NST = (DH <= 64) ? 3 : 2;               // K/V ring depth: as deep as keeps three (dh <= 64) or two CTAs per SM
  static constexpr int TCOLS = (64 + DH <= 128) ? 128 : (64 + DH <= 256) ? 256 : 512;   // 64 score columns + the O accumulator
  static constexpr int SMEM = Q_BYTES + NST * 2 * KV_BYTES + 1024 + 128;
};

template <int DH>
__global__ void __launch_bounds__(128) attn_fwd_tc_kernel(const __grid_constant__ CUtensorMap tmQ,
                                                          const __grid_constant__ CUtensorMap tmKV, bf16* __restrict__ o,
                                                          float* __restrict__ lse, int T, int H, float scale, unsigned* err) {
  using C = FwdCfg<DH>;
  constexpr int NST = C::NST;
  extern __shared__ uint8_t smem_raw[];
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_smem;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sQ = base;
  const uint32_t sK0 = sQ + C::Q_BYTES;                       // the K stages, then the V stages
  const uint32_t sV0 = sK0 + NST * C::KV_BYTES;
  const uint32_t bars = sV0 + NST * C::KV_BYTES;
  const uint32_t bar_q = bars, bar_s = bars + 8, bar_o = bars + 16, bar_drain = bars + 24, bar_kv0 = bars + 32;

  const int tid = threadIdx.x, warp = tid >> 5;
  const int qb = gridDim.x - 1 - blockIdx.x;                  // longest sweeps first
  const int b = blockIdx.y / H, h = blockIdx.y % H;
  const int d = H * DH;
  const int row = qb * TQ + tid;                              // query position of this thread
  int nkv = (qb * TQ + TQ + TK - 1) / TK;
  const int nkv_all = (T + TK - 1) / TK;
  if (nkv > nkv_all) nkv = nkv_all;

  if (tid == 0) {
    abort_flag = 0;
    mbar_init(bar_q, 1);
    for (int s = 0; s < NST; ++s) mbar_init(bar_kv0 + 8 * s, 1);
    mbar_init(bar_s, 1);
    mbar_init(bar_o, 1);
    mbar_init(bar_drain, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmQ);
    tma_prefetch_desc(&tmKV);
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(&tmem_base_smem), C::TCOLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dep_wait();
  const uint32_t tmem_base = tmem_base_smem;                  // scores at columns [0, 64) (then P packed in [0, 32)), O at [64, 64 + dh)
  const uint32_t t_lane = tmem_base + ((uint32_t)(warp * 32) << 16);
  volatile int* abortp = &abort_flag;
  constexpr uint32_t idesc_s = make_idesc_bf16(TQ, TK, 0, 0);
  constexpr uint32_t idesc_o = make_idesc_bf16(TQ, DH, 0, 1);
  int fail = 0;

  auto load_kv = [&](int j) {
    const int st = j % NST;
    mbar_expect_tx(bar_kv0 + 8 * st, 2 * C::KV_BYTES);
#pragma unroll
    for (int c = 0; c < C::NCH; ++c) {
      tma_load_4d(sK0 + st * C::KV_BYTES + c * (TK * 128), &tmKV, c * 64, H + h, j * TK, b, bar_kv0 + 8 * st);
      tma_load_4d(sV0 + st * C::KV_BYTES + c * (TK * 128), &tmKV, c * 64, 2 * H + h, j * TK, b, bar_kv0 + 8 * st);
    }
  };
  if (tid == 0) {
    mbar_expect_tx(bar_q, C::Q_BYTES);
#pragma unroll
    for (int c = 0; c < C::NCH; ++c) tma_load_4d(sQ + c * (TQ * 128), &tmQ, c * 64, h, qb * TQ, b, bar_q);
    for (int i = 0; i < NST; ++i)
      if (i < nkv) load_kv(i);
  }

  const float c2 = scale * IL_LOG2E;
  // Running statistics of this thread's row.  m is the reference maximum the exponentials are taken against; it
  // is only raised when a block's maximum exceeds it by more than 8 (in log2 units), so that the accumulator in
  // TMEM rarely needs rescaling; l and O stay consistent with whatever m is, and O / l is exact either way.
  float m = -INFINITY, l = 0.f;
  const float slack = 8.0f / c2;

  // S_j = Q K_j^T; issued by thread 0 one step ahead (right after the previous block's P V) so that each sweep
  // step waits for the tensor pipe only once
  // descriptors of the operands at their first stage; a sweep step adds its stage's offset (one add per MMA:
  // the issuing thread's own instruction stream is on every step's critical path)
  const SmemDescBase dq_k = make_smem_desc_base(sQ, 16, 1024), dk_k = make_smem_desc_base(sK0, 16, 1024);
  const SmemDescBase dv_mn = make_smem_desc_base(sV0, TK * 128, 1024);
  auto issue_s = [&](int j) {
    const int st = j % NST;
    if (!mbar_wait(bar_kv0 + 8 * st, (uint32_t)(j / NST) & 1u, abortp)) { fail = 1; abort_flag = 1; }
    tc_fence_after();
    const uint32_t so = (uint32_t)(st * C::KV_BYTES);
#pragma unroll
    for (int ks = 0; ks < DH / 16; ++ks)
      umma_bf16(tmem_base, desc_at(dq_k, (ks >> 2) * (TQ * 128) + (ks & 3) * 32),
                desc_at(dk_k, so + (ks >> 2) * (TK * 128) + (ks & 3) * 32), idesc_s, ks ? 1u : 0u);
    umma_commit(bar_s);
  };
  if (tid == 0) {
    if (!mbar_wait(bar_q, 0, abortp)) { fail = 1; abort_flag = 1; }
    issue_s(0);
  }

  for (int j = 0; j < nkv; ++j) {
    const int st = j % NST;
    const uint32_t ph = (uint32_t)j & 1u;
    if (!mbar_wait(bar_s, ph, abortp)) { fail = 1; abort_flag = 1; }
    // the previous block's P V was issued before these scores and the tensor pipe retires in order, so it has
    // landed too (bar_s covers it; only the last P V is committed on its own): the packed P columns, the O
    // accumulator and that block's K/V stage are free
    if (j > 0) {
      if (tid == 0 && j - 1 + NST < nkv) load_kv(j - 1 + NST);
    }
    tc_fence_after();
    // ---- softmax of this thread's row over the 64 keys of the block
    uint32_t r0[32], r1[32];
    tmem_ld_32x32(t_lane, r0);
    tmem_ld_32x32(t_lane + 32, r1);
    tmem_ld_wait();
    float s[64];
#pragma unroll
    for (int i = 0; i < 32; ++i) { s[i] = __uint_as_float(r0[i]); s[32 + i] = __uint_as_float(r1[i]); }
    if (j * TK + TK - 1 > qb * TQ) {              // block touches the diagonal: mask keys after the query
#pragma unroll
      for (int i = 0; i < 64; ++i)
        if (j * TK + i > row) s[i] = -INFINITY;
    }
    float mx4[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
    for (int i = 4; i < 64; i += 4) {
      mx4[0] = fmaxf(mx4[0], s[i]); mx4[1] = fmaxf(mx4[1], s[i + 1]);
      mx4[2] = fmaxf(mx4[2], s[i + 2]); mx4[3] = fmaxf(mx4[3], s[i + 3]);
    }
    const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
    if (__any_sync(0xffffffffu, mx > m + slack)) {            // warp-uniform: raise the reference maximum
      const float mn = fmaxf(m, mx);
      const float alpha = ex2_fast((m - mn) * c2);            // 0 on the first block (m = -inf)
      l *= alpha;
      m = mn;
      if (j > 0) {
#pragma unroll
        for (int c0 = 0; c0 < DH; c0 += 32) {
          if (c0 + 32 <= DH) {
            uint32_t r[32];
            tmem_ld_32x32(t_lane + 64 + c0, r);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * alpha);
            tmem_st_32x32(t_lane + 64 + c0, r);
          } else {
            uint32_t r[16];
            tmem_ld_32x16(t_lane + 64 + c0, r);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) * alpha);
            tmem_st_32x16(t_lane + 64 + c0, r);
          }
        }
        tmem_st_wait();
      }
    }
    const float mc = m * c2;
    float ps4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 64; i += 4) {
      s[i] = ex2_fast(fmaf(s[i], c2, -mc)); s[i + 1] = ex2_fast(fmaf(s[i + 1], c2, -mc));
      s[i + 2] = ex2_fast(fmaf(s[i + 2], c2, -mc)); s[i + 3] = ex2_fast(fmaf(s[i + 3], c2, -mc));
      ps4[0] += s[i]; ps4[1] += s[i + 1]; ps4[2] += s[i + 2]; ps4[3] += s[i + 3];
    }
    l += (ps4[0] + ps4[1]) + (ps4[2] + ps4[3]);
    // P (bf16 pairs, even key in the low half) over the first 32 score columns of this thread's lane
    {
      uint32_t pw[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) pw[i] = pack_bf16x2(s[2 * i], s[2 * i + 1]);
      tmem_st_32x32(t_lane, pw);
      tmem_st_wait();
    }
    tc_fence_before();
    if (__syncthreads_or(fail)) { fail = 1; break; }     // uniform exit if any thread's wait expired
    if (tid == 0) {
      tc_fence_after();
      const uint32_t so = (uint32_t)(st * C::KV_BYTES);
#pragma unroll
      for (int ks = 0; ks < TK / 16; ++ks)       // B = V read MN-major; O accumulates in TMEM
        umma_bf16_ts(tmem_base + 64, tmem_base + 8 * ks, desc_at(dv_mn, so + ks * 2048), idesc_o, (j | ks) ? 1u : 0u);
      // every thread has read S_j (barrier above); the tensor pipe runs the P V just issued, which reads the
      // packed columns, before it overwrites them with the next scores
      if (j + 1 < nkv) issue_s(j + 1);
      else umma_commit(bar_o);
    }
  }
  grid_dep_launch();
  if (!fail && nkv > 0) {
    if (!mbar_wait(bar_o, 0, abortp)) { fail = 1; abort_flag = 1; }
    tc_fence_after();
  }
  fail = __syncthreads_or(fail);
  if (!fail) {
    const float inv = 1.0f / l;
    bf16* orow = o + ((size_t)b * T + row) * d + h * DH;
#pragma unroll
    for (int c0 = 0; c0 < DH; c0 += 32) {
      float v[32];
      if (c0 + 32 <= DH) {
        uint32_t r[32];
        tmem_ld_32x32(t_lane + 64 + c0, r);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]) * inv;
      } else {
        uint32_t r[16];
        tmem_ld_32x16(t_lane + 64 + c0, r);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]) * inv;
      }
      if (row < T) {
#pragma unroll
        for (int i = 0; i < 32 && c0 + i < DH; i += 8) {
          uint4 pk;
          pk.x = pack_bf16x2(v[i], v[i + 1]);
          pk.y = pack_bf16x2(v[i + 2], v[i + 3]);
          pk.z = pack_bf16x2(v[i + 4], v[i + 5]);
          pk.w = pack_bf16x2(v[i + 6], v[i + 7]);
          *reinterpret_cast<uint4*>(orow + c0 + i) = pk;
        }
      }
    }
    if (row < T) lse[((size_t)b * H + h) * T + row] = m * scale + logf(l);
  }
  if (tid == 0) {
    if (fail && err) atomicExch(err, DEV_TIMEOUT_MMA);
    umma_commit(bar_drain);                      // every MMA issued by this CTA has retired before TMEM goes
    int never = 0;
    mbar_wait(bar_drain, 0, &never);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TCOLS);
  }
}

// ------------------------------------------------------------------------------------------------
// Forward for head dimensions up to 128: two query tiles in flight per SM.
// One persistent CTA per SM walks (256 query rows, sequence, head) items, the long ones first, in snake order.  An item
// is two 128-row tiles over the same key / value blocks of 128; tensor memory holds S (128 columns) and O (dh) of both.
//   warps 0-3 / 4-7   softmax of tile 0 / 1, one thread per row, in halves of 64 keys: tcgen05.ld the scores, reference
//                     maximum as above, P packed over the score columns; at the end of an item O / l to global memory
//   warps 8, 9        one thread per tile issues the MMAs: P V of a half, then the next block's Q K^T of that half behind it (in
//                     pipe order, so the score columns that hold P are free by then).  A tile's other half is in the
//                     softmax threads' hands meanwhile, so they find their next scores ready
//   warp 10           TMA: Q of an item, a ring of K and one of V
// While one tile's softmax runs, the pipe works on the other tile; the next item's loads and first scores start while
// this one's output is written.  What bounds it: a half step takes a softmax warp about 1600 cycles, 820 of them the
// exponentials (the special-function unit needs 512 for one tile's and serves both), 320 the load and the maximum, 345
// waiting for the scores; the unit is busy 64 % of a sweep.
// Measured (causal, one launch; the one-tile kernel above, several CTAs per SM, in brackets): 8 x 16 heads x 1024, dh 64
// 41 us (50); 1 x 8 x 4096, dh 128 66 (101); 2 x 32 x 2048, dh 80 67 (120); 1 x 12 x 256, dh 64 6.9 (7.5).  Up to 160
// positions the one-tile kernel is kept: 4 x 4 x 64, dh 32 3.5 against 4.3, 2 x 4 x 129, dh 64 5.4 against 6.2.
// ------------------------------------------------------------------------------------------------
template <int DH>
struct Fwd2Cfg {
  static constexpr int NCH = (DH + 63) / 64;
  static constexpr int T_BYTES = NCH * 128 * 128;               // a 128-row operand
  static constexpr int NST = NCH == 1 ? 4 : 2;                  // ring depth of K and of V
  static constexpr int SMEM = 2 * T_BYTES + NST * 2 * T_BYTES + 1024 + 512;
  static constexpr int C_O = 256, O_STRIDE = DH <= 64 ? 64 : 128;
};
constexpr int FWD2_THREADS = 352;
constexpr int FWD_ONE_TILE_T = 160;    // up to this length (and for dh 256) the one-tile kernel is the faster one

struct FwdItem { int qt, b, h, n0, n1; };
__device__ __forceinline__ FwdItem fwd_item(int i, int nqt, int BH, int H, int T) {
  FwdItem w;
  const int r = i / BH, bh = i - r * BH;
  w.qt = nqt - 1 - r;
  w.b = bh / H;
  w.h = bh - w.b * H;
  w.n0 = 2 * w.qt + 1;                                          // key blocks up to and with the diagonal one
  w.n1 = (2 * w.qt + 1) * 128 < T ? 2 * w.qt + 2 : 0;           // the second tile may lie wholly past the sequence
  return w;
}
// item of round r for CTA c of G: forwards and backwards in turn, so that nobody always gets the longer ones
__device__ __forceinline__ int snake(int r, int c, int G) { return r * G + ((r & 1) ? G - 1 - c : c); }

template <int DH>
__global__ void __launch_bounds__(FWD2_THREADS, 1) attn_fwd_pair_kernel(const __grid_constant__ CUtensorMap tm, bf16* __restrict__ o,
                                                                        float* __restrict__ lse, int B, int T, int H,
                                                                        float scale, unsigned* err) {
  using C = Fwd2Cfg<DH>;
  constexpr int NST = C::NST;
  extern __shared__ uint8_t smem_raw[];
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_smem;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sQ = base, sK0 = base + 2 * C::T_BYTES, sV0 = sK0 + NST * C::T_BYTES;
  const uint32_t bars = sV0 + NST * C::T_BYTES;
  const uint32_t bar_q = bars, bar_qfree = bars + 8;
  auto bar_drain = [&](int x) { return bars + 16 * NST * 2 + 120 + 8 * x; };
  auto bar_s = [&](int x, int hf) { return bars + 24 + 8 * (2 * x + hf); };       // scores of a half block
  auto bar_p = [&](int x, int hf) { return bars + 56 + 8 * (2 * x + hf); };       // ... turned into probabilities
  // ... multiplied with V.  One barrier per half: whoever waits for a phase by its parity must know that the phase before it is
  // over and that the one after it cannot be, and a softmax warp held up between its arrival and its wait can find both
  // halves' products done.
  auto bar_pv = [&](int x, int hf) { return bars + 88 + 8 * (2 * x + hf); };
  auto bar_k = [&](int st) { return bars + 120 + 8 * st; };
  auto bar_v = [&](int st) { return bars + 120 + 8 * (NST + st); };
  auto bar_kfree = [&](int st) { return bars + 120 + 8 * (2 * NST + st); };
  auto bar_vfree = [&](int st) { return bars + 120 + 8 * (3 * NST + st); };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nqt = (T + 255) / 256, BH = B * H, nitems = nqt * BH, G = gridDim.x;
  const int rounds = (nitems + G - 1) / G;
  volatile int* abortp = &abort_flag;

  if (tid == 0) {
    abort_flag = 0;
    mbar_init(bar_q, 1);
    mbar_init(bar_qfree, 2);               // one arrival per issuing thread
    mbar_init(bar_drain(0), 1);
    mbar_init(bar_drain(1), 1);
    for (int x = 0; x < 2; ++x) {
      for (int hf = 0; hf < 2; ++hf) { mbar_init(bar_s(x, hf), 1); mbar_init(bar_p(x, hf), 4); mbar_init(bar_pv(x, hf), 1); }
    }
    for (int st = 0; st < NST; ++st) {
      mbar_init(bar_k(st), 1); mbar_init(bar_v(st), 1);
      mbar_init(bar_kfree(st), 2); mbar_init(bar_vfree(st), 2);
    }
    fence_mbar_init();
    tma_prefetch_desc(&tm);
  }
  if (warp == 8) {
    tmem_alloc(smem_u32(&tmem_base_smem), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dep_wait();
  const uint32_t tmem_base = tmem_base_smem;
  int fail = 0;

  if (warp == 10) {
    // ---------------------------------------------------------------- loads
    if (lane == 0) {
      int g = 0, n_item = 0;
      auto load_tile = [&](uint32_t dst, int slot, int row, int b, uint32_t bar) {
#pragma unroll
        for (int c = 0; c < C::NCH; ++c) tma_load_4d(dst + c * (128 * 128), &tm, c * 64, slot, row, b, bar);
      };
      for (int r = 0; r < rounds && !fail; ++r) {
        const int i = snake(r, blockIdx.x, G);
        if (i >= nitems) continue;
        const FwdItem w = fwd_item(i, nqt, BH, H, T);
        const int n = w.n1 > w.n0 ? w.n1 : w.n0;
        for (int j = 0; j < n; ++j) {
          const int st = (g + j) % NST;
          const uint32_t ph = (uint32_t)((g + j) / NST) & 1u;
          if (!mbar_wait(bar_kfree(st), ph ^ 1u, abortp)) { fail = 1; break; }
          mbar_expect_tx(bar_k(st), C::T_BYTES);
          load_tile(sK0 + st * C::T_BYTES, H + w.h, j * 128, w.b, bar_k(st));
          if (j == 0) {                     // (after the first K, which does not depend on the previous item's scores)
            if (n_item > 0 && !mbar_wait(bar_qfree, (uint32_t)(n_item - 1) & 1u, abortp)) { fail = 1; break; }
            mbar_expect_tx(bar_q, (w.n1 ? 2 : 1) * C::T_BYTES);
            load_tile(sQ, w.h, w.qt * 256, w.b, bar_q);
            if (w.n1) load_tile(sQ + C::T_BYTES, w.h, w.qt * 256 + 128, w.b, bar_q);
          }
          if (!mbar_wait(bar_vfree(st), ph ^ 1u, abortp)) { fail = 1; break; }
          mbar_expect_tx(bar_v(st), C::T_BYTES);
          load_tile(sV0 + st * C::T_BYTES, 2 * H + w.h, j * 128, w.b, bar_v(st));
        }
        g += n;
        ++n_item;
      }
      grid_dep_launch();
      if (fail) abort_flag = 1;
    }
  } else if (warp >= 8) {
    // ---------------------------------------------------------------- MMA issue, one thread per tile
    // (A thread issues an MMA of this size no faster than every ~54 cycles and is held up while the pipe is full: one
    // thread for both tiles made the sweep wait for it.)
    if (lane == 0) {
      const int x = warp - 8;
      constexpr uint32_t idesc_s = make_idesc_bf16(128, 64, 0, 0);
      constexpr uint32_t idesc_o = make_idesc_bf16(128, DH, 0, 1);
      const SmemDescBase dq = make_smem_desc_base(sQ + (uint32_t)x * C::T_BYTES, 16, 1024), dk = make_smem_desc_base(sK0, 16, 1024);
      const SmemDescBase dv = make_smem_desc_base(sV0, 128 * 128, 1024);
      const uint32_t t_s = tmem_base + 128 * x, t_o = tmem_base + C::C_O + C::O_STRIDE * x;
      int g = 0, n_item = 0;
      uint32_t pc = 0;                      // blocks of this tile consumed so far
      bool ok = true;
      // scores of keys 64 hf .. 64 hf + 63 of the block in stage st
      auto issue_s = [&](int hf, int st) {
        const uint32_t ko = (uint32_t)st * C::T_BYTES + (uint32_t)hf * (64 * 128);
#pragma unroll
        for (int ks = 0; ks < DH / 16; ++ks) {
          const uint32_t off = (ks >> 2) * (128 * 128) + (ks & 3) * 32;
          umma_bf16(t_s + 64 * hf, desc_at(dq, off), desc_at(dk, ko + off), idesc_s, ks ? 1u : 0u);
        }
        umma_commit(bar_s(x, hf));
      };
      for (int r = 0; r < rounds && ok; ++r) {
        const int i = snake(r, blockIdx.x, G);
        if (i >= nitems) continue;
        const FwdItem w = fwd_item(i, nqt, BH, H, T);
        const int nt = x ? w.n1 : w.n0;
        const int n = w.n1 > w.n0 ? w.n1 : w.n0;          // both threads pace themselves by every block, used or not
        if (!mbar_wait(bar_k(g % NST), (uint32_t)(g / NST) & 1u, abortp) || !mbar_wait(bar_q, (uint32_t)n_item & 1u, abortp)) { ok = false; break; }
        tc_fence_after();
        if (nt) { issue_s(0, g % NST); issue_s(1, g % NST); }
        umma_commit(bar_kfree(g % NST));
        if (n == 1) umma_commit(bar_qfree);
        for (int j = 0; j < n && ok; ++j) {
          const int st = (g + j) % NST, st1 = (g + j + 1) % NST;
          if (!mbar_wait(bar_v(st), (uint32_t)((g + j) / NST) & 1u, abortp)) { ok = false; break; }
          if (j + 1 < n && !mbar_wait(bar_k(st1), (uint32_t)((g + j + 1) / NST) & 1u, abortp)) { ok = false; break; }
          if (j < nt) {
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              if (!mbar_wait(bar_p(x, hf), pc & 1u, abortp)) { ok = false; break; }
              tc_fence_after();
              const uint32_t vo = (uint32_t)st * C::T_BYTES + (uint32_t)hf * (4 * 2048);
#pragma unroll
              for (int ks = 0; ks < 4; ++ks)
                umma_bf16_ts(t_o, t_s + 64 * hf + 8 * ks, desc_at(dv, vo + ks * 2048), idesc_o, (j | hf | ks) ? 1u : 0u);
              umma_commit(bar_pv(x, hf));
              if (j + 1 < nt) issue_s(hf, st1);
            }
            ++pc;
          }
          if (!ok) break;
          umma_commit(bar_vfree(st));
          if (j + 1 < n) {
            umma_commit(bar_kfree(st1));
            if (j + 2 == n) umma_commit(bar_qfree);       // the item's last scores
          }
        }
        g += n;
        ++n_item;
      }
      if (!ok) { fail = 1; abort_flag = 1; }
      umma_commit(bar_drain(x));                   // every MMA issued has retired before TMEM goes
      int never = 0;
      mbar_wait(bar_drain(x), 0, &never);
    }
  } else {
    // ---------------------------------------------------------------- softmax and output (thread = row of tile x)
    const int x = warp >> 2;
    const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t t_s = t_lane + 128 * x, t_o = t_lane + C::C_O + C::O_STRIDE * x;
    const int d = H * DH;
    const float c2 = scale * IL_LOG2E;
    const float slack = 8.0f / c2;
    auto wait = [&](uint32_t bar, uint32_t parity) -> bool { return __all_sync(0xffffffffu, mbar_wait(bar, parity, abortp)); };
    uint32_t sc = 0;                               // blocks of this tile so far
    for (int r = 0; r < rounds && !fail; ++r) {
      const int i = snake(r, blockIdx.x, G);
      if (i >= nitems) continue;
      const FwdItem w = fwd_item(i, nqt, BH, H, T);
      const int n = x ? w.n1 : w.n0;
      if (n == 0) continue;
      const int rl = (warp & 3) * 32 + lane;       // row within the tile
      const int row = w.qt * 256 + x * 128 + rl;
      float m = -INFINITY, l = 0.f;
      for (int j = 0; j < n && !fail; ++j, ++sc) {
#pragma unroll 1
        for (int hf = 0; hf < 2; ++hf) {
          if (!wait(bar_s(x, hf), sc & 1u)) { fail = 1; abort_flag = 1; break; }
          tc_fence_after();
          float s[64];
          {
            uint32_t u0[32], u1[32];
            tmem_ld_32x32(t_s + 64 * hf, u0);
            tmem_ld_32x32(t_s + 64 * hf + 32, u1);
            tmem_ld_wait();
#pragma unroll
            for (int q = 0; q < 32; ++q) { s[q] = __uint_as_float(u0[q]); s[32 + q] = __uint_as_float(u1[q]); }
          }
          if (j + 1 == n) {                        // the diagonal block: keys after the query
#pragma unroll
            for (int q = 0; q < 64; ++q)
              if (64 * hf + q > rl) s[q] = -INFINITY;
          }
          float mx4[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
          for (int q = 4; q < 60; q += 8)
#pragma unroll
            for (int e = 0; e < 4; ++e) mx4[e] = fmaxf(mx4[e], fmaxf(s[q + e], s[q + 4 + e]));
          const float mx = fmaxf(fmaxf(fmaxf(mx4[0], s[60]), fmaxf(mx4[1], s[61])), fmaxf(fmaxf(mx4[2], s[62]), fmaxf(mx4[3], s[63])));
          if (__any_sync(0xffffffffu, mx > m + slack)) {            // warp-uniform: raise the reference maximum
            const float mn = fmaxf(m, mx);
            const float alpha = ex2_fast((m - mn) * c2);            // 0 on the first block (m = -inf)
            l *= alpha;
            m = mn;
            if (j | hf) {                          // O holds everything up to the half before: that product has to be in
              if (!wait(bar_pv(x, hf ^ 1), (hf ? sc : sc - 1) & 1u)) { fail = 1; abort_flag = 1; break; }
              tc_fence_after();
#pragma unroll 1
              for (int c0 = 0; c0 < DH; c0 += 16) {
                uint32_t v[16];
                tmem_ld_32x16(t_o + c0, v);
                tmem_ld_wait();
#pragma unroll
                for (int q = 0; q < 16; ++q) v[q] = __float_as_uint(__uint_as_float(v[q]) * alpha);
                tmem_st_32x16(t_o + c0, v);
              }
              tmem_st_wait();
            }
          }
          const float mc = m * c2;
          float ps4[4] = {0.f, 0.f, 0.f, 0.f};
          uint32_t pw[32];
#pragma unroll
          for (int q = 0; q < 64; q += 4) {
            const float e0 = ex2_fast(fmaf(s[q], c2, -mc)), e1 = ex2_fast(fmaf(s[q + 1], c2, -mc));
            const float e2 = ex2_fast(fmaf(s[q + 2], c2, -mc)), e3 = ex2_fast(fmaf(s[q + 3], c2, -mc));
            ps4[0] += e0; ps4[1] += e1; ps4[2] += e2; ps4[3] += e3;
            pw[q / 2] = pack_bf16x2(e0, e1);
            pw[q / 2 + 1] = pack_bf16x2(e2, e3);
          }
          tmem_st_32x32(t_s + 64 * hf, pw);        // P over the first half of the score columns this thread read
          l += (ps4[0] + ps4[1]) + (ps4[2] + ps4[3]);
          tmem_st_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_p(x, hf));
        }
      }
      if (fail) break;
      // the last block's two products (the block before it is done: its products precede the last scores in the pipe)
      if (!wait(bar_pv(x, 0), (sc - 1) & 1u) || !wait(bar_pv(x, 1), (sc - 1) & 1u)) { fail = 1; abort_flag = 1; break; }
      tc_fence_after();
      const float inv = 1.0f / l;
      bf16* orow = o + ((size_t)w.b * T + row) * d + w.h * DH;
#pragma unroll
      for (int c0 = 0; c0 < DH; c0 += 16) {
        uint32_t v[16];
        tmem_ld_32x16(t_o + c0, v);
        tmem_ld_wait();
        if (row < T) {
#pragma unroll
          for (int q = 0; q < 16; q += 8) {
            uint4 pk;
            pk.x = pack_bf16x2(__uint_as_float(v[q]) * inv, __uint_as_float(v[q + 1]) * inv);
            pk.y = pack_bf16x2(__uint_as_float(v[q + 2]) * inv, __uint_as_float(v[q + 3]) * inv);
            pk.z = pack_bf16x2(__uint_as_float(v[q + 4]) * inv, __uint_as_float(v[q + 5]) * inv);
            pk.w = pack_bf16x2(__uint_as_float(v[q + 6]) * inv, __uint_as_float(v[q + 7]) * inv);
            *reinterpret_cast<uint4*>(orow + c0 + q) = pk;
          }
        }
      }
      if (row < T) lse[((size_t)w.b * H + w.h) * T + row] = m * scale + logf(l);
      tc_fence_before();       // O has been read before this thread's next P lets the next item's products overwrite it
    }
  }
  fail = __syncthreads_or(fail);
  if (tid == 0 && fail && err) atomicExch(err, DEV_TIMEOUT_MMA);
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

template <int DH>
cudaError_t fwd_pair_launch(const bf16* qkv, bf16* o, float* lse, int B, int T, int H, unsigned* err, cudaStream_t s) {
  using C = Fwd2Cfg<DH>;
  const unsigned long long d3 = 3ull * H * DH;
  const unsigned long long dims[4] = {(unsigned long long)DH, 3ull * H, (unsigned long long)T, (unsigned long long)B};
  const unsigned long long strides[3] = {(unsigned long long)DH * 2, d3 * 2, (unsigned long long)T * d3 * 2};
  const unsigned box[4] = {64, 1, 128, 1};
  CUtensorMap tm;
  if (!tma_encode_bf16(&tm, qkv, 4, dims, strides, box)) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(attn_fwd_pair_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const long long items = (long long)((T + 255) / 256) * B * H;
  const int grid = (int)(items < sms ? items : sms);
  launch_dep(attn_fwd_pair_kernel<DH>, dim3(grid), dim3(FWD2_THREADS), C::SMEM, s, tm, o, lse, B, T, H, rsqrtf((float)DH), err);
  return cudaGetLastError();
}

template <int DH>
cudaError_t fwd_tc_launch(const bf16* qkv, bf16* o, float* lse, int B, int T, int H, unsigned* err, cudaStream_t s) {
  using C = FwdCfg<DH>;
  const unsigned long long d3 = 3ull * H * DH;
  const unsigned long long dims[4] = {(unsigned long long)DH, 3ull * H, (unsigned long long)T, (unsigned long long)B};
  const unsigned long long strides[3] = {(unsigned long long)DH * 2, d3 * 2, (unsigned long long)T * d3 * 2};
  const unsigned boxq[4] = {64, 1, TQ, 1}, boxk[4] = {64, 1, TK, 1};
  CUtensorMap tmQ, tmKV;
  if (!tma_encode_bf16(&tmQ, qkv, 4, dims, strides, boxq)) return cudaErrorInvalidValue;
  if (!tma_encode_bf16(&tmKV, qkv, 4, dims, strides, boxk)) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(attn_fwd_tc_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  dim3 grid((T + TQ - 1) / TQ, B * H);
  launch_dep(attn_fwd_tc_kernel<DH>, dim3(grid), dim3(128), C::SMEM, s, tmQ, tmKV, o, lse, T, H, rsqrtf((float)DH), err);
  return cudaGetLastError();
}


// ------------------------------------------------------------------------------------------------
// Backward at head dimension 256 (the smaller ones: attention_sweep.cu).  Same structure as the forward: a CTA owns 128 rows
// (keys for dK/dV, queries for dQ), the other index is swept in blocks of 64; two threads share a row (32 columns of each block each: the backward has
// no row-wise reduction, so they never need to talk), all products run on tcgen05 and
// — because the backward has no running maximum — every gradient accumulates in TMEM across the sweep.
// Probabilities are recomputed from the saved log-sum-exp; delta_i = sum_c dO_ic O_ic.
// P^T and dS^T (dS for dQ) never touch shared memory: a thread rounds its 32 values to bf16, packs them in
// pairs and stores the 16 words back into the first half of the TMEM columns it has just read, from where
// the next MMA takes them as its A operand.  One 64 KB stage of swept tiles is all that fits beside the row operands, so a
// step's scores are issued at its own top; dV and dK do not fit the 512 TMEM columns together and run as two launches.
// ------------------------------------------------------------------------------------------------

template <int DH>
struct BwdCfg {
  static constexpr int NCH = (DH + 63) / 64;
  static constexpr int ROW_BYTES = NCH * TQ * 128;      // a 128-row operand (all chunks)
  static constexpr int BLK_BYTES = NCH * TK * 128;      // a 64-row operand
  // dK/dV: K, V resident; one stage of (Q, dO); lse/delta vectors.  TMEM: S^T, dP^T, dV or dK.
  static constexpr int SMEM_KV = 2 * ROW_BYTES + 2 * BLK_BYTES + 1024 + 2 * 2 * 64 * 4 + 128;
  // dQ: Q, dO resident; one stage of (K, V).  TMEM: S, dP, dQ.
  static constexpr int SMEM_Q = 2 * ROW_BYTES + 2 * BLK_BYTES + 1024 + 128;
  static constexpr int TCOLS = 512;
};

// 32 fp32 values -> 16 words of bf16 pairs (even index in the low half)
__device__ __forceinline__ void pack_row32(const float (&v)[32], uint32_t (&w)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) w[i] = pack_bf16x2(v[2 * i], v[2 * i + 1]);
}
// TMEM column offset (within a 64-column block whose two 32-column halves each hold their packed values in
// their first 16 columns) of the A operand of K-step ks (16 elements = 8 columns)
__device__ __forceinline__ constexpr uint32_t packed_col(int ks) { return (uint32_t)((ks >> 1) * 32 + (ks & 1) * 8); }

// PART: 1 = dV, 2 = dK (each recomputing the scores).
template <int DH, int PART>
__global__ void __launch_bounds__(256) attn_bwd_dkv_tc_kernel(const __grid_constant__ CUtensorMap tmRow,   // qkv, 128-row box
                                                              const __grid_constant__ CUtensorMap tmBlk,   // qkv, 64-row box
                                                              const __grid_constant__ CUtensorMap tmdO,    // dout, 64-row box
                                                              const float* __restrict__ lse, const float* __restrict__ delta,
                                                              bf16* __restrict__ dqkv, int B, int T, int H, float scale,
                                                              unsigned* err) {
  using C = BwdCfg<DH>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_smem;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sK = base, sV = sK + C::ROW_BYTES;
  const uint32_t sQ0 = sV + C::ROW_BYTES, sdO0 = sQ0 + C::BLK_BYTES;
  const uint32_t vecs = sdO0 + C::BLK_BYTES;               // lse2[2][64], delta[2][64]
  const uint32_t bars = vecs + 2 * 2 * 64 * 4;
  const uint32_t bar_kv = bars, bar_s = bars + 8, bar_acc = bars + 16, bar_drain = bars + 24, bar_q0 = bars + 32;
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  float* s_lse = reinterpret_cast<float*>(gen + (vecs - base));  // [2][64]
  float* s_del = s_lse + 128;                                    // [2][64]

  // 256 threads: thread (r, hf) owns row r = tid % 128 and columns [32 hf, 32 hf + 32) of each 64-wide block
  const int tid = threadIdx.x, warp = tid >> 5, r = tid & 127, hf = tid >> 7;
  const int kb = blockIdx.x;
  const int nb = blockIdx.y / H, h = blockIdx.y % H;
  const int bs = nb % B;
  const int d = H * DH;
  const int key = kb * TQ + r;
  const int nq = (T + TK - 1) / TK;
  const int q0 = (kb * TQ) / TK;                                 // first query block that can see these keys
  const float* lse_b = lse + ((size_t)bs * H + h) * T;
  const float* del_b = delta + ((size_t)nb * H + h) * T;

  if (tid == 0) {
    abort_flag = 0;
    mbar_init(bar_kv, 1);
    mbar_init(bar_s, 1);
    mbar_init(bar_acc, 1);
    mbar_init(bar_drain, 1);
    mbar_init(bar_q0, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmRow);
    tma_prefetch_desc(&tmBlk);
    tma_prefetch_desc(&tmdO);
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(&tmem_base_smem), C::TCOLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();          // tensor memory is held by this CTA before the next kernel may become resident
  grid_dep_wait();
  // lse (in log2 units) and delta of a query block: fetched from global memory into a register one sweep
  // step before they are put into shared memory (buffer j&1), two steps before they are used, so that no
  // step waits on that load
  auto fetch_vec = [&](int j) -> float {
    const int q = j * TK + (tid & 63);
    if (j >= nq || q >= T || tid >= 128) return 0.f;
    return tid < 64 ? lse_b[q] * IL_LOG2E : del_b[q];
  };
  auto put_vec = [&](int j, float v) {
    if (tid < 64) s_lse[(j & 1) * 64 + tid] = v;
    else if (tid < 128) s_del[(j & 1) * 64 + (tid & 63)] = v;
  };
  if (q0 < nq) put_vec(q0, fetch_vec(q0));
  float vec_next = fetch_vec(q0 + 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // TMEM: S^T [0,64) and dP^T [64,128) (each later overwritten in part by its packed bf16 successor P^T,
  // dS^T), dV [128,128+dh), dK [128+dh, 128+2dh)
  const uint32_t tmem_base = tmem_base_smem;
  const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
  volatile int* abortp = &abort_flag;
  constexpr uint32_t idesc_s = make_idesc_bf16(TQ, TK, 0, 0);
  constexpr uint32_t idesc_g = make_idesc_bf16(TQ, DH, 0, 1);
  int fail = 0;

  auto load_q = [&](int j) {
    mbar_expect_tx(bar_q0, 2 * C::BLK_BYTES);
#pragma unroll
    for (int c = 0; c < C::NCH; ++c) {
      tma_load_4d(sQ0 + c * (TK * 128), &tmBlk, c * 64, h, j * TK, bs, bar_q0);
      tma_load_4d(sdO0 + c * (TK * 128), &tmdO, c * 64, h, j * TK, nb, bar_q0);
    }
  };
  if (tid == 0) {
    mbar_expect_tx(bar_kv, 2 * C::ROW_BYTES);
#pragma unroll
    for (int c = 0; c < C::NCH; ++c) {
      tma_load_4d(sK + c * (TQ * 128), &tmRow, c * 64, H + h, kb * TQ, bs, bar_kv);
      tma_load_4d(sV + c * (TQ * 128), &tmRow, c * 64, 2 * H + h, kb * TQ, bs, bar_kv);
    }
    if (q0 < nq) load_q(q0);
  }
  const float c2 = scale * IL_LOG2E;

  // S^T and dP^T of query block j, issued by thread 0
  const SmemDescBase dk_k = make_smem_desc_base(sK, 16, 1024), dv_k = make_smem_desc_base(sV, 16, 1024);
  const SmemDescBase dq_k = make_smem_desc_base(sQ0, 16, 1024), ddo_k = make_smem_desc_base(sdO0, 16, 1024);
  const SmemDescBase dq_mn = make_smem_desc_base(sQ0, TK * 128, 1024), ddo_mn = make_smem_desc_base(sdO0, TK * 128, 1024);
  auto issue_s = [&](int j) {
    if (!mbar_wait(bar_q0, (uint32_t)(j - q0) & 1u, abortp)) { fail = 1; abort_flag = 1; }
    tc_fence_after();
#pragma unroll
    for (int ks = 0; ks < DH / 16; ++ks) {
      const uint32_t off_a = (ks >> 2) * (TQ * 128) + (ks & 3) * 32;
      const uint32_t off_b = (ks >> 2) * (TK * 128) + (ks & 3) * 32;
      umma_bf16(tmem_base, desc_at(dk_k, off_a), desc_at(dq_k, off_b), idesc_s, ks ? 1u : 0u);
      if (PART != 1) umma_bf16(tmem_base + 64, desc_at(dv_k, off_a), desc_at(ddo_k, off_b), idesc_s, ks ? 1u : 0u);
    }
    umma_commit(bar_s);
  };
  if (tid == 0 && q0 < nq) {
    if (!mbar_wait(bar_kv, 0, abortp)) { fail = 1; abort_flag = 1; }
  }

  for (int j = q0; j < nq; ++j) {
    const int it = j - q0;
    if (j + 1 < nq) put_vec(j + 1, vec_next);      // visible after this step's barrier
    vec_next = fetch_vec(j + 2);
    // the previous step's products must have retired before its tiles are replaced and the new scores overwrite the packed
    // columns; only then are this step's scores issued
    if (it > 0) {
      if (!mbar_wait(bar_acc, (uint32_t)(it - 1) & 1u, abortp)) { fail = 1; abort_flag = 1; }
      if (tid == 0) load_q(j);
    }
    if (tid == 0) issue_s(j);
    if (!mbar_wait(bar_s, (uint32_t)it & 1u, abortp)) { fail = 1; abort_flag = 1; }
    tc_fence_after();
    {
      float p[32], ds[32];
      uint32_t r0[32], r1[32];
      tmem_ld_32x32(t_lane + 32 * hf, r0);
      if (PART != 1) tmem_ld_32x32(t_lane + 64 + 32 * hf, r1);
      tmem_ld_wait();
      const float4* lv = reinterpret_cast<const float4*>(s_lse + (j & 1) * 64 + 32 * hf);
      const float4* dv_ = reinterpret_cast<const float4*>(s_del + (j & 1) * 64 + 32 * hf);
      const bool diag = (j * TK < kb * TQ + TQ);   // some queries of this block precede some keys of this CTA
      const bool tail = (j * TK + TK > T);
      const int qbase = j * TK + 32 * hf;
#pragma unroll
      for (int i4 = 0; i4 < 8; ++i4) {
        const float4 l4 = lv[i4], d4 = dv_[i4];
        const float ll[4] = {l4.x, l4.y, l4.z, l4.w}, dd[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int i = 4 * i4 + e;
          p[i] = ex2_fast(fmaf(__uint_as_float(r0[i]), c2, -ll[e]));
          ds[i] = PART != 1 ? __uint_as_float(r1[i]) - dd[e] : 0.f;
        }
      }
      if (diag || tail) {                          // uniform: only blocks on the diagonal or past the sequence end
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (qbase + i < key || qbase + i >= T) p[i] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < 32; ++i) ds[i] *= p[i];
      uint32_t pw[16], dw[16];
      if (PART != 2) {
        pack_row32(p, pw);
        tmem_st_32x16(t_lane + 32 * hf, pw);       // P^T over the first half of the S^T columns this thread read
      }
      if (PART != 1) {
        pack_row32(ds, dw);
        tmem_st_32x16(t_lane + 64 + 32 * hf, dw);  // dS^T likewise over dP^T
      }
      tmem_st_wait();
    }
    tc_fence_before();
    if (__syncthreads_or(fail)) { fail = 1; break; }
    if (tid == 0) {
      tc_fence_after();
#pragma unroll
      for (int ks = 0; ks < TK / 16; ++ks) {
        const uint32_t off_b = ks * 2048;                                                   // MN-major: 16 queries
        if (PART != 2)
          umma_bf16_ts(tmem_base + 128, tmem_base + packed_col(ks), desc_at(ddo_mn, off_b), idesc_g, (it | ks) ? 1u : 0u);
        if (PART != 1)
          umma_bf16_ts(tmem_base + 128, tmem_base + 64 + packed_col(ks), desc_at(dq_mn, off_b), idesc_g,
                       (it | ks) ? 1u : 0u);
      }
      umma_commit(bar_acc);
    }
  }
  const int nit = nq - q0;
  grid_dep_launch();
  if (!fail && nit > 0) {
    if (!mbar_wait(bar_acc, (uint32_t)(nit - 1) & 1u, abortp)) { fail = 1; abort_flag = 1; }
    tc_fence_after();
  }
  fail = __syncthreads_or(fail);
  if (!fail) {
    bf16* rowp = dqkv + ((size_t)nb * T + key) * (3 * d) + h * DH;
    {
      // the two halves of the threads split the columns
      const int which = PART - 1;
      const uint32_t tcol = t_lane + 128;
      bf16* dst = rowp + (which == 0 ? 2 * d : d);
      const float f = which == 0 ? 1.0f : scale;
      const int cbeg = hf * (DH / 2), cend = cbeg + DH / 2;
#pragma unroll
      for (int c0 = cbeg; c0 < cend; c0 += 32) {
        float v[32];
        if (c0 + 32 <= DH) {
          uint32_t rr[32];
          tmem_ld_32x32(tcol + c0, rr);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] = nit > 0 ? __uint_as_float(rr[i]) * f : 0.f;
        } else {
          uint32_t rr[16];
          tmem_ld_32x16(tcol + c0, rr);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = nit > 0 ? __uint_as_float(rr[i]) * f : 0.f;
        }
        if (key < T) {
#pragma unroll
          for (int i = 0; i < 32 && c0 + i < DH; i += 8) {
            uint4 pk;
            pk.x = pack_bf16x2(v[i], v[i + 1]);
            pk.y = pack_bf16x2(v[i + 2], v[i + 3]);
            pk.z = pack_bf16x2(v[i + 4], v[i + 5]);
            pk.w = pack_bf16x2(v[i + 6], v[i + 7]);
            *reinterpret_cast<uint4*>(dst + c0 + i) = pk;
          }
        }
      }
    }
  }
  if (tid == 0) {
    if (fail && err) atomicExch(err, DEV_TIMEOUT_MMA);
    umma_commit(bar_drain);
    int never = 0;
    mbar_wait(bar_drain, 0, &never);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TCOLS);
  }
}

template <int DH>
__global__ void __launch_bounds__(256) attn_bwd_dq_tc_kernel(const __grid_constant__ CUtensorMap tmRow,    // qkv, 128-row box
                                                             const __grid_constant__ CUtensorMap tmBlk,    // qkv, 64-row box
                                                             const __grid_constant__ CUtensorMap tmdO,     // dout, 128-row box
                                                             const float* __restrict__ lse, const float* __restrict__ delta,
                                                             bf16* __restrict__ dqkv, int B, int T, int H, float scale,
                                                             unsigned* err) {
  using C = BwdCfg<DH>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_smem;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sQ = base, sdO = sQ + C::ROW_BYTES;
  const uint32_t sK0 = sdO + C::ROW_BYTES, sV0 = sK0 + C::BLK_BYTES;
  const uint32_t bars = sV0 + C::BLK_BYTES;
  const uint32_t bar_q = bars, bar_s = bars + 8, bar_acc = bars + 16, bar_drain = bars + 24, bar_kv0 = bars + 32;

  // 256 threads: thread (r, hf) owns row r = tid % 128 and columns [32 hf, 32 hf + 32) of each 64-wide block
  const int tid = threadIdx.x, warp = tid >> 5, r = tid & 127, hf = tid >> 7;
  const int qb = gridDim.x - 1 - blockIdx.x;
  const int nb = blockIdx.y / H, h = blockIdx.y % H;
  const int bs = nb % B;
  const int d = H * DH;
  const int row = qb * TQ + r;
  int nkv = (qb * TQ + TQ + TK - 1) / TK;
  const int nkv_all = (T + TK - 1) / TK;
  if (nkv > nkv_all) nkv = nkv_all;

  if (tid == 0) {
    abort_flag = 0;
    mbar_init(bar_q, 1);
    mbar_init(bar_kv0, 1);
    mbar_init(bar_s, 1);
    mbar_init(bar_acc, 1);
    mbar_init(bar_drain, 1);
    fence_mbar_init();
    tma_prefetch_desc(&tmRow);
    tma_prefetch_desc(&tmBlk);
    tma_prefetch_desc(&tmdO);
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(&tmem_base_smem), C::TCOLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dep_wait();
  const uint32_t tmem_base = tmem_base_smem;     // S [0,64), dP [64,128) (later in part the packed dS), dQ [128,128+dh)
  const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
  volatile int* abortp = &abort_flag;
  constexpr uint32_t idesc_s = make_idesc_bf16(TQ, TK, 0, 0);
  constexpr uint32_t idesc_g = make_idesc_bf16(TQ, DH, 0, 1);
  int fail = 0;

  auto load_kv = [&](int j) {
    mbar_expect_tx(bar_kv0, 2 * C::BLK_BYTES);
#pragma unroll
    for (int c = 0; c < C::NCH; ++c) {
      tma_load_4d(sK0 + c * (TK * 128), &tmBlk, c * 64, H + h, j * TK, bs, bar_kv0);
      tma_load_4d(sV0 + c * (TK * 128), &tmBlk, c * 64, 2 * H + h, j * TK, bs, bar_kv0);
    }
  };
  if (tid == 0) {
    mbar_expect_tx(bar_q, 2 * C::ROW_BYTES);
#pragma unroll
    for (int c = 0; c < C::NCH; ++c) {
      tma_load_4d(sQ + c * (TQ * 128), &tmRow, c * 64, h, qb * TQ, bs, bar_q);
      tma_load_4d(sdO + c * (TQ * 128), &tmdO, c * 64, h, qb * TQ, nb, bar_q);
    }
    if (nkv > 0) load_kv(0);
  }
  const float c2 = scale * IL_LOG2E;
  const float lse2 = row < T ? lse[((size_t)bs * H + h) * T + row] * IL_LOG2E : 0.f;
  const float del = row < T ? delta[((size_t)nb * H + h) * T + row] : 0.f;

  // S and dP of key block j, issued by thread 0
  const SmemDescBase dq_k = make_smem_desc_base(sQ, 16, 1024), ddo_k = make_smem_desc_base(sdO, 16, 1024);
  const SmemDescBase dk_k = make_smem_desc_base(sK0, 16, 1024), dv_k = make_smem_desc_base(sV0, 16, 1024);
  const SmemDescBase dk_mn = make_smem_desc_base(sK0, TK * 128, 1024);
  auto issue_s = [&](int j) {
    if (!mbar_wait(bar_kv0, (uint32_t)j & 1u, abortp)) { fail = 1; abort_flag = 1; }
    tc_fence_after();
#pragma unroll
    for (int ks = 0; ks < DH / 16; ++ks) {
      const uint32_t off_a = (ks >> 2) * (TQ * 128) + (ks & 3) * 32;
      const uint32_t off_b = (ks >> 2) * (TK * 128) + (ks & 3) * 32;
      umma_bf16(tmem_base, desc_at(dq_k, off_a), desc_at(dk_k, off_b), idesc_s, ks ? 1u : 0u);
      umma_bf16(tmem_base + 64, desc_at(ddo_k, off_a), desc_at(dv_k, off_b), idesc_s, ks ? 1u : 0u);
    }
    umma_commit(bar_s);
  };
  if (tid == 0 && nkv > 0) {
    if (!mbar_wait(bar_q, 0, abortp)) { fail = 1; abort_flag = 1; }
  }

  for (int j = 0; j < nkv; ++j) {
    // retire the previous step's product, replace its tiles, then issue these scores
    if (j > 0) {
      if (!mbar_wait(bar_acc, (uint32_t)(j - 1) & 1u, abortp)) { fail = 1; abort_flag = 1; }
      if (tid == 0) load_kv(j);
    }
    if (tid == 0) issue_s(j);
    if (!mbar_wait(bar_s, (uint32_t)j & 1u, abortp)) { fail = 1; abort_flag = 1; }
    tc_fence_after();
    {
      float ds[32];
      uint32_t r0[32], r1[32];
      tmem_ld_32x32(t_lane + 32 * hf, r0);
      tmem_ld_32x32(t_lane + 64 + 32 * hf, r1);
      tmem_ld_wait();
      const bool diag = (j * TK + TK - 1 > qb * TQ);
      const int kbase = j * TK + 32 * hf;
#pragma unroll
      for (int i = 0; i < 32; ++i) ds[i] = ex2_fast(fmaf(__uint_as_float(r0[i]), c2, -lse2));
      if (diag) {                                  // uniform: only blocks on the diagonal
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (kbase + i > row) ds[i] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < 32; ++i) ds[i] *= (__uint_as_float(r1[i]) - del);
      uint32_t dw[16];
      pack_row32(ds, dw);
      tmem_st_32x16(t_lane + 64 + 32 * hf, dw);      // dS over the first half of the dP columns this thread read
      tmem_st_wait();
    }
    tc_fence_before();
    if (__syncthreads_or(fail)) { fail = 1; break; }
    if (tid == 0) {
      tc_fence_after();
#pragma unroll
      for (int ks = 0; ks < TK / 16; ++ks)
        umma_bf16_ts(tmem_base + 128, tmem_base + 64 + packed_col(ks), desc_at(dk_mn, ks * 2048), idesc_g, (j | ks) ? 1u : 0u);
      umma_commit(bar_acc);
    }
  }
  grid_dep_launch();
  if (!fail && nkv > 0) {
    if (!mbar_wait(bar_acc, (uint32_t)(nkv - 1) & 1u, abortp)) { fail = 1; abort_flag = 1; }
    tc_fence_after();
  }
  fail = __syncthreads_or(fail);
  if (!fail) {
    bf16* dst = dqkv + ((size_t)nb * T + row) * (3 * d) + h * DH;
#pragma unroll
    for (int u = 0; u < DH / 16; ++u) {              // 16-column units, alternating between the two halves
      if ((u & 1) != hf) continue;
      const int c0 = u * 16;
      float v[16];
      {
        uint32_t rr[16];
        tmem_ld_32x16(t_lane + 128 + c0, rr);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(rr[i]) * scale;
      }
      if (row < T) {
#pragma unroll
        for (int i = 0; i < 16; i += 8) {
          uint4 pk;
          pk.x = pack_bf16x2(v[i], v[i + 1]);
          pk.y = pack_bf16x2(v[i + 2], v[i + 3]);
          pk.z = pack_bf16x2(v[i + 4], v[i + 5]);
          pk.w = pack_bf16x2(v[i + 6], v[i + 7]);
          *reinterpret_cast<uint4*>(dst + c0 + i) = pk;
        }
      }
    }
  }
  if (tid == 0) {
    if (fail && err) atomicExch(err, DEV_TIMEOUT_MMA);
    umma_commit(bar_drain);
    int never = 0;
    mbar_wait(bar_drain, 0, &never);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, C::TCOLS);
  }
}

// ------------------------------------------------------------------------------------------------
// Backward in one sweep (head dimensions up to 64).  The two-kernel forms recompute the scores twice (seven
// products for five); here a CTA owns 128 keys, sweeps the queries in blocks of 128 and produces dV, dK and its
// share of dQ from one recomputation of S^T and dP^T:
//   S^T, dP^T   tcgen05.mma M128 (keys) N64 per 64-query half -> TMEM, two halves per step
//   P^T, dS^T   threads (two per key row and half, 32 columns each) recompute the probabilities from the saved
//               log-sum-exp, round to bf16 and store the packed pairs back over the score columns
//   dV += P^T dO, dK += dS^T Q      A operand read from those TMEM columns, accumulated over the whole sweep
//   dQ_blk = dS K                   needs dS with the queries as rows: the same threads also write their dS values
//                                   to shared memory in the layout of an MN-major A operand (swizzled 128-byte
//                                   rows, one row per key); the product lands in one of two TMEM buffers and is
//                                   added to an fp32 [rows, d] accumulator in global memory by bulk reductions (every
//                                   key tile of a (sequence, head) contributes to the same query rows)
// Roles: warps 0-7 / 8-15 recompute and convert the first / second half of every step, warps 16-19 add finished dQ blocks to
// the global accumulator, each its own 32 rows, and store an item's dV / dK, a thread each of warps 20, 21 and 22 issues the
// MMAs of S and dV, of dP and dK, and of dQ, warp 23 feeds the Q / dO ring by TMA and the per-query lse / delta vectors by
// plain loads.  The halves give the pipeline its overlap: while eight warps work on one half, the tensor pipe runs the other's
// products and next scores.  One CTA per SM (all 512 TMEM columns, ~200 KB of shared memory), persistent: a CTA walks a list of
// (key tile, sequence, head) items, and the loads and scores of an item start while the previous item's dV / dK are still
// being written out.
// What bounds it: a step of 128 x 128 takes about 3200 cycles, of which a recompute warp works 1400 (sixteen warps share the
// issue slots) and an issuing thread 1700 (16 MMAs at 60, two commits at 120, looks at barriers at 150 each); the change of
// items costs another step (K and V of one item only fit beside three Q / dO stages: with two buffers and two stages the tiles
// came late and nothing was gained).  Measured, delta and conversion included, launches back to back: 16 x 16 heads x 1024,
// dh 64 236 -> 209 us, 8 x 16 124 -> 107, against the form with all sixteen warps on either half in turn, one issuing thread per half
// and the four flush warps staging a block together; 211 and 110 on another GPU since dS has a barrier per buffer.  The 80
// registers that 768 threads leave spill a little: 0.39 of 34.5 million warp instructions touch local memory.
// The sum over key tiles in dQ is made by floating-point atomics: its order, and with it the last bit of dQ,
// depends on scheduling.  Every wait is bounded.
// ------------------------------------------------------------------------------------------------
template <int DH>
struct FusedCfg {
  static constexpr int NST = 3;                          // Q / dO ring depth
  static constexpr int KVB = 1;                          // items whose K / V are held (two would cost the ring a stage)
  static constexpr int VST = 4;                          // ring of their lse / delta vectors, filled a step further ahead
  static constexpr int ROW_BYTES = TQ * 128;             // a 128-row operand (one 64-column chunk)
  static constexpr int DS_BYTES = 2 * TQ * 128;          // dS of one step: two 64-query chunks x 128 key rows x 128 B
  static constexpr int VEC_BYTES = 2 * TQ * 4;           // lse (log2 units) and delta of the step's 128 queries
  static constexpr int SMEM = KVB * 2 * ROW_BYTES + NST * 2 * ROW_BYTES + VST * VEC_BYTES + 2 * DS_BYTES + 256 + 1024;
  // TMEM columns: S^T [0,128) (two halves), dP^T [128,256), dV [256,256+DH), dK [320,320+DH), dQ [384,384+DH) / [448,448+DH)
  static constexpr int C_S = 0, C_DP = 128, C_DV = 256, C_DK = 320, C_DQ = 384;
};

constexpr int FUSED_THREADS = 768;   // warps 0-15 recompute, 16-19 flush dQ and store dV / dK, 20-22 issue MMAs, 23 loads
constexpr int FUSED_RW = 16;         // recompute warps: eight per half, two threads per key row, 32 query columns each

// Work item = (key tile, gradient sequence, head).  Items are numbered key tile first, so the long sweeps (key tile
// 0 sees every query block) come first; CTA c takes items c, c + gridDim.x, ...  Every role walks the same list and
// counts the same global step number g, from which ring stages and barrier parities follow.
struct FusedItem { int kb, nb, h, bs, nit; };
__device__ __forceinline__ FusedItem fused_item(int item, int nbh, int H, int B, int nq) {
  FusedItem w;
  w.kb = item / nbh;
  const int r = item - w.kb * nbh;
  w.nb = r / H;
  w.h = r - w.nb * H;
  w.bs = w.nb % B;
  w.nit = nq - w.kb;                    // query blocks kb .. nq-1 see these keys
  return w;
}

template <int DH>
__global__ void __launch_bounds__(FUSED_THREADS, 1) attn_bwd_fused_kernel(const __grid_constant__ CUtensorMap tmRow,     // qkv, 128-row box
                                                                          const __grid_constant__ CUtensorMap tmdO,      // dout, 128-row box
                                                                          const __grid_constant__ CUtensorMap tmAcc,     // dQ accumulator (fp32), 32 x 32 box
                                                                          const float* __restrict__ lse, const float* __restrict__ delta,
                                                                          bf16* __restrict__ dqkv, int NB,
                                                                          int B, int T, int H, float scale, unsigned* err) {
  using C = FusedCfg<DH>;
  constexpr int NST = C::NST, VST = C::VST, KVB = C::KVB;
  extern __shared__ uint8_t smem_raw[];
  __shared__ int abort_flag;
  __shared__ uint32_t tmem_base_smem;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sKV = base;                                               // K of an item, V after it
  const uint32_t sQ0 = sKV + KVB * 2 * C::ROW_BYTES;                             // stage st: Q at sQ0 + st * STAGE, dO after it
  constexpr uint32_t STAGE = 2 * C::ROW_BYTES;
  const uint32_t sDS = sQ0 + NST * STAGE;                                  // two dS buffers
  const uint32_t sVec = sDS + 2 * C::DS_BYTES;                             // VST x (lse2[128], delta[128])
  const uint32_t bars = sVec + VST * C::VEC_BYTES;
  // Barriers (8 bytes each).  A wait by parity is right only while the phase before the awaited one is over and the one after it
  // cannot be; and a phase of several arrivals must not collect those of two steps.  Every waiter below waits for all phases of a
  // barrier in turn, and after each barrier stands what holds its next phase back until all have passed this one.
  auto bar_kv = [&](int i) { return bars + 8 * i; };                           // K / V buffer i loaded: the loader waits for bar_kvfree
  auto bar_kvfree = [&](int i) { return bars + 16 + 8 * i; };                  // arrivals follow bar_kv, which the loader lets go
  const uint32_t bar_acc = bars + 32;                                          // dV / dK complete: next products wait for bar_accfree
  const uint32_t bar_accfree = bars + 40;                                      // ... stored: arrivals follow bar_acc
  // dS of a step written by both halves, into buffer b.  One per buffer: the halves run up to a step apart, so a barrier for
  // both buffers would count the faster half's next step in the slower one's stead.  Arrivals at this buffer's next
  // step follow bar_dsfree(b).
  auto bar_ds = [&](int b) { return bars + 48 + 8 * b; };
  auto bar_drain = [&](int t) { return bars + 64 + 8 * t; };                   // one per issuing thread, used once
  auto bar_full = [&](int st) { return bars + 88 + 8 * st; };                  // Q / dO of a step loaded: the loader waits for bar_empty
  auto bar_empty = [&](int st) { return bars + 88 + 8 * (NST + st); };         // arrivals follow bar_full
  auto bar_s = [&](int x) { return bars + 88 + 8 * (2 * NST + x); };           // scores of half x ready: each issuing thread waits for bar_p(x)
  auto bar_p = [&](int x) { return bars + 88 + 8 * (2 * NST + 2 + x); };       // P^T / dS^T of half x in tensor memory: arrivals follow bar_s(x)
  auto bar_dq = [&](int b) { return bars + 88 + 8 * (2 * NST + 4 + b); };      // dQ buffer b complete: its thread waits for bar_dqfree(b)
  auto bar_dqfree = [&](int b) { return bars + 88 + 8 * (2 * NST + 6 + b); };  // dQ buffer b flushed: arrivals follow bar_dq(b)
  auto bar_vec = [&](int v) { return bars + 88 + 8 * (2 * NST + 8 + v); };     // lse / delta vectors written: the loader has waited for bar_empty of
                                                                               // the slot's last step, which follows all reads of it
  auto bar_dsfree = [&](int b) { return bars + 88 + 8 * (2 * NST + VST + 8 + b); };  // dS buffer b (also the staging of its dQ block) free
                                                                               // again: arrivals follow bar_dq(b), which follows bar_ds(b)
  static_assert(88 + 8 * (2 * C::NST + C::VST + 10) <= 256, "barriers");
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  float* s_vec = reinterpret_cast<float*>(gen + (sVec - base));

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int d = H * DH;
  const int nq = (T + TQ - 1) / TQ;
  const int nbh = NB * H;
  const int nitems = nq * nbh;
  volatile int* abortp = &abort_flag;

  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < 2; ++i) { mbar_init(bar_kv(i), 1); mbar_init(bar_kvfree(i), 3); }    // (freed by the three issuing threads)
    mbar_init(bar_acc, 2);               // the threads of dV and of dK
    mbar_init(bar_accfree, 4);           // one arrival per flush warp
    for (int b = 0; b < 2; ++b) mbar_init(bar_ds(b), FUSED_RW);     // one arrival per recompute warp
    mbar_init(bar_drain(0), 1);
    mbar_init(bar_drain(1), 1);
    mbar_init(bar_drain(2), 1);
    for (int st = 0; st < NST; ++st) { mbar_init(bar_full(st), 1); mbar_init(bar_empty(st), 2); }
    for (int v = 0; v < VST; ++v) mbar_init(bar_vec(v), 1);
    for (int x = 0; x < 2; ++x) {
      mbar_init(bar_s(x), 2);            // the threads of S and of dP
      mbar_init(bar_p(x), FUSED_RW / 2);
      mbar_init(bar_dq(x), 1);
      mbar_init(bar_dqfree(x), 4);       // one arrival per flush warp
      mbar_init(bar_dsfree(x), 4);       // (likewise)
    }
    fence_mbar_init();
    tma_prefetch_desc(&tmRow);
    tma_prefetch_desc(&tmdO);
    tma_prefetch_desc(&tmAcc);
  }
  if (warp == 20) {
    tmem_alloc(smem_u32(&tmem_base_smem), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dep_wait();
  const uint32_t tmem_base = tmem_base_smem;
  const float c2 = scale * IL_LOG2E;
  int fail = 0;

  if (warp == 23) {
    // ---------------------------------------------------------------- loads
    // lse (log2 units) and delta of a step's queries, by plain loads: into registers two steps ahead of the tiles, into shared
    // memory one step ahead.  Slot of step g + 1 = slot of step g - NST, whose readers are done: the stage of that step was
    // waited for.
    static_assert(VST == NST + 1, "a slot is free when the tiles of the step before its next use are requested");
    int v_item = blockIdx.x, v_it = 0, v_g = 0;
    float v_lse[4], v_del[4];
    auto fetch_vectors = [&]() {
      if (v_item >= nitems) return;
      const FusedItem w = fused_item(v_item, nbh, H, B, nq);
      const float* lse_b = lse + ((size_t)w.bs * H + w.h) * T;
      const float* del_b = delta + ((size_t)w.nb * H + w.h) * T;
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) {
        const int q = (w.kb + v_it) * TQ + q4 * 32 + lane;
        v_lse[q4] = q < T ? lse_b[q] : 0.f;
        v_del[q4] = q < T ? del_b[q] : 0.f;
      }
    };
    auto put_vectors = [&]() {                                   // ... and the next ones are asked for
      if (v_item >= nitems) return;
      float* vec = s_vec + (v_g % VST) * (2 * TQ);
#pragma unroll
      for (int q4 = 0; q4 < 4; ++q4) {
        vec[q4 * 32 + lane] = v_lse[q4] * IL_LOG2E;
        vec[TQ + q4 * 32 + lane] = v_del[q4];
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_vec(v_g % VST));            // its release publishes the warp's stores
      ++v_g;
      if (++v_it == fused_item(v_item, nbh, H, B, nq).nit) { v_it = 0; v_item += gridDim.x; }
      fetch_vectors();
    };
    fetch_vectors();
    put_vectors();
    int g = 0, n_item = 0;
    for (int item = blockIdx.x; item < nitems && !fail; item += gridDim.x, ++n_item) {
      const FusedItem w = fused_item(item, nbh, H, B, nq);
      for (int it = 0; it < w.nit; ++it) {
        const int gs = g + it, st = gs % NST, j = w.kb + it;
        int ok = 1;
        if (lane == 0 && gs >= NST) ok = mbar_wait(bar_empty(st), (uint32_t)(gs / NST - 1) & 1u, abortp) ? 1 : 0;
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) { fail = 1; abort_flag = 1; break; }
        if (lane == 0) {
          mbar_expect_tx(bar_full(st), 2 * C::ROW_BYTES);
          tma_load_4d(sQ0 + st * STAGE, &tmRow, 0, w.h, j * TQ, w.bs, bar_full(st));
          tma_load_4d(sQ0 + st * STAGE + C::ROW_BYTES, &tmdO, 0, w.h, j * TQ, w.nb, bar_full(st));
        }
        if (it == 0) {
          // the item's K and V: their buffer is free once the previous item's last products that read them have retired
          int ok2 = 1;
          const int kb = n_item % KVB;
          if (lane == 0 && n_item >= KVB) ok2 = mbar_wait(bar_kvfree(kb), (uint32_t)(n_item / KVB - 1) & 1u, abortp) ? 1 : 0;
          ok2 = __shfl_sync(0xffffffffu, ok2, 0);
          if (!ok2) { fail = 1; abort_flag = 1; break; }
          if (lane == 0) {
            mbar_expect_tx(bar_kv(kb), 2 * C::ROW_BYTES);
            tma_load_4d(sKV + kb * STAGE, &tmRow, 0, H + w.h, w.kb * TQ, w.bs, bar_kv(kb));
            tma_load_4d(sKV + kb * STAGE + C::ROW_BYTES, &tmRow, 0, 2 * H + w.h, w.kb * TQ, w.bs, bar_kv(kb));
          }
        }
        put_vectors();
      }
      g += w.nit;
    }
    grid_dep_launch();
  } else if (warp == 20 || warp == 21) {
    // ---------------------------------------------------------------- MMA issue: S and dV, dP and dK
    // A thread issues small MMAs no faster than one per ~60 cycles, a commit costs it 120, a look at a barrier 150, and every
    // hand-over between threads a round trip of several hundred.  One thread does S and dV, the other dP and dK: in program
    // order (the tensor pipe keeps one thread's MMAs in order) a half's product and then the next step's scores of that half,
    // into the columns the product has just read.  Each accumulator belongs to one thread, so its sums have a fixed order.
    if (lane == 0) {
      const int x = warp - 20;
      constexpr uint32_t idesc_s = make_idesc_bf16(TQ, TK, 0, 0);          // S^T / dP^T half: M128 N64, both K-major
      constexpr uint32_t idesc_g = make_idesc_bf16(TQ, DH, 0, 1);          // dV / dK: A from TMEM, B MN-major
      const SmemDescBase rows = make_smem_desc_base(sKV + (x ? C::ROW_BYTES : 0), 16, 1024);             // K / V
      const SmemDescBase cols = make_smem_desc_base(sQ0 + (x ? C::ROW_BYTES : 0), 16, 1024);             // Q / dO
      const SmemDescBase other = make_smem_desc_base(sQ0 + (x ? 0 : C::ROW_BYTES), TQ * 128, 1024);      // dO / Q
      const uint32_t t_s = tmem_base + (x ? C::C_DP : C::C_S), t_acc = tmem_base + (x ? C::C_DK : C::C_DV);
      bool ok = true;
      // scores of half hf of the step held in stage st: rows 64 hf .. 64 hf + 63 of its tile (8 KB further)
      auto issue_scores = [&](int hf, int st, int kb) {
        const uint32_t so = (uint32_t)st * STAGE + (uint32_t)hf * (TK * 128), ko = (uint32_t)kb * STAGE;
#pragma unroll
        for (int ks = 0; ks < DH / 16; ++ks)
          umma_bf16(t_s + 64 * hf, desc_at(rows, ko + ks * 32), desc_at(cols, so + ks * 32), idesc_s, ks ? 1u : 0u);
        umma_commit(bar_s(hf));
      };
      int g = 0, n_item = 0;
      for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x, ++n_item) {
        const FusedItem w = fused_item(item, nbh, H, B, nq);
        const int kb = n_item % KVB;
        // first step of the item: its scores need the item's K / V and the step's Q / dO (the score columns are free:
        // this thread's own last products of the previous item come before them in the pipe)
        if (!mbar_wait(bar_kv(kb), (uint32_t)(n_item / KVB) & 1u, abortp)) { ok = false; break; }
        if (!mbar_wait(bar_full(g % NST), (uint32_t)(g / NST) & 1u, abortp)) { ok = false; break; }
        tc_fence_after();
        issue_scores(0, g % NST, kb);
        issue_scores(1, g % NST, kb);
        // the accumulator still holds the previous item's dV / dK until it has been stored
        if (n_item > 0 && !mbar_wait(bar_accfree, (uint32_t)(n_item - 1) & 1u, abortp)) { ok = false; break; }
        for (int it = 0; it < w.nit && ok; ++it) {
          const int gs = g + it, st = gs % NST, st1 = (gs + 1) % NST;
          const uint32_t ph = (uint32_t)gs & 1u;
          const bool more = it + 1 < w.nit;
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            if (!mbar_wait(bar_p(hf), ph, abortp)) { ok = false; break; }
            tc_fence_after();
            // dV += P^T dO / dK += dS^T Q: contraction over the half's 64 queries (MN-major B: 16 queries = 2048 B)
            const uint32_t so = (uint32_t)st * STAGE + (uint32_t)hf * (TK * 128);
#pragma unroll
            for (int ks = 0; ks < TK / 16; ++ks)
              umma_bf16_ts(t_acc, t_s + 64 * hf + packed_col(ks), desc_at(other, so + ks * 2048), idesc_g, (it | hf | ks) ? 1u : 0u);
            if (hf == 1) umma_commit(bar_empty(st));          // (one of two arrivals) this thread's products have read the stage
            if (more) {
              if (hf == 0 && !mbar_wait(bar_full(st1), (uint32_t)((gs + 1) / NST) & 1u, abortp)) { ok = false; break; }
              issue_scores(hf, st1, kb);
            }
          }
        }
        if (!ok) break;
        umma_commit(bar_kvfree(kb));                          // (one of three) nothing of this item reads K / V from this thread any more
        umma_commit(bar_acc);                                 // (one of two) dV / dK is complete
        g += w.nit;
      }
      if (!ok) { fail = 1; abort_flag = 1; }
      umma_commit(bar_drain(x));                   // every MMA this thread issued has retired before TMEM goes
      int never = 0;
      mbar_wait(bar_drain(x), 0, &never);
    }
  } else if (warp == 22) {
    // ---------------------------------------------------------------- MMA issue, third thread: dQ
    if (lane == 0) {
      constexpr uint32_t idesc_q = make_idesc_bf16(TQ, DH, 1, 1);          // A = dS (MN-major), B = K (MN-major)
      const SmemDescBase dk_mn = make_smem_desc_base(sKV, TQ * 128, 1024);
      const SmemDescBase dds_mn = make_smem_desc_base(sDS, TQ * 128, 1024);
      bool ok = true;
      int g = 0, n_item = 0;
      for (int item = blockIdx.x; item < nitems && ok; item += gridDim.x, ++n_item) {
        const FusedItem w = fused_item(item, nbh, H, B, nq);
        const int kb = n_item % KVB;
        const uint32_t ko = (uint32_t)kb * STAGE;
        if (!mbar_wait(bar_kv(kb), (uint32_t)(n_item / KVB) & 1u, abortp)) { ok = false; break; }     // this item's K is in place
        for (int it = 0; it < w.nit && ok; ++it) {
          const int gs = g + it, b = gs & 1;
          // dQ(step) = dS K over this tile's 128 keys: both halves of dS are in shared memory (bar_ds; the item's K
          // arrived before the scores that dS came from), buffer b of the accumulator is free once the flush of
          // step gs-2 is done
          if (!mbar_wait(bar_ds(b), (uint32_t)(gs >> 1) & 1u, abortp)) { ok = false; break; }
          if (gs >= 2 && !mbar_wait(bar_dqfree(b), (uint32_t)((gs >> 1) - 1) & 1u, abortp)) { ok = false; break; }
          tc_fence_after();
#pragma unroll
          for (int ks = 0; ks < TQ / 16; ++ks)
            umma_bf16(tmem_base + C::C_DQ + 64 * b, desc_at(dds_mn, (uint32_t)b * C::DS_BYTES + ks * 2048), desc_at(dk_mn, ko + ks * 2048),
                      idesc_q, ks ? 1u : 0u);
          umma_commit(bar_dq(b));
          if (it + 1 == w.nit) umma_commit(bar_kvfree(kb));      // (one of three)
        }
        g += w.nit;
      }
      if (!ok) { fail = 1; abort_flag = 1; }
      umma_commit(bar_drain(2));
      int never = 0;
      mbar_wait(bar_drain(2), 0, &never);
    }
  } else if (warp >= 16 && warp < 20) {
    // ---------------------------------------------------------------- dQ flush and dV / dK store (warps 16-19: thread = row)
    const int r = tid - 512;
    const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    // (a warp's rows are its own throughout: waits, staging and reductions need no meeting of the four)
    auto wait = [&](uint32_t bar, uint32_t parity) -> bool { return __all_sync(0xffffffffu, mbar_wait(bar, parity, abortp)); };
    // an item's dV and dK: this thread's key row, scaled and rounded to bf16
    auto store_item = [&](const FusedItem& w, int n_item) -> bool {
      if (!wait(bar_acc, (uint32_t)n_item & 1u)) return false;
      tc_fence_after();
      const int key = w.kb * TQ + r;
      bf16* rowp = dqkv + ((size_t)w.nb * T + key) * (3 * d) + w.h * DH;
#pragma unroll
      for (int which = 0; which < 2; ++which) {
        bf16* dst = rowp + (which == 0 ? 2 * d : d);
        const float f = which == 0 ? 1.0f : scale;
        const uint32_t tcol = t_lane + (which == 0 ? C::C_DV : C::C_DK);
#pragma unroll
        for (int c0 = 0; c0 < DH; c0 += 32) {
          uint32_t rr[32];
          tmem_ld_32x32(tcol + c0, rr);
          tmem_ld_wait();
          if (key < T) {
#pragma unroll
            for (int i = 0; i < 32; i += 8) {
              uint4 pk;
              pk.x = pack_bf16x2(__uint_as_float(rr[i]) * f, __uint_as_float(rr[i + 1]) * f);
              pk.y = pack_bf16x2(__uint_as_float(rr[i + 2]) * f, __uint_as_float(rr[i + 3]) * f);
              pk.z = pack_bf16x2(__uint_as_float(rr[i + 4]) * f, __uint_as_float(rr[i + 5]) * f);
              pk.w = pack_bf16x2(__uint_as_float(rr[i + 6]) * f, __uint_as_float(rr[i + 7]) * f);
              *reinterpret_cast<uint4*>(dst + c0 + i) = pk;
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_accfree);               // the accumulators may be overwritten by the next item
      return true;
    };
    int g = 0, n_item = 0;
    for (int item = blockIdx.x; item < nitems && !fail; item += gridDim.x, ++n_item) {
      const FusedItem w = fused_item(item, nbh, H, B, nq);
      for (int it = 0; it < w.nit; ++it) {
        const int gs = g + it, b = gs & 1;
        // (before the last dQ block: the next item's first products wait for the accumulators)
        if (it + 1 == w.nit && !store_item(w, n_item)) { fail = 1; abort_flag = 1; break; }
        if (!wait(bar_dq(b), (uint32_t)(gs >> 1) & 1u)) { fail = 1; abort_flag = 1; break; }
        tc_fence_after();
        // The warp's 32 rows go to the global accumulator as one bulk reduction per 32 columns: they are staged in the dS
        // buffer of this step (its dQ product, the only reader, has retired) in the 128-byte-swizzled layout of the tensor
        // map, and one thread issues cp.reduce.async.bulk.tensor (rows past the sequence end are dropped by the map's bounds).
        const uint32_t stage = sDS + (uint32_t)b * C::DS_BYTES;
#pragma unroll
        for (int c0 = 0; c0 < DH; c0 += 32) {
          uint32_t rr[32];
          tmem_ld_32x32(t_lane + C::C_DQ + 64 * b + c0, rr);
          tmem_ld_wait();
          const uint32_t rowaddr = stage + (uint32_t)(c0 / 32) * (TQ * 128) + (uint32_t)r * 128;
#pragma unroll
          for (int t = 0; t < 8; ++t)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(rowaddr + (((uint32_t)t ^ (uint32_t)(r & 7)) * 16)), "r"(rr[4 * t]),
                         "r"(rr[4 * t + 1]), "r"(rr[4 * t + 2]), "r"(rr[4 * t + 3])
                         : "memory");
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_dqfree(b));               // the TMEM buffer has been read
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          const int row0 = (w.kb + it) * TQ + (warp & 3) * 32;
          if (row0 < T) {
#pragma unroll
            for (int c0 = 0; c0 < DH; c0 += 32)
              tma_reduce_add_3d(&tmAcc, stage + (uint32_t)(c0 / 32) * (TQ * 128) + (uint32_t)(warp & 3) * (32 * 128), w.h * DH + c0, row0, w.nb);
          }
          bulk_commit_group();
          bulk_wait_group_read0();                               // the staging has been read: the buffer may be rewritten
          mbar_arrive(bar_dsfree(b));
        }
        __syncwarp();
      }
      if (fail) break;
      g += w.nit;
    }
    if (lane == 0) bulk_wait_group0();                         // every reduction this thread issued has reached memory
  } else if (warp < FUSED_RW) {
    // ---------------------------------------------------------------- recompute and convert (warps 0-15)
    // Warps 0-7 take the first half of every step, 8-15 the second; thread = key row r, query columns 32 hc .. 32 hc + 31 of
    // the half.
    const int x = warp >> 3, hc = (warp >> 2) & 1, r = tid & 127;
    const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t t_s = t_lane + C::C_S + 64 * x + 32 * hc, t_dp = t_lane + C::C_DP + 64 * x + 32 * hc;
    auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
      if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
      return __all_sync(0xffffffffu, mbar_wait(bar, parity, abortp));
    };
    int g = 0;
    for (int item = blockIdx.x; item < nitems && !fail; item += gridDim.x) {
      const FusedItem w = fused_item(item, nbh, H, B, nq);
      const int key = w.kb * TQ + r;
      for (int it = 0; it < w.nit; ++it) {
        const int gs = g + it, b = gs & 1, j = w.kb + it;
        const float4* lv = reinterpret_cast<const float4*>(s_vec + (gs % VST) * (2 * TQ) + 64 * x + 32 * hc);
        const float4* dv_ = reinterpret_cast<const float4*>(s_vec + (gs % VST) * (2 * TQ) + TQ + 64 * x + 32 * hc);
        if (!wait(bar_vec(gs % VST), (uint32_t)(gs / VST) & 1u) || !wait(bar_s(x), (uint32_t)gs & 1u)) { fail = 1; abort_flag = 1; break; }
        tc_fence_after();
        const bool masked = it == 0 || j * TQ + TQ > T;    // uniform: some queries precede some keys, or lie past the sequence
        const int qbase = j * TQ + 64 * x + 32 * hc;
        uint32_t dw[16];
#pragma unroll
        for (int c = 0; c < 2; ++c) {                      // 16 columns at a time: the register budget of 768 threads
          uint32_t s[16], dp[16], pw[8], dc[8];
          tmem_ld_32x16(t_s + 16 * c, s);
          tmem_ld_32x16(t_dp + 16 * c, dp);
          tmem_ld_wait();
          float p[16];
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            const float4 l = lv[4 * c + i / 4];
            p[i] = ex2_fast(fmaf(__uint_as_float(s[i]), c2, -l.x));
            p[i + 1] = ex2_fast(fmaf(__uint_as_float(s[i + 1]), c2, -l.y));
            p[i + 2] = ex2_fast(fmaf(__uint_as_float(s[i + 2]), c2, -l.z));
            p[i + 3] = ex2_fast(fmaf(__uint_as_float(s[i + 3]), c2, -l.w));
          }
          if (masked) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (qbase + 16 * c + i < key || qbase + 16 * c + i >= T) p[i] = 0.f;
          }
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            const float4 e = dv_[4 * c + i / 4];
            dc[i / 2] = pack_bf16x2((__uint_as_float(dp[i]) - e.x) * p[i], (__uint_as_float(dp[i + 1]) - e.y) * p[i + 1]);
            dc[i / 2 + 1] = pack_bf16x2((__uint_as_float(dp[i + 2]) - e.z) * p[i + 2], (__uint_as_float(dp[i + 3]) - e.w) * p[i + 3]);
            pw[i / 2] = pack_bf16x2(p[i], p[i + 1]);
            pw[i / 2 + 1] = pack_bf16x2(p[i + 2], p[i + 3]);
          }
          tmem_st_32x8(t_s + 8 * c, pw);                   // P^T over columns this thread has read
          tmem_st_32x8(t_dp + 8 * c, dc);                  // dS^T likewise
#pragma unroll
          for (int i = 0; i < 8; ++i) dw[8 * c + i] = dc[i];
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_p(x));              // dV / dK of this half can go
        // dS as the A operand of dQ = dS K: row = key, 64 queries of half x = one swizzled 128-byte row of chunk x.  Its
        // buffer is free once the dQ block of step gs-2, staged in it after its product, has been handed to the bulk reduction.
        if (gs >= 2 && !wait(bar_dsfree(b), (uint32_t)((gs >> 1) - 1) & 1u)) { fail = 1; abort_flag = 1; break; }
        const uint32_t rowaddr = sDS + (uint32_t)b * C::DS_BYTES + (uint32_t)x * (TQ * 128) + (uint32_t)r * 128;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const uint32_t unit = (uint32_t)(4 * hc + t) ^ (uint32_t)(r & 7);
          asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(rowaddr + unit * 16), "r"(dw[4 * t]), "r"(dw[4 * t + 1]),
                       "r"(dw[4 * t + 2]), "r"(dw[4 * t + 3])
                       : "memory");
        }
        fence_proxy_async();                               // the dS rows are read by the tensor pipe (async proxy)
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_ds(b));
      }
      g += w.nit;
    }
  }
  fail = __syncthreads_or(fail);
  if (tid == 0 && fail && err) atomicExch(err, DEV_TIMEOUT_MMA);
  tc_fence_before();
  __syncthreads();
  if (warp == 20) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// dqkv[row, h*dh + c] (the Q third) = bf16(scale * dq_acc[row, h*dh + c]): the accumulated dQ leaves fp32 here.
__global__ void __launch_bounds__(256) attn_dq_convert_kernel(const float* __restrict__ acc, bf16* __restrict__ dqkv, size_t rows,
                                                              int d, float scale) {
  grid_dep_wait();
  const int d8 = d >> 3;
  const size_t total = rows * (size_t)d8;
  for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < total; i += (size_t)gridDim.x * 256) {
    const size_t row = i / d8;
    const int c = (int)(i % d8) * 8;
    const float4 a = *reinterpret_cast<const float4*>(acc + row * d + c);
    const float4 b = *reinterpret_cast<const float4*>(acc + row * d + c + 4);
    uint4 o;
    o.x = pack_bf16x2(a.x * scale, a.y * scale);
    o.y = pack_bf16x2(a.z * scale, a.w * scale);
    o.z = pack_bf16x2(b.x * scale, b.y * scale);
    o.w = pack_bf16x2(b.z * scale, b.w * scale);
    *reinterpret_cast<uint4*>(dqkv + row * (size_t)(3 * d) + c) = o;
  }
}

// delta[nb, h, t] = sum_c dO[nb*T+t, h*dh+c] * O[(nb%B)*T+t, h*dh+c].  A thread takes 8 consecutive columns
// (16 bytes of each operand); the dh/8 threads of a (row, head) sit in one warp and combine by shuffles.
// With dq_zero != NULL the same threads also clear their 8 columns of the fp32 dQ accumulator [NB*T, H*dh] that the
// one-sweep backward adds into.
template <int DH>
__global__ void __launch_bounds__(256) attn_delta_tc_kernel(const bf16* __restrict__ dout, const bf16* __restrict__ o,
                                                            float* __restrict__ delta, float* __restrict__ dq_zero, int NB,
                                                            int B, int T, int H) {
  grid_dep_wait();
  constexpr int TPR = (DH == 80) ? 16 : DH / 8;      // threads per (row, head): a power of two (dh 80: 10 of 16 active)
  const long long gid = (long long)blockIdx.x * 256 + threadIdx.x;
  const long long item = gid / TPR;                  // (row, head) index
  const int part = (int)(gid % TPR);
  const long long total = (long long)NB * T * H;
  float s = 0.f;
  int h = 0;
  long long row = 0;
  if (item < total) {
    h = (int)(item % H);
    row = item / H;
    const int nb = (int)(row / T), t = (int)(row % T);
    if (part * 8 < DH) {
      const int d = H * DH;
      if (dq_zero) {
        float4* z = reinterpret_cast<float4*>(dq_zero + (size_t)row * d + h * DH + part * 8);
        z[0] = make_float4(0.f, 0.f, 0.f, 0.f);
        z[1] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
      const uint4 a = *reinterpret_cast<const uint4*>(dout + (size_t)row * d + h * DH + part * 8);
      const uint4 c = *reinterpret_cast<const uint4*>(o + ((size_t)(nb % B) * T + t) * d + h * DH + part * 8);
      const __nv_bfloat162* a2 = reinterpret_cast<const __nv_bfloat162*>(&a);
      const __nv_bfloat162* c2 = reinterpret_cast<const __nv_bfloat162*>(&c);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 x = __bfloat1622float2(a2[i]), y = __bfloat1622float2(c2[i]);
        s += x.x * y.x + x.y * y.y;
      }
    }
  }
  grid_dep_launch();
#pragma unroll
  for (int off = TPR / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (item < total && part == 0) {
    const int nb = (int)(row / T), t = (int)(row % T);
    delta[((size_t)nb * H + h) * T + t] = s;
  }
}

template <int DH>
cudaError_t delta_launch(const bf16* dout, const bf16* o, float* delta, float* dq_zero, int NB, int B, int T, int H, cudaStream_t s) {
  constexpr int TPR = (DH == 80) ? 16 : DH / 8;
  const long long nthreads = (long long)NB * T * H * TPR;
  return launch_dep(attn_delta_tc_kernel<DH>, dim3((unsigned)((nthreads + 255) / 256)), dim3(256), 0, s, dout, o, delta, dq_zero, NB, B, T, H);
}

template <int DH>
cudaError_t bwd_tc_launch(const bf16* qkv, const bf16* o, const float* lse, const bf16* dout, bf16* dqkv, float* delta, int NB,
                          int B, int T, int H, unsigned* err, cudaStream_t s) {
  cudaError_t e = delta_launch<DH>(dout, o, delta, nullptr, NB, B, T, H, s);
  if (e != cudaSuccess) return e;
  if constexpr (DH <= 128) {
    return attention_bwd_sweep(qkv, lse, dout, dqkv, delta, NB, B, T, H, DH, err, s);
  } else {
    using C = BwdCfg<DH>;
    const unsigned long long d3 = 3ull * H * DH, d1 = (unsigned long long)H * DH;
    const unsigned long long dims[4] = {(unsigned long long)DH, 3ull * H, (unsigned long long)T, (unsigned long long)B};
    const unsigned long long strides[3] = {(unsigned long long)DH * 2, d3 * 2, (unsigned long long)T * d3 * 2};
    const unsigned long long ddims[4] = {(unsigned long long)DH, (unsigned long long)H, (unsigned long long)T, (unsigned long long)NB};
    const unsigned long long dstrides[3] = {(unsigned long long)DH * 2, d1 * 2, (unsigned long long)T * d1 * 2};
    const unsigned box128[4] = {64, 1, TQ, 1}, box64[4] = {64, 1, TK, 1};
    CUtensorMap tmRow, tmBlk, tmdO64, tmdO128;
    if (!tma_encode_bf16(&tmRow, qkv, 4, dims, strides, box128) || !tma_encode_bf16(&tmBlk, qkv, 4, dims, strides, box64) ||
        !tma_encode_bf16(&tmdO64, dout, 4, ddims, dstrides, box64) || !tma_encode_bf16(&tmdO128, dout, 4, ddims, dstrides, box128))
      return cudaErrorInvalidValue;
    e = cudaFuncSetAttribute(attn_bwd_dkv_tc_kernel<DH, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_KV);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(attn_bwd_dkv_tc_kernel<DH, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_KV);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(attn_bwd_dq_tc_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM_Q);
    if (e != cudaSuccess) return e;
    dim3 grid((T + TQ - 1) / TQ, NB * H);
    const float scale = rsqrtf((float)DH);
    launch_dep(attn_bwd_dkv_tc_kernel<DH, 1>, dim3(grid), dim3(256), C::SMEM_KV, s, tmRow, tmBlk, tmdO64, lse, delta, dqkv, B, T, H, scale, err);
    launch_dep(attn_bwd_dkv_tc_kernel<DH, 2>, dim3(grid), dim3(256), C::SMEM_KV, s, tmRow, tmBlk, tmdO64, lse, delta, dqkv, B, T, H, scale, err);
    launch_dep(attn_bwd_dq_tc_kernel<DH>, dim3(grid), dim3(256), C::SMEM_Q, s, tmRow, tmBlk, tmdO128, lse, delta, dqkv, B, T, H, scale, err);
    return cudaGetLastError();
  }
}

// One-sweep backward: delta (+ clearing the accumulator), the sweep, then dQ from fp32 to bf16.
template <int DH>
cudaError_t bwd_fused_launch(const bf16* qkv, const bf16* o, const float* lse, const bf16* dout, bf16* dqkv, float* delta,
                             float* dq_acc, int NB, int B, int T, int H, unsigned* err, cudaStream_t s) {
  using C = FusedCfg<DH>;
  const unsigned long long d3 = 3ull * H * DH, d1 = (unsigned long long)H * DH;
  const unsigned long long dims[4] = {(unsigned long long)DH, 3ull * H, (unsigned long long)T, (unsigned long long)B};
  const unsigned long long strides[3] = {(unsigned long long)DH * 2, d3 * 2, (unsigned long long)T * d3 * 2};
  const unsigned long long ddims[4] = {(unsigned long long)DH, (unsigned long long)H, (unsigned long long)T, (unsigned long long)NB};
  const unsigned long long dstrides[3] = {(unsigned long long)DH * 2, d1 * 2, (unsigned long long)T * d1 * 2};
  const unsigned box128[4] = {64, 1, TQ, 1};
  CUtensorMap tmRow, tmdO, tmAcc;
  if (!tma_encode_bf16(&tmRow, qkv, 4, dims, strides, box128) || !tma_encode_bf16(&tmdO, dout, 4, ddims, dstrides, box128))
    return cudaErrorInvalidValue;
  // the fp32 dQ accumulator [NB, T, d] as the target of the bulk reductions: boxes of 32 columns x 32 rows of one sequence
  const unsigned long long adims[3] = {d1, (unsigned long long)T, (unsigned long long)NB};
  const unsigned long long astrides[2] = {d1 * 4, (unsigned long long)T * d1 * 4};
  const unsigned abox[3] = {32, 32, 1};
  if (!tma_encode_f32(&tmAcc, dq_acc, 3, adims, astrides, abox)) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(attn_bwd_fused_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  if ((e = delta_launch<DH>(dout, o, delta, dq_acc, NB, B, T, H, s)) != cudaSuccess) return e;
  // persistent CTAs, one per SM, each walking its share of the (key tile, sequence, head) items
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const long long nitems = (long long)((T + TQ - 1) / TQ) * NB * H;
  const int grid = (int)(nitems < sms ? nitems : sms);
  const float scale = rsqrtf((float)DH);
  launch_dep(attn_bwd_fused_kernel<DH>, dim3(grid), dim3(FUSED_THREADS), C::SMEM, s, tmRow, tmdO, tmAcc, lse, delta, dqkv, NB, B, T, H, scale, err);
  const size_t rows = (size_t)NB * T;
  size_t blocks = (rows * (size_t)(H * DH / 8) + 255) / 256;
  if (blocks > 148 * 16) blocks = 148 * 16;
  launch_dep(attn_dq_convert_kernel, dim3((unsigned)blocks), dim3(256), 0, s, dq_acc, dqkv, rows, H * DH, scale);
  return cudaGetLastError();
}

}  // namespace

cudaError_t attention_fwd(const bf16* qkv, bf16* o, float* lse, int B, int T, int H, int dh, unsigned* err,
                          cudaStream_t s) {
  if (((uintptr_t)qkv % 16) || ((uintptr_t)o % 16) || ((uintptr_t)lse % 4)) return cudaErrorInvalidValue;
  switch (dh) {
    case 32: return T > FWD_ONE_TILE_T ? fwd_pair_launch<32>(qkv, o, lse, B, T, H, err, s) : fwd_tc_launch<32>(qkv, o, lse, B, T, H, err, s);
    case 64: return T > FWD_ONE_TILE_T ? fwd_pair_launch<64>(qkv, o, lse, B, T, H, err, s) : fwd_tc_launch<64>(qkv, o, lse, B, T, H, err, s);
    case 80: return T > FWD_ONE_TILE_T ? fwd_pair_launch<80>(qkv, o, lse, B, T, H, err, s) : fwd_tc_launch<80>(qkv, o, lse, B, T, H, err, s);
    case 128: return T > FWD_ONE_TILE_T ? fwd_pair_launch<128>(qkv, o, lse, B, T, H, err, s) : fwd_tc_launch<128>(qkv, o, lse, B, T, H, err, s);
    case 256: return fwd_tc_launch<256>(qkv, o, lse, B, T, H, err, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t attention_bwd(const bf16* qkv, const bf16* o, const float* lse, const bf16* dout, bf16* dqkv, float* delta,
                          float* dq_acc, int NB, int B, int T, int H, int dh, unsigned* err, cudaStream_t s) {
  // o is read with 16-byte loads by the delta kernel, qkv / dout / dqkv by TMA and 16-byte stores
  if (((uintptr_t)qkv % 16) || ((uintptr_t)o % 16) || ((uintptr_t)dout % 16) || ((uintptr_t)dqkv % 16) ||
      ((uintptr_t)lse % 4) || ((uintptr_t)delta % 4))
    return cudaErrorInvalidValue;
  if (T <= ATTN_BWD_SHORT_T) return attention_bwd_short(qkv, lse, dout, dqkv, NB, B, T, H, dh, err, s);
  if (dq_acc && (dh == 32 || dh == 64)) {        // one sweep, dQ summed over key tiles in the fp32 accumulator
    if ((uintptr_t)dq_acc % 16) return cudaErrorInvalidValue;
    return dh == 32 ? bwd_fused_launch<32>(qkv, o, lse, dout, dqkv, delta, dq_acc, NB, B, T, H, err, s)
                    : bwd_fused_launch<64>(qkv, o, lse, dout, dqkv, delta, dq_acc, NB, B, T, H, err, s);
  }
  switch (dh) {
    case 32: return bwd_tc_launch<32>(qkv, o, lse, dout, dqkv, delta, NB, B, T, H, err, s);
    case 64: return bwd_tc_launch<64>(qkv, o, lse, dout, dqkv, delta, NB, B, T, H, err, s);
    case 80: return bwd_tc_launch<80>(qkv, o, lse, dout, dqkv, delta, NB, B, T, H, err, s);
    case 128: return bwd_tc_launch<128>(qkv, o, lse, dout, dqkv, delta, NB, B, T, H, err, s);
    case 256: return bwd_tc_launch<256>(qkv, o, lse, dout, dqkv, delta, NB, B, T, H, err, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace il

