// The per-use check of the attention D use, and the kernels that evaluate a fresh read of the saved
// output through Eq. dterm itself.
//
// dS = P o (dP - D) is affine in the correction term D, and so are dQ = c dS K and dK = c dS^T Q.
// With D_k = rowsum(dO o O_k) the term under the k-th fresh rounding of the saved output and D* the
// reference's (from the original output), draw k differs from the reference gradient by
//
//     dQ_k - dQ* = -c diag(D_k - D*) (P K)            dK_k - dK* = -c P^T diag(D_k - D*) Q
//
// and dV does not move at all.  The Monte-Carlo check needs exactly these differences (its sums are
// S1 = sum_k (g_k - g*), S2 = sum_k (g_k - g*)^2), so the kernels here form them directly:
//   * dQ: row i of the difference is the row of P K scaled by (D_k - D*)[i], hence
//     S1 = -c (P K) o rowwise sum_k (D_k - D*),  S2 = c^2 (P K)^2 o rowwise sum_k (D_k - D*)^2:
//     one pass for P K (the forward kernel with K in place of V) and an elementwise kernel, whatever K;
//   * dK: one contraction per draw, P^T against the rows of Q scaled by -c (D_k - D*).  The
//     probabilities are formed once per step for four draws: the scaled Q tiles of the four draws lie
//     side by side as one 128 x 256 B operand, so a step is one product for S^T, one pass of the exp2
//     unit, and one 128 x 256 x 128 product.
// Rounding an operand to bf16 now costs 2^-9 of the *difference*, not of the whole dS, so the
// statistics see the read and not the operand format, and no per-draw gradient is ever written.
//
// attn_dk_diff_kernel: persistent, one CTA per SM walking (key block, head, set of draws) items, heaviest
// first; a CTA takes the draws of its set four at a time and adds to the sums in that order (sets as in
// attn_f8.cu, whose sum_sets_kernel joins them).  640 threads: warps 0..15 probabilities, operand scaling and
// epilogue (32 columns of S^T each), warp 16 TMA, warp 17 MMA issue.  Tensor memory: two S^T buffers of 128
// columns, four accumulators of 64.  P^T goes back into the columns its thread read S^T from (two K = 16
// steps per 32 columns, the first 16 of them), so the scores are double-buffered in the room that one buffer
// and a separate operand would take, and S^T of a step is formed under the exponentials and stores of the
// step before (B H = 128, S = 2048, causal, 32 draws: 1.68 ms; with one buffer, eight warps and a launch per four
// draws 1.89).  -LSE enters S^T through one extra K = 16 product step (a tile of ones against rows holding
// -LSE/c as three bf16 terms), written two steps ahead, so P^T = exp2(c2 acc) needs no per-column operand.
#include <limits.h>
#include <string.h>

#include <atomic>

#include "attn_common.cuh"
#include "mc_stats.cuh"

namespace bsp {

constexpr int kDkThreads = 640;
constexpr int kDkWarps = 16;
constexpr int kDkND = kDrawsPerPass;               // draws per pass over the steps
constexpr uint32_t kDkStages = 3;                  // ring of streamed Q tiles
constexpr uint32_t kDkBuf = kDkND * kAtTile;       // one buffer of scaled Q tiles (also the epilogue's 64 KB of staging)
constexpr int kDkBiasTile = AT_BLK * 16 * 2;       // 4 KB: one 128 x 16 bf16 tile of the extra K = 16 step
// shared memory: K tiles [2], Q ring [3], scaled Q tiles [2][4], barriers, the ones tile and three -LSE tiles
constexpr int kDkSmem = 1024 + (2 + (int)kDkStages + 2 * kDkND) * kAtTile + 1024 + 4 * kDkBiasTile;
static_assert(kDkSmem <= 232448, "dynamic shared memory of attn_dk_diff_kernel exceeds the SM's");

struct DkDiffParams {
  int BH, S, nblk, causal;
  float c;                       // softmax scale
  const float* lse;              // [BH*S]
  const float* d_ref;            // [BH*S]      the reference's correction term
  const float* d_draws;          // [K][BH*S]   the draws' correction terms
  int K, sets, passes;           // draws; sets per (block, head); passes of up to four draws per set
  float *s1, *s2;                // what tm_s1 and tm_s2 map
  int walk;                      // items from here on are left as after a wait that ran out (self-test; else all)
  bsp_diag_t* diag;
};

__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

__global__ void __launch_bounds__(kDkThreads, 1)
attn_dk_diff_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                    const __grid_constant__ CUtensorMap tm_s1, const __grid_constant__ CUtensorMap tm_s2,
                    DkDiffParams p) {
  grid_dependency();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  const uint32_t res_base = base;                                   // K tile of the pass, two buffers
  const uint32_t q0 = base + 2 * kAtTile;                           // stage s: q0 + s * kAtTile
  const uint32_t bs0 = q0 + kDkStages * kAtTile;                    // buffer pb, draw d: bs0 + pb * kDkBuf + d * kAtTile
  const uint32_t bars = bs0 + 2 * kDkBuf;
  const uint32_t b_res = bars, b_res_empty = bars + 16, b_sfull = bars + 32, b_sempty = bars + 56,
                 b_s_full = bars + 80 /* [2] */, b_op_ready = bars + 96 /* [2] */, b_op_free = bars + 112 /* [2] */,
                 b_acc = bars + 128, b_acc_free = bars + 136, b_bias = bars + 144 /* [3] */, b_staged = bars + 184,
                 b_stg_free = bars + 192;
  const uint32_t bias0 = bars + 1024;                               // ones tile; buffer b: the -LSE tile at 1 + b
  uint8_t* bars_gen = smem_raw + (bars - raw);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bars_gen + 208);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars_gen + 212);
  volatile int* items_out = abort_flag + 1;                         // items whose sums have been sent off whole

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nwork = p.nblk * p.BH * p.sets;
  // the CTA's n-th item: rounds of gridDim.x items, walked forwards and backwards in turn
  auto item_at = [&](int n) -> int {
    const int b = (int)blockIdx.x, G = (int)gridDim.x;
    return n * G + ((n & 1) ? G - 1 - b : b);
  };
  // draws [d_begin, d_end) of the item, in passes of up to kDkND
  auto decode = [&](int w, int& blk, int& bh, int& set, int& it_begin, int& nsteps, int& d_begin, int& d_end) {
    set = w % p.sets;
    const int i = w / p.sets;
    blk = i / p.BH;                                                 // key block j: steps i = j .. nblk-1 (causal)
    bh = i % p.BH;
    it_begin = p.causal ? blk : 0;
    nsteps = p.nblk - it_begin;
    d_begin = set * p.passes * kDkND;
    d_end = d_begin + p.passes * kDkND < p.K ? d_begin + p.passes * kDkND : p.K;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(b_res + 8 * s, 1); mbar_init(b_res_empty + 8 * s, 1); mbar_init(b_s_full + 8 * s, 1);
      mbar_init(b_op_ready + 8 * s, kDkWarps); mbar_init(b_op_free + 8 * s, 1);
    }
    for (uint32_t s = 0; s < kDkStages; ++s) { mbar_init(b_sfull + 8 * s, 1); mbar_init(b_sempty + 8 * s, 1); }
    for (uint32_t s = 0; s < 3; ++s) mbar_init(b_bias + 8 * s, 4);
    mbar_init(b_acc, 1); mbar_init(b_acc_free, kDkWarps);
    mbar_init(b_staged, kDkWarps); mbar_init(b_stg_free, 1);
    *abort_flag = 0;
    *items_out = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 256) {
    // constant parts of the four extra tiles: thread t clears 16 bytes of each (row t & 127, half t >> 7); the
    // first three columns of the ones tile are 1
    const int t0 = (int)threadIdx.x;
    const uint32_t off = (uint32_t)((t0 & 127) >> 3) * 256u + (uint32_t)(t0 >> 7) * 128u + (uint32_t)(t0 & 7) * 16u;
#pragma unroll
    for (uint32_t t = 0; t < 4; ++t) {
      const bool one = t == 0 && t0 < 128;
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %3};" ::"r"(bias0 + t * kDkBiasTile + off),
                   "r"(one ? 0x3F803F80u : 0u), "r"(one ? 0x00003F80u : 0u), "r"(0u) : "memory");
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 17) tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // two S^T buffers of 128 columns (P^T in place), the accumulator of draw d at t_acc + 64 d
  const uint32_t t_s = tmem, t_acc = tmem + 256;

  const uint32_t id_s = make_idesc(1u, 1u, 128, 128);                          // A, B K-major
  const uint32_t id_acc = make_idesc(1u, 1u, 128, 64 * kDkND) | (1u << 16);    // A from tensor memory, B MN-major

  // the block starts with 640 x 96 registers: the control warpgroup keeps 32 a thread, the others take 112
  if (warp >= kDkWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
    if (warp == 16) {
      // ------------------------------------------------ TMA producer
      if (lane == 0) {
        tma_prefetch_desc(&tm_q); tma_prefetch_desc(&tm_k);
        bool ok = true;
        uint32_t itg = 0, vi = 0;                                   // global step, pass
        int n = 0;
        for (int w = item_at(0); w < p.walk && ok; w = item_at(++n)) {
          int blk, bh, set, it_begin, nsteps, d0, d_end;
          decode(w, blk, bh, set, it_begin, nsteps, d0, d_end);
          for (; d0 < d_end && ok; d0 += kDkND, ++vi) {
            const uint32_t rb = vi & 1u;
            if (!mbar_wait(b_res_empty + 8 * rb, ((vi >> 1) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
            mbar_expect_tx(b_res + 8 * rb, kAtTile);
            tma_load_3d(res_base + rb * kAtTile, &tm_k, b_res + 8 * rb, 0, blk * AT_BLK, bh);
            for (int it = 0; it < nsteps; ++it, ++itg) {
              const uint32_t s = itg % kDkStages, ph = (itg / kDkStages) & 1u;
              if (!mbar_wait(b_sempty + 8 * s, ph ^ 1u, abort_flag)) { ok = false; break; }
              mbar_expect_tx(b_sfull + 8 * s, kAtTile);
              tma_load_3d(q0 + s * kAtTile, &tm_q, b_sfull + 8 * s, 0, (it_begin + it) * AT_BLK, bh);
            }
          }
        }
        if (!ok) for (int i = 0; i < 200; ++i) __nanosleep(1000);   // let copies in flight land
      }
    } else if (warp == 17) {
      // ------------------------------------------------ MMA issuer (the whole warp walks, one lane issues)
      const uint32_t leader = elect_one() ? 1u : 0u;
      auto wait_all = [&](uint32_t bar, uint32_t parity) -> bool {
        return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, abort_flag));
      };
      bool ok = true;
      uint32_t itg = 0, vi = 0;
      int n = 0;
      for (int w = item_at(0); w < p.walk && ok; w = item_at(++n)) {
        int blk, bh, set, it_begin, nsteps, d0, d_end;
        decode(w, blk, bh, set, it_begin, nsteps, d0, d_end);
        for (; d0 < d_end && ok; d0 += kDkND, ++vi) {
          const uint32_t rb = vi & 1u;
          const uint32_t k_t = res_base + rb * kAtTile;
          if (!wait_all(b_res + 8 * rb, (vi >> 1) & 1u)) { ok = false; break; }
          // S^T = K Q^T of global step jt (rows = keys), plus the K = 16 step that subtracts LSE / c, one step
          // ahead; its buffer is free once the product of two steps ago has read P^T there
          auto issue_s = [&](uint32_t jt) -> bool {
            const uint32_t s = jt % kDkStages, sb = jt & 1u, bb = jt % 3u;
            if (!wait_all(b_sfull + 8 * s, (jt / kDkStages) & 1u)) return false;
            if (!wait_all(b_op_free + 8 * sb, ((jt >> 1) & 1u) ^ 1u)) return false;
            if (!wait_all(b_bias + 8 * bb, (jt / 3u) & 1u)) return false;
            tc_fence_after();
            const uint64_t a = make_smem_desc(k_t), b = make_smem_desc(q0 + s * kAtTile);
#pragma unroll
            for (int k = 0; k < 4; ++k) tc_mma_l<false>(leader, t_s + 128u * sb, a + 2u * k, b + 2u * k, id_s, k != 0);
            tc_mma_l<false>(leader, t_s + 128u * sb, make_smem_desc_k16(bias0), make_smem_desc_k16(bias0 + (1u + bb) * kDkBiasTile), id_s, 1u);
            tc_commit_l(leader, b_s_full + 8 * sb);
            return true;
          };
          ok = issue_s(itg);
          for (int it = 0; it < nsteps && ok; ++it) {
            const uint32_t jg = itg + (uint32_t)it, s = jg % kDkStages, pb = jg & 1u;
            if (it + 1 < nsteps && !issue_s(jg + 1)) { ok = false; break; }
            if (!wait_all(b_op_ready + 8 * pb, (jg >> 1) & 1u)) { ok = false; break; }
            // the accumulators are free once the epilogue of the pass before has read them
            if (it == 0 && !wait_all(b_acc_free, (vi & 1u) ^ 1u)) { ok = false; break; }
            tc_fence_after();
            // all four draws at once: P^T (tensor memory, eight columns per 16 queries, 16 of every 32 columns)
            // against the four scaled Q tiles side by side (MN-major, one 128-byte atom of 64 columns per draw)
            const uint64_t bq = make_smem_desc_mn(bs0 + pb * kDkBuf, (uint32_t)kAtTile);
#pragma unroll
            for (uint32_t k = 0; k < 8; ++k)
              tc_mma_ts_l<false>(leader, t_acc, t_s + 128u * pb + 32u * (k >> 1) + 8u * (k & 1u), bq + 128u * k, id_acc,
                                 (it != 0 || k != 0) ? 1u : 0u);
            tc_commit_l(leader, b_op_free + 8 * pb);
            tc_commit_l(leader, b_sempty + 8 * s);
          }
          itg += (uint32_t)nsteps;
          if (ok) {
            tc_commit_l(leader, b_res_empty + 8 * rb);
            tc_commit_l(leader, b_acc);
          }
        }
      }
    }
  } else {
    // ------------------------------------------------ probabilities, operand scaling, epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    const int q4 = warp & 3, h = warp >> 2;                         // lane quarter; 32 of the 128 columns
    const int r = q4 * 32 + lane;                                   // row of the 128-row block: a key (S^T), a query (Q tile)
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    const uint32_t row_off = (uint32_t)r * 128u;
    const float c2 = p.c * kLog2e;
    const float bias_mul = -kLog2e / c2;                            // the accumulator holds s - LSE / c
    const size_t rows = (size_t)p.BH * p.S;
    bool ok = true, store_pending = false;
    uint32_t bias_written = 0, jt = 0, vi = 0, stg_ph = 0;          // -LSE rows written; global step, pass; last epilogue's phase
    // the pass whose accumulators have not been read yet
    bool due = false, e_first = true, e_last = true;
    int e_blk = 0, e_bh = 0, e_set = 0;
    // the -LSE row of one step (the warps of column quarter 0: thread r writes query r of the tile)
    auto bias_fetch = [&](int tbh, int step) -> float {
      const int q = step * AT_BLK + r;
      return q < p.S ? ldg(p.lse + (size_t)tbh * p.S + q) : 0.f;
    };
    auto bias_put = [&](uint32_t j, float rawv) {
      const float x = rawv * bias_mul;
      const __nv_bfloat16 h1 = __float2bfloat16_rn(x);
      const float r1 = x - __bfloat162float(h1);
      const __nv_bfloat16 h2 = __float2bfloat16_rn(r1);
      const __nv_bfloat16 h3 = __float2bfloat16_rn(r1 - __bfloat162float(h2));
      const uint32_t w0 = (uint32_t)__bfloat16_as_ushort(h1) | ((uint32_t)__bfloat16_as_ushort(h2) << 16);
      const uint32_t w1 = (uint32_t)__bfloat16_as_ushort(h3);
      const uint32_t tile = bias0 + (1u + j % 3u) * kDkBiasTile;
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %3};" ::"r"(tile + (uint32_t)(r >> 3) * 256u + (uint32_t)(r & 7) * 16u),
                   "r"(w0), "r"(w1), "r"(0u) : "memory");
    };
    // Reads the accumulators of pass `v` (its last global step: last) and adds the draws' sum and sum of squares to
    // S1 and S2 (the first pass of an item sets them), staged in that step's operand buffer, which no product reads
    // any more.
    auto epilogue = [&](uint32_t v, uint32_t last) -> bool {
      if (!__all_sync(0xFFFFFFFFu, mbar_wait(b_acc, v & 1u, abort_flag))) return false;
      tc_fence_after();
      const uint32_t stg = bs0 + (last & 1u) * kDkBuf;
      float s1[16], s2[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) s1[e] = s2[e] = 0.f;
#pragma unroll
      for (int d = 0; d < kDkND; ++d) {                             // (draws that a pass does not have add zeros)
        uint32_t a[16];
        tmem_ld16(t_acc + 64u * d + lane_off + h * 16, a);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float g = __uint_as_float(a[e]);
          s1[e] += g;
          s2[e] = fmaf(g, g, s2[e]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_acc_free);
      // box h >> 1 of 32 columns, four 16-byte chunks of this thread's half of it
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const uint32_t at = stg + (uint32_t)(h >> 1) * 16384u + row_off + ((uint32_t)(((h & 1) * 4 + t) ^ (r & 7)) << 4);
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at), "f"(s1[4 * t]), "f"(s1[4 * t + 1]), "f"(s1[4 * t + 2]),
                     "f"(s1[4 * t + 3]) : "memory");
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at + 32768u), "f"(s2[4 * t]), "f"(s2[4 * t + 1]),
                     "f"(s2[4 * t + 2]), "f"(s2[4 * t + 3]) : "memory");
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(b_staged);
      if (warp == 0 && !__all_sync(0xFFFFFFFFu, mbar_wait(b_staged, v & 1u, abort_flag))) return false;
      if (warp == 0 && lane == 0) {
        const int y = e_blk * AT_BLK, z = e_set * p.BH + e_bh;
        if (e_first) {
          tma_store_3d(&tm_s1, stg, 0, y, z);
          tma_store_3d(&tm_s1, stg + 16384u, 32, y, z);
          tma_store_3d(&tm_s2, stg + 32768u, 0, y, z);
          tma_store_3d(&tm_s2, stg + 49152u, 32, y, z);
        } else {
          tma_store_wait_all();                                     // this thread's stores of the passes before have landed
          tma_reduce_add_3d(&tm_s1, stg, 0, y, z);
          tma_reduce_add_3d(&tm_s1, stg + 16384u, 32, y, z);
          tma_reduce_add_3d(&tm_s2, stg + 32768u, 0, y, z);
          tma_reduce_add_3d(&tm_s2, stg + 49152u, 32, y, z);
        }
        tma_store_commit();
        if (e_last) *items_out = *items_out + 1;
      }
      store_pending = true;
      stg_ph = v & 1u;
      return true;
    };

    int n = 0;
    for (int w = item_at(0); w < p.walk && ok; w = item_at(++n)) {
      int blk, bh, set, it_begin, nsteps, d0, d_end;
      decode(w, blk, bh, set, it_begin, nsteps, d0, d_end);
      const int d_first = d0;
      for (; d0 < d_end && ok; d0 += kDkND, ++vi) {
        const int nd = d_end - d0 < kDkND ? d_end - d0 : kDkND;
        // the next pass's head and steps: its first two -LSE rows are written under this pass's tail
        int nx_bh = bh, nx_begin = it_begin, nx_total = nsteps;
        if (d0 + kDkND >= d_end) {
          const int wn = item_at(n + 1);
          nx_total = 0;
          if (wn < p.walk) { int b0, s0, x0, x1; decode(wn, b0, nx_bh, s0, nx_begin, nx_total, x0, x1); }
        }
        if (h == 0) {
          while (bias_written < jt + (uint32_t)(nsteps < 2 ? nsteps : 2)) {
            bias_put(bias_written, bias_fetch(bh, it_begin + (int)(bias_written - jt)));
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(b_bias + 8 * (bias_written % 3u));
            ++bias_written;
          }
        }
        const int key = blk * AT_BLK + r;                           // this thread's row of S^T
        for (int it = 0; it < nsteps && ok; ++it, ++jt) {
          const int step = it_begin + it;
          const uint32_t pb = jt & 1u, t_pb = t_s + 128u * pb + lane_off + 32u * (uint32_t)h, bsb = bs0 + pb * kDkBuf + row_off;
          // this step's correction terms of query step*128 + r: requested here, first used after the exponentials
          float draw_raw[kDkND], dref_raw;
          const bool q_in = step * AT_BLK + r < p.S;
          {
            const size_t qi = (size_t)bh * p.S + (q_in ? step * AT_BLK + r : 0);
            dref_raw = ldg(p.d_ref + qi);
#pragma unroll
            for (int d = 0; d < kDkND; ++d) draw_raw[d] = d < nd ? ldg(p.d_draws + (size_t)(d0 + d) * rows + qi) : 0.f;
          }
          // the -LSE row two steps ahead
          const int bt = it + 2;
          const bool bias_due = h == 0 && bias_written == jt + 2u && (bt < nsteps || bt - nsteps < nx_total);
          float bias_next = 0.f;
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(b_s_full + 8 * pb, (jt >> 1) & 1u, abort_flag));
          if (!ok) break;
          tc_fence_after();
          uint32_t sv[32];
          tmem_ld32_nowait(t_pb, sv);
          if (bias_due) bias_next = bt < nsteps ? bias_fetch(bh, it_begin + bt) : bias_fetch(nx_bh, nx_begin + (bt - nsteps));
          // the step's Q tile has landed (S^T read it); this thread still has to see its barrier before it reads it
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(b_sfull + 8 * (jt % kDkStages), (jt / kDkStages) & 1u, abort_flag));
          tmem_wait_ld();
          if (!ok) break;
          const int col0 = step * AT_BLK + h * 32;                  // first query of this thread's 32 columns
          const bool edge = (p.causal && blk == step) || (blk + 1) * AT_BLK > p.S || (step + 1) * AT_BLK > p.S;
          uint32_t pk[16];
          if (!edge) {
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              float a0, a1;
              mul_f32x2(a0, a1, __uint_as_float(sv[j]), __uint_as_float(sv[j + 1]), c2, c2);
              pk[j >> 1] = pack_bf16x2(ex2_approx(a0), ex2_approx(a1));
            }
          } else {
            // valid queries of this key: first <= column < end
            const int first = (p.causal ? key : 0) - col0, end = (key < p.S ? p.S : 0) - col0;
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              float a0, a1;
              mul_f32x2(a0, a1, __uint_as_float(sv[j]), __uint_as_float(sv[j + 1]), c2, c2);
              if (j < first || j >= end) a0 = -INFINITY;
              if (j + 1 < first || j + 1 >= end) a1 = -INFINITY;
              pk[j >> 1] = pack_bf16x2(ex2_approx(a0), ex2_approx(a1));
            }
          }
          tmem_st16(t_pb, pk);                                      // in place: the first 16 of the thread's own 32 columns
          if (store_pending) {                                      // an epilogue's staging has left this buffer
            if (warp == 0 && lane == 0) { tma_store_wait_read(); mbar_arrive(b_stg_free); }
            ok = __all_sync(0xFFFFFFFFu, mbar_wait(b_stg_free, stg_ph, abort_flag));
            if (!ok) break;
            store_pending = false;
          }
          // ---- the B operand: row r of the streamed Q tile times this row's factor of each draw, written at the same
          // (swizzled) place of the draw's tile.  Thread (r, h) takes the 16-byte chunks 2h and 2h + 1; chunk c of row r
          // sits at position c ^ (r & 7), so the lanes of a warp (consecutive rows) spread over all banks.  (The
          // buffer is free: S^T of this step was only formed after the product of two steps ago.)
          {
            uint32_t f2[kDkND];
            asm volatile("" : "+f"(dref_raw));                      // keeps the first use of the loads here
#pragma unroll
            for (int d = 0; d < kDkND; ++d) {
              asm volatile("" : "+f"(draw_raw[d]));
              const float fk = (q_in && d < nd) ? -p.c * (draw_raw[d] - dref_raw) : 0.f;
              f2[d] = pack_bf16x2(fk, fk);
            }
            const uint32_t qt = q0 + (jt % kDkStages) * kAtTile + row_off;
#pragma unroll
            for (int cch = 0; cch < 2; ++cch) {
              uint32_t a0, a1, a2, a3;
              const uint32_t off = (uint32_t)((2 * h + cch) ^ (r & 7)) << 4;
              asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(a0), "=r"(a1), "=r"(a2), "=r"(a3) : "r"(qt + off));
#pragma unroll
              for (int d = 0; d < kDkND; ++d)
                asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(bsb + (uint32_t)d * kAtTile + off),
                             "r"(mul_bf16x2(a0, f2[d])), "r"(mul_bf16x2(a1, f2[d])), "r"(mul_bf16x2(a2, f2[d])),
                             "r"(mul_bf16x2(a3, f2[d])) : "memory");
            }
          }
          if (bias_due) {
            asm volatile("" : "+f"(bias_next));
            bias_put(bias_written, bias_next);
          }
          tmem_wait_st();
          tc_fence_before();
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(b_op_ready + 8 * pb);
            if (bias_due) mbar_arrive(b_bias + 8 * (bias_written % 3u));
          }
          if (bias_due) ++bias_written;
          if (it == 0 && due) {
            ok = epilogue(vi - 1u, jt - 1u);
            due = false;
            if (!ok) break;
          }
        }
        e_blk = blk; e_bh = bh; e_set = set; e_first = d0 == d_first; e_last = d0 + kDkND >= d_end;
        due = true;
      }
    }
    if (ok && due) ok = epilogue(vi - 1u, jt - 1u);
    if (warp == 0 && lane == 0) tma_store_wait_all();
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag && p.diag) atomicMax(&p.diag->status, (int)BSP_ERR_TIMEOUT);
  for (int n = *items_out, w; (w = item_at(n)) < nwork; ++n) {      // none, unless a wait ran out
    int blk, bh, set, a, b, c, d;
    decode(w, blk, bh, set, a, b, c, d);
    attn_fill_nan(p.s1, p.s2, set * p.BH + bh, blk, p.S, kDkThreads);
  }
  if (warp == 17) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// S1[i, :] = -c PK[i, :] a[i], S2[i, :] = c^2 PK[i, :]^2 b[i] with a = sum_k (D_k - D*), b = sum_k (D_k - D*)^2
// (the rowwise sums of the correction term itself): the K draws of dQ in one elementwise pass.
__global__ void __launch_bounds__(256)
attn_dq_sums_kernel(const float* pk, const float* S1d, const float* S2d, float c,
                    float* S1q, float* S2q, size_t n4) {
  grid_dependency();
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  const size_t row = i / (AT_D / 4);
  const float4 v = ldg(reinterpret_cast<const float4*>(pk) + i);
  const float a = -c * ldg(S1d + row), b = c * c * ldg(S2d + row);
  reinterpret_cast<float4*>(S1q)[i] = make_float4(v.x * a, v.y * a, v.z * a, v.w * a);
  reinterpret_cast<float4*>(S2q)[i] = make_float4(v.x * v.x * b, v.y * v.y * b, v.z * v.z * b, v.w * v.w * b);
}

// S1 += times * (g - ref), S2 += times * (g - ref)^2, elementwise (times = 1: one draw).
__global__ void mc_accumulate_kernel(const float* g, const float* ref, float* S1,
                                     float* S2, size_t n4, float times) {
  grid_dependency();
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  const float4 a = ldg(reinterpret_cast<const float4*>(g) + i), r = ldg(reinterpret_cast<const float4*>(ref) + i);
  float4 s1 = reinterpret_cast<float4*>(S1)[i], s2 = reinterpret_cast<float4*>(S2)[i];
  const float d0 = a.x - r.x, d1 = a.y - r.y, d2 = a.z - r.z, d3 = a.w - r.w;
  s1.x = fmaf(times, d0, s1.x); s1.y = fmaf(times, d1, s1.y); s1.z = fmaf(times, d2, s1.z); s1.w = fmaf(times, d3, s1.w);
  s2.x = fmaf(times * d0, d0, s2.x); s2.y = fmaf(times * d1, d1, s2.y);
  s2.z = fmaf(times * d2, d2, s2.z); s2.w = fmaf(times * d3, d3, s2.w);
  reinterpret_cast<float4*>(S1)[i] = s1;
  reinterpret_cast<float4*>(S2)[i] = s2;
}

// The same over nd draws held back to back (g[d * stride + i]), in draw order: one launch instead of
// nd for a tensor as small as the correction term.  Any n (no vector accesses).
__global__ void mc_accumulate_draws_kernel(const float* g, size_t stride, int nd,
                                           const float* ref, float* S1,
                                           float* S2, size_t n) {
  grid_dependency();
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float r = ldg(ref + i);
  float s1 = S1[i], s2 = S2[i];
  for (int d = 0; d < nd; ++d) {
    const float e = ldg(g + (size_t)d * stride + i) - r;
    s1 += e;
    s2 = fmaf(e, e, s2);
  }
  S1[i] = s1;
  S2[i] = s2;
}

// The sums over the K draws of the dK difference; `partials` as in attn_f8_draws (two arrays of it).
static int attn_dk_diff(int BH, int S, int causal, float c, const void* q, const void* k, const float* lse,
                        const float* d_ref, const float* d_draws, int K, float* S1k, float* S2k, float* partials, int walk,
                        bsp_diag_t* diag, cudaStream_t st) {
  DkDiffParams p;
  p.BH = BH; p.S = S; p.nblk = (S + AT_BLK - 1) / AT_BLK; p.causal = causal ? 1 : 0; p.c = c;
  p.lse = lse; p.d_ref = d_ref; p.d_draws = d_draws; p.K = K; p.diag = diag;
  p.sets = partials ? attn_draw_sets(BH, S, K) : 1;
  p.passes = ((K + kDkND - 1) / kDkND + p.sets - 1) / p.sets;
  const size_t n = (size_t)BH * S * AT_D;
  float* o1 = p.sets > 1 ? partials : S1k;
  float* o2 = p.sets > 1 ? partials + (size_t)p.sets * n : S2k;
  CUtensorMap mq, mk, m1, m2;
  int rc;
  if ((rc = make_head_map(&mq, q, BH, S)) != BSP_OK) return rc;
  if ((rc = make_head_map(&mk, k, BH, S)) != BSP_OK) return rc;
  if ((rc = make_out_map(&m1, o1, BH * p.sets, S)) != BSP_OK) return rc;
  if ((rc = make_out_map(&m2, o2, BH * p.sets, S)) != BSP_OK) return rc;
  static std::atomic<bool> attr_set_dev[kMaxDevices];
  std::atomic<bool>& attr_set = attr_set_dev[device_slot()];
  if (!attr_set.load(std::memory_order_acquire)) {
    BSP_CHECK_CUDA(cudaFuncSetAttribute(attn_dk_diff_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDkSmem));
    attr_set.store(true, std::memory_order_release);
  }
  const int nsm = sm_count_or_default();
  const int64_t nwork = (int64_t)p.nblk * BH * p.sets;
  p.s1 = o1; p.s2 = o2;
  p.walk = walk < nwork ? walk : (int)nwork;
  launch_kernel(attn_dk_diff_kernel, (unsigned)(nwork < nsm ? nwork : nsm), kDkThreads, kDkSmem, st, mq, mk, m1, m2, p);
  BSP_LAUNCH_CHECK();
  return p.sets > 1 ? attn_sum_sets(o1, o2, p.sets, S1k, S2k, n, st) : BSP_OK;
}

struct AttnCheckBuffers {
  float *o, *lse, *amax, *scales, *d_ref, *d_pol, *d_draws;
  uint8_t* codes;
  float *g_ref[3], *g_pol[3], *S1[2], *S2[2], *S1d, *S2d;
  // FP8-operand mode: the rounded operands (decoded codes as bf16) and their per-slice scales
  void* op8[4];
  uint8_t* opc[4];                                // the operands' codes (FP8-operand mode)
  float *op_amax[4], *op_scale[4];
  float* partials;                                // sums of the sets of draws (where (block, head) items are few)
  void* ws_stats;
  size_t b_stats;
};

static size_t attn_carve(const bsp_attn_desc_t* op, int K, char* base, AttnCheckBuffers* out, bool room_for_sets = true) {
  size_t off = 0;
  auto take = [&](size_t bytes) -> void* {
    void* p = base ? base + off : nullptr;
    off += round_up(bytes ? bytes : 1, 256);
    return p;
  };
  const size_t BH = (size_t)op->B * op->H, rows = BH * op->S, n = rows * op->Dh;
  AttnCheckBuffers c;
  memset(&c, 0, sizeof(c));
  c.o = (float*)take(n * 4); c.lse = (float*)take(rows * 4);
  c.amax = (float*)take(BH * 4); c.scales = (float*)take(BH * 4);
  c.d_ref = (float*)take(rows * 4); c.d_pol = (float*)take(rows * 4);
  c.d_draws = (float*)take(rows * 4 * (size_t)(K > 0 ? K : 1));
  c.codes = (uint8_t*)take(n);
  for (int t = 0; t < 3; ++t) { c.g_ref[t] = (float*)take(n * 4); c.g_pol[t] = (float*)take(n * 4); }
  for (int t = 0; t < 2; ++t) { c.S1[t] = (float*)take(n * 4); c.S2[t] = (float*)take(n * 4); }
  c.S1d = (float*)take(rows * 4); c.S2d = (float*)take(rows * 4);
  if (op->fp8_operands) {
    for (int t = 0; t < 4; ++t) {
      c.op8[t] = take(n * 2); c.opc[t] = (uint8_t*)take(n); c.op_amax[t] = (float*)take(BH * 4); c.op_scale[t] = (float*)take(BH * 4);
    }
  }
  c.b_stats = kMaxPendingStats * kStatSlotBytes;
  c.ws_stats = take(c.b_stats);
  // last: a workspace without room for them is taken too, and then every item's draws stay in one set
  const size_t sets = room_for_sets ? (size_t)attn_draw_sets((int64_t)BH, op->S, K > 0 ? K : 1) : 1;
  if (sets > 1) c.partials = (float*)take((op->fp8_operands ? 4 : 2) * sets * n * 4);
  if (out) *out = c;
  return off;
}

}  // namespace bsp

using namespace bsp;

extern "C" {

int bsp_mc_accumulate(const float* g, const float* g_ref, float* S1, float* S2, size_t n, void* stream) {
  if (!g || !g_ref || !S1 || !S2) return BSP_ERR_ARG;
  if (n % 4 != 0) return BSP_ERR_UNSUPPORTED;
  if (!aligned16(g) || !aligned16(g_ref) || !aligned16(S1) || !aligned16(S2)) return BSP_ERR_ALIGN;
  if (n == 0) return BSP_OK;
  const size_t n4 = n / 4;
  launch_kernel(mc_accumulate_kernel, (unsigned)((n4 + 255) / 256), 256, 0, (cudaStream_t)stream, g, g_ref, S1, S2, n4, 1.0f);
  BSP_LAUNCH_CHECK();
  return BSP_OK;
}

size_t bsp_mc_check_attn_workspace_bytes(const bsp_attn_desc_t* op, int K) {
  if (!op || op->B <= 0 || op->H <= 0 || op->S <= 0 || op->Dh <= 0) return 0;
  return attn_carve(op, K, nullptr, nullptr);
}

#define BSP_TRY(expr)              \
  do {                             \
    int _rc = (expr);              \
    if (_rc != BSP_OK) return _rc; \
  } while (0)

static int attn_check(const bsp_attn_desc_t* op, int K, const bsp_verdict_rule_t* rule, bsp_use_result_t* results,
                      int* n_results, void* ws, size_t ws_bytes, int walk, bsp_diag_t* diag, void* stream) {
  if (!op || !results || !n_results || K < 4 || !rule_valid(rule)) return BSP_ERR_ARG;
  if (!op->q || !op->k || !op->v || !op->dO) return BSP_ERR_ARG;
  int rc = check_attn_shape(op->B, op->H, op->S, op->Dh, op->dtype);
  if (rc != BSP_OK) return rc;
  const bool fp8 = op->fp8_operands != 0;
  if (fp8 && (!(op->p_scale > 0.f) || !(op->ds_scale > 0.f))) return BSP_ERR_ARG;
  const bool room_for_sets = ws_bytes >= bsp_mc_check_attn_workspace_bytes(op, K);
  if (!ws || ws_bytes < attn_carve(op, K, nullptr, nullptr, false) || (reinterpret_cast<uintptr_t>(ws) & 255u))
    return BSP_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  AttnCheckBuffers b;
  attn_carve(op, K, reinterpret_cast<char*>(ws), &b, room_for_sets);
  const int B = op->B, H = op->H, S = op->S, Dh = op->Dh, dt = op->dtype;
  const size_t BH = (size_t)B * H, rows = BH * S, n = rows * Dh;
  const float c = op->softmax_scale;
  *n_results = 0;

  // ---- FP8-operand mode: the operands as the emulated backward sees them
  const void *q = op->q, *k = op->k, *v = op->v, *dO = op->dO;
  bsp_attn_fp8_t f8;
  const bsp_attn_fp8_t* f = nullptr;
  if (fp8) {
    const void* src[4] = {op->q, op->k, op->v, op->dO};
    for (int t = 0; t < 4; ++t)
      BSP_TRY(bsp_attn_quantize(src[t], (int)BH, (size_t)S * Dh, t == 3 ? BSP_E5M2 : BSP_E4M3, b.op8[t], b.opc[t],
                                b.op_amax[t], b.op_scale[t], diag, st));
    q = b.op8[0]; k = b.op8[1]; v = b.op8[2]; dO = b.op8[3];
    f8.q_scale = b.op_scale[0]; f8.k_scale = b.op_scale[1]; f8.v_scale = b.op_scale[2]; f8.do_scale = b.op_scale[3];
    f8.p_scale = op->p_scale; f8.ds_scale = op->ds_scale;
    f8.q_codes = b.opc[0]; f8.k_codes = b.opc[1]; f8.v_codes = b.opc[2]; f8.do_codes = b.opc[3];
    f = &f8;
  }
  const float* do_scales = fp8 ? f8.do_scale : nullptr;

  // ---- once: forward output and LSE, the output store (per-(b,h) amax scale, stream 0)
  BSP_TRY(attn_fwd_impl(B, H, S, Dh, op->causal, c, q, k, v, dt, f, b.o, b.lse, diag, st));
  BSP_TRY(bsp_amax(b.o, BSP_F32, BH, (size_t)S * Dh, b.amax, diag, st));
  BSP_TRY(bsp_scale_from_amax(b.amax, BH, op->store_fmt, b.scales, st));
  bsp_key_t key;
  key.seed = op->seed; key.tensor_id = op->tensor_id; key.stream = BSP_STREAM_FORWARD; key.draw = 0; key.reserved = 0;
  BSP_TRY(bsp_round_grouped(b.o, BSP_F32, BH, (size_t)S * Dh, op->store_fmt, op->forward_mode, b.scales, key, b.codes,
                            diag, st));
  key.stream = BSP_STREAM_ATTN_D;

  // ---- reference: D reads the original output
  BSP_TRY(attn_dterm_impl(B, H, S, Dh, dO, dt, do_scales, b.o, b.codes, b.scales, op->store_fmt, BSP_READ_ORIGINAL,
                          key, 0, 1, b.d_ref, st));
  BSP_TRY(attn_bwd_dterm_impl(B, H, S, Dh, op->causal, c, q, k, v, dO, dt, f, b.lse, b.d_ref, b.g_ref[0], b.g_ref[1],
                              b.g_ref[2], diag, st));
  // the statistics passes are read behind one synchronisation at the end
  PendingStats pend;
  pend.slots = reinterpret_cast<double*>(b.ws_stats);
  pend.st = st;
  pend.rule = rule;
  int nres = 0;
  const int out_ids[4] = {BSP_OUT_D, BSP_OUT_DQ, BSP_OUT_DK, BSP_OUT_DV};
  auto emit = [&](int out, int pol) -> bsp_use_result_t* {
    bsp_use_result_t* r = &results[nres++];
    memset(r, 0, sizeof(*r));
    r->use_id = BSP_STREAM_ATTN_D; r->output_id = out; r->policy = pol;
    // FP8 operands: dQ and dK pass through the nearest rounding of dS, which is not linear in D
    r->informational = (fp8 && pol == BSP_READ_FRESH && (out == BSP_OUT_DQ || out == BSP_OUT_DK)) ? 1 : 0;
    return r;
  };
  for (int pol = 0; pol < 2; ++pol) {
    if (!((op->policy_mask >> pol) & 1u)) continue;
    const float* dsrc = b.d_ref;
    float* const* gsrc = b.g_ref;
    if (pol == BSP_READ_FORWARD) {
      BSP_TRY(attn_dterm_impl(B, H, S, Dh, dO, dt, do_scales, b.o, b.codes, b.scales, op->store_fmt, BSP_READ_FORWARD,
                              key, 0, 1, b.d_pol, st));
      BSP_TRY(attn_bwd_dterm_impl(B, H, S, Dh, op->causal, c, q, k, v, dO, dt, f, b.lse, b.d_pol, b.g_pol[0],
                                  b.g_pol[1], b.g_pol[2], diag, st));
      dsrc = b.d_pol;
      gsrc = b.g_pol;
    }
    BSP_TRY(pend.add(b.d_ref, dsrc, nullptr, (int64_t)rows, 1, 0, emit(out_ids[0], pol)));
    for (int t = 0; t < 3; ++t)
      BSP_TRY(pend.add(b.g_ref[t], gsrc[t], nullptr, (int64_t)n, 1, 0, emit(out_ids[t + 1], pol)));
  }
  if ((op->policy_mask >> 2) & 1u) {
    // fresh read: all K correction terms in one pass, and the sums of D itself in one launch
    BSP_TRY(attn_dterm_impl(B, H, S, Dh, dO, dt, do_scales, b.o, b.codes, b.scales, op->store_fmt, BSP_READ_FRESH, key,
                            0, K, b.d_draws, st));
    BSP_CHECK_CUDA(cudaMemsetAsync(b.S1d, 0, rows * 4, st));
    BSP_CHECK_CUDA(cudaMemsetAsync(b.S2d, 0, rows * 4, st));
    launch_kernel(mc_accumulate_draws_kernel, (unsigned)((rows + 255) / 256), 256, 0, st, b.d_draws, rows, K, b.d_ref, b.S1d, b.S2d,
                  rows);
    BSP_LAUNCH_CHECK();
    if (!fp8) {
      // dQ: P K once (the forward kernel with K in place of V and the rows' LSE given, so it takes one
      // pass over the keys; g_pol[0] is free by now), then the K draws collapse to one elementwise pass
      BSP_TRY(attn_fwd_impl(B, H, S, Dh, op->causal, c, q, k, k, dt, nullptr, b.g_pol[0], nullptr, diag, st, b.lse));
      launch_kernel(attn_dq_sums_kernel, (unsigned)((n / 4 + 255) / 256), 256, 0, st, b.g_pol[0], b.S1d, b.S2d, c, b.S1[0], b.S2[0],
                    n / 4);
      BSP_LAUNCH_CHECK();
      // dK: all draws in one launch
      BSP_TRY(attn_dk_diff((int)BH, S, op->causal, c, q, k, b.lse, b.d_ref, b.d_draws, K, b.S1[1], b.S2[1], b.partials, walk, diag, st));
    } else {
      // the rounded backward of every draw; dQ and dK go from the accumulators straight into their sums
      BSP_TRY(attn_f8_draws((int)BH, S, op->causal, c, f, b.lse, b.d_draws, K, b.g_ref[0], b.S1[0], b.S2[0], b.g_ref[1], b.S1[1],
                            b.S2[1], b.partials, walk, diag, st));
    }
    BSP_TRY(pend.add(b.d_ref, b.S1d, b.S2d, (int64_t)rows, K, 1, emit(out_ids[0], BSP_READ_FRESH)));
    for (int t = 0; t < 2; ++t)
      BSP_TRY(pend.add(b.g_ref[t], b.S1[t], b.S2[t], (int64_t)n, K, 1, emit(out_ids[t + 1], BSP_READ_FRESH)));
    // dV does not read the correction term: every draw is the reference itself
    pend.add_exact_fresh((int64_t)n, K, emit(out_ids[3], BSP_READ_FRESH));
  }
  *n_results = nres;
  return pend.flush();
}

int bsp_mc_check_attn(const bsp_attn_desc_t* op, int K, const bsp_verdict_rule_t* rule, bsp_use_result_t* results,
                      int* n_results, void* ws, size_t ws_bytes, bsp_diag_t* diag, void* stream) {
  return attn_check(op, K, rule, results, n_results, ws, ws_bytes, INT_MAX, diag, stream);
}

int bsp_selftest_attn_unfinished(const bsp_attn_desc_t* op, int K, int done, bsp_use_result_t* results, int* n_results,
                                 void* ws, size_t ws_bytes, bsp_diag_t* diag, void* stream) {
  if (done < 0) return BSP_ERR_ARG;
  return attn_check(op, K, nullptr, results, n_results, ws, ws_bytes, done, diag, stream);
}

}  // extern "C"
