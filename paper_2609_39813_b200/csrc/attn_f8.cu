// The attention backward of the FP8-operand mode: one evaluation (attn_f8_bwd), and the K draws of a
// fresh read of the correction term with the running sums of the Monte-Carlo check (attn_f8_draws).
//
//   P = exp(c Q K^T - LSE), dP = dO V^T;  dS_k = E5M2(P (dP - D_k) ds_scale) for the correction terms
//   D_k of the draws;  dQ_k = c dS_k K, dK_k = c dS_k^T Q;  dV = E4M3(P p_scale)^T dO.
//
// The scores, dP and the exponentials do not depend on the draw, so a step forms them once for up to
// four draws.  What limits the number of draws is tensor memory: S and dP take 128 columns each, an
// accumulator 64; the operands dS_k therefore go through shared memory (16 KB of codes per draw and
// step) and the four accumulators fill the other 256 columns.  A thread owns a query row
// in both kernels, so LSE and the D_k are scalars of the thread: the dQ kernel reads the codes K-major
// (rows = queries), the dK / dV kernel reads the same layout MN-major (rows = the contraction).
//
// Little that the softmax warps wait for is on their own path: S and dP of the next step are issued as soon as
// they hold this step's in registers; a step's products run under the exponentials of the next, so one buffer
// of operands is enough; an item's accumulators are read after the next item's first step.  The running sums of
// an item stay in shared memory, in the place of a second buffer, from its first pass to its last, and leave
// in one store.  (Bulk reduce-adds per pass instead: 64 KB each, 3000 cycles of every pass spent waiting for
// their staging to be read.)
//
// Measured at B H = 128, S = 2048, causal, 32 draws: both kernels 4.35 ms (a launch per pair of draws, with the
// operands in tensor memory and eight softmax warps, 8.2; two operand buffers and reduce-adds 4.5), the whole
// check 9.54 -> 6.08 ms.  Of a step's 4600 cycles the conversions take 1700 and the exponentials 1200, one after the
// other in all warps (a start half a step apart does not last: a step's products need every warp's codes); 450
// are a pass's end, the rest waits for barriers and tensor memory.
//
// Persistent CTA, one per SM, walking (block, head, set of draws) items, heaviest first.  A CTA takes the
// draws of its set four at a time and adds to the sums in that order; where there are at most half as many
// (block, head) items as SMs the draws are spread over several sets, each with sums of its own, which sum_sets_kernel
// adds in order, so the sums stay reproducible.  640 threads: warps 0..15 softmax and epilogue, warp 16
// TMA, warp 17 MMA issue.  Every wait is bounded (the warps meet on mbarriers, never on a block barrier).
#include <string.h>

#include <atomic>

#include "attn_common.cuh"

namespace bsp {

constexpr int kF8Threads = 640;
constexpr int kF8Warps = 16;                       // softmax warps
constexpr int kF8ND = kDrawsPerPass;               // draws per pass over the steps
constexpr uint32_t kF8Stages = 3;                  // ring of streamed tile pairs
constexpr uint32_t kF8Tile = AT_BLK * AT_D;        // 8 KB: 128 rows of 64 codes
constexpr uint32_t kF8Op = AT_BLK * AT_BLK;        // 16 KB: one operand, 128 x 128 codes
constexpr uint32_t kF8Buf = kF8ND * kF8Op;         // the step's operands
constexpr uint32_t kF8Out = AT_BLK * AT_D * 4;     // 32 KB: an FP32 output tile, as two boxes of 32 columns
// operands [4], two output tiles (the running sums), resident tiles [2][2], ring [3][2], barriers
constexpr int kF8Smem = 1024 + kF8Buf + 2 * kF8Out + 4 * kF8Tile + kF8Stages * 2 * kF8Tile + 512;
static_assert(kF8Smem <= 232448, "dynamic shared memory of attn_f8_kernel exceeds the SM's");

// Two pairs of floats to four FP8 codes in one word (nearest, saturating).
template <int FMT>
__device__ __forceinline__ uint32_t f8_encode4(uint64_t ab, uint64_t cd) {
  uint32_t r;
  float a, b, c, d;
  f2_unpack(ab, a, b);
  f2_unpack(cd, c, d);
  if (FMT == BSP_E4M3)
    asm("{\n\t.reg .b16 lo, hi;\n\tcvt.rn.satfinite.e4m3x2.f32 lo, %2, %1;\n\tcvt.rn.satfinite.e4m3x2.f32 hi, %4, %3;\n\t"
        "mov.b32 %0, {lo, hi};\n\t}" : "=r"(r) : "f"(a), "f"(b), "f"(c), "f"(d));
  else
    asm("{\n\t.reg .b16 lo, hi;\n\tcvt.rn.satfinite.e5m2x2.f32 lo, %2, %1;\n\tcvt.rn.satfinite.e5m2x2.f32 hi, %4, %3;\n\t"
        "mov.b32 %0, {lo, hi};\n\t}" : "=r"(r) : "f"(a), "f"(b), "f"(c), "f"(d));
  return r;
}

struct AttnF8Params {
  int BH, S, nblk, causal;
  float c;
  const float* lse;              // [BH*S]
  const float* dterm;            // [K][BH*S] correction terms of the draws (one for a plain evaluation)
  int K, sets, passes;           // draws; sets per (block, head); passes of up to four draws per set
  const float* mc_ref;           // [BH*S*64]: the sums are of g_k - mc_ref (draws only)
  const float *sc_q, *sc_k, *sc_v, *sc_do;         // [BH]
  float p_scale, ds_scale;
  bsp_diag_t* diag;
};
struct AttnF8Draws : AttnF8Params {
  float *s1, *s2;                // what tm_o0 and tm_o1 map
  int walk;                      // items from here on are left as after a wait that ran out (self-test; else all)
};
template <bool MC> struct AttnF8Arg { using type = AttnF8Params; };
template <> struct AttnF8Arg<true> { using type = AttnF8Draws; };

// MODE: AT_DQ (the CTA owns a query block, streams K_j, V_j) or AT_DKV (owns a key block, streams Q_i, dO_i).
// MC: the draws with their sums S1 (tm_o0), S2 (tm_o1); else one evaluation: dQ (tm_o0), or dK (tm_o1) and,
// with DV, dV (tm_o0).
template <int MODE, bool MC, bool DV>
__global__ void __launch_bounds__(kF8Threads, 1)
attn_f8_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
               const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_do,
               const __grid_constant__ CUtensorMap tm_o0, const __grid_constant__ CUtensorMap tm_o1,
               typename AttnF8Arg<MC>::type p) {
  static_assert(!DV || (MODE == AT_DKV && !MC), "dV: one evaluation of the dK / dV kernel");
  grid_dependency();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  const uint32_t op0 = base, out0 = op0 + kF8Buf;                   // operand o: op0 + o * kF8Op
  const uint32_t res_base = out0 + 2 * kF8Out;                      // resident pair rb: res_base + rb * 2 * kF8Tile
  const uint32_t str0 = res_base + 4 * kF8Tile;                     // stage s: str0 + s * 2 * kF8Tile
  const uint32_t bars = str0 + kF8Stages * 2 * kF8Tile;
  const uint32_t b_res = bars, b_res_empty = bars + 16, b_sfull = bars + 32, b_sempty = bars + 56, b_sdp_full = bars + 80,
                 b_sdp_free = bars + 88, b_op_ready = bars + 96, b_op_free = bars + 112, b_acc = bars + 128,
                 b_acc_free = bars + 136, b_staged = bars + 144, b_stg_free = bars + 152;
  uint8_t* bars_gen = smem_raw + (bars - raw);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bars_gen + 176);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars_gen + 180);
  volatile int* items_out = abort_flag + 1;                         // items whose outputs have been sent off

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nwork = p.nblk * p.BH * p.sets;
  int nwalk = nwork;
  if constexpr (MC) nwalk = p.walk;
  // the CTA's n-th item: rounds of gridDim.x items, walked forwards and backwards in turn
  auto item_at = [&](int n) -> int {
    const int b = (int)blockIdx.x, G = (int)gridDim.x;
    return n * G + ((n & 1) ? G - 1 - b : b);
  };
  // draws [d_begin, d_end) of the item, in passes of up to kF8ND
  auto decode = [&](int w, int& blk, int& bh, int& set, int& it_begin, int& nsteps, int& d_begin, int& d_end) {
    set = w % p.sets;
    const int i = w / p.sets;
    const int rank = i / p.BH;
    bh = i % p.BH;
    if (MODE == AT_DKV) {
      blk = rank;                                                   // key block j: query blocks i = j .. nblk-1 (causal)
      it_begin = p.causal ? blk : 0;
      nsteps = p.nblk - it_begin;
    } else {
      blk = p.nblk - 1 - rank;                                      // query block i: key blocks j = 0 .. i (causal)
      it_begin = 0;
      nsteps = p.causal ? blk + 1 : p.nblk;
    }
    d_begin = set * p.passes * kF8ND;
    d_end = d_begin + p.passes * kF8ND < p.K ? d_begin + p.passes * kF8ND : p.K;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(b_res + 8 * s, 1); mbar_init(b_res_empty + 8 * s, 1);
    }
    mbar_init(b_op_ready, kF8Warps); mbar_init(b_op_free, 1);
    for (uint32_t s = 0; s < kF8Stages; ++s) { mbar_init(b_sfull + 8 * s, 1); mbar_init(b_sempty + 8 * s, 1); }
    mbar_init(b_sdp_full, 1); mbar_init(b_sdp_free, kF8Warps);
    mbar_init(b_acc, 1); mbar_init(b_acc_free, kF8Warps);
    mbar_init(b_staged, kF8Warps); mbar_init(b_stg_free, 1);
    *abort_flag = 0;
    if (MC) *items_out = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 17) tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t t_s = tmem, t_dp = tmem + 128, t_acc = tmem + 256;  // the accumulator of operand o at t_acc + 64 o

  // operand formats (E4M3 = 0, E5M2 = 1): S from Q and K, dP from dO (E5M2) and V, rows = queries
  const uint32_t id_s = make_idesc(0u, 0u, 128, 128), id_dp = make_idesc(1u, 0u, 128, 128);
  // dS (E5M2) x K or Q (E4M3, MN-major); P (E4M3) x dO (E5M2, MN-major).  dK / dV: A MN-major too
  const uint32_t id_ds = make_idesc(1u, 0u, 128, 64) | (1u << 16) | (MODE == AT_DKV ? 1u << 15 : 0u);
  const uint32_t id_p = make_idesc(0u, 1u, 128, 64) | (1u << 16) | (1u << 15);

  // the block starts with 640 x 96 registers: the control warpgroup keeps 32 a thread, the others take 112
  if (warp >= kF8Warps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
    if (warp == 16) {
      // ------------------------------------------------ TMA producer
      if (lane == 0) {
        tma_prefetch_desc(&tm_q); tma_prefetch_desc(&tm_k); tma_prefetch_desc(&tm_v); tma_prefetch_desc(&tm_do);
        bool ok = true;
        uint32_t itg = 0, vi = 0;                                   // global step, pass
        int n = 0;
        for (int w = item_at(0); w < nwalk && ok; w = item_at(++n)) {
          int blk, bh, set, it_begin, nsteps, d0, d_end;
          decode(w, blk, bh, set, it_begin, nsteps, d0, d_end);
          for (; d0 < d_end && ok; d0 += kF8ND, ++vi) {
            const uint32_t rb = vi & 1u;
            if (!mbar_wait(b_res_empty + 8 * rb, ((vi >> 1) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
            const uint32_t r0 = res_base + rb * 2 * kF8Tile, r1 = r0 + kF8Tile;
            mbar_expect_tx(b_res + 8 * rb, 2 * kF8Tile);
            tma_load_3d(r0, MODE == AT_DKV ? &tm_k : &tm_q, b_res + 8 * rb, 0, blk * AT_BLK, bh);
            tma_load_3d(r1, MODE == AT_DKV ? &tm_v : &tm_do, b_res + 8 * rb, 0, blk * AT_BLK, bh);
            for (int it = 0; it < nsteps; ++it, ++itg) {
              const uint32_t s = itg % kF8Stages, ph = (itg / kF8Stages) & 1u;
              if (!mbar_wait(b_sempty + 8 * s, ph ^ 1u, abort_flag)) { ok = false; break; }
              const uint32_t s0 = str0 + s * 2 * kF8Tile, s1 = s0 + kF8Tile;
              mbar_expect_tx(b_sfull + 8 * s, 2 * kF8Tile);
              tma_load_3d(s0, MODE == AT_DKV ? &tm_q : &tm_k, b_sfull + 8 * s, 0, (it_begin + it) * AT_BLK, bh);
              tma_load_3d(s1, MODE == AT_DKV ? &tm_do : &tm_v, b_sfull + 8 * s, 0, (it_begin + it) * AT_BLK, bh);
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
      for (int w = item_at(0); w < nwalk && ok; w = item_at(++n)) {
        int blk, bh, set, it_begin, nsteps, d0, d_end;
        decode(w, blk, bh, set, it_begin, nsteps, d0, d_end);
        for (; d0 < d_end && ok; d0 += kF8ND, ++vi) {
          const uint32_t rb = vi & 1u;
          const uint32_t res0 = res_base + rb * 2 * kF8Tile, res1 = res0 + kF8Tile;
          const int nd = d_end - d0 < kF8ND ? d_end - d0 : kF8ND;
          if (!wait_all(b_res + 8 * rb, (vi >> 1) & 1u)) { ok = false; break; }
          // S = Q K^T and dP = dO V^T of global step jt, 64 = 2 x 32 along K; issued one step ahead
          auto issue_sdp = [&](uint32_t jt) -> bool {
            const uint32_t s = jt % kF8Stages;
            if (!wait_all(b_sfull + 8 * s, (jt / kF8Stages) & 1u)) return false;
            if (!wait_all(b_sdp_free, (jt & 1u) ^ 1u)) return false;
            tc_fence_after();
            const uint32_t st0 = str0 + s * 2 * kF8Tile, st1 = st0 + kF8Tile;
            const uint64_t q = make_smem_desc_sw64(MODE == AT_DKV ? st0 : res0), k = make_smem_desc_sw64(MODE == AT_DKV ? res0 : st0);
            const uint64_t g = make_smem_desc_sw64(MODE == AT_DKV ? st1 : res1), v = make_smem_desc_sw64(MODE == AT_DKV ? res1 : st1);
#pragma unroll
            for (int i = 0; i < 2; ++i) tc_mma_l<true>(leader, t_s, q + 2u * i, k + 2u * i, id_s, i != 0);
#pragma unroll
            for (int i = 0; i < 2; ++i) tc_mma_l<true>(leader, t_dp, g + 2u * i, v + 2u * i, id_dp, i != 0);
            tc_commit_l(leader, b_sdp_full);
            return true;
          };
          ok = issue_sdp(itg);
          for (int it = 0; it < nsteps && ok; ++it) {
            const uint32_t jg = itg + (uint32_t)it, s = jg % kF8Stages;
            if (it + 1 < nsteps && !issue_sdp(jg + 1)) { ok = false; break; }
            if (!wait_all(b_op_ready, jg & 1u)) { ok = false; break; }
            // the accumulators are free once the epilogue of the pass before has read them
            if (it == 0 && !wait_all(b_acc_free, (vi & 1u) ^ 1u)) { ok = false; break; }
            tc_fence_after();
            const uint32_t st0 = str0 + s * 2 * kF8Tile;
            const uint64_t bs = make_smem_desc_mn_sw64(st0), bdo = make_smem_desc_mn_sw64(st0 + kF8Tile);
            const uint32_t acc = it == 0 ? 0u : 1u;
            // 128 = 4 x 32 along the contraction: 32 bytes of a row (K-major A) or 32 rows (MN-major A) per step
            auto products = [&](uint32_t o, uint64_t b, uint32_t id) {
              const uint32_t op = op0 + o * kF8Op;
              const uint64_t a = MODE == AT_DKV ? make_smem_desc_mn(op, 16384u) : make_smem_desc(op);
#pragma unroll
              for (uint32_t i = 0; i < 4; ++i)
                tc_mma_l<true>(leader, t_acc + 64u * o, a + (MODE == AT_DKV ? 256u : 2u) * i, b + 128u * i, id, i != 0 ? 1u : acc);
            };
            if (MC) {
              for (int d = 0; d < nd; ++d) products((uint32_t)d, bs, id_ds);
            } else {
              products(0u, bs, id_ds);
              if (DV) products(1u, bdo, id_p);
            }
            tc_commit_l(leader, b_op_free);
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
    // ------------------------------------------------ softmax warps: P, the draws' dS codes, the epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    const int q4 = warp & 3, h = warp >> 2;                         // lane quarter; 32 of the 128 columns
    const int r = q4 * 32 + lane;                                   // this thread's query row of the score tile
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    const size_t rows = (size_t)p.BH * p.S;
    const uint32_t row_off = (uint32_t)r * 128u;
    const uint32_t ch0 = (uint32_t)((2 * h) ^ (r & 7)) << 4, ch1 = (uint32_t)((2 * h + 1) ^ (r & 7)) << 4;
    bool ok = true;
    uint32_t jt = 0, vi = 0, stored = 0;                            // global step, pass; items whose outputs have been sent off
    // the pass whose accumulators have not been read yet
    bool due = false;
    int e_blk = 0, e_bh = 0, e_set = 0, e_nd = 0;
    bool e_first = true, e_last = true;
    // Reads the accumulators of pass `v` into the item's output tiles; after its last pass the tiles leave.
    auto epilogue = [&](uint32_t v) -> bool {
      const int orow = e_blk * AT_BLK + r;                          // a key (dK / dV) or a query
      float ref[MC ? 16 : 1];
      if (MC) {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
          if (orow < p.S) f = ldg(reinterpret_cast<const float4*>(p.mc_ref + ((size_t)e_bh * p.S + orow) * AT_D + h * 16) + t);
          ref[MC ? 4 * t : 0] = f.x; ref[MC ? 4 * t + 1 : 0] = f.y; ref[MC ? 4 * t + 2 : 0] = f.z; ref[MC ? 4 * t + 3 : 0] = f.w;
        }
      }
      const float inv_q = __fdiv_rn(1.0f, ldg(p.sc_q + e_bh)), inv_k = __fdiv_rn(1.0f, ldg(p.sc_k + e_bh));
      const float mul = p.c * ((MODE == AT_DKV ? inv_q : inv_k) / p.ds_scale);
      if (e_first && stored) {                                      // the stores of the item before have read the tiles
        if (warp == 0 && lane == 0) { tma_store_wait_read(); mbar_arrive(b_stg_free); }
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(b_stg_free, (stored - 1u) & 1u, abort_flag))) return false;
      }
      if (!__all_sync(0xFFFFFFFFu, mbar_wait(b_acc, v & 1u, abort_flag))) return false;
      tc_fence_after();
      // box h >> 1 of 32 columns, four 16-byte chunks of this thread's half of it
      const uint32_t box = out0 + (uint32_t)(h >> 1) * 16384u + row_off;
      auto chunk = [&](int t) -> uint32_t { return box + ((uint32_t)(((h & 1) * 4 + t) ^ (r & 7)) << 4); };
      auto put4 = [&](uint32_t at, float a, float b, float c, float d) {
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
      };
      if (MC) {
        float s1[16], s2[16];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          if (e_first) {
#pragma unroll
            for (int e = 4 * t; e < 4 * t + 4; ++e) s1[e] = s2[e] = 0.f;
          } else {
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(s1[4 * t]), "=f"(s1[4 * t + 1]), "=f"(s1[4 * t + 2]), "=f"(s1[4 * t + 3]) : "r"(chunk(t)));
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(s2[4 * t]), "=f"(s2[4 * t + 1]), "=f"(s2[4 * t + 2]), "=f"(s2[4 * t + 3]) : "r"(chunk(t) + kF8Out));
          }
        }
        for (int d = 0; d < e_nd; ++d) {
          uint32_t a[16];
          tmem_ld16(t_acc + 64u * (uint32_t)d + lane_off + h * 16, a);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const float g = __fmul_rn(__uint_as_float(a[e]), mul) - ref[MC ? e : 0];   // zero where the draw is the reference
            s1[e] += g;
            s2[e] = fmaf(g, g, s2[e]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(b_acc_free);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          put4(chunk(t), s1[4 * t], s1[4 * t + 1], s1[4 * t + 2], s1[4 * t + 3]);
          put4(chunk(t) + kF8Out, s2[4 * t], s2[4 * t + 1], s2[4 * t + 2], s2[4 * t + 3]);
        }
        if (!e_last) return true;
      } else {
        const float mul_v = DV ? __fdiv_rn(1.0f, ldg(p.sc_do + e_bh)) / p.p_scale : 0.f;
#pragma unroll
        for (int o = 0; o < (DV ? 2 : 1); ++o) {                    // operand 0: dS (dQ or dK), operand 1: P (dV)
          uint32_t a[16];
          tmem_ld16(t_acc + 64u * (uint32_t)o + lane_off + h * 16, a);
          tmem_wait_ld();
          const float m = o == 0 ? mul : mul_v;
#pragma unroll
          for (int t = 0; t < 4; ++t)
            put4(chunk(t) + kF8Out * o, __uint_as_float(a[4 * t]) * m, __uint_as_float(a[4 * t + 1]) * m,
                 __uint_as_float(a[4 * t + 2]) * m, __uint_as_float(a[4 * t + 3]) * m);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(b_acc_free);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(b_staged);
      if (warp == 0) {
        if (!__all_sync(0xFFFFFFFFu, mbar_wait(b_staged, stored & 1u, abort_flag))) return false;
        if (lane == 0) {
          // MC: S1, S2; else dQ, or dK and dV
          const CUtensorMap* m0 = !MC && MODE == AT_DKV ? &tm_o1 : &tm_o0;
          const CUtensorMap* m1 = !MC && MODE == AT_DKV ? &tm_o0 : &tm_o1;
          const int y = e_blk * AT_BLK, z = e_set * p.BH + e_bh;
          tma_store_3d(m0, out0, 0, y, z);
          tma_store_3d(m0, out0 + 16384u, 32, y, z);
          if (MC || DV) {
            tma_store_3d(m1, out0 + kF8Out, 0, y, z);
            tma_store_3d(m1, out0 + kF8Out + 16384u, 32, y, z);
          }
          tma_store_commit();
          if (MC) *items_out = (int)stored + 1;
        }
      }
      ++stored;
      return true;
    };

    int n = 0;
    for (int w = item_at(0); w < nwalk && ok; w = item_at(++n)) {
      int blk, bh, set, it_begin, nsteps, d0, d_end;
      decode(w, blk, bh, set, it_begin, nsteps, d0, d_end);
      const int d_first = d0;
      const float inv_q = __fdiv_rn(1.0f, ldg(p.sc_q + bh)), inv_k = __fdiv_rn(1.0f, ldg(p.sc_k + bh));
      const float inv_v = __fdiv_rn(1.0f, ldg(p.sc_v + bh)), inv_do = __fdiv_rn(1.0f, ldg(p.sc_do + bh));
      const float c2 = p.c * kLog2e * inv_q * inv_k, dp_mul = inv_do * inv_v;   // scores and dP arrive as products of codes
      const uint64_t c2_2 = f2_pack(c2, c2), dp_mul_2 = f2_pack(dp_mul, dp_mul);
      const uint64_t ds_2 = f2_pack(p.ds_scale, p.ds_scale), ps_2 = f2_pack(p.p_scale, p.p_scale);
      for (; d0 < d_end && ok; d0 += kF8ND, ++vi) {
        const int nd = MC ? (d_end - d0 < kF8ND ? d_end - d0 : kF8ND) : 1;
        // LSE and the draws' correction terms of the thread's query: of the item (dQ), or of the step (dK / dV,
        // read a step ahead)
        float lse_q, dd[kF8ND];
        auto fetch = [&](int qblk) {
          const int qy = qblk * AT_BLK + r;
          const size_t i = (size_t)bh * p.S + (qy < p.S ? qy : 0);
          lse_q = qy < p.S ? ldg(p.lse + i) : 0.f;
#pragma unroll
          for (int d = 0; d < kF8ND; ++d) dd[d] = (MC ? d < nd : d == 0) && qy < p.S ? ldg(p.dterm + (size_t)(d0 + d) * rows + i) : 0.f;
        };
        fetch(MODE == AT_DKV ? it_begin : blk);
        for (int it = 0; it < nsteps && ok; ++it, ++jt) {
          const int step = it_begin + it;
          const int qblk = MODE == AT_DKV ? step : blk, kblk = MODE == AT_DKV ? blk : step;
          const uint64_t nlse_2 = f2_pack(-lse_q * kLog2e, -lse_q * kLog2e);
          uint64_t ndk_2[kF8ND];
#pragma unroll
          for (int d = 0; d < kF8ND; ++d) ndk_2[d] = f2_pack(-dd[d], -dd[d]);
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(b_sdp_full, jt & 1u, abort_flag));
          if (!ok) break;
          tc_fence_after();
          uint32_t sv[32], dv[32];
          tmem_ld32_nowait(t_s + lane_off + h * 32, sv);
          tmem_ld32_nowait(t_dp + lane_off + h * 32, dv);
          tmem_wait_ld();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(b_sdp_free);
          if (MODE == AT_DKV && it + 1 < nsteps) fetch(step + 1);
          // the probabilities, in place (masking only on the diagonal block and where the sequence ends)
          const int key0 = kblk * AT_BLK + h * 32, qy = qblk * AT_BLK + r;
          const bool edge = (p.causal && kblk >= qblk) || (kblk + 1) * AT_BLK > p.S || (qblk + 1) * AT_BLK > p.S;
          uint64_t pr[16], dp[16];                                  // pairs of columns
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            pr[j] = f2_fma(f2_pack(__uint_as_float(sv[2 * j]), __uint_as_float(sv[2 * j + 1])), c2_2, nlse_2);
            dp[j] = f2_pack(__uint_as_float(dv[2 * j]), __uint_as_float(dv[2 * j + 1]));
          }
          if (edge) {
            // the last valid key of this row, relative to the thread's first column
            const int last = (qy < p.S ? (p.causal && qy < p.S - 1 ? qy : p.S - 1) : -1) - key0;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              float a0, a1;
              f2_unpack(pr[j], a0, a1);
              if (2 * j > last) a0 = -INFINITY;
              if (2 * j + 1 > last) a1 = -INFINITY;
              pr[j] = f2_pack(a0, a1);
            }
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            float a0, a1;
            f2_unpack(pr[j], a0, a1);
            pr[j] = f2_pack(ex2_approx(a0), ex2_approx(a1));
          }
          // the products of the step before have read the operands
          ok = __all_sync(0xFFFFFFFFu, mbar_wait(b_op_free, (jt & 1u) ^ 1u, abort_flag));
          if (!ok) break;
          const uint32_t op = op0 + row_off;
          auto put = [&](uint32_t o, const uint32_t (&w8)[8]) {
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(op + o * kF8Op + ch0), "r"(w8[0]), "r"(w8[1]), "r"(w8[2]), "r"(w8[3]) : "memory");
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(op + o * kF8Op + ch1), "r"(w8[4]), "r"(w8[5]), "r"(w8[6]), "r"(w8[7]) : "memory");
          };
          if (DV) {
            uint32_t w8[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) w8[j] = f8_encode4<BSP_E4M3>(f2_mul(pr[2 * j], ps_2), f2_mul(pr[2 * j + 1], ps_2));
            put(1u, w8);
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) pr[j] = f2_mul(pr[j], ds_2);  // P ds_scale: once for all draws
#pragma unroll
          for (int d = 0; d < (MC ? kF8ND : 1); ++d) {
            if (MC && d >= nd) break;
            uint32_t w8[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
              w8[j] = f8_encode4<BSP_E5M2>(f2_mul(pr[2 * j], f2_fma(dp[2 * j], dp_mul_2, ndk_2[d])),
                                           f2_mul(pr[2 * j + 1], f2_fma(dp[2 * j + 1], dp_mul_2, ndk_2[d])));
            put((uint32_t)d, w8);
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(b_op_ready);
          if (it == 0 && due) {
            ok = epilogue(vi - 1u);
            due = false;
            if (!ok) break;
          }
        }
        e_blk = blk; e_bh = bh; e_set = set; e_nd = nd; e_first = d0 == d_first; e_last = d0 + kF8ND >= d_end;
        due = true;
      }
    }
    if (ok && due) ok = epilogue(vi - 1u);
    if (warp == 0 && lane == 0) tma_store_wait_all();
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag && p.diag) atomicMax(&p.diag->status, (int)BSP_ERR_TIMEOUT);
  if constexpr (MC) {
    for (int n = *items_out, w; (w = item_at(n)) < nwork; ++n) {    // none, unless a wait ran out
      int blk, bh, set, a, b, c, d;
      decode(w, blk, bh, set, a, b, c, d);
      attn_fill_nan(p.s1, p.s2, set * p.BH + bh, blk, p.S, kF8Threads);
    }
  }
  if (warp == 17) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// The sum over the sets, in their order, of both sums of one gradient.
__global__ void __launch_bounds__(256)
sum_sets_kernel(const float* p1, const float* p2, int sets, float* S1, float* S2, size_t n4) {
  grid_dependency();
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  const float* src = blockIdx.y ? p2 : p1;
  float4 s = ldg(reinterpret_cast<const float4*>(src) + i);
  for (int k = 1; k < sets; ++k) {
    const float4 v = ldg(reinterpret_cast<const float4*>(src) + (size_t)k * n4 + i);
    s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
  }
  reinterpret_cast<float4*>(blockIdx.y ? S2 : S1)[i] = s;
}

// ------------------------------------------------------------------------------- host side

static int f8_params(AttnF8Params& p, int BH, int S, int causal, float c, const bsp_attn_fp8_t* f, const float* lse,
                     const float* dterm, bsp_diag_t* diag) {
  if (!f->q_codes || !f->k_codes || !f->v_codes || !f->do_codes) return BSP_ERR_ARG;
  if (!aligned16(f->q_codes) || !aligned16(f->k_codes) || !aligned16(f->v_codes) || !aligned16(f->do_codes)) return BSP_ERR_ALIGN;
  p.BH = BH; p.S = S; p.nblk = (S + AT_BLK - 1) / AT_BLK; p.causal = causal ? 1 : 0; p.c = c;
  p.lse = lse; p.dterm = dterm; p.K = 1; p.sets = 1; p.passes = 1; p.mc_ref = nullptr;
  p.sc_q = f->q_scale; p.sc_k = f->k_scale; p.sc_v = f->v_scale; p.sc_do = f->do_scale;
  p.p_scale = f->p_scale; p.ds_scale = f->ds_scale; p.diag = diag;
  return BSP_OK;
}

template <int MODE, bool MC, bool DV>
static int launch_f8(const bsp_attn_fp8_t* f, float* out0, float* out1, typename AttnF8Arg<MC>::type p, cudaStream_t st) {
  CUtensorMap mq, mk, mv, mdo, mo0, mo1;
  int rc;
  if ((rc = make_head_map_u8(&mq, f->q_codes, p.BH, p.S)) != BSP_OK) return rc;
  if ((rc = make_head_map_u8(&mk, f->k_codes, p.BH, p.S)) != BSP_OK) return rc;
  if ((rc = make_head_map_u8(&mv, f->v_codes, p.BH, p.S)) != BSP_OK) return rc;
  if ((rc = make_head_map_u8(&mdo, f->do_codes, p.BH, p.S)) != BSP_OK) return rc;
  if ((rc = make_out_map(&mo0, out0 ? out0 : out1, p.BH * p.sets, p.S)) != BSP_OK) return rc;
  if ((rc = make_out_map(&mo1, out1 ? out1 : out0, p.BH * p.sets, p.S)) != BSP_OK) return rc;
  static std::atomic<bool> attr_set_dev[kMaxDevices];       // per kernel instantiation and device
  std::atomic<bool>& attr_set = attr_set_dev[device_slot()];
  if (!attr_set.load(std::memory_order_acquire)) {
    BSP_CHECK_CUDA(cudaFuncSetAttribute(attn_f8_kernel<MODE, MC, DV>, cudaFuncAttributeMaxDynamicSharedMemorySize, kF8Smem));
    attr_set.store(true, std::memory_order_release);
  }
  const int nsm = sm_count_or_default();
  const int64_t nwork = (int64_t)p.nblk * p.BH * p.sets;
  if constexpr (MC) {
    p.s1 = out0; p.s2 = out1;
    if (p.walk > nwork) p.walk = (int)nwork;
  }
  launch_kernel(attn_f8_kernel<MODE, MC, DV>, (unsigned)(nwork < nsm ? nwork : nsm), kF8Threads, kF8Smem, st, mq, mk, mv, mdo, mo0,
                mo1, p);
  BSP_LAUNCH_CHECK();
  return BSP_OK;
}

int attn_f8_bwd(int BH, int S, int causal, float c, const bsp_attn_fp8_t* f, const float* lse, const float* dterm, float* dq,
                float* dk, float* dv, bsp_diag_t* diag, cudaStream_t st) {
  AttnF8Params p{};
  int rc = f8_params(p, BH, S, causal, c, f, lse, dterm, diag);
  if (rc != BSP_OK) return rc;
  if (dk && (rc = dv ? launch_f8<AT_DKV, false, true>(f, dv, dk, p, st) : launch_f8<AT_DKV, false, false>(f, nullptr, dk, p, st)) != BSP_OK)
    return rc;
  if (dq) return launch_f8<AT_DQ, false, false>(f, dq, nullptr, p, st);
  return BSP_OK;
}

// Sets the K draws are spread over: as many whole sets of the (block, head) items as the SMs take in one round (so from
// 75 items on one), each of at least one pass.  (The partial sums then stay below 148 x 128 x 64 floats per array.)
int attn_draw_sets(int64_t BH, int S, int K) {
  const int64_t items = ((int64_t)S + AT_BLK - 1) / AT_BLK * BH;
  const int passes = (K + kF8ND - 1) / kF8ND;
  int64_t sets = items > 0 ? kNumSMs / items : 1;
  if (sets > passes) sets = passes;
  if (sets <= 1) return 1;
  const int per = (passes + (int)sets - 1) / (int)sets;
  return (passes + per - 1) / per;                          // no empty set
}

int attn_sum_sets(const float* p1, const float* p2, int sets, float* S1, float* S2, size_t n, cudaStream_t st) {
  const dim3 grid((unsigned)((n / 4 + 255) / 256), 2);
  launch_kernel(sum_sets_kernel, grid, 256, 0, st, p1, p2, sets, S1, S2, n / 4);
  BSP_LAUNCH_CHECK();
  return BSP_OK;
}

int attn_f8_draws(int BH, int S, int causal, float c, const bsp_attn_fp8_t* f, const float* lse, const float* dterm, int K,
                  const float* ref_dq, float* S1q, float* S2q, const float* ref_dk, float* S1k, float* S2k, float* partials,
                  int walk, bsp_diag_t* diag, cudaStream_t st) {
  AttnF8Draws p{};
  int rc = f8_params(p, BH, S, causal, c, f, lse, dterm, diag);
  if (rc != BSP_OK) return rc;
  p.K = K;
  p.walk = walk;
  p.sets = partials ? attn_draw_sets(BH, S, K) : 1;
  p.passes = ((K + kF8ND - 1) / kF8ND + p.sets - 1) / p.sets;
  const size_t n = (size_t)BH * S * AT_D;
  float* part[4] = {S1k, S2k, S1q, S2q};
  if (p.sets > 1)
    for (int i = 0; i < 4; ++i) part[i] = partials + (size_t)i * p.sets * n;
  p.mc_ref = ref_dk;
  if ((rc = launch_f8<AT_DKV, true, false>(f, part[0], part[1], p, st)) != BSP_OK) return rc;
  p.mc_ref = ref_dq;
  if ((rc = launch_f8<AT_DQ, true, false>(f, part[2], part[3], p, st)) != BSP_OK) return rc;
  if (p.sets == 1) return BSP_OK;
  if ((rc = attn_sum_sets(part[0], part[1], p.sets, S1k, S2k, n, st)) != BSP_OK) return rc;
  return attn_sum_sets(part[2], part[3], p.sets, S1q, S2q, n, st);
}

}  // namespace bsp
