// Dense contractions on the 5th-generation tensor cores: C[M,N] = alpha * A[M,K] B[N,K]^T with
// both operands K-major (K contiguous), FP8 (kind::f8f6f4, E5M2/E4M3 in any combination) or BF16
// (kind::f16) operands and FP32 accumulation in tensor memory.
//
// One persistent CTA per SM, 320 threads:
//   warp 0      TMA producer   (cp.async.bulk.tensor, 128-byte swizzle, kStages-deep mbarrier ring)
//   warp 1      MMA issuer     (one elected lane issues tcgen05.mma 128 x 256 x 32B; owns TMEM alloc)
//   warps 2..9  epilogue       (tcgen05.ld 32 lanes x 32 columns -> registers -> global; two warps per
//               lane quarter take every other 32 columns: with one, a tile of a short contraction (K of
//               1024 and below) spent longer in its epilogue than in its products)
// Two accumulator stages (2 x 256 TMEM columns) let the epilogue of one tile overlap the main loop
// of the next.  Work items are (tile, batch): a CTA owns its tiles and walks all batches of a tile
// in order, so the Monte-Carlo epilogue's read-modify-write of the shifted sums is race-free and
// bit-reproducible.  Every wait is bounded; on time-out the kernel records BSP_ERR_TIMEOUT in the
// diagnostics word and unwinds (TMEM is freed on every path).
#include <atomic>
#include <cuda.h>
#include <stdlib.h>

#include "common.cuh"
#include "gemm.cuh"
#include "tc.cuh"

namespace bsp {

// ------------------------------------------------------------------------------- the kernel

constexpr int BM = 128, BN = 256, BKB = 128;      // tile; BKB = K extent of one stage in bytes
constexpr int kStages = 4;
constexpr int kABytes = BM * BKB, kBBytes = BN * BKB, kStageBytes = kABytes + kBBytes;
constexpr int kGemmThreads = 320;
constexpr int kTmemCols = 512;
constexpr int kEpiStage = 8 * 4096;              // one 32-row x 128-byte staging block per epilogue warp
constexpr int kPairStages = 6, kPairStageBytes = kABytes + kBBytes / 2;   // a CTA of a pair holds half of B's tile
static_assert(kPairStages * kPairStageBytes == kStages * kStageBytes, "one ring size");
constexpr size_t kGemmSmem = (size_t)kStages * kStageBytes + 1024 /*alignment slack*/ + 256 /*barriers*/ + kEpiStage;

struct GemmParams {
  int M, N, K;            // K in elements
  int bn;                 // gemm_tc_kernel: tile columns (see tile_columns)
  int nb;                 // batches of B (and of C in plain mode)
  int a_mn, b_mn;         // operand stored [K][M] / [K][N] (MN-major) instead of [M][K] / [N][K]
  uint32_t idesc;
  uint32_t idesc2;               // gemm_mc_kernel: the 128 x 256 product over a pair of draws
  float sa, sb;           // operand scales; alpha = (1/sa) * (1/sb)
  const float* sa_dev;
  const float* sb_dev;
  int mode;               // EPI_*
  void* C;                // float or bf16 [nb][M][ldc]
  int64_t ldc;
  const float* ref;       // EPI_MC
  float* S1;
  float* S2;
  uint16_t* split;        // EPI_SPLIT
  uint16_t* diff;
  float moment_scale;     // EPI_MOMENTS
  int moment_first;
  bsp_diag_t* diag;
};

// Tile t of the persistent walk -> (tm, tn).  The tile columns are taken in bands of kBandTiles: inside
// a band the walk is row-major, so the CTAs of one wave (consecutive t) cover about 148 / 8 tile rows
// by 8 tile columns, and the A and B panels they stream together stay within L2 (for a wide N, a
// plain row-major walk has every CTA of a wave on its own B panel: 32 panels of 2 MB per draw at
// T = 16384).  With at most kBandTiles tile columns this is the plain row-major order.
constexpr int kBandTiles = 8;
__device__ __forceinline__ void tile_coords(int t, int tiles_m, int tiles_n, int& tm, int& tn) {
  const int per_band = kBandTiles * tiles_m;
  const int band = t / per_band, idx = t - band * per_band;
  const int c0 = band * kBandTiles;
  const int wb = tiles_n - c0 < kBandTiles ? tiles_n - c0 : kBandTiles;
  tm = idx / wb;
  tn = c0 + idx - tm * wb;
}

// Four values as two bf16 terms each, packed in pairs: v = hi + lo to 16 bits.
__device__ __forceinline__ void split4(const float4& v, uint2& hi, uint2& lo) {
  const uint32_t h0 = float_to_bf16_bits(v.x), h1 = float_to_bf16_bits(v.y), h2 = float_to_bf16_bits(v.z), h3 = float_to_bf16_bits(v.w);
  hi = make_uint2(h0 | (h1 << 16), h2 | (h3 << 16));
  lo = make_uint2(float_to_bf16_bits(v.x - bf16_bits_to_float(h0)) | (float_to_bf16_bits(v.y - bf16_bits_to_float(h1)) << 16),
                  float_to_bf16_bits(v.z - bf16_bits_to_float(h2)) | (float_to_bf16_bits(v.w - bf16_bits_to_float(h3)) << 16));
}

// PAIR: two CTAs of a cluster take two tile rows of the same columns as one product over 256 rows
// (cta_group::2), each with its own A rows and half of B's columns: (128 + bn / 2) instead of (128 + bn)
// rows through L2 and shared memory per CTA.  The leader (rank 0) issues for both.
template <bool FP8, int MODE, bool PAIR>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b, GemmParams p) {
  grid_dependency();
  constexpr int kStages = PAIR ? kPairStages : bsp::kStages, kStageBytes = PAIR ? kPairStageBytes : bsp::kStageBytes, kCtas = PAIR ? 2 : 1;
  constexpr int kElem = FP8 ? 1 : 2, bk_elems = BKB / kElem, kAtom = 128 / kElem;   // elements per 128 bytes
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles = (raw + 1023u) & ~1023u;                    // 1024-byte aligned operand ring
  const uint32_t bars = tiles + kStages * kStageBytes;              // barriers after the ring
  // barrier layout (8 bytes each): full[kStages], empty[kStages], tfull[2], tempty[2]; then tmem slot, abort flag
  const uint32_t full0 = bars, empty0 = bars + 8 * kStages, tfull0 = bars + 16 * kStages, tempty0 = tfull0 + 16;
  const uint32_t epi_stage = bars + 256;                            // staging blocks of the epilogue warps
  uint8_t* bars_gen = smem_raw + (bars - raw);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bars_gen + 16 * kStages + 32);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars_gen + 16 * kStages + 36);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = PAIR ? (int)cluster_rank() : 0, bn_cta = p.bn / kCtas;   // columns of B this CTA loads
  const int tiles_m = (p.M + kCtas * BM - 1) / (kCtas * BM), tiles_n = (p.N + p.bn - 1) / p.bn;
  const int ntiles = tiles_m * tiles_n;
  const int kblocks = (p.K * kElem + BKB - 1) / BKB;
  // an MN-major B comes in atoms of 128 bytes of N: the last one may reach past the tile's columns
  const int b_atoms = (bn_cta * kElem + 127) / 128, b_bytes = p.b_mn ? b_atoms * bk_elems * 128 : bn_cta * BKB;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull0 + 8 * a, 1); mbar_init(tempty0 + 8 * a, 8 * kCtas); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    if (PAIR) tmem_alloc2(smem_u32(const_cast<uint32_t*>(tmem_slot)), kTmemCols);
    else tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), kTmemCols);
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();                              // both CTAs' barriers exist before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------ TMA producer
    if (lane == 0) {
      tma_prefetch_desc(&tmap_a);
      tma_prefetch_desc(&tmap_b);
      uint32_t it = 0;
      bool ok = true;
      for (int t = blockIdx.x / kCtas; t < ntiles && ok; t += gridDim.x / kCtas) {
        int tm, tn;
      tile_coords(t, tiles_m, tiles_n, tm, tn);
        for (int b = 0; b < p.nb && ok; ++b) {
          for (int kb = 0; kb < kblocks; ++kb, ++it) {
            const uint32_t s = it % kStages, ph = (it / kStages) & 1u;
            if (!mbar_wait(empty0 + 8 * s, ph ^ 1u, abort_flag)) { ok = false; break; }
            const uint32_t sa = tiles + s * kStageBytes, sb = sa + kABytes;
            // the leader's barrier counts both CTAs' bytes
            const uint32_t bar = PAIR ? leader_addr(full0 + 8 * s) : full0 + 8 * s;
            if (rank == 0) mbar_expect_tx(full0 + 8 * s, kCtas * (kABytes + b_bytes));
            const int row0 = (kCtas * tm + rank) * BM, col0 = tn * p.bn + rank * bn_cta;
            if (!p.a_mn) {
              tma_load_2d_c<PAIR>(sa, &tmap_a, bar, kb * bk_elems, row0);
            } else {
              // one box per 128 bytes of M: [bk_elems k rows][128 B]
#pragma unroll
              for (int a = 0; a < BM / kAtom; ++a)
                tma_load_2d_c<PAIR>(sa + a * bk_elems * 128, &tmap_a, bar, row0 + a * kAtom, kb * bk_elems);
            }
            if (!p.b_mn) {
              tma_load_3d_c<PAIR>(sb, &tmap_b, bar, kb * bk_elems, col0, b);
            } else {
#pragma unroll
              for (int a = 0; a < BN / kCtas / kAtom; ++a)
                if (a < b_atoms)
                  tma_load_3d_c<PAIR>(sb + a * bk_elems * 128, &tmap_b, bar, col0 + a * kAtom, kb * bk_elems, b);
            }
          }
        }
      }
      if (!ok) {
        // let copies already in flight land before the CTA's shared memory is released
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------ MMA issuer
    if (lane == 0 && rank == 0) {
      uint32_t it = 0, tc = 0;
      bool ok = true;
      for (int t = blockIdx.x / kCtas; t < ntiles && ok; t += gridDim.x / kCtas) {
        for (int b = 0; b < p.nb && ok; ++b, ++tc) {
          const uint32_t as = tc & 1u, aph = (tc >> 1) & 1u;
          if (!mbar_wait(tempty0 + 8 * as, aph ^ 1u, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t tmem_d = tmem_base + as * BN;
          for (int kb = 0; kb < kblocks; ++kb, ++it) {
            const uint32_t s = it % kStages, ph = (it / kStages) & 1u;
            if (!mbar_wait(full0 + 8 * s, ph, abort_flag)) { ok = false; break; }
            tc_fence_after();
            const uint32_t sa = tiles + s * kStageBytes, sb = sa + kABytes;
            // K-major: one MMA advances 32 bytes along K inside the swizzle atom (+2 in 16-byte
            // units).  MN-major: it advances 32/elem_bytes k rows of 128 bytes.
            const uint32_t atom_bytes = (uint32_t)bk_elems * 128u;
            const uint32_t mn_step = (32u / (uint32_t)kElem) * 128u >> 4;
            const uint64_t adesc = p.a_mn ? make_smem_desc_mn(sa, atom_bytes) : make_smem_desc(sa);
            const uint64_t bdesc = p.b_mn ? make_smem_desc_mn(sb, atom_bytes) : make_smem_desc(sb);
            const uint32_t astep = p.a_mn ? mn_step : 2u, bstep = p.b_mn ? mn_step : 2u;
#pragma unroll
            for (int k = 0; k < BKB / 32; ++k)
              if (PAIR) tc_mma2<FP8>(tmem_d, adesc + astep * k, bdesc + bstep * k, p.idesc, (kb | k) != 0 ? 1u : 0u);
              else tc_mma<FP8>(tmem_d, adesc + astep * k, bdesc + bstep * k, p.idesc, (kb | k) != 0 ? 1u : 0u);
            if (PAIR) tc_commit2(empty0 + 8 * s);   // frees the stage when these MMAs have read it
            else tc_commit(empty0 + 8 * s);
          }
          if (ok) {                                 // accumulator complete
            if (PAIR) tc_commit2(tfull0 + 8 * as);
            else tc_commit(tfull0 + 8 * as);
          }
        }
      }
    }
  } else {
    // ------------------------------------------------ epilogue (warps 2..9)
    const int q = warp & 3;                      // TMEM lane quarter this warp may access
    const float inv_a = __fdiv_rn(1.0f, p.sa_dev ? ldg(p.sa_dev) : p.sa);
    const float inv_b = __fdiv_rn(1.0f, p.sb_dev ? ldg(p.sb_dev) : p.sb);
    uint32_t tc = 0;
    bool ok = true;
    for (int t = blockIdx.x / kCtas; t < ntiles && ok; t += gridDim.x / kCtas) {
      int tm, tn;
      tile_coords(t, tiles_m, tiles_n, tm, tn);
      const int row0 = (kCtas * tm + rank) * BM, row = row0 + q * 32 + lane;
      const int nlim = p.N < (tn + 1) * p.bn ? p.N : (tn + 1) * p.bn;   // columns from here on are not this tile's
      for (int b = 0; b < p.nb && ok; ++b, ++tc) {
        const uint32_t as = tc & 1u, aph = (tc >> 1) & 1u;
        // every lane polls; the outcome is made warp-uniform before any .aligned instruction
        ok = __all_sync(0xFFFFFFFFu, mbar_wait_suspend(tfull0 + 8 * as, aph, abort_flag));
        if (!ok) break;
        tc_fence_after();
        const uint32_t taddr = tmem_base + as * BN + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
        for (int ch = (warp - 2) >> 2; ch < BN / 32; ch += 2) {
          const int col0 = tn * p.bn + ch * 32;
          if (col0 >= nlim) break;               // warp-uniform
          uint32_t r[32];
          // what the warp will write goes row by row (row 4 t + lane / 8, four columns from 4 (lane % 8)); the
          // values that an epilogue reads back there are fetched before the accumulator
          constexpr bool by_rows = MODE != EPI_STORE_BF16;
          const int row8 = row0 + q * 32 + (lane >> 3), col4 = col0 + 4 * (lane & 7);
          float4 old1[8], old2[8];
          const bool reads1 = (MODE == EPI_SPLIT && p.ref) || (MODE == EPI_MOMENTS && !p.moment_first);
          if (reads1) {
            const float* src = MODE == EPI_SPLIT ? p.ref : p.S1;
#pragma unroll
            for (int t8 = 0; t8 < 8; ++t8)
              if (row8 + 4 * t8 < p.M && col4 < nlim) {
                old1[t8] = *reinterpret_cast<const float4*>(src + (size_t)(row8 + 4 * t8) * p.ldc + col4);
                if (MODE == EPI_MOMENTS) old2[t8] = *reinterpret_cast<const float4*>(p.S2 + (size_t)(row8 + 4 * t8) * p.ldc + col4);
              }
          }
          tmem_ld32(taddr + ch * 32, r);
          if (by_rows) {
            // A lane holds 128 bytes of its own row; written as they are, a warp's store touches 32
            // rows with 16 bytes each.  Through the warp's 4 KB staging block the warp instead writes
            // four rows of 128 contiguous bytes per instruction (row 4 t + lane / 8, chunk lane % 8).
            const uint32_t wb = epi_stage + (uint32_t)(warp - 2) * 4096u;
#pragma unroll
            for (int j = 0; j < 8; ++j)
              asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(wb + (uint32_t)lane * 128u + ((uint32_t)(j ^ (lane & 7)) << 4)),
                           "f"(__uint_as_float(r[4 * j]) * inv_a * inv_b), "f"(__uint_as_float(r[4 * j + 1]) * inv_a * inv_b),
                           "f"(__uint_as_float(r[4 * j + 2]) * inv_a * inv_b), "f"(__uint_as_float(r[4 * j + 3]) * inv_a * inv_b)
                           : "memory");
            __syncwarp();
            float* cbase = reinterpret_cast<float*>(p.C) + (size_t)b * p.M * p.ldc;
#pragma unroll
            for (int t8 = 0; t8 < 8; ++t8) {
              const int rl = 4 * t8 + (lane >> 3), c4 = lane & 7;
              float4 o;
              asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                           : "=f"(o.x), "=f"(o.y), "=f"(o.z), "=f"(o.w)
                           : "r"(wb + (uint32_t)rl * 128u + ((uint32_t)(c4 ^ (rl & 7)) << 4)));
              const int orow = row0 + q * 32 + rl, ocol = col0 + 4 * c4;
              if (orow < p.M && ocol < nlim) {
                const size_t off = (size_t)orow * p.ldc + ocol;
                if (MODE == EPI_STORE_F32) {
                  *reinterpret_cast<float4*>(cbase + off) = o;
                } else if (MODE == EPI_SPLIT) {
                  if (p.C) *reinterpret_cast<float4*>(cbase + off) = o;
                  uint2 hi, lo;
                  split4(o, hi, lo);
                  uint16_t* sp = p.split + (size_t)orow * 2 * p.N + ocol;
                  *reinterpret_cast<uint2*>(sp) = hi;
                  *reinterpret_cast<uint2*>(sp + p.N) = lo;
                  if (p.ref) {
                    const float4 a = old1[t8];
                    split4(make_float4(a.x - o.x, a.y - o.y, a.z - o.z, a.w - o.w), hi, lo);
                    uint16_t* df = p.diff + (size_t)orow * p.N + ocol;
                    *reinterpret_cast<uint2*>(df) = hi;
                    *reinterpret_cast<uint2*>(df + (size_t)p.M * p.N) = lo;
                  }
                } else {
                  const float f = p.moment_scale;
                  float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b2 = a;
                  if (!p.moment_first) { a = old1[t8]; b2 = old2[t8]; }
                  a.x = fmaf(f, o.x, a.x); a.y = fmaf(f, o.y, a.y); a.z = fmaf(f, o.z, a.z); a.w = fmaf(f, o.w, a.w);
                  b2.x = fmaf(f * o.x, o.x, b2.x); b2.y = fmaf(f * o.y, o.y, b2.y);
                  b2.z = fmaf(f * o.z, o.z, b2.z); b2.w = fmaf(f * o.w, o.w, b2.w);
                  *reinterpret_cast<float4*>(p.S1 + off) = a;
                  *reinterpret_cast<float4*>(p.S2 + off) = b2;
                }
              }
            }
            __syncwarp();
          }
          if (row < p.M) {
            const size_t off = (size_t)row * p.ldc + col0;
            if (!by_rows) {
              uint16_t* dst = reinterpret_cast<uint16_t*>(p.C) + (size_t)b * p.M * p.ldc + off;
#pragma unroll
              for (int j = 0; j < 32; j += 4) {
                if (col0 + j < nlim) {
                  const uint32_t lo = float_to_bf16_bits(__uint_as_float(r[j]) * inv_a * inv_b) |
                                      (float_to_bf16_bits(__uint_as_float(r[j + 1]) * inv_a * inv_b) << 16);
                  const uint32_t hi = float_to_bf16_bits(__uint_as_float(r[j + 2]) * inv_a * inv_b) |
                                      (float_to_bf16_bits(__uint_as_float(r[j + 3]) * inv_a * inv_b) << 16);
                  *reinterpret_cast<uint2*>(dst + j) = make_uint2(lo, hi);
                }
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (PAIR) mbar_arrive_cluster(leader_addr(tempty0 + 8 * as));
          else mbar_arrive(tempty0 + 8 * as);
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();                              // nothing of this CTA is used by the other any more
  if (threadIdx.x == 0 && *abort_flag && p.diag) atomicMax(&p.diag->status, (int)BSP_ERR_TIMEOUT);
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    if (PAIR) tmem_dealloc2(tmem_base, kTmemCols);
    else tmem_dealloc(tmem_base, kTmemCols);
  }
}

// ------------------------------------------------------------------------------- Monte-Carlo contraction

// Contraction over nb draws of B with the per-element shifted sums kept on chip: for every output tile
// the CTA walks the draws b and accumulates
//   S1 += alpha*acc_b - ref,   S2 += (alpha*acc_b - ref)^2
// without ever writing a per-draw gradient.  Tile 128 x 128, draws two at a time: a stage of the ring
// holds the A tile and the B tiles of both draws, so one 128 x 256 product per K slice fills both
// accumulators and the A tile is fetched (from L2 and from shared memory) once for two draws.
//
// 384 threads: warp 0 TMA, warp 1 MMA, warps 4..11 epilogue (two warps per TMEM lane quarter, each
// owning 64 of the 128 columns).  The reference and both sums of a tile sit in the epilogue threads'
// registers (3 x 64), to which the producer's warpgroup gives up its share; that leaves all 512 columns
// of tensor memory to two pairs of accumulators, so the products of a pair run under the epilogue of
// the pair before.  With the sums in tensor memory (one pair of accumulators) every pair ended in an
// epilogue the tensor pipe waited for: 4096 x 1024 x 4096, 64 draws (with the split below): 847 -> 767 us.
//
// PAIR: two CTAs of a cluster take two tile rows of the same columns as one product over 256 rows
// (cta_group::2): each loads its own A rows and one of the two draws' B tiles, 32 KB per 128 bytes of K
// instead of 48, which is what L2 has to deliver to every SM (96 bytes per cycle at the tensor rate
// without pairs, of about 80 that the times of unpaired products allow; no counter was read): see mc_pairs for what it measured.  The leader's (rank 0) warp 1
// issues for both; its full barriers count both CTAs' bytes, its commits arrive in both.
//
// The walk is over units (tile, range of draws).  Whole waves of tiles take all their draws; the tiles
// of a last, partial wave (or of a problem with fewer tiles than SMs) are cut into nseg ranges, range
// by range over the tiles, so that CTAs which run together read the same draws.  Range 0 adds to S1 and
// S2, range s > 0 writes its sums to slot (s - 1) of the split workspace, and gemm_mc_merge_kernel adds
// the slots in order: every sum has one order, whatever the scheduling.
constexpr int MC_BN = 128;
constexpr int kMcABytes = BM * BKB, kMcBBytes = MC_BN * BKB;
template <bool PAIR> struct McRing {
  static constexpr int kStages = PAIR ? 6 : 4, kStageBytes = kMcABytes + (PAIR ? 1 : 2) * kMcBBytes;
};
static_assert(McRing<true>::kStages * McRing<true>::kStageBytes == McRing<false>::kStages * McRing<false>::kStageBytes, "one ring size");
constexpr int kMcThreads = 384;
constexpr int kMcRegsProducer = 40, kMcRegsEpilogue = 232;   // 40 + 2 * 232 = 3 * 168: the launch's registers
constexpr size_t kMcSmem = (size_t)McRing<true>::kStages * McRing<true>::kStageBytes + 1024 + 256;
constexpr size_t kMcSplitTileFloats = (size_t)2 * BM * MC_BN;   // S1 and S2 of one tile in a split slot

// Units of the walk: tiles [0, whole) with all draws, then nseg ranges over the other tiles.
struct McSplit {
  int whole, rest, nseg, pairs_per_seg;
  int first;                             // the sums start with this launch's draws
};
__device__ __forceinline__ void mc_unit(const McSplit& sp, int u, int npairs, int& tile, int& seg, int& p0, int& p1) {
  if (u < sp.whole) { tile = u; seg = 0; p0 = 0; p1 = npairs; return; }
  const int v = u - sp.whole;
  seg = v / sp.rest;
  tile = sp.whole + v - seg * sp.rest;
  p0 = seg * sp.pairs_per_seg;
  p1 = p0 + sp.pairs_per_seg < npairs ? p0 + sp.pairs_per_seg : npairs;
}

template <bool FP8, bool PAIR>
__global__ void __launch_bounds__(kMcThreads, 1)
gemm_mc_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b, GemmParams p,
               McSplit sp, float* split_ws) {
  grid_dependency();
  constexpr int kMcStages = McRing<PAIR>::kStages, kMcStageBytes = McRing<PAIR>::kStageBytes, kCtas = PAIR ? 2 : 1;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles = (raw + 1023u) & ~1023u;
  const uint32_t bars = tiles + kMcStages * kMcStageBytes;
  const uint32_t full0 = bars, empty0 = bars + 8 * kMcStages, tfull0 = bars + 16 * kMcStages, tempty0 = tfull0 + 16;
  uint8_t* bars_gen = smem_raw + (bars - raw);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(bars_gen + 16 * kMcStages + 32);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars_gen + 16 * kMcStages + 36);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = PAIR ? (int)cluster_rank() : 0;
  const int tiles_m = (p.M + kCtas * BM - 1) / (kCtas * BM), tiles_n = (p.N + MC_BN - 1) / MC_BN;
  const int nunits = sp.whole + sp.rest * sp.nseg, npairs = (p.nb + 1) / 2;
  constexpr int kElemsPerStage = FP8 ? BKB : BKB / 2;   // K extent of one 128-byte stage in elements
  const int kblocks = (p.K + kElemsPerStage - 1) / kElemsPerStage;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMcStages; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull0 + 8 * a, 1); mbar_init(tempty0 + 8 * a, 8 * kCtas); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    if (PAIR) tmem_alloc2(smem_u32(const_cast<uint32_t*>(tmem_slot)), kTmemCols);
    else tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), kTmemCols);
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();                              // both CTAs' barriers exist before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kMcRegsProducer));
    if (warp == 0 && lane == 0) {
      tma_prefetch_desc(&tmap_a);
      tma_prefetch_desc(&tmap_b);
      // the dY panel of a tile row is read again by every pass over a pair of draws (and by the
      // other tiles of the row): it should outlive the fresh-code panels, which a wave reads once
      const uint64_t keep = l2_policy_evict_last();
      uint32_t it = 0;
      bool ok = true;
      for (int u = blockIdx.x / kCtas; u < nunits && ok; u += gridDim.x / kCtas) {
        int t, seg, p0, p1, tm, tn;
        mc_unit(sp, u, npairs, t, seg, p0, p1);
        tile_coords(t, tiles_m, tiles_n, tm, tn);
        for (int pr = p0; pr < p1 && ok; ++pr) {
          const int b = 2 * pr;
          const bool two = b + 1 < p.nb;                       // an odd count ends with a single draw
          for (int kb = 0; kb < kblocks; ++kb, ++it) {
            const uint32_t s = it % kMcStages, ph = (it / kMcStages) & 1u;
            if (!mbar_wait(empty0 + 8 * s, ph ^ 1u, abort_flag)) { ok = false; break; }
            const uint32_t sa = tiles + s * kMcStageBytes, sb = sa + kMcABytes;
            if (PAIR) {
              // one draw's B tile per CTA; of a single draw's tile a CTA provides half the columns (the box
              // is whole all the same).  Bytes that arrive before the leader announces them only make
              // its count negative for a while: the phase still waits for the leader's own arrival.
              const uint32_t bar = leader_addr(full0 + 8 * s);
              if (rank == 0) mbar_expect_tx(full0 + 8 * s, 2 * kMcStageBytes);
              tma_load_2d_pair(sa, &tmap_a, bar, kb * kElemsPerStage, (2 * tm + rank) * BM, keep);
              tma_load_3d_pair(sb, &tmap_b, bar, kb * kElemsPerStage, tn * MC_BN + (two ? 0 : rank * (MC_BN / 2)),
                               two ? b + rank : b);
              continue;
            }
            mbar_expect_tx(full0 + 8 * s, kMcABytes + (two ? 2 : 1) * kMcBBytes);
            tma_load_2d_hint(sa, &tmap_a, full0 + 8 * s, kb * kElemsPerStage, tm * BM, keep);
            tma_load_3d(sb, &tmap_b, full0 + 8 * s, kb * kElemsPerStage, tn * MC_BN, b);
            if (two) tma_load_3d(sb + kMcBBytes, &tmap_b, full0 + 8 * s, kb * kElemsPerStage, tn * MC_BN, b + 1);
          }
        }
      }
      if (!ok) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
      }
    } else if (warp == 1 && lane == 0 && rank == 0) {
      uint32_t it = 0, tc = 0;
      bool ok = true;
      for (int u = blockIdx.x / kCtas; u < nunits && ok; u += gridDim.x / kCtas) {
        int t, seg, p0, p1;
        mc_unit(sp, u, npairs, t, seg, p0, p1);
        for (int pr = p0; pr < p1 && ok; ++pr, ++tc) {
          const uint32_t as = tc & 1u, aph = (tc >> 1) & 1u;
          // the epilogue of the pair before last must be through with this pair of accumulators
          if (!mbar_wait(tempty0 + 8 * as, aph ^ 1u, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint32_t idesc = 2 * pr + 1 < p.nb ? p.idesc2 : p.idesc, tmem_d = tmem_base + as * 2 * MC_BN;
          for (int kb = 0; kb < kblocks; ++kb, ++it) {
            const uint32_t s = it % kMcStages, ph = (it / kMcStages) & 1u;
            if (!mbar_wait(full0 + 8 * s, ph, abort_flag)) { ok = false; break; }
            tc_fence_after();
            const uint32_t sa = tiles + s * kMcStageBytes, sb = sa + kMcABytes;
            const uint64_t adesc = make_smem_desc(sa), bdesc = make_smem_desc(sb);   // B: 128 or 256 rows
#pragma unroll
            for (int k = 0; k < BKB / 32; ++k) {
              if (PAIR) tc_mma2<FP8>(tmem_d, adesc + 2u * k, bdesc + 2u * k, idesc, (kb | k) != 0 ? 1u : 0u);
              else tc_mma<FP8>(tmem_d, adesc + 2u * k, bdesc + 2u * k, idesc, (kb | k) != 0 ? 1u : 0u);
            }
            if (PAIR) tc_commit2(empty0 + 8 * s);
            else tc_commit(empty0 + 8 * s);
          }
          if (ok) {
            if (PAIR) tc_commit2(tfull0 + 8 * as);
            else tc_commit(tfull0 + 8 * as);
          }
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kMcRegsEpilogue));
    const int q = warp & 3;                  // TMEM lane quarter
    const int h = (warp - 4) >> 2;           // column half
    const float inv_a = __fdiv_rn(1.0f, p.sa_dev ? ldg(p.sa_dev) : p.sa);
    const float inv_b = __fdiv_rn(1.0f, p.sb_dev ? ldg(p.sb_dev) : p.sb);
    const uint32_t lane_base = tmem_base + ((uint32_t)(q * 32) << 16) + h * 64;
    uint32_t tc = 0;
    bool ok = true;
    for (int u = blockIdx.x / kCtas; u < nunits && ok; u += gridDim.x / kCtas) {
      int t, seg, p0, p1, tm, tn;
      mc_unit(sp, u, npairs, t, seg, p0, p1);
      tile_coords(t, tiles_m, tiles_n, tm, tn);
      const int row = (kCtas * tm + rank) * BM + q * 32 + lane;
      const int colbase = tn * MC_BN + h * 64;
      float refv[64], s1[64], s2[64];
      // ---- unit start: the reference, and the sums so far when this unit continues them
#pragma unroll
      for (int c = 0; c < 64; c += 4) {
        float4 g0 = make_float4(0.f, 0.f, 0.f, 0.f), v1 = g0, v2 = g0;
        if (row < p.M && colbase + c < p.N) {
          const size_t off = (size_t)row * p.ldc + colbase + c;
          // no reference: the products are differences to the reference already
          if (p.ref) g0 = *reinterpret_cast<const float4*>(p.ref + off);
          if (seg == 0 && !sp.first) {
            v1 = *reinterpret_cast<const float4*>(p.S1 + off);
            v2 = *reinterpret_cast<const float4*>(p.S2 + off);
          }
        }
        refv[c] = g0.x; refv[c + 1] = g0.y; refv[c + 2] = g0.z; refv[c + 3] = g0.w;
        s1[c] = v1.x; s1[c + 1] = v1.y; s1[c + 2] = v1.z; s1[c + 3] = v1.w;
        s2[c] = v2.x; s2[c + 1] = v2.y; s2[c + 2] = v2.z; s2[c + 3] = v2.w;
      }
      // ---- the unit's draws
      for (int pr = p0; pr < p1 && ok; ++pr, ++tc) {
        const uint32_t as = tc & 1u, aph = (tc >> 1) & 1u;
        ok = __all_sync(0xFFFFFFFFu, mbar_wait_suspend(tfull0 + 8 * as, aph, abort_flag));
        if (!ok) break;
        tc_fence_after();
        const uint32_t acc_base = lane_base + as * 2 * MC_BN;  // draw 2 pr; draw 2 pr + 1 is MC_BN columns further
        // the sums take the draws in order, as a one-draw-at-a-time pass would
#pragma unroll
        for (int d = 0; d < 2; ++d) {
          if (d == 0 || 2 * pr + 1 < p.nb) {
#pragma unroll
            for (int c = 0; c < 64; c += 16) {
              uint32_t acc[16];
              tmem_ld16(acc_base + d * MC_BN + c, acc);
              tmem_wait_ld();
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const float e = __uint_as_float(acc[j]) * inv_a * inv_b - refv[c + j];
                s1[c + j] += e;
                s2[c + j] = fmaf(e, e, s2[c + j]);
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (PAIR) mbar_arrive_cluster(leader_addr(tempty0 + 8 * as));
          else mbar_arrive(tempty0 + 8 * as);
        }
      }
      if (!ok) break;
      // ---- unit end: the sums back to S1 and S2, or to the unit's split slot
      if (seg == 0) {
#pragma unroll
        for (int c = 0; c < 64; c += 4)
          if (row < p.M && colbase + c < p.N) {
            const size_t off = (size_t)row * p.ldc + colbase + c;
            *reinterpret_cast<float4*>(p.S1 + off) = make_float4(s1[c], s1[c + 1], s1[c + 2], s1[c + 3]);
            *reinterpret_cast<float4*>(p.S2 + off) = make_float4(s2[c], s2[c + 1], s2[c + 2], s2[c + 3]);
          }
      } else {
        // [S1 | S2][column / 4][row] as groups of four columns: a warp writes 512 consecutive bytes
        float4* slot = reinterpret_cast<float4*>(split_ws + (((size_t)(seg - 1) * sp.rest + (t - sp.whole)) * kCtas + rank) * kMcSplitTileFloats) +
                       (h * 16) * BM + q * 32 + lane;
#pragma unroll
        for (int c = 0; c < 64; c += 4) {
          slot[(c / 4) * BM] = make_float4(s1[c], s1[c + 1], s1[c + 2], s1[c + 3]);
          slot[(MC_BN / 4 + c / 4) * BM] = make_float4(s2[c], s2[c + 1], s2[c + 2], s2[c + 3]);
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();                              // nothing of this CTA is used by the other any more
  if (threadIdx.x == 0 && *abort_flag && p.diag) atomicMax(&p.diag->status, (int)BSP_ERR_TIMEOUT);
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    if (PAIR) tmem_dealloc2(tmem_base, kTmemCols);
    else tmem_dealloc(tmem_base, kTmemCols);
  }
}

// S1 += slot sums, S2 likewise, of the tiles whose draws were split.  Block (t, y): tile whole + t / ctas
// (its row tile t % ctas), a
// thread takes four columns of one row; slots are added in the order of their draws.
__global__ void __launch_bounds__(256)
gemm_mc_merge_kernel(const float* split_ws, McSplit sp, int ctas, int M, int N, int64_t ldc, float* S1,
                     float* S2) {
  grid_dependency();
  const int tiles_m = (M + ctas * BM - 1) / (ctas * BM), tiles_n = (N + MC_BN - 1) / MC_BN;
  int tm, tn;
  tile_coords(sp.whole + (int)blockIdx.x / ctas, tiles_m, tiles_n, tm, tn);
  tm = tm * ctas + (int)blockIdx.x % ctas;
  const int i = (int)blockIdx.y * 256 + threadIdx.x, second = i >= BM * MC_BN / 4, k = i - second * (BM * MC_BN / 4);
  const int row = tm * BM + (k & (BM - 1)), col = tn * MC_BN + 4 * (k / BM);
  if (row >= M || col >= N) return;
  float4* dst = reinterpret_cast<float4*>((second ? S2 : S1) + (size_t)row * ldc + col);
  float4 s = *dst;
  const float4* src = reinterpret_cast<const float4*>(split_ws + (size_t)blockIdx.x * kMcSplitTileFloats) + i;
#pragma unroll 4
  for (int g = 1; g < sp.nseg; ++g, src += (size_t)sp.rest * ctas * (kMcSplitTileFloats / 4)) {
    const float4 v = ldg(src);
    s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
  }
  *dst = s;
}

// ------------------------------------------------------------------------------- diagnostic SIMT path

// Plain shared-memory tiled contraction on the CUDA cores; selected only by BSP_GEMM_SIMT=1 in
// the environment, to tell a tensor-core-path defect from a defect elsewhere.
template <bool FP8>
__global__ void __launch_bounds__(256)
gemm_simt_kernel(const void* A, const void* B, int a_fmt, int b_fmt, int64_t lda,
                 int64_t ldb, int64_t b_batch_stride, GemmParams p) {
  grid_dependency();
  __shared__ float sa[16][17], sb[16][17];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int m = blockIdx.y * 16 + ty, n = blockIdx.x * 16 + tx;
  const int b = blockIdx.z;
  const float inv_a = __fdiv_rn(1.0f, p.sa_dev ? ldg(p.sa_dev) : p.sa);
  const float inv_b = __fdiv_rn(1.0f, p.sb_dev ? ldg(p.sb_dev) : p.sb);
  float acc = 0.f;
  for (int k0 = 0; k0 < p.K; k0 += 16) {
    const int ka = k0 + tx;
    float av = 0.f, bv = 0.f;
    const int mr = blockIdx.y * 16 + ty, nr = blockIdx.x * 16 + ty;
    if (mr < p.M && ka < p.K) {
      if (FP8) {
        const uint32_t c = reinterpret_cast<const uint8_t*>(A)[p.a_mn ? (size_t)ka * lda + mr : (size_t)mr * lda + ka];
        av = a_fmt == BSP_E4M3 ? f8_decode<BSP_E4M3>(c) : f8_decode<BSP_E5M2>(c);
      } else {
        av = bf16_bits_to_float(reinterpret_cast<const uint16_t*>(A)[p.a_mn ? (size_t)ka * lda + mr : (size_t)mr * lda + ka]);
      }
    }
    if (nr < p.N && ka < p.K) {
      const size_t idx = (size_t)b * b_batch_stride + (p.b_mn ? (size_t)ka * ldb + nr : (size_t)nr * ldb + ka);
      if (FP8) {
        const uint32_t c = reinterpret_cast<const uint8_t*>(B)[idx];
        bv = b_fmt == BSP_E4M3 ? f8_decode<BSP_E4M3>(c) : f8_decode<BSP_E5M2>(c);
      } else {
        bv = bf16_bits_to_float(reinterpret_cast<const uint16_t*>(B)[idx]);
      }
    }
    sa[ty][tx] = av;
    sb[ty][tx] = bv;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k) acc = fmaf(sa[ty][k], sb[tx][k], acc);
    __syncthreads();
  }
  if (m < p.M && n < p.N) {
    const float v = acc * inv_a * inv_b;
    const size_t off = (size_t)m * p.ldc + n;
    if (p.mode == EPI_STORE_F32) {
      reinterpret_cast<float*>(p.C)[(size_t)b * p.M * p.ldc + off] = v;
    } else if (p.mode == EPI_STORE_BF16) {
      reinterpret_cast<uint16_t*>(p.C)[(size_t)b * p.M * p.ldc + off] = (uint16_t)float_to_bf16_bits(v);
    } else if (p.mode == EPI_SPLIT) {
      if (p.C) reinterpret_cast<float*>(p.C)[off] = v;
      const uint32_t hi = float_to_bf16_bits(v);
      p.split[(size_t)m * 2 * p.N + n] = (uint16_t)hi;
      p.split[(size_t)m * 2 * p.N + p.N + n] = (uint16_t)float_to_bf16_bits(v - bf16_bits_to_float(hi));
      if (p.ref) {
        const float e = p.ref[off] - v;
        const uint32_t eh = float_to_bf16_bits(e);
        p.diff[(size_t)m * p.N + n] = (uint16_t)eh;
        p.diff[(size_t)(p.M + m) * p.N + n] = (uint16_t)float_to_bf16_bits(e - bf16_bits_to_float(eh));
      }
    } else if (p.mode == EPI_MOMENTS) {
      const float f = p.moment_scale;
      p.S1[off] = fmaf(f, v, p.moment_first ? 0.f : p.S1[off]);
      p.S2[off] = fmaf(f * v, v, p.moment_first ? 0.f : p.S2[off]);
    } else {
      const float d = v - (p.ref ? p.ref[off] : 0.f);
      p.S1[off] += d;
      p.S2[off] = fmaf(d, d, p.S2[off]);
    }
  }
}

// ------------------------------------------------------------------------------- host side

// Tensor map over an operand.  K-major: matrix [batch][rows][K] (row pitch ld elements), box =
// 128 bytes of K x box_rows.  MN-major: matrix [batch][K][rows] (pitch ld), box = 128 bytes of MN x
// (128 / elem_bytes) k rows.
static int make_operand_map(CUtensorMap* map, const void* base, int elem_bytes, int64_t K, int64_t rows, int64_t ld,
                            int64_t nbatch, int64_t batch_stride_elems, int box_rows, bool mn_major = false) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return BSP_ERR_CUDA;
  const CUtensorMapDataType dt = elem_bytes == 1 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  cuuint64_t gdim[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)nbatch};
  cuuint64_t gstr[2] = {(cuuint64_t)ld * elem_bytes, (cuuint64_t)batch_stride_elems * elem_bytes};
  cuuint32_t box[3] = {(cuuint32_t)(BKB / elem_bytes), (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  const cuuint32_t rank = nbatch > 0 ? 3 : 2;
  if (mn_major) {
    gdim[0] = (cuuint64_t)rows; gdim[1] = (cuuint64_t)K;
    box[0] = (cuuint32_t)(128 / elem_bytes); box[1] = (cuuint32_t)(BKB / elem_bytes);
  }
  if (rank == 3 && nbatch == 1) gstr[1] = (cuuint64_t)gdim[1] * ld * elem_bytes;   // any valid stride
  CUresult r = fn(map, dt, rank, const_cast<void*>(base), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? BSP_OK : BSP_ERR_CUDA;
}

static bool simt_forced() {
  const char* e = getenv("BSP_GEMM_SIMT");
  return e && e[0] == '1';
}

static int device_sms() {
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
    return v;
  return kNumSMs;
}

// How a plain contraction is tiled: columns of a tile, 64 .. 256 in steps of 16 (of 32 for a pair of CTAs),
// and whether pairs take two tile rows together.  The time goes with the number of rounds the tiles take
// over the SMs times what a tile costs: per 32 bytes of K the product's bn / 2 cycles or, with every SM
// loading, the 32 bytes of each operand row at the 80 bytes per cycle and SM that fit the times
// (alone, 256 columns reach 0.83 of the tensor rate, 128 columns 0.6), and the epilogue of the last tile
// (about 12 cycles a column).  Fewer columns only where they save a twentieth (3001 x 1552 x 4112 bf16, 144 columns: 66 -> 54 us); pairs wherever they
// cost no more (16384 x 4096 x 11008 bf16: 1070 -> 954 us; 4096 x 1024 x 8192: 63 -> 55).
struct TilePlan {
  int bn;
  bool pair;
};
static TilePlan plan_tiles(int64_t M, int64_t N, int64_t k_bytes, int nsm) {
  const int64_t slices = (k_bytes + 31) / 32;
  TilePlan best = {BN, false};
  double least = 0.0;
  for (int ctas = 1; ctas <= 2; ++ctas) {
    if (ctas == 2 && M <= BM) break;
    const int64_t tm = (M + ctas * BM - 1) / (ctas * BM);
    TilePlan mine = {BN, ctas == 2};
    double cost_mine = 0.0;
    for (int bn = BN; bn >= 64; bn -= 16 * ctas) {
      const int64_t rounds = (tm * ((N + bn - 1) / bn) + nsm / ctas - 1) / (nsm / ctas);
      const double feed = 0.4 * (128 + bn / ctas), slice = bn / 2.0 > feed ? bn / 2.0 : feed;
      const double cost = (double)rounds * (double)slices * slice + 12.0 * bn;
      if (bn == BN || cost < 0.95 * cost_mine) { cost_mine = cost; mine.bn = bn; }
    }
    if (ctas == 1 || cost_mine <= least) { least = cost_mine; best = mine; }
  }
  return best;
}

// How the draws of a Monte-Carlo contraction are cut.  Costs are in pairs of draws per CTA: a pair's
// products take kblocks ring stages of about 0.27 us, and a cut adds the merge launch (about 3 us) and
// 128 KB written and read per slot.  Cuts are of at least four pairs, so that a range's start (the
// reference from memory) stays small beside its products.
static bool mc_pairs(int64_t M, int64_t k_bytes) {
  // An odd count of tile rows leaves half a pair idle: worth it when that is one in nine or fewer.  Pairs win
  // 4 to 14 % (A of 17, 34, 90 MB: 1012 -> 931 us, 1850 -> 1755, 5400 -> 4800) until A, which every pass over a
  // pair of draws reads again, is larger than L2: 180 MB, 16 draws, 8.75 ms alone and 8.9 in pairs.
  const int64_t tm = (M + BM - 1) / BM;
  return (tm % 2 == 0 || tm >= 9) && M * k_bytes <= (int64_t)120 << 20;
}
static McSplit mc_split_plan(int64_t M, int64_t N, int64_t k_bytes, int nb, int nsm) {
  const int ctas = mc_pairs(M, k_bytes) ? 2 : 1;         // CTAs per unit of the walk
  const int ntiles = (int)(((M + ctas * BM - 1) / (ctas * BM)) * ((N + MC_BN - 1) / MC_BN)), npairs = (nb + 1) / 2;
  nsm /= ctas;
  McSplit sp;
  sp.whole = ntiles / nsm * nsm;
  sp.rest = ntiles - sp.whole;
  sp.nseg = 1;
  sp.pairs_per_seg = npairs;
  sp.first = 0;
  if (sp.rest == 0) return sp;
  const double pair_us = 1.0 + 0.27 * (double)((k_bytes + BKB - 1) / BKB);
  double best = npairs * pair_us;
  for (int s = 2; s <= 32 && npairs >= 4 * s; ++s) {
    const int per = (npairs + s - 1) / s, nseg = (npairs + per - 1) / per;
    const int rounds = (sp.rest * nseg + nsm - 1) / nsm;
    const double cost = (double)rounds * per * pair_us + 3.0 + 0.05 * sp.rest * ctas * (nseg - 1) + 1.0 * (rounds - 1);
    if (cost < 0.97 * best) { best = cost; sp.nseg = nseg; sp.pairs_per_seg = per; }
  }
  return sp;
}
static size_t mc_split_bytes(const McSplit& sp, int64_t M, int64_t k_bytes) {
  return (size_t)(sp.nseg - 1) * (size_t)sp.rest * (mc_pairs(M, k_bytes) ? 2 : 1) * kMcSplitTileFloats * sizeof(float);
}
size_t gemm_mc_split_bytes(int64_t M, int64_t N, int64_t K, bool fp8, int nb) {
  if (M <= 0 || N <= 0 || K <= 0 || nb <= 0) return 0;
  const int64_t k_bytes = K * (fp8 ? 1 : 2);
  return mc_split_bytes(mc_split_plan(M, N, k_bytes, nb, device_sms()), M, k_bytes);
}

template <bool FP8, bool PAIR>
static int gemm_mc_launch(const CUtensorMap& ma, const CUtensorMap& mb, const GemmParams& p, const McSplit& sp, float* split_ws,
                          int grid, cudaStream_t st) {
  static std::atomic<bool> attr_set_dev[kMaxDevices];
  std::atomic<bool>& attr_set = attr_set_dev[device_slot()];
  if (!attr_set.load(std::memory_order_acquire)) {
    BSP_CHECK_CUDA(cudaFuncSetAttribute(gemm_mc_kernel<FP8, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMcSmem));
    attr_set.store(true, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // as launch_kernel does
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = PAIR ? 2 : 1; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kMcThreads); cfg.dynamicSmemBytes = kMcSmem; cfg.stream = st;
  cfg.attrs = attr; cfg.numAttrs = PAIR ? 2 : 1;
  BSP_CHECK_CUDA(cudaLaunchKernelEx(&cfg, gemm_mc_kernel<FP8, PAIR>, ma, mb, p, sp, split_ws));
  BSP_LAUNCH_CHECK();
  return BSP_OK;
}

template <bool FP8, int MODE, bool PAIR>
static int gemm_tc_launch_as(const CUtensorMap& ma, const CUtensorMap& mb, const GemmParams& p, int nsm, cudaStream_t st) {
  static std::atomic<bool> attr_set_dev[kMaxDevices];
  std::atomic<bool>& attr_set = attr_set_dev[device_slot()];
  if (!attr_set.load(std::memory_order_acquire)) {
    BSP_CHECK_CUDA(cudaFuncSetAttribute(gemm_tc_kernel<FP8, MODE, PAIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGemmSmem));
    attr_set.store(true, std::memory_order_release);
  }
  constexpr int ctas = PAIR ? 2 : 1;
  const int ntiles = ((p.M + ctas * BM - 1) / (ctas * BM)) * ((p.N + p.bn - 1) / p.bn);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // as launch_kernel does
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = ctas; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(ctas * (ntiles < nsm / ctas ? ntiles : nsm / ctas)));
  cfg.blockDim = dim3(kGemmThreads); cfg.dynamicSmemBytes = kGemmSmem; cfg.stream = st;
  cfg.attrs = attr; cfg.numAttrs = PAIR ? 2 : 1;
  BSP_CHECK_CUDA(cudaLaunchKernelEx(&cfg, gemm_tc_kernel<FP8, MODE, PAIR>, ma, mb, p));
  BSP_LAUNCH_CHECK();
  return BSP_OK;
}
template <bool FP8, int MODE>
static int gemm_tc_launch(const CUtensorMap& ma, const CUtensorMap& mb, const GemmParams& p, bool pair, int nsm, cudaStream_t st) {
  return pair ? gemm_tc_launch_as<FP8, MODE, true>(ma, mb, p, nsm, st) : gemm_tc_launch_as<FP8, MODE, false>(ma, mb, p, nsm, st);
}

int gemm_run(const GemmArgs& g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.nb <= 0) return BSP_OK;
  if (g.K <= 0) return BSP_ERR_ARG;
  const int eb = g.fp8 ? 1 : 2;
  if ((g.lda * eb) % 16 != 0 || (g.ldb * eb) % 16 != 0 || !aligned16(g.A) || !aligned16(g.B)) return BSP_ERR_ALIGN;
  if (g.ldc % 4 != 0 || !aligned16(g.C) || !aligned16(g.ref) || !aligned16(g.S1) || !aligned16(g.S2))
    return BSP_ERR_ALIGN;
  if ((g.b_batch_stride * eb) % 16 != 0) return BSP_ERR_ALIGN;
  GemmParams p;
  p.M = (int)g.M; p.N = (int)g.N; p.K = (int)g.K; p.nb = g.nb;
  p.a_mn = g.a_mn ? 1 : 0; p.b_mn = g.b_mn ? 1 : 0;
  p.idesc = 0u; p.idesc2 = 0u; p.bn = BN;
  if ((g.a_mn || g.b_mn) && g.mode == EPI_MC) return BSP_ERR_UNSUPPORTED;
  if (g.mode >= EPI_SPLIT && g.nb != 1) return BSP_ERR_UNSUPPORTED;
  p.sa = g.sa; p.sb = g.sb; p.sa_dev = g.sa_dev; p.sb_dev = g.sb_dev;
  p.mode = g.mode; p.C = g.C; p.ldc = g.ldc; p.ref = g.ref; p.S1 = g.S1; p.S2 = g.S2; p.diag = g.diag;
  p.split = g.split; p.diff = g.diff; p.moment_scale = g.moment_scale; p.moment_first = g.moment_first ? 1 : 0;

  if (simt_forced()) {
    dim3 grid((unsigned)((g.N + 15) / 16), (unsigned)((g.M + 15) / 16), (unsigned)g.nb);
    if (g.mode == EPI_MC && g.mc_first) {
      BSP_CHECK_CUDA(cudaMemsetAsync(g.S1, 0, (size_t)g.M * g.ldc * sizeof(float), st));
      BSP_CHECK_CUDA(cudaMemsetAsync(g.S2, 0, (size_t)g.M * g.ldc * sizeof(float), st));
    }
    // the MC epilogue is a read-modify-write: batches must run one after another
    if (g.mode == EPI_MC && g.nb > 1) {
      for (int b = 0; b < g.nb; ++b) {
        grid.z = 1;
        const void* Bb = reinterpret_cast<const uint8_t*>(g.B) + (size_t)b * g.b_batch_stride * eb;
        if (g.fp8) launch_kernel(gemm_simt_kernel<true>, grid, 256, 0, st, g.A, Bb, g.a_fmt, g.b_fmt, g.lda, g.ldb, 0, p);
        else launch_kernel(gemm_simt_kernel<false>, grid, 256, 0, st, g.A, Bb, g.a_fmt, g.b_fmt, g.lda, g.ldb, 0, p);
      }
    } else {
      if (g.fp8) launch_kernel(gemm_simt_kernel<true>, grid, 256, 0, st, g.A, g.B, g.a_fmt, g.b_fmt, g.lda, g.ldb, g.b_batch_stride, p);
      else launch_kernel(gemm_simt_kernel<false>, grid, 256, 0, st, g.A, g.B, g.a_fmt, g.b_fmt, g.lda, g.ldb, g.b_batch_stride, p);
    }
    BSP_LAUNCH_CHECK();
    return BSP_OK;
  }

  const int nsm = device_sms();
  CUtensorMap ma, mb;
  int rc = make_operand_map(&ma, g.A, eb, g.K, g.M, g.lda, 0, 0, BM, g.a_mn);
  if (rc != BSP_OK) return rc;

  if (g.mode == EPI_MC) {
    // shifted sums on chip over all draws of a tile
    if (g.N % 16 != 0 || !g.S1 || !g.S2) return BSP_ERR_ARG;
    rc = make_operand_map(&mb, g.B, eb, g.K, g.N, g.ldb, g.nb, g.b_batch_stride, MC_BN);
    if (rc != BSP_OK) return rc;
    const uint32_t fa = g.fp8 ? (g.a_fmt == BSP_E5M2 ? 1u : 0u) : 1u, fb = g.fp8 ? (g.b_fmt == BSP_E5M2 ? 1u : 0u) : 1u;
    const bool pair = mc_pairs(g.M, g.K * eb);
    const int ctas = pair ? 2 : 1;
    p.idesc = make_idesc(fa, fb, ctas * BM, MC_BN);
    p.idesc2 = make_idesc(fa, fb, ctas * BM, 2 * MC_BN);
    McSplit sp = mc_split_plan(g.M, g.N, g.K * eb, g.nb, nsm);
    sp.first = g.mc_first ? 1 : 0;
    if (!g.split_ws || g.split_ws_bytes < mc_split_bytes(sp, g.M, g.K * eb)) {      // no room: every tile takes all its draws
      sp.whole += sp.rest;
      sp.rest = 0;
      sp.nseg = 1;
    }
    const int nunits = sp.whole + sp.rest * sp.nseg, grid_mc = ctas * (nunits < nsm / ctas ? nunits : nsm / ctas);
    if (g.fp8) rc = pair ? gemm_mc_launch<true, true>(ma, mb, p, sp, g.split_ws, grid_mc, st) : gemm_mc_launch<true, false>(ma, mb, p, sp, g.split_ws, grid_mc, st);
    else rc = pair ? gemm_mc_launch<false, true>(ma, mb, p, sp, g.split_ws, grid_mc, st) : gemm_mc_launch<false, false>(ma, mb, p, sp, g.split_ws, grid_mc, st);
    if (rc != BSP_OK) return rc;
    if (sp.nseg > 1) {
      launch_kernel(gemm_mc_merge_kernel, dim3((unsigned)(sp.rest * ctas), 2 * BM * MC_BN / 4 / 256), 256, 0, st, g.split_ws, sp, ctas, p.M, p.N, p.ldc,
                    p.S1, p.S2);
      BSP_LAUNCH_CHECK();
    }
    return BSP_OK;
  }

  const TilePlan plan = plan_tiles(g.M, g.N, g.K * eb, nsm);
  const int ctas = plan.pair ? 2 : 1;
  p.bn = plan.bn;
  const uint32_t fa = g.fp8 ? (g.a_fmt == BSP_E5M2 ? 1u : 0u) : 1u, fb = g.fp8 ? (g.b_fmt == BSP_E5M2 ? 1u : 0u) : 1u;
  p.idesc = make_idesc(fa, fb, ctas * BM, (uint32_t)p.bn) | (g.a_mn ? 1u << 15 : 0u) | (g.b_mn ? 1u << 16 : 0u);   // operand major bits
  rc = make_operand_map(&mb, g.B, eb, g.K, g.N, g.ldb, g.nb, g.b_batch_stride, p.bn / ctas, g.b_mn);
  if (rc != BSP_OK) return rc;
  if (g.fp8) return g.mode == EPI_STORE_F32 ? gemm_tc_launch<true, EPI_STORE_F32>(ma, mb, p, plan.pair, nsm, st) : BSP_ERR_UNSUPPORTED;
  switch (g.mode) {
    case EPI_STORE_F32: return gemm_tc_launch<false, EPI_STORE_F32>(ma, mb, p, plan.pair, nsm, st);
    case EPI_STORE_BF16: return gemm_tc_launch<false, EPI_STORE_BF16>(ma, mb, p, plan.pair, nsm, st);
    case EPI_SPLIT: return gemm_tc_launch<false, EPI_SPLIT>(ma, mb, p, plan.pair, nsm, st);
    case EPI_MOMENTS: return gemm_tc_launch<false, EPI_MOMENTS>(ma, mb, p, plan.pair, nsm, st);
    default: return BSP_ERR_UNSUPPORTED;
  }
}

// ------------------------------------------------------------------------------- operand preparation

// codes -> bf16 (exact), same layout; sixteen codes per thread through the hardware conversions
// (bound by its 3 B per code; field by field it was bound by instructions; 180 M codes: 146 -> 95 us).
template <int FMT>
__global__ void __launch_bounds__(256)
decode_to_bf16_kernel(const uint8_t* codes, size_t n16, uint16_t* out) {
  grid_dependency();
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n16) return;
  const uint4 c = ldg(reinterpret_cast<const uint4*>(codes) + t);
  const uint2 a = f8_to_bf16x4<FMT>(c.x), b = f8_to_bf16x4<FMT>(c.y), d = f8_to_bf16x4<FMT>(c.z), e = f8_to_bf16x4<FMT>(c.w);
  uint4* dst = reinterpret_cast<uint4*>(out) + 2 * t;
  dst[0] = make_uint4(a.x, a.y, b.x, b.y);
  dst[1] = make_uint4(d.x, d.y, e.x, e.y);
}

// FP32 -> bf16, same layout.
__global__ void __launch_bounds__(256)
to_bf16_kernel(const float* in, size_t n8, uint16_t* out) {
  grid_dependency();
  const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n8) return;
  const float4 a = ldg(reinterpret_cast<const float4*>(in) + 2 * t), b = ldg(reinterpret_cast<const float4*>(in) + 2 * t + 1);
  reinterpret_cast<uint4*>(out)[t] =
      make_uint4(float_to_bf16_bits(a.x) | (float_to_bf16_bits(a.y) << 16), float_to_bf16_bits(a.z) | (float_to_bf16_bits(a.w) << 16),
                 float_to_bf16_bits(b.x) | (float_to_bf16_bits(b.y) << 16), float_to_bf16_bits(b.z) | (float_to_bf16_bits(b.w) << 16));
}

// out[c*ld_out + r] = bf16(in[r*cols + c]); 32 x 32 tiles.
template <int DT>
__global__ void __launch_bounds__(256)
to_bf16_transpose_kernel(const void* in, int64_t rows, int64_t cols, uint16_t* out,
                         int64_t ld_out) {
  grid_dependency();
  __shared__ uint16_t tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t r0 = (int64_t)blockIdx.y * 32, c0 = (int64_t)blockIdx.x * 32;
  for (int i = ty; i < 32; i += 8) {
    const int64_t r = r0 + i, c = c0 + tx;
    tile[i][tx] = (r < rows && c < cols) ? (uint16_t)float_to_bf16_bits(load1<DT>(in, (size_t)r * cols + c)) : 0;
  }
  __syncthreads();
  for (int i = ty; i < 32; i += 8) {
    const int64_t c = c0 + i, r = r0 + tx;
    if (c < cols && r < ld_out) out[(size_t)c * ld_out + r] = r < rows ? tile[tx][i] : 0;
  }
}

static bool valid_enum(int v, int hi) { return v >= 0 && v <= hi; }

}  // namespace bsp

using namespace bsp;

extern "C" {

size_t bsp_linear_wgrad_workspace_bytes(int64_t T, int64_t O, int64_t C, int x_read) {
  (void)C;
  if (T <= 0 || O <= 0) return 0;
  if (x_read != BSP_READ_ORIGINAL) return 256;
  return round_up((size_t)O * round_up((size_t)T, 16) * 2, 256);
}

int bsp_linear_wgrad(int64_t T, int64_t O, int64_t C, const uint8_t* dy_codes_t, bsp_quant_t q_dy, int x_read,
                     const void* x_t, bsp_quant_t q_x, int64_t ld_t, float* dW, const float* mc_ref, float* mc_S1,
                     float* mc_S2, void* ws, size_t ws_bytes, bsp_diag_t* diag, void* stream) {
  if (T < 0 || O < 0 || C < 0 || !valid_enum(x_read, 2) || !valid_enum(q_dy.fmt, 1) || !valid_enum(q_x.fmt, 1))
    return BSP_ERR_ARG;
  if (O == 0 || C == 0) return BSP_OK;
  const bool mc = mc_ref != nullptr;
  if (mc ? (!mc_S1 || !mc_S2) : !dW) return BSP_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (T == 0) {
    if (!mc) BSP_CHECK_CUDA(cudaMemsetAsync(dW, 0, (size_t)O * C * sizeof(float), st));
    return BSP_OK;
  }
  if (!dy_codes_t || !x_t) return BSP_ERR_ARG;
  if (ld_t < T || ld_t % 16 != 0 || C % 4 != 0) return BSP_ERR_ALIGN;
  GemmArgs g;
  g.M = O; g.N = C; g.K = T; g.nb = 1;
  g.lda = ld_t; g.ldb = ld_t; g.b_batch_stride = (int64_t)C * ld_t;
  g.sa = q_dy.scale; g.sa_dev = q_dy.scale_dev; g.sb = q_x.scale; g.sb_dev = q_x.scale_dev;
  g.mode = mc ? EPI_MC : EPI_STORE_F32;
  g.C = dW; g.ldc = C; g.ref = mc_ref; g.S1 = mc_S1; g.S2 = mc_S2; g.diag = diag;
  if (x_read == BSP_READ_ORIGINAL) {
    // BF16 contraction: decode dY's codes to bf16 (exact) into the workspace; x_t is bf16 already
    const size_t need = bsp_linear_wgrad_workspace_bytes(T, O, C, x_read);
    if (!ws || ws_bytes < need || (reinterpret_cast<uintptr_t>(ws) & 255u)) return BSP_ERR_WORKSPACE;
    const size_t n16 = (size_t)O * ld_t / 16;
    uint16_t* dyb = reinterpret_cast<uint16_t*>(ws);
    if (q_dy.fmt == BSP_E5M2)
      launch_kernel(decode_to_bf16_kernel<BSP_E5M2>, (unsigned)((n16 + 255) / 256), 256, 0, st, dy_codes_t, n16, dyb);
    else
      launch_kernel(decode_to_bf16_kernel<BSP_E4M3>, (unsigned)((n16 + 255) / 256), 256, 0, st, dy_codes_t, n16, dyb);
    BSP_LAUNCH_CHECK();
    g.fp8 = false; g.A = dyb; g.B = x_t; g.a_fmt = 0; g.b_fmt = 0;
    g.sb = 1.0f; g.sb_dev = nullptr;          // the original is unscaled
  } else {
    g.fp8 = true; g.A = dy_codes_t; g.B = x_t; g.a_fmt = q_dy.fmt; g.b_fmt = q_x.fmt;
  }
  return gemm_run(g, st);
}

int bsp_gemm(int64_t M, int64_t N, int64_t K, int elem, const void* A, int64_t lda, int a_mn, int a_fmt,
             const void* B, int64_t ldb, int b_mn, int b_fmt, float alpha, float* C, int64_t ldc, bsp_diag_t* diag,
             void* stream) {
  if (M < 0 || N < 0 || K <= 0 || (elem != 1 && elem != 2) || !valid_enum(a_fmt, 1) || !valid_enum(b_fmt, 1))
    return BSP_ERR_ARG;
  if (M == 0 || N == 0) return BSP_OK;
  if (!A || !B || !C || alpha == 0.f) return BSP_ERR_ARG;
  GemmArgs g;
  g.M = M; g.N = N; g.K = K; g.nb = 1; g.fp8 = elem == 1; g.a_fmt = a_fmt; g.b_fmt = b_fmt;
  g.A = A; g.B = B; g.a_mn = a_mn != 0; g.b_mn = b_mn != 0; g.lda = lda; g.ldb = ldb;
  g.b_batch_stride = (b_mn ? K : N) * ldb;
  g.sa = 1.0f / alpha; g.sb = 1.0f; g.mode = EPI_STORE_F32; g.C = C; g.ldc = ldc; g.diag = diag;
  return gemm_run(g, (cudaStream_t)stream);
}

int bsp_linear_wgrad_mc(int64_t T, int64_t O, int64_t C, const uint8_t* dy_codes_t, bsp_quant_t q_dy,
                        const uint8_t* x_t_draws, bsp_quant_t q_x, int64_t ld_t, int n_draws, const float* g_ref,
                        float* S1, float* S2, bsp_diag_t* diag, void* stream) {
  return bsp::linear_wgrad_mc_run(T, O, C, dy_codes_t, q_dy, x_t_draws, q_x, ld_t, n_draws, g_ref, S1, S2, false, nullptr,
                                  0, diag, stream);
}

}  // extern "C"

// The same with room for split ranges of draws (gemm_mc_split_bytes).
int bsp::linear_wgrad_mc_run(int64_t T, int64_t O, int64_t C, const uint8_t* dy_codes_t, bsp_quant_t q_dy,
                             const uint8_t* x_t_draws, bsp_quant_t q_x, int64_t ld_t, int n_draws, const float* g_ref,
                             float* S1, float* S2, bool first, float* split_ws, size_t split_ws_bytes, bsp_diag_t* diag, void* stream) {
  if (T < 0 || O < 0 || C < 0 || n_draws < 0 || !valid_enum(q_dy.fmt, 1) || !valid_enum(q_x.fmt, 1)) return BSP_ERR_ARG;
  if (O == 0 || C == 0 || n_draws == 0) return BSP_OK;
  if (!g_ref || !S1 || !S2) return BSP_ERR_ARG;
  if (T == 0) return BSP_ERR_UNSUPPORTED;       // every draw would add (0 - ref): not a case the check produces
  if (!dy_codes_t || !x_t_draws) return BSP_ERR_ARG;
  if (ld_t < T || ld_t % 16 != 0 || C % 16 != 0) return BSP_ERR_ALIGN;
  GemmArgs g;
  g.M = O; g.N = C; g.K = T; g.nb = n_draws; g.fp8 = true;
  g.A = dy_codes_t; g.B = x_t_draws; g.a_fmt = q_dy.fmt; g.b_fmt = q_x.fmt;
  g.lda = ld_t; g.ldb = ld_t; g.b_batch_stride = (int64_t)C * ld_t;
  g.sa = q_dy.scale; g.sa_dev = q_dy.scale_dev; g.sb = q_x.scale; g.sb_dev = q_x.scale_dev;
  g.mode = EPI_MC; g.C = nullptr; g.ldc = C; g.ref = g_ref; g.S1 = S1; g.S2 = S2; g.diag = diag;
  g.mc_first = first; g.split_ws = split_ws; g.split_ws_bytes = split_ws_bytes;
  return gemm_run(g, (cudaStream_t)stream);
}

extern "C" {

size_t bsp_linear_dgrad_workspace_bytes(int64_t T, int64_t O, int64_t C) {
  if (T <= 0 || O <= 0 || C <= 0) return 0;
  const size_t ldo = round_up((size_t)O, 16);
  return round_up((size_t)T * ldo * 2, 256) + round_up((size_t)C * ldo * 2, 256);
}

int bsp_linear_dgrad(int64_t T, int64_t O, int64_t C, const uint8_t* dy_codes, bsp_quant_t q_dy, const void* W,
                     int w_dt, void* du, int du_dt, void* ws, size_t ws_bytes, bsp_diag_t* diag, void* stream) {
  if (T < 0 || O <= 0 || C < 0 || !valid_enum(q_dy.fmt, 1) || !valid_enum(w_dt, 1) || !valid_enum(du_dt, 1))
    return BSP_ERR_ARG;
  if (T == 0 || C == 0) return BSP_OK;
  if (!dy_codes || !W || !du) return BSP_ERR_ARG;
  if (O % 16 != 0 || C % 4 != 0) return BSP_ERR_UNSUPPORTED;
  if (!ws || ws_bytes < bsp_linear_dgrad_workspace_bytes(T, O, C) || (reinterpret_cast<uintptr_t>(ws) & 255u))
    return BSP_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  uint16_t* dyb = reinterpret_cast<uint16_t*>(ws);             // (bsp_mc_check reads it here afterwards)
  uint16_t* wt = reinterpret_cast<uint16_t*>(reinterpret_cast<char*>(ws) + round_up((size_t)T * O * 2, 256));
  const size_t n16 = (size_t)T * O / 16;
  if (q_dy.fmt == BSP_E5M2)
    launch_kernel(decode_to_bf16_kernel<BSP_E5M2>, (unsigned)((n16 + 255) / 256), 256, 0, st, dy_codes, n16, dyb);
  else
    launch_kernel(decode_to_bf16_kernel<BSP_E4M3>, (unsigned)((n16 + 255) / 256), 256, 0, st, dy_codes, n16, dyb);
  BSP_LAUNCH_CHECK();
  // W [O][C] is the B operand with the contraction index outermost and is read as it lies (MN-major): a
  // bf16 W in place, an FP32 W from a bf16 copy of the same layout (a transposed copy, a quarter of the
  // speed at 4112 x 1552: 21 us against 7, is left for a C that breaks the 16-byte pitch)
  const bool pitch_ok = C % 8 == 0 && aligned16(W), w_in_place = pitch_ok && w_dt == BSP_BF16;
  if (pitch_ok && !w_in_place) {
    const size_t n8 = (size_t)O * C / 8;
    launch_kernel(to_bf16_kernel, (unsigned)((n8 + 255) / 256), 256, 0, st, reinterpret_cast<const float*>(W), n8, wt);
    BSP_LAUNCH_CHECK();
  } else if (!pitch_ok) {
    dim3 tg((unsigned)((C + 31) / 32), (unsigned)((O + 31) / 32));
    if (w_dt == BSP_F32) launch_kernel(to_bf16_transpose_kernel<BSP_F32>, tg, 256, 0, st, W, O, C, wt, O);
    else launch_kernel(to_bf16_transpose_kernel<BSP_BF16>, tg, 256, 0, st, W, O, C, wt, O);
    BSP_LAUNCH_CHECK();
  }
  GemmArgs g;
  g.M = T; g.N = C; g.K = O; g.nb = 1; g.fp8 = false; g.a_fmt = 0; g.b_fmt = 0;
  g.A = dyb; g.lda = O;
  if (pitch_ok) { g.B = w_in_place ? W : wt; g.b_mn = true; g.ldb = C; g.b_batch_stride = (int64_t)O * C; }
  else { g.B = wt; g.ldb = O; g.b_batch_stride = (int64_t)C * O; }
  g.sa = q_dy.scale; g.sa_dev = q_dy.scale_dev; g.sb = 1.0f; g.sb_dev = nullptr;
  g.mode = du_dt == BSP_F32 ? EPI_STORE_F32 : EPI_STORE_BF16;
  g.C = du; g.ldc = C; g.ref = nullptr; g.S1 = nullptr; g.S2 = nullptr; g.diag = diag;
  return gemm_run(g, st);
}

}  // extern "C"
