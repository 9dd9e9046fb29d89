// The rounded-probability averages on the tensor cores, for rows of up to 128 entries and 64 value
// columns.  A draw of a row needs h = V^T p_q, dp = V h and two outer products with h: per row and draw
// 4 n d multiply-adds, which on the CUDA cores ran at a quarter of the FP32 rate (V and h from shared
// memory for every draw: 16384 rows of 128 x 64, 256 draws, 14.7 ms; here 4.06).  Here the draws of a row are
// the M dimension of small contractions.
//
// Everything a draw rounds is two-valued: p_q = lo + s q with a bit q per entry (s = param for the grid,
// 2 param for the +-param law), likewise a and b.  The bits enter the products as exact bf16 0 / 1 and
// the FP32 factors as three bf16 terms:
//   H   = bits V            128 slots x 64, for the bits of p_q, a and b        3 x 3 products
//   delta = s H_q + V^T (lo - p),  h = V^T p + delta  (p_q's; a's and b's likewise), and with them the
//           dot products x . dp = (V^T x) . h of the operators, one thread per slot
//   dp^T = V (V^T p) + V delta^T    128 entries x 128 slots, delta in three terms   6 products
//   sum_k q delta^T, sum_k a delta^T  per row, 128 entries x 64 each, over the row's slots
// V's terms are multiples of 2^-8, 2^-17 and 2^-26 of its column's scale, nine bits each, so the first term's
// sums (one accumulator) and the other two's (another) are integers below 2^24 of their unit: H is exact for this V.
// That matters because tensor-core accumulation truncates: a truncated H is off to one side in every draw, and such
// an error, unlike a rounded one, survives the average over the draws.  An entry of V is held to 2^-27 of its
// column's scale, which is FP32's own precision for entries of at least an eighth of it and less below; for a V whose
// rows differ by more than that bears (probs_wide) the kernel forms the sums in FP32 (probs_fp32_rows).
// Summing against delta = h - V^T p, whose mean over the draws is zero, rather than against h keeps the
// sums as small as their results: sum (p - p_q) h^T = -w (V^T p)^T + (p - lo) (sum delta)^T - s sum q delta^T
// with the scalar w_j = sum_k (p_q - p)_j known from the count of up-roundings.
// Against 64-bit arithmetic, 128 x 64, 256 draws, grid 1/64: the operators' sums are off by 0.8 - 2.7e-7 (the FP32
// kernel: 2.3 - 3.8e-7), their squares by 0.4 - 0.8e-7 (2.0 - 2.7e-7), the gradient-of-V sums by 1.3 - 1.7e-7 (2.2 - 3.4e-7).
//
// A block keeps V's terms in shared memory and walks groups of rows: sixteen warps compute, one issues the
// products.  A tile is 128 slots: one row's 128 draws, or two rows' 64.  Per tile: the generator (three streams)
// under the H products of the stream before, the slot pass, the dp and outer products, and the entry pass, in
// which a thread owns an entry and walks 32 slots (the five operators' errors and their squares, in packed
// FP32 pairs of slots).  Of a tile's 32 thousand cycles at 128 draws and two tiles a row, the generator and
// the bits take 14, the entry pass 6, the slot pass 3, waits for products 4, and the row's start and end 7:
// no unit is full (issue slots 48 %, the generator's multiplier 45 %, tensor pipe 15 %), the phases following one
// another with four warps per scheduler; a second set of bit matrices, to overlap them, does not fit.
#pragma once

#include "common.cuh"
#include "tc.cuh"

namespace bsp {

constexpr int kPtWorkers = 512, kPtThreads = kPtWorkers + 128, kPtN = 128, kPtD = 64, kPtSlots = 128, kPtVals = 10;
constexpr uint32_t kPtCodePitch = kPtSlots + 4;               // codes are [entry][slot]: neighbouring entries on neighbouring banks
constexpr int kPtSegment = 256;
constexpr uint32_t kPtMat = 32768, kPtTerm = 16384;           // a bit matrix (two halves of 64 entries); one bf16 term
constexpr uint32_t kPtBits = 0, kPtV = 3 * kPtMat, kPtDelta = kPtV + 3 * kPtTerm, kPtCodes = kPtDelta + 3 * kPtTerm,
                   kPtDots = kPtCodes + kPtN * kPtCodePitch,  // float [4][128]: minus p.dp, (p_q - p).dp, (a - p).dp, (b - p).dp
                   kPtDotPart = kPtDots + kPtSlots * 16,      // float4 [4][128]
                   kPtSumA = kPtDotPart + 4 * kPtSlots * 16,  // float [128]: 1^T a - 1
                   kPtP = kPtSumA + kPtSlots * 4,             // float [2][128]
                   kPtX = kPtP + 2 * kPtN * 4,                // float [2][128]: lo, then V (V^T p), then w
                   kPtHp = kPtX + 2 * kPtN * 4,               // float [2][64]: V^T p
                   kPtHl = kPtHp + 2 * kPtD * 4,              // float [2][64]: V^T (lo - p)
                   kPtSd = kPtHl + 2 * kPtD * 4,              // float [4][64]: sums of delta, per 32 slots
                   kPtThr = kPtSd + 4 * kPtD * 4,             // uint32 [2][128]: the thresholds
                   kPtBar = kPtThr + 2 * kPtN * 4, kPtEnd = kPtBar + 96;
constexpr size_t kPtSmemBytes = kPtEnd + 1024;
static_assert(kPtSmemBytes <= 232448, "shared memory of the tensor-core probability kernel");
// scratch over the delta terms: column partials double2 [2][2][16][32] at a group's start, at its end partial
// sums [4][10][128], counts [2][16][32] words of four entries each, and the counts per row [2][2][128]
constexpr uint32_t kPtCnt4 = 4 * kPtVals * kPtN * 4, kPtCnt = kPtCnt4 + 2 * 16 * 32 * 4;
static_assert(kPtCnt + 2 * 2 * kPtN * 4 <= 3 * kPtTerm && 2 * 2 * 16 * 32 * 16 <= 3 * kPtTerm, "scratch over the delta terms");
// tensor memory columns: H (two accumulators per stream), over it dp^T and the second row's sums once the
// slot pass has read it, and the first row's sums, which live through all tiles of a row
constexpr uint32_t kPtTmH = 0, kPtTmDp = 0, kPtTmAcc1 = 128, kPtTmAcc0 = 384;

// Two FP32 values in one 64-bit register pair, for the packed instructions.
__device__ __forceinline__ uint64_t f2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_get(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Two FP32 values as three bf16 terms each, a term's two in one word.
__device__ __forceinline__ void bf16_split3(float a, float b, uint32_t (&t)[3]) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(t[i]) : "f"(b), "f"(a));
    a -= __uint_as_float(t[i] << 16);
    b -= __uint_as_float(t[i] & 0xFFFF0000u);
  }
}

// Whether V's rows differ too widely in size for terms of fixed position: the smallest of the rows' largest
// magnitudes (rows of zeros aside) below a sixteenth of the power of two above V's largest, or V not finite.  A row of
// probabilities may lie on the smallest row alone, and then the error of h is 2^-27 of the largest over the
// smallest.  The line lies where the two forms cross: relative errors of the operators' sums, of their squares and of
// the gradient-of-V sums against 64 bits, the worst of twelve rows, with one row of V scaled up and unlikely, fixed
// terms and FP32: x 6 3.4, 3.4, 1.4e-7 and 3.8, 2.6, 2.1e-7; x 100 1.7, 3.9, 0.8e-6 and 1.6, 0.8, 0.2e-6; x 1000 1.1, 2.2,
// 1.0e-5 and 2.1, 0.2, 0.2e-6.  Scaled down and all but certain: 1/8 0.6, 1.1, 1.2e-6 and 1.3, 1.2, 1.2e-6; 1/32 1.5, 4.0,
// 0.5e-6 and 1.9, 2.1, 0.9e-6; 1/1000 0.9, 1.0, 0.2e-4 and 1.8, 1.5, 1.5e-6.
// Also the largest magnitude of each column, to col_max ([64] words).  The kernel's whole block; found is two words.
__device__ __forceinline__ bool probs_wide(const float* V, int n, int d, uint32_t* found, uint32_t* col_max) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr int kWarps = kPtThreads / 32, kRows = (kPtN + kWarps - 1) / kWarps;
  if (threadIdx.x < kPtD) col_max[threadIdx.x] = 0u;
  if (threadIdx.x == 0) { found[0] = 0u; found[1] = 0xFFFFFFFFu; }
  uint32_t v[kRows][2];                                               // d <= 64: two columns a lane
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
    const int j = w + kWarps * i;
    v[i][0] = j < n && lane < d ? __float_as_uint(ldg(V + (size_t)j * d + lane)) & 0x7FFFFFFFu : 0u;
    v[i][1] = j < n && lane + 32 < d ? __float_as_uint(ldg(V + (size_t)j * d + lane + 32)) & 0x7FFFFFFFu : 0u;
  }
  __syncthreads();
  uint32_t c0 = 0u, c1 = 0u, most = 0u, least = 0xFFFFFFFFu;
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
    c0 = max(c0, v[i][0]);
    c1 = max(c1, v[i][1]);
    const uint32_t row = __reduce_max_sync(0xFFFFFFFFu, max(v[i][0], v[i][1]));
    most = max(most, row);
    if (row) least = min(least, row);
  }
  if (lane < d) atomicMax(&col_max[lane], c0);
  if (lane + 32 < d) atomicMax(&col_max[lane + 32], c1);
  if (lane == 0) { atomicMax(&found[0], most); atomicMin(&found[1], least); }
  __syncthreads();
  most = found[0]; least = found[1];
  if (most == 0u) return false;
  if (most >= 0x7F800000u) return true;
  int ex;
  frexpf(__uint_as_float(most), &ex);                                 // most < 2^ex
  return scalbnf(__uint_as_float(least), 4 - ex) < 1.f;
}
// Where an entry sits between its two rounded values (law 0: the uniform grid; law 1: +-param).
// Up iff the word is below thr (law 0) or above it (law 1: its top bit is set).
__device__ __forceinline__ void probs_cell(float p, int law, float param, float& lo, float& hi, uint32_t& thr) {
  if (law == 1) { lo = p - param; hi = p + param; thr = 0x7FFFFFFFu; return; }
  const float t = __fdiv_rn(p, param), n0 = floorf(t);
  lo = n0 * param; hi = (n0 + 1.f) * param;
  thr = __float2uint_rd(__fsub_rn(t, n0) * 4294967296.0f);
}

// Barriers of the worker warps alone; the second carries their common verdict on a wait.
__device__ __forceinline__ void pt_sync() { asm volatile("barrier.cta.sync.aligned 1, %0;" ::"n"(kPtWorkers) : "memory"); }
__device__ __forceinline__ bool pt_sync_and(bool ok) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.and.aligned.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(r) : "r"((uint32_t)ok), "n"(kPtWorkers) : "memory");
  return r != 0;
}
// A worker warp's shared-memory writes and tensor-memory reads are done as far as the products go.
__device__ __forceinline__ void pt_arrive(uint32_t bar, int lane) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive(bar);
}

// The sums in FP32 on the CUDA cores, for few draws (probs.cu) and for a V that terms of fixed position do not hold
// (probs_wide).  The whole block; sixteen draws of a row at a time.  Phase 1, a warp per draw: a lane owns four consecutive entries, one
// generator block per stream; h = V^T p_q with the lane owning two columns, dp = V h from a transposed copy of V;
// the dot products are warp sums.  Phase 2, a thread per entry and quarter of the columns: adds the draws to its
// sums.  4096 rows, 32 draws: 128 x 64 662 us (probs_mc_128x64_kernel 663), 64 x 64 523 (probs_mc_kernel 771), 100 x 16
// 367 (1278), 16 x 16 257 (299).
constexpr int kPwDraws = 16;
constexpr size_t kPwFloats = (size_t)2 * kPtN * kPtD + kPwDraws * (3 * kPtN /*pq, eu, ea*/ + kPtD /*h*/ + 5 * kPtN /*err*/);
static_assert(kPwFloats * sizeof(float) <= kPtEnd, "the FP32 form's shared memory");
template <int law>
__device__ __forceinline__ void probs_fp32_rows(float* sm, const float* p_all, const float* V, int n, int d, float param,
                                                PhiloxKey kq, int draw0, int K, float* ds_sum, float* ds_sq, float* dV_sum,
                                                size_t rows) {
  float* Vs = sm;                                                     // [128][64]
  float* Vt = Vs + kPtN * kPtD;                                       // [64][128]
  float* pq_s = Vt + kPtN * kPtD;                                     // [16][128]
  float* eu_s = pq_s + kPwDraws * kPtN;                               // [16][128]: p - p_q
  float* ea_s = eu_s + kPwDraws * kPtN;                               // [16][128]: a - p_q
  float* h_s = ea_s + kPwDraws * kPtN;                                // [16][64]
  float* err_s = h_s + kPwDraws * kPtD;                               // [16][5][128]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  __syncthreads();
  for (int i = tid; i < kPtN * kPtD; i += kPtThreads) {
    const int j = i >> 6, c = i & (kPtD - 1);
    const float v = j < n && c < d ? ldg(V + (size_t)j * d + c) : 0.f;
    Vs[i] = v;
    Vt[c * kPtN + j] = v;
  }
  const int j2 = tid & (kPtN - 1), hh = tid >> 7;                     // phase 2: entry, quarter (the fifth is idle)
  const int op0 = hh == 0 ? 0 : hh + 1, nops = hh == 0 ? 2 : 1;       // its operators: two in the first, one in the others
  const bool on = 4 * lane < n, on2 = hh < 4 && j2 < n;
  const uint32_t c3 = kq.c3 & ~0xFFu;
  __syncthreads();
  for (size_t row = blockIdx.x; row < rows; row += gridDim.x) {
    float pv[4], lo[4], hi[4];
    uint32_t thr[4];
    double sum_p = 0.0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      pv[e] = lo[e] = hi[e] = 0.f;
      thr[e] = 0u;                                                    // an entry that is not there stays zero either way
      if (on) {
        pv[e] = ldg(p_all + row * n + 4 * lane + e);
        probs_cell(pv[e], law, param, lo[e], hi[e], thr[e]);
      }
      sum_p += (double)pv[e];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum_p += __shfl_xor_sync(0xFFFFFFFFu, sum_p, o);
    const float sum_p_m1 = (float)(sum_p - 1.0);
    const uint64_t q = (row * (uint64_t)n) / 4 + (uint64_t)lane;
    float acc_u[16], acc_a[16], acc_s[2] = {0.f, 0.f}, acc_q[2] = {0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 16; ++c) acc_u[c] = acc_a[c] = 0.f;
    for (int k0 = 0; k0 < K; k0 += kPwDraws) {
      const int nd = K - k0 < kPwDraws ? K - k0 : kPwDraws;
      if (w < nd) {
        float pq[4], a[4], b[4];
        auto draw = [&](uint32_t stream, float (&x)[4]) {
          const uint4 r = philox4x32_10((uint32_t)q, (uint32_t)(q >> 32), (uint32_t)(draw0 + k0 + w), c3 | stream, kq.k0, kq.k1);
          const uint32_t u[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) x[e] = (law == 1 ? u[e] > thr[e] : u[e] < thr[e]) ? hi[e] : lo[e];
        };
        draw(0u, pq); draw(1u, a); draw(2u, b);
        float* pqw = pq_s + w * kPtN;
        *reinterpret_cast<float4*>(pqw + 4 * lane) = make_float4(pq[0], pq[1], pq[2], pq[3]);
        __syncwarp();
        float h0 = 0.f, h1 = 0.f, g0 = 0.f, g1 = 0.f;
#pragma unroll 2
        for (int j = 0; j < n; j += 4) {
          const float4 x = *reinterpret_cast<const float4*>(pqw + j);
          const float2* v = reinterpret_cast<const float2*>(Vs + j * kPtD) + lane;
          const float2 v0 = v[0], v1 = v[kPtD / 2], v2 = v[kPtD], v3 = v[3 * kPtD / 2];
          h0 = fmaf(v0.x, x.x, h0); h1 = fmaf(v0.y, x.x, h1);
          g0 = fmaf(v1.x, x.y, g0); g1 = fmaf(v1.y, x.y, g1);
          h0 = fmaf(v2.x, x.z, h0); h1 = fmaf(v2.y, x.z, h1);
          g0 = fmaf(v3.x, x.w, g0); g1 = fmaf(v3.y, x.w, g1);
        }
        float* hw = h_s + w * kPtD;
        *reinterpret_cast<float2*>(hw + 2 * lane) = make_float2(h0 + g0, h1 + g1);
        __syncwarp();
        float dp[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
        for (int c = 0; c < d; ++c) {
          const float hv = hw[c];
          const float4 t = *reinterpret_cast<const float4*>(Vt + c * kPtN + 4 * lane);
          dp[0] = fmaf(t.x, hv, dp[0]); dp[1] = fmaf(t.y, hv, dp[1]); dp[2] = fmaf(t.z, hv, dp[2]); dp[3] = fmaf(t.w, hv, dp[3]);
        }
        float dots[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          dots[0] = fmaf(pv[e], dp[e], dots[0]);
          dots[1] = fmaf(pq[e] - pv[e], dp[e], dots[1]);
          dots[2] = fmaf(a[e] - pv[e], dp[e], dots[2]);
          dots[3] = fmaf(b[e] - pv[e], dp[e], dots[3]);
          dots[4] += a[e] - pv[e];
        }
#pragma unroll
        for (int i = 0; i < 5; ++i) dots[i] = warp_sum(dots[i]);
        float er[5][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {                                 // as in the entry pass below
          const float c = dp[e] - dots[0], dq = pq[e] - pv[e], da = a[e] - pv[e], db = b[e] - pv[e];
          er[0][e] = dq * c - pq[e] * dots[1];
          er[1][e] = da * c - a[e] * dots[2];
          er[2][e] = a[e] * (dots[4] + sum_p_m1) * dp[e] + er[1][e];
          er[3][e] = 0.5f * ((da + db) * c - (a[e] * dots[3] + b[e] * dots[2]));
          er[4][e] = 0.5f * ((dq + db) * c - (pq[e] * dots[3] + b[e] * dots[1]));
        }
#pragma unroll
        for (int o = 0; o < 5; ++o)
          *reinterpret_cast<float4*>(err_s + (w * 5 + o) * kPtN + 4 * lane) = make_float4(er[o][0], er[o][1], er[o][2], er[o][3]);
        *reinterpret_cast<float4*>(eu_s + w * kPtN + 4 * lane) = make_float4(pv[0] - pq[0], pv[1] - pq[1], pv[2] - pq[2], pv[3] - pq[3]);
        *reinterpret_cast<float4*>(ea_s + w * kPtN + 4 * lane) = make_float4(a[0] - pq[0], a[1] - pq[1], a[2] - pq[2], a[3] - pq[3]);
      }
      __syncthreads();
      if (on2)
        for (int k = 0; k < nd; ++k) {
          const float eu = eu_s[k * kPtN + j2], ea = ea_s[k * kPtN + j2];
          if (16 * hh < d)
#pragma unroll
            for (int c = 0; c < 16; c += 4) {
              const float4 hv = *reinterpret_cast<const float4*>(h_s + k * kPtD + 16 * hh + c);
              acc_u[c] = fmaf(eu, hv.x, acc_u[c]); acc_u[c + 1] = fmaf(eu, hv.y, acc_u[c + 1]);
              acc_u[c + 2] = fmaf(eu, hv.z, acc_u[c + 2]); acc_u[c + 3] = fmaf(eu, hv.w, acc_u[c + 3]);
              acc_a[c] = fmaf(ea, hv.x, acc_a[c]); acc_a[c + 1] = fmaf(ea, hv.y, acc_a[c + 1]);
              acc_a[c + 2] = fmaf(ea, hv.z, acc_a[c + 2]); acc_a[c + 3] = fmaf(ea, hv.w, acc_a[c + 3]);
            }
#pragma unroll
          for (int i = 0; i < 2; ++i)
            if (i < nops) {
              const float v = err_s[(k * 5 + op0 + i) * kPtN + j2];
              acc_s[i] += v;
              acc_q[i] = fmaf(v, v, acc_q[i]);
            }
        }
      __syncthreads();
    }
    if (on2) {
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (i < nops) {
          const size_t at = ((size_t)(op0 + i) * rows + row) * n + j2;
          ds_sum[at] = acc_s[i];
          if (ds_sq) ds_sq[at] = acc_q[i];
        }
      float* o_u = dV_sum + (row * (size_t)n + j2) * d + 16 * hh;
      float* o_a = o_u + rows * (size_t)n * d;
#pragma unroll
      for (int c = 0; c < 16; c += 4) {
        if (16 * hh + c >= d) break;
        if ((d & 3) == 0) {
          *reinterpret_cast<float4*>(o_u + c) = make_float4(acc_u[c], acc_u[c + 1], acc_u[c + 2], acc_u[c + 3]);
          *reinterpret_cast<float4*>(o_a + c) = make_float4(acc_a[c], acc_a[c + 1], acc_a[c + 2], acc_a[c + 3]);
        } else {
#pragma unroll
          for (int e = c; e < c + 4; ++e)
            if (16 * hh + e < d) { o_u[e] = acc_u[e]; o_a[e] = acc_a[e]; }
        }
      }
    }
  }
}

template <int law>
__global__ void __launch_bounds__(kPtThreads, 1)
probs_mc_tc_kernel(const float* p_all, const float* V, int n, int d, float param,
                   PhiloxKey kq, int draw0, int K_all, int g /* slots per row: 64 or 128 */, float* ds_sum,
                   float* ds_sq, float* dV_sum, size_t rows, bool few /* draws: the FP32 form */,
                   size_t stop /* groups from here on are left undone (self-test) */) {
  grid_dependency();
  extern __shared__ uint8_t pt_raw[];
  const uint32_t raw = smem_u32(pt_raw), base = (raw + 1023u) & ~1023u;
  uint8_t* sm = pt_raw + (base - raw);
  float* dots_s = reinterpret_cast<float*>(sm + kPtDots);
  float4* dotp_s = reinterpret_cast<float4*>(sm + kPtDotPart);
  float* suma_s = reinterpret_cast<float*>(sm + kPtSumA);
  float* p_s = reinterpret_cast<float*>(sm + kPtP);
  float* x_s = reinterpret_cast<float*>(sm + kPtX);
  float* hp_s = reinterpret_cast<float*>(sm + kPtHp);
  float* hl_s = reinterpret_cast<float*>(sm + kPtHl);
  float* sd_s = reinterpret_cast<float*>(sm + kPtSd);
  uint32_t* thr_s = reinterpret_cast<uint32_t*>(sm + kPtThr);
  float* comb_s = reinterpret_cast<float*>(sm + kPtDelta);
  // bits of stream m written (0..2), delta written (3); H complete, dp^T complete, the row sums complete
  const uint32_t bar_go = base + kPtBar, bar_h = bar_go + 32, bar_d = bar_go + 40, bar_v = bar_go + 48;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sm + kPtBar + 56);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + kPtBar + 60);
  double* sumlo_s = reinterpret_cast<double*>(sm + kPtBar + 64);      // [2]: sum of lo - 1
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, wq = w & 3, wg = w >> 2;

  if (few) {
    probs_fp32_rows<law>(reinterpret_cast<float*>(sm), p_all, V, n, d, param, kq, draw0, K_all, ds_sum, ds_sq, dV_sum, rows);
    return;
  }
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) mbar_init(bar_go + 8 * i, kPtWorkers / 32);
    mbar_init(bar_h, 1); mbar_init(bar_d, 1); mbar_init(bar_v, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (w == 16) tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), 512);
  uint32_t* vmax_s = reinterpret_cast<uint32_t*>(hp_s);
  if (probs_wide(V, n, d, vmax_s + kPtD, vmax_s)) {
    if (w == 16) tmem_dealloc(*tmem_slot, 512);
    probs_fp32_rows<law>(reinterpret_cast<float*>(sm), p_all, V, n, d, param, kq, draw0, K_all, ds_sum, ds_sq, dV_sum, rows);
    return;
  }
  // V's three terms, [entry][column] rows of 128 bytes in the 128-byte swizzle: the K-major A operand of
  // dp^T and the MN-major B operand of H.  The scale of a column is the power of two at or above its
  // largest magnitude.
  for (int i = tid; i < kPtN * kPtD; i += kPtThreads) {
    const int j = i >> 6, c = i & 63;
    const float m = __uint_as_float(vmax_s[c]);
    int ex = 0;
    if (m > 0.f) frexpf(m, &ex);                                      // m < 2^ex
    float v = j < n && c < d ? ldg(V + (size_t)j * d + c) : 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int sh = 8 + 9 * k - ex;                                  // unit 2^-sh
      const uint32_t t = float_to_bf16_bits(scalbnf(rintf(scalbnf(v, sh)), -sh));
      v -= bf16_bits_to_float(t);
      *reinterpret_cast<uint16_t*>(sm + kPtV + k * kPtTerm + j * 128 + ((((uint32_t)c >> 3) ^ (j & 7)) << 4) + (c & 7) * 2) =
          (uint16_t)t;
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = *tmem_slot, tm_lane = tm + ((uint32_t)(wq * 32) << 16);

  // a row's draws in segments: the products' accumulators truncate, so they are read out and added to the
  // sums in memory every kPtSegment draws
  const int R = kPtSlots / g, nsegs = (K_all + kPtSegment - 1) / kPtSegment;
  const size_t ngroups = (rows + R - 1) / R;
  uint32_t tile = 0;
  bool ok = true;
  // 640 threads start with 96 registers each; the warpgroup of the issuing warp leaves the workers 112
  if (w >= 16) {
    // ------------------------------------------------ the products, issued by one lane
    asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
    if (w == 16 && lane == 0) {
      const int nk = (n + 15) / 16, nkd = (d + 15) / 16;
      const uint32_t idesc_h = make_idesc(1u, 1u, 128, 64) | (1u << 16), idesc_d = make_idesc(1u, 1u, 128, 128),
                     idesc_v = make_idesc(1u, 1u, 128, 64) | (1u << 15) | (1u << 16);
      const uint64_t bits_k = make_smem_desc(base + kPtBits), bits_mn = make_smem_desc_mn(base + kPtBits, kPtTerm),
                     v_k = make_smem_desc(base + kPtV), v_mn = make_smem_desc_mn(base + kPtV, kPtTerm),
                     dl_k = make_smem_desc(base + kPtDelta), dl_mn = make_smem_desc_mn(base + kPtDelta, kPtTerm);
      constexpr uint32_t mat = kPtMat >> 4, term = kPtTerm >> 4;      // descriptor addresses count 16 bytes
      for (size_t grp = blockIdx.x; grp < stop && ok; grp += gridDim.x)
        for (int unit = 0; unit < K_all && ok; unit += g, ++tile) {   // (a segment is a whole number of tiles)
          const uint32_t ph = tile & 1u;
          const bool fresh = unit % kPtSegment == 0;
          for (int m = 0; m < 3 && ok; ++m) {
            ok = mbar_wait(bar_go + 8 * m, ph, abort_flag);
            if (!ok) break;
            tc_fence_after();
            for (int t = 2; t >= 0; --t)                              // the first term alone, the other two together
              for (int ks = 0; ks < nk; ++ks)
                tc_mma<false>(tm + kPtTmH + m * 128 + (t ? 64 : 0), bits_k + m * mat + (ks >> 2) * term + 2u * (ks & 3),
                              v_mn + t * term + 128u * ks, idesc_h, t == 1 || ks != 0 ? 1u : 0u);
          }
          if (!ok) break;
          tc_commit(bar_h);
          ok = mbar_wait(bar_go + 24, ph, abort_flag);
          if (!ok) break;
          tc_fence_after();
          // dp^T: products of V's and delta's terms down to 2^-24, the smallest first
#pragma unroll
          for (int i = 0; i < 6; ++i) {
            constexpr int tv[6] = {2, 0, 1, 1, 0, 0}, td[6] = {0, 2, 1, 0, 1, 0};
            for (int ks = 0; ks < nkd; ++ks)
              tc_mma<false>(tm + kPtTmDp, v_k + tv[i] * term + 2u * ks, dl_k + td[i] * term + 2u * ks, idesc_d,
                            (i | ks) != 0 ? 1u : 0u);
          }
          tc_commit(bar_d);
          // sum over the row's slots of q delta^T and a delta^T
          for (int r = 0; r < R; ++r)
            for (int m = 0; m < 2; ++m)
              for (int t = 2; t >= 0; --t)
                for (int ks = 0; ks < g / 16; ++ks) {
                  const uint32_t at = (uint32_t)(r * g * 8) + 128u * ks;
                  tc_mma<false>(tm + (r ? kPtTmAcc1 : kPtTmAcc0) + m * 64, bits_mn + m * mat + at, dl_mn + t * term + at, idesc_v,
                                !fresh || t != 2 || ks != 0 ? 1u : 0u);
                }
          tc_commit(bar_v);
        }
      if (!ok)                                                        // let the products in flight end
        for (int i = 0; i < 200; ++i) __nanosleep(1000);
    }
  } else {
    // ------------------------------------------------ sixteen worker warps
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    const float step = law == 1 ? 2.f * param : param;
    const uint32_t c3 = kq.c3 & ~0xFFu;
    const float inv_param = 1.f / param;
    size_t it = (size_t)blockIdx.x * nsegs;
    for (; it < stop * nsegs && ok;
         it += (it + 1) % nsegs ? 1 : ((size_t)gridDim.x - 1) * nsegs + 1) {      // group by group, its segments in order
      const size_t row0 = it / nsegs * R;
      const int seg = (int)(it % nsegs), k_seg = seg * kPtSegment, K = K_all - k_seg < kPtSegment ? K_all - k_seg : kPtSegment,
                nchunks = (K + g - 1) / g;
      // ---- the group's rows: probabilities, V^T p and V^T (lo - p) (in double: their error would be
      // the same in every draw), V (V^T p)
      for (int i = tid; i < R * kPtN; i += kPtWorkers) {
        const size_t row = row0 + (i >> 7);
        const int j = i & (kPtN - 1);
        const float p = row < rows && j < n ? ldg(p_all + row * n + j) : 0.f;
        float lo = 0.f, hi;
        uint32_t thr = law == 1 ? 0xFFFFFFFFu : 0u;                   // never up
        if (j < n && row < rows) probs_cell(p, law, param, lo, hi, thr);
        p_s[i] = p;
        x_s[i] = lo;
        thr_s[i] = thr;
      }
      pt_sync();
      if (w < R) {
        double t = 0.0;
        for (int j = lane; j < kPtN; j += 32) t += (double)x_s[w * kPtN + j];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
        if (lane == 0) sumlo_s[w] = t - 1.0;
      }
      const int gen_r = 8 * w / g;                                    // the row this warp draws for
      const uint4 thr4 = *reinterpret_cast<const uint4*>(thr_s + gen_r * kPtN + 4 * lane);
      const uint32_t thr[4] = {thr4.x, thr4.y, thr4.z, thr4.w};
      // the entry pass's ownership: entry ej, slots 32 wg ..
      const int ej = 32 * wq + lane, er = 32 * wg / g;
      const bool e_on = row0 + er < rows && 32 * wq < n;              // (warp-uniform)
      const float ep = p_s[er * kPtN + ej], elo = x_s[er * kPtN + ej];
      // as probs_cell: lo = n0 param (n0 is found again without its division, up to where that is exact)
      float ehi = law == 1 ? ep + param : (rintf(elo * inv_param) + 1.f) * param;
      if (law == 0 && elo > 1e6f * param) {
        float lo;
        uint32_t t;
        probs_cell(ep, law, param, lo, ehi, t);
      }
      const float dlo = elo - ep, dhi = ehi - ep;
      const uint64_t gq = ((row0 + gen_r) * (uint64_t)n) / 4 + lane;  // n % 4 == 0: a generator block per lane
      // column partials: warp w takes entries 8 w .. 8 w + 7, a lane columns 2 lane and 2 lane + 1
      double2* colp_s = reinterpret_cast<double2*>(sm + kPtDelta);
      {
        double acc[2][4] = {{0.0, 0.0, 0.0, 0.0}, {0.0, 0.0, 0.0, 0.0}};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int j = 8 * w + i;
          const uint32_t off = kPtV + j * 128 + ((((uint32_t)lane >> 2) ^ i) << 4) + (lane & 3) * 4;
          float v0 = 0.f, v1 = 0.f;
#pragma unroll
          for (int k = 2; k >= 0; --k) {
            const uint32_t u = *reinterpret_cast<const uint32_t*>(sm + off + k * kPtTerm);
            v0 += __uint_as_float(u << 16);
            v1 += __uint_as_float(u & 0xFFFF0000u);
          }
#pragma unroll
          for (int r = 0; r < 2; ++r)
            if (r < R) {
              const double d0 = (double)v0, d1 = (double)v1, p = (double)p_s[r * kPtN + j], l = (double)x_s[r * kPtN + j] - p;
              acc[r][0] = fma(d0, p, acc[r][0]); acc[r][1] = fma(d1, p, acc[r][1]);
              acc[r][2] = fma(d0, l, acc[r][2]); acc[r][3] = fma(d1, l, acc[r][3]);
            }
        }
#pragma unroll
        for (int r = 0; r < 2; ++r)
          if (r < R) {
            colp_s[((2 * r) * 16 + w) * 32 + lane] = make_double2(acc[r][0], acc[r][1]);
            colp_s[((2 * r + 1) * 16 + w) * 32 + lane] = make_double2(acc[r][2], acc[r][3]);
          }
      }
      pt_sync();
      if (tid < 2 * R * kPtD) {                                       // (row, which, column)
        const int c = tid & 63, which = (tid >> 6) & 1, r = tid >> 7;
        const double* q = reinterpret_cast<const double*>(colp_s + ((2 * r + which) * 16) * 32) + c;
        double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int k = 0; k < 16; ++k) s[k & 3] += q[k * 64];
        (which ? hl_s : hp_s)[r * kPtD + c] = (float)((s[0] + s[1]) + (s[2] + s[3]));
      }
      pt_sync();
      for (int r = 0; r < R; ++r) {                                   // V (V^T p): four threads per entry, 16 columns each
        const int j = tid >> 2, q = tid & 3;
        float s = 0.f;
#pragma unroll
        for (int h8 = 0; h8 < 2; ++h8) {
          const uint32_t off = kPtV + j * 128 + (((uint32_t)(2 * q + h8) ^ (j & 7)) << 4);
          float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int k = 2; k >= 0; --k) {
            const uint4 u = *reinterpret_cast<const uint4*>(sm + off + k * kPtTerm);
            const uint32_t uu[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) { v[2 * e] += bf16_bits_to_float(uu[e] & 0xFFFFu); v[2 * e + 1] += bf16_bits_to_float(uu[e] >> 16); }
          }
#pragma unroll
          for (int e = 0; e < 8; ++e) s = fmaf(v[e], hp_s[r * kPtD + 16 * q + 8 * h8 + e], s);
        }
        s += __shfl_xor_sync(0xFFFFFFFFu, s, 1);
        s += __shfl_xor_sync(0xFFFFFFFFu, s, 2);
        if (q == 0) x_s[r * kPtN + j] = s;                            // (lo was last read before the barriers above)
      }
      float sd = 0.f;
      uint64_t acc_s[5], acc_q[5];                                    // over even and odd slots
#pragma unroll
      for (int o = 0; o < 5; ++o) acc_s[o] = acc_q[o] = 0ull;
      uint32_t cnt_q4 = 0u, cnt_a4 = 0u;                              // up-roundings of this lane's four entries, a byte each
      const double sumlo = sumlo_s[gen_r];

      for (int chunk = 0; chunk < nchunks; ++chunk, ++tile) {
        const uint32_t ph = tile & 1u;
        // ---- bits of the three streams; the H products of a stream run under the generator of the next
        uint32_t code[8];
#pragma unroll
        for (int s8 = 0; s8 < 8; ++s8) code[s8] = 0u;
        const int nv = K - (chunk * g + ((8 * w) & (g - 1)));           // draws left for this warp's eight slots
        // (unrolled, so that a stream does only its own counting: 4.23 -> 4.06 ms; a second body for whole groups of
        // eight draws, without their limit, is no faster)
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          uint32_t ups[2] = {0u, 0u};                                 // up-roundings of a, a byte per slot (at most 128)
          if (nv <= 0) {                                              // (warp-uniform)
#pragma unroll
            for (int s8 = 0; s8 < 8; ++s8)
              *reinterpret_cast<uint2*>(sm + kPtBits + m * kPtMat + (lane >> 4) * kPtTerm + (8 * w + s8) * 128 +
                                        ((((uint32_t)(lane & 15) >> 1) ^ s8) << 4) + (lane & 1) * 8) = make_uint2(0u, 0u);
            pt_arrive(bar_go + 8 * m, lane);
            continue;
          }
#pragma unroll
          for (int s8 = 0; s8 < 8; ++s8) {
            const int slot = 8 * w + s8, k = chunk * g + (slot & (g - 1));
            // the four bits as bf16 0 / 1; no branch, so that the slots' generator chains interleave (entries past
            // n and rows past the end have thresholds nothing passes)
            const uint4 x = philox4x32_10((uint32_t)gq, (uint32_t)(gq >> 32), (uint32_t)(draw0 + k_seg + k), c3 | (uint32_t)m, kq.k0, kq.k1);
            auto up = [&](uint32_t word, uint32_t t) { return law == 1 ? word > t : word < t; };
            uint32_t lo2 = (up(x.x, thr[0]) ? 0x3F80u : 0u) | (up(x.y, thr[1]) ? 0x3F800000u : 0u);
            uint32_t hi2 = (up(x.z, thr[2]) ? 0x3F80u : 0u) | (up(x.w, thr[3]) ? 0x3F800000u : 0u);
            if (s8 >= nv) lo2 = hi2 = 0u;
            const uint32_t t4 = __byte_perm(lo2, hi2, 0x7531);        // 0x3F or 0 per entry
            code[s8] |= t4 & (0x01010101u << m);
            if (m == 0) cnt_q4 += t4 & 0x01010101u;
            if (m == 1) {
              cnt_a4 += t4 & 0x01010101u;
              ups[s8 >> 2] += (uint32_t)__popc(t4 & 0x01010101u) << (8 * (s8 & 3));
            }
            *reinterpret_cast<uint2*>(sm + kPtBits + m * kPtMat + (lane >> 4) * kPtTerm + slot * 128 +
                                      ((((uint32_t)(lane & 15) >> 1) ^ s8) << 4) + (lane & 1) * 8) = make_uint2(lo2, hi2);
          }
          if (m == 1) {
            const uint32_t u0 = __reduce_add_sync(0xFFFFFFFFu, ups[0]), u1 = __reduce_add_sync(0xFFFFFFFFu, ups[1]);
            // 1^T a - 1, in double from the count
            if (lane < 8)
              suma_s[8 * w + lane] = (float)(sumlo + (double)step * (double)(((lane & 4 ? u1 : u0) >> (8 * (lane & 3))) & 0xFFu));
          }
          pt_arrive(bar_go + 8 * m, lane);
        }
#pragma unroll
        for (int h8 = 0; h8 < 2; ++h8) {                              // codes by entry: four slots to a word
          const uint32_t* c4 = code + 4 * h8;
          const uint32_t t0 = __byte_perm(c4[0], c4[1], 0x5140), t1 = __byte_perm(c4[2], c4[3], 0x5140);
          const uint32_t t2 = __byte_perm(c4[0], c4[1], 0x7362), t3 = __byte_perm(c4[2], c4[3], 0x7362);
          uint32_t* dst = reinterpret_cast<uint32_t*>(sm + kPtCodes + 4 * lane * kPtCodePitch + 8 * w + 4 * h8);
          dst[0] = __byte_perm(t0, t1, 0x5410);
          dst[kPtCodePitch / 4] = __byte_perm(t0, t1, 0x7632);
          dst[2 * kPtCodePitch / 4] = __byte_perm(t2, t3, 0x5410);
          dst[3 * kPtCodePitch / 4] = __byte_perm(t2, t3, 0x7632);
        }
        // ---- slot pass: a thread is a slot and takes 16 of its 64 columns
        ok = __all_sync(0xFFFFFFFFu, mbar_wait_suspend(bar_h, ph, abort_flag));
        if (ok) {
          tc_fence_after();
          const int slot = 32 * wq + lane, r = 32 * wq / g;
          const float* hp = hp_s + r * kPtD + 16 * wg;
          const float* hl = hl_s + r * kPtD + 16 * wg;
          float4 dt = make_float4(0.f, 0.f, 0.f, 0.f);
          float dq[16];
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            uint32_t h1[16], h2[16];
            tmem_ld16(tm_lane + kPtTmH + m * 128 + 16 * wg, h1);
            tmem_ld16(tm_lane + kPtTmH + m * 128 + 64 + 16 * wg, h2);
            tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 16; ++c) {
              const float x = fmaf(step, __uint_as_float(h2[c]), fmaf(step, __uint_as_float(h1[c]), hl[c]));
              if (m == 0) {
                dq[c] = x;
                const float h = hp[c] + x;
                dt.x = fmaf(hp[c], h, dt.x);
                dt.y = fmaf(x, h, dt.y);
              } else if (m == 1) {
                dt.z = fmaf(x, hp[c] + dq[c], dt.z);
              } else {
                dt.w = fmaf(x, hp[c] + dq[c], dt.w);
              }
            }
          }
          dotp_s[wg * kPtSlots + slot] = dt;
#pragma unroll
          for (int h8 = 0; h8 < 2; ++h8) {
            uint32_t pk[3][4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              uint32_t t3[3];
              bf16_split3(dq[8 * h8 + 2 * c], dq[8 * h8 + 2 * c + 1], t3);
#pragma unroll
              for (int t = 0; t < 3; ++t) pk[t][c] = t3[t];
            }
#pragma unroll
            for (int t = 0; t < 3; ++t)
              *reinterpret_cast<uint4*>(sm + kPtDelta + t * kPtTerm + slot * 128 + (((uint32_t)(2 * wg + h8) ^ (slot & 7)) << 4)) =
                  make_uint4(pk[t][0], pk[t][1], pk[t][2], pk[t][3]);
          }
          pt_arrive(bar_go + 24, lane);
          // the sum of delta over the warp's slots: lane pair l holds column l / 2 of the warp's sixteen
          if (chunk * g + (slot & (g - 1)) >= K)
#pragma unroll
            for (int c = 0; c < 16; ++c) dq[c] = 0.f;
#pragma unroll
          for (int o = 8; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < o; ++c) {
              const bool up = lane & (2 * o);
              const float keep = up ? dq[c + o] : dq[c], give = up ? dq[c] : dq[c + o];
              dq[c] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, 2 * o);
            }
          sd += dq[0] + __shfl_xor_sync(0xFFFFFFFFu, dq[0], 1);
        }
        ok = pt_sync_and(ok);
        if (!ok) break;
        if (tid >= kPtWorkers - kPtSlots) {
          const int slot = tid - (kPtWorkers - kPtSlots);
          float4 s = dotp_s[slot];
#pragma unroll
          for (int k = 1; k < 4; ++k) {
            const float4 v = dotp_s[k * kPtSlots + slot];
            s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
          }
          dots_s[slot] = -s.x; dots_s[kPtSlots + slot] = -s.y;
          dots_s[2 * kPtSlots + slot] = -s.z; dots_s[3 * kPtSlots + slot] = -s.w;
        }
        ok = mbar_wait_suspend(bar_d, ph, abort_flag);
        ok = pt_sync_and(ok);
        if (!ok) break;
        tc_fence_after();
        // ---- entry pass: with J(x) dp = x o dp - x (x.dp) and x = p + dx,
        // (J(x) - J(p)) dp = dx (dp - p.dp) - x (dx.dp): no error is formed as a difference of large terms
        // Four slots at a time, two to a packed instruction; J2's errors are kept doubled.
        const int left = K - (chunk * g + ((32 * wg) & (g - 1))), nval = left < 32 ? left : 32;
        if (e_on && nval > 0) {
          const float dp0 = x_s[er * kPtN + ej];
          const uint64_t dp02 = f2(dp0, dp0), p2 = f2(ep, ep);
          const uint32_t* cp = reinterpret_cast<const uint32_t*>(sm + kPtCodes + ej * kPtCodePitch + 32 * wg);
          const float4* sp = reinterpret_cast<const float4*>(dots_s + 32 * wg);
          const float4* sa = reinterpret_cast<const float4*>(suma_s + 32 * wg);
#pragma unroll 1
          for (int c0 = 0; c0 < nval; c0 += 8) {
            uint32_t dv[8];
            tmem_ld8(tm_lane + kPtTmDp + 32 * wg + c0, dv);
            tmem_wait_ld();
#pragma unroll
            for (int q4 = 0; q4 < 2; ++q4) {
              if (c0 + 4 * q4 >= nval) break;                         // (warp-uniform)
              const int s4 = (c0 >> 2) + q4;
              const uint32_t cd = cp[s4];
              const float4 n0 = sp[s4], nq = sp[kPtSlots / 4 + s4], na = sp[2 * kPtSlots / 4 + s4], nb = sp[3 * kPtSlots / 4 + s4],
                           S = sa[s4];
              const bool part = c0 + 4 * q4 + 4 > nval;               // the last slots of a row whose draws end here
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                const uint32_t b0 = cd >> (16 * h), b1 = cd >> (16 * h + 8);
                const uint64_t N0 = h ? f2(n0.z, n0.w) : f2(n0.x, n0.y), NQ = h ? f2(nq.z, nq.w) : f2(nq.x, nq.y),
                               NA = h ? f2(na.z, na.w) : f2(na.x, na.y), NB = h ? f2(nb.z, nb.w) : f2(nb.x, nb.y),
                               SA = h ? f2(S.z, S.w) : f2(S.x, S.y);
                const uint64_t dq = f2(b0 & 1u ? dhi : dlo, b1 & 1u ? dhi : dlo), da = f2(b0 & 2u ? dhi : dlo, b1 & 2u ? dhi : dlo),
                               db = f2(b0 & 4u ? dhi : dlo, b1 & 4u ? dhi : dlo);
                const uint64_t pq = f2_add(dq, p2), a = f2_add(da, p2), b = f2_add(db, p2);
                const uint64_t dp = f2_add(f2(__uint_as_float(dv[4 * q4 + 2 * h]), __uint_as_float(dv[4 * q4 + 2 * h + 1])), dp02);
                const uint64_t c = f2_add(dp, N0), tq = f2_mul(dq, c), ta = f2_mul(da, c), tb = f2_mul(db, c);
                uint64_t er5[5];
                er5[0] = f2_fma(pq, NQ, tq);                                          // J(p_q)
                er5[1] = f2_fma(a, NA, ta);                                           // J(a)
                er5[2] = f2_fma(f2_mul(a, SA), dp, er5[1]);                           // K(a): + a (1^T a - 1) dp
                er5[3] = f2_fma(a, NB, f2_fma(b, NA, f2_add(ta, tb)));                // 2 J2(a, b)
                er5[4] = f2_fma(pq, NB, f2_fma(b, NQ, f2_add(tq, tb)));               // 2 J2(p_q, b)
                if (part) {
                  const int s0 = c0 + 4 * q4 + 2 * h;
                  const uint64_t on = f2(s0 < nval ? 1.f : 0.f, s0 + 1 < nval ? 1.f : 0.f);
#pragma unroll
                  for (int o = 0; o < 5; ++o) er5[o] = f2_mul(er5[o], on);
                }
#pragma unroll
                for (int o = 0; o < 5; ++o) { acc_s[o] = f2_add(acc_s[o], er5[o]); acc_q[o] = f2_fma(er5[o], er5[o], acc_q[o]); }
              }
            }
          }
        }
        // the bits and delta are free and the row sums complete; everyone is through with codes and dots
        ok = mbar_wait_suspend(bar_v, ph, abort_flag);
        ok = pt_sync_and(ok);
        if (!ok) break;
        tc_fence_after();
      }
      if (!ok) break;
      // ---- row end: the four slot groups' sums, in order
      uint32_t* cnt4_s = reinterpret_cast<uint32_t*>(sm + kPtDelta + kPtCnt4);
      float* cnt_s = reinterpret_cast<float*>(sm + kPtDelta + kPtCnt);
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        float s0, s1, q0, q1;
        f2_get(acc_s[v], s0, s1);
        f2_get(acc_q[v], q0, q1);
        comb_s[(wg * kPtVals + v) * kPtN + ej] = (s0 + s1) * (v < 3 ? 1.f : 0.5f);
        comb_s[(wg * kPtVals + 5 + v) * kPtN + ej] = (q0 + q1) * (v < 3 ? 1.f : 0.25f);
      }
      cnt4_s[w * 32 + lane] = cnt_q4;
      cnt4_s[(16 + w) * 32 + lane] = cnt_a4;
      if (!(lane & 1)) sd_s[wq * kPtD + 16 * wg + (lane >> 1)] = sd;
      pt_sync();
      const int per = g / 32;                                         // slot groups per row
      for (int i = tid; i < R * kPtVals * kPtN; i += kPtWorkers) {
        const int r = i / (kPtVals * kPtN), v = (i >> 7) % kPtVals, j = i & (kPtN - 1);
        float s = 0.f;
        for (int k = 0; k < per; ++k) s += comb_s[((r * per + k) * kPtVals + v) * kPtN + j];
        const size_t row = row0 + r;
        float* out = v < 5 ? ds_sum : ds_sq;
        if (out && row < rows && j < n) {
          out += ((size_t)(v < 5 ? v : v - 5) * rows + row) * n + j;
          *out = seg ? *out + s : s;
        }
      }
      for (int i = tid; i < 2 * R * kPtN; i += kPtWorkers) {          // (which, row, entry): counts over the row's warps
        const int which = i / (R * kPtN), r = (i >> 7) % R, j = i & (kPtN - 1);
        uint32_t c = 0u;
        for (int k = 0; k < g / 8; ++k) c += (cnt4_s[(16 * which + r * (g / 8) + k) * 32 + (j >> 2)] >> (8 * (j & 3))) & 0xFFu;
        cnt_s[(2 * r + which) * kPtN + j] = (float)c;
        if (which == 0) {
          const float p = p_s[r * kPtN + j];
          float lo = 0.f, hi = 0.f;
          uint32_t t;
          if (j < n) probs_cell(p, law, param, lo, hi, t);
          x_s[r * kPtN + j] = fmaf(hi - lo, (float)c, -((float)K * (p - lo)));   // w_j = sum over the draws of p_q - p
        }
      }
      pt_sync();
      // the gradient-of-V rows go through shared memory (over the bits, which the products have read): a
      // warp holds 32 entries of 16 columns, which straight to memory would be 32 rows per store
      for (int r = 0; r < R; ++r) {
        const size_t row = row0 + r;
        if (r) pt_sync();
        if (row < rows && 32 * wq < n && 16 * wg < d) {               // (warp-uniform)
          uint32_t aq[16], aa[16];
          const uint32_t acc = tm_lane + (r ? kPtTmAcc1 : kPtTmAcc0) + 16 * wg;
          tmem_ld16(acc, aq);
          tmem_ld16(acc + 64, aa);
          tmem_wait_ld();
          const float p = p_s[r * kPtN + ej], wj = x_s[r * kPtN + ej];
          float lo = 0.f, hi = 0.f;
          uint32_t t;
          if (ej < n) probs_cell(p, law, param, lo, hi, t);
          const float cq = cnt_s[2 * r * kPtN + ej], ca = cnt_s[(2 * r + 1) * kPtN + ej];
          const float wa = (hi - lo) * (ca - cq), pl = p - lo;
#pragma unroll
          for (int c = 0; c < 16; c += 4) {
            const float4 hp = *reinterpret_cast<const float4*>(hp_s + r * kPtD + 16 * wg + c);
            float4 sd4 = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int k = 0; k < per; ++k) {
              const float4 v = *reinterpret_cast<const float4*>(sd_s + (r * per + k) * kPtD + 16 * wg + c);
              sd4.x += v.x; sd4.y += v.y; sd4.z += v.z; sd4.w += v.w;
            }
            const float h4[4] = {hp.x, hp.y, hp.z, hp.w}, s4[4] = {sd4.x, sd4.y, sd4.z, sd4.w};
            float ou[4], oa[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float q = __uint_as_float(aq[c + e]);
              ou[e] = fmaf(-wj, h4[e], fmaf(pl, s4[e], -step * q));                 // p - p_q
              oa[e] = fmaf(wa, h4[e], step * (__uint_as_float(aa[c + e]) - q));     // a - p_q
            }
            const uint32_t off = kPtBits + ej * 256 + ((((uint32_t)(16 * wg + c) >> 2) ^ (ej & 15)) << 4);
            *reinterpret_cast<float4*>(sm + off) = make_float4(ou[0], ou[1], ou[2], ou[3]);
            *reinterpret_cast<float4*>(sm + off + kPtMat) = make_float4(oa[0], oa[1], oa[2], oa[3]);
          }
        }
        pt_sync();
        if (row < rows) {
          float* o_u = dV_sum + row * (size_t)n * d;
          float* o_a = o_u + rows * (size_t)n * d;
          if ((d & 3) == 0) {
            const int dq4 = d >> 2;
            for (int i = tid; i < n * dq4; i += kPtWorkers) {
              const int j = i / dq4, c4 = i - j * dq4;
              const uint32_t off = kPtBits + j * 256 + ((uint32_t)(c4 ^ (j & 15)) << 4);
              float4 u = *reinterpret_cast<const float4*>(sm + off), a = *reinterpret_cast<const float4*>(sm + off + kPtMat);
              if (seg) {
                const float4 u0 = reinterpret_cast<const float4*>(o_u)[i], a0 = reinterpret_cast<const float4*>(o_a)[i];
                u.x += u0.x; u.y += u0.y; u.z += u0.z; u.w += u0.w;
                a.x += a0.x; a.y += a0.y; a.z += a0.z; a.w += a0.w;
              }
              reinterpret_cast<float4*>(o_u)[i] = u;
              reinterpret_cast<float4*>(o_a)[i] = a;
            }
          } else {
            for (int i = tid; i < n * d; i += kPtWorkers) {
              const int j = i / d, c = i - j * d;
              const uint32_t off = kPtBits + j * 256 + ((((uint32_t)c >> 2) ^ (j & 15)) << 4) + (c & 3) * 4;
              const float u = *reinterpret_cast<const float*>(sm + off), a = *reinterpret_cast<const float*>(sm + off + kPtMat);
              o_u[i] = seg ? o_u[i] + u : u;
              o_a[i] = seg ? o_a[i] + a : a;
            }
          }
        }
      }
      tc_fence_before();
      pt_sync();                                                      // the scratch is reused
      tc_fence_after();
    }
    // a bounded wait ran out: the sums of this block's rows that are not complete do not look valid
    for (size_t grp = it / nsegs; grp < ngroups; grp += gridDim.x) {
      const size_t r0 = grp * R, nr = rows - r0 < (size_t)R ? rows - r0 : (size_t)R;
      for (int o = 0; o < 5; ++o)
        for (size_t i = tid; i < nr * n; i += kPtWorkers) {
          ds_sum[(o * rows + r0) * n + i] = NAN;
          if (ds_sq) ds_sq[(o * rows + r0) * n + i] = NAN;
        }
      for (int o = 0; o < 2; ++o)
        for (size_t i = tid; i < nr * n * d; i += kPtWorkers) dV_sum[(o * rows + r0) * (size_t)n * d + i] = NAN;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (w == 16) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tm, 512);
  }
}

}  // namespace bsp
