// Averages over the forward's rounding (Appendix "What the checker reads and reports"; Appendix "The
// same dependence in a normalization backward"; the continuation probes of Appendix "The
// normalization store").
//
// Setting: normalisation -> FP8 store u_q = u + r -> y = u_q W^T with the loss ||y||^2 / 2, so that the
// incoming gradients dy = y and du = dy W depend on the rounding the forward consumed.  The forward
// is drawn again and again (generator stream 0, draws 0, 1, 2, ...; pair k = draws 2k, 2k + 1) and
// the following are averaged:
//   * the gain-use error under read R, sum_t (r / gamma) o du, with its split into a mean part
//     sum_t (E r / gamma) o E du and a coupling (the rest); and the same error under a fresh read;
//   * per pair T = <r_a - r_b, du_a - du_b> / 2 and the control <du_a, r_b>;
//   * X = -(r_a - r_b)^T (dy_a - dy_b) / 2, which averages to the weight-use error -r^T dy.
//
// Tensor cores carry the three contractions with no operand rounded below 16 bits: u_q (decoded
// codes) and W are bf16 values, dy is split into hi + lo bf16 terms against W twice over, and for X
// the difference of two roundings of one value is a single grid step (exact in bf16) against the
// hi + lo split of dy_a - dy_b.  The contractions' epilogues write what the next step reads (the split of
// y, the split of y_a - y_b, the running sums of X), and both operands of X and the second of du are
// read as they lie in memory (contraction index outermost), so no transposed copy is made.
//
// Per forward two passes over [T, C] remain, each element touched once: cp_forward_kernel (the store's
// rounding as the bf16 operand) and cp_sums_kernel (both gain-use errors with the fresh rounding formed on
// the fly, and for the second forward of a pair the dot products and the sums of r and du).
// 16 forwards of 4096 x 1024 -> 4096: 5.27 -> 3.1 ms (the contractions 2.2 of them).
#include <string.h>

#include <vector>

#include "common.cuh"
#include "gemm.cuh"

namespace bsp {

// u of four columns from the saved statistics: the chain of FP32 operations of the FP8 store.
__device__ __forceinline__ void cp_chain(int kind, const float4& x, float rs, float mu, const float4& g, const float4& b,
                                         float (&u)[4]) {
  if (kind == BSP_RMSNORM) {
    u[0] = __fmul_rn(__fmul_rn(x.x, rs), g.x); u[1] = __fmul_rn(__fmul_rn(x.y, rs), g.y);
    u[2] = __fmul_rn(__fmul_rn(x.z, rs), g.z); u[3] = __fmul_rn(__fmul_rn(x.w, rs), g.w);
  } else {
    u[0] = __fadd_rn(__fmul_rn(__fmul_rn(__fsub_rn(x.x, mu), rs), g.x), b.x);
    u[1] = __fadd_rn(__fmul_rn(__fmul_rn(__fsub_rn(x.y, mu), rs), g.y), b.y);
    u[2] = __fadd_rn(__fmul_rn(__fmul_rn(__fsub_rn(x.z, mu), rs), g.z), b.z);
    u[3] = __fadd_rn(__fmul_rn(__fmul_rn(__fsub_rn(x.w, mu), rs), g.w), b.w);
  }
}

__device__ __forceinline__ void bf16x4_to_float(const uint2& b, float (&v)[4]) {
  v[0] = bf16_bits_to_float(b.x & 0xFFFFu); v[1] = bf16_bits_to_float(b.x >> 16);
  v[2] = bf16_bits_to_float(b.y & 0xFFFFu); v[3] = bf16_bits_to_float(b.y >> 16);
}

// One forward's rounding: code = round(u scale), uq = decode(code) as bf16 (exact).  uq_a given: also
// dr[t] = dr[T + t] = uq_a - uq, the first operand of X (twice, to meet both terms of the second; zero or
// one grid step, exact in bf16).
// Block (64, 4): 64 groups of four columns by 16 rows; the rows along grid.x, which holds any T.
constexpr int kCpRows = 16;
template <int DT, int FMT, bool SR>
__global__ void __launch_bounds__(256)
cp_forward_kernel(int kind, const void* x, int64_t T, int64_t C, const float* gamma,
                  const float* beta, const float* rstd, const float* mean,
                  const float* scale_dev, PhiloxKey key, uint16_t* uq,
                  const uint16_t* uq_a, uint16_t* dr, bsp_diag_t* diag) {
  grid_dependency();
  const int64_t c = 4 * ((int64_t)blockIdx.y * 64 + threadIdx.x);
  const float scale = ldg(scale_dev);
  DiagCounters dc;
  if (c < C) {
    const float4 g4 = ldg(reinterpret_cast<const float4*>(gamma + c));
    float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (kind == BSP_LAYERNORM) b4 = ldg(reinterpret_cast<const float4*>(beta + c));
    // the loads of the thread's rows are all requested before the first is used (4096 x 1024: 17.6 -> 15.4 us)
    constexpr int R = kCpRows / 4;
    const int64_t t0 = (int64_t)blockIdx.x * kCpRows + threadIdx.y;
    float4 xr[R];
    float rs[R], mu[R];
    uint2 qa_r[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int64_t t = t0 + 4 * j < T ? t0 + 4 * j : T - 1;
      xr[j] = load4<DT>(x, (size_t)t * C + c);
      rs[j] = ldg(rstd + t);
      mu[j] = kind == BSP_LAYERNORM ? ldg(mean + t) : 0.f;
      qa_r[j] = uq_a ? ldg(reinterpret_cast<const uint2*>(uq_a + (size_t)t * C + c)) : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int64_t t = t0 + 4 * j;
      if (t >= T) break;
      const size_t i = (size_t)t * C + c;
      float u[4];
      cp_chain(kind, xr[j], rs[j], mu[j], g4, b4, u);
      const float v[4] = {__fmul_rn(u[0], scale), __fmul_rn(u[1], scale), __fmul_rn(u[2], scale), __fmul_rn(u[3], scale)};
      uint32_t packed = 0;
      if (SR) {
        packed = f8_encode4_sr<FMT>(v, philox_block(key, (uint64_t)i >> 2, key.c2), dc);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) packed |= f8_encode<FMT, false>(v[e], 0u, dc) << (8 * e);
      }
      const uint2 q = f8_to_bf16x4<FMT>(packed);
      *reinterpret_cast<uint2*>(uq + i) = q;
      if (uq_a) {
        const uint2 a = qa_r[j];
        float qa[4], qb[4];
        bf16x4_to_float(a, qa);
        bf16x4_to_float(q, qb);
        const uint2 d = make_uint2(float_to_bf16_bits(qa[0] - qb[0]) | (float_to_bf16_bits(qa[1] - qb[1]) << 16),
                                   float_to_bf16_bits(qa[2] - qb[2]) | (float_to_bf16_bits(qa[3] - qb[3]) << 16));
        *reinterpret_cast<uint2*>(dr + i) = d;
        *reinterpret_cast<uint2*>(dr + (size_t)T * C + i) = d;
      }
    }
  }
  diag_flush_warp(diag, dc);
}

// W as bf16, twice: Wd[o][c] = Wd[O + o][c].  (W need not be aligned.)
template <int DT>
__global__ void __launch_bounds__(256)
cp_weight_kernel(const void* W, size_t n4, uint16_t* Wd) {
  grid_dependency();
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  const float4 v = (reinterpret_cast<uintptr_t>(W) & 15u) == 0
                       ? load4<DT>(W, 4 * i)
                       : make_float4(load1<DT>(W, 4 * i), load1<DT>(W, 4 * i + 1), load1<DT>(W, 4 * i + 2), load1<DT>(W, 4 * i + 3));
  const uint2 o = make_uint2(float_to_bf16_bits(v.x) | (float_to_bf16_bits(v.y) << 16), float_to_bf16_bits(v.z) | (float_to_bf16_bits(v.w) << 16));
  reinterpret_cast<uint2*>(Wd)[i] = o;
  reinterpret_cast<uint2*>(Wd)[n4 + i] = o;
}

// What a forward contributes once its du is there, in one walk over [T, C]: the gain-use sums of its own
// error r = uq / scale - u, sum_t r du, and of a fresh read's, sum_t (fresh(u) - u) du (generator stream of
// `key`, formed on the fly).  With the pair's first forward (uq_a, dua) given also sum (ra - r)(dua - du)
// and sum dua r, and both forwards join sum_r and sum_du (or start them, first).  u is formed from x
// again, which costs less traffic than an FP32 r would.  Block (x, y) walks slab y of rows for 128
// columns, a thread four columns of every eighth row; its two column sums join partial[2][slab][C] (or
// start it), so every sum has one writer and a fixed order.  A column's sum is an FP32
// chain of a thread's rows (cp_slab_rows bounds them); the dot products are summed in double from the products on
// (eight FP32 chains per thread instead took more registers than there are: 16 forwards of 4096 x 1024 -> 64
// 1277 -> 1202 us, and an error of T of 5e-8 of the terms' norm, not 1e-8).
constexpr int kCpSlabs = 64, kCpResident = 3;                       // slabs at most; blocks per SM
template <int DT, int FMT>
__global__ void __launch_bounds__(256, kCpResident)
cp_sums_kernel(int kind, const void* x, int64_t T, int64_t C, const float* gamma,
               const float* beta, const float* rstd, const float* mean,
               const float* scale_dev, PhiloxKey key, int64_t slab_rows, const uint16_t* uq,
               const float* du, const uint16_t* uq_a, const float* dua,
               float* sum_r, float* sum_du, bool first, float* partial,
               double* dots, bsp_diag_t* diag) {
  grid_dependency();
  __shared__ __align__(16) float sm[2][8][128];
  __shared__ double sd[2][8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t c = (int64_t)blockIdx.x * 128 + 4 * lane;
  const float scale = ldg(scale_dev), inv = __fdiv_rn(1.0f, scale);
  const int64_t t0 = (int64_t)blockIdx.y * slab_rows, t1 = t0 + slab_rows < T ? t0 + slab_rows : T;
  float own[4] = {0.f, 0.f, 0.f, 0.f}, fresh[4] = {0.f, 0.f, 0.f, 0.f};
  double da = 0.0, db = 0.0;
  DiagCounters dc;
  if (c < C) {
    const float4 g4 = ldg(reinterpret_cast<const float4*>(gamma + c));
    float4 b4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (kind == BSP_LAYERNORM) b4 = ldg(reinterpret_cast<const float4*>(beta + c));
    const int rows = (int)(t1 - t0);
#pragma unroll 1
    for (int n = w; n < rows; n += 8) {
      const int64_t t = t0 + n;
      const size_t i = (size_t)t * C + c;
      const float4 xv = load4<DT>(x, i), dv = ldg(reinterpret_cast<const float4*>(du + i));
      const uint2 qv = ldg(reinterpret_cast<const uint2*>(uq + i));
      uint2 qav = make_uint2(0u, 0u);
      float4 ya = make_float4(0.f, 0.f, 0.f, 0.f), sr = ya, sdu = ya;
      if (uq_a) {
        qav = ldg(reinterpret_cast<const uint2*>(uq_a + i));
        ya = ldg(reinterpret_cast<const float4*>(dua + i));
        if (!first) {
          sr = *reinterpret_cast<const float4*>(sum_r + i);
          sdu = *reinterpret_cast<const float4*>(sum_du + i);
        }
      }
      float u[4], q4[4], dec[4];
      cp_chain(kind, xv, ldg(rstd + t), kind == BSP_LAYERNORM ? ldg(mean + t) : 0.f, g4, b4, u);
      const float v[4] = {__fmul_rn(u[0], scale), __fmul_rn(u[1], scale), __fmul_rn(u[2], scale), __fmul_rn(u[3], scale)};
      const uint32_t packed = f8_encode4_sr<FMT>(v, philox_block(key, (uint64_t)i >> 2, key.c2), dc);
      f8_decode4<FMT>(packed, dec);
      bf16x4_to_float(qv, q4);
      const float d4[4] = {dv.x, dv.y, dv.z, dv.w};
      float r4[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        r4[e] = q4[e] * inv - u[e];
        own[e] = fmaf(r4[e], d4[e], own[e]);
        fresh[e] = fmaf(dec[e] * inv - u[e], d4[e], fresh[e]);
      }
      if (uq_a) {
        const float y4[4] = {ya.x, ya.y, ya.z, ya.w};
        float qa[4], ra[4];
        bf16x4_to_float(qav, qa);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          ra[e] = qa[e] * inv - u[e];
          da += (double)((ra[e] - r4[e]) * (y4[e] - d4[e]));
          db += (double)(y4[e] * r4[e]);
        }
        *reinterpret_cast<float4*>(sum_r + i) =
            make_float4((sr.x + ra[0]) + r4[0], (sr.y + ra[1]) + r4[1], (sr.z + ra[2]) + r4[2], (sr.w + ra[3]) + r4[3]);
        *reinterpret_cast<float4*>(sum_du + i) =
            make_float4((sdu.x + y4[0]) + d4[0], (sdu.y + y4[1]) + d4[1], (sdu.z + y4[2]) + d4[2], (sdu.w + y4[3]) + d4[3]);
      }
    }
  }
  diag_flush_warp(diag, dc);
  *reinterpret_cast<float4*>(&sm[0][w][4 * lane]) = make_float4(own[0], own[1], own[2], own[3]);
  *reinterpret_cast<float4*>(&sm[1][w][4 * lane]) = make_float4(fresh[0], fresh[1], fresh[2], fresh[3]);
  if (uq_a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) { da += __shfl_xor_sync(0xFFFFFFFFu, da, o); db += __shfl_xor_sync(0xFFFFFFFFu, db, o); }
    if (lane == 0) { sd[0][w] = da; sd[1][w] = db; }
  }
  __syncthreads();
  const int which = threadIdx.x >> 7, cl = threadIdx.x & 127;
  const int64_t cc = (int64_t)blockIdx.x * 128 + cl;
  if (cc < C) {
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += sm[which][k][cl];
    float* dst = partial + ((size_t)which * gridDim.y + blockIdx.y) * C + cc;
    *dst = first && !uq_a ? s : *dst + s;
  }
  if (uq_a && threadIdx.x < 2) {
    double s = 0.0;
    for (int k = 0; k < 8; ++k) s += sd[threadIdx.x][k];
    dots[2 * ((size_t)blockIdx.y * gridDim.x + blockIdx.x) + threadIdx.x] = s;
  }
}

// Rows of a slab: the fewest rounds of blocks over the SMs times eight rows of a block (and about two such steps of
// a block's own start and end), from kCpSlabs slabs down.  4096 x 1024: 52 slabs, 416 blocks in one round of 444
// places, where 64 slabs are 512 blocks in two (26.7 -> 20.1 us a pass on average).  Up to kCpMostRows rows, 64 of a
// thread: with terms of random signs the rounding of a column's sum has the variance T r / 16 in the threads' chains
// and T^2 / 2 r over the slabs, and at r = 512 that is what 64 slabs give for any T; more tokens take 64 slabs.
constexpr int64_t kCpMostRows = 512;
static int64_t cp_slab_rows(int64_t T, int64_t C) {
  const int64_t columns = (C + 127) / 128, places = kCpResident * kNumSMs;
  int64_t best = 0, cost = INT64_MAX;
  for (int64_t n = kCpSlabs; n > 0; --n) {
    const int64_t r = ((T + n - 1) / n + 7) & ~(int64_t)7;
    if (best && r > kCpMostRows) break;
    const int64_t rounds = (columns * ((T + r - 1) / r) + places - 1) / places;
    if (rounds * (r / 8 + 2) < cost) { cost = rounds * (r / 8 + 2); best = r; }
  }
  return best;
}

// out[k] = { T, control } of pair k from its blocks' dot products, in a fixed order.  One block per pair.
__global__ void __launch_bounds__(256)
cp_dots_final_kernel(const double* partial, int nblocks, double* out) {
  grid_dependency();
  __shared__ double sm[2][256];
  const double* p = partial + (size_t)blockIdx.x * 2 * nblocks;
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < nblocks; i += 256) { a += p[2 * i]; b += p[2 * i + 1]; }
  sm[0][threadIdx.x] = a; sm[1][threadIdx.x] = b;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) { sm[0][threadIdx.x] += sm[0][threadIdx.x + o]; sm[1][threadIdx.x] += sm[1][threadIdx.x + o]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) { out[2 * blockIdx.x] = 0.5 * sm[0][0]; out[2 * blockIdx.x + 1] = sm[1][0]; }
}

// The column sums sum_t a[t][c] b[t][c] per slab of rows (the mean part of the gain error at the end).
__global__ void __launch_bounds__(256)
cp_mean_part_kernel(const float* a, const float* b, int64_t T, int64_t C, int64_t slab_rows,
                    float* partial /* [slab][C] */) {
  grid_dependency();
  __shared__ float sm[8][33];
  const int cl = threadIdx.x & 31, rl = threadIdx.x >> 5;
  const int64_t c = (int64_t)blockIdx.x * 32 + cl;
  const int64_t t0 = (int64_t)blockIdx.y * slab_rows, t1 = t0 + slab_rows < T ? t0 + slab_rows : T;
  float s = 0.f;
  if (c < C)
    for (int64_t t = t0 + rl; t < t1; t += 8) s = fmaf(a[(size_t)t * C + c], b[(size_t)t * C + c], s);
  sm[rl][cl] = s;
  __syncthreads();
  if (rl == 0 && c < C) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += sm[w][cl];
    partial[(size_t)blockIdx.y * C + c] = t;
  }
}

// out_y[c] = f_y / gamma[c] times the slabs' sum y (0: own error, 1: fresh read, 2: mean part), in order.
__global__ void __launch_bounds__(256)
cp_gain_final_kernel(const float* partial /* [3][slab][C] */, int nslabs, const float* gamma, int64_t C,
                     float inv_n, float* own, float* fresh, float* mean_part) {
  grid_dependency();
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= C) return;
  const int y = blockIdx.y;
  const float* p = partial + (size_t)y * nslabs * C + c;
  float t = 0.f;
#pragma unroll 8
  for (int k = 0; k < nslabs; ++k) t += p[(size_t)k * C];
  (y == 0 ? own : y == 1 ? fresh : mean_part)[c] = t * (y == 2 ? inv_n * inv_n : inv_n) / gamma[c];
}

struct CouplingBuffers {
  float *rstd, *mean, *amax, *scale;
  uint16_t *uq[2], *Wd, *ysplit, *dr, *dy;
  float *ya, *du[2], *sum_r, *sum_du;
  float *gain_total, *gain_mean_part, *gain_fresh, *X, *X_sq, *gain_partial;
  double *dot_partial, *dots;
  int64_t slab_rows;
  int nslabs, nblocks;
};

static size_t coupling_carve(const bsp_coupling_desc_t* op, int pairs, char* base, CouplingBuffers* out) {
  size_t off = 0;
  auto take = [&](size_t bytes) -> void* {
    void* p = base ? base + off : nullptr;
    off += round_up(bytes ? bytes : 1, 256);
    return p;
  };
  const size_t T = (size_t)op->T, C = (size_t)op->C, O = (size_t)op->O;
  CouplingBuffers c;
  memset(&c, 0, sizeof(c));
  c.slab_rows = cp_slab_rows(op->T, (int64_t)C);
  c.nslabs = (int)((op->T + c.slab_rows - 1) / c.slab_rows);
  c.nblocks = c.nslabs * (int)((C + 127) / 128);
  c.rstd = (float*)take(T * 4); c.mean = (float*)take(T * 4); c.amax = (float*)take(4); c.scale = (float*)take(4);
  c.Wd = (uint16_t*)take(2 * O * C * 2);
  c.ysplit = (uint16_t*)take(T * 2 * O * 2); c.ya = (float*)take(T * O * 4);
  c.dr = (uint16_t*)take(2 * T * C * 2); c.dy = (uint16_t*)take(2 * T * O * 2);
  for (int i = 0; i < 2; ++i) { c.uq[i] = (uint16_t*)take(T * C * 2); c.du[i] = (float*)take(T * C * 4); }
  c.sum_r = (float*)take(T * C * 4); c.sum_du = (float*)take(T * C * 4);
  c.gain_total = (float*)take(C * 4); c.gain_mean_part = (float*)take(C * 4); c.gain_fresh = (float*)take(C * 4);
  c.X = (float*)take(C * O * 4); c.X_sq = (float*)take(C * O * 4);
  const size_t np = (size_t)(pairs > 0 ? pairs : 1);
  c.dot_partial = (double*)take(np * c.nblocks * 2 * sizeof(double));
  c.dots = (double*)take(np * 2 * sizeof(double));
  c.gain_partial = (float*)take((size_t)3 * c.nslabs * C * 4);
  if (out) *out = c;
  return off;
}

}  // namespace bsp

using namespace bsp;

extern "C" {

size_t bsp_coupling_check_workspace_bytes(const bsp_coupling_desc_t* op, int pairs) {
  if (!op || op->T <= 0 || op->C <= 0 || op->O <= 0 || pairs <= 0) return 0;
  return coupling_carve(op, pairs, nullptr, nullptr);
}

int bsp_coupling_layout(const bsp_coupling_desc_t* op, int pairs, bsp_coupling_layout_t* layout) {
  if (!op || !layout || op->T <= 0 || op->C <= 0 || op->O <= 0 || pairs <= 0) return BSP_ERR_ARG;
  CouplingBuffers b;
  char* const base = reinterpret_cast<char*>((uintptr_t)4096);
  coupling_carve(op, pairs, base, &b);
  auto off = [&](const void* p) { return (size_t)(reinterpret_cast<const char*>(p) - base); };
  layout->gain_total = off(b.gain_total); layout->gain_mean_part = off(b.gain_mean_part); layout->gain_fresh = off(b.gain_fresh);
  layout->X = off(b.X); layout->X_sq = off(b.X_sq);
  return BSP_OK;
}

#define BSP_TRY(expr)              \
  do {                             \
    int _rc = (expr);              \
    if (_rc != BSP_OK) return _rc; \
  } while (0)

int bsp_coupling_check(const bsp_coupling_desc_t* op, int pairs, double* T_out, double* control_out, void* ws,
                       size_t ws_bytes, bsp_diag_t* diag, void* stream) {
  if (!op || !T_out || !control_out || pairs <= 0) return BSP_ERR_ARG;
  if (op->T <= 0 || op->C <= 0 || op->O <= 0) return BSP_ERR_ARG;
  if (!op->x || !op->gamma || !op->W || (op->norm_kind == BSP_LAYERNORM && !op->beta)) return BSP_ERR_ARG;
  if (op->norm_kind < 0 || op->norm_kind > 1 || op->dtype < 0 || op->dtype > 1 || op->store_fmt < 0 || op->store_fmt > 1 ||
      op->forward_mode < 0 || op->forward_mode > 1 || op->tensor_id >= (1u << 24))
    return BSP_ERR_ARG;
  if (op->C % 16 != 0 || op->O % 16 != 0 || op->C > 8192) return BSP_ERR_UNSUPPORTED;
  if (!ws || ws_bytes < bsp_coupling_check_workspace_bytes(op, pairs) || (reinterpret_cast<uintptr_t>(ws) & 255u))
    return BSP_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  CouplingBuffers b;
  coupling_carve(op, pairs, reinterpret_cast<char*>(ws), &b);
  const int64_t T = op->T, C = op->C, O = op->O;
  const int dt = op->dtype, kind = op->norm_kind, fmt = op->store_fmt;

  BSP_TRY(bsp_norm_stats(kind, op->x, dt, T, C, op->gamma, op->beta, op->eps, b.rstd, b.mean, b.amax, diag, st));
  BSP_TRY(bsp_scale_from_amax(b.amax, 1, fmt, b.scale, st));
  const size_t w4 = (size_t)O * C / 4;
  if (dt == BSP_BF16) launch_kernel(cp_weight_kernel<BSP_BF16>, (unsigned)((w4 + 255) / 256), 256, 0, st, op->W, w4, b.Wd);
  else launch_kernel(cp_weight_kernel<BSP_F32>, (unsigned)((w4 + 255) / 256), 256, 0, st, op->W, w4, b.Wd);
  BSP_LAUNCH_CHECK();

  bsp_key_t key;
  key.seed = op->seed; key.tensor_id = op->tensor_id; key.reserved = 0;
  const dim3 gf((unsigned)((T + kCpRows - 1) / kCpRows), (unsigned)((C / 4 + 63) / 64));
  const dim3 gs((unsigned)((C + 127) / 128), (unsigned)b.nslabs);

  auto forward = [&](int draw, int slot) -> int {
    const bool first = draw < 2;                                    // the first pair
    key.stream = BSP_STREAM_FORWARD; key.draw = (uint32_t)draw;
    const PhiloxKey pk = make_key(key);
    const uint16_t* uq_a = slot ? b.uq[0] : nullptr;
#define BSP_CP_FWD(DT, FMT, SR)                                                                                          \
  launch_kernel(cp_forward_kernel<DT, FMT, SR>, gf, dim3(64, 4), 0, st, kind, op->x, T, C, op->gamma, op->beta, b.rstd, b.mean,     \
                                                             b.scale, pk, b.uq[slot], uq_a, b.dr, diag)
#define BSP_CP_MODE(DT, FMT)                                                   \
  do {                                                                         \
    if (op->forward_mode == BSP_ROUND_STOCHASTIC) BSP_CP_FWD(DT, FMT, true);   \
    else BSP_CP_FWD(DT, FMT, false);                                           \
  } while (0)
    if (dt == BSP_F32 && fmt == BSP_E4M3) BSP_CP_MODE(BSP_F32, BSP_E4M3);
    else if (dt == BSP_F32) BSP_CP_MODE(BSP_F32, BSP_E5M2);
    else if (fmt == BSP_E4M3) BSP_CP_MODE(BSP_BF16, BSP_E4M3);
    else BSP_CP_MODE(BSP_BF16, BSP_E5M2);
#undef BSP_CP_MODE
#undef BSP_CP_FWD
    BSP_LAUNCH_CHECK();
    // y = u_q W^T (decoded codes times bf16 W, the store's scale in the epilogue); dy = y.  The first
    // forward of a pair keeps y in FP32 for the second, whose epilogue writes the split of y_a - y_b
    GemmArgs g;
    g.M = T; g.N = O; g.K = C; g.nb = 1; g.fp8 = false;
    g.A = b.uq[slot]; g.lda = C; g.B = b.Wd; g.ldb = C; g.b_batch_stride = O * C;
    g.sa = 1.f; g.sa_dev = b.scale; g.sb = 1.f; g.mode = EPI_SPLIT; g.split = b.ysplit; g.ldc = O; g.diag = diag;
    if (slot == 0) g.C = b.ya;
    else { g.ref = b.ya; g.diff = b.dy; }
    BSP_TRY(gemm_run(g, st));
    // du = dy W: the split of dy against W twice
    GemmArgs h;
    h.M = T; h.N = C; h.K = 2 * O; h.nb = 1; h.fp8 = false;
    h.A = b.ysplit; h.lda = 2 * O; h.B = b.Wd; h.b_mn = true; h.ldb = C; h.b_batch_stride = 2 * O * C;
    h.sa = 1.f; h.sb = 1.f; h.mode = EPI_STORE_F32; h.C = b.du[slot]; h.ldc = C; h.diag = diag;
    BSP_TRY(gemm_run(h, st));
    // gain-use errors: read R (this forward's own error) and a fresh read (stream 1, same draw)
    key.stream = BSP_STREAM_GAIN;
    const PhiloxKey pg = make_key(key);
#define BSP_CP_SUMS(DT, FMT)                                                                                          \
  launch_kernel(cp_sums_kernel<DT, FMT>, gs, 256, 0, st, kind, op->x, T, C, op->gamma, op->beta, b.rstd, b.mean, b.scale, pg,    \
                                              b.slab_rows, b.uq[slot], b.du[slot], uq_a, slot ? b.du[0] : nullptr,    \
                                              b.sum_r, b.sum_du, first, b.gain_partial,                               \
                                              b.dot_partial + (size_t)(draw / 2) * b.nblocks * 2, diag)
    if (dt == BSP_F32 && fmt == BSP_E4M3) BSP_CP_SUMS(BSP_F32, BSP_E4M3);
    else if (dt == BSP_F32) BSP_CP_SUMS(BSP_F32, BSP_E5M2);
    else if (fmt == BSP_E4M3) BSP_CP_SUMS(BSP_BF16, BSP_E4M3);
    else BSP_CP_SUMS(BSP_BF16, BSP_E5M2);
#undef BSP_CP_SUMS
    BSP_LAUNCH_CHECK();
    return BSP_OK;
  };

  for (int k = 0; k < pairs; ++k) {
    BSP_TRY(forward(2 * k, 0));
    BSP_TRY(forward(2 * k + 1, 1));
    // X_k = -(r_a - r_b)^T (dy_a - dy_b) / 2 as [C, O], averaged with its square over the pairs
    GemmArgs x;
    x.M = C; x.N = O; x.K = 2 * T; x.nb = 1; x.fp8 = false;
    x.A = b.dr; x.a_mn = true; x.lda = C; x.B = b.dy; x.b_mn = true; x.ldb = O; x.b_batch_stride = 2 * T * O;
    x.sa = 1.f; x.sa_dev = b.scale; x.sb = -2.0f;                   // alpha = -1 / (2 scale): the codes' scale and the -1/2
    x.mode = EPI_MOMENTS; x.S1 = b.X; x.S2 = b.X_sq; x.ldc = O; x.diag = diag;
    x.moment_scale = 1.0f / (float)pairs; x.moment_first = k == 0;
    BSP_TRY(gemm_run(x, st));
  }
  launch_kernel(cp_dots_final_kernel, (unsigned)pairs, 256, 0, st, b.dot_partial, b.nblocks, b.dots);
  BSP_LAUNCH_CHECK();
  // mean part of the gain error, sum_t (sum_r / n) (sum_du / n) / gamma, and the averages over the forwards
  launch_kernel(cp_mean_part_kernel, dim3((unsigned)((C + 31) / 32), (unsigned)b.nslabs), 256, 0, st,
                b.sum_r, b.sum_du, T, C, b.slab_rows, b.gain_partial + (size_t)2 * b.nslabs * C);
  BSP_LAUNCH_CHECK();
  launch_kernel(cp_gain_final_kernel, dim3((unsigned)((C + 255) / 256), 3), 256, 0, st,
                b.gain_partial, b.nslabs, op->gamma, C, 1.0f / (float)(2 * pairs), b.gain_total, b.gain_fresh, b.gain_mean_part);
  BSP_LAUNCH_CHECK();
  std::vector<double> host((size_t)pairs * 2);
  BSP_CHECK_CUDA(cudaMemcpyAsync(host.data(), b.dots, host.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
  count_d2h(host.size() * sizeof(double));
  BSP_CHECK_CUDA(cudaStreamSynchronize(st));
  for (int k = 0; k < pairs; ++k) { T_out[k] = host[2 * k]; control_out[k] = host[2 * k + 1]; }
  return BSP_OK;
}

}  // extern "C"
