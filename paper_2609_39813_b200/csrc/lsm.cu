// Log-softmax backward with a +-eps error injected into its saved output (Appendix "Log-softmax").
//
// The operator's backward takes the incoming gradient h and the saved output S and returns
// h - exp(S) (1^T h).  The saved output is S = l + r, r_j = +-eps independently; under reuse the
// backward reads this S, under an independent copy l + r'.  With p = exp(l), g the returned gradient
// and g* what the operator returns from l with the same h, a trial's statistic is the mean over rows
// and classes of (g_j - g*_j) / p_j, under two losses: the likelihood with a fixed target (h = -e_y)
// and the constructed loss whose incoming gradient is the error itself (h = r).  Six statistics per
// trial (see bsp_lsm_stat_id), then mean, standard error over trials and z.
//
// What a class contributes depends on its error's sign alone: with A = (exp(l + r) - p) / p and
// B = (exp(l + r) / cosh(eps) - p) / p the six terms are A, A' (of the copy's sign), -A sum_r, -A' sum_r,
// B and -B sum_r, because h itself cancels between g and g* and sum_r = 1^T h of the constructed loss
// is common to the row.  So lsm_prep_kernel forms A and B for both signs once per row and class, and a
// trial adds up the entries its signs select.
//
// lsm_trial_kernel: a thread is a trial and walks the classes of its rows, so a row's sums stay in one
// thread: no shuffle, no barrier, and a warp reads one table entry at one address.  Per four classes
// two generator blocks and about 36 instructions of selection and addition: generator-bound.  The block
// per trial it replaces, which evaluated the exponentials per trial and reduced every row over the
// block, took 293 us for 64 x 128, 4096 trials; this one takes 57 us (two words per entry and trial
// at the generator's 1690 G words/s are 40 us).
// lsm_collect_kernel: sums over row chunks per trial, then the column sums over trials in double.
#include "common.cuh"

namespace bsp {

constexpr int kLsmThreads = 256;
constexpr int kLsmStats = 6, kLsmCols = 8;

__global__ void __launch_bounds__(kLsmThreads)
lsm_prep_kernel(const float* logits, int classes, float eps, float4* table) {
  grid_dependency();
  __shared__ float red[kLsmThreads / 32];
  __shared__ float bc;
  const size_t row = blockIdx.x;
  const float* x = logits + row * classes;
  float m = -INFINITY;
  for (int j = threadIdx.x; j < classes; j += kLsmThreads) m = fmaxf(m, x[j]);
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = red[0];
    for (int w = 1; w < kLsmThreads / 32; ++w) t = fmaxf(t, red[w]);
    bc = t;
  }
  __syncthreads();
  m = bc;
  float s = 0.f;
  for (int j = threadIdx.x; j < classes; j += kLsmThreads) s += expf(x[j] - m);
  s = warp_sum(s);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < kLsmThreads / 32; ++w) t += red[w];
    bc = logf(t);
  }
  __syncthreads();
  const float lz = bc;
  const float inv_c = 1.0f / coshf(eps);
  for (int j = threadIdx.x; j < classes; j += kLsmThreads) {
    const float l = (x[j] - m) - lz, p = expf(l), up = expf(l + eps), dn = expf(l - eps);
    table[row * classes + j] = make_float4((up - p) / p, (dn - p) / p, (up * inv_c - p) / p, (dn * inv_c - p) / p);
  }
}

// What a trial's signs select of `left` groups of a row (t: their table, q0: their first generator block): the sums
// of A, of A' and of B, and the count of +eps.  In lumps of 256 groups, so that a long row is no chain of thousands of
// additions: 16 x 8192, errors against 64 bits of the first four statistics 1.1, 1.2, 6.3, 3.6e-5 in one chain, 0.4, 0.4,
// 0.3, 0.5e-5 so.
constexpr int kLsmLump = 256;
__device__ __forceinline__ void lsm_walk(const float4* t, uint64_t q0, int left, PhiloxKey key_reuse, PhiloxKey key_copy,
                                         uint32_t trial, float& a1, float& a2, float& b1, int& cnt) {
  a1 = a2 = b1 = 0.f;
  cnt = 0;
#pragma unroll 1
  while (left > 0) {
    const int groups = left < kLsmLump ? left : kLsmLump;
    float l1 = 0.f, l2 = 0.f, m1 = 0.f;
#pragma unroll 2
    for (int g = 0; g < groups; ++g) {
      const uint4 w1 = philox_block(key_reuse, q0 + g, trial), w2 = philox_block(key_copy, q0 + g, trial);
      const uint32_t u1[4] = {w1.x, w1.y, w1.z, w1.w}, u2[4] = {w2.x, w2.y, w2.z, w2.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float4 v = ldg(t + 4 * g + e);
        l1 += (int)u1[e] < 0 ? v.x : v.y;                           // the top bit set: +eps
        m1 += (int)u1[e] < 0 ? v.z : v.w;
        l2 += (int)u2[e] < 0 ? v.x : v.y;
        cnt += (int)(u1[e] >> 31);
      }
    }
    a1 += l1; b1 += m1; a2 += l2;
    t += 4 * groups; q0 += groups; left -= groups;
  }
}

// Block (x, y): trials x * blockDim.x .., rows of chunk y; partial[y][statistic][trial].
__global__ void __launch_bounds__(kLsmThreads)
lsm_trial_kernel(const float4* table, int rows, int rows_per_chunk, int classes, float eps, PhiloxKey key_reuse,
                 PhiloxKey key_copy, int trials, float* partial) {
  grid_dependency();
  const int trial = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  const int row0 = (int)blockIdx.y * rows_per_chunk;
  const int row1 = row0 + rows_per_chunk < rows ? row0 + rows_per_chunk : rows;
  const int groups = classes / 4;                                   // classes % 4 == 0: groups never straddle rows
  float acc[kLsmStats] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int row = row0; row < row1; ++row) {
    float a1, a2, b1;
    int cnt;
    lsm_walk(table + (size_t)row * classes, (uint64_t)row * groups, groups, key_reuse, key_copy, (uint32_t)trial, a1, a2, b1, cnt);
    const float sum_r = eps * (float)(2 * cnt - classes);           // 1^T h of the constructed loss
    acc[0] += a1;
    acc[1] += a2;
    acc[2] -= a1 * sum_r;
    acc[3] -= a2 * sum_r;
    acc[4] += b1;
    acc[5] -= b1 * sum_r;
  }
  if (trial < trials)
#pragma unroll
    for (int i = 0; i < kLsmStats; ++i) partial[((size_t)blockIdx.y * kLsmStats + i) * trials + trial] = acc[i];
}

// The same for few trials of few rows, with the classes of a row cut as well: block (x, y) takes range y % nranges of row
// y / nranges, its threadIdx.y parts of `per` groups each; ranges[y][4][trial] the sums of A, A', B and the count.
__global__ void __launch_bounds__(kLsmThreads)
lsm_range_kernel(const float4* table, int nranges, int per, int classes, PhiloxKey key_reuse, PhiloxKey key_copy, int trials,
                 float* ranges) {
  grid_dependency();
  __shared__ float sm[4][kLsmThreads];
  const int trial = (int)(blockIdx.x * blockDim.x + threadIdx.x), row = (int)blockIdx.y / nranges;
  const int groups = classes / 4, g0 = ((int)(blockIdx.y % nranges) * (int)blockDim.y + (int)threadIdx.y) * per;
  float a1, a2, b1;
  int cnt;
  lsm_walk(table + (size_t)row * classes + 4 * g0, (uint64_t)row * groups + g0, groups - g0 < per ? groups - g0 : per, key_reuse, key_copy,
           (uint32_t)trial, a1, a2, b1, cnt);
  const int at = (int)(threadIdx.y * blockDim.x + threadIdx.x);
  sm[0][at] = a1; sm[1][at] = a2; sm[2][at] = b1; sm[3][at] = (float)cnt;
  __syncthreads();
  if (threadIdx.y == 0 && trial < trials)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float v = 0.f;
      for (int y = 0; y < (int)blockDim.y; ++y) v += sm[i][y * blockDim.x + threadIdx.x];
      ranges[((size_t)blockIdx.y * 4 + i) * trials + trial] = v;
    }
}

// The ranges of a row together, and its six terms, as lsm_trial_kernel leaves them for a chunk of one row.  Block (x, y):
// 32 trials of row y, eight threads sharing a trial's ranges.
__global__ void __launch_bounds__(256)
lsm_join_kernel(const float* ranges, int nranges, int classes, float eps, int trials, float* partial) {
  grid_dependency();
  __shared__ float sm[8][4][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, t = (int)blockIdx.x * 32 + lane;
  float s[4] = {0.f, 0.f, 0.f, 0.f};
  if (t < trials)
#pragma unroll 4
    for (int r = w; r < nranges; r += 8)
#pragma unroll
      for (int i = 0; i < 4; ++i) s[i] += ldg(ranges + (((size_t)blockIdx.y * nranges + r) * 4 + i) * trials + t);
#pragma unroll
  for (int i = 0; i < 4; ++i) sm[w][i][lane] = s[i];
  __syncthreads();
  if (w != 0 || t >= trials) return;
#pragma unroll
  for (int k = 1; k < 8; ++k)
#pragma unroll
    for (int i = 0; i < 4; ++i) s[i] += sm[k][i][lane];
  const float sum_r = eps * (2.f * s[3] - (float)classes);            // (the count is below 2^24: exact)
  const float v[kLsmStats] = {s[0], s[1], -s[0] * sum_r, -s[1] * sum_r, s[2], -s[2] * sum_r};
#pragma unroll
  for (int i = 0; i < kLsmStats; ++i) partial[((size_t)blockIdx.y * kLsmStats + i) * trials + t] = v[i];
}

// Per trial the statistics as means over rows and classes (FP32 out), and per block the sums over its
// trials: column c < 6 the statistic itself, 6 and 7 the paired contrasts reuse - independent
// (likelihood, constructed); out[block][2c], [2c + 1] = sum and sum of squares in double.  A block takes
// 32 trials at a time, eight threads sharing a trial's row chunks; fixed order throughout.
__global__ void __launch_bounds__(256)
lsm_collect_kernel(const float* partial, int nchunks, int trials, double inv_n, float* per_trial,
                   double* out) {
  grid_dependency();
  __shared__ double part[8][kLsmStats][33];
  __shared__ double sh[2 * kLsmCols][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double s1[kLsmCols], s2[kLsmCols];
#pragma unroll
  for (int c = 0; c < kLsmCols; ++c) s1[c] = s2[c] = 0.0;
  for (int t0 = (int)blockIdx.x * 32; t0 < trials; t0 += (int)gridDim.x * 32) {
    const int t = t0 + lane;
    double a[kLsmStats] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if (t < trials)
      for (int y = w; y < nchunks; y += 8)
#pragma unroll
        for (int i = 0; i < kLsmStats; ++i) a[i] += (double)ldg(partial + ((size_t)y * kLsmStats + i) * trials + t);
#pragma unroll
    for (int i = 0; i < kLsmStats; ++i) part[w][i][lane] = a[i];
    __syncthreads();
    if (w == 0 && t < trials) {
      double x[kLsmCols];
#pragma unroll
      for (int i = 0; i < kLsmStats; ++i) {
        double v = 0.0;
        for (int k = 0; k < 8; ++k) v += part[k][i][lane];
        const float f = (float)(v * inv_n);
        per_trial[(size_t)t * kLsmStats + i] = f;
        x[i] = (double)f;
      }
      x[6] = x[0] - x[1];
      x[7] = x[2] - x[3];
#pragma unroll
      for (int c = 0; c < kLsmCols; ++c) { s1[c] += x[c]; s2[c] += x[c] * x[c]; }
    }
    __syncthreads();
  }
  if (w == 0)
#pragma unroll
    for (int c = 0; c < kLsmCols; ++c) { sh[2 * c][lane] = s1[c]; sh[2 * c + 1][lane] = s2[c]; }
  __syncthreads();
  if (threadIdx.x < 2 * kLsmCols) {
    double v = 0.0;
    for (int k = 0; k < 32; ++k) v += sh[threadIdx.x][k];
    out[(size_t)blockIdx.x * 2 * kLsmCols + threadIdx.x] = v;
  }
}

// How a call is cut: blocks of up to 256 trials by chunks of rows, about seven blocks per SM (one wave
// of the eight that fit) where the rows allow it.  Where a chunk is one row and that leaves an eighth of the threads or
// fewer, each row's groups of classes are cut too, into parts of at least 16 groups; a block takes as many parts of a
// row as make it 256 threads, the rest go over nranges blocks.  Thread per trial and so: 16 x 8192, 64 trials 637 and
// 70 us; 16 x 512, 256 trials 71 and 47; 16 x 4096, 1024 trials (an eighth and less) 380 and 182; 64 x 512, 1024 (a quarter)
// 106 and 112.
struct LsmPlan {
  int threads, tblocks, rows_per_chunk, nchunks, cblocks;
  int parts, per, nranges;                                          // nranges 0: classes are not cut
  LsmPlan(int rows, int classes, int trials) {
    threads = trials >= kLsmThreads ? kLsmThreads : (trials + 31) / 32 * 32;
    tblocks = (trials + threads - 1) / threads;
    int want = (kNumSMs * 7 + tblocks - 1) / tblocks;
    if (want > rows) want = rows;
    rows_per_chunk = (rows + want - 1) / want;
    nchunks = (rows + rows_per_chunk - 1) / rows_per_chunk;
    cblocks = (trials + 31) / 32;
    if (cblocks > kNumSMs) cblocks = kNumSMs;
    const int groups = classes / 4;
    int64_t cuts = (int64_t)kNumSMs * 7 * kLsmThreads / ((int64_t)tblocks * threads * rows);   // of the threads wanted over those there
    parts = 1; per = groups; nranges = 0;
    if (rows_per_chunk > 1 || cuts < 8 || groups < 32) return;
    if (cuts > groups / 16) cuts = groups / 16;
    parts = kLsmThreads / threads < cuts ? kLsmThreads / threads : (int)cuts;
    nranges = (int)((cuts + parts - 1) / parts);
    per = (groups + nranges * parts - 1) / (nranges * parts);
  }
  // floats: the chunks' terms, and before them the ranges' sums
  size_t partials(int trials) const { return (size_t)nchunks * kLsmStats * trials; }
  size_t ranges(int trials) const { return (size_t)nchunks * nranges * 4 * trials; }
};

}  // namespace bsp

using namespace bsp;

extern "C" {

size_t bsp_lsm_check_workspace_bytes(int rows, int classes, int trials) {
  if (rows <= 0 || classes <= 0 || trials <= 0) return 0;
  const LsmPlan plan(rows, classes, trials);
  return round_up((size_t)rows * classes * sizeof(float4), 256) +
         round_up(plan.ranges(trials) * sizeof(float), 256) + round_up(plan.partials(trials) * sizeof(float), 256) +
         round_up((size_t)trials * kLsmStats * sizeof(float), 256) + (size_t)kNumSMs * 2 * kLsmCols * sizeof(double);
}

int bsp_lsm_check(const float* logits, const int32_t* target, int rows, int classes, float eps, int trials, uint64_t seed,
                  uint32_t tensor_id, float* per_trial, bsp_lsm_stat_t* stats, void* ws, size_t ws_bytes, void* stream) {
  if (!logits || !target || !stats || rows <= 0 || classes <= 0 || trials < 2 || !(eps > 0.f) || tensor_id >= (1u << 24))
    return BSP_ERR_ARG;
  if (classes % 4 != 0 || classes > 32 * 4 * kLsmThreads / 4) return BSP_ERR_UNSUPPORTED;   // <= 32 classes per thread
  if (!aligned16(logits)) return BSP_ERR_ALIGN;
  if (!ws || ws_bytes < bsp_lsm_check_workspace_bytes(rows, classes, trials) || (reinterpret_cast<uintptr_t>(ws) & 255u))
    return BSP_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t n = (size_t)rows * classes;
  const LsmPlan plan(rows, classes, trials);
  char* base = reinterpret_cast<char*>(ws);
  float4* table = reinterpret_cast<float4*>(base);
  base += round_up(n * sizeof(float4), 256);
  float* ranges = reinterpret_cast<float*>(base);
  base += round_up(plan.ranges(trials) * sizeof(float), 256);
  float* partial = reinterpret_cast<float*>(base);
  base += round_up(plan.partials(trials) * sizeof(float), 256);
  float* pt = per_trial ? per_trial : reinterpret_cast<float*>(base);
  base += round_up((size_t)trials * kLsmStats * sizeof(float), 256);
  double* sums = reinterpret_cast<double*>(base);
  bsp_key_t k;
  k.seed = seed; k.tensor_id = tensor_id; k.stream = BSP_STREAM_FORWARD; k.draw = 0; k.reserved = 0;
  const PhiloxKey kr = make_key(k);
  k.stream = BSP_STREAM_GAIN;                                       // the independent copy's own stream
  const PhiloxKey kc = make_key(k);
  launch_kernel(lsm_prep_kernel, (unsigned)rows, kLsmThreads, 0, st, logits, classes, eps, table);
  BSP_LAUNCH_CHECK();
  if (plan.nranges) {
    launch_kernel(lsm_range_kernel, dim3((unsigned)plan.tblocks, (unsigned)(rows * plan.nranges)), dim3(plan.threads, plan.parts), 0, st,
                  table, plan.nranges, plan.per, classes, kr, kc, trials, ranges);
    launch_kernel(lsm_join_kernel, dim3((unsigned)((trials + 31) / 32), (unsigned)rows), 256, 0, st, ranges, plan.nranges, classes, eps,
                  trials, partial);
  } else {
    launch_kernel(lsm_trial_kernel, dim3((unsigned)plan.tblocks, (unsigned)plan.nchunks), plan.threads, 0, st,
                  table, rows, plan.rows_per_chunk, classes, eps, kr, kc, trials, partial);
  }
  BSP_LAUNCH_CHECK();
  launch_kernel(lsm_collect_kernel, (unsigned)plan.cblocks, 256, 0, st, partial, plan.nchunks, trials, 1.0 / ((double)rows * classes), pt, sums);
  BSP_LAUNCH_CHECK();
  double parts[kNumSMs * 2 * kLsmCols], host[2 * kLsmCols];
  const size_t bytes = (size_t)plan.cblocks * 2 * kLsmCols * sizeof(double);
  BSP_CHECK_CUDA(cudaMemcpyAsync(parts, sums, bytes, cudaMemcpyDeviceToHost, st));
  count_d2h(bytes);
  BSP_CHECK_CUDA(cudaStreamSynchronize(st));
  for (int c = 0; c < 2 * kLsmCols; ++c) {
    host[c] = 0.0;
    for (int k = 0; k < plan.cblocks; ++k) host[c] += parts[k * 2 * kLsmCols + c];
  }
  for (int c = 0; c < kLsmCols; ++c) {
    const double mean = host[2 * c] / trials;
    double var = (host[2 * c + 1] - host[2 * c] * mean) / (trials - 1);
    if (var < 0) var = 0;
    const double se = sqrt(var / trials);
    stats[c].mean = mean;
    stats[c].se = se;
    stats[c].z = se > 0 ? fabs(mean) / se : (mean == 0 ? 0.0 : INFINITY);
  }
  return BSP_OK;
}

}  // extern "C"
