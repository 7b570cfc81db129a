// split_aux.cu -- tour preparation, feasible-arc counting, the deterministic
// FP64 scenario mean, and the Split adjoint's backtrack / gradient assembly.
#include "dependent.cuh"
#include "sdp_internal.cuh"

namespace sdp {

// Travel cost c(a,b).  Coordinates: FP32 Euclidean distance with IEEE
// rounding at every step (no contraction, correctly rounded sqrt), so every
// launch and every kernel sees the same bits.  Matrix: dist[a*(n+1)+b].
__device__ __forceinline__ float travel(const float* coords, const float* dist,
                                        int n, int a, int b) {
  if (dist) return __ldg(dist + (size_t)a * (n + 1) + b);
  float dx = __fsub_rn(__ldg(coords + 2 * a), __ldg(coords + 2 * b));
  float dy = __fsub_rn(__ldg(coords + 2 * a + 1), __ldg(coords + 2 * b + 1));
  return __fsqrt_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)));
}

// One CTA per tour (Sec. 2 Instantiation A: the route cost W(p,i) depends on
// the tour only through c(0,s_{p+1}), the consecutive arcs and c(s_i,0)).
__global__ void __launch_bounds__(256) tour_prep_kernel(
    const int32_t* __restrict__ tour, int n, const float* __restrict__ coords,
    const float* __restrict__ dist, TourPrep prep, uint32_t* status,
    CallCounters counters, LoadSample sample) {
  __shared__ double red[256];
  __shared__ uint32_t load[kLoadSample];
  static_assert(kLoadSample == 256 / 32, "a warp each");
  dep_launch();
  if (sample.below) {
    const int j = threadIdx.x >> 5;
    const int32_t* q = sample.demands + (sample.S - 1) * j / (kLoadSample - 1) * n;
    uint32_t v = 0u;
#pragma unroll 8
    for (int k = threadIdx.x & 31; k < n; k += 32) v += (uint32_t)min(max(__ldg(q + k), 0), sample.Q + 1);
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) load[j] = v;
  }
  if (threadIdx.x == 0) {  // the call's counters, for the kernels that follow
    if (counters.flagged) *counters.flagged = 0u;
    if (counters.tiles) *counters.tiles = 0ull;
    if (counters.mean) *counters.mean = 0u;
  }
  if (counters.routes)
    for (int k = threadIdx.x; k < 2 * n + 1; k += blockDim.x) counters.routes[k] = 0ull;
  double acc = 0.0;
  bool bad = false;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    int si = __ldg(tour + i);
    if (si < 1 || si > n) { bad = true; si = 1; }
    float c0 = travel(coords, dist, n, 0, si);
    float ce = travel(coords, dist, n, si, 0);
    float e = 0.f;
    if (i > 0) {
      int sp = __ldg(tour + i - 1);
      if (sp < 1 || sp > n) sp = 1;
      e = travel(coords, dist, n, sp, si);
      acc += (double)e;  // D(n) = sum of the n-1 consecutive arcs
    }
    StepRec r;
    r.col = (uint32_t)(si - 1);
    r.a = __fsub_rn(c0, e);
    r.ce = ce;
    r.pad = 0u;
    prep.rec[i] = r;
    prep.cols[i] = (uint16_t)(si - 1);
  }
  if (bad) atomicOr(status, SDP_FLAG_DEVICE_CHECK);
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    *prep.Dn = red[0];
    if (sample.below) {
      uint32_t v = 0u;
      for (int j = 0; j < kLoadSample; ++j) v += load[j];
      *sample.out = v < sample.below ? 1u : 0u;
    }
  }
}

void launch_tour_prep(const int32_t* tour, int n, const float* coords,
                      const float* dist, TourPrep prep, uint32_t* status,
                      CallCounters counters, cudaStream_t st, LoadSample sample) {
  tour_prep_kernel<<<1, 256, 0, st>>>(tour, n, coords, dist, prep, status, counters, sample);
}

// ----------------------------------------------------------- arc counting
// Feasible arcs of scenario s: sum_i (i - pmin(i)), pmin(i) the smallest p
// with load(s_{p+1..i}) <= Q (two pointers; the load is monotone).
__global__ void __launch_bounds__(256) count_arcs_kernel(
    int n, int Q, int64_t S, const StepRec* __restrict__ rec,
    const int32_t* __restrict__ demands, int64_t* __restrict__ arcs,
    unsigned long long* total) {
  unsigned long long mine = 0;
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < S;
       s += (int64_t)gridDim.x * blockDim.x) {
    const int32_t* q = demands + s * n;
    int64_t W = 0, cnt = 0;
    int pm = 0;
    for (int i = 1; i <= n; ++i) {
      W += max(__ldg(q + __ldg(&rec[i - 1].col)), 0);
      while (W > Q && pm < i) {
        ++pm;
        W -= max(__ldg(q + __ldg(&rec[pm - 1].col)), 0);
      }
      cnt += i - pm;
    }
    if (arcs) arcs[s] = cnt;
    mine += (unsigned long long)cnt;
  }
  if (total) {
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, o);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(total, mine);
  }
}

void launch_count_arcs(int n, int Q, int64_t S, const StepRec* rec,
                       const int32_t* demands, int64_t* arcs,
                       unsigned long long* total, int grid, cudaStream_t st) {
  count_arcs_kernel<<<grid, 256, 0, st>>>(n, Q, S, rec, demands, arcs, total);
}

// ------------------------------------------------------------- FP64 mean
// Eight values as the pair of floats (their rounded sum, the sum of its rounding
// errors by Knuth's two-sum) and then one FP64 number.  GB300 has few FP64 units
// (a conversion and an addition per value took 48 us for 1,025 x 10^4 values;
// 0.25 of each per value here).  The pair is taken only where it is exact:
// where the largest magnitude M and the least one above zero, m, are at most 19
// binary exponents apart.  With u the last place of m, all sums and errors are
// multiples of u; a partial sum is at most 8 M, so the seven errors add up to
// at most 28 last places of M <= 2^24 u, which a float holds, and the two parts
// to 46 bits, which a double holds.  Other groups (a spread of 2^20 or more, an
// infinity, a NaN, a sum beyond the largest float) are added in FP64.
__device__ __forceinline__ double sum8(const float* v) {
  float hi = v[0], lo = 0.f, big = fabsf(v[0]);
  uint32_t least = 2u * __float_as_uint(v[0]) - 1u;  // magnitudes in order, zero as the last
#pragma unroll
  for (int k = 1; k < 8; ++k) {
    const float s = __fadd_rn(hi, v[k]);
    const float t = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(v[k], t)));
    hi = s;
    big = fmaxf(big, fabsf(v[k]));
    least = min(least, 2u * __float_as_uint(v[k]) - 1u);
  }
  // (all zeros: least is the largest word, and the test holds)
  if (fabsf(hi) <= 3.0e38f && (__float_as_uint(big) >> 23) <= (least >> 24) + 19u)
    return (double)hi + (double)lo;
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < 8; ++k) acc += (double)v[k];
  return acc;
}

// sum of red[0 .. 256) in the order of a binary tree (valid in thread 0; the
// last five levels within a warp)
__device__ __forceinline__ double block_tree(double* red) {
  for (int w = 128; w > 16; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  double v = red[threadIdx.x & 31];
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) v += __shfl_down_sync(0xffffffffu, v, w);
  return v;
}

// sum of x[lo .. hi) over the CTA's 256 threads, in a fixed order (every
// thread takes x[lo + thread + 256 j]; the result is valid in thread 0).  A
// thread's last values are a group filled up with zeros: one load latency and
// one FP64 addition instead of up to seven of each (1,025 x 10^4 values:
// 24.8 -> 19.0 us; one block of 1,000: 5.1 -> 4.3).
__device__ double block_sum(const float* x, int64_t lo, int64_t hi, double* red) {
  double acc = 0.0;
  for (int64_t k = lo + threadIdx.x; k < hi; k += 8 * 256) {
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = k + j * 256 < hi ? x[k + j * 256] : 0.f;
    acc += sum8(v);
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  return block_tree(red);
}

// One launch: block b sums its contiguous chunk, the block that finishes last
// (counter, zero at launch) the partial sums in their order, so the result
// does not depend on scheduling (bit-reproducible).  One block needs no
// counter.
__global__ void __launch_bounds__(256) mean_kernel(const float* x, int64_t count, double* partial, uint32_t* counter, double* out) {
  __shared__ double red[256];
  __shared__ bool last;
  dep_wait();
  const int64_t chunk = (count + gridDim.x - 1) / gridDim.x;
  const int64_t lo = blockIdx.x * chunk;
  double total = block_sum(x, lo, min(count, lo + chunk), red);
  if (gridDim.x > 1) {
    if (threadIdx.x == 0) {
      partial[blockIdx.x] = total;
      __threadfence();
      last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    red[threadIdx.x] = threadIdx.x < gridDim.x ? __ldcg(partial + threadIdx.x) : 0.0;
    __syncthreads();
    total = block_tree(red);
  }
  if (threadIdx.x == 0) *out = count > 0 ? total / (double)count : 0.0;
}

// up to 4,096 values a block, at most 256 blocks (the counter sits behind the
// partial sums: mean_counter)
void launch_mean(const float* x, int64_t count, double* partial, double* out,
                 cudaStream_t st) {
  const int64_t blocks = (count + 4095) / 4096;
  const int grid = blocks < 1 ? 1 : (int)imin64(blocks, 256);
  launch_dependent(true, mean_kernel, grid, 256, 0, st, x, count, partial, mean_counter(partial), out);
}

// ------------------------------------------------------------------ adjoint
// Backtrack of stored predecessors: for each scenario walk i = n -> pred(i)
// -> ... -> 0; route p+1..i starts at position p+1 and ends at position i.
// hist[0..n) = starts, hist[n..2n) = ends, hist[2n] = scenarios counted.
template <typename PT>
__global__ void __launch_bounds__(256) backtrack_hist_kernel(
    int n, int64_t S, const PT* __restrict__ pred,
    unsigned long long* __restrict__ hist, uint32_t* status) {
  extern __shared__ unsigned int sh[];
  const bool use_smem = (2 * n + 1) * 4 <= 48 * 1024;
  if (use_smem)
    for (int k = threadIdx.x; k < 2 * n + 1; k += blockDim.x) sh[k] = 0u;
  __syncthreads();
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < S;
       s += (int64_t)gridDim.x * blockDim.x) {
    const PT* ps = pred + s * n;
    bool ok = true;
    for (int i = n; i > 0;) {
      long long p = (long long)ps[i - 1];
      if (sizeof(PT) == 2 && p == 0xFFFF) p = -1;
      if (p < 0 || p >= i) { ok = false; break; }
      i = (int)p;
    }
    if (!ok) continue;
    for (int i = n; i > 0;) {
      int p = (int)ps[i - 1];
      if (use_smem) {
        atomicAdd(&sh[p], 1u);
        atomicAdd(&sh[n + i - 1], 1u);
      } else {
        atomicAdd(&hist[p], 1ull);
        atomicAdd(&hist[n + i - 1], 1ull);
      }
      i = p;
    }
    if (use_smem) atomicAdd(&sh[2 * n], 1u);
    else atomicAdd(&hist[2 * n], 1ull);
  }
  __syncthreads();
  if (use_smem)
    for (int k = threadIdx.x; k < 2 * n + 1; k += blockDim.x)
      if (sh[k]) atomicAdd(&hist[k], (unsigned long long)sh[k]);
}

void launch_backtrack_hist(int n, int64_t S, const void* pred, int pred_dtype,
                           unsigned long long* hist, uint32_t* status,
                           cudaStream_t st) {
  int grid = 2 * num_sms();
  size_t smem = (2 * (size_t)n + 1) * 4 <= 48 * 1024 ? (2 * (size_t)n + 1) * 4 : 0;
  if (pred_dtype == SDP_PRED_U16)
    backtrack_hist_kernel<uint16_t><<<grid, 256, smem, st>>>(
        n, S, (const uint16_t*)pred, hist, status);
  else
    backtrack_hist_kernel<int32_t><<<grid, 256, smem, st>>>(
        n, S, (const int32_t*)pred, hist, status);
}

// Each route p+1..i uses (0,s_{p+1}), (s_k,s_{k+1}) for p+1 <= k < i and
// (s_i,0).  Position k either ends its route (arc (s_k,0)) or continues to
// s_{k+1}: continue(k) = counted scenarios - ends(k).  Every entry of the
// matrix is written once: a block inverts the tour in shared memory (position
// of each customer, 0 where the tour does not hold it) and takes whole rows.
// GT: the type of the incoming gradient, taken as a float.
template <typename GT>
__global__ void __launch_bounds__(256) grad_kernel(int n, int64_t S, const int32_t* __restrict__ tour,
                                                   const unsigned long long* __restrict__ hist,
                                                   const GT* __restrict__ grad_mean,
                                                   float* __restrict__ grad, int64_t* hist_out) {
  extern __shared__ int32_t pos[];  // [n + 1], 1-based
  const int m = n + 1;
  for (int k = threadIdx.x; k < m; k += blockDim.x) pos[k] = 0;
  __syncthreads();
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const int sk = __ldg(tour + k);
    if (sk >= 1 && sk <= n) pos[sk] = k + 1;  // (an invalid entry is flagged by tour_prep)
  }
  __syncthreads();
  const bool any = n > 0 && S > 0;
  const double scale = any ? (double)(float)__ldg(grad_mean) / (double)S : 0.0;
  const unsigned long long used = any ? hist[2 * n] : 0ull;
  for (int a = blockIdx.x; a < m; a += gridDim.x) {
    const int pa = pos[a];
    const unsigned long long ends = any && pa ? hist[n + pa - 1] : 0ull;
    for (int b = threadIdx.x; b < m; b += blockDim.x) {
      const int pb = pos[b];
      float g = 0.f;
      if (any) {
        if (a == 0) {
          if (pb) g = (float)((double)hist[pb - 1] * scale);
        } else if (pa) {
          if (b == 0) g = (float)((double)ends * scale);
          else if (pb == pa + 1) g = (float)((double)(used - ends) * scale);
        }
      }
      grad[(size_t)a * m + b] = g;
    }
  }
  if (hist_out && blockIdx.x == 0 && any)
    for (int k = threadIdx.x; k < 2 * n; k += blockDim.x) hist_out[k] = (int64_t)hist[k];
}

// The same over a zeroed matrix, for tours whose inverse does not fit shared
// memory (n > 58,000): position k writes its own arcs, which are distinct
// because the tour is a permutation.
template <typename GT>
__global__ void __launch_bounds__(256) grad_scatter_kernel(int n, int64_t S,
                                                           const int32_t* __restrict__ tour,
                                                           const unsigned long long* __restrict__ hist,
                                                           const GT* __restrict__ grad_mean,
                                                           float* __restrict__ grad, int64_t* hist_out) {
  const double scale = (double)(float)__ldg(grad_mean) / (double)S;
  const unsigned long long used = hist[2 * n];
  const int m = n + 1;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    const int sk = __ldg(tour + k);
    if (sk < 1 || sk > n) continue;
    const unsigned long long st = hist[k], en = hist[n + k];
    grad[(size_t)sk] = (float)((double)st * scale);
    grad[(size_t)sk * m] = (float)((double)en * scale);
    if (k + 1 < n) {
      const int sn = __ldg(tour + k + 1);
      if (sn >= 1 && sn <= n) grad[(size_t)sk * m + sn] = (float)((double)(used - en) * scale);
    }
    if (hist_out) {
      hist_out[k] = (int64_t)st;
      hist_out[n + k] = (int64_t)en;
    }
  }
}

namespace {
template <typename GT>
int launch_grad_t(int n, int64_t S, const int32_t* tour, const unsigned long long* hist,
                  const GT* grad_mean, float* grad, int64_t* hist_out, cudaStream_t st) {
  const size_t smem = (size_t)(n + 1) * 4;
  if (smem > 227 * 1024) {
    const cudaError_t e = cudaMemsetAsync(grad, 0, (size_t)(n + 1) * (size_t)(n + 1) * sizeof(float), st);
    if (e != cudaSuccess) return (int)e;
    if (S > 0)
      grad_scatter_kernel<GT><<<(n + 255) / 256, 256, 0, st>>>(n, S, tour, hist, grad_mean, grad, hist_out);
    return (int)cudaGetLastError();
  }
  if (smem > 48 * 1024) {
    const cudaError_t e =
        cudaFuncSetAttribute(grad_kernel<GT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
  }
  const int grid = (int)imin64(n + 1, 4 * (int64_t)num_sms());
  grad_kernel<GT><<<grid, 256, smem, st>>>(n, S, tour, hist, grad_mean, grad, hist_out);
  return (int)cudaGetLastError();
}
}  // namespace

int launch_grad(int n, int64_t S, const int32_t* tour, const unsigned long long* hist,
                const void* grad_mean, bool grad_is_double, float* grad, int64_t* hist_out,
                cudaStream_t st) {
  return grad_is_double
             ? launch_grad_t(n, S, tour, hist, (const double*)grad_mean, grad, hist_out, st)
             : launch_grad_t(n, S, tour, hist, (const float*)grad_mean, grad, hist_out, st);
}

}  // namespace sdp

namespace sdp {

// ------------------------------------------------------------ batched Split
// Tour prep for every tour of a batch: one CTA per tour, same arithmetic as
// tour_prep_kernel.  With a.prefix, tour 0's records are made alongside, to
// count the leading ones that the tour shares with it.
__global__ void __launch_bounds__(256) batch_prep_kernel(BatchPrepArgs a) {
  __shared__ double red[256];
  const int b = blockIdx.x;
  const int n = a.n[b];
  const int32_t* tour = a.tours + a.tour_off[b];
  const float* coords = a.coords + 2 * a.coord_off[b];
  StepRec* rec = a.rec + a.rec_off[b];
  if (b == 0 && threadIdx.x == 0) {
    *a.counter = 0ull;
    *a.fb_count = 0u;
  }
  __shared__ int same;
  if (threadIdx.x == 0) same = n;
  __syncthreads();
  double acc = 0.0;
  bool bad = false;
  int differs = n;
  // record i of a tour, and its arc from the position before
  auto record = [&](const int32_t* t, const float* xy, int i, float* arc) -> StepRec {
    int si = __ldg(t + i);
    if (si < 1 || si > n) { bad = true; si = 1; }
    const float c0 = travel(xy, nullptr, n, 0, si);
    const float ce = travel(xy, nullptr, n, si, 0);
    float e = 0.f;
    if (i > 0) {
      int sp = __ldg(t + i - 1);
      if (sp < 1 || sp > n) sp = 1;
      e = travel(xy, nullptr, n, sp, si);
    }
    *arc = e;
    StepRec r;
    r.col = (uint32_t)(si - 1);
    r.a = __fsub_rn(c0, e);
    r.ce = ce;
    r.pad = 0u;
    return r;
  };
  const int32_t* tour0 = a.tours + a.tour_off[0];
  const float* coords0 = a.coords + 2 * a.coord_off[0];
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    float e;
    const StepRec r = record(tour, coords, i, &e);
    if (i > 0) acc += (double)e;
    rec[i] = r;
    if (a.prefix && b > 0 && differs == n) {
      const StepRec r0 = record(tour0, coords0, i, &e);
      if (r.col != r0.col || __float_as_uint(r.a) != __float_as_uint(r0.a) ||
          __float_as_uint(r.ce) != __float_as_uint(r0.ce))
        differs = i;
    }
  }
  if (bad) atomicOr(a.status, SDP_FLAG_DEVICE_CHECK);
  if (differs < n) atomicMin(&same, differs);
  red[threadIdx.x] = acc;
  __syncthreads();
  if (a.prefix && threadIdx.x == 0) a.prefix[b] = same;
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) a.Dn[b] = red[0];
}

void launch_batch_prep(const BatchPrepArgs& a, int B, cudaStream_t st) {
  batch_prep_kernel<<<B, 256, 0, st>>>(a);
}

// Per-tour FP64 mean of costs[b*S .. b*S+S): one CTA per tour, fixed order.
__global__ void __launch_bounds__(256) batch_mean_kernel(const float* costs, int64_t S,
                                                         double* means) {
  __shared__ double red[256];
  dep_wait();
  const double total = block_sum(costs + (int64_t)blockIdx.x * S, 0, S, red);
  if (threadIdx.x == 0) means[blockIdx.x] = total / (double)S;
}

void launch_batch_means(const float* costs, int B, int64_t S, double* means, cudaStream_t st) {
  launch_dependent(true, batch_mean_kernel, B, 256, 0, st, costs, S, means);
}

// Feasible arcs of every (tour, scenario) of a batch.
__global__ void __launch_bounds__(256) batch_count_kernel(BatchPrepArgs a, int B, int64_t S,
                                                          int Q, const int64_t* dem_off,
                                                          const int32_t* demands,
                                                          unsigned long long* total) {
  unsigned long long mine = 0;
  const int64_t N = (int64_t)B * S;
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < N;
       g += (int64_t)gridDim.x * blockDim.x) {
    const int b = (int)(g / S);
    const int64_t s = g - (int64_t)b * S;
    const int n = a.n[b];
    const StepRec* rec = a.rec + a.rec_off[b];
    const int32_t* q = demands + dem_off[b] + s * n;
    int64_t W = 0, cnt = 0;
    int pm = 0;
    for (int i = 1; i <= n; ++i) {
      W += max(__ldg(q + __ldg(&rec[i - 1].col)), 0);
      while (W > Q && pm < i) {
        ++pm;
        W -= max(__ldg(q + __ldg(&rec[pm - 1].col)), 0);
      }
      cnt += i - pm;
    }
    mine += (unsigned long long)cnt;
  }
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, o);
  if ((threadIdx.x & 31) == 0 && mine) atomicAdd(total, mine);
}

void launch_batch_count(const BatchPrepArgs& a, int B, int64_t S, int Q, const int64_t* dem_off,
                        const int32_t* demands, unsigned long long* total, cudaStream_t st) {
  batch_count_kernel<<<8 * num_sms(), 256, 0, st>>>(a, B, S, Q, dem_off, demands, total);
}

}  // namespace sdp
