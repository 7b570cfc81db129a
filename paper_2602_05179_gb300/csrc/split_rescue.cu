// split_rescue.cu -- recomputation of the scenarios a deque kernel flagged
// (its deque outgrew the ring, or its staging could not hold a demand), one
// warp per scenario, for sm_103a.
//
// Eq. eqdpA in the K-form of sdp_internal.cuh: K(i) = min over p < i of
// psi(p) (+ beta per unit of load above Q with soft capacity, p within the
// capacity window otherwise) + ce_i, psi(p) = K(p) + a_{p+1}.  Positions go 32
// at a time, one per lane.  The candidates before the block are known: each
// lane takes the minimum over its own, no lane waiting for another.  Those
// inside it are pushed: position u's psi, final once the positions before it
// have been pushed, goes to every lane by one shuffle, and the lanes above
// whose window holds it take the minimum.  So a position costs one shuffle
// and half a dozen operations on the dependent chain, where spreading its
// candidates over the lanes and reducing them cost a chain of ten shuffles
// and several loads: 112 us for the flagged scenarios of an n = 333 call with
// that form, 25 us with this one.
//   Soft capacity lets every earlier p compete.  A lane scans them downward
// and stops where even the least psi so far (PM, a running minimum) with the
// penalty reached exceeds its best: penalties only grow as p falls and
// rounding is monotone, so no later candidate is below or ties.  With the
// one-thread-per-scenario plain kernel, which relaxes every pair, the flagged
// scenarios of an n = 500 call took about 14.7 ms, here 0.1 ms.
//   The adjoint's flagged scenarios also count their routes: predecessors in
// shared memory, walked back from position n.
// The FP32 arithmetic is the plain kernel's, operation for operation (psi,
// the penalty added to it, the minimum with ties to the smallest p, then
// + ce_i), so the results are the same bits whichever kernel ran.  With hard
// capacity demands are clamped to [0, Q+1]: a route holding a demand above Q
// is infeasible whatever its value.
#include <math_constants.h>

#include <algorithm>

#include "dependent.cuh"
#include "sdp_internal.cuh"

namespace sdp {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRescueMaxWarps = 8;                 // warps per CTA
constexpr size_t kRescueCtaBudget = 96u * 1024u;   // shared memory per CTA we aim for
constexpr size_t kRescueWarpMax = 200u * 1024u;    // one warp's rows at most

// per warp, [n+1] each: prefix loads, psi; soft: the running minimum of psi;
// route counts: predecessors
size_t rescue_per_warp(int n_max, bool soft, bool hist) {
  return (size_t)(8 + (soft ? 4 : 0) + (hist ? 4 : 0)) * ((size_t)n_max + 1);
}

// PT: predecessor type; HIST: count route starts / ends into a.hist (costs only
// where a.cost is set)
template <typename PT, bool BATCH, bool SOFT, bool HIST>
__global__ void __launch_bounds__(kRescueMaxWarps * 32) split_rescue_kernel(RescueArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  const int wpb = blockDim.x >> 5;
  dep_launch();
  dep_wait();
  const int64_t nwork = (int64_t)(*a.fb_count);
  const int64_t nw = (int64_t)gridDim.x * wpb;
  constexpr int kArrays = 2 + (SOFT ? 1 : 0) + (HIST ? 1 : 0);
  const int64_t stride = (int64_t)a.n_max + 1;
  int32_t* L = reinterpret_cast<int32_t*>(smem) + (int64_t)wib * kArrays * stride;
  float* psi = reinterpret_cast<float*>(L + stride);
  float* PM = psi + stride;                                        // SOFT
  int32_t* prs = reinterpret_cast<int32_t*>(psi + (SOFT ? 2 : 1) * stride);  // HIST
  const int Q = a.Q;
  bool neg = false, inf_any = false;
  for (int64_t w = (int64_t)blockIdx.x * wpb + wib; w < nwork; w += nw) {
    int n;
    const StepRec* rec;
    const int32_t* q;
    double Dn;
    int64_t out;
    if (BATCH) {
      const unsigned long long g = a.fb_list[w];
      const int b = (int)(g / (unsigned long long)a.S);
      const int64_t s = (int64_t)(g - (unsigned long long)b * (unsigned long long)a.S);
      n = a.n[b];
      rec = a.rec + a.rec_off[b];
      q = a.demands + a.dem_off[b] + s * n;
      Dn = a.Dn[b];
      out = (int64_t)g;
    } else {
      const int64_t s = (int64_t)a.fb_list1[w];
      n = a.n1;
      rec = a.rec;
      q = a.demands + s * n;
      Dn = n > 0 ? *a.Dn : 0.0;
      out = s;
    }
    __syncwarp();  // the previous scenario's reads of the rows are done
    // demands by customer (staged in psi), then prefix loads in tour order
    int32_t* stage = reinterpret_cast<int32_t*>(psi);
#pragma unroll 4
    for (int k = lane; k < n; k += 32) stage[k] = __ldg(q + k);
    __syncwarp();
    int carry = 0;
    float total = 0.f;  // soft: the load as a float, to see sums beyond 2^31
    if (lane == 0) L[0] = 0;
#pragma unroll 2
    for (int i0 = 1; i0 <= n; i0 += 32) {
      const int i = i0 + lane;
      int v = 0;
      if (i <= n) {
        const int raw = stage[__ldg(&rec[i - 1].col)];
        neg |= raw < 0;
        v = SOFT ? max(raw, 0) : min(max(raw, 0), Q + 1);
        if (SOFT) total += (float)v;
      }
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(kFull, v, d);
        if (lane >= d) v += t;
      }
      if (i <= n) L[i] = carry + v;
      carry += __shfl_sync(kFull, v, 31);
    }
    // a load that wraps (the plain kernel's does too) is not monotone
    const bool wraps = SOFT && __any_sync(kFull, total > 6.0e7f);
    __syncwarp();
    const float psi0 = n > 0 ? __fadd_rn(0.f, __ldg(&rec[0].a)) : 0.f;
    if (lane == 0) {
      psi[0] = psi0;
      if (SOFT) PM[0] = psi0;
    }
    __syncwarp();
    float pm_carry = psi0;  // soft: the least psi so far
    float Kn = 0.f;
    int lo = 0;             // hard: this lane's window start, which only grows
    for (int b0 = 0; b0 < n; b0 += 32) {
      const int i = b0 + 1 + lane;
      const bool on = i <= n;
      const int ic = min(i, n);
      const int Li = L[ic];
      const float ce = __ldg(&rec[ic - 1].ce);
      const float an = i < n ? __ldg(&rec[i].a) : 0.f;
      float m = CUDART_INF_F;
      int bp = -1;
      // ---- candidates up to position b0
      uint32_t take = (1u << lane) - 1u;  // the positions of the block below this one
      if (!SOFT) {
        int hi = ic;
        while (lo < hi) {  // the smallest p with L(i) - L(p) <= Q (i itself: none)
          const int mid = (lo + hi) >> 1;
          if (Li - L[mid] <= Q) hi = mid; else lo = mid + 1;
        }
#pragma unroll 4
        for (int p = lo; p <= b0; ++p) {
          const float x = psi[p];
          if (x < m) {
            m = x;
            bp = p;
          }
        }
        const int first = lo - b0 - 1;  // window starts inside the block
        if (first > 0) take = first >= 32 ? 0u : take & ~((1u << first) - 1u);
      } else {
#pragma unroll 2
        for (int p = b0; p >= 0; --p) {
          const int load = Li - L[p];
          float x = psi[p];
          if (load > Q) {
            const float pen = __fmul_rn(a.beta, (float)(load - Q));
            if (!wraps && __fadd_rn(PM[p], pen) > m) break;
            x = __fadd_rn(x, pen);
          }
          if (x <= m) {  // p descends: "<=" keeps the smallest p on ties
            m = x;
            bp = p;
          }
        }
        if (m == CUDART_INF_F) bp = -1;
      }
      // ---- the block's own positions, pushed in order
      __syncwarp();
      const int cnt = min(32, n - b0);
#pragma unroll
      for (int u = 0; u < 32; ++u) {
        // (lane u's minimum is final here; a position past n reaches no other)
        const float pu = __shfl_sync(kFull, __fadd_rn(__fadd_rn(m, ce), an), u);
        float x = pu;
        if (SOFT) {
          const int load = Li - L[min(b0 + 1 + u, n)];
          if (load > Q) x = __fadd_rn(x, __fmul_rn(a.beta, (float)(load - Q)));
        }
        if (((take >> u) & 1u) && x < m) {
          m = x;
          bp = b0 + 1 + u;
        }
      }
      const float K = __fadd_rn(m, ce);
      float v = __fadd_rn(K, an);
      if (on) psi[i] = v;
      if (SOFT) {
        v = on ? v : CUDART_INF_F;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) v = fminf(v, __shfl_up_sync(kFull, v, d));
        v = fminf(v, pm_carry);
        if (on) PM[i] = v;
        pm_carry = __shfl_sync(kFull, v, 31);
      }
      if (on) {
        if (HIST) prs[i] = bp;
        else if (!BATCH && a.pred) reinterpret_cast<PT*>(a.pred)[out * n + i - 1] = (PT)bp;
      }
      Kn = __shfl_sync(kFull, K, cnt - 1);
      __syncwarp();
    }
    const bool inf = n > 0 && Kn == CUDART_INF_F;
    inf_any |= inf;
    if (HIST) {
      if (lane == 0 && !inf) {
        for (int i = n; i > 0;) {
          const int p = prs[i];
          if (p < 0 || p >= i) break;
          atomicAdd(&a.hist[p], 1ull);
          atomicAdd(&a.hist[n + i - 1], 1ull);
          i = p;
        }
        atomicAdd(&a.hist[2 * n], 1ull);
      }
    }
    if (lane == 0 && (!HIST || a.cost)) {
      const float c = inf ? CUDART_INF_F : (float)((double)Kn + Dn);
      if (BATCH) a.costs[out] = c;
      else a.cost[out] = c;
    }
  }
  const bool any_neg = __any_sync(kFull, neg);
  if (lane == 0) {
    if (any_neg) atomicOr(a.status, SDP_FLAG_NEG_INPUT);
    if (inf_any) atomicOr(a.status, SDP_FLAG_INFEASIBLE);
  }
}

template <typename PT, bool BATCH, bool SOFT, bool HIST>
int launch_r(const RescueArgs& a, int wpb, size_t smem, int grid, cudaStream_t st) {
  auto k = split_rescue_kernel<PT, BATCH, SOFT, HIST>;
  if (smem > 48u * 1024u) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
  }
  return (int)launch_dependent(false, k, grid, wpb * 32, smem, st, a);
}

}  // namespace

bool rescue_supported(int n_max, bool soft, bool hist) {
  return n_max >= 0 && rescue_per_warp(n_max, soft, hist) <= kRescueWarpMax;
}

int launch_split_rescue(const RescueArgs& a, int64_t max_work, cudaStream_t st) {
  const bool hist = a.hist != nullptr;
  const size_t per = rescue_per_warp(a.n_max, a.soft != 0, hist);
  const int wpb = (int)std::min<size_t>(kRescueMaxWarps, std::max<size_t>(1, kRescueCtaBudget / per));
  const size_t smem = (size_t)wpb * per;
  // a few CTAs per SM at most: the list is short unless the rings were far too small
  const int64_t want = (max_work + wpb - 1) / wpb;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, 2 * (int64_t)num_sms()));
  const bool u16 = a.pred && a.pred_dtype == SDP_PRED_U16;
  if (a.batched) return launch_r<uint16_t, true, false, false>(a, wpb, smem, grid, st);
  if (hist) return launch_r<int32_t, false, false, true>(a, wpb, smem, grid, st);
  if (a.soft)
    return u16 ? launch_r<uint16_t, false, true, false>(a, wpb, smem, grid, st)
               : launch_r<int32_t, false, true, false>(a, wpb, smem, grid, st);
  return u16 ? launch_r<uint16_t, false, false, false>(a, wpb, smem, grid, st)
             : launch_r<int32_t, false, false, false>(a, wpb, smem, grid, st);
}

}  // namespace sdp
