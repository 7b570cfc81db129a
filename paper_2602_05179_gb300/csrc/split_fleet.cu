// split_fleet.cu -- fleet-limited Split (at most K routes) for sm_103a.
//
// The extensive model of Appendix A bounds the vehicles used per scenario
// (constraint eq:fleet_size); its giant-tour example has "three vehicles
// available".  With hard capacity as in Eq. eqdpA and at most K routes, the
// recursion gains a route-count dimension:
//     J_k(i) = min over capacity-feasible p < i of J_{k-1}(p) + W(p,i),
//     J_0(0) = 0, J_0(i > 0) = J_k(0) = +inf, cost = min_{k <= K} J_k(n),
// ties to the smallest p at every (k, i), then to the fewest routes.  In the
// K-form of sdp_internal.cuh, layer k is the window minimum of
// psi_{k-1}(p) = K_{k-1}(p) + a_{p+1} -- the Split recursion fed by the layer
// below -- and every layer has the same capacity window.
//
// split_fleet_band_kernel (AUTO up to n = 1,855 to 1,879, by K): one warp per
// scenario, layer after layer, over the band of positions that matter.  A
// split into at most K routes passes (k, i) only if n can be reached from i
// with K - k more routes, i >= lo_k, and i from 0 with k, i <= hi_k: both
// ends follow from the prefix loads alone (lo by filling routes greedily from
// the tour's end, hi from its start), every feasible p of a position in the
// band lies in the band below, so the values in it are those of the full
// recursion.  A binding fleet leaves few routes of slack, and the band is
// slack routes wide: at n = 500, Q = 200, K = 42 (about 41 needed) 19
// positions of 500 on average.  Within a layer the positions are independent: a lane
// each, windows by minima of blocks of B positions (built once per layer in
// shared memory), values only.  The layers' psi rows go to a scratch of the
// warp (band only, in L2), and the path is found from the last layer back,
// 32 candidates at a time.
//   Windows of at most 32 positions take blocks of 4; a scenario with a
// longer one is flagged and recomputed by the same kernel with blocks of 16
// (its list, SDP_FLAG_FALLBACK).
//   n = 500, K = 42, S = 65,536: 1.12 ms where the deque kernel
// below, which steps every layer through every position, took 5.43 ms and
// 0.32 ms of recomputation.
//   A fleet with much slack makes the band the whole tour: such calls it leaves
// to the deque kernel (fleet_loose_load), which hands back the scenarios whose
// deque outgrows its ring.
//
// split_fleet_kernel (longer tours, calls with much slack): one warp per
// scenario, the layers across its lanes:
// lane l's slot j holds layer k = 32 j + l + 1 (two slots: K <= 64).  Every
// lane walks the same positions i = 1..n in lockstep, so the demand of s_i
// and the tour record are broadcast loads; layer k's input psi_{k-1}(i-1) =
// K_{k-1}(i-1) + a_i comes from the lane below (a shuffle; lane 0 of slot 0
// takes layer 0: K_0(0) = 0, else +inf), and each lane keeps its layer's
// window candidates in a monotone deque (entries (psi bits, L(p) << 16 | p),
// rings [slot][entry][lane] in shared memory): pop the back while its psi is
// larger (an equal one is older: smallest p), push p = i - 1 unless its state
// is unreachable (+inf), pop the front while the route p+1..i exceeds Q; an
// empty window reads +inf (a demand above Q at position i empties it, and
// the first such position makes every later J infinite).  With route output, i - p of every
// (i, k) goes to the warp's scratch row [i][k] and lane 0 walks the optimal
// split back.  A deque that outgrows its ring flags the scenario and
// split_fleet_rescue_kernel recomputes it, one warp per scenario and the same
// FP32 operations as split_fleet_plain_kernel (one thread per scenario, every
// feasible p of every layer: PLAIN, and the recomputation for n too long for
// the rescue's shared memory).
#include <math_constants.h>

#include <algorithm>

#include "dependent.cuh"
#include "sdp_internal.cuh"

namespace sdp {

namespace {

constexpr int kFRing = 16;                          // deque entries per layer and lane
constexpr uint32_t kFRingBytes = kFRing * 256u;     // one layer's ring for 32 lanes
constexpr int kFMaxWarps = 24;                      // warps per CTA at most (as shared memory allows)
constexpr int kFAhead = 8;                          // demands loaded ahead

__device__ __forceinline__ float flds(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint2 flds2(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ void fsts2(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.u32 [%0], {%1,%2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}

// One layer's deque of one lane (checked form: emptiness tests, any demand).
struct FleetDeque {
  uint32_t rb;          // shared address of the lane's entry in ring slot 0
  uint32_t head, tail;  // byte offsets (multiples of 256), unwrapped
  uint32_t fent;        // front entry L(p) << 16 | p
  float fpsi, bpsi, K;  // front psi, back psi, K_k(i) of the last position
  bool full;
  __device__ __forceinline__ uint32_t at(uint32_t off) const {
    return rb + (off & ((kFRing - 1) << 8));
  }
  __device__ __forceinline__ void init(uint32_t ring, int lane) {
    rb = ring + 8u * (uint32_t)lane;
    head = tail = 0u;
    fent = 0u;
    fpsi = CUDART_INF_F;
    bpsi = -CUDART_INF_F;
    K = CUDART_INF_F;
    full = false;
  }
  // push entry (psi, ent) of p = i-1, then drop expired fronts; Lc = L(i)<<16.
  // An unreachable state (psi = +inf) is not pushed: it could only be the
  // minimum of an empty window, which reads +inf anyway (pushed, such entries
  // would pile up behind each other over a long unreachable stretch).
  __device__ __forceinline__ void step(float psi, uint32_t ent, uint32_t Lc, uint32_t Qc,
                                       float ce) {
    if (psi != CUDART_INF_F) {
      while (bpsi > psi) {
        tail -= 256u;
        bpsi = tail == head ? -CUDART_INF_F : flds(at(tail - 256u));
      }
      if (tail == head) {
        fpsi = psi;
        fent = ent;
      }
      if (tail - head >= kFRingBytes) {  // full: flagged, restart at the new entry
        full = true;
        head = tail;
        fpsi = psi;
        fent = ent;
      }
      fsts2(at(tail), __float_as_uint(psi), ent);
      tail += 256u;
      bpsi = psi;
    }
    while (tail != head && ((Lc | 0xFFFFu) - fent) > Qc) {
      head += 256u;
      if (head != tail) {
        const uint2 e = flds2(at(head));
        fpsi = __uint_as_float(e.x);
        fent = e.y;
      }
    }
    if (tail == head) {  // nothing feasible in the window
      fpsi = CUDART_INF_F;
      bpsi = -CUDART_INF_F;
    }
    K = __fadd_rn(fpsi, ce);
  }
};

// KS: slots per lane (layers = 32 KS >= K); ROUTES: keep i - p of every
// (i, k) in the warp's scratch for the backtrack.
template <int KS, bool ROUTES>
__global__ void __launch_bounds__(kFMaxWarps * 32) split_fleet_kernel(SplitFleetArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int n = a.n, Q = a.Q, K = a.K;
  dep_launch();
  const bool shared_call = a.loose != nullptr;  // with the band kernel: one of them takes the call
  if (shared_call && *a.loose == 0u) return;
  // shared: (a_i, ce_i) and columns of the tour | per warp: KS rings,
  // route boundaries
  float2* rec = reinterpret_cast<float2*>(smem);
  uint16_t* cols = reinterpret_cast<uint16_t*>(rec + n);
  const size_t head_bytes = (((size_t)n * 8 + (size_t)n * 2) + 255) & ~(size_t)255;
  const size_t per_warp = (size_t)KS * kFRingBytes + 256 * 4;
  unsigned char* wb = smem + head_bytes + per_warp * warp;
  const uint32_t rings = (uint32_t)__cvta_generic_to_shared(wb);
  int32_t* bounds = reinterpret_cast<int32_t*>(wb + (size_t)KS * kFRingBytes);
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const StepRec r = a.rec[k];
    rec[k] = make_float2(r.a, r.ce);
    cols[k] = (uint16_t)r.col;
  }
  __syncthreads();
  const uint32_t Qh = (uint32_t)Q << 16, Qc = Qh | 0xFFFFu;
  const double Dn = *a.Dn;
  const int64_t wslot = (int64_t)blockIdx.x * nw + warp;
  // the warp's delta scratch: [i][k] uint16, 32 KS layers per position
  uint16_t* dsc = ROUTES ? a.dscratch + wslot * (int64_t)n * 32 * KS : nullptr;
  bool neg = false, any_fb = false, any_inf = false;
  for (int64_t s = wslot; s < a.S; s += (int64_t)gridDim.x * nw) {
    if (shared_call && s != wslot) {
      // rings outgrow on a tour more than on a scenario: where one in eight so
      // far has, the rest goes to the band kernel too
      uint32_t back = 0u;
      if (lane == 0) back = __ldcg(a.fb_count);
      if ((int64_t)__shfl_sync(0xffffffffu, back, 0) > 16 + s / 8) {
        if (lane == 0) a.fb_list[atomicAdd(a.fb_count, 1u)] = (uint32_t)s;
        continue;
      }
    }
    const int32_t* qrow = a.demands + s * n;
    FleetDeque dq[KS];
#pragma unroll
    for (int j = 0; j < KS; ++j) dq[j].init(rings + (uint32_t)j * kFRingBytes, lane);
    // demands of positions i .. i + kFAhead - 1 (broadcast loads, ahead)
    int qa[kFAhead];
#pragma unroll
    for (int u = 0; u < kFAhead; ++u) qa[u] = u < n ? __ldg(qrow + cols[u]) : 0;
    uint32_t Lc = 0u;  // L(i-1) << 16 (mod 2^32)
    uint32_t first_inf = (uint32_t)n + 1u;
    for (int i0 = 1; i0 <= n; i0 += kFAhead) {
#pragma unroll
      for (int u = 0; u < kFAhead; ++u) {
        const int i = i0 + u;
        if (i > n) break;
        const int q = qa[u];
        qa[u] = i + kFAhead <= n ? __ldg(qrow + cols[i + kFAhead - 1]) : 0;
        neg |= q < 0;
        const uint32_t qh = (uint32_t)min(max(q, 0), Q + 1) << 16;
        if (qh > Qh && first_inf > (uint32_t)n) first_inf = (uint32_t)i;
        const float2 r = rec[i - 1];
        const uint32_t ent = Lc | (uint32_t)(i - 1);
        const uint32_t Lnew = Lc + qh;
        // inputs from the layer below as it stood before this position
        float below[KS];
#pragma unroll
        for (int j = 0; j < KS; ++j) {
          const float up = __shfl_up_sync(0xffffffffu, dq[j].K, 1);
          const float wrap = j > 0 ? __shfl_sync(0xffffffffu, dq[j > 0 ? j - 1 : 0].K, 31)
                                   : (i == 1 ? 0.f : CUDART_INF_F);
          below[j] = lane > 0 ? up : wrap;
        }
#pragma unroll
        for (int j = 0; j < KS; ++j) {
          if (32 * j + lane < K) {
            dq[j].step(__fadd_rn(below[j], r.x), ent, Lnew, Qc, r.y);
            if (ROUTES)
              dsc[(int64_t)(i - 1) * 32 * KS + 32 * j + lane] =
                  (uint16_t)(i - (int)(dq[j].fent & 0xFFFFu));
          }
        }
        Lc = Lnew;
      }
      if (shared_call && __any_sync(0xffffffffu, dq[0].full || dq[KS - 1].full)) break;
    }
    // the best layer k <= K, fewest routes on ties
    float best = CUDART_INF_F;
    int bk = 0;
    bool full = false;
#pragma unroll
    for (int j = KS - 1; j >= 0; --j) {
      if (32 * j + lane < K) {
        full |= dq[j].full;
        if (dq[j].K <= best) {
          best = dq[j].K;
          bk = 32 * j + lane + 1;
        }
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const float ob = __shfl_xor_sync(0xffffffffu, best, off);
      const int ok = __shfl_xor_sync(0xffffffffu, bk, off);
      if (ob < best || (ob == best && ok != 0 && (bk == 0 || ok < bk))) {
        best = ob;
        bk = ok;
      }
    }
    full = __any_sync(0xffffffffu, full);
    const bool infeasible = first_inf <= (uint32_t)n || bk == 0 || best == CUDART_INF_F;
    if (full) {
      if (lane == 0) {
        const uint32_t f = atomicAdd(a.fb_count, 1u);
        a.fb_list[f] = (uint32_t)s;
      }
      any_fb = true;
      continue;
    }
    any_inf |= infeasible;
    if (lane == 0) {
      a.cost[s] = infeasible ? CUDART_INF_F : (float)((double)best + Dn);
      if (a.nroutes) a.nroutes[s] = infeasible ? 0 : bk;
    }
    if (ROUTES) {
      uint8_t* ro = a.route + s * n;
      if (infeasible) {
        for (int m = lane; m < n; m += 32) ro[m] = 0xFFu;
      } else {
        // route k (1-based) covers positions bounds[k-1]+1 .. bounds[k]
        __syncwarp();
        if (lane == 0) {
          int i = n, k = bk;
          bounds[k] = n;
          while (k > 0) {
            if (i > 0) i = max(0, i - (int)dsc[(int64_t)(i - 1) * 32 * KS + (k - 1)]);
            bounds[--k] = i;
          }
        }
        __syncwarp();
        for (int m = lane; m < n; m += 32) {
          int k = 0;
          while (bounds[k + 1] <= m) ++k;
          ro[m] = (uint8_t)k;
        }
        __syncwarp();
      }
    }
  }
  if (lane == 0) {
    if (any_fb) atomicOr(a.status, SDP_FLAG_FALLBACK);
    if (any_inf) atomicOr(a.status, SDP_FLAG_INFEASIBLE);
  }
  if (__any_sync(0xffffffffu, neg) && lane == 0) atomicOr(a.status, SDP_FLAG_NEG_INPUT);
}

// Every feasible p of every layer, one thread per scenario (PLAIN for the
// fleet-limited Split, and the recomputation of flagged scenarios): layer k
// from layer k - 1 held in the thread's scratch rows, the same FP32
// operations and tie rules as split_fleet_kernel.
__global__ void __launch_bounds__(256) split_fleet_plain_kernel(SplitFleetArgs a) {
  const int n = a.n, Q = a.Q, K = a.K;
  const int64_t nslots = a.nslots;
  const int64_t count = a.fb_list ? (int64_t)*a.fb_count : a.S;
  for (int64_t slot = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; slot < nslots;
       slot += (int64_t)gridDim.x * blockDim.x) {
    float* Kp = a.kscratch + slot * 2 * (int64_t)(n + 1);
    float* Kc = Kp + (n + 1);
    uint16_t* P = a.pscratch ? a.pscratch + slot * (int64_t)K * n : nullptr;
    for (int64_t it = slot; it < count; it += nslots) {
      const int64_t s = a.fb_list ? (int64_t)a.fb_list[it] : it;
      const int32_t* q = a.demands + s * n;
      Kp[0] = 0.f;
      for (int i = 1; i <= n; ++i) Kp[i] = CUDART_INF_F;
      float best = CUDART_INF_F;
      int bk = 0;
      bool infeasible = false;
      for (int i = 1; i <= n && !infeasible; ++i) infeasible = q[a.rec[i - 1].col] > Q;
      for (int k = 1; k <= K && !infeasible; ++k) {
        Kc[0] = CUDART_INF_F;
        for (int i = 1; i <= n; ++i) {
          float bv = CUDART_INF_F;
          int bp = -1;
          int load = 0;
          for (int p = i - 1; p >= 0; --p) {
            load += max(__ldg(q + a.rec[p].col), 0);
            if (load > Q) break;
            const float psi = __fadd_rn(Kp[p], a.rec[p].a);
            if (psi <= bv) {  // p runs downwards: the smallest p on ties
              bv = psi;
              bp = p;
            }
          }
          Kc[i] = bp < 0 ? CUDART_INF_F : __fadd_rn(bv, a.rec[i - 1].ce);
          if (P) P[(int64_t)(k - 1) * n + (i - 1)] = (uint16_t)(bp < 0 ? 0 : i - bp);
        }
        if (Kc[n] < best) {  // the fewest routes on ties
          best = Kc[n];
          bk = k;
        }
        float* t = Kp;
        Kp = Kc;
        Kc = t;
      }
      infeasible = infeasible || bk == 0 || best == CUDART_INF_F;
      a.cost[s] = infeasible ? CUDART_INF_F : (float)((double)best + *a.Dn);
      if (a.nroutes) a.nroutes[s] = infeasible ? 0 : bk;
      if (a.route) {
        uint8_t* ro = a.route + s * n;
        if (infeasible) {
          for (int m = 0; m < n; ++m) ro[m] = 0xFFu;
        } else {
          int i = n, k = bk;
          while (k > 0 && i > 0) {
            const int p = max(0, i - (int)P[(int64_t)(k - 1) * n + (i - 1)]);
            for (int m = p; m < i; ++m) ro[m] = (uint8_t)(k - 1);
            i = p;
            --k;
          }
        }
      }
      if (infeasible) atomicOr(a.status, SDP_FLAG_INFEASIBLE);
    }
  }
}

// Recomputation of the flagged scenarios, one warp per scenario.  Layer k
// depends only on layer k - 1, so within a layer every position is
// independent: lane l takes positions i = 1 + l, 33 + l, ... and scans its
// window p = i - 1 down to pmin(i), the smallest p whose route p+1..i fits Q
// (the same for every layer: found once per scenario by a binary search of
// the prefix loads).  K_{k-1} and K_k sit in shared memory, and the tour's
// a_{p+1} and ce_i once per CTA; the FP32 operations, the order of p and the
// tie rules are split_fleet_plain_kernel's, so the results are its bits, and
// the route deltas go to the same per-slot scratch for the same backtrack.
constexpr int kFRescueWarps = 8;
// per warp: K_{k-1}, K_k, prefix loads L and window starts pmin, [n+1] each
__host__ __device__ inline size_t fleet_rescue_per_warp(int n) { return (size_t)4 * 4 * ((size_t)n + 1); }
__host__ __device__ inline size_t fleet_rescue_head(int n) { return ((size_t)8 * (size_t)n + 15) & ~(size_t)15; }

__global__ void __launch_bounds__(kFRescueWarps * 32) split_fleet_rescue_kernel(SplitFleetArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  const int n = a.n, Q = a.Q, K = a.K;
  float* as = reinterpret_cast<float*>(smem);  // a_{p+1} at [p], ce_i at [n + i - 1]
  float* ces = as + n;
  float* Kp = reinterpret_cast<float*>(smem + fleet_rescue_head(n) + (size_t)wib * fleet_rescue_per_warp(n));
  float* Kc = Kp + (n + 1);
  int32_t* L = reinterpret_cast<int32_t*>(Kc + (n + 1));
  int32_t* pmin = L + (n + 1);
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    as[k] = a.rec[k].a;
    ces[k] = a.rec[k].ce;
  }
  __syncthreads();
  const int64_t slot = (int64_t)blockIdx.x * wpb + wib;  // < nslots (the launch sees to it)
  uint16_t* P = a.pscratch ? a.pscratch + slot * (int64_t)K * n : nullptr;
  const int64_t count = (int64_t)*a.fb_count;
  const int64_t nw = (int64_t)gridDim.x * wpb;
  for (int64_t it = slot; it < count; it += nw) {
    const int64_t s = (int64_t)a.fb_list[it];
    const int32_t* q = a.demands + s * n;
    __syncwarp();  // the previous scenario's reads are done
    int carry = 0;
    bool over = false;
    if (lane == 0) L[0] = 0;
    for (int i0 = 1; i0 <= n; i0 += 32) {
      const int i = i0 + lane;
      int v = 0;
      if (i <= n) {
        const int raw = __ldg(q + __ldg(&a.rec[i - 1].col));
        over |= raw > Q;
        v = max(raw, 0);
      }
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += t;
      }
      if (i <= n) L[i] = carry + v;
      carry += __shfl_sync(0xffffffffu, v, 31);
    }
    const bool infeasible0 = __any_sync(0xffffffffu, over);
    __syncwarp();
    // pmin(i): L is non-decreasing, so the feasible p < i form [pmin, i - 1]
    // (pmin = i: none; only with a demand above Q, which makes the scenario
    // infeasible anyway)
    for (int i = 1 + lane; i <= n; i += 32) {
      const int Li = L[i];
      int lo = 0, hi = i;  // smallest p in [0, i) with Li - L[p] <= Q, else i
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (Li - L[mid] <= Q) hi = mid; else lo = mid + 1;
      }
      pmin[i] = lo;
    }
    for (int i = lane; i <= n; i += 32) Kp[i] = i == 0 ? 0.f : CUDART_INF_F;
    __syncwarp();
    float* kp = Kp;
    float* kc = Kc;
    float best = CUDART_INF_F;
    int bk = 0;
    for (int k = 1; k <= K && !infeasible0; ++k) {
      if (lane == 0) kc[0] = CUDART_INF_F;
      for (int i = 1 + lane; i <= n; i += 32) {
        const int pm = pmin[i];
        float bv = CUDART_INF_F;
        int bp = -1;
#pragma unroll 4
        for (int p = i - 1; p >= pm; --p) {
          const float psi = __fadd_rn(kp[p], as[p]);
          if (psi <= bv) {  // p runs downwards: the smallest p on ties
            bv = psi;
            bp = p;
          }
        }
        kc[i] = bp < 0 ? CUDART_INF_F : __fadd_rn(bv, ces[i - 1]);
        if (P) P[(int64_t)(k - 1) * n + (i - 1)] = (uint16_t)(bp < 0 ? 0 : i - bp);
      }
      __syncwarp();  // layer k complete before it is read
      if (kc[n] < best) {  // the fewest routes on ties
        best = kc[n];
        bk = k;
      }
      float* t = kp;
      kp = kc;
      kc = t;
    }
    const bool infeasible = infeasible0 || bk == 0 || best == CUDART_INF_F;
    if (lane == 0) {
      a.cost[s] = infeasible ? CUDART_INF_F : (float)((double)best + *a.Dn);
      if (a.nroutes) a.nroutes[s] = infeasible ? 0 : bk;
      if (infeasible) atomicOr(a.status, SDP_FLAG_INFEASIBLE);
    }
    if (a.route) {
      __syncwarp();  // the route deltas of every lane, for lane 0's backtrack
      uint8_t* ro = a.route + s * n;
      if (infeasible) {
        for (int m = lane; m < n; m += 32) ro[m] = 0xFFu;
      } else if (lane == 0) {
        int i = n, k = bk;
        while (k > 0 && i > 0) {
          const int p = max(0, i - (int)P[(int64_t)(k - 1) * n + (i - 1)]);
          for (int m = p; m < i; ++m) ro[m] = (uint8_t)(k - 1);
          i = p;
          --k;
        }
      }
    }
  }
}

// -------------------------------------------------------------- the band
constexpr int kBandMaxWarps = 24;
constexpr int kBandMinWarps = 8;   // per SM: fewer hide too little latency
constexpr int kBandWindow = 32;    // longest window of the narrow form
constexpr int kBandNarrow = 4, kBandWide = 16;  // positions per block minimum

// CTA: a_{p+1} and ce_i [n+1] floats each, columns [n]; per warp: prefix
// loads, psi and block minima [n+1 .. +16] (each on 16 bytes), window starts [n+1] uint16, and
// the layers' ends and route bounds [K+2] uint16 x 3.
__host__ __device__ constexpr size_t band_head(int n) {
  return ((size_t)(n + 1) * 8 + (size_t)n * 2 + 15) & ~(size_t)15;
}
__host__ __device__ constexpr size_t band_floats(int n) { return ((size_t)n + 1 + kBandWide + 3) & ~(size_t)3; }
__host__ __device__ constexpr size_t band_per_warp(int n, int K) {
  return (band_floats(n) * 12 + (size_t)(n + 1) * 2 + (size_t)(K + 2) * 6 + 15) & ~(size_t)15;
}

// B: positions per block minimum.  LIST: the flagged scenarios (fb_list);
// otherwise all, flagging those with a window above kBandWindow, or none where
// the tour preparation's sample says that the fleet has much slack (loose).
template <int B, bool LIST, bool ROUTES>
__global__ void __launch_bounds__(kBandMaxWarps * 32) split_fleet_band_kernel(SplitFleetArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int n = a.n, Q = a.Q, K = a.K;
  float* as = reinterpret_cast<float*>(smem);  // a_{p+1} at [p], 0 at [n]
  float* ces = as + n + 1;                     // ce_i at [i]
  uint16_t* cols = reinterpret_cast<uint16_t*>(ces + n + 1);
  unsigned char* wb = smem + band_head(n) + band_per_warp(n, K) * warp;
  int32_t* L = reinterpret_cast<int32_t*>(wb);
  float* psi = reinterpret_cast<float*>(L + band_floats(n));
  float* blk = psi + band_floats(n);
  uint16_t* pm = reinterpret_cast<uint16_t*>(blk + band_floats(n));
  uint16_t* lo_of = pm + n + 1;      // [m]: the first position that m more routes take to n
  uint16_t* hi_of = lo_of + K + 2;   // [k]: the last position that k routes reach
  uint16_t* bound = hi_of + K + 2;   // route k covers positions bound[k] + 1 .. bound[k+1]
  if (LIST) dep_wait();
  const uint32_t leave = !LIST && a.loose ? *a.loose : 0u;  // (in flight with the records)
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const StepRec r = a.rec[k];
    as[k] = r.a;
    ces[k + 1] = r.ce;
    cols[k] = (uint16_t)r.col;
  }
  if (threadIdx.x == 0) as[n] = 0.f;
  __syncthreads();
  if (!LIST && leave) return;
  const double Dn = *a.Dn;
  const int64_t slot = (int64_t)blockIdx.x * nw + warp;
  float* rows = ROUTES ? reinterpret_cast<float*>(a.dscratch) + slot * K * (int64_t)(n + 1) : nullptr;
  bool neg = false;
  uint32_t any_fb = 0, any_inf = 0;
  const int64_t count = LIST ? (int64_t)*a.fb_count : a.S;
  const int64_t stride = (int64_t)gridDim.x * nw;
  const bool vec = (n & 3) == 0 && (reinterpret_cast<uintptr_t>(a.demands) & 15) == 0;
  for (int64_t it = slot; it < count; it += stride) {
    const int64_t s = LIST ? (int64_t)a.fb_list[it] : it;
    const int32_t* qrow = a.demands + s * n;
    if (!LIST && it + stride < count) {  // the next scenario's row into L2
      const char* nx = reinterpret_cast<const char*>(a.demands + (s + stride) * n);
      for (int o = lane * 128; o < n * 4; o += 32 * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(nx + o));
    }
    // ---- demands by customer (staged in psi), then prefix loads in tour order
    int32_t* stage = reinterpret_cast<int32_t*>(psi);
    if (vec) {
      for (int k = lane; k < n / 4; k += 32)
        reinterpret_cast<int4*>(blk)[k] = __ldg(reinterpret_cast<const int4*>(qrow) + k);
      stage = reinterpret_cast<int32_t*>(blk);
    } else {
      for (int k = lane; k < n; k += 32) stage[k] = __ldg(qrow + k);
    }
    __syncwarp();
    bool over = false;
    int carry = 0;
    if (lane == 0) L[0] = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
      const int i = i0 + lane;
      int v = i < n ? stage[cols[i]] : 0;
      neg |= v < 0;
      over |= v > Q;
      v = min(max(v, 0), Q + 1);
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(kAll, v, d);
        if (lane >= d) v += t;
      }
      if (i < n) L[i + 1] = carry + v;
      carry += __shfl_sync(kAll, v, 31);
    }
    bool infeasible = __any_sync(kAll, over);
    __syncwarp();
    float best = CUDART_INF_F;
    int bk = 0;
    if (!infeasible) {
      // ---- window starts: the smallest p with L(i) - L(p) <= Q.  They only
      // grow with i, so a lane's search begins at its last one's.
      int lo = 0, longest = 0;
      for (int i0 = 1; i0 <= n; i0 += 32) {
        const int i = min(i0 + lane, n);
        const int need = L[i] - Q;
        int hi = i;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (L[mid] >= need) hi = mid; else lo = mid + 1;
        }
        pm[i] = (uint16_t)lo;
        longest = max(longest, i - lo);
      }
      if (lane == 0) pm[0] = 0;
      __syncwarp();
      if (!LIST && __any_sync(kAll, longest > kBandWindow)) {
        if (lane == 0) a.fb_list[atomicAdd(a.fb_count, 1u)] = (uint32_t)s;
        any_fb = 1;
        continue;
      }
      // ---- the band's lower end, from the tour's end
      {
        int x = n, m = 0;
        for (; m <= K && x > 0; ++m) {
          if (lane == 0) lo_of[m] = (uint16_t)x;
          x = pm[x];
        }
        infeasible = x > 0;  // more than K routes (x reached 0 after m of them)
        for (int k = m + lane; k <= K; k += 32) lo_of[k] = 0;
      }
      infeasible = infeasible || (__syncwarp(), lo_of[K] != 0);
    }
    if (!infeasible) {
      // ---- layer 0
      for (int p = lane; p < (int)band_floats(n); p += 32) {
        psi[p] = p == 0 ? as[0] : CUDART_INF_F;
        blk[p] = CUDART_INF_F;
      }
      if (lane == 0) hi_of[0] = 0;
      __syncwarp();
      int hi = 0, lo_prev = 0;
      for (int k = 1; k <= K; ++k) {
        // block minima of the layer below: blk[p] = min psi[p .. p + B - 1]
        for (int p = lo_prev + lane; p <= hi; p += 32) {
          float m = psi[p];
#pragma unroll
          for (int e = 1; e < B; ++e) m = fminf(m, psi[p + e]);
          blk[p] = m;
        }
        // the last position that k routes reach
        int nh = hi;
        {
          const int reach = L[hi] + Q;
          for (;;) {
            const int i = nh + 1 + lane;
            const unsigned ok = __ballot_sync(kAll, i <= n && L[min(i, n)] <= reach);
            nh += __popc(ok);
            if (ok != kAll) break;
          }
        }
        const int lo = max((int)lo_of[K - k], 1);
        __syncwarp();
        float* row = ROUTES ? rows + (int64_t)(k - 1) * (n + 1) : nullptr;
        for (int top = nh; top >= lo; top -= 32) {
          const int i = max(top - lane, lo);
          const int pi = pm[i];
          float m = CUDART_INF_F;
          const int last = i - B;  // the block that ends at i - 1
          if (last >= pi) {
            m = blk[last];
            for (int p = pi; p < last; p += B) m = fminf(m, blk[p]);
          } else {
            for (int p = pi; p < i; ++p) m = fminf(m, psi[p]);
          }
          const float Ki = __fadd_rn(m, ces[i]);
          __syncwarp();  // this round's reads come before its writes
          if (top - lane >= lo) {
            const float v = __fadd_rn(Ki, as[i]);
            psi[i] = v;
            if (ROUTES) row[i] = v;
          }
          if (top == n) {
            const float Kn = __shfl_sync(kAll, Ki, 0);
            if (Kn < best) {  // the fewest routes on ties
              best = Kn;
              bk = k;
            }
          }
        }
        if (k == 1 && lane == 0) psi[0] = CUDART_INF_F;  // J_k(0), k >= 1
        if (lane == 0) hi_of[k] = (uint16_t)nh;
        hi = nh;
        lo_prev = lo_of[K - k];
        __syncwarp();
      }
      infeasible = bk == 0;
    }
    any_inf |= infeasible;
    if (lane == 0) {
      a.cost[s] = infeasible ? CUDART_INF_F : (float)((double)best + Dn);
      if (a.nroutes) a.nroutes[s] = infeasible ? 0 : bk;
    }
    if (ROUTES) {
      uint8_t* out = a.route + s * n;
      uint8_t* st = reinterpret_cast<uint8_t*>(psi);
      if (infeasible) {
        for (int m = lane; m < n; m += 32) out[m] = 0xFFu;
      } else {
        // ---- the path, last route first: the smallest p of the window with
        // the least psi of the layer below
        int i = n;
        for (int k = bk; k >= 1; --k) {
          if (lane == 0) bound[k] = (uint16_t)i;
          int p = 0;
          if (k > 1) {
            const float* row = rows + (int64_t)(k - 2) * (n + 1);
            const int p0 = max((int)pm[i], 1), p1 = min(i - 1, (int)hi_of[k - 1]);
            p = p0;
            uint32_t least = 0xFFFFFFFFu;
            for (int c = p0; c <= p1; c += 32) {
              // floats as unsigned keys in their order (-0 taken as 0)
              uint32_t key = 0xFFFFFFFFu;
              if (c + lane <= p1) {
                const uint32_t b = __float_as_uint(__fadd_rn(row[c + lane], 0.f));
                key = b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
              }
              const uint32_t m = __reduce_min_sync(kAll, key);
              if (m < least) {
                least = m;
                p = c + __ffs(__ballot_sync(kAll, key == m)) - 1;
              }
            }
          }
          i = p;
        }
        if (lane == 0) bound[0] = 0;
        __syncwarp();
        if (LIST) {
          for (int k = 0; k < bk; ++k)
            for (int m = bound[k] + lane; m < (int)bound[k + 1]; m += 32) st[m] = (uint8_t)k;
        } else {
          for (int k = lane; k < bk; k += 32)
            for (int m = bound[k]; m < (int)bound[k + 1]; ++m) st[m] = (uint8_t)k;
        }
        __syncwarp();
        if ((n & 3) == 0 && (reinterpret_cast<uintptr_t>(a.route) & 3) == 0) {
          for (int m = lane; m < n / 4; m += 32)
            reinterpret_cast<uint32_t*>(out)[m] = reinterpret_cast<const uint32_t*>(st)[m];
        } else {
          for (int m = lane; m < n; m += 32) out[m] = st[m];
        }
      }
    }
    __syncwarp();  // the scenario's shared rows are read before the next one's writes
  }
  if (lane == 0) {
    if (any_fb) atomicOr(a.status, SDP_FLAG_FALLBACK);
    if (any_inf) atomicOr(a.status, SDP_FLAG_INFEASIBLE);
  }
  if (__any_sync(kAll, neg) && lane == 0) atomicOr(a.status, SDP_FLAG_NEG_INPUT);
}

size_t fleet_head(int n) { return (((size_t)n * 8 + (size_t)n * 2) + 255) & ~(size_t)255; }
size_t fleet_per_warp(int ks) { return (size_t)ks * kFRingBytes + 256 * 4; }

template <int KS, bool ROUTES>
int launch_fleet_k(const SplitFleetArgs& a, int warps, int grid, cudaStream_t st) {
  auto k = split_fleet_kernel<KS, ROUTES>;
  const size_t smem = fleet_head(a.n) + fleet_per_warp(KS) * warps;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return (int)e;
  k<<<grid, warps * 32, smem, st>>>(a);
  return (int)cudaGetLastError();
}

int launch_deque(const SplitFleetArgs& a, int warps, int grid, cudaStream_t st) {
  if (a.K <= 32)
    return a.route ? launch_fleet_k<1, true>(a, warps, grid, st) : launch_fleet_k<1, false>(a, warps, grid, st);
  return a.route ? launch_fleet_k<2, true>(a, warps, grid, st) : launch_fleet_k<2, false>(a, warps, grid, st);
}

template <bool ROUTES>
int launch_band(const SplitFleetArgs& a, const FleetConfig& c, cudaStream_t st) {
  const size_t smem = band_head(a.n) + band_per_warp(a.n, a.K) * c.warps;
  auto narrow = split_fleet_band_kernel<kBandNarrow, false, ROUTES>;
  auto wide = split_fleet_band_kernel<kBandWide, true, ROUTES>;
  cudaError_t e = cudaFuncSetAttribute(narrow, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(wide, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return (int)e;
  narrow<<<c.grid, c.warps * 32, smem, st>>>(a);
  if (a.loose) {
    const int d = launch_deque(a, c.loose_warps, c.loose_grid, st);
    if (d) return d;
  }
  // placed while the deque kernel finds that it has nothing to do; placed early
  // behind the narrow form it slows that one (n = 500, K = 42: 1128 -> 1153 us)
  return (int)launch_dependent(a.loose != nullptr, wide, c.grid, c.warps * 32, smem, st, a);
}

// The deque kernel's shape: one CTA per SM with as many warps as its shared
// memory holds; fewer CTAs when there are fewer scenarios.
void deque_shape(int n, int K, int64_t S, int* warps, int* grid) {
  const size_t budget = 226 * 1024;  // dynamic shared memory of one CTA per SM
  const size_t head = fleet_head(n);
  const int w = head >= budget ? 0 : (int)((budget - head) / fleet_per_warp(K <= 32 ? 1 : 2));
  *warps = w > kFMaxWarps ? kFMaxWarps : w;
  if (*warps < 1) return;
  const int64_t need = (S + *warps - 1) / *warps;
  *grid = (int)imin64(need < 1 ? 1 : need, (int64_t)num_sms());
}

// The load of the kLoadSample scenarios below which the deque kernel takes a
// call rather than the band kernel: kLoadSample Q times the mean m of the routes
// that they need at least.
//   The band of a scenario holds about n (K - m) states.  On 65,536 scenarios
// (n = 31..500, K up to 64, windows of 4 to n positions, random and sweep tours)
// the band kernel takes about 12.3 K + 0.25 n (K - m) us beyond what both do,
// 0.34 n (K - m) for windows of n / 3 positions and more; the deque kernel 6.5 n
// (K <= 32) or 10.3 n (two layers a lane) while its rings hold, which the lines
// below take 5% higher.  Up to a scenario per warp of the chip the band kernel
// spreads them over all SMs, and the line lies higher.  Everything in the band,
// K = 64 and windows of 32 of n = 100 took 3.45 ms, the deque kernel 1.30;
// n = 300, window 46: 5.71 and 3.70.  A tight fleet (n = 500, K = 42, 39 to 42
// needed): 1.13 and 5.75.
//   With the choice, 1,500 sizes from S = 200 on take at most 1.08 of the deque
// kernel's time (eight of them up to 1.20).  It costs tight fleets a launch (1 to
// 4 us; n = 500, K = 42: 1,124 -> 1,128).  The sample taken by the band kernel's
// CTAs cost 3 us more, the deques inlined into the band kernel, or called from
// it, 2 to 13%.  Calls whose rings do outgrow (windows of 22 to n / 3 positions;
// the deque kernel and its recomputation took 2 to 20 times the band's time
// there) lose the time until the scenarios are handed back: up to 12% of the
// band's time, up to 78% where each warp has one scenario.
uint32_t fleet_loose_load(int n, int Q, int K, int64_t S) {
  const double idle = std::max(0.0, 1.0 - (double)S / (kFMaxWarps * num_sms()));
  // per position, in units of 0.25 us on 65,536 scenarios
  const double deque = (K <= 32 ? 27.0 + 6.0 * idle : 43.0 + 3.0 * idle) + 1200.0 * idle / n - 49.0 * K / n;
  const double m = std::max(K - deque, std::min(3.0, K - deque / 1.35));
  // (less than one route: hardly a call, and the choice costs each call a launch)
  return m >= 1.0 ? (uint32_t)(kLoadSample * std::min(m, K + 1.0) * Q) : 0u;
}

}  // namespace

// The band kernel: one CTA per SM with as many warps as its shared memory
// holds, spread over all SMs when there are few scenarios; else the deque
// kernel alone.
FleetConfig fleet_config(int n, int Q, int K, int64_t S) {
  FleetConfig c{};
  if (band_head(n) + band_per_warp(n, K) * kBandMinWarps <= 226 * 1024) {
    int warps = (int)((226 * 1024 - band_head(n)) / band_per_warp(n, K));
    warps = warps > kBandMaxWarps ? kBandMaxWarps : warps;
    // few scenarios: as many SMs as possible
    const int64_t share = (S + num_sms() - 1) / num_sms();
    c.band = true;
    c.warps = (int)imin64(warps, share < 1 ? 1 : share);
    const int64_t need = (S + c.warps - 1) / c.warps;
    c.grid = (int)imin64(need < 1 ? 1 : need, (int64_t)num_sms());
    c.loose_load = fleet_loose_load(n, Q, K, S);
    if (c.loose_load) deque_shape(n, K, S, &c.loose_warps, &c.loose_grid);
    if (c.loose_warps < 1) c.loose_load = 0u;
    return c;
  }
  deque_shape(n, K, S, &c.warps, &c.grid);
  return c;
}

// the band's rows (floats) and the deque kernel's route deltas share it, one
// kernel after the other
size_t fleet_dscratch_elems(int n, int K, const FleetConfig& c) {
  const size_t deltas = (size_t)n * 32 * (K <= 32 ? 1 : 2);
  if (!c.band) return (size_t)c.grid * c.warps * deltas;
  const size_t rows = (size_t)c.grid * c.warps * (size_t)K * (size_t)(n + 1) * 2;
  return c.loose_load ? std::max(rows, (size_t)c.loose_grid * c.loose_warps * deltas) : rows;
}

int launch_split_fleet(const SplitFleetArgs& a, const FleetConfig& c, cudaStream_t st) {
  if (c.warps < 1) return (int)cudaErrorInvalidValue;
  if (c.band) return a.route ? launch_band<true>(a, c, st) : launch_band<false>(a, c, st);
  return launch_deque(a, c.warps, c.grid, st);
}

bool fleet_rescue_supported(int n) { return fleet_rescue_head(n) + fleet_rescue_per_warp(n) <= 200u * 1024u; }

int launch_split_fleet_rescue(const SplitFleetArgs& a, cudaStream_t st) {
  const size_t per = fleet_rescue_per_warp(a.n);
  int wpb = (int)std::min<size_t>(kFRescueWarps, std::max<size_t>(1, (96u * 1024u) / per));
  if (wpb > a.nslots) wpb = (int)a.nslots;
  const size_t smem = fleet_rescue_head(a.n) + (size_t)wpb * per;
  // one scratch slot per warp: wpb * grid <= nslots
  const int grid = (int)std::max<int64_t>(1, a.nslots / wpb);
  auto k = split_fleet_rescue_kernel;
  if (smem > 48u * 1024u) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
  }
  k<<<grid, wpb * 32, smem, st>>>(a);
  return (int)cudaGetLastError();
}

int launch_split_fleet_plain(const SplitFleetArgs& a, cudaStream_t st) {
  const int grid = (int)((a.nslots + 255) / 256);
  split_fleet_plain_kernel<<<grid, 256, 0, st>>>(a);
  return (int)cudaGetLastError();
}

}  // namespace sdp
