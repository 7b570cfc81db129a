// split_shared.cu -- batched Split of many tours over one demand array (the
// candidate loop: every neighbour of a tour scored on the same scenarios) for
// sm_103a.
//
// Why.  The pipelined batched kernel (split_pipe.cu) narrows and permutes a
// tile's demands into tour order for each (tour, tile): with 1,025 tours on
// the same scenarios the same 32 rows are staged 1,025 times, by 9 of a CTA's
// 32 warps, through L2.  Here a CTA stages a tile of 32 scenarios once, in
// shared memory and by customer ([customer][32 scenarios], uint8 for Q <= 254,
// else uint16), and all 32 warps run tours on it: position i of a tour needs
// the 32 demands of customer s_i, one conflict-free shared load.  The (tile,
// tour) pairs, tile by tile, are cut into one run per CTA, so that a CTA
// stages two or three tiles of a launch of 313 tiles x 1,025 tours and
// meets a barrier only between them; within a tile its warps claim tours
// from a shared counter.  Launches of less than two tours per warp give each
// tile its own CTAs instead (launch_split_shared).
//
// The recursion is that of split_pipe.cu (Eq. eqdpA in the K-form of
// sdp_internal.cuh with a monotone deque per lane, entries (psi bits,
// L(p) << 16 | p), ring of 16): see there for the entry arithmetic, the ring
// test and the checked step of tiles with a demand above Q.  The lean step
// takes its pops under warp votes: what leaves the deque at the back is mostly
// decided by the tour, not by the scenario (at n = 100 the lanes pop 0.79
// entries a step, the busiest lane of a warp 0.91, and half the steps none),
// so one vote skips the back and the warp does not diverge.
//
// Neighbours of a tour begin as it does.  batch_prep_kernel counts the leading
// records that a tour shares with tour 0; on each tile warp 0 runs tour 0 once
// more and keeps the deques' state (ring and registers, 5 KB) after every
// a.snap_step positions, and a tour is resumed from the last state that lies
// within its shared records -- the same steps on the same values, not taken
// again.  States that warp 0 has not reached yet are not waited for.  Four
// iterations of a search (n = 100, 1,024 neighbours by 2-opt, relocation and
// swap, 10^4 scenarios): 6.23 -> 5.41 ms.  Tours that share too little for
// tour 0's extra run (twice its length in all) are run as they are.
//
// Bound: instruction issue, 43 warp instructions per DP step with 82% of the
// slots filled: 1,025 tours of n = 100 on 10^4 scenarios, each run whole, in
// 1.37 ms, where the pipelined kernel took 2.74 ms (85 instructions a step, staging included).
// Tiles staged by each warp in its own L2 slot took 2.05 ms.
#include <math_constants.h>

#include <algorithm>

#include "async_copy.cuh"
#include "sdp_internal.cuh"

namespace sdp {

namespace {

constexpr unsigned kAll = 0xffffffffu;
constexpr int kSWarps = 32;                    // one CTA per SM: 64 registers a thread
constexpr int kSRing = 16;                     // deque entries per lane
constexpr uint32_t kSRingBytes = (uint32_t)kSRing * 256u;
constexpr uint32_t kSRingMask = (uint32_t)(kSRing - 1) << 8;
constexpr int kSRecs = 32;                     // records of a warp's tour on chip
constexpr int kSBlock = kSRecs / 2;            // ... filled a block ahead
constexpr int kSCheckEvery = 2;                // steps between ring tests (lean step)
constexpr uint32_t kSMaxAtCheck = 14u;         // entries allowed at a test (+2 pushes <= 16)
static_assert(kSMaxAtCheck + kSCheckEvery <= (uint32_t)kSRing && kSBlock % kSCheckEvery == 0,
              "a test must leave room for the pushes until the next one");

__device__ __forceinline__ float4 lds_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_f4(uint32_t addr, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z),
               "f"(v.w) : "memory");
}
template <typename QT>
__device__ __forceinline__ uint32_t lds_q(uint32_t addr) {
  uint32_t v;
  if (sizeof(QT) == 1) {
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(addr));
  } else {
    unsigned short h;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(h) : "r"(addr));
    v = h;
  }
  return v;
}

// One lane's deque, as in split_pipe.cu; ring slots are byte offsets,
// multiples of 256 (32 lanes x 8 bytes), kept unwrapped and masked on use.
struct SharedLane {
  uint32_t rb;          // shared address of this lane's entry in ring slot 0
  uint32_t head, tail;  // offsets of the front and of the next free slot
  uint32_t Lent;        // L(i) << 16 | i (lean); L(i) << 16 (checked)
  uint32_t fent;        // front entry: L(p) << 16 | p
  float K, fpsi, bpsi;
  bool ovf;             // the deque outgrew the ring: recompute the scenario

  __device__ __forceinline__ uint32_t at(uint32_t off) const { return rb | (off & kSRingMask); }
  // lean: the first step restarts the deque at p = 0 (any psi is below +inf);
  // checked: the deque is empty (a back psi of -inf)
  __device__ __forceinline__ void init(uint32_t ring, int lane, bool lean) {
    rb = ring + 8u * (uint32_t)lane;
    head = tail = 0u;
    Lent = fent = 0u;
    K = 0.f;
    fpsi = CUDART_INF_F;
    bpsi = lean ? CUDART_INF_F : -CUDART_INF_F;
    ovf = false;
  }
  __device__ __forceinline__ void load_front() {
    const uint2 e = lds_u2(at(head));
    fpsi = __uint_as_float(e.x);
    fent = e.y;
  }
  // position i with demand q and record (a_i, ce_i); no demand above Q in the
  // tile, so neither loop empties the deque
  __device__ __forceinline__ void step(uint32_t q, float a, float ce, uint32_t Qc) {
    const float psi = __fadd_rn(K, a);
    const uint32_t ent = Lent;
    Lent += (q << 16) + 1u;
    if (__any_sync(kAll, bpsi > psi)) {
      if (__any_sync(kAll, psi < fpsi)) {
        if (psi < fpsi) {  // below the minimum: every entry pops
          tail = head;
          fpsi = psi;
          fent = ent;
          bpsi = -CUDART_INF_F;
        }
      }
      do {
        if (bpsi > psi) {
          tail -= 256u;
          bpsi = lds_f32(at(tail - 256u));
        }
      } while (__any_sync(kAll, bpsi > psi));
    }
    sts_u2(at(tail), __float_as_uint(psi), ent);
    tail += 256u;
    bpsi = psi;
    do {
      if (Lent - fent > Qc) {
        head += 256u;
        load_front();
      }
    } while (__any_sync(kAll, Lent - fent > Qc));
    K = __fadd_rn(fpsi, ce);
  }
  // every kSCheckEvery lean steps: more than kSMaxAtCheck entries flags the
  // lane and restarts its deque at the newest entry
  __device__ __forceinline__ void check() {
    if (tail - head > kSMaxAtCheck * 256u) {
      ovf = true;
      head = tail - 256u;
      load_front();
    }
  }
  // a demand above Q in the tile (Lent = L(i-1) << 16 here): emptiness and
  // exact ring tests
  __device__ __forceinline__ void step_chk(int i, uint32_t q, float a, float ce, uint32_t Qc, int Q,
                                           int n, uint32_t& first_inf) {
    const float psi = __fadd_rn(K, a);
    const uint32_t ent = Lent | (uint32_t)(i - 1);
    while (bpsi > psi) {
      tail -= 256u;
      bpsi = tail == head ? -CUDART_INF_F : lds_f32(at(tail - 256u));
    }
    if (tail == head) {
      fpsi = psi;
      fent = ent;
    }
    if (tail - head >= kSRingBytes) {  // full: flagged, restart at the new entry
      ovf = true;
      head = tail;
      fpsi = psi;
      fent = ent;
    }
    const uint32_t newest = tail;
    sts_u2(at(tail), __float_as_uint(psi), ent);
    tail += 256u;
    bpsi = psi;
    Lent += q << 16;
    if (q > (uint32_t)Q && first_inf > (uint32_t)n) first_inf = (uint32_t)i;
    // the newest entry stays even when q_i > Q
    while (((Lent | 0xFFFFu) - fent) > Qc && head != newest) {
      head += 256u;
      load_front();
    }
    K = __fadd_rn(fpsi, ce);
  }
};

// States of tour 0's deques, kept at every step-th position in shared memory.
constexpr uint32_t kSStateBytes = kSRingBytes + 8u * 128u;
struct Snapshots {
  uint32_t base;    // shared address of the first state
  int step;         // positions between them, a multiple of kSCheckEvery; 0: none
  int count;        // states that fit
  uint32_t* ready;  // states written so far
};
__device__ __forceinline__ uint32_t lds_u1(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sts_u1(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void save_state(const SharedLane& st, uint32_t at, int lane) {
#pragma unroll 4
  for (int k = 0; k < kSRing; ++k) {
    const uint2 e = lds_u2(st.rb + 256u * (uint32_t)k);
    sts_u2(at + 256u * (uint32_t)k + 8u * (uint32_t)lane, e.x, e.y);
  }
  const uint32_t w = at + kSRingBytes + 4u * (uint32_t)lane;
  sts_u1(w, st.head);
  sts_u1(w + 128u, st.tail);
  sts_u1(w + 256u, st.Lent);
  sts_u1(w + 384u, st.fent);
  sts_u1(w + 512u, __float_as_uint(st.K));
  sts_u1(w + 640u, __float_as_uint(st.fpsi));
  sts_u1(w + 768u, __float_as_uint(st.bpsi));
  sts_u1(w + 896u, st.ovf ? 1u : 0u);
}
__device__ __forceinline__ void load_state(SharedLane& st, uint32_t at, int lane) {
#pragma unroll 4
  for (int k = 0; k < kSRing; ++k) {
    const uint2 e = lds_u2(at + 256u * (uint32_t)k + 8u * (uint32_t)lane);
    sts_u2(st.rb + 256u * (uint32_t)k, e.x, e.y);
  }
  const uint32_t w = at + kSRingBytes + 4u * (uint32_t)lane;
  st.head = lds_u1(w);
  st.tail = lds_u1(w + 128u);
  st.Lent = lds_u1(w + 256u);
  st.fent = lds_u1(w + 384u);
  st.K = __uint_as_float(lds_u1(w + 512u));
  st.fpsi = __uint_as_float(lds_u1(w + 640u));
  st.bpsi = __uint_as_float(lds_u1(w + 768u));
  st.ovf = lds_u1(w + 896u) != 0u;
}

// One tour on the staged tile: lane l runs scenario row l.  SAVE: its states
// are kept (lean steps only); else it resumes from state `from` (0: from the
// start), after from * snap.step positions.  recs: the warp's
// kSRecs records (a, ce, shared address of the lane-0 demand of the customer),
// position k at k % kSRecs, filled a block of kSBlock ahead.
template <typename QT, bool CHECK, bool SAVE>
__device__ __forceinline__ void run_tour(int n, int Q, uint32_t tile, uint32_t ring, uint32_t recs,
                                         const StepRec* __restrict__ rec, int lane,
                                         const Snapshots& snap, int from, float* K_out,
                                         uint32_t* first_inf_out, bool* bad) {
  const uint32_t Qc = ((uint32_t)Q << 16) | 0xFFFFu;
  const uint32_t lq = (uint32_t)(lane * (int)sizeof(QT));
  SharedLane st;
  st.init(ring, lane, !CHECK);
  uint32_t first_inf = (uint32_t)n + 1u;
  if (!CHECK && !SAVE && from > 0) {
    load_state(st, snap.base + kSStateBytes * (uint32_t)(from - 1), lane);
    rec += from * snap.step;
    n -= from * snap.step;
  }
  auto fetch = [&](int k) -> float4 {  // record of position k + 1
    const float4 v = __ldg(reinterpret_cast<const float4*>(rec + min(k, n - 1)));
    return make_float4(v.y, v.z, __uint_as_float(tile + __float_as_uint(v.x) * 32u * (uint32_t)sizeof(QT)), 0.f);
  };
  auto slot = [&](int k) -> uint32_t { return recs + 16u * (uint32_t)(k & (kSRecs - 1)); };
  __syncwarp();  // the last tour's reads of the records are done
  sts_f4(slot(lane), fetch(lane));
  __syncwarp();
  // demand and record are read one and two positions ahead
  float4 r = lds_f4(slot(0)), rn = lds_f4(slot(1));
  uint32_t q = lds_q<QT>(__float_as_uint(r.z) + lq);
  auto do_step = [&](int i, bool test) {
    const uint32_t qi = q;
    const float a = r.x, ce = r.y;
    q = lds_q<QT>(__float_as_uint(rn.z) + lq);
    r = rn;
    rn = lds_f4(slot(i + 1));
    if (CHECK) {
      st.step_chk(i, qi, a, ce, Qc, Q, n, first_inf);
    } else {
      st.step(qi, a, ce, Qc);
      if (test) st.check();
    }
  };
  int i = 1, kept = 0;
  auto keep = [&]() {  // after position i
    if (kept < snap.count && i == (kept + 1) * snap.step) {
      save_state(st, snap.base + kSStateBytes * (uint32_t)kept, lane);
      __syncwarp();
      if (lane == 0) st_release_shared(snap.ready, (uint32_t)++kept);
      kept = __shfl_sync(kAll, kept, 0);
    }
  };
  for (int b0 = kSBlock; b0 <= n; b0 += kSBlock) {
    // records b0 + kSBlock .. : the half of the ring that the last block read
    const float4 nx = fetch(b0 + kSBlock + (lane & (kSBlock - 1)));
#pragma unroll(SAVE ? 2 : kSBlock)
    for (int u = 0; u < kSBlock; ++u, ++i) {
      do_step(i, u % kSCheckEvery == kSCheckEvery - 1);
      if (SAVE && u % kSCheckEvery == kSCheckEvery - 1) keep();
    }
    __syncwarp();
    if (lane < kSBlock) sts_f4(slot(b0 + kSBlock + lane), nx);
    __syncwarp();
  }
  for (; i <= n; ++i) {
    do_step(i, true);
    if (SAVE) keep();
  }
  *K_out = st.K;
  *first_inf_out = first_inf;
  *bad = st.ovf;
}

template <typename QT>
__global__ void __launch_bounds__(kSWarps * 32, 1) split_shared_kernel(PipeArgs a, int per_tile, int snap_step, int snap_count) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ uint32_t tile_inf;
  __shared__ int next_tour;
  __shared__ uint32_t snap_ready;
  __shared__ int saved;  // states' distances that the run's tours need not take again
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = a.n_max, Q = a.Q;
  const int64_t S = a.S;
  // shared: deque rings (on 4 KB) | records | the tile's demands
  const uint32_t rings = (smem_u32(smem) + kSRingBytes - 1) & ~(kSRingBytes - 1);
  const uint32_t recs = rings + kSWarps * kSRingBytes + (uint32_t)warp * kSRecs * 16u;
  const uint32_t tile = rings + kSWarps * kSRingBytes + kSWarps * kSRecs * 16u;
  QT* tile_p = reinterpret_cast<QT*>(smem + (tile - smem_u32(smem)));
  const uint32_t ring = rings + kSRingBytes * (uint32_t)warp;
  const int32_t* dem = a.demands + a.dem_off[0];
  const int64_t tpt = (S + 31) / 32;
  // this CTA's run of the pairs (tile, tour), tile by tile
  const int64_t pairs = tpt * a.B;
  int64_t lo = pairs * blockIdx.x / gridDim.x, hi = pairs * (blockIdx.x + 1) / gridDim.x;
  if (per_tile > 0) {  // or its share of one tile's tours
    const int64_t t = blockIdx.x / per_tile, j = blockIdx.x % per_tile;
    lo = t * a.B + a.B * j / per_tile;
    hi = t * a.B + a.B * (j + 1) / per_tile;
  }
  const Snapshots snap{(tile + (uint32_t)(n * 32 * (int)sizeof(QT)) + 15u) & ~15u, snap_step, snap_count, &snap_ready};
  uint32_t any_inf = 0, any_fb = 0;
  bool neg = false;
  for (int64_t at = lo; at < hi;) {
    const int64_t t = at / a.B;
    const int b_lo = (int)(at - t * a.B);
    const int b_hi = (int)imin64(a.B, b_lo + (hi - at));
    at += b_hi - b_lo;
    const int64_t s0 = t * 32;
    const int rows = (int)imin64(32, S - s0);
    __syncthreads();  // every warp is done with the last tile
    if (threadIdx.x == 0) {
      tile_inf = 0u;
      next_tour = b_lo;
      snap_ready = 0u;
      saved = 0;
    }
    __syncthreads();
    // ---- the tile by customer; rows past the last are zeros
    {
      constexpr int kPer = 4 / (int)sizeof(QT);  // rows per 32-bit word
      const int32_t* src = dem + s0 * n;
      for (int k = threadIdx.x; k < n * (32 / kPer); k += blockDim.x) {
        const int g = k / n, c = k - g * n;
        uint32_t word = 0u, inf = 0u;
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
          const int row = g * kPer + e;
          const int v = row < rows ? __ldg(src + (int64_t)row * n + c) : 0;
          if (v > Q) inf |= 1u << row;
          neg |= v < 0;
          word |= (uint32_t)min(max(v, 0), Q + 1) << (8 * (int)sizeof(QT) * e);
        }
        reinterpret_cast<uint32_t*>(tile_p)[c * (32 / kPer) + g] = word;
        if (inf) atomicOr(&tile_inf, inf);
      }
    }
    if (snap_step > 0) {
      int mine = 0;
      for (int b = b_lo + (int)threadIdx.x; b < b_hi; b += blockDim.x)
        mine += min(a.prefix[b] / snap_step, snap_count);
      mine = __reduce_add_sync(kAll, mine);
      if (lane == 0 && mine) atomicAdd(&saved, mine);
    }
    __syncthreads();
    const uint32_t tf = tile_inf;
    any_inf |= tf;
    const bool live = lane < rows;
    // worth tour 0's extra run: some of it is another warp's idle time
    const bool resume = tf == 0u && (int64_t)saved * snap_step > 2 * (int64_t)n;
    if (resume && warp == 0) {
      float K;
      uint32_t first_inf;
      bool bad;
      run_tour<QT, false, true>(n, Q, tile, ring, recs, a.rec + a.rec_off[0], lane, snap, 0, &K, &first_inf, &bad);
    }
    for (;;) {
      int b = 0;
      if (lane == 0) b = atomicAdd(&next_tour, 1);
      b = __shfl_sync(kAll, b, 0);
      if (b >= b_hi) break;
      const StepRec* rec = a.rec + a.rec_off[b];
      float K;
      uint32_t first_inf;
      bool bad;
      int from = 0;
      if (resume) {
        if (lane == 0) from = min(a.prefix[b] / snap_step, (int)ld_acquire_shared(&snap_ready));
        // lane 0's acquire orders its own reads only; the barrier carries the
        // order to the lanes that read the state with it (a shuffle does not)
        __syncwarp();
        from = __shfl_sync(kAll, from, 0);
      }
      if (tf) run_tour<QT, true, false>(n, Q, tile, ring, recs, rec, lane, snap, 0, &K, &first_inf, &bad);
      else run_tour<QT, false, false>(n, Q, tile, ring, recs, rec, lane, snap, from, &K, &first_inf, &bad);
      bad = bad && live;
      if (live) {
        const int64_t g = (int64_t)b * S + s0 + lane;
        if (bad) a.fb_list[atomicAdd(a.fb_count, 1u)] = (unsigned long long)g;
        else a.cost[g] = first_inf <= (uint32_t)n ? CUDART_INF_F : (float)((double)K + a.Dn[b]);
      }
      any_fb |= __ballot_sync(kAll, bad);
    }
  }
  const bool any_neg = __any_sync(kAll, neg);
  if (lane == 0) {
    if (any_inf) atomicOr(a.status, SDP_FLAG_INFEASIBLE);
    if (any_fb) atomicOr(a.status, SDP_FLAG_FALLBACK);
    if (any_neg) atomicOr(a.status, SDP_FLAG_NEG_INPUT);
  }
}

// dynamic shared memory of a CTA: 227 KB less the kernel's own variables
constexpr size_t kSSmemMax = 227 * 1024 - 256;
size_t shared_smem(int n, int Q) {
  return (size_t)(kSWarps + 1) * kSRingBytes + (size_t)kSWarps * kSRecs * 16 +
         (size_t)n * 32 * (Q <= 254 ? 1 : 2) + 16;
}

template <typename QT>
int launch_s(const PipeArgs& a, int grid, int per_tile, cudaStream_t st) {
  auto k = split_shared_kernel<QT>;
  // tour 0's states: as many as fit, every 8 positions at best (the last one
  // before position n)
  const size_t tiles = shared_smem(a.n_max, a.Q);
  const int fit = tiles < kSSmemMax ? (int)((kSSmemMax - tiles) / kSStateBytes) : 0;
  int step = 0, count = 0;
  if (a.prefix && fit > 0 && a.n_max > 8) {
    step = (((a.n_max - 1) / 8 + fit - 1) / fit) * 8;
    count = std::min(fit, (a.n_max - 1) / step);
  }
  const size_t smem = tiles + (size_t)count * kSStateBytes;
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return (int)e;
  k<<<grid, kSWarps * 32, smem, st>>>(a, per_tile, step, count);
  return (int)cudaGetLastError();
}

}  // namespace

// At least two tours per warp, so that a staged tile keeps the warps busy.
bool shared_supported(int n, int Q, int B) {
  return n >= 1 && n <= 65535 && Q >= 1 && Q <= 32767 && B >= 2 * kSWarps &&
         shared_smem(n, Q) <= kSSmemMax;
}

// Below two tours per warp of the chip, a run of pairs that crosses from one
// tile into the next takes a barrier and one more tour's time for a few pairs,
// and a run of at least 32 leaves SMs without any where there are few: there
// every tile gets an equal number of CTAs, as many as there are SMs for, if its
// warps then take fewer tours one after the other than the worst run would, or
// as many on no fewer SMs.  Against runs, where these took one tour more than
// the pipelined kernel had (n = 1000, Q = 100): 100 tours x 16 tiles 423 -> 220
// us (pipelined 300), 64 x 1 257 -> 182 (222), 100 x 63 562 -> 443 (613).
int launch_split_shared(const PipeArgs& a, cudaStream_t st) {
  const int64_t tiles = (a.S + 31) / 32, pairs = tiles * a.B, sms = num_sms();
  int per_tile = 0;
  int64_t grid = imin64(sms, (pairs + kSWarps - 1) / kSWarps);
  if (pairs < 2 * kSWarps * sms) {  // so tiles < SMs, as B >= 64, and a run crosses once
    const int64_t run = (pairs + grid - 1) / grid;
    const int64_t run_tours = tiles == 1 ? (run + kSWarps - 1) / kSWarps : (run - 2) / kSWarps + 2;
    const int64_t share = imin64(a.B, sms / tiles);
    const int64_t own_tours = ((a.B + share - 1) / share + kSWarps - 1) / kSWarps;
    if (own_tours < run_tours || (own_tours == run_tours && tiles * share >= grid)) {
      per_tile = (int)share;
      grid = tiles * share;
    }
  }
  return a.Q <= 254 ? launch_s<uint8_t>(a, (int)grid, per_tile, st)
                    : launch_s<uint16_t>(a, (int)grid, per_tile, st);
}

}  // namespace sdp
