// reinsert_chain.cu -- order-up-to reinsertion over the states that a policy
// can reach (Sec. 2 "Instantiation B", Eq. eqdp2; Algorithm "SolveBatchDP"),
// one scenario per lane, for sm_103a.
//
// Why.  After a delivery on day t the inventory is U - d_t whatever it was
// before, so on day s the state is max(0, U - d_t - ... - d_{s-1}) for the
// day t of the last delivery (or I0 minus the consumption so far): at most
// t + 1 states a day out of U + 1, and only those above zero differ, about
// U / mean consumption of them.  The kernels of reinsert.cu evaluate all U + 1
// states (T U = 12,060 at T = 60, U = 200; the reachable ones are about
// 1,500).  Where only the value from I0 and its policy are wanted, this
// kernel evaluates the reachable states alone, with the FP32 operations of
// those kernels on each (same bits).
//
// Chains.  With P(s) = d_0 + ... + d_{s-1}, "chain t" is the run of states
// after a delivery on day t: A = U + P(t), I_s = A - P(s) for s = t+1 .. z-1,
// z the first day (or T) that starts empty; from z on every chain is the
// empty chain, whose C_s(0) is kept per day.  Backward along a chain
//     nd_s = e(I_s - d_s) + C_{s+1},  C_s = min(dv_s, nd_s),
//     dv_s = base_s = f_s + G_{s+1}(U - d_s)   (+ c (U - I_s)),
// down to s = t + 1, and its last nd (s = t) is G_{t+1}(U - d_t), from which
// base_t follows.  Days run backward and chain t needs base_s of s > t only,
// so four chains t .. t - 3 walk down together to day t + 1 (one shared load
// of (base_s, P(s)) serves four cells of four instructions), and the last
// days close them one after the other.  Where the warp's lanes become empty
// on different days (from zhi down to zlo) a cell carries the choice between
// a running and an empty chain; below zlo all of them run.  The days are the
// warp's (uniform), so no loop diverges.  The delivery days are not kept:
// only the few chains on the path from I0 matter, and they are walked again.
//
// What bounds it: the fixed latencies of a cell's dependent operations with
// 8 warps per SM (14 bytes of shared memory per scenario-day).  At T = 60,
// U = 200, mean consumption 8, S = 10^6: 230 warp instructions per day and 32
// scenarios against about 2,100 for the lane kernel; 0.64 ms, the lane kernel
// 5.20 ms.  Four routes: 2.11 ms against 9.9.  Loading a day's record while
// the day above runs gave 5% of that (routes 1%), the L2 prefetch of the next
// tile's rows 4% (3%).  11 warps per SM (16-bit prefix sums, decisions as bits)
// took 263 instructions a day and the same time.  One chain at a time with
// loops of each lane's own length took 1.14 ms (the decisions recorded in
// every cell); two chains the same.
//
// Tiles with a daily cost below zero, or a day that consumes 2^24 / (T + 1) or
// more, take tests that the others do without (ChainTile::days<true>, out of
// line).  In long horizons of little consumption that is the slower way: with
// costs below zero up to 1.7 of the lane kernel's time (U = 40, T = 120, one a
// day), with such days 3.6; at U = 200, T = 60 0.9.
#include <math.h>
#include <math_constants.h>

#include "async_copy.cuh"
#include "dependent.cuh"
#include "sdp_internal.cuh"

namespace sdp {

namespace {

constexpr int kChains = 4;          // chains walked together
constexpr int kChainMaxWarps = 16;
constexpr int kChainMinWarps = 4;   // per SM (reinsert_chain_supported)
constexpr int kChainMaxT = 254;     // days are kept in bytes
constexpr int kChainSample = 8;     // scenarios that the choice of kernel looks at
constexpr size_t kChainSmem = 227 * 1024 - 64;  // dynamic shared memory of a CTA, less the kernel's own

// Per warp: float2 (base, P) [T+1][32], the empty state's cost [T+1][32], its
// first delivery from each day on [T+1][32] bytes, the policy rows [32][T]
// bytes (T + 1 of them to keep 16 bytes) and the packed route capacities
// [RK/4][T][32].
__host__ __device__ constexpr size_t chain_warp_bytes(int T, int rk) {
  return (size_t)(T + 1) * 32 * 14 + (size_t)(rk / 4) * T * 32 * 4;
}
// CTA: daily costs (f_t, or the route costs [T][RK]), then the table
__host__ __device__ constexpr size_t chain_head_bytes(int T, int U, bool table, int rk) {
  return (((size_t)T * (rk ? rk : 1) + (table ? U + 1 : 0)) * 4 + 15) & ~(size_t)15;
}

// A tile's chains: pointers are the lane's own (shared rows are strided by 32).
template <bool TABLE, bool UNIT, int RK>
struct ChainTile {
  static constexpr int CW = RK / 4;            // capacity words per scenario-day
  static constexpr int DW = RK > 0 ? RK : 1;   // daily costs per day
  int T, lane;
  float h, p, np, c, fU, e0;
  int dmax;                // consumptions enter the prefix sums up to dmax
  bool negc;               // some daily cost is negative
  const float* day_sm;     // [T][DW]
  const float* tab_sm;
  float2* bp;              // (base, P) [s * 32]
  float* zs;               // the empty state's cost [s * 32]
  unsigned char* nz;       // its first delivery [s * 32]
  unsigned char* pol;      // the warp's room for the policy
  const uint32_t* cap;     // [(w T + s) * 32]
  const int32_t* crow;     // the scenario's consumption
  float zc, zn;            // C_{t+1}(0); what `left` adds: C, or e(0) + C in linear mode
  int zfirst;

  // the routes of a day: costs, and capacities as floats 2^23 + capacity (a
  // byte under the exponent 0x4B)
  struct Routes {
    float cost[DW], cap[DW];
  };
  __device__ __forceinline__ Routes routes_of(int s) const {
    Routes r;
#pragma unroll
    for (int w = 0; w < CW; ++w) {
      const uint32_t cw = cap[(w * T + s) * 32];
      const float4 rc = *reinterpret_cast<const float4*>(day_sm + s * DW + 4 * w);
      const float cs[4] = {rc.x, rc.y, rc.z, rc.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        r.cost[(4 * w + e) % DW] = cs[e];
        r.cap[(4 * w + e) % DW] = __uint_as_float(__byte_perm(cw, 0x4B000000u, 0x7540u | e));
      }
    }
    return r;
  }
  // the delivery's value from state I of a day (v: its base): the cheapest
  // route that carries U - I, +inf when none does
  __device__ __forceinline__ float deliver(const Routes& r, float v, float I) const {
    float dv = v;
    if (RK > 0) {
      const float qm = __fsub_rn(fU + 8388608.f, I);
      float F = CUDART_INF_F;
#pragma unroll
      for (int k = 0; k < RK; ++k)
        if (qm <= r.cap[k]) F = fminf(F, r.cost[k]);
      dv = __fadd_rn(F, v);
    }
    if (UNIT) dv = __fadd_rn(dv, __fmul_rn(c, __fsub_rn(fU, I)));
    return dv;
  }
  // nd of the day before day s >= 1, whose state x = A - P(s) this is: e(x)
  // + C for x > 0; below, the stockout's cost on the empty state's zv.
  // far (EXACT): what day s - 1 consumes if that is dmax or more, else 0; it is
  // taken as it stands where the chain was still running on it, which is where
  // this nd is used.
  template <bool EXACT>
  __device__ __forceinline__ float left(float A, float x, float C, float zv, int s, int far) const {
    const bool on = x > 0.f;
    if (TABLE) return __fadd_rn(tab_sm[max((int)x, 0)], on ? C : zv);
    float m = x;
    if (EXACT && far > 0 && !on)
      m = -(float)(far - (int)fmaxf(__fsub_rn(A, bp[(s - 1) * 32].y), 0.f));
    return __fadd_rn(__fmul_rn(on ? h : np, m), on ? C : zv);
  }
  // what day s - 1 consumes if that is dmax or more (of a day that mark() marked)
  __device__ __forceinline__ int beyond(int s) const {
    if (TABLE || !pol[s - 1] || __fsub_rn(bp[s * 32].y, bp[(s - 1) * 32].y) < (float)dmax) return 0;
    return __ldg(crow + s - 1);
  }
  // the days on which some lane consumes dmax or more, in the policy's room
  __device__ __forceinline__ void mark() {
    for (int t = 0; t < T; ++t) {
      const bool any = __any_sync(0xffffffffu, __fsub_rn(bp[(t + 1) * 32].y, bp[t * 32].y) >= (float)dmax);
      if (lane == 0) pol[t] = any;
    }
    __syncwarp();
  }

  // day s of a chain at (A, nd); JOIN: it may still be empty
  template <bool SLOW, bool JOIN>
  __device__ __forceinline__ void cell(int s, float2 v, const Routes& r, float z, int far, float A, float& nd) const {
    const float I = __fsub_rn(A, v.y);
    const float dv = deliver(r, v.x, I);
    float C;
    if (SLOW) C = dv < nd && (!negc || I < fU) ? dv : nd;
    else if (TABLE) C = dv < nd ? dv : nd;
    else C = fminf(dv, nd);
    if (JOIN) nd = left<SLOW>(A, I, C, z, s, far);
    else nd = __fadd_rn(TABLE ? tab_sm[(int)I] : __fmul_rn(h, I), C);
  }
  // day s of the four chains
  template <bool SLOW, bool JOIN>
  __device__ __forceinline__ void cells(int s, float2 v, float z, const float* A, float* nd) const {
    const Routes r = routes_of(s);
    const int far = SLOW && JOIN ? beyond(s) : 0;
#pragma unroll
    for (int j = 0; j < kChains; ++j) cell<SLOW, JOIN>(s, v, r, z, far, A[j], nd[j]);
  }

  // All the days of the tile.  SLOW: some daily cost is negative or some
  // consumption above dmax; otherwise no state equal to U gains by a delivery of
  // nothing, and stockouts are the prefix loads' own.  (The minimum is an FMNMX:
  // with h, p and c bounded, nd is never NaN, and a NaN delivery is not chosen
  // either way.)
  template <bool SLOW>
  __device__ __forceinline__ void days() {
    if (SLOW) mark();
    // all chains of the warp are empty from day zhi on (or zhi = T), and
    // all four are running from day zlo - 1 down (both only fall)
    int zhi = T, zlo = T;
    for (int t = T - 1; t >= 0; t -= kChains) {
      float A[kChains], P[kChains], nd[kChains];
#pragma unroll
      for (int j = 0; j < kChains; ++j) {
        P[j] = bp[max(t - j, 0) * 32].y;
        A[j] = __fadd_rn(fU, P[j]);
      }
      while (zhi - 1 > t && !__any_sync(0xffffffffu, A[0] > bp[(zhi - 1) * 32].y)) --zhi;
      zlo = min(zlo, zhi);
      while (zlo - 1 > t && !__all_sync(0xffffffffu, A[kChains - 1] > bp[(zlo - 1) * 32].y)) --zlo;
      {
        const float Pz = bp[zhi * 32].y, z = zs[zhi * 32];
        const int far = SLOW ? beyond(zhi) : 0;
#pragma unroll
        for (int j = 0; j < kChains; ++j)
          nd[j] = left<SLOW>(A[j], __fsub_rn(A[j], Pz), -0.f, z, zhi, far);
      }
      // the next day's record is loaded while this day's cells run
      int s = zhi - 1;
      float2 v = bp[max(s, 0) * 32];
#pragma unroll 1
      for (; s >= zlo; --s) {
        const float2 vn = bp[max(s - 1, 0) * 32];
        cells<SLOW, true>(s, v, zs[s * 32], A, nd);
        v = vn;
      }
#pragma unroll 4
      for (; s > t; --s) {
        const float2 vn = bp[max(s - 1, 0) * 32];
        cells<SLOW, false>(s, v, 0.f, A, nd);
        v = vn;
      }
      // days t .. t - 3: each chain comes down to its day, which gives that
      // day's base and empty state, and the chains below take the day
      float Pn = bp[(t + 1) * 32].y;
#pragma unroll
      for (int j = 0; j < kChains; ++j) {
        const int d0 = t - j;
        if (d0 < 0) break;
        const float base = RK > 0 ? nd[j] : __fadd_rn(day_sm[d0], nd[j]);
        float d = __fsub_rn(Pn, P[j]);
        Pn = P[j];
        if (SLOW && d >= (float)dmax) d = (float)max(__ldg(crow + d0), 0);
        const Routes r = routes_of(d0);
        const float G0 = TABLE ? __fadd_rn(e0, zc) : zn;
        const float n0 = (TABLE || d == 0.f) ? G0 : __fadd_rn(G0, __fmul_rn(p, d));
        const float dv = deliver(r, base, 0.f);
        const bool dec = fU > 0.f && dv < n0;
        zc = dec ? dv : n0;
        zfirst = dec ? d0 : zfirst;
        nz[d0 * 32] = (unsigned char)zfirst;
        zn = TABLE ? zc : __fadd_rn(e0, zc);
        bp[d0 * 32].x = base;
        zs[d0 * 32] = zn;
        if (d0 > 0) {
          const int far = SLOW ? beyond(d0) : 0;
#pragma unroll
          for (int k = j + 1; k < kChains; ++k)
            cell<SLOW, true>(d0, make_float2(base, P[j]), r, zn, far, A[k], nd[k]);
        }
      }
    }
    if (SLOW) __syncwarp();  // the marks are read before the policy takes their room
  }
};

// Out of line: inlined, the tests of the rare tiles cost the others 1.5% (5% with
// four routes).  A copy keeps the members in registers, and pointers made from
// the block's own array are known to be shared memory.
template <bool TABLE, bool UNIT, int RK>
__device__ __noinline__ float slow_days(const ChainTile<TABLE, UNIT, RK>& tile) {
  extern __shared__ __align__(16) unsigned char smem[];
  auto at = [&](const void* q) -> unsigned char* { return smem + (smem_u32(q) - smem_u32(smem)); };
  ChainTile<TABLE, UNIT, RK> t = tile;
  t.day_sm = reinterpret_cast<const float*>(at(tile.day_sm));
  t.tab_sm = reinterpret_cast<const float*>(at(tile.tab_sm));
  t.bp = reinterpret_cast<float2*>(at(tile.bp));
  t.zs = reinterpret_cast<float*>(at(tile.zs));
  t.nz = at(tile.nz);
  t.pol = at(tile.pol);
  t.cap = reinterpret_cast<const uint32_t*>(at(tile.cap));
  t.template days<true>();
  return t.zc;
}

template <bool TABLE, bool UNIT, int RK>
__global__ void __launch_bounds__(kChainMaxWarps * 32, 1) reinsert_chain_kernel(ReinsertArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  dep_launch();
  if (a.mean_counter && blockIdx.x == 0 && threadIdx.x == 0) *a.mean_counter = 0u;
  constexpr int CW = RK / 4;                // capacity words per scenario-day
  constexpr int DW = RK > 0 ? RK : 1;       // daily costs per day
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int T = a.T, U = a.U;
  const int K = RK > 0 ? a.n_routes : 0;
  if ((TABLE || RK > 0) && a.sparse_load) {  // every CTA adds up the same scenarios' consumption
    __shared__ uint32_t used;
    if (threadIdx.x == 0) used = 0u;
    __syncthreads();
    uint32_t v = 0u;
#pragma unroll 4
    for (int k = threadIdx.x; k < kChainSample * T; k += blockDim.x) {
      const int64_t s = (a.S - 1) * (k / T) / (kChainSample - 1);
      v += (uint32_t)min(max(__ldg(a.cons + s * T + k % T), 0), U);
    }
    v = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) atomicAdd(&used, v);
    __syncthreads();
    const bool leave = used < a.sparse_load;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.sparse = leave ? 1u : 0u;
    if (leave) return;
  }
  float* day_sm = reinterpret_cast<float*>(smem);  // [T][DW]
  float* tab_sm = day_sm + T * DW;
  unsigned char* wb = smem + chain_head_bytes(T, U, TABLE, RK) + chain_warp_bytes(T, RK) * warp;
  float2* bp = reinterpret_cast<float2*>(wb) + lane;                           // [s * 32]
  float* zs = reinterpret_cast<float*>(wb + (size_t)(T + 1) * 256) + lane;     // [s * 32]
  unsigned char* nz = wb + (size_t)(T + 1) * 384 + lane;                       // [s * 32]
  unsigned char* pol = wb + (size_t)(T + 1) * 416;
  uint32_t* cap = reinterpret_cast<uint32_t*>(wb + (size_t)(T + 1) * 448) + lane;  // [(w T + t) * 32]
  // a negative cost can make delivering nothing look cheaper than not
  // delivering: only then a chain's states equal to U need a test
  bool negc = false;
  for (int i = threadIdx.x; i < T * DW; i += blockDim.x) {
    float v;
    if (RK > 0) {
      const int t = i / DW, r = i % DW;
      v = r < K ? __ldg(a.route_cost + t * K + r) : CUDART_INF_F;
    } else {
      v = __ldg(a.fixed + i);
    }
    day_sm[i] = v;
    negc |= v < 0.f;
  }
  if (TABLE)
    for (int i = threadIdx.x; i <= U; i += blockDim.x) tab_sm[i] = __ldg(a.table + i);
  negc = __syncthreads_or(negc);

  const float h = a.h, p = a.p, c = a.c;
  const float np = -p;
  const float fU = (float)U;
  const float e0 = TABLE ? tab_sm[0] : __fmul_rn(h, 0.f);
  // consumptions enter the prefix sums up to dmax, so that sums stay below
  // 2^24 (exact); what a day consumes beyond it counts in its stockout only
  const int dmax = (1 << 24) / (T + 1) - 1;
  bool neg = false;
  const int64_t tiles = (a.S + 31) / 32;
  const bool vec = (T & 3) == 0 && (reinterpret_cast<uintptr_t>(a.cons) & 15) == 0;
  const bool vcap = RK > 0 && K == 4 && (reinterpret_cast<uintptr_t>(a.route_cap) & 15) == 0;

  for (int64_t tile = (int64_t)blockIdx.x * nwarps + warp; tile < tiles;
       tile += (int64_t)gridDim.x * nwarps) {
    const int64_t s0 = tile * 32;
    const bool live = lane < a.S - s0;
    // the warp's next rows on their way to L2 meanwhile
    const int64_t next = s0 + 32 * (int64_t)gridDim.x * nwarps;
    if (lane == 0 && next < a.S) {
      const int64_t rows = imin64(32, a.S - next);
      auto ahead = [&](const int32_t* p, int64_t row) {
        p += next * row;
        if ((reinterpret_cast<uintptr_t>(p) & 15) == 0 && rows * row >= 4)
          bulk_prefetch_l2(p, (uint32_t)(rows * row * 4) & ~15u);
      };
      ahead(a.cons, T);
      if (RK > 0) ahead(a.route_cap, (int64_t)T * K);
    }
    // a lane without a scenario follows the tile's first
    const int32_t* crow = a.cons + (s0 + (live ? lane : 0)) * T;
    const int32_t* caprow = RK > 0 ? a.route_cap + (s0 + (live ? lane : 0)) * (int64_t)T * K : nullptr;
    bool big = false;  // a consumption above dmax
    {
      float P = 0.f;
      auto put = [&](int t, int d) {
        neg |= live && d < 0;
        big |= d > dmax;
        bp[t * 32].y = P;
        P = __fadd_rn(P, (float)min(max(d, 0), dmax));
      };
      if (vec) {
#pragma unroll 4
        for (int t = 0; t < T; t += 4) {
          const int4 v = __ldg(reinterpret_cast<const int4*>(crow + t));
          put(t, v.x);
          put(t + 1, v.y);
          put(t + 2, v.z);
          put(t + 3, v.w);
        }
      } else {
#pragma unroll 4
        for (int t = 0; t < T; ++t) put(t, __ldg(crow + t));
      }
      bp[T * 32].y = P;
    }
    // route capacities, a byte each (a refill is at most U <= 255)
    if (RK > 0) {
      auto pack = [](int x, int y, int z, int w) -> uint32_t {
        auto b = [](int v) -> uint32_t { return (uint32_t)min(max(v, 0), 255); };
        return b(x) | b(y) << 8 | b(z) << 16 | b(w) << 24;
      };
      if (vcap) {
#pragma unroll 4
        for (int t = 0; t < T; ++t) {
          const int4 v = __ldg(reinterpret_cast<const int4*>(caprow) + t);
          cap[t * 32] = pack(v.x, v.y, v.z, v.w);
        }
      } else {
#pragma unroll 2
        for (int t = 0; t < T; ++t)
#pragma unroll
          for (int w = 0; w < CW; ++w) {
            int v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = 4 * w + e < K ? __ldg(caprow + t * K + 4 * w + e) : 0;
            cap[(w * T + t) * 32] = pack(v[0], v[1], v[2], v[3]);
          }
      }
    }
    ChainTile<TABLE, UNIT, RK> ct;
    ct.T = T; ct.lane = lane;
    ct.h = h; ct.p = p; ct.np = np; ct.c = c; ct.fU = fU; ct.e0 = e0;
    ct.dmax = dmax; ct.negc = negc;
    ct.day_sm = day_sm; ct.tab_sm = tab_sm;
    ct.bp = bp; ct.zs = zs; ct.nz = nz; ct.pol = pol; ct.cap = cap; ct.crow = crow;
    ct.zc = -0.f;
    ct.zn = TABLE ? ct.zc : __fadd_rn(e0, ct.zc);
    ct.zfirst = T;
    zs[T * 32] = ct.zn;
    nz[T * 32] = (unsigned char)T;
    const bool slow = negc || __any_sync(0xffffffffu, big);
    if (slow) {
      const ChainTile<TABLE, UNIT, RK> copy = ct;
      ct.zc = slow_days(copy);
    } else {
      ct.template days<false>();
    }

    // ---- the path from I0.  Only a few chains are on it, so the days on
    // which a chain delivers are found by walking it again.
    // From the state A - P(t0) > 0 of day t0 on: the first day that delivers
    // (T: none); C: the value at t0.
    auto walk = [&](float A, int t0, float& C) -> int {
      int z = t0, hi = T;  // the first day from t0 on that starts empty, or T
      while (z < hi) {
        const int mid = (z + hi) >> 1;
        if (bp[mid * 32].y >= A) hi = mid; else z = mid + 1;
      }
      int first = nz[z * 32];
      if (z == t0) return first;
      const float x = __fsub_rn(A, bp[z * 32].y);
      const int far = slow && !TABLE ? max(__ldg(crow + z - 1), 0) : 0;
      float nd = slow ? ct.template left<true>(A, x, -0.f, zs[z * 32], z, far >= dmax ? far : 0)
                      : ct.template left<false>(A, x, -0.f, zs[z * 32], z, 0);
#pragma unroll 2
      for (int s = z - 1; s >= t0; --s) {
        const float2 v = bp[s * 32];
        const float I = __fsub_rn(A, v.y);
        const float dv = ct.deliver(ct.routes_of(s), v.x, I);
        const bool dec = dv < nd && (!negc || I < fU);
        C = dec ? dv : nd;
        if (dec) first = s;
        nd = __fadd_rn(TABLE ? tab_sm[(int)I] : __fmul_rn(h, I), C);
      }
      return first;
    };
    float A = (float)a.I0, C = ct.zc;
    int day = walk(A, 0, C);
    if (live) a.value[s0 + lane] = __fadd_rn(0.f, C);
    if (a.policy) {
      // rows of zeros and the delivery days, in the room kept for them
      unsigned char* st = pol;  // [32][T]
      for (int k = lane; k < 2 * T; k += 32) reinterpret_cast<uint4*>(st)[k] = make_uint4(0u, 0u, 0u, 0u);
      __syncwarp();
      while (day < T) {
        const float Pd = bp[day * 32].y;
        int pv = 1;
        if (RK > 0) {  // the cheapest route that holds U - I, the first on ties
          const int q = U - (int)fmaxf(__fsub_rn(A, Pd), 0.f);
          float best = CUDART_INF_F;
          pv = 0;
          for (int r = 0; r < K; ++r) {
            const float fr = day_sm[day * DW + r];
            const int cr = (int)((cap[((r >> 2) * T + day) * 32] >> (8 * (r & 3))) & 0xFFu);
            if (cr >= q && fr < best) {
              best = fr;
              pv = r + 1;
            }
          }
        }
        st[lane * T + day] = (unsigned char)pv;
        A = __fadd_rn(fU, Pd);
        day = walk(A, day + 1, C);
      }
      __syncwarp();
      uint8_t* dst = a.policy + s0 * T;
      const int bytes = (int)imin64(32, a.S - s0) * T;
      int done = 0;
      if ((reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
        done = bytes & ~15;
        for (int k = lane; k < done / 16; k += 32)
          reinterpret_cast<uint4*>(dst)[k] = reinterpret_cast<const uint4*>(st)[k];
      }
      for (int k = done + lane; k < bytes; k += 32) dst[k] = st[k];
    }
    __syncwarp();  // the tile's rows are read before the next one's are written
  }
  if (__any_sync(0xffffffffu, neg) && lane == 0) atomicOr(a.status, SDP_FLAG_NEG_INPUT);
}

int chain_rk(int n_routes) { return n_routes == 0 ? 0 : n_routes <= 4 ? 4 : 8; }

int chain_warps(int T, int U, bool table, int n_routes) {
  const int rk = chain_rk(n_routes);
  int w = kChainMaxWarps;
  while (w > 0 && chain_head_bytes(T, U, table, rk) + chain_warp_bytes(T, rk) * w > kChainSmem) --w;
  return w;
}

template <bool TABLE, bool UNIT, int RK>
int launch_chain(const ReinsertArgs& a, cudaStream_t st) {
  auto k = reinsert_chain_kernel<TABLE, UNIT, RK>;
  const int64_t tiles = (a.S + 31) / 32;
  // few tiles: as many SMs as possible, a warp each
  const int warps = (int)imin64(chain_warps(a.T, a.U, TABLE, a.n_routes),
                                (tiles + num_sms() - 1) / num_sms());
  const size_t smem = chain_head_bytes(a.T, a.U, TABLE, RK) + chain_warp_bytes(a.T, RK) * warps;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return (int)e;
  const int grid = (int)imin64((tiles + warps - 1) / warps, (int64_t)num_sms());
  if (grid > 0) k<<<grid, warps * 32, smem, st>>>(a);
  return (int)cudaGetLastError();
}

}  // namespace

// A chain has at most T / 2 cells a day (no consumption), the lane kernel 32
// ceil((U + 1) / 32) states, and with table costs or routes a cell costs more
// than a state.  Against the lane kernel on 10^5 scenarios that consume next to
// nothing, the longest T that did not lose:
//   no routes: 2.5 x states (32 states, T = 80: 0.93), with unit costs 72 of 32
//     states (80: 1.07);
//   table: 72 (80: 1.29) of 32 states, 80 of 64 (128: 1.31), 120 of 96;
//   1 to 4 routes: 56 (72: 1.71) of 32, 80 of 64 (99: 1.11);
//   5 to 8 routes: 48 of 64 (80: 1.87), 64 of 96 (80: 1.36), 80 of 128, and no
//     gain worth having at 32 states (T = 20: 0.94-1.17, T = 80: 3.1).
// At 32 states these are the limits.  From 64 states on, longer T with what
// stock is held for takes 0.4 to 0.8 of the lane kernel's time: there a sample
// decides (reinsert_sparse_load).
//   The other end, with few warps per SM: four (T = 128; 99 with routes, 80 with
// five and more) at U = 200, 8 a day, S = 2 10^5: 582 us, the lane kernel 2,644
// (1,174 and 3,886 with four routes; 2,176 and 4,721 with eight).  Fewer were
// not tried.
//
// h, p and c are bounded so that no cost of a state is infinite or NaN (the
// kernel takes minima, and multiplies p by shortfalls of 0).
bool reinsert_chain_supported(int T, int U, bool table, int n_routes, float h, float p, float c) {
  if (!(fabsf(h) <= 1e25f && fabsf(p) <= 1e25f && fabsf(c) <= 1e25f)) return false;
  if (T < 1 || T > kChainMaxT || U < 0 || U > 1023 || n_routes < 0 || n_routes > 8) return false;
  if (n_routes > 0 && (U > 255 || table)) return false;
  const int states = 32 * ((U + 1 + 31) / 32);
  if (states == 32 && (n_routes > 4 || T > (n_routes ? 56 : table || c != 0.f ? 72 : 80))) return false;
  return 2 * T <= 5 * states && chain_warps(T, U, table, n_routes) >= kChainMinWarps;
}

// The consumption of the kChainSample scenarios, each day's up to U, below which
// the chains leave a call to the lane kernel.  With T0 the limits above, the
// chains take about (T / T0)^1.5 of its time without consumption, and in between
// in proportion to a day's cells plus 20; a chain lasts U / (mean consumption)
// days.  (64 states, 8 routes, T = 80, U = 40: the sides meet at 4.8 a day;
// measured 1.12 at 3 a day, 0.74 at 8.)
uint32_t reinsert_sparse_load(int T, int U, bool table, int n_routes) {
  const double states = 32 * ((U + 1 + 31) / 32);
  const double t0 = n_routes > 4 ? 16.0 + states / 2 : n_routes > 0 ? 32.0 + 0.75 * states : 1.25 * states;
  if (states < 64 || !(table || n_routes) || T <= t0) return 0u;
  const double cells = (T / 2.0 + 20.0) / pow(T / t0, 1.5) - 20.0;  // a day's, where the sides meet
  const double days = T * (1.0 - sqrt(fmax(0.0, 1.0 - 2.0 * cells / T)));
  return (uint32_t)(kChainSample * T * (double)U / fmax(days, 1.0));
}

int launch_reinsert_chain(const ReinsertArgs& a, cudaStream_t st) {
  const bool unit = a.c != 0.f;
  if (a.n_routes > 4)
    return unit ? launch_chain<false, true, 8>(a, st) : launch_chain<false, false, 8>(a, st);
  if (a.n_routes > 0)
    return unit ? launch_chain<false, true, 4>(a, st) : launch_chain<false, false, 4>(a, st);
  if (a.table) return unit ? launch_chain<true, true, 0>(a, st) : launch_chain<true, false, 0>(a, st);
  return unit ? launch_chain<false, true, 0>(a, st) : launch_chain<false, false, 0>(a, st);
}

}  // namespace sdp
