// Range resolution, segment mask and range-aware strategy selection
// (Section 4.2: Strategy A's skip-list descent lands on the first in-range object;
// Algorithm 7: the segments that intersect [l, h]; range-aware selection:
// A if Y <= tau_A, B if Y >= tau_B, otherwise C).
//
// The skip list's bottom layer is the attribute order, so the descent to the first
// object with attribute >= lo is a lower_bound on the attribute-sorted values, and
// the in-range objects are the positions [pa, pb) of that order.
#include "common.cuh"
#include "internal.h"

namespace unify {

constexpr int kRouteWarps = 8;  // queries per CTA, one warp each

// The first position of the attribute order whose value is not below x (strict), or
// above x (!strict): the 16 lanes of a half warp probe 16 positions per step, so that n =
// 1M takes 6 dependent loads instead of 20. Both halves search at once, each its own x.
__device__ __forceinline__ int half_warp_bound(const int64_t* a, int n, int64_t x, bool strict) {
  const int lane = lane_id(), l16 = lane & 15;
  int lo = 0, hi = n;  // the answer lies in [lo, hi]
  while (__any_sync(kFull, lo < hi)) {
    const int len = hi - lo;
    const int at = lo + (int)((int64_t)(l16 + 1) * len / 17);  // below hi while len > 0, ascending over the lanes
    bool below = false;
    if (len > 0) {
      const int64_t v = __ldg(a + at);
      below = strict ? v < x : v <= x;
    }
    const unsigned bal = (__ballot_sync(kFull, below) >> (lane & 16)) & 0xffffu;
    const int c = __popc(bal);
    const int last = __shfl_sync(kFull, at, (lane & 16) + (c > 0 ? c - 1 : 0));
    const int next = __shfl_sync(kFull, at, (lane & 16) + (c < 16 ? c : 15));
    if (len > 0) {
      if (c < 16) hi = next;
      if (c > 0) lo = last + 1;
    }
  }
  return lo;
}

struct RouteArgs {
  const int64_t* sorted_attr;
  int64_t n;
  int S;
  const int64_t* lo;
  const int64_t* hi;
  int64_t nq;
  int64_t tau_a, tau_b;
  int forced;        // -1: range-aware, else the strategy for every query
  int scan_rows;
  int max_items;     // scan work items per query, at most (the scratch's share of this batch)
  int build_queues;
  int ef_h, ef_p;    // beams of hybrid and post-filter walks
  int32_t* pa;
  int32_t* pb;
  uint32_t* mask;
  int32_t* strat;
  int32_t* nblk;
  int32_t* qbase;
  int32_t* done;
  int32_t* queues;
  int64_t cap_nq;
  int2* items;
  int32_t* counters;
  int32_t* out_counters;  // may be null
  // tensor-core scan: its tables to clear (slots to -1, spans to 0); null without it
  int32_t* tc_slotpos;
  int32_t* tc_spans;
  int64_t tc_slots, tc_spans_n;
};

// One warp per query finds its bounds, mask and strategy; then the CTA's first warp takes
// places in the queues and in the item list for all of its queries (an atomic per queue
// and CTA, not per query), and every warp writes its query's items. Bound by the chain of
// dependent loads of the search. Measured on GB300 (n = 1M; a thread per query and binary
// searches before): 5,000 queries 18 -> 8 us.
__global__ void __launch_bounds__(32 * kRouteWarps) route_kernel(RouteArgs a, const int64_t* __restrict__ seg_bounds,
                                                                 const int32_t* __restrict__ seg_start) {
  __shared__ int s_strat[kRouteWarps], s_nb[kRouteWarps], s_base[kRouteWarps], s_rows[kRouteWarps];
  const int warp = threadIdx.x >> 5, lane = lane_id();
  const int64_t i = (int64_t)blockIdx.x * kRouteWarps + warp;
  const bool valid = i < a.nq;
  int st = -1, nb = 0, Y = 0;
  bool shrt = false;
  if (a.tc_slotpos) {
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = t0; t < a.tc_slots / 4; t += stride)  // tc_slots is a multiple of 128
      reinterpret_cast<int4*>(a.tc_slotpos)[t] = make_int4(-1, -1, -1, -1);
    for (int64_t t = t0; t < a.tc_spans_n; t += stride) a.tc_spans[t] = 0;
  }
  if (valid) {
    const int64_t lo = a.lo[i], hi = a.hi[i];
    const int p = half_warp_bound(a.sorted_attr, (int)a.n, lane < 16 ? lo : hi, lane < 16);
    const int p0 = __shfl_sync(kFull, p, 0);
    int p1 = __shfl_sync(kFull, p, 16);
    if (p1 < p0) p1 = p0;
    bool hit = false;
    if (lane < a.S && lo <= hi) {
      const bool nonempty = __ldg(seg_start + lane + 1) > __ldg(seg_start + lane);
      const bool lower_ok = lane == 0 || __ldg(seg_bounds + lane) <= hi;
      const bool upper_ok = lane == a.S - 1 || lo < __ldg(seg_bounds + lane + 1);
      hit = nonempty && lower_ok && upper_ok;
    }
    const uint32_t m = __ballot_sync(kFull, hit);
    Y = p1 - p0;
    st = a.forced;
    if (st < 0) st = (Y <= a.tau_a) ? UNIFY_PRE : ((Y >= a.tau_b) ? UNIFY_POST : UNIFY_HYBRID);
    if (st == UNIFY_HYBRID) {
      // A hybrid walk expands until ef_h of the objects it met are in range, about one in
      // (rows of its segments) / Y of them; a post-filter walk expands about ef_p. The
      // longest work should start first: hybrid walks that expect to take longer than a
      // post-filter walk (an expansion of theirs costs about 1.5 of one) go before those,
      // the others after. Measured on GB300, 10,000 auto-routed queries over 1M x 128 (4,000
      // short hybrid walks, 2,000 post-filter walks; all hybrid walks first before):
      // float32 1,259 -> 1,096 us, bfloat16 1,182 -> 1,010 us. Post-filter walks before every
      // hybrid one lost 8 % on a batch with ranges that fill a tenth of their segments.
      const unsigned rows = hit ? (unsigned)(__ldg(seg_start + lane + 1) - __ldg(seg_start + lane)) : 0u;
      const int64_t met = __reduce_add_sync(kFull, rows);
      shrt = 3 * (int64_t)a.ef_h * met <= 2 * (int64_t)a.ef_p * Y;
    }
    if (st == UNIFY_PRE) {
      nb = (Y + a.scan_rows - 1) / a.scan_rows;
      nb = nb < 1 ? 1 : nb > a.max_items ? a.max_items : nb;
    }
    if (lane == 0) {
      if (a.pa) a.pa[i] = p0;
      if (a.pb) a.pb[i] = p1;
      if (a.mask) a.mask[i] = m;
      if (a.strat) a.strat[i] = st;
    }
  }
  if (!a.build_queues) return;
  if (lane == 0) {
    s_strat[warp] = st == UNIFY_HYBRID && shrt ? 3 : st;
    s_nb[warp] = nb;
    s_rows[warp] = Y;
  }
  __syncthreads();
  if (warp == 0) {
    const int qst = lane < kRouteWarps ? s_strat[lane] : -1;
    const int qnb = lane < kRouteWarps ? s_nb[lane] : 0;
    const int64_t qi = (int64_t)blockIdx.x * kRouteWarps + lane;
    for (int q = 0; q < 4; ++q) {
      // pre-filter, long hybrid, post-filter, short hybrid
      const bool mine = qst == (q == 0 ? UNIFY_PRE : q == 1 ? UNIFY_HYBRID : q == 2 ? UNIFY_POST : 3);
      const unsigned bal = __ballot_sync(kFull, mine);
      if (bal == 0) continue;
      int base = 0;
      if (lane == 0) base = atomicAdd(&a.counters[q < 3 ? CNT_QA + q : CNT_QS], __popc(bal));
      base = __shfl_sync(kFull, base, 0) + __popc(bal & lanemask_lt());
      if (mine) a.queues[q < 3 ? q * a.cap_nq + base : 2 * a.cap_nq - 1 - base] = (int32_t)qi;
    }
    int incl = qnb;  // inclusive sum of the item counts
    for (int off = 1; off < kRouteWarps; off <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, off);
      if (lane >= off) incl += v;
    }
    int base = 0;
    const int total = __shfl_sync(kFull, incl, kRouteWarps - 1);
    if (lane == 0 && total > 0) base = atomicAdd(&a.counters[CNT_ITEMS], total);
    base = __shfl_sync(kFull, base, 0) + incl - qnb;
    if (a.tc_slotpos) {
      const unsigned y = qst == UNIFY_PRE ? (unsigned)s_rows[lane] : 0u;
      const unsigned long long sum = __reduce_add_sync(kFull, y & 0xffffu) + ((unsigned long long)__reduce_add_sync(kFull, y >> 16) << 16);
      if (lane == 0 && sum > 0) atomicAdd(reinterpret_cast<unsigned long long*>(a.counters + CNT_TC_SUMY), sum);
    }
    if (qst == UNIFY_PRE) {
      s_base[lane] = base;
      a.nblk[qi] = qnb;
      a.qbase[qi] = base;
      a.done[qi] = 0;
    }
  }
  __syncthreads();
  if (st == UNIFY_PRE) {
    for (int t = lane; t < nb; t += 32) a.items[s_base[warp] + t] = make_int2((int)i, t);
    if (a.out_counters && lane == 0) {
      a.out_counters[4 * i] = Y;
      a.out_counters[4 * i + 1] = 0;
      a.out_counters[4 * i + 2] = 0x7fffffff;  // earliest item start (atomicMin)
      a.out_counters[4 * i + 3] = 0;           // latest item end (atomicMax)
    }
  }
}

cudaError_t launch_route(const DeviceIndex& ix, const Scratch& sc, const int64_t* lo, const int64_t* hi,
                         int64_t nq, int64_t tau_a, int64_t tau_b, int forced, int scan_rows,
                         int build_queues, int32_t* out_pa, int32_t* out_pb, uint32_t* out_mask,
                         int32_t* out_strat, const Outputs* outs, const Params* p, cudaStream_t st, bool tc) {
  RouteArgs a;
  a.sorted_attr = ix.sorted_attr;
  a.n = ix.n;
  a.S = ix.S;
  a.lo = lo;
  a.hi = hi;
  a.nq = nq;
  a.tau_a = tau_a;
  a.tau_b = tau_b;
  a.forced = forced;
  a.scan_rows = scan_rows > 0 ? scan_rows : 8192;
  // items and partial lists of cap_nq * kMaxScanBlocks work items, shared by nq <= cap_nq queries
  a.max_items = kMaxScanBlocks;
  if (build_queues && nq > 0) {
    const int64_t share = sc.cap_nq * kMaxScanBlocks / nq;
    a.max_items = (int)(share < kMaxItemsPerQuery ? share : kMaxItemsPerQuery);
  }
  a.build_queues = build_queues;
  a.ef_h = p ? (p->ef > p->k ? p->ef : p->k) : 0;
  a.ef_p = p ? (p->ef_post > p->k ? p->ef_post : p->k) : 0;
  a.pa = out_pa;
  a.pb = out_pb;
  a.mask = out_mask;
  a.strat = out_strat;
  a.nblk = sc.nblk;
  a.qbase = sc.qbase;
  a.done = sc.done;
  a.queues = sc.queues;
  a.cap_nq = sc.cap_nq;
  a.items = sc.items;
  a.counters = sc.counters;
  a.out_counters = outs ? outs->counters : nullptr;
  a.tc_slotpos = tc ? sc.tc_slotpos : nullptr;
  a.tc_slots = sc.tc_slots;
  a.tc_spans = sc.tc_spans;
  a.tc_spans_n = sc.tc_spans_cap;
  if (nq == 0) return cudaSuccess;
  int64_t blocks = (nq + kRouteWarps - 1) / kRouteWarps;
  if (tc) {
    // The tables to clear are as large as the largest batch the handle has seen: CTAs without
    // queries help, four steps of the clearing loop each. Measured on GB300, one query after a
    // batch of 100,000 (6.4 MB of tables): 156 us for the call with a single CTA, 63 with them.
    const int64_t clear = (a.tc_slots + 16 * 32 * kRouteWarps - 1) / (16 * 32 * kRouteWarps);
    const int64_t most = 4ll * ix.num_sms;
    if (blocks < clear) blocks = clear < most ? clear : (blocks < most ? most : blocks);
  }
  route_kernel<<<(unsigned)blocks, 32 * kRouteWarps, 0, st>>>(a, ix.seg_bounds, ix.seg_start);
  return cudaGetLastError();
}

}  // namespace unify
