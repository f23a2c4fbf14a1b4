// The search of one batch in one persistent kernel: hybrid filtering (Strategy
// C), post-filtering (Strategy B) and pre-filtering (Strategy A) of Section 4.2.
//
// Work queue. The router appends every query to a queue per strategy and splits
// each pre-filter query into scan items. One warp takes one work unit at a time
// from a single device counter, in the order: long hybrid walks, post-filter walks,
// short hybrid walks (route.cu tells them apart), scan items. The long graph searches
// start first and the short scan items fill the tail, so the batch has one tail instead of
// one per strategy. A pre-filter query split into several items is merged by the warp that
// completes its last item (release/acquire through a per-query counter).
//
// Graph search (Algorithm 2's scheme; Algorithm 1 for B over bitmap-marked
// slots; Algorithm 7 for C over the first ceil(m/S') slots of each intersected
// chunk). One warp per query. Per-warp shared memory holds
//   E    the candidate buffer: every visited object that can still matter, sorted
//        by key (distance, id), the lowest key bit an "expanded" flag; popping the
//        nearest candidate is taking the first unexpanded entry;
//   ann  the result heap of Algorithms 1/7 as a sorted array of capacity ef;
//   vis  a direct-mapped visited filter (ids; a slot may be overwritten).
// Equivalence with the heap formulation: once ann holds ef entries its worst key
// w only decreases, and an object with key > w can neither enter cand or ann nor
// be expanded (the loop stops first), so E keeps exactly the visited objects with
// key <= w (all visited objects while ann is not full). An object the filter
// forgot is re-checked against E and ann by key, which is exact because its
// distance is recomputed bit-identically (a fixed reduction tree). The neighbours of
// one expansion are processed in batches against the ann of the start of the batch;
// objects the sequential loop would have rejected after an earlier insertion of the
// same batch end above the final w and are dropped from E, so the outcome is the
// same however the neighbours are split into batches, as long as E has room. The
// visible differences are the capacity of E (UNIFY_Q_TRUNCATED) and the expansion
// bound (UNIFY_Q_LIMIT). So that the capacity acts on the same entries at any batch
// size, a batch that might overflow E goes in by the blocks of 32 slots it came from.
//
// What bounds a graph query is the chain of dependent steps of one expansion, run by
// one warp (a few thousand cycles, issuing about every fifth), and in large batches the
// issue slots of the 16 to 20 warps per SM; DRAM stays far from busy. So the steps are
// laid out for a short chain and few instructions:
//   - the adjacency of the next candidate is copied into shared memory
//     (cp.async) while the current one's distances are computed; when an insertion
//     changes the order, it is fetched anew;
//   - all slots of an expansion pass the visited filter first, then the survivors of
//     several 32-slot blocks share distance groups and one insertion;
//   - a group's row loads are all in flight together (group_dist);
//   - the insertion needs no sort: ranks by counting, and every position of a sorted
//     array finds its source by a ballot (sorted_insert);
//   - few registers are spilled: with shared memory full, L1 is small and swept by the row
//     gathers, and a reload of a spilled register comes from L2. State that an expansion
//     seldom needs lives in shared memory, scan and re-rank run out of line, hybrid and post
//     walks share one body, and addresses are recomputed (WarpMem). The builds for rows of up
//     to 128 elements still report 16 to 72 bytes of spill stores with 128 and 96 registers and
//     96 to 142 with 80; how many of them lie inside the loop was not established.
// Measured on GB300 against lanes-per-row of 32, a bitonic sort, a merge by binary
// searches and 32 to 136 bytes of spills per thread: one query, 120 expansions 399 -> 276
// us; 10,000 auto-routed queries over 1M x 128 (graph walks and the tensor-core scan
// before them) float32 1,680 -> 1,230 us, bfloat16 1,721 -> 1,143 us; 1,622 walks for k =
// 100 over 200K x 96 3,308 -> 2,203 us; FP8 log-uniform batch of 5,001 1,705 -> 1,071 us.
//
// Scan (Strategy A): rows [pa, pb) of the attribute-ordered vectors; a warp
// computes 32 rows per step, eight lanes per row (4 shuffles per 16 rows instead of 16,
// all loads of a batch in flight); keys beating the current k-th are inserted into a
// sorted top-k. Bound by the latency of a step's loads and by L2 and HBM: 301 queries over
// 4,150 rows of 3,840 B each gather 8 TB/s (609 us), 4,000 queries over 1M x 128 float32 8.4
// TB/s (1,347 us).
//
// Bounds (checked by reading, against the buffers the launch receives):
// E[< cand_cap], ann[< ann_cap], vis[< 2^vis_log2], clist[< 32], SK[< 32], nadj and
// table[< kSlotTable]; S1 keeps its 64 keys in nadj(1) and the table's first 32 ints, its
// list of 32 ids after them; ids come from validated adjacency
// (0 <= id < n < 2^30), and where a row repeats one only its first place is inserted
// (sorted_insert keeps positions apart by distinct keys); upper-layer rows exist for every
// object reached on that layer (validated levels); scan rows lie in [pa, pb) and loads
// clamp to the last valid row.
#pragma once

#include "common.cuh"
#include "internal.h"
#include "warp_ops.cuh"

namespace unify {

struct BatchArgs {
  const float* vec;                // float32 rows by id (re-rank, and traversal for FP32)
  const unsigned char* vt;         // traversal rows by id in the storage format
  const unsigned char* vts;        // the same rows in attribute order (scan)
  const float* scale;              // FP8 per-vector scales by id (else null)
  const float* scale_sorted;       // FP8 scales in attribute order
  int row_bytes;                   // bytes per stored row
  int rerank;                      // candidates re-ranked in FP32 (0: FP32 storage, none)
  const int32_t* sorted_ids;
  int dp4, d;
  int S, M, max_level, entry_global;
  const int32_t* adj0;
  const int32_t* gadj0;            // bitmap-marked neighbours of layer 0, GW per row, in slot order
  const int32_t* adjU;
  const int32_t* gadjU;
  int GW;
  const int32_t* upper_base;
  const int32_t* pos;
  const int32_t* seg_start;
  const float* q;
  const int32_t* pa;
  const int32_t* pb;
  const uint32_t* mask;
  const int32_t* queues;
  int64_t cap_nq;
  const int32_t* nblk;
  const int32_t* qbase;
  int32_t* done;
  const int2* items;
  uint64_t* part;
  int32_t* counters;
  int k, ef_h, ef_p, m, cand_cap, ann_cap, vis_log2, max_exp;
  Conj cj;  // second-attribute predicate (attr2 == nullptr: none)
  int repeats;  // a row of the file may name a neighbour more than once
  int s1;  // hybrid selection S1 (the m neighbours nearest to the expanded object) instead of S2
  int warp_bytes, off_q, off_E, off_ann;
  int scan_only;  // every query is a pre-filter query: no walks' buffers, a large L1
  int skip_scan;  // the pre-filter queries were searched by the tensor-core scan
  Outputs o;
};

constexpr int kSlotTable = 96;  // slots of an expansion handled at a time (a multiple of 32, at least 64)

extern __shared__ __align__(16) unsigned char smem_raw[];

// The kernel's arguments are copied to the front of shared memory, for the parts that run
// out of line (a function that is not inlined cannot name the kernel's parameters).
__device__ __forceinline__ const BatchArgs& shared_args() { return *reinterpret_cast<const BatchArgs*>(smem_raw); }
constexpr int kArgsBytes = (sizeof(BatchArgs) + 15) & ~15;

// A warp's shared memory. Its place is held as an offset that the walk's loop declares
// unknown in every iteration (renew), so that the compiler keeps that one register across
// an expansion instead of a dozen derived addresses: what it spilled otherwise went
// through an L1 that the row gathers keep sweeping. State that an expansion seldom reads
// lives here as well.
struct WarpMem {
  saddr off;
  const BatchArgs& a;
  static constexpr int kNadj = 256, kTable = kNadj + 2 * kSlotTable * 4, kSegs = kTable + kSlotTable * 4,
                       kRange = kSegs + 32, kCold = kRange + 32, kFixed = kCold + 64;
  __device__ void renew() { asm volatile("" : "+r"(off)); }
  __device__ saddr SK() const { return off; }  // 32 keys
  // neighbour ids of an expansion: two buffers of kSlotTable ints, one being filled ahead
  __device__ saddr nadj(int i) const { return off + kNadj + i * (kSlotTable * 4); }
  __device__ saddr clist() const { return nadj(0); }  // 32 ids, outside a walk
  // hybrid S2: slot per selection index, bit 31 set where its segment is only partly in
  // the range
  __device__ saddr table() const { return off + kTable; }
  __device__ saddr vis() const { return off + kFixed; }
  __device__ saddr q() const { return off + a.off_q; }         // dp4 chunks
  __device__ saddr xo() const { return q() + 16 * a.dp4; }     // S1: the expanded object's row (else not there)
  __device__ saddr E() const { return off + a.off_E; }
  __device__ saddr ann() const { return off + a.off_ann; }
  // the same memory by pointer, for what an expansion seldom needs
  __device__ unsigned char* at(saddr x) const { return smem_raw + (x - sa(smem_raw)); }
  __device__ uint8_t* segs() const { return at(off + kSegs); }  // intersected segments
  // in-range positions [x, y), and the range on the second attribute
  __device__ int2* range() const { return reinterpret_cast<int2*>(at(off + kRange)); }
  __device__ longlong2* range2() const { return reinterpret_cast<longlong2*>(at(off + kRange + 16)); }
  __device__ struct Cold* cold() const { return reinterpret_cast<struct Cold*>(at(off + kCold)); }
};

// Fills the offsets and the size of a warp's shared memory.
inline void layout(BatchArgs& a) {
  a.off_q = WarpMem::kFixed + (4 << a.vis_log2);
  a.off_E = a.off_q + a.dp4 * 16 * (a.s1 ? 2 : 1);
  a.off_ann = a.off_E + a.cand_cap * 8;
  a.warp_bytes = (a.off_ann + a.ann_cap * 8 + 15) & ~15;
}

// Keys of the graph search: (distance bits) << 32 | id << 1 | expanded. They order as
// (distance, id); the flag only tells copies of one object apart.
__device__ __forceinline__ uint64_t graph_key(float d, int id) {
  return ((uint64_t)__float_as_uint(d) << 32) | ((uint32_t)id << 1);
}
__device__ __forceinline__ int graph_id(uint64_t k) { return (int)((uint32_t)k >> 1); }

__device__ __forceinline__ uint32_t vis_hash(int id, int log2) {
  return ((uint32_t)id * 0x9E3779B1u) >> (32 - log2);
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Microseconds since the first work unit of this launch started (instrumented runs).
__device__ __forceinline__ int us_since_start(int32_t* counters) {
  unsigned long long* t0 = reinterpret_cast<unsigned long long*>(counters + CNT_T0);
  const unsigned long long now = global_ns();
  unsigned long long base = atomicCAS(t0, 0ull, now);
  if (base == 0ull) base = now;
  return (int)((now - base) / 1000ull);
}

// Copies one int into shared memory without a register in between (cp.async).
__device__ __forceinline__ void async_copy4(saddr dst, const int* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void async_copy16(saddr dst, const int* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The second-attribute predicate for object id (true without a second attribute).
__device__ __forceinline__ bool conj_ok(const BatchArgs& a, int id, int64_t l2, int64_t h2) {
  if (!a.cj.attr2) return true;
  const int64_t v = __ldg(a.cj.attr2 + id);
  return v >= l2 && v <= h2;
}

// Whether object id at attribute-order position p satisfies the query's ranges.
__device__ __forceinline__ bool in_range(const BatchArgs& a, const WarpMem& w, int id, int p) {
  const int2 r = *w.range();
  if (p < r.x || p >= r.y) return false;
  if (!a.cj.attr2) return true;
  const longlong2 r2 = *w.range2();
  return conj_ok(a, id, r2.x, r2.y);
}

// A query's state outside the walk's loop, in shared memory.
struct Cold {
  int qi, t_start, per, slots, l, efl0;
  int n_dist, n_exp;
  uint32_t status, mask;
};

// Tables the slots (segment * M + s) of kSlotTable selection indexes from sb on of a hybrid
// S2 query: the first `per` slots of every intersected segment.
__device__ __forceinline__ void table_slots(const BatchArgs& a, const WarpMem& w, int sb) {
  const int per = w.cold()->per, slots = w.cold()->slots;
  const int2 r = *w.range();
  for (int ci = sb + lane_id(); ci < slots && ci < sb + kSlotTable; ci += 32) {
    const int kseg = ci / per;
    const int seg = w.segs()[kseg];
    const bool inside = __ldg(a.seg_start + seg) >= r.x && __ldg(a.seg_start + seg + 1) <= r.y;
    sts32(w.table() + 4 * (ci - sb), (seg * a.M + (ci - kseg * per)) | (inside ? 0u : 0x80000000u));
  }
  __syncwarp();
}

// Starts copying the neighbour ids of n slots of object o on layer l into dst: the tabled
// slots (hybrid), or the bitmap-marked ones (post).
__device__ __forceinline__ void fetch_adjacency(const BatchArgs& a, const WarpMem& w, bool hy, saddr dst, int o, int l,
                                                int n) {
  const int lane = lane_id();
  const int64_t row = l == 0 ? (int64_t)o : (int64_t)__ldg(a.upper_base + o) + (l - 1);
  if (hy) {
    const int32_t* adj = (l == 0 ? a.adj0 : a.adjU) + row * (a.S * a.M);
#pragma unroll 1
    for (int ci = lane; ci < n; ci += 32) async_copy4(dst + 4 * ci, adj + (lds32(w.table() + 4 * ci) & 0x7fffffff));
  } else {
    const int32_t* adj = (l == 0 ? a.gadj0 : a.gadjU) + row * a.GW;
    if (4 * lane < n) async_copy16(dst + 16 * lane, adj + 4 * lane);  // n = GW <= 64, a multiple of 4
  }
}

// Selection S1: every neighbour of o in the intersected chunks, by (distance to o, id),
// the first m, into nadj(0) (these owner distances are not query distance evaluations and
// are not counted). Returns how many.
template <class T, int CH, int G>
__device__ __forceinline__ int select_s1(const BatchArgs& a, const WarpMem& w, int nseg, int o, int l) {
  const int lane = lane_id();
  const int64_t row = l == 0 ? (int64_t)o : (int64_t)__ldg(a.upper_base + o) + (l - 1);
  const int32_t* adj = (l == 0 ? a.adj0 : a.adjU) + row * (a.S * a.M);
  const unsigned char* orow = a.vt + (int64_t)o * a.row_bytes;
  const float sc = a.scale ? __ldg(a.scale + o) : 1.f;
  __syncwarp();
  float4* const xo = reinterpret_cast<float4*>(w.at(w.xo()));
  for (int c = lane; c < a.dp4; c += 32) xo[c] = value4<T>(T::load(orow, c, sc), sc);
  __syncwarp();
  const saddr selk = w.nadj(1), scratch = w.table() + 128;  // 64 keys; 32 ids
  const int tot = nseg * a.M;
  int ns = 0;
  auto neighbour = [&](int ci) {
    if (ci >= tot) return -1;
    const int kseg = ci / a.M;
    return (int)__ldg(adj + w.segs()[kseg] * a.M + (ci - kseg * a.M));
  };
  int next = neighbour(lane);
#pragma unroll 1
  for (int b0 = 0; b0 < tot; b0 += 32) {
    const int cid = next;
    next = neighbour(b0 + 32 + lane);
    const float dv = batch_dist<T, CH, G>(w.xo(), cid, a.vt, a.row_bytes, a.scale, a.dp4, scratch);
    ns = topk_offer(selk, ns, a.m < 64 ? a.m : 64, cid >= 0 ? make_key(dv, cid) : kKeyMax, w.SK(), a.repeats != 0);
  }
  for (int t = lane; t < ns; t += 32) sts32(w.nadj(0) + 4 * t, key_id(lds64(selk + 8 * t)));
  __syncwarp();
  return ns;
}

// Inserts the candidates of the lanes in kb (keys below the threshold of the batch's
// start) into E and, for hybrid, the in-range ones into ann.
__device__ __forceinline__ void insert_batch(const BatchArgs& a, const WarpMem& w, bool hy, int efl, uint64_t key, bool inr,
                                             unsigned kb, int& nE, int& nA, int& cursor, bool& truncated) {
  const int lane = lane_id();
  const saddr E = hy ? w.E() : w.ann();
  const int capE = hy ? a.cand_cap : efl;
  bool keep = (kb >> lane) & 1u;
  const int rk = warp_rank(E, nE, key, kb);
  // a visited object the filter forgot is still in E (or, after an overflow of E,
  // possibly only in ann): drop it
  if (keep) keep = rk >= nE || (lds64(E + 8 * rk) ^ key) > 1ull;
  if (hy && truncated && keep) keep = !contains_u64(w.ann(), nA, key);
  kb = __ballot_sync(kFull, keep);
  if (kb == 0) return;
  int in_less = 0;
  const int less = rank_among(key, kb, w.SK(), hy && inr ? 1u : 0u, &in_less);
  if (hy && nE + __popc(kb) > capE) truncated = true;
  nE = sorted_insert(E, nE, capE, key, rk, less, kb);
  const int r0 = (int)__reduce_min_sync(kFull, keep ? (unsigned)rk : 0x7fffffffu);
  if (r0 < cursor) cursor = r0;
  if (!hy) {
    nA = nE;  // cand and ann share the buffer; dropping beyond ef is ann's pop
    if (cursor > nE) cursor = nE;
    return;
  }
  const unsigned ab = __ballot_sync(kFull, keep && inr);
  if (ab == 0) return;  // w did not change, and every key kept was below it
  const int ra = warp_rank(w.ann(), nA, key, ab);
  nA = sorted_insert(w.ann(), nA, efl, key, ra, in_less, ab);
  if (nA >= efl) {
    nE = warp_count_le(E, nE, lds64(w.ann() + 8 * (efl - 1)) | 1ull);
    if (cursor > nE) cursor = nE;
  }
}

// One layer (cold()->l; base: layer 0) of Algorithm 1 (post) or Algorithm 7 (hybrid, hy;
// S1: with that selection) over cold()->slots slots per expansion. Returns |ann|; the ann
// array is w.ann for hybrid. For post every candidate push is also an ann push, so cand is
// a subset of ann and one sorted buffer of capacity efl holds both: the result is then in
// w.ann as well (the buffer is w.ann itself, its flags set).
template <class T, int CH, int G, bool S1>
__device__ __forceinline__ int search_layer(const BatchArgs& a, WarpMem w, bool hy, bool base, int efl, uint64_t ep_key,
                                            bool ep_in) {
  const int lane = lane_id();
  int4* const vis4 = reinterpret_cast<int4*>(w.at(w.vis()));
  for (int t = lane; t < (1 << a.vis_log2) / 4; t += 32) vis4[t] = make_int4(-1, -1, -1, -1);
  __syncwarp();
  if (lane == 0) {
    sts64(hy ? w.E() : w.ann(), ep_key);
    if (hy && ep_in) sts64(w.ann(), ep_key);
    sts32(w.vis() + 4 * vis_hash(graph_id(ep_key), a.vis_log2), graph_id(ep_key));
  }
  __syncwarp();
  const int slots = w.cold()->slots;
  int nE = 1, nA = hy ? (ep_in ? 1 : 0) : 1, cursor = 0, exp_l = 0, n_dist = 0;
  int fetched = -1;  // object whose neighbour ids are in nadj(buf), or on their way
  int buf = 0;
  bool truncated = false;
#pragma unroll 1
  for (;;) {
    w.renew();
    // the nearest unexpanded candidate and, among the next 31 entries, the one after it
    int o = -1, o2 = -1;
#pragma unroll 1
    while (cursor < nE) {
      const saddr e = (hy ? w.E() : w.ann()) + 8 * (cursor + lane);  // the key's low word
      const uint32_t lo = cursor + lane < nE ? lds32(e) : 1u;
      const unsigned bal = __ballot_sync(kFull, (lo & 1u) == 0u);
      if (bal) {
        const int at = __ffs(bal) - 1;
        const unsigned rest = bal & (bal - 1);
        o = (int)(__shfl_sync(kFull, lo, at) >> 1);
        o2 = (int)(__shfl_sync(kFull, lo, rest ? __ffs(rest) - 1 : at) >> 1);
        if (!rest) o2 = -1;
        if (exp_l < a.max_exp && lane == at) sts32(e, lo | 1u);
        cursor += at;
        break;
      }
      cursor += 32;
    }
    if (o < 0) break;
    if (exp_l >= a.max_exp) {
      if (lane == 0) w.cold()->status |= UNIFY_Q_LIMIT;
      break;
    }
    ++exp_l;
    int total = slots;
    const bool s1 = S1 && hy;
    if (s1) {
      total = select_s1<T, CH, G>(a, w, slots, o, w.cold()->l);
      // the next candidate's adjacency into L2
      if (base && o2 >= 0)
        for (int t = 32 * lane; t < a.S * a.M; t += 32 * 32)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(a.adj0 + (int64_t)o2 * (a.S * a.M) + t));
    }
#pragma unroll 1
    for (int sb = 0; sb < total; sb += kSlotTable) {
      const int n = total - sb < kSlotTable ? total - sb : kSlotTable;
      if (!s1) {
        if (fetched != o || sb > 0) {
          async_wait_all();  // of a fetch for another object
          __syncwarp();
          if (hy && slots > kSlotTable) table_slots(a, w, sb);
          fetch_adjacency(a, w, hy, w.nadj(buf), o, base ? 0 : w.cold()->l, n);
        }
        async_wait_all();
        __syncwarp();
      }
      // blocks of 32 slots through the visited filter; the survivors move to the front of
      // the list. Bit 31: layer 0 of a hybrid query tests the range by position where the
      // segment is only partly inside. Bit 30 changes from block to block.
      const saddr list = w.nadj(buf);
      int nc = 0;
      int block = 0;
#pragma unroll 1
      for (int b = 0; b < n; b += 32) {
        const int ci = b + lane;
        int c = ci < n ? (int)lds32(list + 4 * ci) : -1;
        uint32_t need = 0;
        if (hy && base) need = s1 ? 0x80000000u : (ci < n ? lds32(w.table() + 4 * ci) : 0u) & 0x80000000u;
        const saddr v = w.vis() + 4 * vis_hash(c, a.vis_log2);
        const int seen = (int)lds32(v);  // of some slot where c is -1: no object has id -1
        const bool fresh = c >= 0 && seen != c;
        if (fresh) sts32(v, c);
        const unsigned m = __ballot_sync(kFull, fresh);
        if (fresh) sts32(list + 4 * (nc + __popc(m & lanemask_lt())), (uint32_t)(c | block) | need);
        nc += __popc(m);
        if (m) block ^= 1 << 30;
        __syncwarp();
      }
      // the next candidate's neighbour ids, on their way behind this one's rows (on layer 0;
      // above it the next object is nearly always one found just now)
      if (!s1 && slots <= kSlotTable) {
        buf ^= 1;
        fetched = base ? o2 : -1;
        if (fetched >= 0) fetch_adjacency(a, w, hy, w.nadj(buf), o2, 0, slots);
      }
      n_dist += nc;
#pragma unroll 1
      for (int c0 = 0; c0 < nc;) {
        int m = nc - c0;
        if (m > 32) {
          // as many whole blocks as fit
          const uint32_t d = (lds32(list + 4 * (c0 + lane)) ^ lds32(list + 4 * (c0 + lane + 1))) & (1u << 30);
          m = 32 - __clz(__ballot_sync(kFull, d != 0));
        }
        const int c = lane < m ? (int)lds32(list + 4 * (c0 + lane)) : 0;
        const int id = c & kIdMask;
        // where a row of the file may name a neighbour twice, its first place counts
        // (sorted_insert wants distinct keys)
        unsigned cand = m < 32 ? (1u << m) - 1u : kFull;
        if (a.repeats)
          cand &= __ballot_sync(kFull, (__match_any_sync(kFull, lane < m ? id : ~lane) & lanemask_lt()) == 0);
        const int pv = hy && c < 0 ? __ldg(a.pos + id) : 0;
        const bool two = hy && base && a.cj.attr2 != nullptr;
        const int64_t v2 = two && lane < m ? __ldg(a.cj.attr2 + id) : 0;
        const float dist = group_dist<T, CH, G>(w.q(), list + 4 * c0, m, a.vt, a.row_bytes, a.scale, a.dp4);
        c0 += m;
        bool inr = lane < m;
        if (hy && c < 0) {
          const int2 r = *w.range();
          inr = pv >= r.x && pv < r.y;
        }
        if (two) {
          const longlong2 r = *w.range2();
          inr = inr && v2 >= r.x && v2 <= r.y;
        }
        const uint64_t key = graph_key(dist, id);
        const saddr last = w.ann() + 8 * (efl - 1);  // for post, E is w.ann
        unsigned kb = cand & __ballot_sync(kFull, key < (nA >= efl ? lds64(last) & ~1ull : kKeyMax));
        if (kb == 0) continue;
        // where E might overflow: block by block, each against the ann of its own start
        unsigned ends = 0;
        if (hy && nE + __popc(kb) > a.cand_cap) {
          const int nx = __shfl_down_sync(kFull, c, 1);
          ends = __ballot_sync(kFull, lane == m - 1 || (lane < m && ((c ^ nx) & (1 << 30)) != 0));
          kb = 0;
        }
        int b0 = 0;
        do {
          if (hy && ends) {
            const int b1 = __ffs(ends);
            ends &= ends - 1;
            kb = cand & __ballot_sync(kFull, lane >= b0 && lane < b1 && key < (nA >= efl ? lds64(last) : kKeyMax));
            b0 = b1;
          }
          if (kb) insert_batch(a, w, hy, efl, key, inr, kb, nE, nA, cursor, truncated);
        } while (hy && ends);
      }
    }
  }
  if (lane == 0) {
    w.cold()->n_exp += exp_l;
    w.cold()->n_dist += n_dist;
    if (truncated) w.cold()->status |= UNIFY_Q_TRUNCATED;
  }
  async_wait_all();  // a copy that was not needed has landed before nadj is used again
  __syncwarp();
  return nA;
}

// FP32 re-rank: exact float32 distances (direct difference against the float32
// rows) of the nc candidates of E or ann (plain keys, or graph keys), the k best written
// to row qi (the other buffer holds them meanwhile). Returns the number written.
// Out of line, as scan_item: both run once per query or item, and inlined into the work
// loop they cost the walk's loop its registers.
template <int CH, int G, bool kGraphKeys>
__device__ __noinline__ int rerank_write(uint32_t off, bool from_E, int nc, int64_t qi) {
  const BatchArgs& a = shared_args();
  const WarpMem w{off, a};
  const saddr keys = from_E ? w.E() : w.ann(), tmp = from_E ? w.ann() : w.E();
  const int lane = lane_id();
  int nt = 0;
#pragma unroll 1
  for (int base = 0; base < nc; base += 32) {
    const int t = base + lane;
    const int cid = t < nc ? (kGraphKeys ? graph_id(lds64(keys + 8 * t)) : key_id(lds64(keys + 8 * t))) : -1;
    const float dist = batch_dist<StoreF32, CH, G>(w.q(), cid, reinterpret_cast<const unsigned char*>(a.vec), a.dp4 * 16,
                                                   nullptr, a.dp4, w.clist());
    nt = topk_offer(tmp, nt, a.k, cid >= 0 ? make_key(dist, cid) : kKeyMax, w.SK());
  }
  write_row(reinterpret_cast<const uint64_t*>(w.at(tmp)), nt, a.k, qi, a.o);
  return nt;
}

template <class T, int CH, int G, int GF, bool S1>
__device__ __forceinline__ void graph_query(const BatchArgs& a, const WarpMem& w, int qi, bool hy) {
  const int lane = lane_id();
  Cold* const cold = w.cold();
  int cnt = 0;
  {
    const uint32_t mask = a.mask[qi];
    const int2 r = make_int2(a.pa[qi], a.pb[qi]);
    const int Sp = __popc(mask);
    int per = Sp > 0 ? (a.m + Sp - 1) / Sp : 0;
    if (per > a.M) per = a.M;
    __syncwarp();
    if (lane == 0) {
      cold->qi = qi;
      cold->t_start = a.o.counters ? us_since_start(a.counters) : 0;
      cold->per = per;
      cold->slots = !hy ? a.GW : S1 ? Sp : Sp * per;  // S1: select_s1 takes the number of segments
      cold->efl0 = hy ? (a.ef_h > a.k ? a.ef_h : a.k) : (a.ef_p > a.k ? a.ef_p : a.k);
      cold->n_dist = 0;
      cold->n_exp = 0;
      cold->status = 0;
      cold->mask = mask;
      *w.range() = r;
      if (a.cj.attr2) *w.range2() = make_longlong2(a.cj.lo2[qi], a.cj.hi2[qi]);
    }
    // the intersected segments and, for S2, the slots it selects from every expanded
    // object: the same for the whole query
    if ((mask >> lane) & 1u) w.segs()[__popc(mask & lanemask_lt())] = (uint8_t)lane;
    __syncwarp();
  }
  if (hy ? cold->mask != 0 : w.range()->y > w.range()->x) {  // nothing can be in range otherwise
    load_query(reinterpret_cast<float4*>(w.at(w.q())), a.q + (int64_t)qi * a.d, a.d, a.dp4);
    if (hy && !S1 && cold->slots <= kSlotTable) table_slots(a, w, 0);
    // entry point: the first object on the top layer
    const float d0 = batch_dist<T, CH, G>(w.q(), lane == 0 ? a.entry_global : -1, a.vt, a.row_bytes, a.scale, a.dp4,
                                          w.clist());
    uint64_t ep_key = graph_key(__shfl_sync(kFull, d0, 0), a.entry_global);
    if (lane == 0) cold->n_dist = 1;
    int nA = 0;
#pragma unroll 1
    for (int l = a.max_level; l >= 0; --l) {
      const int ep = graph_id(ep_key);
      bool ep_in = true;
      if (hy) {
        const int p = __ldg(a.pos + ep);
        if (l == 0) {
          ep_in = in_range(a, w, ep, p);
        } else {
          // the last segment that starts at or before p (segment 0 otherwise)
          const unsigned at = __ballot_sync(kFull, lane > 0 && lane < a.S && __ldg(a.seg_start + lane) <= p);
          ep_in = (cold->mask >> (at ? 31 - __clz(at) : 0)) & 1u;
        }
      }
      if (lane == 0) cold->l = l;
      nA = search_layer<T, CH, G, S1>(a, w, hy, l == 0, l > 0 ? 1 : cold->efl0, ep_key, ep_in);
      if (l > 0 && nA > 0) ep_key = lds64(w.ann()) & ~1ull;
      l = cold->l;
      __syncwarp();  // lane 0 stores the next layer's number only after every lane has read this one's
    }
    qi = cold->qi;
    if (a.rerank > 0) {
      // reduced-precision storage: re-rank the first rerank_mult * k candidates in FP32
      int nc = nA;
      if (!hy) {
        // Strategy B: the range filter first, compacted into E (free after the search)
        nc = 0;
        for (int base = 0; base < nA && nc < a.rerank; base += 32) {
          const int t = base + lane;
          bool inr = false;
          uint64_t key = kKeyMax;
          if (t < nA) {
            key = lds64(w.ann() + 8 * t);
            inr = in_range(a, w, graph_id(key), __ldg(a.pos + graph_id(key)));
          }
          const unsigned bal = __ballot_sync(kFull, inr);
          const int dst = nc + __popc(bal & lanemask_lt());
          if (inr && dst < a.rerank) sts64(w.E() + 8 * dst, key);
          nc += __popc(bal);
        }
        __syncwarp();
      }
      if (nc > a.rerank) nc = a.rerank;
      cnt = rerank_write<CH, GF, true>(w.off, !hy, nc, qi);
    } else {
      // the first k of ann; Strategy B filters ann by the range first
      for (int base = 0; base < nA && cnt < a.k; base += 32) {
        const int t = base + lane;
        bool inr = t < nA;
        uint64_t key = kKeyMax;
        if (t < nA) {
          key = lds64(w.ann() + 8 * t);
          if (!hy) {
            inr = in_range(a, w, graph_id(key), __ldg(a.pos + graph_id(key)));
          }
        }
        const unsigned bal = __ballot_sync(kFull, inr);
        const int dst = cnt + __popc(bal & lanemask_lt());
        if (inr && dst < a.k) {
          a.o.ids[(int64_t)qi * a.k + dst] = graph_id(key);
          a.o.dist[(int64_t)qi * a.k + dst] = key_dist(key);
        }
        cnt += __popc(bal);
      }
      if (cnt > a.k) cnt = a.k;
      for (int t = cnt + lane; t < a.k; t += 32) {
        a.o.ids[(int64_t)qi * a.k + t] = -1;
        a.o.dist[(int64_t)qi * a.k + t] = __int_as_float(0x7f800000);
      }
    }
  } else {
    write_row(nullptr, 0, a.k, qi, a.o);
  }
  if (lane == 0) {
    a.o.count[qi] = cnt;
    if (a.o.status) a.o.status[qi] = cold->status;
    if (a.o.counters) {
      a.o.counters[4 * (int64_t)qi] = cold->n_dist;
      a.o.counters[4 * (int64_t)qi + 1] = cold->n_exp;
      a.o.counters[4 * (int64_t)qi + 2] = cold->t_start;
      a.o.counters[4 * (int64_t)qi + 3] = us_since_start(a.counters);
    }
  }
  __syncwarp();
}

// The kk smallest keys of nb ascending lists of kk keys each, into ann; returns how many.
// Each lane walks one list from its front and stops at the first key that cannot enter
// any more, the next key of its list already in flight.
static __device__ __noinline__ int merge_lists(saddr off, const uint64_t* lists, int nb, int kk) {
  const WarpMem w{off, shared_args()};
  const saddr topk = w.ann();
  const int lane = lane_id();
  int nt = 0;
  for (int b0 = 0; b0 < nb; b0 += 32) {
    bool has = b0 + lane < nb;
    const unsigned long long* list =
        reinterpret_cast<const unsigned long long*>(lists) + (int64_t)(has ? b0 + lane : 0) * kk;
    uint64_t next = has ? __ldcg(list) : kKeyMax;
    for (int t = 0; t < kk; ++t) {
      const uint64_t key = next;
      next = has && t + 1 < kk ? __ldcg(list + t + 1) : kKeyMax;
      has = has && key < (nt >= kk ? lds64(topk + 8 * (kk - 1)) : kKeyMax);
      if (!__any_sync(kFull, has)) break;
      nt = topk_offer(topk, nt, kk, has ? key : kKeyMax, w.SK());
    }
  }
  return nt;
}

template <class T, int CH, int RB, int GF, bool kL1, bool kEarly>
__device__ __noinline__ void scan_item(uint32_t off, int it) {
  const BatchArgs& a = shared_args();
  const WarpMem w{off, a};
  const int lane = lane_id();
  const saddr topk = w.ann();  // ann_cap >= kk
  const int kk = a.rerank > 0 ? a.rerank : a.k;  // keys kept per list
  const int2 item = a.items[it];
  const int qi = item.x, b = item.y;
  if (a.o.counters && lane == 0) atomicMin(&a.o.counters[4 * (int64_t)qi + 2], us_since_start(a.counters));
  const int pa = a.pa[qi], pb = a.pb[qi], nb = a.nblk[qi];
  const int Y = pb - pa;
  const int rpb = (Y + nb - 1) / (nb > 0 ? nb : 1);
  const int r0 = pa + b * rpb;
  const int r1 = min(pb, r0 + rpb);
  const int64_t l2 = a.cj.attr2 ? a.cj.lo2[qi] : 0, h2 = a.cj.attr2 ? a.cj.hi2[qi] : 0;
  load_query(reinterpret_cast<float4*>(w.at(w.q())), a.q + (int64_t)qi * a.d, a.d, a.dp4);
  // Eight lanes per row (as group_dist): row base + 4 r + g, r < 8, is lanes 8 g .. 8 g + 7's;
  // RB of the eight steps r load together, 32 chunks of each row at a time. The arguments are
  // copied out of shared memory first: every insertion would make them be read again. The
  // loop over a row's chunk blocks stays a loop: unrolled, the row loads of all blocks crowd
  // the registers (1.1 KB of spills at 960 elements, 90 bytes so).
  const int dp4 = a.dp4, row_bytes = a.row_bytes;
  const unsigned char* const rows = a.vts;
  const float* const row_scale = a.scale_sorted;
  const int32_t* const sorted_ids = a.sorted_ids;
  const saddr qs = w.q();
  const int j = lane & 7, g = lane >> 3;
  int nt = 0;
#pragma unroll 1
  for (int base = r0; base < r1; base += 32) {
    // the ids of short rows on their way with them (4,000 queries over 1M x 128 BF16 954 ->
    // 907 us; long rows lose 4 %, the smaller builds up to 3 %)
    const int32_t id0 = kEarly ? __ldg(sorted_ids + min(base + 4 * j + g, r1 - 1)) : 0;
    float part[8];
#pragma unroll
    for (int h = 0; h < 8; h += RB) {
      const unsigned char* src[RB];
      float sc[RB];
      float acc[RB][4];
#pragma unroll
      for (int r = 0; r < RB; ++r) {
        const int row = min(base + 4 * (h + r) + g, r1 - 1);
        src[r] = rows + (int64_t)row * row_bytes;
        sc[r] = T::kScaled ? __ldg(row_scale + row) : 1.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[r][i] = 0.f;
      }
#pragma unroll 1
      for (int c0 = 0; CH == 1 ? c0 < 1 : c0 < dp4; c0 += 32) {
        Held<T> x[RB][4];
#pragma unroll
        for (int r = 0; r < RB; ++r)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = c0 + 8 * i + j;
            x[r][i] = c < dp4 ? T::template load_raw<kL1>(src[r], c) : T::zero_raw();
          }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int c = c0 + 8 * i + j;
          if (c < dp4) {
            const float4 q = lds_f4(qs + 16 * c);
#pragma unroll
            for (int r = 0; r < RB; ++r) acc[r][i] = sum_sq<T>(q, T::decode(x[r][i]), sc[r], acc[r][i]);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < RB; ++r) part[h + r] = (acc[r][0] + acc[r][2]) + (acc[r][1] + acc[r][3]);
    }
    const float dist = oct_transpose_reduce<8>(part);  // lane 8 g + r: row base + 4 r + g
    const int row = base + 4 * j + g;
    uint64_t key = kKeyMax;
    if (row < r1) {
      const int32_t id = kEarly ? id0 : __ldg(sorted_ids + row);
      if (conj_ok(a, id, l2, h2)) key = make_key(dist, id);
    }
    nt = topk_offer(topk, nt, kk, key, w.SK());
  }
  if (nb > 1) {
    // split query: publish the partial list; the warp finishing the last item merges
    uint64_t* dst = a.part + (int64_t)it * kk;
    for (int t = lane; t < kk; t += 32) dst[t] = t < nt ? lds64(topk + 8 * t) : kKeyMax;
    __threadfence();
    __syncwarp();
    int prev = 0;
    if (lane == 0) prev = atomicAdd(&a.done[qi], 1);
    prev = __shfl_sync(kFull, prev, 0);
    if (prev != nb - 1) {
      if (a.o.counters && lane == 0) atomicMax(&a.o.counters[4 * (int64_t)qi + 3], us_since_start(a.counters));
      return;
    }
    __threadfence();
    nt = merge_lists(off, a.part + (int64_t)a.qbase[qi] * kk, nb, kk);
    nt = min(nt, Y);
  }
  int cnt;
  if (a.rerank > 0) {
    cnt = rerank_write<CH, GF, false>(off, false, nt, qi);
  } else {
    cnt = min(nt, a.k);
    write_row(reinterpret_cast<const uint64_t*>(w.at(topk)), cnt, a.k, qi, a.o);
  }
  if (lane == 0) {
    a.o.count[qi] = cnt;
    if (a.o.status) a.o.status[qi] = 0u;
    if (a.o.counters) atomicMax(&a.o.counters[4 * (int64_t)qi + 3], us_since_start(a.counters));
  }
  __syncwarp();
}

// MINB: minimum resident CTAs of 128 threads per SM the register allocation must
// allow (4 -> 128 registers, 5 -> 96, 6 -> 80). A group of distances holds up to 64
// registers of row chunks in flight (32 in the smaller builds), the scan as well.
template <class T, int CH, int MINB, bool S1>
__global__ void __launch_bounds__(128, MINB) batch_kernel(const __grid_constant__ BatchArgs a) {
  // rows per distance group: 64 registers of row chunks in flight, 32 in the smaller builds
  // and for rows of more than 128 elements (there a block of each row at a time). Selection
  // S1 over FP8 rows takes 8: its expansions decode up to 256 neighbours next to the query's
  // (GB300, 3,696 queries over 1M x 128: 1,877 -> 1,625 us; 2,000 hybrid ones 2,327 -> 2,209;
  // 5,000 log-uniform ones over 200K x 96 3,266 -> 3,378).
  constexpr int G = T::kRawRegs == 4 ? (CH == 1 && MINB == 4 ? 16 : 8) : S1 && T::kRawRegs == 1 ? 8 : 16,
                GF = CH == 1 && MINB == 4 ? 16 : 8;
  // rows of a scan step in flight per lane: 64 registers, 32 in the smaller builds
  constexpr int kRows = (MINB == 4 ? 16 : 8) / T::kRawRegs, RB = kRows > 8 ? 8 : kRows;
  // Scans keep the lines of short narrow rows in L1, of which each load takes a part, and
  // beside the walks' buffers, which leave L1 little room for loads that bypass it, also those
  // of float32 rows where no walk shares L1 (decided below). GB300, without / with: 10,000
  // auto-routed queries over 1M x 128 BF16 1,627 / 1,581 us (96 registers 1,674 / 1,603, 80
  // registers 2,317 / 1,858), 4,000 short ranges BF16 1,211 / 1,133, 4,000 over 200K x 96 BF16
  // 321 / 296, float32 331 / 277; against it: 1,003 float32 queries with walks 1,900 / 1,938,
  // 4,000 forced pre-filter ones BF16 907 / 932 (a second copy of the scan for these cost the
  // BF16 walks 1.5 %).
  constexpr bool kL1 = CH == 1 && T::kRawRegs < 4, kEarly = CH == 1 && MINB == 4;
  for (int t = threadIdx.x; t < (int)(sizeof(BatchArgs) / 4); t += blockDim.x)
    reinterpret_cast<uint32_t*>(smem_raw)[t] = reinterpret_cast<const uint32_t*>(&a)[t];
  __syncthreads();
  const int lane = lane_id();
  const WarpMem w{sa(smem_raw) + kArgsBytes + (threadIdx.x >> 5) * (uint32_t)a.warp_bytes, a};
#pragma unroll 1
  for (;;) {
    int idx = 0;
    if (lane == 0) idx = atomicAdd(&a.counters[CNT_TAKE], 1);
    idx = __shfl_sync(kFull, idx, 0);
    // queue lengths: read again for every unit (in L1), not held across it
    const int nL = __ldg(a.counters + CNT_QC), nLB = nL + __ldg(a.counters + CNT_QB);
    const int nG = nLB + __ldg(a.counters + CNT_QS);
    if (idx < nG) {
      // long hybrid walks, post-filter walks, short hybrid walks (from the queue's end)
      const bool hy = idx < nL || idx >= nLB;
      const int64_t at = idx < nL ? a.cap_nq + idx : idx < nLB ? 2 * a.cap_nq + (idx - nL) : 2 * a.cap_nq - 1 - (idx - nLB);
      graph_query<T, CH, G, GF, S1>(a, w, a.queues[at], hy);
    } else if (!a.skip_scan && idx - nG < __ldg(a.counters + CNT_ITEMS)) {
      if (CH == 1 && MINB == 4 && nG == 0 && !a.scan_only) scan_item<T, CH, RB, GF, true, kEarly>(w.off, idx - nG);
      else scan_item<T, CH, RB, GF, kL1, kEarly>(w.off, idx - nG);
    } else {
      break;
    }
  }
}

template <class T, int CH, int MINB, bool S1 = false>
static cudaError_t launch_t(const BatchArgs& a, int wpb, int num_sms, cudaStream_t st) {
  const int threads = 32 * wpb;
  const size_t smem = kArgsBytes + (size_t)wpb * a.warp_bytes;
  cudaError_t e = cudaFuncSetAttribute(batch_kernel<T, CH, MINB, S1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel<T, CH, MINB, S1>, threads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  batch_kernel<T, CH, MINB, S1><<<num_sms * per_sm, threads, smem, st>>>(a);
  return cudaGetLastError();
}

// The build for a row width (CH * 32 chunks of 4 elements hold a row), a register budget
// (rows of up to 128 elements) and the hybrid selection. S1 has the 128-register build alone:
// the smaller ones spill more (GB300, 3,696 queries over 1M x
// 128, 128 / 96 / 80 registers: float32 1,805 / 1,935 / 2,065 us, BF16 1,815 / 2,050 / 2,250).
template <class T>
static cudaError_t launch_dt(const BatchArgs& a, int wpb, int regs, int num_sms, cudaStream_t st) {
  const int ch = (a.dp4 + 31) / 32;
  if (a.s1) {
    if (ch <= 1) return launch_t<T, 1, 4, true>(a, wpb, num_sms, st);
    if (ch <= 2) return launch_t<T, 2, 4, true>(a, wpb, num_sms, st);
    if (ch <= 4) return launch_t<T, 4, 4, true>(a, wpb, num_sms, st);
    return launch_t<T, 8, 4, true>(a, wpb, num_sms, st);
  }
  if (ch <= 1) {
    if (regs == 80) return launch_t<T, 1, 5>(a, wpb, num_sms, st);
    if (regs == 64) return launch_t<T, 1, 6>(a, wpb, num_sms, st);
    return launch_t<T, 1, 4>(a, wpb, num_sms, st);
  }
  if (ch <= 2) return launch_t<T, 2, 4>(a, wpb, num_sms, st);
  if (ch <= 4) return launch_t<T, 4, 4>(a, wpb, num_sms, st);
  return launch_t<T, 8, 4>(a, wpb, num_sms, st);
}

// One translation unit per storage format (they compile in parallel).
cudaError_t launch_batch_f32(const BatchArgs& a, int wpb, int regs, int num_sms, cudaStream_t st);
cudaError_t launch_batch_bf16(const BatchArgs& a, int wpb, int regs, int num_sms, cudaStream_t st);
cudaError_t launch_batch_fp8(const BatchArgs& a, int wpb, int regs, int num_sms, cudaStream_t st);

}  // namespace unify
