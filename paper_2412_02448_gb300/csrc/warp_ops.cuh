// Warp-level helpers shared by the search kernel and the tensor-core scan:
// writing a result row, grouped distance evaluation and top-k insertion.
#pragma once

#include "common.cuh"
#include "internal.h"

namespace unify {

// Writes keys[0, cnt) as result row qi (ids and distances), padded with -1 / +inf.
__device__ __forceinline__ void write_row(const uint64_t* keys, int cnt, int k, int64_t qi, const Outputs& o) {
  const int lane = lane_id();
  for (int t = lane; t < k; t += 32) {
    const bool v = t < cnt;
    const uint64_t key = v ? keys[t] : kKeyMax;
    o.ids[qi * k + t] = v ? (int64_t)key_id(key) : (int64_t)-1;
    o.dist[qi * k + t] = v ? key_dist(key) : __int_as_float(0x7f800000);
  }
}

constexpr int kIdMask = 0x3fffffff;  // an object id (n < 2^30) in an int that carries flags above it

// Distances from the query in qs (shared memory, dp4 float4 chunks) to the rows of
// clist[0, nv) (ids in the low 30 bits, nv <= 32), in storage format T: lane c < nv gets
// the distance of clist[c].
//
// Eight lanes take a row, so one load instruction fetches 128 contiguous bytes (FP32)
// of four rows: lane 8 g + j holds the chunks j, j + 8, j + 16, j + 24 (and, for longer
// rows, those plus 32, 64, ...) of row 4 r + g, r < G / 4. All loads of a group of G rows are
// issued before any is used, so a group costs one memory latency.
//
// The sum of a row is a fixed tree over 32 partial sums, one per chunk index mod 32
// (each accumulated over the chunks in ascending order): pairs 16 apart, then 8, 4, 2
// and 1 apart. The first two levels lie within a lane here; a distance has the same
// bits in whichever slot, group size or kernel it is computed. Against 32 lanes per row
// this takes 4 shuffles per 16 rows instead of 16, 4 row addresses per lane instead of
// 16, and no idle lanes on rows of fewer than 32 chunks.
template <class T, int CH, int R>
__device__ __forceinline__ float oct_dist(saddr qs, saddr clist, int n, const unsigned char* rows, int row_bytes,
                                          const float* scale, int dp4) {
  const int lane = lane_id();
  const int j = lane & 7, g = lane >> 3;
  const unsigned char* row[R];
  float sc[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int c = 4 * r + g;
    const int id = lds32(clist + 4 * (c < n ? c : n - 1)) & kIdMask;
    row[r] = rows + (int64_t)id * row_bytes;
    sc[r] = T::kScaled ? __ldg(scale + id) : 1.f;
  }
  float acc[R][4];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[r][i] = 0.f;
  if constexpr (CH == 1) {
    Held<T> x[R][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = 8 * i + j;
      if (8 * i < dp4) {  // uniform
        const int cc = c < dp4 ? c : dp4 - 1;  // past the row's end: a chunk that is not used
#pragma unroll
        for (int r = 0; r < R; ++r) x[r][i] = T::load_raw(row[r], cc);
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) x[r][i] = T::zero_raw();
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (8 * i < dp4) {
        const int c = 8 * i + j;
        const bool in = c < dp4;
        const float4 q = lds_f4(qs + 16 * (in ? c : dp4 - 1));
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const float s = sum_sq<T>(q, T::decode(x[r][i]), sc[r], acc[r][i]);
          acc[r][i] = in ? s : acc[r][i];
        }
      }
    }
  } else {
    // long rows: blocks of 32 TB chunks, each block's loads (64 registers' worth per lane)
    // without a branch between them, so that they stay in flight together
    constexpr int kFit = 16 / T::kRawRegs / R, TB = kFit > 1 ? 2 : 1;
#pragma unroll 1
    for (int t0 = 0; 32 * t0 < dp4; t0 += TB) {
      Held<T> x[R][4 * TB];
#pragma unroll
      for (int i = 0; i < 4 * TB; ++i) {
        const int c = 32 * t0 + 8 * i + j, cc = c < dp4 ? c : dp4 - 1;
#pragma unroll
        for (int r = 0; r < R; ++r) x[r][i] = T::load_raw(row[r], cc);
      }
#pragma unroll
      for (int i = 0; i < 4 * TB; ++i) {
        const int c = 32 * t0 + 8 * i + j;
        const bool in = c < dp4;
        const float4 q = lds_f4(qs + 16 * (in ? c : dp4 - 1));
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const float s = sum_sq<T>(q, T::decode(x[r][i]), sc[r], acc[r][i & 3]);
          acc[r][i & 3] = in ? s : acc[r][i & 3];
        }
      }
    }
  }
  float part[R];
#pragma unroll
  for (int r = 0; r < R; ++r) part[r] = (acc[r][0] + acc[r][2]) + (acc[r][1] + acc[r][3]);
  const float red = oct_transpose_reduce<R>(part);
  // candidate c = 4 r + g sits in lane 8 g + r * (8 / R)
  return __shfl_sync(kFull, red, ((lane & 3) * 8 + (lane >> 2) * (8 / R)) & 31);
}

// The same for long rows (CH >= 4 blocks of 32 chunks): sixteen lanes take a row, all of it
// in flight at once, 2 R rows per group: lane 16 g + j holds the chunks j, j + 16, ... of row
// 2 r + g. Taking such rows in pieces of 1 KB, eight lanes each, made the float32 re-rank of
// 40 rows of 3,840 B for 5,000 queries 2.3 times slower (115 -> 262 us on GB300).
template <class T, int CH, int R>
__device__ __forceinline__ float hex_dist(saddr qs, saddr clist, int n, const unsigned char* rows, int row_bytes,
                                          const float* scale, int dp4) {
  const int lane = lane_id();
  const int j = lane & 15, g = lane >> 4;
  Held<T> x[R][2 * CH];
  float sc[R], acc[R][2];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int c = 2 * r + g;
    const int id = lds32(clist + 4 * (c < n ? c : n - 1)) & kIdMask;
    const unsigned char* row = rows + (int64_t)id * row_bytes;
    sc[r] = T::kScaled ? __ldg(scale + id) : 1.f;
    acc[r][0] = acc[r][1] = 0.f;
#pragma unroll
    for (int i = 0; i < 2 * CH; ++i) x[r][i] = T::load_raw(row, min(16 * i + j, dp4 - 1));
  }
#pragma unroll
  for (int i = 0; i < 2 * CH; ++i) {
    const bool in = 16 * i + j < dp4;
    const float4 q = lds_f4(qs + 16 * (in ? 16 * i + j : dp4 - 1));
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float s = sum_sq<T>(q, T::decode(x[r][i]), sc[r], acc[r][i & 1]);
      acc[r][i & 1] = in ? s : acc[r][i & 1];
    }
  }
  float v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = acc[r][0] + acc[r][1];
  int off = 8;
#pragma unroll
  for (int cnt = R; cnt > 1; cnt >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < cnt / 2; ++i) {
      const float send = up ? v[i] : v[i + cnt / 2];
      const float keep = up ? v[i + cnt / 2] : v[i];
      v[i] = keep + __shfl_xor_sync(kFull, send, off);
    }
  }
#pragma unroll
  for (; off >= 1; off >>= 1) v[0] += __shfl_xor_sync(kFull, v[0], off);
  // candidate c = 2 r + g sits in lane 16 g + r * (16 / R)
  return __shfl_sync(kFull, v[0], ((lane & 1) * 16 + (lane >> 1) * (16 / R)) & 31);
}

template <class T, int CH, int G>
__device__ __forceinline__ float group_dist(saddr qs, saddr clist, int nv, const unsigned char* rows, int row_bytes,
                                            const float* scale, int dp4) {
  const int lane = lane_id();
  float result = 0.f;
  // what does not fit into the first group, on its way into L2 meanwhile (short rows: of
  // long ones the warps of the device together would ask for more than L2 holds)
  if (CH == 1 && nv > G && lane >= G && lane < nv) {
    const unsigned char* row = rows + (int64_t)(lds32(clist + 4 * lane) & kIdMask) * row_bytes;
#pragma unroll 1
    for (int c = 0; c < row_bytes; c += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + c));
  }
  // long rows: as many as fit in 64 registers per lane, 2 to 8
  constexpr int kFit = 64 / (2 * CH * T::kRawRegs), kStep = CH >= 4 ? 2 * (kFit < 1 ? 1 : kFit > 4 ? 4 : kFit) : G;
#pragma unroll 1
  for (int base = 0; base < nv; base += kStep) {
    const int n = nv - base;
    float v;
    if constexpr (CH >= 4) {
      v = hex_dist<T, CH, kStep / 2>(qs, clist + 4 * base, n, rows, row_bytes, scale, dp4);
    } else {
      // half a group where that is enough: half the instructions
      if (G >= 16 && n <= G / 2) v = oct_dist<T, CH, (G >= 16 ? G / 8 : 2)>(qs, clist + 4 * base, n, rows, row_bytes, scale, dp4);
      else v = oct_dist<T, CH, G / 4>(qs, clist + 4 * base, n, rows, row_bytes, scale, dp4);
    }
    v = base ? __shfl_sync(kFull, v, lane - base) : v;
    if (lane >= base && lane < base + kStep) result = v;
  }
  return result;
}

// The same for candidates held by the lanes (cid >= 0): each such lane gets its own
// candidate's distance. clist is 32 ints of per-warp shared scratch.
template <class T, int CH, int G>
__device__ __forceinline__ float batch_dist(saddr qs, int cid, const unsigned char* rows, int row_bytes,
                                            const float* scale, int dp4, saddr clist) {
  const unsigned vm = __ballot_sync(kFull, cid >= 0);
  const int my = __popc(vm & lanemask_lt());
  __syncwarp();
  if (cid >= 0) sts32(clist + 4 * my, cid);
  __syncwarp();
  const float d = group_dist<T, CH, G>(qs, clist, __popc(vm), rows, row_bytes, scale, dp4);
  return __shfl_sync(kFull, d, my & 31);
}

// lower_bound of the keys of the lanes in kb (the others: any value), the cheaper way.
__device__ __forceinline__ int warp_rank(saddr a, int n, uint64_t key, unsigned kb) {
  return __popc(kb) <= 4 ? warp_lower_bound(a, n, key, kb) : lower_bound_u64(a, n, key);
}

// Inserts the keys of the lanes in kb (distinct from each other and from arr's entries)
// into the sorted array arr[0, n), n <= cap; entries that fall beyond cap are dropped
// (the largest). rank is lower_bound(arr, n, key) on those lanes, nless the number of
// keys of kb below this lane's. Returns the new size.
//
// Every position of the new array finds its source directly: the new keys' positions
// rank + nless are distinct; a position that is none of them takes the old entry at its
// index less the number of new keys before it, a ballot and a bit mask per 32 positions.
// Positions are moved from the top in blocks of 128 whose loads are all in flight
// together; a block reads no position that an earlier block wrote.
__device__ __forceinline__ int sorted_insert(saddr arr, int n, int cap, uint64_t key, int rank, int nless,
                                             unsigned kb) {
  const int lane = lane_id();
  const bool mine = (kb >> lane) & 1u;
  const int D = mine ? rank + nless : 0x7fffffff;
  const int dmin = (int)__reduce_min_sync(kFull, (unsigned)D);
  const int nk = __popc(kb);
  const int nn = n + nk < cap ? n + nk : cap;
  const int wlo = dmin >> 5;
#pragma unroll 1
  for (int w0 = (nn - 1) >> 5; w0 >= wlo; w0 -= 4) {
    uint64_t v[4];
    bool wr[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int w = w0 - u;
      wr[u] = false;
      if (w >= wlo) {  // uniform
        const unsigned m = __reduce_or_sync(kFull, (D >> 5) == w ? 1u << (D & 31) : 0u);
        const int before = __popc(__ballot_sync(kFull, D < 32 * w)) + __popc(m & lanemask_lt());
        const int p = 32 * w + lane;
        wr[u] = p < nn && !((m >> lane) & 1u) && before > 0;
        if (wr[u]) v[u] = lds64(arr + 8 * (p - before));
      }
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (wr[u]) sts64(arr + 8 * (32 * (w0 - u) + lane), v[u]);
  }
  if (D < cap) sts64(arr + 8 * D, key);
  __syncwarp();
  return nn;
}

// Number of keys below this lane's key among the lanes in kb; SK is 32 keys of per-warp
// shared scratch (16-byte aligned). With tag != 0 on some of these lanes, *tagged gets
// the number of tagged ones among them; the lowest bit of a key does not order keys.
__device__ __forceinline__ int rank_among(uint64_t key, unsigned kb, saddr SK, unsigned tag = 0,
                                          int* tagged = nullptr) {
  const int lane = lane_id();
  const int nk = __popc(kb);
  __syncwarp();
  if ((kb >> lane) & 1u) sts64(SK + 8 * __popc(kb & lanemask_lt()), (key & ~1ull) | tag);
  if (lane == 0 && (nk & 1)) sts64(SK + 8 * nk, kKeyMax);  // pads the last pair (nk < 32 then)
  __syncwarp();
  int c = 0, ct = 0;
  const uint64_t k1 = key & ~1ull;
#pragma unroll 2
  for (int i = 0; i < nk; i += 2) {
    const ulonglong2 y = lds64x2(SK + 8 * i);
    const unsigned b0 = y.x < k1, b1 = y.y < k1;
    c += b0 + b1;
    ct += (b0 & (unsigned)y.x) + (b1 & (unsigned)y.y);
  }
  if (tagged) *tagged = ct;
  return c;
}

// The same over all bits of the keys, without tags.
__device__ __forceinline__ int rank_plain(uint64_t key, unsigned kb, saddr SK) {
  const int lane = lane_id();
  const int nk = __popc(kb);
  __syncwarp();
  if ((kb >> lane) & 1u) sts64(SK + 8 * __popc(kb & lanemask_lt()), key);
  if (lane == 0 && (nk & 1)) sts64(SK + 8 * nk, kKeyMax);
  __syncwarp();
  int c = 0;
#pragma unroll 2
  for (int i = 0; i < nk; i += 2) {
    const ulonglong2 y = lds64x2(SK + 8 * i);
    c += (y.x < key) + (y.y < key);
  }
  return c;
}

// Keeps the k smallest keys: inserts the lanes' keys (plain (distance, id) keys) that
// beat the current k-th into topk[0, nt). SK as in rank_among. The keys of one call are
// distinct, or twins is set: equal ones then take a place each, in the lanes' order.
__device__ __forceinline__ int topk_offer(saddr topk, int nt, int k, uint64_t key, saddr SK, bool twins = false) {
  const uint64_t thr = (nt >= k) ? lds64(topk + 8 * (k - 1)) : kKeyMax;
  const bool pass = key < thr;
  const unsigned bal = __ballot_sync(kFull, pass);
  if (bal == 0) return nt;
  int less = rank_plain(key, bal, SK);
  if (twins) less += __popc(__match_any_sync(kFull, (unsigned long long)key) & bal & lanemask_lt());
  const int rank = warp_rank(topk, nt, key, bal);
  return sorted_insert(topk, nt, k, key, rank, less, bal);
}

}  // namespace unify
