// Warp-level device primitives shared by the search kernels.
//
// Keys: a candidate (distance, id) is packed into one uint64 as
// (bits of the non-negative float32 distance) << 32 | id. For non-negative
// floats the IEEE bit pattern orders like the value, so comparing keys compares
// (distance, id) lexicographically: the tie rule "equal distance -> smaller id".
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace unify {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint64_t kKeyMax = ~0ull;

__device__ __forceinline__ uint64_t make_key(float d, int32_t id) {
  return ((uint64_t)__float_as_uint(d) << 32) | (uint32_t)id;
}
__device__ __forceinline__ float key_dist(uint64_t k) { return __uint_as_float((uint32_t)(k >> 32)); }
__device__ __forceinline__ int32_t key_id(uint64_t k) { return (int32_t)(uint32_t)(k & 0xffffffffu); }

// The lane, in a form that the compiler does not connect between calls: values derived
// from it are recomputed where they are needed (an instruction or two) instead of being
// kept in registers, or spilled, across a whole kernel.
__device__ __forceinline__ int lane_id() {
  int l = threadIdx.x & 31;
  asm volatile("" : "+r"(l));
  return l;
}
__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Shared memory by 32-bit address: plain ld.shared / st.shared whatever the compiler can
// prove about a pointer, and one register per address. Volatile: they keep their order
// among each other and with __syncwarp.
using saddr = uint32_t;
__device__ __forceinline__ saddr sa(const void* p) { return static_cast<saddr>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ uint64_t lds64(saddr a) {
  uint64_t v;
  asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds32(saddr a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ ulonglong2 lds64x2(saddr a) {
  ulonglong2 v;
  asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ float4 lds_f4(saddr a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts64(saddr a, uint64_t v) { asm volatile("st.shared.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory"); }
__device__ __forceinline__ void sts32(saddr a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

// Number of entries of the sorted array of n keys at a that are below x (per lane): a
// binary search of a fixed number of steps (n is the same on every lane).
__device__ __forceinline__ int lower_bound_u64(saddr a, int n, uint64_t x) {
  int lo = 0;
#pragma unroll 1
  for (int step = n > 0 ? 1 << (31 - __clz(n)) : 0; step > 0; step >>= 1) {
    const int i = lo + step;
    if (i <= n && lds64(a + 8 * (i - 1)) < x) lo = i;
  }
  return lo;
}

// The same for the lanes in kb, by the whole warp: 32 equally spaced entries are read
// once; then every key takes a ballot over them and one over the stretch it falls into.
// Lanes outside kb get 0. Used where few lanes hold a key: a per-lane search is a chain
// of dependent loads, this is two.
__device__ __forceinline__ int warp_lower_bound(saddr a, int n, uint64_t x, unsigned kb) {
  const int lane = lane_id();
  const int step = (n + 31) >> 5;
  const int li = (lane + 1) * step - 1;
  const uint64_t sample = (unsigned)li < (unsigned)n ? lds64(a + 8 * li) : kKeyMax;  // li is -1 where n = 0
  int rank = 0;
#pragma unroll 1
  for (unsigned rest = kb; rest; rest &= rest - 1) {
    const int src = __ffs(rest) - 1;
    const uint64_t y = __shfl_sync(kFull, x, src);
    int at = __popc(__ballot_sync(kFull, sample < y)) * step;  // whole stretches below y
    const int end = at + step - 1 < n ? at + step - 1 : n;     // entry at + step - 1 is not below y
#pragma unroll 1
    for (int b = at; b < end; b += 32) at += __popc(__ballot_sync(kFull, b + lane < end && lds64(a + 8 * (b + lane)) < y));
    if (lane == src) rank = at;
  }
  return rank;
}

__device__ __forceinline__ bool contains_u64(saddr a, int n, uint64_t x) {
  const int i = lower_bound_u64(a, n, x);
  return i < n && lds64(a + 8 * i) == x;
}

// Number of entries of the sorted array of n keys at a that are <= x, the same x on every
// lane: the warp probes 32 equally spaced entries per step.
__device__ __forceinline__ int warp_count_le(saddr a, int n, uint64_t x) {
  const int lane = lane_id();
  int lo = 0;  // entries below lo are <= x, entries from hi on are > x
  int hi = n;
#pragma unroll 1
  while (hi > lo) {
    const int step = (hi - lo + 31) >> 5;
    const int i = lo + (lane + 1) * step - 1;  // the last entry of this lane's stretch
    const unsigned over = __ballot_sync(kFull, i >= hi || lds64(a + 8 * i) > x);
    const int f = over ? __ffs(over) - 1 : 32;  // the first stretch that is not wholly <= x
    const int nlo = lo + f * step;
    hi = f == 32 ? nlo : (nlo + step - 1 < hi ? nlo + step - 1 : hi);
    lo = nlo < n ? nlo : n;
    if (hi < lo) hi = lo;
  }
  return lo;
}

// Transposed reduction over groups of eight lanes of V partial values per lane (V in
// {2, 4, 8}): lane 8 g + u * (8 / V) (and the lanes after it, up to the next) ends with
// value u of its group, summed over pairs of lanes 4, 2 and 1 apart, in this order.
template <int V>
__device__ __forceinline__ float oct_transpose_reduce(float (&v)[V]) {
  const int lane = lane_id();
  int off = 4;
#pragma unroll
  for (int cnt = V; cnt > 1; cnt >>= 1, off >>= 1) {
    const int half = cnt >> 1;
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float send = up ? v[i] : v[i + half];
      const float keep = up ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(kFull, send, off);
    }
  }
#pragma unroll
  for (; off >= 1; off >>= 1) v[0] += __shfl_xor_sync(kFull, v[0], off);
  return v[0];
}

// Vector storage formats. A row is dp4 chunks of 4 elements; every format gives a chunk
// to the same lane, so the reduction tree is the same and only the load width differs
// (16, 8 or 4 bytes per chunk).
//
// Raw is a chunk as loaded (16, 8 or 4 bytes: 4, 2 or 1 registers); decode() turns it
// into four floats, at use.
//
// Read-only loads that leave no line in L1 (kL1: that do): a row is read once by its warp,
// and the L1 beside a full shared memory is small. Volatile: all loads of a group stay
// together in front of the arithmetic. Otherwise the compiler moves each into the branch
// that uses its chunk, and a group costs four memory latencies instead of one.
template <bool kL1>
__device__ __forceinline__ float4 load_stream16(const void* p) {
  float4 v;
  if constexpr (kL1)
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "l"(p));
  else
    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "l"(p));
  return v;
}
template <bool kL1>
__device__ __forceinline__ uint2 load_stream8(const void* p) {
  uint2 v;
  if constexpr (kL1)
    asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  else
    asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
template <bool kL1>
__device__ __forceinline__ uint32_t load_stream4(const void* p) {
  uint32_t v;
  if constexpr (kL1)
    asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v) : "l"(p));
  else
    asm volatile("ld.global.nc.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

struct StoreF32 {
  static constexpr int kChunkBytes = 16;
  static constexpr bool kScaled = false;
  using Raw = float4;
  static constexpr int kRawRegs = 4;
  template <bool kL1 = false>
  __device__ static __forceinline__ Raw load_raw(const unsigned char* row, int c) {
    return load_stream16<kL1>(row + 16 * c);
  }
  __device__ static __forceinline__ Raw zero_raw() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ static __forceinline__ float4 decode(const Raw& r) { return r; }
  __device__ static __forceinline__ float4 load(const unsigned char* row, int c, float) { return load_raw(row, c); }
};
struct StoreBF16 {  // bfloat16, converted from float32 with round-to-nearest-even
  static constexpr int kChunkBytes = 8;
  static constexpr bool kScaled = false;
  using Raw = uint2;
  static constexpr int kRawRegs = 2;
  template <bool kL1 = false>
  __device__ static __forceinline__ Raw load_raw(const unsigned char* row, int c) {
    return load_stream8<kL1>(row + 8 * c);
  }
  __device__ static __forceinline__ Raw zero_raw() { return make_uint2(0u, 0u); }
  __device__ static __forceinline__ float4 decode(const Raw& u) {
    // a bfloat16 is the upper half of a float32
    return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                       __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
  }
  __device__ static __forceinline__ float4 load(const unsigned char* row, int c, float) {
    return decode(load_raw(row, c));
  }
};
// E4M3 codes of x / s with s = max|x| / 448 per vector. load() returns the decoded
// codes without the scale: the distance loops apply s inside their first FMA
// (q - s x as one fused operation, see diff4), so the scale costs no multiply.
struct StoreFP8 {
  static constexpr int kChunkBytes = 4;
  static constexpr bool kScaled = true;
  using Raw = uint32_t;
  static constexpr int kRawRegs = 1;
  template <bool kL1 = false>
  __device__ static __forceinline__ Raw load_raw(const unsigned char* row, int c) {
    return load_stream4<kL1>(row + 4 * c);
  }
  __device__ static __forceinline__ Raw zero_raw() { return 0u; }
  __device__ static __forceinline__ float4 decode(const Raw& u) {
    const __half2_raw lo = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(u & 0xffffu), __NV_E4M3);
    const __half2_raw hi = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(u >> 16), __NV_E4M3);
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&lo));
    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&hi));
    return make_float4(a.x, a.y, b.x, b.y);
  }
  __device__ static __forceinline__ float4 load(const unsigned char* row, int c, float) {
    return decode(load_raw(row, c));
  }
};

template <class T>
using Held = typename T::Raw;  // a chunk as distance groups and the scan hold it

// q - x for a chunk loaded by T::load: for scaled formats x holds codes and the
// difference is q - scale * code, fused.
template <class T>
__device__ __forceinline__ float4 diff4(const float4& q, const float4& x, float scale) {
  if constexpr (T::kScaled) {
    return make_float4(fmaf(-scale, x.x, q.x), fmaf(-scale, x.y, q.y), fmaf(-scale, x.z, q.z),
                       fmaf(-scale, x.w, q.w));
  } else {
    return make_float4(q.x - x.x, q.y - x.y, q.z - x.z, q.w - x.w);
  }
}

// acc + sum (q - x)^2 over a chunk, element by element in one chain; the differences of
// unscaled formats are taken two at a time (packed float32, the same rounding).
template <class T>
__device__ __forceinline__ float sum_sq(const float4& q, const float4& x, float scale, float acc) {
  float4 e;
  if constexpr (T::kScaled) {
    e = diff4<T>(q, x, scale);
  } else {
    asm("{\n .reg .b64 q0, q1, x0, x1;\n mov.b64 q0, {%4, %5};\n mov.b64 q1, {%6, %7};\n mov.b64 x0, {%8, %9};\n"
        " mov.b64 x1, {%10, %11};\n sub.rn.f32x2 q0, q0, x0;\n sub.rn.f32x2 q1, q1, x1;\n mov.b64 {%0, %1}, q0;\n"
        " mov.b64 {%2, %3}, q1;\n}"
        : "=f"(e.x), "=f"(e.y), "=f"(e.z), "=f"(e.w)
        : "f"(q.x), "f"(q.y), "f"(q.z), "f"(q.w), "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w));
  }
  acc = fmaf(e.x, e.x, acc);
  acc = fmaf(e.y, e.y, acc);
  acc = fmaf(e.z, e.z, acc);
  return fmaf(e.w, e.w, acc);
}

// The value of a chunk loaded by T::load (the scale applied for scaled formats).
template <class T>
__device__ __forceinline__ float4 value4(const float4& x, float scale) {
  if constexpr (T::kScaled) return make_float4(scale * x.x, scale * x.y, scale * x.z, scale * x.w);
  else return x;
}

// Copies the query (d floats, any alignment) into qs, dp4 float4 chunks of shared
// memory, zero beyond d. Called by a whole warp, which may read qs afterwards.
__device__ __forceinline__ void load_query(float4* qs, const float* qrow, int d, int dp4) {
  const int lane = lane_id();
  float* f = reinterpret_cast<float*>(qs);
  __syncwarp();
  for (int c = lane; c < 4 * dp4; c += 32) f[c] = c < d ? __ldg(qrow + c) : 0.f;
  __syncwarp();
}

}  // namespace unify
