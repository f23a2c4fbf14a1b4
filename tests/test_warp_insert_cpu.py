"""The sorted-array primitives of the walks, the scan and the construction on an emulated
warp: their text is taken from the CUDA headers and compiled for the host, with 32 threads
that meet at every warp intrinsic and a shared memory that checks each access against the
arrays it holds. Answers are compared with std::sort."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_02448_gb300", "csrc")
FROM = {"common.cuh": ["lower_bound_u64", "warp_lower_bound", "warp_count_le"],
        "warp_ops.cuh": ["warp_rank", "sorted_insert", "rank_among", "rank_plain", "topk_offer"]}

PRELUDE = r"""
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstring>
#include <thread>
#include <vector>
#define __device__
#define __forceinline__ inline
using saddr = uint32_t;
struct ulonglong2 { uint64_t x, y; };
constexpr unsigned kFull = 0xffffffffu;
constexpr uint64_t kKeyMax = ~0ull;
// Shared memory: SK (32 keys) at 4096, the array (kRoom keys) at 8192; anything else is a fault.
constexpr saddr kSK = 4096, kArr = 8192;
constexpr int kRoom = 600;
static uint64_t g_sk[32], g_arr[kRoom];
static std::atomic<int> g_faults{0};
static int g_len = kRoom;  // entries of the array that may be read
static uint64_t* at(saddr a, bool write) {
  static uint64_t dummy;
  if (a >= kSK && a < kSK + 256 && a % 8 == 0) return g_sk + (a - kSK) / 8;
  if (a >= kArr && a < kArr + 8u * (write ? kRoom : g_len) && a % 8 == 0) return g_arr + (a - kArr) / 8;
  ++g_faults;
  return &dummy;
}
static uint64_t lds64(saddr a) { return *at(a, false); }
static void sts64(saddr a, uint64_t v) { *at(a, true) = v; }
static ulonglong2 lds64x2(saddr a) { return {lds64(a), lds64(a + 8)}; }
static thread_local int t_lane;
static std::atomic<int> g_wait{0}, g_turn{0};
static void meet() {
  const int turn = g_turn.load();
  if (g_wait.fetch_add(1) == 31) { g_wait = 0; ++g_turn; return; }
  while (g_turn.load() == turn) std::this_thread::yield();
}
static uint64_t g_x[32];
static int lane_id() { return t_lane; }
static unsigned lanemask_lt() { return (1u << t_lane) - 1u; }
static void __syncwarp() { meet(); }
template <class T, class F> static T all(T v, F f) {
  g_x[t_lane] = 0;
  std::memcpy(&g_x[t_lane], &v, sizeof v);
  meet();
  T r = f();
  meet();
  return r;
}
static unsigned x32(int i) { return (unsigned)g_x[i]; }
static unsigned __ballot_sync(unsigned, bool p) {
  return all<unsigned>(p, [] { unsigned b = 0; for (int i = 0; i < 32; ++i) b |= (x32(i) & 1u) << i; return b; });
}
static unsigned __reduce_or_sync(unsigned, unsigned v) {
  return all<unsigned>(v, [] { unsigned b = 0; for (int i = 0; i < 32; ++i) b |= x32(i); return b; });
}
static unsigned __reduce_min_sync(unsigned, unsigned v) {
  return all<unsigned>(v, [] { unsigned b = ~0u; for (int i = 0; i < 32; ++i) b = std::min(b, x32(i)); return b; });
}
static unsigned __match_any_sync(unsigned, unsigned long long v) {
  return all<uint64_t>(v, [v] { unsigned b = 0; for (int i = 0; i < 32; ++i) b |= (unsigned)(g_x[i] == v) << i; return b; });
}
static uint64_t __shfl_sync(unsigned, uint64_t v, int src) {
  return all<uint64_t>(v, [src] { return g_x[src & 31]; });
}
static int __popc(unsigned v) { return __builtin_popcount(v); }
static int __ffs(unsigned v) { return __builtin_ffs((int)v); }
static int __clz(unsigned v) { return v ? __builtin_clz(v) : 32; }
"""

MAIN = r"""
template <class F> static void warp(F f) {
  std::vector<std::thread> t;
  for (int i = 0; i < 32; ++i) t.emplace_back([&f, i] { t_lane = i; f(i); });
  for (auto& x : t) x.join();
}
// Offers `rounds` x 32 keys to a list of k (twins: equal keys among those of a round); returns its length (list in out), or -1 after
// an access outside the arrays. One array entry beyond the list may not be read.
extern "C" int offer(const uint64_t* keys, int rounds, int k, int twins, uint64_t* out) {
  g_faults = 0;
  std::fill(g_arr, g_arr + kRoom, 0x5555555555555555ull);
  int n = 0;
  for (int r = 0; r < rounds; ++r) {
    int nn[32];
    g_len = std::max(k, n);
    warp([&](int i) {nn[i] = topk_offer(kArr, n, k, keys[32 * r + i], kSK, twins != 0); });
    n = nn[0];
  }
  std::copy(g_arr, g_arr + n, out);
  return g_faults ? -1 : n;
}
// warp_rank, lower_bound_u64 and warp_count_le over a sorted array of n keys for the keys of
// the lanes in kb; 0, or what went wrong.
extern "C" int ranks(const uint64_t* a, int n, const uint64_t* keys, unsigned kb) {
  g_faults = 0;
  g_len = n;
  std::copy(a, a + n, g_arr);
  std::atomic<int> bad{0};
  warp([&](int i) {
    const int want = (int)(std::lower_bound(a, a + n, keys[i]) - a);
    const int w = warp_lower_bound(kArr, n, keys[i], kb), r = warp_rank(kArr, n, keys[i], kb);
    if ((kb >> i) & 1u) { if (w != want) bad = 2; if (r != want) bad = 3; }
    if (lower_bound_u64(kArr, n, keys[i]) != want) bad = 4;
    if (warp_count_le(kArr, n, keys[0]) != (int)(std::upper_bound(a, a + n, keys[0]) - a)) bad = 5;
  });
  return g_faults ? 1 : (int)bad;
}
"""


def _function(text, name):
    m = re.search(r"^__device__ __forceinline__ \w+ " + name + r"\(", text, re.M)
    depth, i = 0, text.index("{", m.start())
    for j in range(i, len(text)):
        depth += (text[j] == "{") - (text[j] == "}")
        if depth == 0:
            return text[m.start():j + 1]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("warp")
    body = "\n".join(_function(open(os.path.join(CSRC, f)).read(), n) for f, ns in FROM.items() for n in ns)
    src = d / "w.cpp"
    src.write_text(PRELUDE + re.sub(r"#pragma unroll.*", "", body) + MAIN)
    so = str(d / "w.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-pthread", str(src), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.offer.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    lib.ranks.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p, ctypes.c_uint]
    return lib


@pytest.mark.parametrize("n", [0, 1, 2, 31, 32, 33, 64, 95, 512])
@pytest.mark.parametrize("lanes", [1, 4, 5, 32])
def test_ranks(lib, n, lanes):
    """Every search finds std::lower_bound / upper_bound and reads inside the array, also an
    empty one."""
    rng = np.random.default_rng([n, lanes])
    a = np.sort(rng.choice(4 * n + 8, size=n, replace=False)).astype(np.uint64)
    keys = rng.integers(0, 4 * n + 8, 32).astype(np.uint64)
    kb = int(sum(1 << int(i) for i in rng.choice(32, lanes, replace=False)))
    assert lib.ranks(a.ctypes.data, n, keys.ctypes.data, kb) == 0


@pytest.mark.parametrize("k", [1, 10, 33, 256])
@pytest.mark.parametrize("lanes", [1, 3, 32])
def test_topk_offer(lib, k, lanes):
    """The k smallest of several offers of `lanes` keys, the first into an empty list."""
    rng = np.random.default_rng([k, lanes])
    rounds = 12
    keys = np.full((rounds, 32), np.iinfo(np.uint64).max, np.uint64)
    keys[:, :lanes] = rng.choice(1 << 20, size=rounds * lanes, replace=False).reshape(rounds, lanes)
    out = np.zeros(600, np.uint64)
    n = lib.offer(keys.ctypes.data, rounds, k, 0, out.ctypes.data)
    want = np.sort(keys[:, :lanes].ravel())[:k]
    assert n == len(want)
    np.testing.assert_array_equal(out[:n], want)


@pytest.mark.parametrize("k", [1, 7, 40, 256])
def test_topk_offer_twins(lib, k):
    """Offers that repeat keys, within themselves and of earlier ones: the k smallest of the
    multiset, every position of the list written."""
    rng = np.random.default_rng([k, 9])
    keys = rng.integers(0, 60, (12, 32)).astype(np.uint64)
    out = np.zeros(600, np.uint64)
    n = lib.offer(keys.ctypes.data, 12, k, 1, out.ctypes.data)
    want = np.sort(keys.ravel())[:k]
    assert n == len(want)
    np.testing.assert_array_equal(out[:n], want)
