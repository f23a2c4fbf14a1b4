// Host side of the fused search kernel (search_kernel.cuh): its arguments, its limits
// and the choice of the storage format's launcher.
#include "search_kernel.cuh"

namespace unify {

// Rows per scan work item, at most p.scan_rows. An item is one warp's, so it is the
// granularity of the batch's tail and, when there are few queries, all the parallelism
// there is: with fewer queries than resident warps (16 per SM) it shrinks in proportion,
// from 1 MB of float32 rows down to 64 KB, and it grows with a pre-filter batch up to 4 MB;
// never below 64 rows, nor below 4 rows per key kept (each item sorts its own list of the
// kept keys, which the query's last item merges). In a routed batch the graph walks hold most
// warps for longer than an item takes, and finer items only take issue slots from them (2 %
// slower at 1,003 queries with 64 KB): there a batch counts sixteenfold, up to 1 MB. Above
// that the items behind the walks are too few for an even end, below it they slow the long
// walks. With 4 MB / 1 MB / 512 KB / 256 KB, 1M x 128 at the tuned parameters: 5,000
// log-uniform queries 2,108 / 1,867 / 1,878 / 1,917 us, 10,000 of five widths 2,061 / 1,970 /
// 1,973 / 2,002; 5,001 log-uniform queries over 200K x 96 FP8 1,281 / 1,276 / 1,299 / 1,305.
// Measured on GB300 against items of 8,192 rows: 17 queries over 15,000 rows of 512 B
// each 585 -> 50 us; 301 queries over 4,200 rows of 3,840 B 4,900 -> 609 us.
int scan_item_rows(const DeviceIndex& ix, const Params& p, int64_t nq, int strategy) {
  const int64_t row_bytes = (int64_t)ix.dp * 4;  // a row's arithmetic is the same in every storage format
  const int64_t slots = 16ll * ix.num_sms;
  int64_t bytes = (1ll << 20) * (strategy == UNIFY_AUTO ? 16 : 1) * nq / slots;
  if (bytes < (64 << 10)) bytes = 64 << 10;
  const int64_t most = strategy == UNIFY_AUTO ? 1 << 20 : 4 << 20;
  if (bytes > most) bytes = most;
  const int64_t kept = rerank_count(p) > p.k ? rerank_count(p) : p.k;
  int64_t rows = bytes / row_bytes;
  if (rows < 64) rows = 64;
  if (rows < 4 * kept) rows = 4 * kept;
  return (int)(rows < p.scan_rows ? rows : p.scan_rows);
}

int rerank_count(const Params& p) { return p.dtype == UNIFY_FP32 ? 0 : p.rerank_mult * p.k; }

int batch_ann_cap(const Params& p) {
  int c = p.ef > p.ef_post ? p.ef : p.ef_post;
  if (c < p.k) c = p.k;
  if (c < rerank_count(p)) c = rerank_count(p);
  return c;
}

// The limit that parameters are checked against: buffers, one flag byte per buffer entry
// and 768 bytes of lists per warp. A configuration within it also runs where the row's
// copy in shared memory makes a warp's share larger: with fewer warps per CTA.
int batch_smem_per_warp(const Params& p) {
  const int ann = batch_ann_cap(p), big = p.cand_cap > ann ? p.cand_cap : ann;
  return (p.cand_cap * 8 + ann * 8 + (4 << p.vis_log2) + ((big + 15) & ~15) + 768 + 15) & ~15;
}

// The build that reg_budget asks for, or the next larger one where shared memory admits no
// more warps per SM than that holds (16 at 128 registers, 20 at 96): a smaller build then
// only has fewer rows in flight per warp. An SM has 228 KB, 1 KB of it lost per CTA.
// Measured on GB300 with the default buffers (12 warps fit), reg_budget 64 in the
// 80-register build / in the 128-register build: 6,000 hybrid queries over 1M x 128 float32
// 3,871 / 2,956 us, 6,000 post-filter ones 1,604 / 1,266, 2,111 short ranges 505 / 408.
static int usable_reg_budget(int asked, int cta_bytes, int wpb) {
  const int warps = 228 * 1024 / (cta_bytes + 1024) * wpb;
  if (warps <= 16) return 128;
  return warps <= 20 && asked == 64 ? 80 : asked;
}

cudaError_t launch_batch(const DeviceIndex& ix, const Scratch& sc, const float* q, const Params& p,
                         const Outputs& o, cudaStream_t st, bool skip_scan, const Conj* cj, bool scan_only) {
  BatchArgs a;
  a.cj = cj ? *cj : Conj{};
  a.skip_scan = skip_scan ? 1 : 0;
  a.vec = ix.vec;
  a.dp4 = ix.dp / 4;
  a.rerank = rerank_count(p);
  if (p.dtype == UNIFY_BF16) {
    a.vt = ix.vt_bf16;
    a.vts = ix.vts_bf16;
    a.scale = a.scale_sorted = nullptr;
    a.row_bytes = a.dp4 * 8;
  } else if (p.dtype == UNIFY_FP8E4M3) {
    a.vt = ix.vt_fp8;
    a.vts = ix.vts_fp8;
    a.scale = ix.scale_fp8;
    a.scale_sorted = ix.scale_fp8_sorted;
    a.row_bytes = a.dp4 * 4;
  } else {
    a.vt = reinterpret_cast<const unsigned char*>(ix.vec);
    a.vts = reinterpret_cast<const unsigned char*>(ix.vec_sorted);
    a.scale = a.scale_sorted = nullptr;
    a.row_bytes = a.dp4 * 16;
  }
  a.sorted_ids = ix.sorted_ids;
  a.d = ix.d;
  a.S = ix.S;
  a.M = ix.M;
  a.max_level = ix.max_level;
  a.entry_global = ix.entry_global;
  a.adj0 = ix.adj0;
  a.gadj0 = ix.gadj0;
  a.adjU = ix.adjU;
  a.gadjU = ix.gadjU;
  a.GW = ix.GW;
  a.repeats = ix.repeats;
  a.upper_base = ix.upper_base;
  a.pos = ix.pos;
  a.seg_start = ix.seg_start;
  a.q = q;
  a.pa = sc.pa;
  a.pb = sc.pb;
  a.mask = sc.mask;
  a.queues = sc.queues;
  a.cap_nq = sc.cap_nq;
  a.nblk = sc.nblk;
  a.qbase = sc.qbase;
  a.done = sc.done;
  a.items = sc.items;
  a.part = sc.part;
  a.counters = sc.counters;
  a.k = p.k;
  a.ef_h = p.ef;
  a.ef_p = p.ef_post;
  a.m = p.m;
  a.s1 = p.selection == 1 ? 1 : 0;
  a.cand_cap = p.cand_cap;
  a.ann_cap = batch_ann_cap(p);
  a.vis_log2 = p.vis_log2;
  a.max_exp = p.max_exp;
  a.scan_only = scan_only ? 1 : 0;
  if (scan_only) {
    // Nothing walks: no visited filter, the lists alone. With the default parameters 16 warps
    // per SM instead of the 12 that fit beside the walks' buffers (the 128-register build):
    // 4,000 queries over 1M x 128 BF16 1,300 -> 955 us, float32 1,552 -> 1,346.
    a.cand_cap = p.k;
    a.ann_cap = p.k > a.rerank ? p.k : a.rerank;
    a.vis_log2 = 6;
  }
  layout(a);
  a.o = o;
  const int fit = (227 * 1024 - kArgsBytes) / a.warp_bytes;
  const int wpb = p.warps_per_block < fit ? p.warps_per_block : fit;
  if (wpb < 1) return cudaErrorInvalidConfiguration;
  const int regs = usable_reg_budget(p.reg_budget, kArgsBytes + wpb * a.warp_bytes, wpb);
  if (p.dtype == UNIFY_BF16) return launch_batch_bf16(a, wpb, regs, ix.num_sms, st);
  if (p.dtype == UNIFY_FP8E4M3) return launch_batch_fp8(a, wpb, regs, ix.num_sms, st);
  return launch_batch_f32(a, wpb, regs, ix.num_sms, st);
}

}  // namespace unify
