// Span metadata, by one block per sequence: validates a sequence's spans and
// scans (k_i - 1); the last block to finish builds the prefix sums over the
// sequences.
#pragma once

#include "plan.cuh"

namespace umim {
namespace {

constexpr int kPlanThreads = 1024;

// Spans a thread takes per pass, consecutive ones: their loads are in flight
// together and a sequence of up to 8192 spans needs one block-wide scan.  With
// one span a thread, four sequences of 4369 spans took five passes of loads,
// scan and barriers (18.4 us against 16.2).
// A pass of fewer spans branches past the items it does not need: predicated off
// instead, in 32 warps, they cost the plan of 1000 prompts of 64 tokens 2 us (28.6
// against 26.5; 2000 prompts of 20 tokens 42.9 against 38.9).
constexpr int kPlanItems = 8;

// Inclusive block-wide scan of four sums at once; every thread gets the totals.
__device__ inline int4 block_scan_incl(int4 v, int4 &total) {
  __shared__ int4 warp_sums[kPlanThreads / 32];
  static_assert(kPlanThreads / 32 == 32, "one lane per warp");
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  auto warp_scan = [&](int4 x) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int4 y = make_int4(__shfl_up_sync(0xffffffffu, x.x, o), __shfl_up_sync(0xffffffffu, x.y, o),
                               __shfl_up_sync(0xffffffffu, x.z, o), __shfl_up_sync(0xffffffffu, x.w, o));
      if (lane >= o) {
        x.x += y.x;
        x.y += y.y;
        x.z += y.z;
        x.w += y.w;
      }
    }
    return x;
  };
  v = warp_scan(v);
  if (lane == 31) warp_sums[w] = v;
  __syncthreads();
  const int4 s = warp_scan(warp_sums[lane]);   // every warp scans the warps' sums
  auto from = [&](int src) {
    return make_int4(__shfl_sync(0xffffffffu, s.x, src), __shfl_sync(0xffffffffu, s.y, src),
                     __shfl_sync(0xffffffffu, s.z, src), __shfl_sync(0xffffffffu, s.w, src));
  };
  total = from(31);
  const int4 add = from(w > 0 ? w - 1 : 0);
  if (w > 0) {
    v.x += add.x;
    v.y += add.y;
    v.z += add.z;
    v.w += add.w;
  }
  __syncthreads();
  return v;
}

// The same for one sum.
__device__ inline int block_scan_incl(int v, int &total) {
  __shared__ int warp_sums[kPlanThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  auto warp_scan = [&](int x) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    return x;
  };
  v = warp_scan(v);
  if (lane == 31) warp_sums[w] = v;
  __syncthreads();
  const int s = warp_scan(warp_sums[lane]);
  total = __shfl_sync(0xffffffffu, s, 31);
  const int add = __shfl_sync(0xffffffffu, s, w > 0 ? w - 1 : 0);
  __syncthreads();
  return v + (w > 0 ? add : 0);
}

// One sequence's spans in shared memory, for a kernel that goes on with them.
struct SpanCopy {
  int32_t *new_idx, *r_incl, *start, *end;   // [cap]
  int cap;                                   // spans beyond it are left out (valid ones never are)
};

struct PlanSeq {
  int L, Lp, lo, hi, first_page, n_dest;   // n_dest 0: nothing to write, or invalid input
  bool last;                               // this block was the last to get here: it calls plan_totals
};

// The block's sequence (blockIdx.x): validates its spans, scans (k_i - 1) and
// writes their compressed indices; every thread gets the result.
__device__ inline PlanSeq plan_sequence(const PlanArgs &a, const PlanArrays &arr, const SpanCopy *copy) {
  const int b = blockIdx.x;
  __shared__ int s_err, s_last;
  if (threadIdx.x == 0) {
    s_err = 0;
    s_last = 0;
  }
  __syncthreads();
  const int L = a.seq_lens ? a.seq_lens[b] : a.fixed_len;
  const int lo = a.span_offsets[b], hi = a.span_offsets[b + 1];
  bool bad = (lo < 0) || (hi < lo) || (hi > a.S) || (L < 0);
  if (a.block_table && (int64_t)L > (int64_t)a.max_pages * kPageSize) bad = true;
  if (bad && threadIdx.x == 0) s_err = 1;
  int removed = 0;   // by the spans of the passes so far
  if (!bad) {        // (the same in every thread)
    if (a.block_table) {
      const int np = ceil_div(L, kPageSize);
      for (int p = threadIdx.x; p < np; p += kPlanThreads) {
        const int pg = a.block_table[(int64_t)b * a.max_pages + p];
        if (pg < 0 || pg >= a.n_pages) s_err = 1;
      }
    }
    for (int base = lo; base < hi; base += kPlanThreads * kPlanItems) {
      const int per = min(kPlanItems, ceil_div(hi - base, kPlanThreads));
      const int i0 = min(base + (int)threadIdx.x * per, hi), n = min(per, hi - i0);
      int s[kPlanItems], k[kPlanItems];
#pragma unroll
      for (int u = 0; u < kPlanItems; ++u) {
        if (u >= per) break;   // (the same in every thread)
        if (u < n) {
          s[u] = a.span_start[i0 + u];
          k[u] = a.span_len[i0 + u];
        }
      }
      // the end of the span before: positions up to it are taken
      int64_t end = n > 0 && i0 > lo ? (int64_t)a.span_start[i0 - 1] + a.span_len[i0 - 1] : 0;
      int sum = 0;
      bool ok = true;
#pragma unroll
      for (int u = 0; u < kPlanItems; ++u) {
        if (u >= per) break;   // (the same in every thread)
        if (u < n) {
          const bool good = k[u] >= 1 && s[u] >= 0 && (int64_t)s[u] + k[u] <= L && end <= s[u] &&
                            !(a.max_span_len > 0 && k[u] > a.max_span_len);
          end = (int64_t)s[u] + k[u];
          ok = ok && good;
          sum += good ? k[u] - 1 : 0;
        }
      }
      if (!ok) s_err = 1;
      int tot;
      int r = removed + block_scan_incl(sum, tot) - sum;   // removed before this thread's spans
#pragma unroll
      for (int u = 0; u < kPlanItems; ++u) {
        if (u >= per) break;   // (the same in every thread)
        if (u < n) {
          const int at = s[u] - r;
          arr.new_idx[i0 + u] = at;
          r += k[u] - 1;
          arr.r_incl[i0 + u] = r;
          if (copy && i0 + u - lo < copy->cap) {
            copy->new_idx[i0 + u - lo] = at;
            copy->r_incl[i0 + u - lo] = r;
            copy->start[i0 + u - lo] = s[u];
            copy->end[i0 + u - lo] = s[u] + k[u];
          }
        }
      }
      removed += tot;
    }
  }
  __syncthreads();
  const int err = s_err;
  const int Lp = err ? L : L - removed;
  int fp = 0, nd = 0;
  if (!err && hi > lo) {
    fp = a.span_start[lo] / kPageSize;
    nd = ceil_div(Lp, kPageSize) - fp;
  }
  if (threadIdx.x == 0) {
    arr.seq_L[b] = L;
    arr.seq_Lp[b] = Lp;
    arr.first_page[b] = fp;
    arr.n_dest[b] = nd;
    if (err) atomicOr(&arr.hdr->error, 1);
    s_last = arrive_is_last(&arr.hdr->blocks_done, (int)gridDim.x);
  }
  __syncthreads();
  return {L, Lp, lo, hi, fp, nd, s_last != 0};
}

// The totals and the per-call header reset, by one thread.
__device__ inline void plan_finish(const PlanArgs &a, const PlanArrays &arr, int err, int4 tot, int max_dest,
                                   int32_t epoch) {
  arr.unit_base[a.B] = tot.x;
  arr.row_base[a.B] = tot.y;
  arr.freed_base[a.B] = tot.z;
  if (a.cu_seqlens_out && !err) a.cu_seqlens_out[a.B] = tot.y;
  PlanHeader *h = arr.hdr;
  h->total_units = err ? 0 : tot.x;
  h->total_rows = tot.y;
  h->max_dest = err ? 0 : max_dest;
  h->n_active = err ? 0 : tot.w;
  h->skip = err ? 1 : 0;
  h->epoch = epoch + 1;
  h->ticket = 0;
  h->done_ctas = 0;
  h->blocks_done = 0;
  h->error = 0;
  if (err) set_error(a.status, UMIM_ERR_INVALID_ARG);
  __threadfence();
}

// Up to 128 sequences: one warp, kTotItems consecutive sequences a lane, every
// load in flight at once.  By the block (below) the serial trips through L2 and
// the barriers took 7000 cycles for four sequences.  The plan of four sequences
// of 4369 spans, traced: 16.4 -> 14.3 us; of a compaction of 64 prompts 12.2 ->
// 10.1.  128 is what a lane's registers hold with ease; the block's scan beyond
// it costs the same 7000 cycles up to 1024 sequences.
constexpr int kTotItems = 4;

__device__ inline void plan_totals_warp(const PlanArgs &a, const PlanArrays &arr) {
  const int lane = threadIdx.x & 31;
  int err = lane == 0 ? atomicOr(&arr.hdr->error, 0) : 0;
  const int32_t epoch = lane == 0 ? __ldcg(&arr.hdr->epoch) : 0;
  int L[kTotItems], Lp[kTotItems], nd[kTotItems];
#pragma unroll
  for (int i = 0; i < kTotItems; ++i) {
    const int j = lane * kTotItems + i;
    L[i] = j < a.B ? __ldcg(arr.seq_L + j) : 0;
    Lp[i] = j < a.B ? __ldcg(arr.seq_Lp + j) : 0;
    nd[i] = j < a.B ? __ldcg(arr.n_dest + j) : 0;
  }
  int4 v = make_int4(0, 0, 0, 0);
  int most = 0;
#pragma unroll
  for (int i = 0; i < kTotItems; ++i) {
    v.x += a.n_lanes * nd[i];
    v.y += Lp[i];
    v.z += ceil_div(L[i], kPageSize) - ceil_div(Lp[i], kPageSize);
    v.w += nd[i] > 0;
    most = max(most, nd[i]);
  }
  most = __reduce_max_sync(0xffffffffu, most);
  err = __shfl_sync(0xffffffffu, err, 0);
  int4 c = v;   // inclusive, then the lane's first sequence
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int4 y = make_int4(__shfl_up_sync(0xffffffffu, c.x, o), __shfl_up_sync(0xffffffffu, c.y, o),
                             __shfl_up_sync(0xffffffffu, c.z, o), __shfl_up_sync(0xffffffffu, c.w, o));
    if (lane >= o) {
      c.x += y.x;
      c.y += y.y;
      c.z += y.z;
      c.w += y.w;
    }
  }
  const int4 tot = make_int4(__shfl_sync(0xffffffffu, c.x, 31), __shfl_sync(0xffffffffu, c.y, 31),
                             __shfl_sync(0xffffffffu, c.z, 31), __shfl_sync(0xffffffffu, c.w, 31));
  c = make_int4(c.x - v.x, c.y - v.y, c.z - v.z, c.w - v.w);
#pragma unroll
  for (int i = 0; i < kTotItems; ++i) {
    const int j = lane * kTotItems + i;
    if (j >= a.B) break;
    arr.unit_base[j] = c.x;
    arr.row_base[j] = c.y;
    arr.freed_base[j] = c.z;
    if (nd[i] > 0) arr.active[c.w++] = j;
    if (a.cu_seqlens_out && !err) a.cu_seqlens_out[j] = c.y;
    c.x += a.n_lanes * nd[i];
    c.y += Lp[i];
    c.z += ceil_div(L[i], kPageSize) - ceil_div(Lp[i], kPageSize);
  }
  if (lane == 0) plan_finish(a, arr, err, tot, most, epoch);
}

// The last block: prefix sums over the sequences, per-call header reset.
__device__ inline void plan_totals(const PlanArgs &a, const PlanArrays &arr) {
  if (a.B <= 32 * kTotItems) {
    if (threadIdx.x < 32) plan_totals_warp(a, arr);
    return;
  }
  const int err = atomicOr(&arr.hdr->error, 0);
  int cu_units = 0, cu_rows = 0, cu_freed = 0, cu_active = 0;
  __shared__ int s_max_dest;
  if (threadIdx.x == 0) s_max_dest = 0;
  __syncthreads();
  for (int j = threadIdx.x; j < a.B; j += kPlanThreads) atomicMax(&s_max_dest, arr.n_dest[j]);
  for (int base = 0; base < a.B; base += kPlanThreads) {
    const int j = base + threadIdx.x;
    int u = 0, r = 0, f = 0;
    if (j < a.B) {
      const int L = arr.seq_L[j], Lp = arr.seq_Lp[j];
      u = a.n_lanes * arr.n_dest[j];
      r = Lp;
      f = ceil_div(L, kPageSize) - ceil_div(Lp, kPageSize);
    }
    const int act = (j < a.B && arr.n_dest[j] > 0) ? 1 : 0;
    int4 tot;
    const int4 incl = block_scan_incl(make_int4(u, r, f, act), tot);
    if (j < a.B) {
      arr.unit_base[j] = cu_units + incl.x - u;
      arr.row_base[j] = cu_rows + incl.y - r;
      arr.freed_base[j] = cu_freed + incl.z - f;
      if (act) arr.active[cu_active + incl.w - 1] = j;
      if (a.cu_seqlens_out && !err) a.cu_seqlens_out[j] = cu_rows + incl.y - r;
    }
    cu_units += tot.x;
    cu_rows += tot.y;
    cu_freed += tot.z;
    cu_active += tot.w;
  }
  if (threadIdx.x == 0)
    plan_finish(a, arr, err, make_int4(cu_units, cu_rows, cu_freed, cu_active), s_max_dest, arr.hdr->epoch);
}

}  // namespace
}  // namespace umim
