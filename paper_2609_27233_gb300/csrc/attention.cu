// Grouped-query decode attention over the compacted paged bf16 cache
// (App. I.1: decode attends to the accumulated, now shorter, KV cache).
//
// Balanced split-K: the (sequence b, KV head g, page) triples of the whole
// batch are flattened, (b, g)-major, and every warp of a persistent grid
// takes an equal contiguous range of them.  A range piece that lies in one
// (b, g) segment produces one partial (running max m, sum l, unnormalised
// output acc) for the G query heads sharing KV head g; a small combine
// kernel merges the pieces of each segment with log-sum-exp weights.  The plan
// is one prefix sum of pages over the sequences: every CTA of the decode kernel
// derives it from the lengths in shared memory (up to 4096 sequences, 16 KB next
// to the rings; a kernel of its own before it otherwise), and the piece of
// segment s that warp w holds has number s + w, which no two pieces share.  A
// plan kernel before every call cost 3 us of a call of 16 (four sequences of
// 24 000 entries: rollback and attention 178.3 -> 175.8 us).
//
// Per warp: a private ring of NST stages; an elected lane issues TMA tensor loads of
// whole pages (K and V tiles of 16 x D bf16, 128-byte swizzled) into the
// ring and each stage completes an mbarrier.  S = Q K^T (G <= 16 query heads
// as the M=16 side) and O += P V run as mma.sync m16n8k16 on operands read
// with ldmatrix from the swizzled tiles; softmax is online in fp32 with the
// row statistics shared across the 4 threads of an mma row by shuffles.
// Each KV byte is read once from HBM for all G query heads.
#include <algorithm>

#include "common.cuh"
#include "mma.cuh"

namespace umim {
namespace {

// 12 warps x 2 stages (168 registers a thread, 192 KB of rings) moved more bytes
// than 8 x 3, 9 x 3, 10 x 2, 7 x 4, 6 x 4 or 4 x 6; 13 or more warps spill.
constexpr int kAttnWarps = 12;
constexpr int kAttnStages = 2;
constexpr int kPlanThreadsA = 1024;

constexpr int kSmemPlanBatch = 4096;   // sequences whose prefix sum a decode CTA keeps in shared memory

struct AttnPlan {
  int32_t W;          // pages per warp
  int32_t pad[63];
};

struct AttnWs {
  AttnPlan *plan;
  int32_t *pref;      // [B + 1] pages before sequence b (of one KV head)
  float2 *part_ml;    // [pieces][16]      (m in log2 units, l)
  float *part_acc;    // [pieces][16][D]
};

inline size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

inline size_t attn_ws_bytes(int B, int Hkv, int D, int total_warps) {
  const size_t nseg = (size_t)B * Hkv;
  const size_t pieces = nseg + total_warps;
  size_t b = a256(sizeof(AttnPlan)) + a256(sizeof(int32_t) * (B + 1));
  b += a256(sizeof(float2) * pieces * 16);
  b += a256(sizeof(float) * pieces * 16 * D);
  return b;
}

inline AttnWs attn_carve(void *ws, int B, int Hkv, int D, int total_warps) {
  const size_t nseg = (size_t)B * Hkv;
  const size_t pieces = nseg + total_warps;
  char *p = static_cast<char *>(ws);
  AttnWs w;
  w.plan = reinterpret_cast<AttnPlan *>(p);
  p += a256(sizeof(AttnPlan));
  w.pref = reinterpret_cast<int32_t *>(p);
  p += a256(sizeof(int32_t) * (B + 1));
  w.part_ml = reinterpret_cast<float2 *>(p);
  p += a256(sizeof(float2) * pieces * 16);
  w.part_acc = reinterpret_cast<float *>(p);
  return w;
}

// ---------------------------------------------------------------------------
// plan
// ---------------------------------------------------------------------------
// Exclusive prefix sum of every sequence's pages into pref[0 .. B] by a block of
// T threads; returns the total (every thread).  A length outside the block
// table counts as 0 and is recorded when `report` is set.
template <int T>
__device__ int plan_prefix(const int32_t *seq_lens, int B, int max_pages, int32_t *pref, bool report,
                           int32_t *status) {
  static_assert(T <= 1024, "one warp scans the warps' sums");
  __shared__ int s_sum[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int carry = 0;
  for (int b0 = 0; b0 < B; b0 += T) {
    const int b = b0 + threadIdx.x;
    int n = 0;
    if (b < B) {
      int L = seq_lens[b];
      if (L < 0 || (int64_t)L > (int64_t)max_pages * kPageSize) {
        if (report) set_error(status, UMIM_ERR_INVALID_ARG);
        L = 0;
      }
      n = ceil_div(L, kPageSize);
    }
    int x = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_sum[w] = x;
    __syncthreads();
    int v = lane < T / 32 ? s_sum[lane] : 0;   // every warp scans the warps' sums
#pragma unroll
    for (int o = 1; o < T / 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += y;
    }
    const int before = w ? __shfl_sync(0xffffffffu, v, w - 1) : 0;
    if (b < B) pref[b] = carry + before + x - n;
    carry += __shfl_sync(0xffffffffu, v, T / 32 - 1);
    __syncthreads();
  }
  if (threadIdx.x == 0) pref[B] = carry;
  __syncthreads();
  return carry;
}

// more than kSmemPlanBatch sequences: the prefix sum in a kernel of its own (one block)
__global__ void __launch_bounds__(kPlanThreadsA)
    attn_plan_kernel(const int32_t *seq_lens, int B, int max_pages, AttnWs ws, int32_t *status) {
  griddep_wait();
  plan_prefix<kPlanThreadsA>(seq_lens, B, max_pages, ws.pref, true, status);
}

// ---------------------------------------------------------------------------
// main kernel
// ---------------------------------------------------------------------------
struct AttnArgs {
  const __nv_bfloat16 *q;
  const int32_t *block_table;
  const int32_t *seq_lens;
  int32_t B, Hq, Hkv, G, max_pages, n_pages, layer, n_layers;
  int32_t smem_plan;
  float scale_log2;
  int32_t *status;
};

// swizzled byte offset of 16-byte chunk c16 (0 .. D/8-1) of row r in a tile
// stored as D/64 boxes of [16 rows][128 B] with 128-byte swizzling
__device__ __forceinline__ uint32_t sw_off(int r, int c16) {
  const int box = c16 >> 3, cc = c16 & 7;
  return box * 2048 + r * 128 + ((cc ^ (r & 7)) << 4);
}

template <int D>
__global__ void __launch_bounds__(kAttnWarps * 32, 1)
    attn_decode_kernel(const __grid_constant__ CUtensorMap kv_map, AttnArgs a, AttnWs ws) {
  constexpr int kTile = 16 * D * 2;        // bytes of one K (or V) tile
  constexpr int kStage = 2 * kTile;
  constexpr int NB = D / 64;               // 128-byte boxes per tile row
  constexpr int NT = D / 8;                // n-tiles of the output
  constexpr int KC = D / 16;               // k-chunks of Q K^T
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ uint64_t bars[kAttnWarps][kAttnStages];

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int gw = blockIdx.x * kAttnWarps + warp, total_warps = gridDim.x * kAttnWarps;
  uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *wbuf = base + warp * kAttnStages * kStage;

  if (lane == 0) {
    for (int s = 0; s < kAttnStages; ++s) mbar_init(&bars[warp][s], 1);
    fence_mbar_init();
    if (warp == 0) prefetch_tensormap(&kv_map);
  }
  __syncwarp();
  griddep_wait();

  const int G = a.G, Hkv = a.Hkv;
  const int32_t *pref = ws.pref;
  int pages;
  if (a.smem_plan) {
    int32_t *mine = reinterpret_cast<int32_t *>(base + kAttnWarps * kAttnStages * kStage);
    pages = plan_prefix<kAttnWarps * 32>(a.seq_lens, a.B, a.max_pages, mine, blockIdx.x == 0, a.status);
    pref = mine;
    if (blockIdx.x == 0)   // for the combine kernel
      for (int b = threadIdx.x; b <= a.B; b += kAttnWarps * 32) ws.pref[b] = mine[b];
  } else {
    pages = pref[a.B];
  }
  const int total = Hkv * pages;
  const int W = max(1, ceil_div(total, total_warps));
  if (blockIdx.x == 0 && threadIdx.x == 0) ws.plan->W = W;
  const int start = (int)min((int64_t)gw * W, (int64_t)total);
  const int end = min(total, start + W);
  if (start >= end) return;

  const uint64_t pol = policy_evict_first();

  // (sequence, KV head, page) of a flattened position: the last sequence whose
  // first page is at or before it (sequences without pages share their successor's)
  auto locate = [&](int pos, int &b, int &g, int &pi) {
    int l = 0, h = a.B;
    while (h - l > 1) {
      const int m = (l + h) >> 1;
      if (Hkv * pref[m] <= pos) l = m;
      else h = m;
    }
    b = l;
    const int n = pref[b + 1] - pref[b];
    const int r = pos - Hkv * pref[b];
    g = r / n;
    pi = r - g * n;
  };

  // ---- compute cursor and loader cursor (every lane keeps both; one issues the copies) ----
  int cb, cg, cpi;
  locate(start, cb, cg, cpi);
  int cn = pref[cb + 1] - pref[cb], cL = a.seq_lens[cb];
  int ld_pos = start, lb = cb, lg = cg, lpi = cpi, ln = cn;
  auto issue = [&](int stage) {
    const int page = in_bounds(lpi, a.max_pages, a.status, kSiteAttnTable)
                         ? a.block_table[(int64_t)lb * a.max_pages + lpi] : -1;
    int c4 = a.layer * a.n_pages + page;
    if (page < 0 || page >= a.n_pages) {
      // a coordinate past the tensor's last page: the copy reads zeros
      set_error(a.status, UMIM_ERR_INVALID_ARG);
      c4 = a.n_layers * a.n_pages;
    }
    if (elect_one()) {
      uint64_t *bar = &bars[warp][stage];
      uint8_t *dst = wbuf + stage * kStage;
      mbar_arrive_expect_tx(bar, kStage);
#pragma unroll
      for (int c = 0; c < NB; ++c) {
        tma_load_5d(dst + c * 2048, &kv_map, bar, c * 64, 0, lg, 0, c4, pol);
        tma_load_5d(dst + kTile + c * 2048, &kv_map, bar, c * 64, 0, lg, 1, c4, pol);
      }
    }
    if (++ld_pos < end && ++lpi == ln) {
      lpi = 0;
      if (++lg == Hkv) {
        lg = 0;
        do ++lb;
        while (pref[lb + 1] == pref[lb]);
        ln = pref[lb + 1] - pref[lb];
      }
    }
  };
  for (int s = 0; s < kAttnStages && ld_pos < end; ++s) issue(s);

  // ---- compute state ----
  const int qr = lane >> 2, qc = lane & 3;      // mma fragment row / column group
  uint32_t qa[KC][4];
  auto load_q = [&]() {
    const __nv_bfloat16 *qbase = a.q + ((int64_t)cb * a.Hq + (int64_t)cg * G) * D;
#pragma unroll
    for (int c = 0; c < KC; ++c) {
      const int k0 = c * 16 + 2 * qc;
      const uint32_t *r0 = reinterpret_cast<const uint32_t *>(qbase + (int64_t)qr * D + k0);
      const uint32_t *r1 = reinterpret_cast<const uint32_t *>(qbase + (int64_t)(qr + 8) * D + k0);
      qa[c][0] = qr < G ? r0[0] : 0u;
      qa[c][1] = qr + 8 < G ? r1[0] : 0u;
      qa[c][2] = qr < G ? r0[4] : 0u;
      qa[c][3] = qr + 8 < G ? r1[4] : 0u;
    }
  };
  load_q();
  float acc[NT][4];
  float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
#pragma unroll
  for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;

  auto flush = [&]() {
    // complete the row sums across the 4 threads of each row
    float s0 = l0, s1 = l1;
    s0 += __shfl_xor_sync(0xffffffffu, s0, 1);
    s0 += __shfl_xor_sync(0xffffffffu, s0, 2);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 2);
    const int piece = cb * Hkv + cg + gw;
    if (!in_bounds(piece, (int64_t)a.B * Hkv + total_warps, a.status, kSiteAttnPiece)) return;
    float2 *ml = ws.part_ml + (int64_t)piece * 16;
    float *pacc = ws.part_acc + (int64_t)piece * 16 * D;
    if (qc == 0) {
      if (qr < G) ml[qr] = make_float2(m0, s0);
      if (qr + 8 < G) ml[qr + 8] = make_float2(m1, s1);
    }
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      const int col = j * 8 + 2 * qc;
      if (qr < G) *reinterpret_cast<float2 *>(pacc + qr * D + col) = make_float2(acc[j][0], acc[j][1]);
      if (qr + 8 < G) *reinterpret_cast<float2 *>(pacc + (qr + 8) * D + col) = make_float2(acc[j][2], acc[j][3]);
    }
  };

  int it = 0;
  for (int pos = start; pos < end; ++pos, ++it) {
    // next segment?
    if (cpi == cn) {
      flush();
      cpi = 0;
      if (++cg == Hkv) {
        cg = 0;
        do ++cb;
        while (pref[cb + 1] == pref[cb]);
        cn = pref[cb + 1] - pref[cb];
        cL = a.seq_lens[cb];
      }
      load_q();
      m0 = m1 = -INFINITY;
      l0 = l1 = 0.f;
#pragma unroll
      for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    }
    const int stage = it % kAttnStages;
    const uint32_t parity = (it / kAttnStages) & 1;
    if (!mbar_wait(&bars[warp][stage], parity)) {
      set_error(a.status, UMIM_ERR_TIMEOUT);
      // let the copies still in flight land (each wait bounded) before leaving
      for (int k = 1; k < kAttnStages && pos + k < ld_pos; ++k)
        mbar_wait(&bars[warp][(it + k) % kAttnStages], ((it + k) / kAttnStages) & 1);
      return;
    }
    uint8_t *kt = wbuf + stage * kStage;
    uint8_t *vt = kt + kTile;
    const int nvalid = min(16, cL - cpi * 16);
    ++cpi;
    if (nvalid < 16) {
      // zero V rows past the end so that 0 * garbage cannot make a NaN
      for (int idx = lane; idx < (16 - nvalid) * NB * 8; idx += 32) {
        const int r = nvalid + idx / (NB * 8);
        const int c16 = idx % (NB * 8);
        *reinterpret_cast<uint4 *>(vt + sw_off(r, c16)) = make_uint4(0, 0, 0, 0);
      }
      // order these generic-proxy writes before the next TMA write of the stage
      fence_proxy_async_smem();
      __syncwarp();
    }
    const uint32_t ks = smem_u32(kt), vs = smem_u32(vt);

    // S = Q K^T   (16 x 16 keys as two n-tiles of 8); even and odd k-chunks
    // accumulate separately to halve the dependent mma chain
    float s[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    float s2[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int c = 0; c < KC; ++c) {
      const int key = (lane & 7) + ((lane >> 4) << 3);
      const int c16 = 2 * c + ((lane >> 3) & 1);
      uint32_t b0, b1, b2, b3;
      ldsm_x4(ks + sw_off(key, c16), b0, b1, b2, b3);
      if (c & 1) {
        mma_bf16(s2[0], qa[c], b0, b1);
        mma_bf16(s2[1], qa[c], b2, b3);
      } else {
        mma_bf16(s[0], qa[c], b0, b1);
        mma_bf16(s[1], qa[c], b2, b3);
      }
    }
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) s[nt][e] += s2[nt][e];
    // scale to log2 units and mask keys past the end
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int key = nt * 8 + 2 * qc + (e & 1);
        s[nt][e] = key < nvalid ? s[nt][e] * a.scale_log2 : -INFINITY;
      }
    float mx0 = fmaxf(fmaxf(s[0][0], s[0][1]), fmaxf(s[1][0], s[1][1]));
    float mx1 = fmaxf(fmaxf(s[0][2], s[0][3]), fmaxf(s[1][2], s[1][3]));
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
    const float was0 = m0, was1 = m1;
    m0 = fmaxf(m0, mx0);
    m1 = fmaxf(m1, mx1);
    // no finite score so far: weights from 0, so that a score of -inf weighs 0 and NaN stays NaN
    const float n0 = m0 == -INFINITY ? 0.f : m0, n1 = m1 == -INFINITY ? 0.f : m1;
    const float c0 = exp2f(was0 - n0), c1 = exp2f(was1 - n1);
    float p[2][4];
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      p[nt][0] = exp2f(s[nt][0] - n0);
      p[nt][1] = exp2f(s[nt][1] - n0);
      p[nt][2] = exp2f(s[nt][2] - n1);
      p[nt][3] = exp2f(s[nt][3] - n1);
    }
    l0 = l0 * c0 + p[0][0] + p[0][1] + p[1][0] + p[1][1];
    l1 = l1 * c1 + p[0][2] + p[0][3] + p[1][2] + p[1][3];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      acc[j][0] *= c0;
      acc[j][1] *= c0;
      acc[j][2] *= c1;
      acc[j][3] *= c1;
    }
    // P as the A operand, split into a bf16 high part and a bf16 remainder
    uint32_t ph[4], pl[4];
    {
      const float v[4][2] = {{p[0][0], p[0][1]}, {p[0][2], p[0][3]}, {p[1][0], p[1][1]}, {p[1][2], p[1][3]}};
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v[r][0], v[r][1]);
        ph[r] = *reinterpret_cast<const uint32_t *>(&h);
        pl[r] = pack_bf16(v[r][0] - __low2float(h), v[r][1] - __high2float(h));
      }
    }
    // O += P V
#pragma unroll
    for (int j = 0; j < D / 16; ++j) {
      const int key = (lane & 7) + (((lane >> 3) & 1) << 3);
      const int c16 = 2 * j + (lane >> 4);
      uint32_t b0, b1, b2, b3;
      ldsm_x4_t(vs + sw_off(key, c16), b0, b1, b2, b3);
      mma_bf16(acc[2 * j], ph, b0, b1);
      mma_bf16(acc[2 * j + 1], ph, b2, b3);
      mma_bf16(acc[2 * j], pl, b0, b1);
      mma_bf16(acc[2 * j + 1], pl, b2, b3);
    }
    __syncwarp();
    // refill this stage
    if (ld_pos < end) issue(stage);
  }
  flush();
}

// ---------------------------------------------------------------------------
// combine: WPR warps per (b, query head) row, 256 threads per CTA.  The warps
// of a row split its segment's pieces, each merges its share in one pass with
// a running maximum, and (WPR > 1) the warps' (m, l, acc) are merged through
// shared memory.  WPR grows with the pieces per segment (few, long sequences
// split into many pieces).
// ---------------------------------------------------------------------------
constexpr int kCombineThreads = 256;

template <int D, int WPR>
__global__ void __launch_bounds__(kCombineThreads)
    attn_combine_kernel(AttnWs ws, int B, int Hq, int Hkv, int G, __nv_bfloat16 *out) {
  constexpr int E = D / 32;
  constexpr int RPB = kCombineThreads / 32 / WPR;   // rows per CTA
  __shared__ float s_m[kCombineThreads / 32], s_l[kCombineThreads / 32];
  __shared__ float s_acc[WPR > 1 ? kCombineThreads / 32 : 1][D];
  griddep_wait();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row_g = blockIdx.x * RPB + warp / WPR, sub = warp % WPR;
  const bool live = row_g < B * Hq;
  const int b = live ? row_g / Hq : 0, h = live ? row_g % Hq : 0;
  const int seg = b * Hkv + h / G, row = h % G;
  // the segment's pieces: seg + w for the warps w whose ranges meet its positions
  int p0 = 0, p1 = 0;
  if (live) {
    const int first = ws.pref[b], n = ws.pref[b + 1] - first, W = ws.plan->W;
    const int o = Hkv * first + h / G * n;
    if (n > 0) {
      p0 = seg + o / W;
      p1 = seg + (o + n - 1) / W + 1;
    }
  }
  float M = -INFINITY, l = 0.f, o[E];
#pragma unroll
  for (int e = 0; e < E; ++e) o[e] = 0.f;
  // pieces whose loads are in flight together: one at a time, a row of 76 pieces
  // (long context, 16.4 us with eight warps a row) waits for memory ten times over;
  // four at a time 8.3 us
  constexpr int U = 4;
  for (int pc = p0 + sub; pc < p1; pc += U * WPR) {
    float2 ml[U];
    float av[U][E];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t at = (int64_t)(pc + u * WPR) * 16 + row;
      ml[u] = make_float2(-INFINITY, 0.f);
#pragma unroll
      for (int e = 0; e < E; ++e) av[u][e] = 0.f;
      if (pc + u * WPR < p1) {
        ml[u] = ws.part_ml[at];
        if constexpr (E == 4) {
          const float4 f = *reinterpret_cast<const float4 *>(ws.part_acc + at * D + lane * E);
          av[u][0] = f.x, av[u][1] = f.y, av[u][2] = f.z, av[u][3] = f.w;
        } else {
          const float2 f = *reinterpret_cast<const float2 *>(ws.part_acc + at * D + lane * E);
          av[u][0] = f.x, av[u][1] = f.y;
        }
      }
    }
    float nm = M;
#pragma unroll
    for (int u = 0; u < U; ++u) nm = fmaxf(nm, ml[u].x);
    // (a piece whose scores are all NaN has no maximum either, but a NaN sum: weighted, not skipped)
    const float from = nm == -INFINITY ? 0.f : nm;
    const float c_old = exp2f(M - from);
    l *= c_old;
#pragma unroll
    for (int e = 0; e < E; ++e) o[e] *= c_old;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float c = exp2f(ml[u].x - from);   // 0 for an absent or empty piece
      l = fmaf(ml[u].y, c, l);
#pragma unroll
      for (int e = 0; e < E; ++e) o[e] = fmaf(av[u][e], c, o[e]);
    }
    M = nm;
  }
  if constexpr (WPR > 1) {
    if (lane == 0) {
      s_m[warp] = M;
      s_l[warp] = l;
    }
#pragma unroll
    for (int e = 0; e < E; ++e) s_acc[warp][lane * E + e] = o[e];
    __syncthreads();
    if (sub != 0) return;
    float Mx = -INFINITY;
#pragma unroll
    for (int w = 0; w < WPR; ++w) Mx = fmaxf(Mx, s_m[warp + w]);
    l = 0.f;
#pragma unroll
    for (int e = 0; e < E; ++e) o[e] = 0.f;
    if (Mx == -INFINITY) Mx = 0.f;
#pragma unroll
    for (int w = 0; w < WPR; ++w) {
      const float c = exp2f(s_m[warp + w] - Mx);
      l += c * s_l[warp + w];
#pragma unroll
      for (int e = 0; e < E; ++e) o[e] += c * s_acc[warp + w][lane * E + e];
    }
  }
  if (!live) return;
  const float inv = p1 > p0 ? 1.f / l : 0.f;   // (no entries: zeros)
  __nv_bfloat16 *dst = out + ((int64_t)b * Hq + h) * D + lane * E;
#pragma unroll
  for (int e = 0; e < E; ++e) dst[e] = __float2bfloat16_rn(o[e] * inv);
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                   CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                   CUtensorMapFloatOOBfill);
EncodeTiledFn get_encode_tiled();

int attn_total_warps(int num_sms) { return std::max(1, num_sms) * kAttnWarps; }

size_t decode_attention_workspace_bytes(int B, int Hq, int Hkv, int D, int num_sms) {
  (void)Hq;
  return attn_ws_bytes(B, Hkv, D, attn_total_warps(num_sms));
}

template <int D>
static umim_status run_attention(const void *q, int Hq, const umim_paged_kv *kv, int layer,
                                 const int32_t *block_table, int max_pages, const int32_t *seq_lens, int B,
                                 float scale, void *out, void *workspace, int32_t *status, cudaStream_t stream,
                                 int num_sms) {
  EncodeTiledFn enc = get_encode_tiled();
  if (!enc) return UMIM_ERR_CUDA;
  CUtensorMap map;
  const cuuint64_t dims[5] = {(cuuint64_t)D, 16, (cuuint64_t)kv->n_kv_heads, 2,
                              (cuuint64_t)kv->n_layers * (cuuint64_t)kv->n_pages};
  const cuuint64_t strides[4] = {(cuuint64_t)D * 2, (cuuint64_t)16 * D * 2,
                                 (cuuint64_t)kv->n_kv_heads * 16 * D * 2,
                                 (cuuint64_t)2 * kv->n_kv_heads * 16 * D * 2};
  const cuuint32_t box[5] = {64, 16, 1, 1, 1};
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, kv->base, dims, strides, box, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return UMIM_ERR_CUDA;
  const int total_warps = attn_total_warps(num_sms);
  const int Hkv = kv->n_kv_heads;
  AttnWs ws = attn_carve(workspace, B, Hkv, D, total_warps);
  const bool smem_plan = B <= kSmemPlanBatch;
  if (!smem_plan) {
    trace_mark(stream, "attention.plan");
    if (launch_pdl(attn_plan_kernel, dim3(1), dim3(kPlanThreadsA), 0, stream, seq_lens, B, max_pages, ws, status) !=
        cudaSuccess)
      return UMIM_ERR_CUDA;
  }

  AttnArgs a{};
  a.smem_plan = smem_plan ? 1 : 0;
  a.q = static_cast<const __nv_bfloat16 *>(q);
  a.block_table = block_table;
  a.seq_lens = seq_lens;
  a.B = B;
  a.Hq = Hq;
  a.Hkv = Hkv;
  a.G = Hq / Hkv;
  a.max_pages = max_pages;
  a.n_pages = kv->n_pages;
  a.layer = layer;
  a.n_layers = kv->n_layers;
  a.scale_log2 = scale * 1.4426950408889634f;
  a.status = status;
  constexpr size_t kRings = (size_t)kAttnWarps * kAttnStages * 2 * 16 * D * 2 + 1024;
  const size_t smem = kRings + (smem_plan ? sizeof(int32_t) * ((size_t)B + 1) : 0);
  auto kern = attn_decode_kernel<D>;
  if (!allow_smem(kern, kRings + sizeof(int32_t) * (kSmemPlanBatch + 1))) return UMIM_ERR_CUDA;
  trace_mark(stream, "attention.decode");
  if (launch_pdl(kern, dim3(total_warps / kAttnWarps), dim3(kAttnWarps * 32), smem, stream, map, a, ws) !=
      cudaSuccess)
    return UMIM_ERR_CUDA;
  trace_mark(stream, "attention.combine");
  // warps per row: about half the pieces a segment has (1 + warps / segments)
  const int per_seg = 1 + total_warps / std::max(1, B * Hkv);
  const int wpr = per_seg >= 16 ? 8 : per_seg >= 8 ? 4 : per_seg >= 4 ? 2 : 1;
  const int rows_per_cta = kCombineThreads / 32 / wpr;
  auto comb = wpr == 8 ? attn_combine_kernel<D, 8>
              : wpr == 4 ? attn_combine_kernel<D, 4>
              : wpr == 2 ? attn_combine_kernel<D, 2> : attn_combine_kernel<D, 1>;
  if (launch_pdl(comb, dim3((unsigned)((B * Hq + rows_per_cta - 1) / rows_per_cta)), dim3(kCombineThreads), 0, stream,
                 ws, B, Hq, Hkv, a.G, static_cast<__nv_bfloat16 *>(out)) != cudaSuccess)
    return UMIM_ERR_CUDA;
  trace_mark(stream, nullptr);
  return cudaGetLastError() == cudaSuccess ? UMIM_OK : UMIM_ERR_CUDA;
}

umim_status decode_attention(const void *q, int Hq, const umim_paged_kv *kv, int layer, const int32_t *block_table,
                             int max_pages, const int32_t *seq_lens, int B, float scale, void *out,
                             void *workspace, int32_t *status, cudaStream_t stream, int num_sms) {
  if (kv->head_dim == 128)
    return run_attention<128>(q, Hq, kv, layer, block_table, max_pages, seq_lens, B, scale, out, workspace,
                              status, stream, num_sms);
  return run_attention<64>(q, Hq, kv, layer, block_table, max_pages, seq_lens, B, scale, out, workspace, status,
                           stream, num_sms);
}

}  // namespace umim
