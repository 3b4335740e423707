// Causal grouped-query prefill attention over packed compressed prompts (App.
// E "Prompt Merging", App. C.5: the compressed embeddings, with contiguous
// positions, go through the frozen backbone's prefill, whose self-attention
// then runs over the shorter sequences).  Sequence b owns rows
// cu_seqlens[b] .. cu_seqlens[b+1]-1 of q [T][Hq][D], k, v [T][Hkv][D].
//
// On the 5th-generation tensor cores, in one of two kernels: one head at a
// time, described here, or two heads of an even group at a time (below), for
// enough work.  One head: a persistent kernel, two CTAs per SM (each allocates
// half of the tensor memory, so one CTA's products fill the tensor cores while
// the other's softmax runs), each walking work units of 128 query rows of one
// sequence for one query head, heaviest first; the next unit's Q and K loads
// and first S products overlap the current unit's last tiles and epilogue.
// Warp 0 loads tiles with TMA (a unit's Q; 64-key K tiles into a 2-stage ring
// running a tile ahead of the V^T tiles' 2-stage ring), warp 1 issues the S = Q
// K^T products (tcgen05.mma into one of two tensor-memory buffers, reused once
// the P V product that read it is done), warp 6 the O += P V products into a
// tensor-memory accumulator (a separate issuing thread, so that a P V product
// never waits behind an S product that waits for the previous P V), and warps
// 2-5 run the online softmax, one thread per query row: S from tensor memory
// (tcgen05.ld), causal mask, running max, P = exp2(S - max) written back in
// fp16 over the S columns it came from (tcgen05.st; the P V product reads its A
// operand from tensor memory, so P never touches shared memory), row sums.  P V
// runs on fp16 operands (V^T is converted when it is transposed): fp16's 11-bit
// significand keeps P's and V's rounding near 3e-4 relative, where bf16 P would
// cost 1e-3 of the output's error budget; P <= 2^8 by construction and |v| <
// 65504 is checked (UMIM_ERR_UNSUPPORTED otherwise).  The running max is only
// moved when it grows by more than 2^8, so the accumulator in tensor memory is
// rescaled rarely (the result is the same: P and the row sum use the same stale
// max).
//
// V is transposed first (per sequence, padded to a multiple of 64 keys) so
// that both products read K-major operands and every TMA copy starts on a
// 16-byte boundary.  The transposing CTAs turn cu_seqlens into per-sequence tile
// offsets and padded key offsets (and validate them) in shared memory, each for
// itself, and write every query tile's record; beyond kPfSmemBatch sequences a plan
// kernel ahead of them derives the offsets.  Tiles run heaviest (last in their
// sequence) first.
#include <cuda_fp16.h>

#include "common.cuh"

namespace umim {

using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                   CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                   CUtensorMapFloatOOBfill);
EncodeTiledFn get_encode_tiled();

namespace {

constexpr int kPfRows = 128;             // query rows per CTA (the MMA's M)
constexpr int kPfKeys = 64;              // keys per K / V tile (the S MMA's N)
constexpr int kPfKStages = 2;            // K ring (K runs kPfKStages - 1 tiles ahead of V^T)
constexpr int kPfVStages = 2;            // V^T ring
constexpr int kPfThreads = 224;          // warp 0 TMA, warp 1 S products + tensor memory, warps 2-5 softmax
                                         // (thread = query row), warp 6 P V products
constexpr int kPfPlanThreads = 1024, kPfVtThreads = 256;
constexpr int kPfSmemBatch = 2048;       // sequences whose prefix sums a V^T CTA keeps in shared memory
constexpr uint32_t kPfTmemCols = 256;    // S buffers at 0 and 64, O at 128: two CTAs per SM

struct PfArgs {
  __nv_bfloat16 *out;               // [T][Hq][D]
  const int32_t *cu;                // [B + 1]
  int32_t *cu_tiles;                // [B + 1] workspace: query-tile offsets
  int32_t *pcu;                     // [B + 1] workspace: key offsets padded to 64 in V^T
  int4 *tiles;                      // [query tiles] workspace: first row, length, first query, V^T column of the sequence
  const __nv_bfloat16 *v;           // [T][Hkv][D]
  __half *vt;                       // [Hkv][D][Tp] workspace, fp16
  int64_t Tp;                       // row length of V^T (a multiple of 64)
  int32_t B, T, Hq, Hkv, G;
  float scale_log2;
  int32_t *status;
};

// Exclusive prefix sums over the sequences of query tiles (cu_tiles) and of
// lengths rounded up to 64 keys (pcu), [0 .. B], by a block of T threads, which
// also validates cu_seqlens: invalid offsets leave totals of 0, no work at all.
template <int T>
__device__ void pf_prefix(const PfArgs &a, int32_t *cu_tiles, int32_t *pcu, bool report) {
  __shared__ int s_wsum[2][32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int err = a.cu[0] != 0 || a.cu[a.B] > a.T;
  int carry_t = 0, carry_p = 0;
  for (int base = 0; base < a.B; base += T) {
    const int b = base + tid;
    int n = 0, pk = 0;
    if (b < a.B) {
      const int len = a.cu[b + 1] - a.cu[b];
      if (len < 0) err = 1;
      n = len > 0 ? (len + kPfRows - 1) / kPfRows : 0;
      pk = len > 0 ? (len + kPfKeys - 1) / kPfKeys * kPfKeys : 0;
    }
    int it = n, ip = pk;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, it, o), z = __shfl_up_sync(0xffffffffu, ip, o);
      if (lane >= o) {
        it += y;
        ip += z;
      }
    }
    if (lane == 31) {
      s_wsum[0][wid] = it;
      s_wsum[1][wid] = ip;
    }
    __syncthreads();
    int bt = 0, tt = 0, bp = 0, tp = 0;
#pragma unroll
    for (int w = 0; w < T / 32; ++w) {
      if (w < wid) {
        bt += s_wsum[0][w];
        bp += s_wsum[1][w];
      }
      tt += s_wsum[0][w];
      tp += s_wsum[1][w];
    }
    if (b < a.B) {
      cu_tiles[b] = carry_t + bt + it - n;
      pcu[b] = carry_p + bp + ip - pk;
    }
    carry_t += tt;
    carry_p += tp;
    __syncthreads();
  }
  err = __syncthreads_or(err);
  if (tid == 0) {
    if (err && report) set_error(a.status, UMIM_ERR_INVALID_ARG);
    cu_tiles[a.B] = err ? 0 : carry_t;
    pcu[a.B] = err ? 0 : carry_p;
  }
  __syncthreads();
}

// more than kPfSmemBatch sequences: the prefix sums in a kernel of its own (one block)
__global__ void __launch_bounds__(kPfPlanThreads) prefill_plan_kernel(PfArgs a) {
  griddep_wait();
  pf_prefix<kPfPlanThreads>(a, a.cu_tiles, a.pcu, true);
}

// last index b in [0, B) with key[b] <= x
__device__ __forceinline__ int pf_find(const int32_t *key, int B, int x) {
  int lo = 0, hi = B;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (key[mid] <= x) lo = mid;
    else hi = mid;
  }
  return lo;
}

// V^T: vt[g][d][pcu[b] + t] = v[cu[b] + t][g][d] for t < len_b, 0 up to the
// next multiple of 64.  CTAs walk the (64 padded keys, KV head) blocks, each
// through a shared-memory tile.  The blocks of KV head 0 whose keys start a
// query tile also write that tile's record.  With PLAN the CTAs derive the
// prefix sums themselves, in shared memory, once each: as a kernel before this
// one they cost a launch and a trip through memory (five short prompts: 12.7 ->
// 10.0 us; 64 of 1500 rows: both kernels 80 -> 71 us).
template <int D, bool PLAN>
__global__ void __launch_bounds__(kPfVtThreads) vt_kernel(PfArgs a) {
  griddep_wait();
  __shared__ uint32_t tile[kPfKeys][D / 2 + 1];   // bf16 pairs, padded against bank conflicts
  extern __shared__ int32_t s_plan[];             // PLAN: the prefix sums, [B + 1] each
  const int32_t *cu_tiles = a.cu_tiles, *pcu = a.pcu;
  if (PLAN) {
    pf_prefix<kPfVtThreads>(a, s_plan, s_plan + a.B + 1, blockIdx.x == 0);
    cu_tiles = s_plan;
    pcu = s_plan + a.B + 1;
    if (blockIdx.x == 0 && threadIdx.x == 0) a.cu_tiles[a.B] = cu_tiles[a.B];   // for the attention kernel
  }
  const int blocks = pcu[a.B] / kPfKeys * a.Hkv;
  constexpr int CPR = D / 8;                             // 16-byte chunks per key row
  constexpr int NU = kPfKeys * CPR / kPfVtThreads;       // chunks a thread loads
  uint4 u[NU];
  // a block's rows; the next block's are loaded while this one is written
  auto load = [&](int it) {
    const int k0 = it / a.Hkv * kPfKeys, g = it % a.Hkv;
    const int b = pf_find(pcu, a.B, k0);
    const int first = a.cu[b], len = a.cu[b + 1] - first;
    const int t0 = k0 - pcu[b];
    if (g == 0 && threadIdx.x == 0 && t0 % kPfRows == 0)
      a.tiles[cu_tiles[b] + t0 / kPfRows] = make_int4(first, len, t0, pcu[b]);
#pragma unroll
    for (int k = 0; k < NU; ++k) {
      const int i = threadIdx.x + k * kPfVtThreads, r = i / CPR, c = i % CPR;
      u[k] = make_uint4(0, 0, 0, 0);
      if (t0 + r < len)
        u[k] = __ldg(reinterpret_cast<const uint4 *>(a.v + ((int64_t)(first + t0 + r) * a.Hkv + g) * D) + c);
    }
  };
  bool too_big = false;
  if ((int)blockIdx.x < blocks) load(blockIdx.x);
  for (int it = blockIdx.x; it < blocks; it += gridDim.x) {
    const int k0 = it / a.Hkv * kPfKeys, g = it % a.Hkv;
#pragma unroll
    for (int k = 0; k < NU; ++k) {
      const int i = threadIdx.x + k * kPfVtThreads, r = i / CPR, c = i % CPR;
      tile[r][4 * c] = u[k].x;
      tile[r][4 * c + 1] = u[k].y;
      tile[r][4 * c + 2] = u[k].z;
      tile[r][4 * c + 3] = u[k].w;
    }
    __syncthreads();
    if (it + (int)gridDim.x < blocks) load(it + gridDim.x);
    // each thread writes 8 keys of one d row (16 bytes), converted to fp16
    for (int i = threadIdx.x; i < D * (kPfKeys / 8); i += kPfVtThreads) {
      const int d = i / (kPfKeys / 8), c = i % (kPfKeys / 8);
      uint32_t w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t x0 = tile[8 * c + 2 * j][d >> 1], x1 = tile[8 * c + 2 * j + 1][d >> 1];
        const float f0 = __uint_as_float((d & 1) ? (x0 & 0xffff0000u) : (x0 << 16));
        const float f1 = __uint_as_float((d & 1) ? (x1 & 0xffff0000u) : (x1 << 16));
        too_big |= !(fabsf(f0) < 65504.f) || !(fabsf(f1) < 65504.f);
        const __half2 hh = __floats2half2_rn(f0, f1);
        w[j] = *reinterpret_cast<const uint32_t *>(&hh);
      }
      *reinterpret_cast<uint4 *>(a.vt + ((int64_t)g * D + d) * a.Tp + k0 + 8 * c) =
          make_uint4(w[0], w[1], w[2], w[3]);
    }
    __syncthreads();   // the tile is filled again
  }
  if (too_big) set_error(a.status, UMIM_ERR_UNSUPPORTED);   // |v| outside fp16's range (or not finite)
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0, int c1, int c2,
                                            uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

// 32 lanes x 64 consecutive fp32 columns from tensor memory in one load
// (thread i: row lane base + i), waited for inside the same statement so no
// register is read before it has landed
__device__ __forceinline__ void tmem_ld_32x32b_x64(uint32_t taddr, float (&v)[64]) {
  uint32_t r[64];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 64; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 lanes x 32 consecutive fp32 columns back into tensor memory (thread i: row lane base + i)
__device__ __forceinline__ void tmem_st_32x32b_x32(uint32_t taddr, const float (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
      "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]), "f"(v[16]), "f"(v[17]), "f"(v[18]),
      "f"(v[19]), "f"(v[20]), "f"(v[21]), "f"(v[22]), "f"(v[23]), "f"(v[24]), "f"(v[25]), "f"(v[26]), "f"(v[27]),
      "f"(v[28]), "f"(v[29]), "f"(v[30]), "f"(v[31])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// the hardware's approximate base-2 exponential (PTX ex2.approx.ftz: relative
// error about 2^-22, -inf -> 0)
__device__ __forceinline__ float max3f(float x, float y, float z) {   // max of three, one instruction
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(x), "f"(y), "f"(z));
  return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&p);
}

// D[tmem] (+)= A[tmem] * B[smem]^T (kind::f16): A's rows in the 128 lanes,
// two 16-bit values of consecutive K per 32-bit column
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// shared-memory layout of the attention kernel (bytes, every piece 1024-aligned)
template <int D>
struct PfSmem {
  static constexpr int kQ = kPfRows * D * 2;              // Q of one head: D/64 atoms of [128 rows][128 B]
  static constexpr int kK = kPfKeys * D * 2;              // K tile: D/64 atoms of [64 keys][128 B]
  static constexpr int kV = D * kPfKeys * 2;              // V^T tile: [D rows][128 B]
  static constexpr int kKoff = kQ;
  static constexpr int kVoff = kKoff + kPfKStages * kK;
  static constexpr int kOoff = kVoff + kPfVStages * kV;   // per softmax warp: 32 rows x 32 columns of the output
  static constexpr int kTotal = kOoff + 4 * 2048;
};

template <int D>
__global__ void __launch_bounds__(kPfThreads, 2)
    prefill_tc_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                      const __grid_constant__ CUtensorMap vt_map, PfArgs a) {
  using L = PfSmem<D>;
  constexpr int DA = D / 64;   // 64-wide atoms along the head dimension
  extern __shared__ __align__(1024) uint8_t pf_raw[];
  __shared__ __align__(8) uint64_t q_full, q_empty, k_full[kPfKStages], k_empty[kPfKStages], v_full[kPfVStages],
      v_empty[kPfVStages], s_full[2], s_empty[2], p_full[2], p_empty, o_done, o_free, mma_done[2];
  __shared__ uint32_t tmem_base;
  __shared__ int s_abort;
  __shared__ int4 s_rec[4];   // the records of the CTA's units k & 3 (written by the copy thread before it loads Q)
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(pf_raw) + 1023) & ~uintptr_t(1023));
  const int warp = warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    s_abort = 0;
    mbar_init(&q_full, 1);
    mbar_init(&q_empty, 1);    // committed once a unit's S products have read Q
    for (int s = 0; s < kPfKStages; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);
    }
    for (int s = 0; s < kPfVStages; ++s) {
      mbar_init(&v_full[s], 1);
      mbar_init(&v_empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s_full[i], 1);
      mbar_init(&s_empty[i], 1);   // committed once the P V product that read P from it is done
      mbar_init(&p_full[i], 4);    // P ready, by tile parity (the four softmax warps)
    }
    mbar_init(&p_empty, 1);       // a P V product has landed
    mbar_init(&o_done, 1);        // a unit's products have landed in O
    mbar_init(&o_free, 4);        // a unit's epilogue has read O (the four softmax warps)
    mbar_init(&mma_done[0], 1);
    mbar_init(&mma_done[1], 1);
    fence_mbar_init();
    prefetch_tensormap(&q_map);
    prefetch_tensormap(&k_map);
    prefetch_tensormap(&vt_map);
  }
  if (warp == 1) {
    tmem_alloc(&tmem_base, kPfTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  griddep_wait();

  // Work units: (query tile, query head), the tiles heaviest first (a
  // sequence's last tiles) and the heads of a tile consecutive, so CTAs that
  // run at the same time share K and V tiles in L2.  CTA c takes units c,
  // c + G, c + 2G, ...; every barrier keeps counting across units (tile
  // counters run over the CTA's units).
  const int total = a.cu_tiles[a.B];
  const int n_units = total * a.Hq;
  const int G = (int)gridDim.x;
  struct Unit {
    int s0, len, q0, h, g, n_kv, kbase;
  };
  // The copy thread reads a unit's record a unit ahead and leaves it in s_rec; the
  // others find it there once the unit's first barrier has let them through (it
  // loads Q of unit k + 1 only when unit k's S products are done, so at most
  // units k - 1 to k + 1 are in use at once).  Looked up by every warp when it
  // was needed, with a binary search over the sequences, a unit began 1000 to
  // 5000 cycles late.  With this and the turned stores of the epilogue (64 x 1500
  // rows, 32/8 heads, D = 128) the call went from 1300 to 1238 us.
  auto unit_of = [&](int u, int4 rec) {   // a sequence's last (heaviest) tiles come first
    Unit w;
    w.s0 = rec.x;
    w.len = rec.y;
    w.q0 = rec.z;
    w.kbase = rec.w;
    w.h = u % a.Hq;
    w.g = w.h / a.G;
    w.n_kv = (min(w.q0 + kPfRows, w.len) + kPfKeys - 1) / kPfKeys;   // causal key tiles
    return w;
  };
  // a warp that gave up tells the others, so that no wait is left to time out on its own
  auto aborted = [&]() { return *reinterpret_cast<volatile int *>(&s_abort) != 0; };
  auto give_up = [&]() {
    set_error(a.status, UMIM_ERR_TIMEOUT);
    *reinterpret_cast<volatile int *>(&s_abort) = 1;
  };

  if (warp == 0) {
    if (elect_one()) {
      const uint64_t pol_q = policy_evict_first(), pol_kv = policy_evict_last();
      // K runs kPfKStages - 1 tiles ahead of V^T: a K load never waits behind
      // the P V product that frees a V^T stage
      constexpr int kLead = kPfKStages - 1;
      int nk = 0, nv = 0, nq = 0;   // K and V^T tiles (ring positions) and Q tiles loaded so far
      bool ok = true;
      int k_unit = 0;
      auto record = [&](int u) {
        return u < n_units ? a.tiles[total - 1 - u / a.Hq] : make_int4(0, 0, 0, 0);
      };
      int4 rec = record((int)blockIdx.x);
      for (int u = (int)blockIdx.x; u < n_units && ok; u += G, ++k_unit) {
        const Unit w = unit_of(u, rec);
        const int4 here = rec;
        rec = record(u + G);
        // the unit's last K row and V^T column (a TMA copy past the end of
        // its tensor reads zeros, so these checks only record)
        (void)in_bounds((int64_t)w.s0 + (w.n_kv - 1) * kPfKeys, a.T, a.status, kSitePrefillKvRow);
        (void)in_bounds(w.kbase + (int64_t)(w.n_kv - 1) * kPfKeys, a.Tp, a.status, kSitePrefillKvRow);
        // Q of the previous unit has been read by its last S product
        if (k_unit > 0 && (aborted() || !mbar_wait(&q_empty, (uint32_t)(k_unit - 1) & 1u))) {
          ok = false;
          break;
        }
        s_rec[k_unit & 3] = here;
        mbar_arrive_expect_tx(&q_full, L::kQ);
#pragma unroll
        for (int d = 0; d < DA; ++d)
          tma_load_3d(smem + d * (kPfRows * 128), &q_map, &q_full, d * 64, w.h, w.s0 + w.q0, pol_q);
        ++nq;
        for (int i = 0; i < w.n_kv + kLead && ok; ++i) {
          if (i < w.n_kv) {
            const int s = nk % kPfKStages;
            if (aborted() || !mbar_wait(&k_empty[s], ((nk / kPfKStages) & 1) ^ 1)) {
              ok = false;
              break;
            }
            mbar_arrive_expect_tx(&k_full[s], L::kK);
#pragma unroll
            for (int d = 0; d < DA; ++d)
              tma_load_3d(smem + L::kKoff + s * L::kK + d * (kPfKeys * 128), &k_map, &k_full[s], d * 64, w.g,
                          w.s0 + i * kPfKeys, pol_kv);
            ++nk;
          }
          const int j = i - kLead;
          if (j >= 0 && j < w.n_kv) {
            const int s = nv % kPfVStages;
            if (aborted() || !mbar_wait(&v_empty[s], ((nv / kPfVStages) & 1) ^ 1)) {
              ok = false;
              break;
            }
            mbar_arrive_expect_tx(&v_full[s], L::kV);
            tma_load_3d(smem + L::kVoff + s * L::kV, &vt_map, &v_full[s], w.kbase + j * kPfKeys, 0, w.g, pol_kv);
            ++nv;
          }
        }
      }
      if (!ok) give_up();
      // copies still in flight when a consumer gave up: wait for them (bounded)
      for (int i = max(0, nk - kPfKStages); i < nk; ++i)
        mbar_wait_for(&k_full[i % kPfKStages], (i / kPfKStages) & 1, kWaitLimitNs);
      for (int i = max(0, nv - kPfVStages); i < nv; ++i)
        mbar_wait_for(&v_full[i % kPfVStages], (i / kPfVStages) & 1, kWaitLimitNs);
      if (nq > 0) mbar_wait_for(&q_full, (uint32_t)(nq - 1) & 1u, kWaitLimitNs);
    }
  } else if (warp == 1) {
    // ---- S = Q K(i)^T into S buffer (tile counter) & 1, once the P V product that read that buffer is done ----
    if (elect_one()) {
      constexpr uint32_t idesc_s = idesc_f32acc(kPfRows, kPfKeys, false);
      bool ok = true;
      int nt = 0, k_unit = 0;   // tiles and units so far
      for (int u = (int)blockIdx.x; u < n_units && ok; u += G, ++k_unit) {
        if (aborted() || !mbar_wait(&q_full, (uint32_t)k_unit & 1u)) {
          ok = false;
          break;
        }
        const Unit w = unit_of(u, s_rec[k_unit & 3]);
        tc_fence_after();
        const uint32_t q_base = smem_u32(smem);
        for (int i = 0; i < w.n_kv; ++i, ++nt) {
          const int s = nt % kPfKStages, sb = nt & 1;
          if (aborted() || !mbar_wait(&k_full[s], (nt / kPfKStages) & 1) ||
              !mbar_wait(&s_empty[sb], ((nt >> 1) & 1) ^ 1)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t k_base = smem_u32(smem + L::kKoff + s * L::kK);
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint32_t off = (kk & 3) * 32;
            tc_mma_bf16(tmem + sb * kPfKeys, sw128_kmajor_desc(q_base + (kk >> 2) * (kPfRows * 128) + off),
                        sw128_kmajor_desc(k_base + (kk >> 2) * (kPfKeys * 128) + off), idesc_s, kk != 0 ? 1u : 0u);
          }
          tc_commit(&s_full[sb]);
          tc_commit(&k_empty[s]);
        }
        if (ok) tc_commit(&q_empty);   // the unit's S products have read Q
      }
      if (!ok) give_up();
      // every product this thread issued has finished before tensor memory is released
      tc_commit(&mma_done[0]);
      mbar_wait_for(&mma_done[0], 0, kWaitLimitNs);
    }
  } else if (warp == 6) {
    // ---- O += P V(i) (fp16 operands, P from tensor memory), as soon as P(i) is ready; frees V(i)'s
    // stage and S(i)'s buffer.  A separate issuing thread, so that a P V product never waits behind
    // an S product that waits for the previous P V.  A unit's first product overwrites O once the
    // previous unit's epilogue has read it ----
    if (elect_one()) {
      constexpr uint32_t idesc_o = idesc_f32acc(kPfRows, D, true);   // P and V^T in fp16
      bool ok = true;
      int nt = 0, k_unit = 0;
      for (int u = (int)blockIdx.x; u < n_units && ok; u += G, ++k_unit) {
        if ((k_unit > 0 && (aborted() || !mbar_wait(&o_free, (uint32_t)(k_unit - 1) & 1u))) || aborted() ||
            !mbar_wait(&p_full[nt & 1], (nt >> 1) & 1)) {   // the unit's first P: its record is there
          ok = false;
          break;
        }
        const Unit w = unit_of(u, s_rec[k_unit & 3]);
        for (int i = 0; i < w.n_kv; ++i, ++nt) {
          const int s = nt % kPfVStages, sb = nt & 1;
          if (aborted() || !mbar_wait(&v_full[s], (nt / kPfVStages) & 1) ||
              !mbar_wait(&p_full[sb], (nt >> 1) & 1)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t v_base = smem_u32(smem + L::kVoff + s * L::kV);
          const uint32_t p_tmem = tmem + sb * kPfKeys;   // P(i) sits where S(i) was
#pragma unroll
          for (int kk = 0; kk < kPfKeys / 16; ++kk)
            tc_mma_ts(tmem + 128, p_tmem + kk * 8, sw128_kmajor_desc(v_base + kk * 32), idesc_o,
                      (i | kk) != 0 ? 1u : 0u);
          tc_commit(&p_empty);
          tc_commit(&s_empty[sb]);
          tc_commit(&v_empty[s]);
        }
        if (ok) tc_commit(&o_done);   // the unit's products have landed in O
      }
      if (!ok) give_up();
      tc_commit(&mma_done[1]);
      mbar_wait_for(&mma_done[1], 0, kWaitLimitNs);
    }
  } else if (warp >= 2 && warp < 6) {
    // ---- softmax and epilogue: four warps, thread = query row ----
    const int quad = warp & 3;                 // tensor-memory lanes this warp may access
    const int r = quad * 32 + lane;            // query row within the tile
    const uint32_t t_s = tmem + ((uint32_t)(quad * 32) << 16);   // this row's S buffers
    const uint32_t t_o = t_s + 128;                                // and O
    const float sl2 = a.scale_log2;
    bool ok = true;
    // every lane waits (each needs the acquire), the warp goes on only if all saw the phase:
    // the .sync.aligned tensor-memory instructions below need the whole warp
    auto wwait = [&](uint64_t *m, uint32_t parity) {
      return __all_sync(0xffffffffu, !aborted() && mbar_wait(m, parity)) != 0;
    };
    // The output of a unit: O / l once its last product has landed, then O is
    // free for the next unit.  Thread = row holds 32 columns at a time; the warp
    // turns them through shared memory so that a store writes 64 contiguous
    // bytes of eight rows (one row per lane took 16-byte pieces of 32 rows).
    auto epilogue = [&](const Unit &w, float l_run, int k) -> bool {   // of the CTA's k-th unit
      if (!wwait(&o_done, (uint32_t)k & 1u)) return false;
      tc_fence_after();
      uint8_t *stage = smem + L::kOoff + (warp - 2) * 2048;
      const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
      const int first = w.q0 + quad * 32;        // position of the warp's first row
      __nv_bfloat16 *obase = a.out + (((int64_t)w.s0 + first) * a.Hq + w.h) * D;
#pragma unroll 1
      for (int c = 0; c < D / 32; ++c) {
        float o[32];
        tmem_ld_32x32b_x32(t_o + c * 32, o);
        __syncwarp();   // the lanes have read the columns before
#pragma unroll
        for (int e = 0; e < 4; ++e)
          *reinterpret_cast<uint4 *>(stage + lane * 64 + ((e ^ ((lane >> 1) & 3)) << 4)) =
              make_uint4(pack_bf16x2(o[8 * e] * inv, o[8 * e + 1] * inv),
                         pack_bf16x2(o[8 * e + 2] * inv, o[8 * e + 3] * inv),
                         pack_bf16x2(o[8 * e + 4] * inv, o[8 * e + 5] * inv),
                         pack_bf16x2(o[8 * e + 6] * inv, o[8 * e + 7] * inv));
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int row = k * 8 + (lane >> 2), ch = lane & 3;
          const uint4 x = *reinterpret_cast<const uint4 *>(stage + row * 64 + ((ch ^ ((row >> 1) & 3)) << 4));
          if (first + row < w.len && in_bounds((int64_t)w.s0 + first + row, a.T, a.status, kSitePrefillOutRow))
            *reinterpret_cast<uint4 *>(obase + (int64_t)row * a.Hq * D + c * 32 + ch * 8) = x;
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&o_free);
      return true;
    };
    int nt = 0, k_unit = 0;
    for (; (int)blockIdx.x + k_unit * G < n_units && ok; ++k_unit) {
      if (!wwait(&s_full[nt & 1], (nt >> 1) & 1)) {   // the unit's first S: its record is there
        ok = false;
        break;
      }
      const Unit w = unit_of((int)blockIdx.x + k_unit * G, s_rec[k_unit & 3]);
      const int qpos = w.q0 + r;                  // position within the sequence
      const int kmax = min(qpos, w.len - 1);      // last key this row sees
      float m_run = -INFINITY, l_run = 0.f;       // running max (log2 units, moved in steps > 8) and row sum
      for (int j = 0; j < w.n_kv; ++j, ++nt) {
        const int sb = nt & 1;
        if (!wwait(&s_full[sb], (nt >> 1) & 1)) {
          ok = false;
          break;
        }
        tc_fence_after();
        float s[kPfKeys];
        tmem_ld_32x32b_x64(t_s + sb * kPfKeys, s);
        const int k0 = j * kPfKeys;
        if (k0 + kPfKeys - 1 > kmax) {   // the diagonal tile (or a row past the sequence)
#pragma unroll
          for (int c = 0; c < kPfKeys; ++c) s[c] = (k0 + c <= kmax) ? s[c] : -INFINITY;
        }
        float m4[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
        for (int c = 4; c < kPfKeys; c += 2) m4[(c >> 1) & 3] = max3f(m4[(c >> 1) & 3], s[c], s[c + 1]);
        const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * sl2;
        // move the running max only when it grows by more than 2^8
        const bool grow = mx > m_run + 8.f;
        float alpha = 1.f;
        if (grow) {
          alpha = (m_run == -INFINITY) ? 0.f : ex2_approx(m_run - mx);
          m_run = mx;
          l_run *= alpha;
        }
        const float nm = (m_run == -INFINITY) ? 0.f : -m_run;
        // exp2(s * scale - max) and the row sum, two columns per packed instruction
        const float2 sl2x2 = make_float2(sl2, sl2), nm2 = make_float2(nm, nm);
        float2 la = make_float2(0.f, 0.f), lb = la;
        float pk[kPfKeys / 2];   // P in fp16 pairs (P <= 2^8)
#pragma unroll
        for (int c = 0; c < kPfKeys; c += 2) {
          const float2 x = __ffma2_rn(make_float2(s[c], s[c + 1]), sl2x2, nm2);
          const float2 e = make_float2(ex2_approx(x.x), ex2_approx(x.y));   // masked (-inf): 0
          if (c & 2) lb = __fadd2_rn(lb, e);
          else la = __fadd2_rn(la, e);
          const __half2 hh = __floats2half2_rn(e.x, e.y);
          pk[c / 2] = __uint_as_float(*reinterpret_cast<const uint32_t *>(&hh));
        }
        const float2 lab = __fadd2_rn(la, lb);
        l_run += lab.x + lab.y;
        // O is rescaled only once the product of tile j - 1 has landed
        if (j > 0 && __any_sync(0xffffffffu, grow)) {
          if (!wwait(&p_empty, (uint32_t)(nt - 1) & 1u)) {
            ok = false;
            break;
          }
          tc_fence_after();
#pragma unroll 1
          for (int c = 0; c < D / 32; ++c) {
            float o[32];
            tmem_ld_32x32b_x32(t_o + c * 32, o);
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] *= alpha;
            tmem_st_32x32b_x32(t_o + c * 32, o);
          }
          tc_fence_before();
        }
        // P(j) over S(j)'s columns (this thread has read them), for the P V product
        tmem_st_32x32b_x32(t_s + sb * kPfKeys, pk);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[sb]);
      }
      if (ok) ok = epilogue(w, l_run, k_unit);
    }
    if (!ok) give_up();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kPfTmemCols);
  }
}

// ---------------------------------------------------------------------------
// Two heads at a time
// ---------------------------------------------------------------------------
// An even group's heads h, h + 1 read the same K and V: one CTA per SM walks
// units of (query tile, pair of heads), each head in a slot of its own (Q, S, O
// and four softmax warps), over 128-key tiles that are loaded once for both.
// What bounds the one-head kernel above is shared memory: per 128 x 64 tile it
// copies K and V^T in (256 cycles at 128 B a cycle) and its S product reads all
// of Q beside 64 keys (384), its P V product V^T (128), for 512 cycles of tensor
// cores.  Here a slot's 128 x 128 tile takes 256 + 512 + 256 for 1024.
// Tensor memory: S of the slots at columns 0 and 128 (P over it), O at 256 and
// 384, all 512, so S is not double-buffered: a slot's P V and next S products
// take the tensor cores while the other slot's softmax runs.  A steady pair of
// tiles takes 2650 cycles: 4 x 512 of products, twice the 220 between the end of
// a P V product and the S product that waits for it, and the softmax's tail; a
// unit's diagonal masks and epilogue cost 2000 more.
// The call, 64 x 1500 rows, 32/8 heads, D = 128: 1206 -> 1060 us; 48 x 1500 rows,
// 8/2 heads, D = 64: 196 -> 178.
constexpr int kPpTile = 128;       // keys per K / V^T tile (the S MMA's N); V^T is loaded by halves
constexpr int kPpStages = 2;       // K ring and V^T ring
constexpr int kPpThreads = 352;    // warp 0 TMA, warps 1-2 a slot's products each, warps 3-6 and 7-10 a slot's
                                   // softmax each (thread = query row)
constexpr uint32_t kPpTmemCols = 512;

__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap *map, int c0, int c1, int c2) {   // into L2
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(c0), "r"(c1), "r"(c2)
               : "memory");
}

__device__ __forceinline__ void tma_store_3d(const CUtensorMap *map, const void *src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(src))
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// 32 lanes x 128 consecutive fp32 columns (as the x64 load above)
__device__ __forceinline__ void tmem_ld_32x32b_x128(uint32_t taddr, float (&v)[128]) {
  uint32_t r[128];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x128.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63, %64, %65, %66, %67, %68, %69, %70, %71, %72, %73, %74, %75, %76, %77, %78, %79, %80, %81, %82, %83, %84, %85, %86, %87, %88, %89, %90, %91, %92, %93, %94, %95, %96, %97, %98, %99, %100, %101, %102, %103, %104, %105, %106, %107, %108, %109, %110, %111, %112, %113, %114, %115, %116, %117, %118, %119, %120, %121, %122, %123, %124, %125, %126, %127}, [%128];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63]), "=r"(r[64]), "=r"(r[65]), "=r"(r[66]), "=r"(r[67]), "=r"(r[68]), "=r"(r[69]), "=r"(r[70]), "=r"(r[71]), "=r"(r[72]), "=r"(r[73]), "=r"(r[74]), "=r"(r[75]), "=r"(r[76]), "=r"(r[77]), "=r"(r[78]), "=r"(r[79]), "=r"(r[80]), "=r"(r[81]), "=r"(r[82]), "=r"(r[83]), "=r"(r[84]), "=r"(r[85]), "=r"(r[86]), "=r"(r[87]), "=r"(r[88]), "=r"(r[89]), "=r"(r[90]), "=r"(r[91]), "=r"(r[92]), "=r"(r[93]), "=r"(r[94]), "=r"(r[95]), "=r"(r[96]), "=r"(r[97]), "=r"(r[98]), "=r"(r[99]), "=r"(r[100]), "=r"(r[101]), "=r"(r[102]), "=r"(r[103]), "=r"(r[104]), "=r"(r[105]), "=r"(r[106]), "=r"(r[107]), "=r"(r[108]), "=r"(r[109]), "=r"(r[110]), "=r"(r[111]), "=r"(r[112]), "=r"(r[113]), "=r"(r[114]), "=r"(r[115]), "=r"(r[116]), "=r"(r[117]), "=r"(r[118]), "=r"(r[119]), "=r"(r[120]), "=r"(r[121]), "=r"(r[122]), "=r"(r[123]), "=r"(r[124]), "=r"(r[125]), "=r"(r[126]), "=r"(r[127])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 128; ++i) v[i] = __uint_as_float(r[i]);
}

// shared-memory layout (bytes, every piece 1024-aligned)
template <int D>
struct PpSmem {
  static constexpr int kQ = kPfRows * D * 2;              // Q of a slot: D/64 atoms of [128 rows][128 B]
  static constexpr int kK = kPpTile * D * 2;              // K tile: D/64 atoms of [128 keys][128 B]
  static constexpr int kVh = D * kPfKeys * 2;             // half a V^T tile: [D rows][128 B]
  static constexpr int kV = 2 * kVh;
  static constexpr int kKoff = 2 * kQ;
  static constexpr int kVoff = kKoff + kPpStages * kK;
  static constexpr int kOoff = kVoff + kPpStages * kV;    // per softmax warp: 32 rows x 64 columns of the output
  static constexpr int kTotal = kOoff + 8 * 4096;
};

template <int D>
__global__ void __launch_bounds__(kPpThreads, 1)
    prefill_pair_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map,
                        const __grid_constant__ CUtensorMap vt_map, const __grid_constant__ CUtensorMap out_map,
                        PfArgs a) {
  using L = PpSmem<D>;
  constexpr int DA = D / 64;   // 64-wide atoms along the head dimension
  extern __shared__ __align__(1024) uint8_t pf_raw[];
  __shared__ __align__(8) uint64_t q_full[2], q_empty[2], k_full[kPpStages], k_empty[kPpStages], v_full[kPpStages],
      v_empty[kPpStages], s_full[2], p_full[2][2], pv_done[2], o_free[2], turn[2], mma_done[2];
  __shared__ uint32_t tmem_base;
  __shared__ int s_abort;
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(pf_raw) + 1023) & ~uintptr_t(1023));
  const int warp = warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    s_abort = 0;
    for (int s = 0; s < kPpStages; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 2);   // read by both slots' products
      mbar_init(&v_full[s], 1);
      mbar_init(&v_empty[s], 2);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(&q_full[t], 1);
      mbar_init(&q_empty[t], 1);     // a unit's S products have read the slot's Q
      mbar_init(&s_full[t], 1);
      mbar_init(&p_full[t][0], 4);   // keys 0-63 of P ready (the slot's four softmax warps)
      mbar_init(&p_full[t][1], 4);   // keys 64-127
      mbar_init(&pv_done[t], 1);     // a tile's P V product has landed
      mbar_init(&o_free[t], 4);      // a unit's epilogue has read O (four softmax warps)
      mbar_init(&turn[t], 1);        // the other slot's products are issued
      mbar_init(&mma_done[t], 1);
    }
    fence_mbar_init();
    prefetch_tensormap(&q_map);
    prefetch_tensormap(&k_map);
    prefetch_tensormap(&vt_map);
    prefetch_tensormap(&out_map);
  }
  if (warp == 1) {
    tmem_alloc(&tmem_base, kPpTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base;
  griddep_wait();

  // Units in the order of the one-head kernel's: the tiles heaviest first, the
  // pairs of a tile consecutive.  The unit number is kept in mixed radix (query
  // tile, KV head, pair within the group): divided anew, the next unit's number
  // kept its first products waiting for 800 cycles.
  const int total = a.cu_tiles[a.B];
  struct Unit {
    int tile, g, p;
  };
  auto unit_of = [&](int u) {
    const int pairs = a.G / 2, tile = u / (a.Hkv * pairs), x = u - tile * (a.Hkv * pairs), g = x / pairs;
    return Unit{tile, g, x - g * pairs};
  };
  const Unit first = unit_of((int)blockIdx.x), step = unit_of((int)gridDim.x);
  auto next_of = [&](Unit u) {
    u.p += step.p;
    u.g += step.g;
    u.tile += step.tile;
    if (u.p >= a.G / 2) {
      u.p -= a.G / 2;
      ++u.g;
    }
    if (u.g >= a.Hkv) {
      u.g -= a.Hkv;
      ++u.tile;
    }
    return u;
  };
  // A unit's record is read a unit ahead (past the last unit: record 0, not
  // used).  Volatile: the compiler would move the load to the record's use.
  auto record = [&](const Unit &u) {
    int4 v;
    const int4 *p = a.tiles + max(total - 1 - u.tile, 0);
    asm volatile("ld.global.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
  };
  struct Tile {
    int s0, len, q0, kbase;
    int kend, n;   // keys the unit reads (causal) and tiles of them
  };
  auto tile_of = [&](int4 rec) {
    Tile w;
    w.s0 = rec.x;
    w.len = rec.y;
    w.q0 = rec.z;
    w.kbase = rec.w;
    w.kend = min(w.q0 + kPfRows, w.len);
    w.n = (w.kend + kPpTile - 1) / kPpTile;
    return w;
  };
  auto head_of = [&](const Unit &u, int t) { return u.g * a.G + 2 * u.p + t; };
  // a warp that gave up tells the others, so that no wait is left to time out on its own
  auto aborted = [&]() { return *reinterpret_cast<volatile int *>(&s_abort) != 0; };
  auto give_up = [&]() {
    set_error(a.status, UMIM_ERR_TIMEOUT);
    *reinterpret_cast<volatile int *>(&s_abort) = 1;
  };

  if (warp == 0) {
    if (elect_one()) {
      const uint64_t pol_q = policy_evict_first(), pol_kv = policy_evict_last();
      int nk = 0, nv = 0, nq[2] = {0, 0};   // K and V^T tiles (ring positions) and the slots' Q loaded so far
      bool ok = true;
      int4 rec = record(first);
      for (Unit u = first, v; u.tile < total && ok; u = v) {
        const Tile w = tile_of(rec);
        v = next_of(u);
        rec = record(v);
        // the unit's last K row and V^T column (a TMA copy past the end of
        // its tensor reads zeros, so these checks only record)
        (void)in_bounds((int64_t)w.s0 + w.kend - 1, a.T, a.status, kSitePrefillKvRow);
        (void)in_bounds(w.kbase + (int64_t)w.kend - 1, a.Tp, a.status, kSitePrefillKvRow);
        // a slot's Q, once the last S product of the slot's unit before has read it
        auto load_q = [&](int t) {
          if (nq[t] > 0 && (aborted() || !mbar_wait(&q_empty[t], (uint32_t)(nq[t] - 1) & 1u))) return false;
          mbar_arrive_expect_tx(&q_full[t], L::kQ);
#pragma unroll
          for (int d = 0; d < DA; ++d)
            tma_load_3d(smem + t * L::kQ + d * (kPfRows * 128), &q_map, &q_full[t], d * 64, head_of(u, t), w.s0 + w.q0,
                        pol_q);
          ++nq[t];
          return true;
        };
        ok = load_q(0);
        // K runs a tile ahead of V^T: a K load never waits behind the P V product that frees a V^T stage
        for (int i = 0; i <= w.n && ok; ++i) {
          if (i < w.n) {
            const int s = nk % kPpStages;
            if (aborted() || !mbar_wait(&k_empty[s], ((nk / kPpStages) & 1) ^ 1)) {
              ok = false;
              break;
            }
            const int halves = w.kend - i * kPpTile > kPfKeys ? 2 : 1;
            mbar_arrive_expect_tx(&k_full[s], L::kK / 2 * halves);
            for (int e = 0; e < halves; ++e)
#pragma unroll
              for (int d = 0; d < DA; ++d)
                tma_load_3d(smem + L::kKoff + s * L::kK + d * (kPpTile * 128) + e * (kPfKeys * 128), &k_map, &k_full[s],
                            d * 64, u.g, w.s0 + i * kPpTile + e * kPfKeys, pol_kv);
            ++nk;
          }
          if (i == 0 && !load_q(1)) {
            ok = false;
            break;
          }
          const int j = i - 1;
          if (j >= 0) {
            const int s = nv % kPpStages;
            if (aborted() || !mbar_wait(&v_empty[s], ((nv / kPpStages) & 1) ^ 1)) {
              ok = false;
              break;
            }
            const int halves = w.kend - j * kPpTile > kPfKeys ? 2 : 1;
            mbar_arrive_expect_tx(&v_full[s], L::kVh * halves);
            for (int e = 0; e < halves; ++e)
              tma_load_3d(smem + L::kVoff + s * L::kV + e * L::kVh, &vt_map, &v_full[s],
                          w.kbase + j * kPpTile + e * kPfKeys, 0, u.g, pol_kv);
            ++nv;
          }
          // the next unit's Q on its way into L2: its load starts when this unit's last S product
          // has read Q, and from HBM it took 3000 cycles, longer than the rest of the unit
          if (i == 1 && v.tile < total)
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
              for (int d = 0; d < DA; ++d) tma_prefetch_3d(&q_map, d * 64, head_of(v, t), rec.x + rec.z);
        }
      }
      if (!ok) give_up();
      // copies still in flight when a consumer gave up: wait for them (bounded)
      for (int i = max(0, nk - kPpStages); i < nk; ++i)
        mbar_wait_for(&k_full[i % kPpStages], (i / kPpStages) & 1, kWaitLimitNs);
      for (int i = max(0, nv - kPpStages); i < nv; ++i)
        mbar_wait_for(&v_full[i % kPpStages], (i / kPpStages) & 1, kWaitLimitNs);
#pragma unroll
      for (int t = 0; t < 2; ++t)
        if (nq[t] > 0) mbar_wait_for(&q_full[t], (uint32_t)(nq[t] - 1) & 1u, kWaitLimitNs);
    }
  } else if (warp <= 2) {
    // ---- the products of slot t, turn by turn: O += P V of a tile as the halves of P
    // become ready, then S = Q K^T of the next (of this unit or the next one) once
    // that P V has landed (P lies over S).  The slots take turns, so that one's
    // softmax runs while the other has the tensor cores; left to themselves both
    // wait for softmax together and then for the tensor cores (3300 cycles a pair
    // of tiles).  A unit's first P V overwrites O once the previous unit's epilogue
    // has read it ----
    const int t = warp - 1;
    if (elect_one()) {
      constexpr uint32_t idesc_s = idesc_f32acc(kPfRows, kPpTile, false), idesc_s1 = idesc_f32acc(kPfRows, kPfKeys, false);
      constexpr uint32_t idesc_o = idesc_f32acc(kPfRows, D, true);   // P and V^T in fp16
      const uint32_t t_s = tmem + t * kPpTile, t_o = tmem + 256 + t * 128;
      const uint64_t q_desc = sw128_kmajor_desc(smem_u32(smem) + t * L::kQ);
      int nt = 0, nu = 0;                  // tiles and units whose S is issued
      int first_of = 0;                    // tile nt - 1 is its unit's first
      bool both = false;                   // and of more than 64 keys
      // P V of tile nt - 1 and, unless that was the last, S of tile nt, the i-th of a unit
      auto take_turn = [&](const Tile &w, int i, bool last) {
        const int sv = (nt + 1) & 1, sk = nt & 1;   // ring stages
        const uint32_t pt = (uint32_t)(nt - 1) & 1u;
        if (nt > 0) {
          if (aborted() || !mbar_wait(&v_full[sv], (uint32_t)(nt - 1) >> 1 & 1u) || !mbar_wait(&p_full[t][0], pt) ||
              (first_of && nu > 1 && !mbar_wait(&o_free[t], (uint32_t)nu & 1u)))
            return false;
        }
        if ((t == 1 || nt > 0) && !mbar_wait(&turn[t], (uint32_t)(nt + t + 1) & 1u)) return false;
        if (nt > 0) {
          const uint64_t v_desc = sw128_kmajor_desc(smem_u32(smem + L::kVoff + sv * L::kV));
          tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < kPfKeys / 16; ++kk)
            tc_mma_ts(t_o, t_s + kk * 8, v_desc + kk * 2, idesc_o, !first_of || kk != 0 ? 1u : 0u);
          if (!mbar_wait(&p_full[t][1], pt)) return false;
          if (both) {
            tc_fence_after();
#pragma unroll
            for (int kk = 0; kk < kPfKeys / 16; ++kk)
              tc_mma_ts(t_o, t_s + kPfKeys / 2 + kk * 8, v_desc + L::kVh / 16 + kk * 2, idesc_o, 1u);
          }
          tc_commit(&pv_done[t]);
        }
        if (last) {
          mbar_arrive(&turn[t ^ 1]);
          return true;
        }
        if (aborted() || !mbar_wait(&k_full[sk], (uint32_t)nt >> 1 & 1u) ||
            (i == 0 && !mbar_wait(&q_full[t], (uint32_t)nu & 1u)) || (nt > 0 && !mbar_wait(&pv_done[t], pt)))
          return false;
        const uint64_t k_desc = sw128_kmajor_desc(smem_u32(smem + L::kKoff + sk * L::kK));
        both = w.kend - i * kPpTile > kPfKeys;   // more than half of the tile's keys
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk)
          tc_mma_bf16(t_s, q_desc + (kk >> 2) * (kPfRows * 8) + (kk & 3) * 2,
                      k_desc + (kk >> 2) * (kPpTile * 8) + (kk & 3) * 2, both ? idesc_s : idesc_s1, kk != 0 ? 1u : 0u);
        tc_commit(&s_full[t]);
        mbar_arrive(&turn[t ^ 1]);
        tc_commit(&k_empty[sk]);
        if (i + 1 == w.n) tc_commit(&q_empty[t]);   // the unit's S products have read Q
        if (nt > 0) tc_commit(&v_empty[sv]);
        first_of = i == 0;
        nu += first_of;
        ++nt;
        return true;
      };
      bool ok = true;
      int4 rec = record(first);
      Tile w{};
      for (Unit u = first; u.tile < total && ok;) {
        w = tile_of(rec);
        u = next_of(u);
        rec = record(u);
        for (int i = 0; i < w.n && ok; ++i) ok = take_turn(w, i, false);
      }
      if (ok && nt > 0) ok = take_turn(w, 0, true);
      if (!ok) give_up();
      // every product this thread issued has finished before tensor memory is released
      tc_commit(&mma_done[t]);
      mbar_wait_for(&mma_done[t], 0, kWaitLimitNs);
    }
  } else {
    // ---- softmax and epilogue of slot t: four warps, thread = query row ----
    const int t = (warp - 3) >> 2;
    const int quad = warp & 3;                 // tensor-memory lanes this warp may access
    const int r = quad * 32 + lane;            // query row within the tile
    const uint32_t t_s = tmem + ((uint32_t)(quad * 32) << 16) + t * kPpTile;          // this row's S
    const uint32_t t_o = tmem + ((uint32_t)(quad * 32) << 16) + 256 + t * 128;        // and O
    const float sl2 = a.scale_log2;
    bool ok = true;
    // every lane waits (each needs the acquire), the warp goes on only if all saw the phase:
    // the .sync.aligned tensor-memory instructions below need the whole warp
    auto wwait = [&](uint64_t *m, uint32_t parity) {
      return __all_sync(0xffffffffu, !aborted() && mbar_wait(m, parity)) != 0;
    };
    // The output of a unit: O / l once its last product has landed, then O is
    // free for the next unit.  Thread = row puts 64 columns at a time into shared
    // memory, from where they are stored by a TMA copy, or by the lanes where the
    // sequence ends among the warp's rows.  (Stores by the lanes held the warp for
    // 2400 cycles a unit, these for 1700.)  A loop, not unrolled: unrolled, with all
    // of O in registers, the call took 5 % longer.
    auto epilogue = [&](const Tile &w, int h, float l_run, uint32_t last) -> bool {   // last: parity of its last tile
      uint8_t *stage = smem + L::kOoff + (warp - 3) * 4096;
      const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
      const int first_row = w.s0 + w.q0 + quad * 32, n_rows = w.len - w.q0 - quad * 32;   // of the warp
      if (!wwait(&pv_done[t], last)) return false;
      tc_fence_after();
#pragma unroll 1
      for (int c = 0; c < D; c += 64) {
        float o[64];
        tmem_ld_32x32b_x64(t_o + c, o);
        // (the elected lane is the same one each time, so these are its own copies)
        if (elect_one()) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the columns before are read
        __syncwarp();
#pragma unroll
        for (int e = 0; e < 8; ++e)   // the layout of the 128-byte swizzle
          *reinterpret_cast<uint4 *>(stage + lane * 128 + ((e ^ (lane & 7)) << 4)) =
              make_uint4(pack_bf16x2(o[8 * e] * inv, o[8 * e + 1] * inv),
                         pack_bf16x2(o[8 * e + 2] * inv, o[8 * e + 3] * inv),
                         pack_bf16x2(o[8 * e + 4] * inv, o[8 * e + 5] * inv),
                         pack_bf16x2(o[8 * e + 6] * inv, o[8 * e + 7] * inv));
        if (n_rows >= 32) {
          fence_proxy_async_smem();
          __syncwarp();
          if (elect_one() && in_bounds((int64_t)first_row + 31, a.T, a.status, kSitePrefillOutRow))
            tma_store_3d(&out_map, stage, c, h, first_row);
        } else {
          __syncwarp();
          for (int k = lane >> 3; k < n_rows; k += 4) {
            const uint4 x = *reinterpret_cast<const uint4 *>(stage + k * 128 + (((lane & 7) ^ (k & 7)) << 4));
            if (in_bounds((int64_t)first_row + k, a.T, a.status, kSitePrefillOutRow))
              *reinterpret_cast<uint4 *>(a.out + (((int64_t)first_row + k) * a.Hq + h) * D + c + (lane & 7) * 8) = x;
          }
          __syncwarp();   // the rows are read before the next columns are written
        }
      }
      tc_fence_before();
      __syncwarp();
      if (elect_one()) mbar_arrive(&o_free[t]);
      return true;
    };
    int nt = 0;
    int4 rec = record(first);
    for (Unit u = first; u.tile < total && ok;) {
      const Tile w = tile_of(rec);
      const int h = head_of(u, t);
      u = next_of(u);
      rec = record(u);
      const int kmax = min(w.q0 + r, w.len - 1);               // last key this row sees
      const int kmax0 = min(w.q0 + quad * 32, w.len - 1);      // and the warp's first row
      float m_run = -INFINITY, l_run = 0.f;       // running max (log2 units, moved in steps > 8) and row sum
      for (int j = 0; j < w.n; ++j, ++nt) {
        if (!wwait(&s_full[t], (uint32_t)nt & 1u)) {
          ok = false;
          break;
        }
        tc_fence_after();
        float s[kPpTile];
        tmem_ld_32x32b_x128(t_s, s);
        const int lim = kmax - j * kPpTile, lim0 = kmax0 - j * kPpTile;
        if (lim0 < kPpTile - 1) {   // the diagonal tile, or the sequence's end in it
#pragma unroll
          for (int x = 0; x < kPpTile; x += 32)
            if (lim0 < x + 31) {
              const uint32_t bits = lim < x ? 0u : ~0u >> max(x + 31 - lim, 0);   // keys this row sees
#pragma unroll
              for (int c = 0; c < 32; ++c) s[x + c] = bits >> c & 1u ? s[x + c] : -INFINITY;
            }
        }
        float m4[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
        for (int c = 4; c < kPpTile; c += 2) m4[(c >> 1) & 3] = max3f(m4[(c >> 1) & 3], s[c], s[c + 1]);
        const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3])) * sl2;
        // move the running max only when it grows by more than 2^8
        const bool grow = mx > m_run + 8.f;
        float alpha = 1.f;
        if (grow) {
          alpha = (m_run == -INFINITY) ? 0.f : ex2_approx(m_run - mx);
          m_run = mx;
          l_run *= alpha;
        }
        const float nm = (m_run == -INFINITY) ? 0.f : -m_run;
        // exp2(s * scale - max) and the row sum, two columns per packed instruction
        const float2 sl2x2 = make_float2(sl2, sl2), nm2 = make_float2(nm, nm);
        float2 la = make_float2(0.f, 0.f), lb = la;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float pk[kPfKeys / 2];   // P in fp16 pairs (P <= 2^8)
#pragma unroll
          for (int c = 0; c < kPfKeys; c += 2) {
            const float2 x = __ffma2_rn(make_float2(s[e * kPfKeys + c], s[e * kPfKeys + c + 1]), sl2x2, nm2);
            const float2 y = make_float2(ex2_approx(x.x), ex2_approx(x.y));   // masked (-inf): 0
            if (c & 2) lb = __fadd2_rn(lb, y);
            else la = __fadd2_rn(la, y);
            const __half2 hh = __floats2half2_rn(y.x, y.y);
            pk[c / 2] = __uint_as_float(*reinterpret_cast<const uint32_t *>(&hh));
          }
          // O is rescaled before the tile's first product (tile j - 1's has landed: S(j) followed it)
          if (e == 0 && j > 0 && __any_sync(0xffffffffu, grow)) {
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {
              float o[32];
              tmem_ld_32x32b_x32(t_o + c * 32, o);
#pragma unroll
              for (int i = 0; i < 32; ++i) o[i] *= alpha;
              tmem_st_32x32b_x32(t_o + c * 32, o);
            }
          }
          // P over S's columns (this thread has read them all), for the P V product
          tmem_st_32x32b_x32(t_s + e * (kPfKeys / 2), pk);
          tc_fence_before();
          __syncwarp();
          if (elect_one()) mbar_arrive(&p_full[t][e]);
        }
        const float2 lab = __fadd2_rn(la, lb);
        l_run += lab.x + lab.y;
      }
      if (ok) ok = epilogue(w, h, l_run, (uint32_t)(nt - 1) & 1u);
    }
    if (elect_one()) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    if (!ok) give_up();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kPpTmemCols);
  }
}

bool encode_3d(EncodeTiledFn enc, CUtensorMap *map, const void *base, uint64_t d0, uint64_t d1, uint64_t d2,
               uint64_t stride1, uint64_t stride2, uint32_t b0, uint32_t b1, uint32_t b2, bool fp16 = false) {
  const cuuint64_t dims[3] = {d0, d1, d2};
  const cuuint64_t strides[2] = {stride1, stride2};
  const cuuint32_t box[3] = {b0, b1, b2};
  const cuuint32_t es[3] = {1, 1, 1};
  return enc(map, fp16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
             const_cast<void *>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// bytes before V^T: the prefix sums and the query tiles' records
size_t pf_plan_bytes(int B, int T) {
  const size_t sums = ((size_t)2 * (B + 1) * sizeof(int32_t) + 15) & ~size_t(15);
  return (sums + ((size_t)T / kPfRows + B) * sizeof(int4) + 1023) & ~size_t(1023);
}

// row length of V^T: room for every sequence padded to 64 keys
int64_t vt_row(int B, int T) { return ((int64_t)T + 63LL * B + 63) / 64 * 64; }

}  // namespace

size_t prefill_attention_workspace_bytes(int B, int T, int Hkv, int D) {
  return pf_plan_bytes(B, T) + (size_t)Hkv * D * vt_row(B, T) * 2;
}

umim_status prefill_attention(const void *q, const void *k, const void *v, int T, int Hq, int Hkv, int D,
                              const int32_t *cu_seqlens, int B, float scale, void *out, void *ws, int32_t *status,
                              cudaStream_t stream, int num_sms) {
  EncodeTiledFn enc = get_encode_tiled();
  if (!enc) return UMIM_ERR_CUDA;
  PfArgs a{};
  a.out = static_cast<__nv_bfloat16 *>(out);
  a.cu = cu_seqlens;
  a.cu_tiles = static_cast<int32_t *>(ws);
  a.pcu = a.cu_tiles + (B + 1);
  a.v = static_cast<const __nv_bfloat16 *>(v);
  a.tiles = reinterpret_cast<int4 *>(static_cast<char *>(ws) +
                                     (((size_t)2 * (B + 1) * sizeof(int32_t) + 15) & ~size_t(15)));
  a.vt = reinterpret_cast<__half *>(static_cast<char *>(ws) + pf_plan_bytes(B, T));
  a.Tp = vt_row(B, T);
  a.B = B;
  a.T = T;
  a.Hq = Hq;
  a.Hkv = Hkv;
  a.G = Hq / Hkv;
  a.scale_log2 = (scale > 0.f ? scale : 1.0f / sqrtf((float)D)) * 1.4426950408889634f;
  a.status = status;
  CUtensorMap qm, km, vm, om;
  if (!encode_3d(enc, &qm, q, D, Hq, T, (uint64_t)D * 2, (uint64_t)Hq * D * 2, 64, 1, kPfRows) ||
      !encode_3d(enc, &km, k, D, Hkv, T, (uint64_t)D * 2, (uint64_t)Hkv * D * 2, 64, 1, kPfKeys) ||
      !encode_3d(enc, &vm, a.vt, a.Tp, D, Hkv, (uint64_t)a.Tp * 2, (uint64_t)D * a.Tp * 2, kPfKeys, D, 1, true))
    return UMIM_ERR_CUDA;
  const bool plan = B <= kPfSmemBatch;
  if (!plan) {
    trace_mark(stream, "prefill.plan");
    if (launch_pdl(prefill_plan_kernel, dim3(1), dim3(kPfPlanThreads), 0, stream, a) != cudaSuccess)
      return UMIM_ERR_CUDA;
  }
  trace_mark(stream, "prefill.v_transpose");
  auto vk = plan ? (D == 128 ? vt_kernel<128, true> : vt_kernel<64, true>)
                 : (D == 128 ? vt_kernel<128, false> : vt_kernel<64, false>);
  const int64_t vt_blocks = a.Tp / kPfKeys * Hkv;
  // eight CTAs an SM are launched: five (D = 128) or six (64) of them are resident by
  // their registers, the others follow as those finish (with six an SM in all, 96 000
  // rows of 8 heads took 82 us, with eight 71)
  const unsigned vt_grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(vt_blocks, 8LL * std::max(num_sms, 1)));
  if (launch_pdl(vk, dim3(vt_grid), dim3(kPfVtThreads), plan ? 2 * sizeof(int32_t) * ((size_t)B + 1) : 0, stream, a) !=
      cudaSuccess)
    return UMIM_ERR_CUDA;
  // Units of the pair kernel, an upper bound (each sequence wastes less than one
  // tile).  It takes the even groups whose units go 3.5 times around the SMs:
  // fewer leave SMs idle, where the one-head kernel has twice the CTAs and half the
  // work in each.  Measured (one-head, pair), 32/8 heads, D = 128: 272 units 43.7,
  // 46.6 us; 528 57.4, 54.8; 704 73.6, 70.6; 1424 128, 117; of short sequences 448
  // units 15.4, 15.9; 768 28.4, 27.1.  8/2 heads, D = 64: 508 56.6, 57.2; 640 26.6, 24.9.
  const int64_t tiles_max = (int64_t)T / kPfRows + B;
  const int sms = std::max(num_sms, 1);
  if (a.G % 2 == 0 && 2 * tiles_max * (Hq / 2) >= 7LL * sms) {
    if (!encode_3d(enc, &om, out, D, Hq, T, (uint64_t)D * 2, (uint64_t)Hq * D * 2, 64, 1, 32)) return UMIM_ERR_CUDA;
    auto kern = D == 128 ? prefill_pair_kernel<128> : prefill_pair_kernel<64>;
    const size_t smem = (size_t)(D == 128 ? PpSmem<128>::kTotal : PpSmem<64>::kTotal) + 1024;
    if (!allow_smem(kern, smem)) return UMIM_ERR_CUDA;
    trace_mark(stream, "prefill.attention");
    if (launch_pdl(kern, dim3((unsigned)sms), dim3(kPpThreads), smem, stream, qm, km, vm, om, a) != cudaSuccess)
      return UMIM_ERR_CUDA;
    trace_mark(stream, nullptr);
    return UMIM_OK;
  }
  auto kern = D == 128 ? prefill_tc_kernel<128> : prefill_tc_kernel<64>;
  const size_t smem = (size_t)(D == 128 ? PfSmem<128>::kTotal : PfSmem<64>::kTotal) + 1024;
  if (!allow_smem(kern, smem)) return UMIM_ERR_CUDA;
  // persistent: two CTAs per SM walk the (query tile, head) units; no more
  // CTAs than an upper bound of the units (each sequence wastes less than one tile)
  const int64_t units_max = ((int64_t)(T + kPfRows - 1) / kPfRows + B) * Hq;
  const unsigned gx = (unsigned)std::max<int64_t>(1, std::min<int64_t>(2LL * std::max(num_sms, 1), units_max));
  trace_mark(stream, "prefill.attention");
  if (launch_pdl(kern, dim3(gx), dim3(kPfThreads), smem, stream, qm, km, vm, a) != cudaSuccess)
    return UMIM_ERR_CUDA;
  trace_mark(stream, nullptr);
  return UMIM_OK;
}

}  // namespace umim
