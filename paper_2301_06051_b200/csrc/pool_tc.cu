// Attention-style 3D pooling (Eq. 6, Eq. 7) with the four projections on the 5th-generation tensor cores
// (tcgen05 + TMEM), bfloat16 operands, fp32 accumulation.
//
// A tile is whole regions of together at most 128 rows.  The rows are the voxels in (region, slot) order; where empty
// slots are keys with a term of their own they are rows too, all slots of a region.  (Otherwise an empty slot's key is
// the bias alone: its score is one more term of the region's sum, its value adds nothing, and no row is spent on it.)
// Per tile: the compute warps gather the rows (plus the slot term) into a bf16 A operand X~ and take the Eq. 6 maxima over
// the regions' rows into another, P, repeated for every row of a region; the tensor pipe forms K = X~ W_k^T and
// Q = P W_q^T (M = 128, N = C) into TMEM; each thread reads its row's quarter of Q and K straight from TMEM, takes the
// scores of its heads, and exchanges them with the other rows of its region through shared memory.  V = X~ W_v^T follows
// into the query's columns; its weighted rows are summed towards a region's first row by shuffles and go back to TMEM
// as the A operand of the output projection, whose first rows are the regions' outputs.  All arithmetic on Q, K and V
// is fp32.
//
// A tile is a chain of dependent phases, so the time is the number of tiles times the chain's length: 22,000 cycles for
// 125 rows with C = 192, 4,600 of them the tensor pipe's.  Longest: maxima 2.0, waits for Q 2.6, gather 3.0, sums of the
// values 1.9, output rows 3.4 thousand.  The next tile's rows are gathered, and their keys formed, while the output
// projection of this one runs (in one sequence 31,600 cycles).  What a phase costs is mostly its address arithmetic: the
// gather took 8,200 cycles in lane-linear units with a division and a swizzle per 16 bytes.
//
// Roles (608 threads): warps 0-15 compute; warp 16 streams the four weight matrices through a three-stage ring
// with plain (single-CTA) TMA loads, tile after tile; warp 17 allocates TMEM and issues the tcgen05.mma
// instructions; warp 18 cuts the row list into tiles, one ahead.  Every mbarrier wait is bounded (DSVT_STATUS_TIMEOUT).
#include <cuda.h>

#include "dsvt_common.cuh"
#include "tc_ptx.cuh"

namespace {
using namespace dsvt_tc;

constexpr int kComputeWarps = 16;
constexpr int kComputeThreads = 32 * kComputeWarps;
constexpr int kTmaWarp = kComputeWarps, kMmaWarp = kComputeWarps + 1, kListWarp = kComputeWarps + 2;
constexpr int kThreads = kComputeThreads + 96;
constexpr int kStages = 3;

struct PoolTcMaps {
  CUtensorMap w[4];  // W_q, W_k, W_v, W_o: boxes of 64 input columns x C rows, 128-byte swizzle
};

struct PoolMisc {
  unsigned long long full[kStages], empty[kStages], acc_full[2], acc_free[2];
  unsigned long long x_ready;   // compute -> MMA: X~ is in place
  unsigned long long p_ready;   // compute -> MMA: P is in place
  unsigned long long ao_ready;  // compute -> MMA: the attention output is in place
  unsigned long long list_ready[2], list_free[2];  // row lists: list warp <-> compute
  unsigned long long drain;
  uint32_t tmem_base;
  int abort_flag;
  int rowvox[2][kTM];  // tile row -> voxel (-1: empty slot)
  int row_seg[2][kTM];  // tile row -> first row of its region | the region's rows << 8 | slot << 16 | region of the tile << 24
  int tile[2][3];      // rows, regions, rank of the first region
  float logit[8][kTM];  // [head][row]
  alignas(16) float carry[kComputeWarps][48];  // a warp's part of a region that starts in the previous one
};
__shared__ PoolMisc s_pm;

__device__ __forceinline__ void quarter_sync(int q) { asm volatile("bar.sync %0, 128;" ::"r"(2 + q) : "memory"); }
__device__ __forceinline__ void compute_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kComputeThreads) : "memory"); }

// fp32 output staging: row r, 16-byte chunk c4 XORed with the row (conflict-free for row-per-thread and row-per-warp
// access alike).
template <int C>
__device__ __forceinline__ uint32_t out_off(int r, int c4) {
  return (uint32_t)(r * (C * 4) + ((c4 ^ (r & 7)) << 4));
}

// ================= weight stream (one thread) ===========================================================
template <int C>
__device__ __noinline__ void pool_producer(const PoolTcMaps& maps, uint32_t st_base, int my_tiles) {
  constexpr int NKB = C / 64;
  constexpr uint32_t STAGE_BYTES = C * 128;
  volatile int* abort_flag = &s_pm.abort_flag;
  int stage = 0;
  uint32_t phase = 0;
  int issued[kStages] = {0, 0, 0};
  for (int t = 0; t < my_tiles; ++t) {
    for (int i = 0; i < 4; ++i) {
      const int c = i == 0 ? 1 : i == 1 ? 0 : i;  // W_k, W_q, W_v, W_o
      for (int kb = 0; kb < NKB; ++kb) {
        if (!mbar_wait(&s_pm.empty[stage], phase ^ 1u, abort_flag)) goto done;
        mbar_expect_tx(&s_pm.full[stage], STAGE_BYTES);
        tma_load_2d(st_base + stage * STAGE_BYTES, &maps.w[c], kb * 64, 0, &s_pm.full[stage]);
        ++issued[stage];
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
    }
  }
done:
  if (*abort_flag) {  // leaving early: no load may still be writing into this CTA's shared memory when it retires
#pragma unroll
    for (int i = 0; i < kStages; ++i)
      if (issued[i] > 0) {
        const uint32_t par = (uint32_t)(issued[i] - 1) & 1u;
        for (int it = 0; it < kMaxPolls && !mbar_try(&s_pm.full[i], par); ++it) {}
      }
  }
}

// ================= MMA issuer (one warp) ================================================================
// Chunks of a tile: K (A = X~, region 1 once the scores have read the previous tile's K), Q (A = P, region 0),
// V (A = X~, region 0 once the scores have read Q), O (A = attention output in TMEM, region 0 once V has been read).
// Warp-uniform code, an elected lane issues (from one divergent thread an MMA took 46 cycles and more to issue).
template <int C>
__device__ __forceinline__ void pool_mma(uint32_t x_base, uint32_t p_base, uint32_t st_base, uint32_t tmem, int my_tiles) {
  constexpr int NKB = C / 64;
  constexpr uint32_t STAGE16 = C * 128 / 16, kRows16 = kTM * 128 / 16, SW = kDescHiSwizzled;
  volatile int* abort_flag = &s_pm.abort_flag;
  const uint32_t x_lo = desc_lo_swizzled(x_base), p_lo = desc_lo_swizzled(p_base), w_lo = desc_lo_swizzled(st_base);
  int stage = 0;
  uint32_t phase = 0;
  for (int t = 0; t < my_tiles; ++t) {
    for (int c = 0; c < 4; ++c) {
      const uint32_t bar = c == 0 ? 1u : 0u;
      unsigned long long* ready = c == 0 ? &s_pm.x_ready : c == 1 ? &s_pm.p_ready : &s_pm.ao_ready;
      if (c != 2 && !mbar_wait(ready, (uint32_t)t & 1u, abort_flag)) goto done;
      const uint32_t uses = c == 0 ? (uint32_t)t : 3u * (uint32_t)t + (uint32_t)(c - 1);  // of the accumulator, so far
      if (!mbar_wait(&s_pm.acc_free[bar], (uses & 1u) ^ 1u, abort_flag)) goto done;
      tc_fence_after();
      const uint32_t a_lo = c == 1 ? p_lo : x_lo, d_tmem = tmem + bar * C;
      for (int kb = 0; kb < NKB; ++kb) {
        if (!mbar_wait(&s_pm.full[stage], phase, abort_flag)) goto done;
        tc_fence_after();
        if (elect_one()) {
#pragma unroll
          for (int k4 = 0; k4 < 4; ++k4) {
            if (c == 3)
              umma_ts(d_tmem, tmem + 2 * C + 32 * kb + 8 * k4, w_lo + stage * STAGE16 + 2 * k4, SW, umma_idesc(C), (kb | k4) != 0 ? 1u : 0u);
            else umma_ss(d_tmem, a_lo + kb * kRows16 + 2 * k4, SW, w_lo + stage * STAGE16 + 2 * k4, SW, umma_idesc(C),
                         (kb | k4) != 0 ? 1u : 0u);
          }
          umma_commit(&s_pm.empty[stage]);
          if (kb == NKB - 1) umma_commit(&s_pm.acc_full[bar]);
        }
        __syncwarp();
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
    }
  }
done:
  if (*abort_flag) {  // the MMAs already issued must have completed before the TMEM columns are returned
    if (elect_one()) umma_commit(&s_pm.drain);
    __syncwarp();
    for (int it = 0; it < kMaxPolls && !mbar_try(&s_pm.drain, 0u); ++it) {}
  }
}

struct PoolTcArgs {
  const float* feats;
  const int4* rows;
  const int32_t* num_rows;
  const int32_t* cell_map;
  const int32_t* region_key;
  const int32_t* num_out;
  int32_t cap_m;
  const float *b_q, *b_k, *b_v, *b_o, *slot_pe;
  float* out_feats;
  int32_t nslots, mask_empty;
  int32_t* status;
};

// ================= list warp: the rows of every tile ===================================================
// Tile t: the regions that start in rows [t * step, (t + 1) * step) of the list.  With step <= 129 - ns its rows are
// within 128 from t * step; with all slots as rows regions start at multiples of ns and step is 128.
struct PoolRows {
  bool padded;  // all slots are rows
  int n_rows, step;
};
__device__ __forceinline__ void pool_list(const PoolTcArgs& a, const PoolRows& pr, int my_tiles, int C) {
  constexpr int W = kTM / 32;
  volatile int* abort_flag = &s_pm.abort_flag;
  const int lane = threadIdx.x & 31, ns = a.nslots;
  for (int tl = 0; tl < my_tiles; ++tl) {
    const int b = tl & 1, row0 = (int)(blockIdx.x + tl * gridDim.x) * pr.step;
    int4 v[W];  // (voxel, rows of its region | slot << 8 | starts the region << 16, rank)
#pragma unroll
    for (int q = 0; q < W; ++q) {
      const int i = row0 + 32 * q + lane, slot = i & (ns - 1);
      v[q] = make_int4(-1, 0, 0, 0);
      if (i >= pr.n_rows) continue;
      if (pr.padded)
        v[q] = make_int4(__ldg(a.cell_map + (size_t)__ldg(a.region_key + i / ns) * ns + slot), ns | (slot << 8) | ((slot == 0) << 16), i / ns, 0);
      else v[q] = __ldg(a.rows + i);
    }
    uint32_t st[W];
    int lo = kTM, hi = pr.step < kTM ? kTM : min(kTM, pr.n_rows - row0);
    // (all starts, then only those at or after step: the next tile's)
#pragma unroll
    for (int q = W - 1; q >= 0; --q) {
      st[q] = __ballot_sync(0xffffffffu, (v[q].y >> 16) != 0);
      if (st[q]) lo = 32 * q + __ffs(st[q]) - 1;
      if (pr.step < kTM) {
        const int o = pr.step - 32 * q;
        const uint32_t after = o >= 32 ? 0u : o > 0 ? st[q] & (0xffffffffu << o) : st[q];
        if (after) hi = 32 * q + __ffs(after) - 1;
      }
    }
    hi = min(hi, pr.n_rows - row0);
    lo = min(lo, hi);
    if (!mbar_wait(&s_pm.list_free[b], ((uint32_t)(tl >> 1) & 1u) ^ 1u, abort_flag)) break;
    int before = 0, first = 0;  // starts in the words so far; the last start so far
#pragma unroll
    for (int q = 0; q < W; ++q) {
      const int o = 32 * q + lane;
      const uint32_t upto = st[q] & (0xffffffffu >> (31 - lane));
      const int ri = before + __popc(upto) - 1, f = upto ? 32 * q + 31 - __clz(upto) : first;
      if (o >= lo && o < hi) {
        s_pm.rowvox[b][o - lo] = v[q].x;
        s_pm.row_seg[b][o - lo] = (f - lo) | ((v[q].y & 255) << 8) | (((v[q].y >> 8) & 255) << 16) | (ri << 24);
        if (o == lo) s_pm.tile[b][2] = v[q].z;
        if (o == hi - 1) s_pm.tile[b][1] = ri + 1;
      }
      before += __popc(st[q]);
      if (st[q]) first = 32 * q + 31 - __clz(st[q]);
    }
    if (lane == 0) {
      s_pm.tile[b][0] = hi - lo;
      if (hi == lo) s_pm.tile[b][1] = 0;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&s_pm.list_ready[b]);
    // the rows are gathered a tile's time from now: bring them into L2
#pragma unroll
    for (int q = 0; q < W; ++q) {
      const int o = 32 * q + lane;
      if (o >= lo && o < hi && v[q].x >= 0)
        for (int c = 0; c < C; c += 32) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.feats + (size_t)v[q].x * C + c));
    }
  }
}

// ================= compute warps: gather + Eq. 6 ========================================================
// 16 lanes to a row (256 bytes), all loads of a thread in flight together, as bf16 to dst; with PE plus the slot term.
// A thread's rows are 32 apart, its chunks 16: all its addresses are one base plus constants.
template <int C, bool PE>
__device__ __forceinline__ void pool_gather(const PoolTcArgs& a, uint32_t dst, int b) {
  constexpr int ROWS = kComputeThreads / 16, P = kTM / ROWS, J = C / 64;
  const int nrow = s_pm.tile[b][0], r0 = threadIdx.x / 16, c0 = threadIdx.x % 16;
  const uint32_t to = dst + swz(r0, c0 >> 1) + 8 * (c0 & 1);
  float4 f[P][J];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int r = r0 + ROWS * p, v = r < nrow ? s_pm.rowvox[b][r] : -1;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      f[p][j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (v >= 0) f[p][j] = __ldg(reinterpret_cast<const float4*>(a.feats + (size_t)v * C) + c0 + 16 * j);
    }
  }
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const float* pe = nullptr;
    if (PE && r0 + ROWS * p < nrow) pe = a.slot_pe + (size_t)((s_pm.row_seg[b][r0 + ROWS * p] >> 16) & 255) * C;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      float4 g = f[p][j];
      if (PE && pe) {
        const float4 e = __ldg(reinterpret_cast<const float4*>(pe) + c0 + 16 * j);
        g.x += e.x; g.y += e.y; g.z += e.z; g.w += e.w;
      }
      sts2(to + p * (ROWS * 128) + j * (kTM * 128), make_uint2(pack_bf16(g.x, g.y), pack_bf16(g.z, g.w)));
    }
  }
}

// Every row of P becomes the maximum over its region's rows of src (rounding to bf16 is monotone, so the maximum of
// rounded values is the rounded maximum), with the zero row of the region's empty slots if those count.  src may be P
// itself: a row that already holds the maximum changes nothing.
template <int C>
__device__ __forceinline__ void pool_max(uint32_t src, uint32_t ps, int b, int ns, int full) {
  constexpr int ROWS = kComputeThreads / 8, J = C / 64;
  const int nrow = s_pm.tile[b][0], c = threadIdx.x % 8;
  auto max4 = [](uint32_t (&m)[4], float4 u) {
    const uint32_t w[4] = {__float_as_uint(u.x), __float_as_uint(u.y), __float_as_uint(u.z), __float_as_uint(u.w)};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const __nv_bfloat162 t = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&m[k]), *reinterpret_cast<const __nv_bfloat162*>(&w[k]));
      m[k] = *reinterpret_cast<const uint32_t*>(&t);
    }
  };
#pragma unroll
  for (int h = 0; h < kTM / ROWS; ++h) {
    const int r = threadIdx.x / 8 + ROWS * h;
    if (r >= nrow) continue;
    const int seg = s_pm.row_seg[b][r], j0 = seg & 255, cnt = (seg >> 8) & 255;
    const uint32_t init = cnt < full ? 0u : 0xff80ff80u;  // zero, minus infinity
    uint32_t m[J][4];
#pragma unroll
    for (int j = 0; j < J; ++j) m[j][0] = m[j][1] = m[j][2] = m[j][3] = init;
    if (ns <= 4) {  // (no loop: the loads overlap)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (k < cnt) {
          const uint32_t at = src + swz(j0 + k, c);
#pragma unroll
          for (int j = 0; j < J; ++j) max4(m[j], lds4(at + j * (kTM * 128)));
        }
      }
    } else {
      for (int k = 0; k < cnt; ++k) {
        const uint32_t at = src + swz(j0 + k, c);
#pragma unroll
        for (int j = 0; j < J; ++j) max4(m[j], lds4(at + j * (kTM * 128)));
      }
    }
    const uint32_t to = ps + swz(r, c);
#pragma unroll
    for (int j = 0; j < J; ++j) sts4(to + j * (kTM * 128), make_uint4(m[j][0], m[j][1], m[j][2], m[j][3]));
  }
}

// ================= the kernel ===========================================================================
// Thread (row, quarter): warp w owns TMEM lanes 32 (w % 4) .. + 31 (tile rows) and the column quarter w / 4, which
// holds HQ = (C / 4) / D whole heads.
template <int C, int D>
__global__ void __launch_bounds__(kThreads, 1) pool_tc_kernel(const __grid_constant__ PoolTcArgs a,
                                                              const __grid_constant__ PoolTcMaps maps) {
  constexpr int QC = C / 4, HQ = QC / D;
  constexpr uint32_t TILE_BYTES = kTM * C * 2;
  extern __shared__ unsigned char pool_tc_smem[];
  const uint32_t raw = smem_u32(pool_tc_smem);
  const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
  unsigned char* sm = pool_tc_smem + pad;
  const uint32_t sbase = raw + pad;
  // X~; P, later the fp32 output staging (half a tile's rows)
  const uint32_t st_base = sbase + 2 * TILE_BYTES;
  const uint32_t xs_s = sbase, ps_s = sbase + TILE_BYTES, par_s = st_base + kStages * C * 128;
  float* par = reinterpret_cast<float*>(sm + 2 * TILE_BYTES + kStages * C * 128);  // b_q, b_k, b_v, b_o
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int ns = a.nslots;
  volatile int* abort_flag = &s_pm.abort_flag;
  if (tid == 0) {
    s_pm.abort_flag = 0;
    for (int i = 0; i < 2; ++i)
      for (int k = 0; k < 3; ++k) s_pm.tile[i][k] = 0;
    for (int i = 0; i < kStages; ++i) { mbar_init(&s_pm.full[i], 1); mbar_init(&s_pm.empty[i], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&s_pm.acc_full[i], 1); mbar_init(&s_pm.acc_free[i], kComputeThreads); }
    mbar_init(&s_pm.x_ready, kComputeThreads);
    mbar_init(&s_pm.p_ready, kComputeThreads);
    for (int i = 0; i < 2; ++i) { mbar_init(&s_pm.list_ready[i], 1); mbar_init(&s_pm.list_free[i], kComputeThreads); }
    mbar_init(&s_pm.ao_ready, kComputeThreads);
    mbar_init(&s_pm.drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_pm.tmem_base)),
                 "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // everything above touched this CTA's own state; what follows reads what the kernels before it in the stream wrote
  // (the row list, the number of regions; the weights and biases too: every launch of the call may start early, the first
  // of them under the tail of a kernel that writes them): wait for them if this launch was allowed to start early
  pdl_enter();
  const int m = min(*a.num_out, a.cap_m);
  PoolRows pr;
  pr.padded = a.rows == nullptr;
  pr.n_rows = pr.padded ? m * ns : *a.num_rows;
  for (int i = tid; i < 4 * C; i += kThreads) {
    const int which = i / C;
    const float* v = which == 0 ? a.b_q : which == 1 ? a.b_k : which == 2 ? a.b_v : a.b_o;
    par[i] = v ? __ldg(v + i % C) : 0.f;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_pm.tmem_base;
  pr.step = pr.padded ? kTM : kTM + 1 - ns;
  if (!pr.padded) {  // as many rounds of tiles as steps of that length take, evenly filled
    const int rounds = max(1, (pr.n_rows + pr.step * (int)gridDim.x - 1) / (pr.step * (int)gridDim.x));
    pr.step = max(1, (pr.n_rows + rounds * (int)gridDim.x - 1) / (rounds * (int)gridDim.x));
  }
  const int full = pr.padded || a.mask_empty ? 0 : ns;  // regions of fewer rows have empty slots that count
  const int num_tiles = (pr.n_rows + pr.step - 1) / pr.step;
  const int my_tiles = (int)blockIdx.x < num_tiles ? (num_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;

  if (warp == kTmaWarp) {
    if (lane == 0) pool_producer<C>(maps, st_base, my_tiles);
    __syncwarp();
  } else if (warp == kMmaWarp) {
    pool_mma<C>(sbase, sbase + TILE_BYTES, st_base, __shfl_sync(0xffffffffu, tmem, 0), my_tiles);
    __syncwarp();
  } else if (warp == kListWarp) {
    pool_list(a, pr, my_tiles, C);
    __syncwarp();
  } else {
    const int row = 32 * (warp & 3) + lane, hq = warp >> 2;
    const uint32_t taddr = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + hq * QC;
    const float scale = rsqrtf((float)D);
    uint32_t uses[2] = {0u, 0u};
    bool ok = true;
    auto acc_wait = [&](int bar) {
      ok = mbar_wait(&s_pm.acc_full[bar], uses[bar] & 1u, abort_flag) && ok;
      ++uses[bar];
      tc_fence_after();
    };
    // the rows of a tile, one tile ahead of its maxima: X~ has been read by the value projection of the one before
    auto gather = [&](int tl) {
      ok = mbar_wait(&s_pm.list_ready[tl & 1], (uint32_t)(tl >> 1) & 1u, abort_flag) && ok;
      if (a.slot_pe) pool_gather<C, true>(a, xs_s, tl & 1);
      else pool_gather<C, false>(a, xs_s, tl & 1);
      fence_proxy_async();
      mbar_arrive(&s_pm.x_ready);
    };
    if (my_tiles > 0) gather(0);
    for (int tl = 0; tl < my_tiles; ++tl) {
      const int b = tl & 1;
      compute_sync();  // X~ is complete; the previous tile's staging rows have been stored
      const int nrow = s_pm.tile[b][0], nr = s_pm.tile[b][1], rank0 = s_pm.tile[b][2];
      if (a.slot_pe) {  // the maxima are over the plain rows
        pool_gather<C, false>(a, ps_s, b);
        compute_sync();
      }
      pool_max<C>(a.slot_pe ? ps_s : xs_s, ps_s, b, ns, full);
      fence_proxy_async();
      mbar_arrive(&s_pm.p_ready);
      // ---- scores: q . k per head of this quarter, softmax over the region's rows ----
      const int seg = row < nrow ? s_pm.row_seg[b][row] : 0, j0 = seg & 255, cnt = (seg >> 8) & 255;
      mbar_arrive(&s_pm.list_free[b]);
      const float empty = cnt > 0 && cnt < full ? (float)(full - cnt) : 0.f;  // empty slots that count
      float p[HQ], pe[HQ];  // scores of this row, and of an empty slot (whose key is the bias)
      float v[QC];  // this thread's query columns: read at once, so that the value projection can take their region
      acc_wait(0);
      tmem_ld_row(taddr, v);
      tmem_wait_ld();
      tc_fence_before();
      mbar_arrive(&s_pm.acc_free[0]);
      acc_wait(1);
#pragma unroll
      for (int j = 0; j < HQ; ++j) {  // one head at a time: D query and D key columns of this thread's row
        float k[D];
        tmem_ld_row(taddr + C + j * D, k);
        tmem_wait_ld();
        float acc = 0.f, acc_e = 0.f;
#pragma unroll
        for (int c = 0; c < D; c += 4) {
          const int cc = hq * QC + j * D + c;
          const float4 bq = lds4(par_s + 4u * (uint32_t)cc), bk = lds4(par_s + 4u * (uint32_t)(C + cc));
          const float q0 = v[j * D + c] + bq.x, q1 = v[j * D + c + 1] + bq.y, q2 = v[j * D + c + 2] + bq.z, q3 = v[j * D + c + 3] + bq.w;
          acc = fmaf(q0, k[c], acc); acc_e = fmaf(q0, bk.x, acc_e);
          acc = fmaf(q1, k[c + 1], acc); acc_e = fmaf(q1, bk.y, acc_e);
          acc = fmaf(q2, k[c + 2], acc); acc_e = fmaf(q2, bk.z, acc_e);
          acc = fmaf(q3, k[c + 3], acc); acc_e = fmaf(q3, bk.w, acc_e);
        }
        pe[j] = acc_e * scale;
        p[j] = (acc + acc_e) * scale;
        s_pm.logit[hq * HQ + j][row] = p[j];
      }
      tc_fence_before();
      mbar_arrive(&s_pm.acc_free[1]);
      quarter_sync(hq);
#pragma unroll
      for (int j = 0; j < HQ; ++j) {
        const float* l = s_pm.logit[hq * HQ + j] + j0;
        float l4[4];
        float mx = empty > 0.f ? pe[j] : -INFINITY;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          l4[k] = k < cnt ? l[k] : -INFINITY;
          mx = fmaxf(mx, l4[k]);
        }
        for (int k = 4; k < cnt; ++k) mx = fmaxf(mx, l[k]);
        float sum = empty > 0.f ? empty * __expf(pe[j] - mx) : 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) sum += __expf(l4[k] - mx);
        for (int k = 4; k < cnt; ++k) sum += __expf(l[k] - mx);
        p[j] = cnt > 0 ? __expf(p[j] - mx) / sum : 0.f;
      }
      __syncwarp();
      // ---- values, weighted, summed towards the region's first row: by shuffles inside the warp, through shared memory
      // where a region lies across two warps' rows (it has at most 32) ----
      acc_wait(0);
      tmem_ld_row(taddr, v);
      tmem_wait_ld();
      tc_fence_before();
      mbar_arrive(&s_pm.acc_free[0]);
#pragma unroll
      for (int c = 0; c < QC; ++c) v[c] *= p[c / D];
      const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)cnt);
      for (int o = 1; o < most; o <<= 1) {
        const bool take = lane + o < 32 && row + o < j0 + cnt;
#pragma unroll
        for (int c = 0; c < QC; ++c) {
          const float got = __shfl_down_sync(0xffffffffu, v[c], o);
          if (take) v[c] += got;
        }
      }
      if (lane == 0 && row > j0 && cnt > 0) {
#pragma unroll
        for (int c = 0; c < QC; ++c) s_pm.carry[warp][c] = v[c];
      }
      quarter_sync(hq);
      const bool start = cnt > 0 && row == j0;
      if (start && lane + cnt > 32) {
#pragma unroll
        for (int c = 0; c < QC; ++c) v[c] += s_pm.carry[warp + 1][c];
      }
      __syncwarp();
      {
        const uint32_t t_a = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + 2 * C + hq * (QC / 2);
#pragma unroll
        for (int c = 0; c < QC / 16; ++c) {  // the probabilities sum to one: + b_v once
          uint32_t w[8];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float4 bv = lds4(par_s + 4u * (uint32_t)(2 * C + hq * QC + 16 * c + 4 * k));
            const float* t = v + 16 * c + 4 * k;
            w[2 * k] = pack_bf16(t[0] + bv.x, t[1] + bv.y);
            w[2 * k + 1] = pack_bf16(t[2] + bv.z, t[3] + bv.w);
          }
          tmem_st8_u32(t_a + 8 * c, w);
        }
        tmem_wait_st();
        tc_fence_before();
      }
      mbar_arrive(&s_pm.ao_ready);
      if (tl + 1 < my_tiles) gather(tl + 1);
      // ---- output projection: the regions' first rows, staged half a tile at a time ----
      acc_wait(0);
      tmem_ld_row(taddr, v);
      tmem_wait_ld();
      tc_fence_before();
      mbar_arrive(&s_pm.acc_free[0]);
      const int n_out = min(nr, m - rank0);  // (regions beyond the output's capacity are dropped)
      for (int r0 = 0; r0 < n_out; r0 += kTM / 2) {
        const int ri = (int)((unsigned)seg >> 24) - r0;
        if (r0 > 0) compute_sync();
        if (start && ri >= 0 && ri < kTM / 2) {
#pragma unroll
          for (int q4 = 0; q4 < QC / 4; ++q4) {
            const float4 bo = lds4(par_s + 4u * (uint32_t)(3 * C + hq * QC + 4 * q4));
            sts4(ps_s + out_off<C>(ri, hq * (QC / 4) + q4),
                 make_float4(v[4 * q4] + bo.x, v[4 * q4 + 1] + bo.y, v[4 * q4 + 2] + bo.z, v[4 * q4 + 3] + bo.w));
          }
        }
        compute_sync();
        const int n = min(n_out - r0, kTM / 2), r1 = tid / 16, c1 = tid % 16;
#pragma unroll
        for (int p = 0; p < kTM / 2; p += kComputeThreads / 16) {  // (addresses as in the gather)
#pragma unroll
          for (int j = 0; j < C / 64; ++j)
            if (r1 + p < n)
              reinterpret_cast<float4*>(a.out_feats + (size_t)(rank0 + r0 + r1 + p) * C)[c1 + 16 * j] =
                  lds4(ps_s + out_off<C>(r1, c1) + p * (C * 4) + j * 256);
        }
      }
    }
    if (!ok || *abort_flag) {
      if (tid == 0) atomicOr(a.status, DSVT_STATUS_TIMEOUT);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

}  // namespace

bool dsvt_pool_tc_supported(int C, int heads, int nslots) {
  if (heads < 1 || C % heads != 0) return false;
  const int d = C / heads;
  if (!((C == 192 && d == 24) || (C == 128 && (d == 16 || d == 32)) || (C == 64 && d == 16))) return false;
  return nslots >= 1 && nslots <= 32 && (nslots & (nslots - 1)) == 0;
}

namespace {
template <int C, int D>
int launch_pool_tc(dsvt_ctx* ctx, const PoolTcArgs& a, const PoolTcMaps& maps, int grid, unsigned flag) {
  const size_t smem = 2 * (size_t)kTM * C * 2 + kStages * (size_t)C * 128 + 4 * (size_t)C * sizeof(float) + 1024;
  if (!(ctx->attr_flags & flag)) {  // (once per context: the attribute belongs to its device)
    DSVT_CUDA_TRY(ctx, cudaFuncSetAttribute(pool_tc_kernel<C, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    ctx->attr_flags |= flag;
  }
  DSVT_CUDA_TRY(ctx, launch_pdl(pool_tc_kernel<C, D>, dim3(grid), dim3(kThreads), smem, ctx->stream, a, maps));
  DSVT_LAUNCHED(ctx);
  return DSVT_OK;
}
}  // namespace

int dsvt_launch_pool_tc(dsvt_ctx* ctx, const dsvt_pool_tc_call& c) {
  PoolTcArgs a;
  a.feats = c.feats; a.rows = c.rows; a.num_rows = c.num_rows; a.cell_map = c.cell_map; a.region_key = c.region_key; a.num_out = c.num_out; a.cap_m = c.cap_m;
  a.b_q = c.b_q; a.b_k = c.b_k; a.b_v = c.b_v; a.b_o = c.b_o; a.slot_pe = c.slot_pe;
  a.out_feats = c.out_feats; a.nslots = c.nslots; a.mask_empty = c.mask_empty;
  a.status = ctx->status;
  PoolTcMaps maps;
  for (int i = 0; i < 4; ++i)
    if (!dsvt_cached_weight_map(ctx, &maps.w[i], c.W[i], c.C, c.C, c.C)) return DSVT_ERR_CUDA;
  const int64_t most = c.n < c.cap_m ? c.n : c.cap_m;  // regions
  const int64_t tiles = c.rows ? dsvt_ceil_div(c.n, kTM + 1 - c.nslots) : dsvt_ceil_div(most * c.nslots, kTM);
  int64_t grid = tiles < ctx->sm_count ? tiles : ctx->sm_count;
  if (grid < 1) grid = 1;
  const int d = c.C / c.heads;
  if (c.C == 192) return launch_pool_tc<192, 24>(ctx, a, maps, (int)grid, 16u);
  if (c.C == 128 && d == 16) return launch_pool_tc<128, 16>(ctx, a, maps, (int)grid, 32u);
  if (c.C == 128) return launch_pool_tc<128, 32>(ctx, a, maps, (int)grid, 64u);
  return launch_pool_tc<64, 16>(ctx, a, maps, (int)grid, 128u);
}
