// Fused DSVT layer in fp32 for the shapes of the paper (C = 64 / 128 / 192, hidden 0 / C / 2C): gather (Eq. 4) ->
// QKV projection -> per-set multi-head attention (Eq. 5) -> output projection -> residual + LayerNorm -> MLP with
// GELU -> residual + LayerNorm -> scatter (App. B.1.1).  All arithmetic is fp32 on the FMA pipes; other shapes, and
// bfloat16 weights that the tensor-core kernel does not cover, take layer_fma.cu.
//
// One thread block (16 warps, one block per SM) works on a tile of whole sets.
// Shared memory holds three row buffers [TM][C + 4]: A (x, then Q, the attention output and x1 in turn), B1 (K, Z,
// first half of the MLP hidden), B2 (V, second half), and a ring of three weight stages [C outputs][32 k] that TMA
// fills (128-byte swizzle; the warps take turns at issuing the next stage).  Weights are never transposed: both operands of a product are read along k as float4, and
// an accumulator is a float2 of the even-k and odd-k partial sums, so that one packed multiply-add takes its operands
// as they were loaded.  A first version staged weights by cp.async from all threads, 16 k at a time with a block-wide
// barrier per stage: a third of its instructions were copies and their addresses.
//
// Every wait is bounded; one that gives up raises DSVT_STATUS_TIMEOUT, and the block leaves at the end of its tile
// without having stored any of its rows.
//
// Measured (B200): two full layers, 12,345 pillars, C = 192: 0.78 ms, 19 TFLOP/s = 27 % of the FMA peak (layer_fma.cu:
// 1.79 ms); two attention-only layers, 2,000 pillars, C = 128: 0.11 ms (0.38 ms).  A C x C product of a 41-row tile takes
// 29 k cycles where the FMA pipes need 13 k: shared-memory loads and FMAs contend, and a block's share of the rows
// varies by a third.  Not kept: single multiply-adds with twice the columns per thread (0.88 ms), two k groups for 5
// and 6 rows per thread (0.82 ms, spills), a warp of its own for the weights (17 warps leave 96 registers per thread).
#include <limits.h>

#include "dsvt_common.cuh"
#include "fma_tile.cuh"
#include "tc_ptx.cuh"

namespace {
using namespace dsvt_tc;  // mbarriers, TMA

constexpr int kT = 512;    // compute threads
constexpr int kW = kT / 32;
constexpr int kKS = 32;    // k per weight stage: a 128-byte row
constexpr int kSt = 3;     // weight stages in the ring

struct F32Geom {
  int hidden, heads, tau;
  int rb_len, rb_sx, rb_sy, rb_centre;  // relative position bias (see dsvt_layer_params)
};

template <int C>
struct Shape {
  static constexpr int LD = C + 4;
  static constexpr int TM = C == 192 ? 64 : 96;  // most rows of a tile
  static constexpr int stages = C / kKS;         // weight stages of a C-deep product
  static constexpr uint32_t stage_bytes = C * kKS * 4;
  static constexpr size_t bytes = 1024 + (size_t)kSt * stage_bytes + sizeof(float) * 3 * (size_t)TM * LD;
};

struct F32Args {
  CUtensorMap qkv, o, w1, w2;  // boxes of 32 k x C outputs
  dsvt_fused_args a;
  F32Geom g;
  int32_t* status;
};

struct Ring {  // weight stage g of the launch lives in slot g % kSt
  unsigned long long full[kSt], empty[kSt];
  int abort_flag;
};
__shared__ Ring s_ring;

struct Job {  // one product: Dst[r][n] (+)= act(sum_k A[r][k] W[n][k] + bias[n])
  const float* A;      // first k; k >= C continues in the next row buffer
  float* D;
  const float* bias;   // or NULL
  int s0, ns;          // weight stages of the launch
  int t0, total;       // first stage of the tile, stages of a tile
  bool gelu, add, sync;  // sync: the destination is (part of) the operand
};

__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// One thread: stage g of the launch, stage g - t0 of its tile: chunks V, K, Q, O, MLP-1 pieces (each C outputs, C
// deep), then MLP-2 (hidden deep), once every warp is done with the stage that had the slot before.
template <int C>
__device__ __forceinline__ void issue_stage(const F32Args& f, uint32_t ring, int g, int t0) {
  constexpr int per = Shape<C>::stages;
  const int chunks = 4 + f.g.hidden / C, s = g - t0, slot = g % kSt, c = min(s / per, chunks);
  const CUtensorMap* map = c < 3 ? &f.qkv : c == 3 ? &f.o : c < chunks ? &f.w1 : &f.w2;
  const int row0 = c < 3 ? (2 - c) * C : c == 3 || c == chunks ? 0 : (c - 4) * C;
  if (g >= kSt && !mbar_wait(&s_ring.empty[slot], (uint32_t)(g / kSt - 1) & 1u, &s_ring.abort_flag)) return;
  mbar_expect_tx(&s_ring.full[slot], Shape<C>::stage_bytes);
  tma_load_2d(ring + slot * Shape<C>::stage_bytes, map, (s - c * per) * kKS, row0, &s_ring.full[slot]);
}

// Rows ty + 8 i (i < RM), columns tx + TX j (j < NJ) per thread; KG = 2: two groups of eight warps each take half of
// a stage's k and the sums meet in the destination, so that few rows still leave every thread RM x NJ sums.  Bound by
// shared-memory bandwidth and the FMA pipes alike: RM + NJ 16-byte loads, two wavefronts each, per 2 RM NJ packed
// multiply-adds.  The lane order (lanes 2i and 2i + 1 share a column, lanes i and i + 16 as well) is what lets a
// warp's 16-byte load with eight distinct addresses go out as two wavefronts; with eight distinct addresses in
// consecutive lanes it takes four.
template <int C, int RM, int KG>
__device__ __noinline__ void product(const F32Args& f, const unsigned char* ring, const Job jb) {
  constexpr int LD = Shape<C>::LD, TX = 64 / KG, NJ = C / TX;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int kg = KG == 2 ? warp >> 3 : 0, wc = KG == 2 ? (warp >> 1) & 3 : warp >> 1;
  const int tx = wc * 8 + ((lane >> 1) & 7), ty = (warp & 1) * 4 + ((lane & 1) | ((lane >> 3) & 2));
  float2 acc[RM][NJ];
#pragma unroll
  for (int i = 0; i < RM; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[i][j] = make_float2(0.f, 0.f);
  int slot = jb.s0 % kSt;
  uint32_t phase = (uint32_t)(jb.s0 / kSt) & 1u;
  __syncthreads();  // the operand is in place
  for (int s = 0; s < jb.ns; ++s) {
    mbar_wait(&s_ring.full[slot], phase, &s_ring.abort_flag);
    const int k = s * kKS;
    const float* a = jb.A + ty * LD + k + kg * (kKS / 2);
    if (k >= C) a += (size_t)Shape<C>::TM * LD - C;  // (the second row buffer of a 2C-deep operand)
    // row n of a stage is 128 bytes, its 16-byte chunk q stored at q ^ (n & 7); n & 7 is the same for all columns of a thread
    const unsigned char* w = ring + slot * Shape<C>::stage_bytes + tx * 128;
    const int swz = (tx & 7) << 4;
#pragma unroll
    for (int kk = 0; kk < kKS / KG; kk += 4) {
      float4 wv[NJ];
      const int q = ((4 * kk) ^ swz) ^ (kg * (2 * kKS));
#pragma unroll
      for (int j = 0; j < NJ; ++j) wv[j] = *reinterpret_cast<const float4*>(w + TX * 128 * j + q);
#pragma unroll
      for (int i = 0; i < RM; ++i) {
        const float4 av = lds4(a + 8 * i * LD + kk);
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          acc[i][j] = __ffma2_rn(make_float2(av.x, av.y), make_float2(wv[j].x, wv[j].y), acc[i][j]);
          acc[i][j] = __ffma2_rn(make_float2(av.z, av.w), make_float2(wv[j].z, wv[j].w), acc[i][j]);
        }
      }
    }
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(&s_ring.empty[slot]);
      const int next = jb.s0 + s + kSt;
      if ((next & (kW - 1)) == warp && next < jb.t0 + jb.total) issue_stage<C>(f, smem_u32(ring), next, jb.t0);
    }
    if (++slot == kSt) { slot = 0; phase ^= 1u; }
  }
  if (jb.sync) __syncthreads();
  if (KG == 2) {
    if (kg == 1) {
#pragma unroll
      for (int j = 0; j < NJ; ++j)
#pragma unroll
        for (int i = 0; i < RM; ++i) {
          float* d = jb.D + (ty + 8 * i) * LD + tx + TX * j;
          const float v = acc[i][j].x + acc[i][j].y;
          *d = jb.add ? *d + v : v;
        }
    }
    __syncthreads();
    if (kg == 1) return;
  }
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    const int n = tx + TX * j;
    const float b = jb.bias ? __ldg(jb.bias + n) : 0.f;
#pragma unroll
    for (int i = 0; i < RM; ++i) {
      float* d = jb.D + (ty + 8 * i) * LD + n;
      float v = acc[i][j].x + acc[i][j].y + b;
      if (KG == 2 || jb.add) v += *d;
      *d = jb.gelu ? dsvt_fma::gelu_erf(v) : v;
    }
  }
}

template <int C>
__device__ __forceinline__ void run_product(int rm, const F32Args& f, const unsigned char* ring, const Job& jb) {
  switch (rm) {
    case 1: product<C, 1, 2>(f, ring, jb); break;
    case 2: product<C, 2, 2>(f, ring, jb); break;
    case 3: product<C, 3, 2>(f, ring, jb); break;
    case 4: product<C, 4, 2>(f, ring, jb); break;
    case 5: product<C, 5, 1>(f, ring, jb); break;
    case 6: product<C, 6, 1>(f, ring, jb); break;
    case 7: case 8: product<C, 8, 1>(f, ring, jb); break;
    default:
      if constexpr (Shape<C>::TM > 64) product<C, 12, 1>(f, ring, jb);
  }
}

// LayerNorm of (x + z) for one row by one warp, two passes in registers; g == NULL: the plain sum.
template <int C>
__device__ __forceinline__ void norm_row(float (&t)[C / 32], const float* __restrict__ g, const float* __restrict__ b, float eps) {
  if (!g) return;
  const int lane = threadIdx.x & 31;
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < C / 32; ++i) s += t[i];
  const float mean = dsvt_fma::warp_sum(s) / (float)C;
  float q = 0.f;
#pragma unroll
  for (int i = 0; i < C / 32; ++i) { const float d = t[i] - mean; q += d * d; }
  const float inv = rsqrtf(dsvt_fma::warp_sum(q) / (float)C + eps);
#pragma unroll
  for (int i = 0; i < C / 32; ++i) t[i] = (t[i] - mean) * inv * __ldg(g + lane + 32 * i) + (b ? __ldg(b + lane + 32 * i) : 0.f);
}

// First index m in [lo, hi] with rowoff[m] >= v (hi if there is none below it), by one warp: each round narrows the
// range to a 32nd with one load per lane (two rounds for a thousand sets; a scalar binary search would be ten
// dependent loads).
__device__ __forceinline__ int warp_lower_bound(const int32_t* __restrict__ rowoff, int lo, int hi, int v) {
  const int lane = threadIdx.x & 31;
  while (lo < hi) {
    const int step = (hi - lo + 31) / 32;
    const int i = lo + lane * step;
    const bool less = i < hi && __ldg(rowoff + i) < v;
    const int cnt = __popc(__ballot_sync(0xffffffffu, less));  // (row offsets ascend: the first cnt probes are below v)
    if (cnt == 0) return lo;
    hi = min(hi, lo + cnt * step);
    lo += (cnt - 1) * step + 1;
  }
  return lo;
}

template <int C, int D>
__global__ void __launch_bounds__(kT, 1) layer_f32_kernel(const __grid_constant__ F32Args f) {
  constexpr int LD = Shape<C>::LD, TM = Shape<C>::TM, per = Shape<C>::stages, V4 = C / 4;
  const dsvt_fused_args& a = f.a;
  const F32Geom& g = f.g;
  int32_t* status = f.status;
  volatile int* abort_flag = &s_ring.abort_flag;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* ring = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  float* bufA = reinterpret_cast<float*>(ring + kSt * Shape<C>::stage_bytes);
  float* bufK = bufA + TM * LD;
  float* bufV = bufK + TM * LD;
  __shared__ int rowvox[TM], rowlin[TM];
  __shared__ unsigned char row_lo[TM], row_n[TM];
  __shared__ int bounds[2];
  const dsvt_layer_params& p = a.p;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int hidden = g.hidden, tau = g.tau;
  if (tid == 0) {
    s_ring.abort_flag = 0;
    for (int i = 0; i < kSt; ++i) { mbar_init(&s_ring.full[i], 1); mbar_init(&s_ring.empty[i], kW); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  pdl_enter();  // everything below may read what earlier kernels of the stream wrote
  __syncthreads();
  const int total = (4 + hidden / C) * per + hidden / kKS;
  int stage0 = 0;  // weight stages consumed by the tiles so far

  const int S = min(__ldg(a.num_sets), a.cap_sets);
  const int R = S > 0 ? __ldg(a.rowoff + S) : 0;
  // This block's sets: those whose first row lies in its equal share of the rows.  They are cut into tiles of at most
  // TM rows, of about the same height.
  if (warp < 2) {
    const int b = S <= 0 ? 0 : warp_lower_bound(a.rowoff, 0, S, (int)((int64_t)R * (blockIdx.x + warp) / gridDim.x));
    if (lane == 0) bounds[warp] = warp == 1 && blockIdx.x + 1 == gridDim.x ? S : b;
  }
  __syncthreads();
  const int s_end = bounds[1];
  for (int s_lo = bounds[0], nsets; s_lo < s_end; s_lo += nsets) {
    if (__syncthreads_or(*abort_flag)) break;  // (also orders the previous tile's last reads)
    const int base = __ldg(a.rowoff + s_lo), left = __ldg(a.rowoff + s_end) - base;
    if (warp == 0) {
      const int cuts = (left + TM - 1) / TM, want = cuts > 1 ? min(TM, (left + cuts - 1) / cuts + tau / 2) : TM;
      const int e = warp_lower_bound(a.rowoff, s_lo + 1, s_end + 1, base + want + 1) - 1;  // last boundary within `want` rows
      if (lane == 0) bounds[0] = max(e, s_lo + 1);
    }
    // (rows that no set fills, where the offsets claim more than a set has, are keys and queries of their own)
    for (int r = tid; r < TM; r += kT) { rowvox[r] = -1; rowlin[r] = 0; row_lo[r] = (unsigned char)r; row_n[r] = 1; }
    __syncthreads();
    nsets = bounds[0] - s_lo;
    const int rows = __ldg(a.rowoff + s_lo + nsets) - base;
    if (rows > TM || rows <= 0 || nsets > TM) {  // row offsets that do not describe this table
      if (tid == 0) atomicOr(status, DSVT_STATUS_BAD_INDEX);
      continue;
    }
    if (tid == 0)
      for (int s = 0; s < kSt; ++s) issue_stage<C>(f, smem_u32(ring), stage0 + s, stage0);
    // ---- distinct slots of each set -> tile rows (Eq. 4), one warp per set ----
    for (int si = warp; si < nsets; si += kW) {
      const int32_t* row = a.table + (size_t)(s_lo + si) * tau;
      const int off = __ldg(a.rowoff + s_lo + si);
      const int lb = off - base, cap = __ldg(a.rowoff + s_lo + si + 1) - off;
      const bool inside = lb >= 0 && lb < TM;
      const int cnt_max = inside ? min(cap, TM - lb) : 0;
      int cnt = 0;
      int lo3[3] = {INT_MAX, INT_MAX, INT_MAX}, hi3[3] = {INT_MIN, INT_MIN, INT_MIN};
      for (int k0 = 0; k0 < tau; k0 += 32) {
        const int k = k0 + lane;
        int v = -1;
        bool uniq = false;
        if (k < tau) {
          v = row[k];
          uniq = (k == 0) || (v != row[k - 1]);
        }
        const unsigned bal = __ballot_sync(0xffffffffu, uniq);
        const int pos = cnt + __popc(bal & ((1u << lane) - 1u));
        if (uniq && pos < cnt_max) {
          if (v < 0 || v >= a.n) { atomicOr(status, DSVT_STATUS_BAD_INDEX); v = -1; }
          rowvox[lb + pos] = v;
          row_lo[lb + pos] = (unsigned char)lb;
          row_n[lb + pos] = (unsigned char)cnt_max;
          if (p.rpb && v >= 0) {
            const int4 c = __ldg(reinterpret_cast<const int4*>(p.coords) + v);
            lo3[0] = min(lo3[0], c.y); hi3[0] = max(hi3[0], c.y);
            lo3[1] = min(lo3[1], c.z); hi3[1] = max(hi3[1], c.z);
            lo3[2] = min(lo3[2], c.w); hi3[2] = max(hi3[2], c.w);
            rowlin[lb + pos] = c.y * g.rb_sx + c.z * g.rb_sy + c.w;
          }
        }
        cnt += __popc(bal);
      }
      bool bad = cnt != cap;
      if (p.rpb) {  // a set spread wider than the table's extent is reported
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int l = -dsvt_fma::warp_max_int(-lo3[q]), h = dsvt_fma::warp_max_int(hi3[q]);
          bad |= (h >= l) && (h - l > p.rpb_extent[q] - 1);
        }
      }
      if (bad && lane == 0) atomicOr(status, DSVT_STATUS_BAD_INDEX);
    }
    __syncthreads();
    const int rm = (rows + 7) >> 3, rows_pad = rm <= 6 ? 8 * rm : rm <= 8 ? 64 : TM;
    auto gather = [&](bool with_pe) {
      for (int i = tid; i < rows_pad * V4; i += kT) {
        const int r = i / V4, c4 = i - r * V4;
        const int v = r < rows ? rowvox[r] : -1;
        float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
        if (v >= 0) {
          f = reinterpret_cast<const float4*>(a.x + (size_t)v * C)[c4];
          if (with_pe) {
            const float4 e = __ldg(reinterpret_cast<const float4*>(p.pe + (size_t)v * C) + c4);
            f.x += e.x; f.y += e.y; f.z += e.z; f.w += e.w;
          }
        }
        *reinterpret_cast<float4*>(bufA + r * LD + 4 * c4) = f;
      }
    };
    // ---- projections; values come from the bare rows, keys and queries from the rows with the positional term ----
    gather(false);
    run_product<C>(rm, f, ring, Job{bufA, bufV, p.b_qkv ? p.b_qkv + 2 * C : nullptr, stage0, per, stage0, total, false, false, false});
    if (p.pe) {
      __syncthreads();
      gather(true);
    }
    run_product<C>(rm, f, ring, Job{bufA, bufK, p.b_qkv ? p.b_qkv + C : nullptr, stage0 + per, per, stage0, total, false, false, false});
    run_product<C>(rm, f, ring, Job{bufA, bufA, p.b_qkv, stage0 + 2 * per, per, stage0, total, false, false, true});
    __syncthreads();
    // ---- attention inside each set: two threads per (query row, head), each takes every other key with a running
    // softmax, and the two halves are merged at the end ----
    {
      const float scale = rsqrtf((float)D);
      const int par = tid & 1;
      const int items = rows * g.heads;
      for (int it0 = 0; it0 < items; it0 += kT / 2) {
        const int it = it0 + (tid >> 1);
        const bool on = it < items;
        const int h = on ? it / rows : 0, r = on ? it - h * rows : 0;
        const int k_lo = row_lo[r], m = on ? row_n[r] : 0;
        float q[D], o[D];
        float mx = -INFINITY, den = 0.f;
        float* qrow = bufA + r * LD + h * D;
#pragma unroll
        for (int c = 0; c < D; c += 4) {
          const float4 v = lds4(qrow + c);
          q[c] = v.x; q[c + 1] = v.y; q[c + 2] = v.z; q[c + 3] = v.w;
          o[c] = o[c + 1] = o[c + 2] = o[c + 3] = 0.f;
        }
        const float* kb = bufK + k_lo * LD + h * D;
        const float* vb = bufV + k_lo * LD + h * D;
        const float* tab = p.rpb ? p.rpb + (size_t)h * g.rb_len : nullptr;
        for (int k = par; k < m; k += 4) {  // keys k and k + 2
          const bool two = k + 2 < m;
          const int kk[2] = {k, two ? k + 2 : k};
          float lg[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            float s0 = 0.f, s1 = 0.f;
#pragma unroll
            for (int c = 0; c < D; c += 4) {
              const float4 v = lds4(kb + kk[u] * LD + c);
              s0 = fmaf(q[c], v.x, s0); s1 = fmaf(q[c + 1], v.y, s1);
              s0 = fmaf(q[c + 2], v.z, s0); s1 = fmaf(q[c + 3], v.w, s1);
            }
            lg[u] = (s0 + s1) * scale;
            if (tab) {
              const int idx = rowlin[r] - rowlin[k_lo + kk[u]] + g.rb_centre;
              lg[u] += __ldg(tab + min(max(idx, 0), g.rb_len - 1));
            }
          }
          if (!two) lg[1] = -INFINITY;
          const float nm = fmaxf(mx, fmaxf(lg[0], lg[1])), from = nm == -INFINITY ? 0.f : nm;  // (a bias may rule out all keys so far)
          const float al = expf(mx - from), e0 = expf(lg[0] - from), e1 = expf(lg[1] - from);  // (exp(-inf) = 0)
          mx = nm;
          den = den * al + (e0 + e1);
#pragma unroll
          for (int c = 0; c < D; c += 4) {
            const float4 v0 = lds4(vb + kk[0] * LD + c), v1 = lds4(vb + kk[1] * LD + c);
            o[c] = fmaf(o[c], al, fmaf(e0, v0.x, e1 * v1.x));
            o[c + 1] = fmaf(o[c + 1], al, fmaf(e0, v0.y, e1 * v1.y));
            o[c + 2] = fmaf(o[c + 2], al, fmaf(e0, v0.z, e1 * v1.z));
            o[c + 3] = fmaf(o[c + 3], al, fmaf(e0, v0.w, e1 * v1.w));
          }
        }
        // merge the two threads' halves (the second one has no keys if the set holds one voxel)
        const float om = __shfl_xor_sync(0xffffffffu, mx, 1), nm = fmaxf(mx, om);
        const float al = nm == -INFINITY ? 0.f : expf(mx - nm);
        den *= al;
        den += __shfl_xor_sync(0xffffffffu, den, 1);
        const float inv = 1.0f / den;
#pragma unroll
        for (int c = 0; c < D; ++c) {
          o[c] *= al;
          o[c] = (o[c] + __shfl_xor_sync(0xffffffffu, o[c], 1)) * inv;
        }
        if (on) {  // both threads have read the query: its slot takes the output, half from each
          if (par == 0) {
#pragma unroll
            for (int c = 0; c < D / 2; c += 4) *reinterpret_cast<float4*>(qrow + c) = make_float4(o[c], o[c + 1], o[c + 2], o[c + 3]);
          } else {
#pragma unroll
            for (int c = (D / 2 + 3) / 4 * 4; c < D; c += 4)
              *reinterpret_cast<float4*>(qrow + c) = make_float4(o[c], o[c + 1], o[c + 2], o[c + 3]);
          }
        }
      }
    }
    // ---- output projection into the key buffer ----
    run_product<C>(rm, f, ring, Job{bufA, bufK, p.b_o, stage0 + 3 * per, per, stage0, total, false, false, false});
    __syncthreads();
    const bool mlp = hidden > 0;
    // ---- x1 = LN1(x + Z): to the operand buffer, or to y where the layer ends here ----
    for (int r = *abort_flag ? rows : warp; r < rows; r += kW) {  // (a wait that gave up did so before the barrier)
      const int v = rowvox[r];
      float tr[C / 32];
#pragma unroll
      for (int i = 0; i < C / 32; ++i)
        tr[i] = bufK[r * LD + lane + 32 * i] + (v >= 0 && !a.attention_only ? a.x[(size_t)v * C + lane + 32 * i] : 0.f);
      if (!a.attention_only) norm_row<C>(tr, p.ln1_g, p.ln1_b, p.ln_eps);
#pragma unroll
      for (int i = 0; i < C / 32; ++i) {
        if (mlp) bufA[r * LD + lane + 32 * i] = tr[i];
        else if (v >= 0) a.y[(size_t)v * C + lane + 32 * i] = tr[i];
      }
    }
    if (!mlp) { stage0 += total; continue; }
    // ---- MLP: H = gelu(x1 W_1^T + b_1) into B1 (and B2), x1 += H W_2^T + b_2 ----
    for (int c = 0; c < hidden / C; ++c)
      run_product<C>(rm, f, ring, Job{bufA, bufK + c * TM * LD, p.b_1 ? p.b_1 + c * C : nullptr, stage0 + (4 + c) * per, per, stage0, total, true, false, false});
    run_product<C>(rm, f, ring, Job{bufK, bufA, p.b_2, stage0 + (4 + hidden / C) * per, hidden / kKS, stage0, total, false, true, false});
    __syncthreads();
    // ---- y = LN2(x1 + M) ----
    for (int r = *abort_flag ? rows : warp; r < rows; r += kW) {
      const int v = rowvox[r];
      float tr[C / 32];
#pragma unroll
      for (int i = 0; i < C / 32; ++i) tr[i] = bufA[r * LD + lane + 32 * i];
      norm_row<C>(tr, p.ln2_g, p.ln2_b, p.ln_eps);
      if (v >= 0) {
#pragma unroll
        for (int i = 0; i < C / 32; ++i) a.y[(size_t)v * C + lane + 32 * i] = tr[i];
      }
    }
    stage0 += total;
  }
  __syncthreads();
  if (tid == 0 && *abort_flag) {
    atomicOr(status, DSVT_STATUS_TIMEOUT);
    // no load may still be writing into this block's shared memory when it retires
    for (int g0 = max(stage0 - kSt, 0); g0 < stage0; ++g0)
      for (int it = 0; it < kMaxPolls && !mbar_try(&s_ring.full[g0 % kSt], (uint32_t)(g0 / kSt) & 1u); ++it) {}
  }
}

template <int C, int D>
int launch_f32(dsvt_ctx* ctx, const F32Args& f, int grid, unsigned flag) {
  if (!(ctx->attr_flags & flag)) {
    DSVT_CUDA_TRY(ctx, cudaFuncSetAttribute(layer_f32_kernel<C, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Shape<C>::bytes));
    ctx->attr_flags |= flag;
  }
  DSVT_CUDA_TRY(ctx, launch_pdl(layer_f32_kernel<C, D>, dim3((unsigned)grid), dim3(kT), Shape<C>::bytes, ctx->stream, f));
  DSVT_LAUNCHED(ctx);
  return DSVT_OK;
}

}  // namespace

bool dsvt_layer_f32_supported(const dsvt_fused_args& a) {
  const dsvt_layer_params& p = a.p;
  if (p.precision != DSVT_FP32 || !dsvt_tensor_maps_available()) return false;
  const int d = p.C / p.heads, hidden = a.attention_only ? 0 : p.hidden;
  if (hidden != 0 && hidden != p.C && hidden != 2 * p.C) return false;
  if (p.C == 192) return d == 24 && p.set_size <= 64;
  return ((p.C == 128 && (d == 16 || d == 32)) || (p.C == 64 && d == 16)) && p.set_size <= 96;
}

int dsvt_launch_layer_f32(dsvt_ctx* ctx, const dsvt_fused_args& a) {
  const dsvt_layer_params& p = a.p;
  F32Args f = {};
  F32Geom& g = f.g;
  g.hidden = a.attention_only ? 0 : p.hidden; g.heads = p.heads; g.tau = p.set_size;
  if (p.rpb) {
    const int L = p.rpb_extent[0], W = p.rpb_extent[1], H = p.rpb_extent[2];
    g.rb_sy = 2 * H - 1;
    g.rb_sx = (2 * W - 1) * g.rb_sy;
    g.rb_len = (2 * L - 1) * g.rb_sx;
    g.rb_centre = (L - 1) * g.rb_sx + (W - 1) * g.rb_sy + (H - 1);
  }
  int64_t rmax = (int64_t)a.cap_sets * p.set_size;
  if (rmax > a.n) rmax = a.n;
  int64_t grid = ctx->sm_count;  // one block per SM, no more blocks than rows
  if (grid > rmax) grid = rmax;
  if (grid < 1) grid = 1;
  f.a = a;
  f.status = ctx->status;
  if (!dsvt_cached_weight_map(ctx, &f.qkv, p.W_qkv, 3 * p.C, p.C, p.C, true) || !dsvt_cached_weight_map(ctx, &f.o, p.W_o, p.C, p.C, p.C, true))
    return DSVT_ERR_CUDA;
  f.w1 = f.w2 = f.o;
  if (g.hidden > 0 && (!dsvt_cached_weight_map(ctx, &f.w1, p.W_1, g.hidden, p.C, p.C, true) ||
                       !dsvt_cached_weight_map(ctx, &f.w2, p.W_2, p.C, g.hidden, p.C, true)))
    return DSVT_ERR_CUDA;
  const int d = p.C / p.heads;
  if (p.C == 192) return launch_f32<192, 24>(ctx, f, (int)grid, 1u << 16);
  if (p.C == 128 && d == 16) return launch_f32<128, 16>(ctx, f, (int)grid, 1u << 17);
  if (p.C == 128) return launch_f32<128, 32>(ctx, f, (int)grid, 1u << 18);
  return launch_f32<64, 16>(ctx, f, (int)grid, 1u << 19);
}
