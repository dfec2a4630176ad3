// DSVT layers in fp32 (C = 64 / 128 / 192) with the matrix products on the tensor cores: gather (Eq. 4) -> QKV
// projection -> per-set multi-head attention (Eq. 5) -> output projection -> residual + LayerNorm -> MLP with GELU ->
// residual + LayerNorm -> scatter (App. B.1.1).
//
// A layer is five kernels over the rows of its sets, in the order of the table (a row's place there is its position):
// QKV, attention, output projection + LayerNorm, first MLP product + GELU, second MLP product + LayerNorm; one more in front
// of every two layers prepares weights and row lists.  Between them the rows lie in the context's workspace,
// [position][Q, attention output or x1 | K, then MLP hidden | V].  One fused kernel cannot hold a tile: its operands take 144 KB
// in three parts (below) and Q, K and V 295 KB.  The workspace is bounded, so a layer of many rows runs in passes of whole sets.
//
// An fp32 product on tcgen05 (Henry, Tang, Heinecke, "Leveraging the bfloat16 artificial intelligence datatype for
// higher-precision computations", ARITH 2019): each operand is the sum of three bfloat16 parts, exact together, and of the nine
// partial products the six largest are formed, each exact in fp32.  With all parts rounded the three that are left out are at most
// 0.9 x 2^-24 of a product (with the first part truncated: 3.5 x 2^-24).  The tensor cores' additions truncate (for which reason
// Ootomo and Yokota, "Recovering single precision accuracy from tensor cores while surpassing the FP32 theoretical peak
// performance", 2022, add partial sums outside of them): with all six in one accumulator the error is 1.2e-6 of the result's
// 2-norm at K = 192, seven times that of fp32 multiply-adds with two running sums (1.8e-7).  So the leading product has an
// accumulator of its own, which is read out and cleared every kChunk stages, and the five small ones share another, where truncation
// is 2^-8 as large.
// Error against float64 of two layers, kernel on the FMA pipes -> now (12 seeds; 2-norm, and largest error in units of the
// result's root mean square):
//   C = 192, hidden 384       3.1e-7 -> 1.9e-7    2.1e-6 -> 1.5e-6
//   C = 192, hidden 256       4.0e-7 -> 1.9e-7    2.6e-6 -> 1.4e-6
//   C = 192, attention alone  1.4e-7 -> 1.1e-7    8.9e-7 -> 7.9e-7
//   C = 128, attention alone  1.23e-7 -> 0.98e-7  7.2e-7 -> 6.5e-7
//   C = 64, hidden 128        1.9e-7 -> 1.6e-7    1.2e-6 -> 1.1e-6
// One attention with positive weights and features, where truncations add up: 0.8e-7 -> 1.2e-7.
//
// Measured (B200): two full layers and their partition, 12,345 pillars, C = 192: 775.8 us on the FMA pipes (27 % of their peak:
// shared-memory reads for the products, and the phases between them), 290.5 us now; two attention-only layers, 2,000 pillars,
// C = 128: 110.3 us and 90.9.  A single voxel, which then was one launch of a tile of eight rows, has got slower: a full layer
// 50.4 us -> 65.0 (60 voxels 84.9 -> 73.2).  A product's tile of 128 rows takes 9 to 11 k cycles, the start of each of its kernels 4 k
// (first instructions, lists, operands) and its epilogue 6 k.
//
// Every wait is bounded; one that gives up raises DSVT_STATUS_TIMEOUT, its block stores nothing more, and no later kernel of
// the call's fp32 layers stores to y (what lies in the workspace for its rows is another call's).
#include <limits.h>

#include "dsvt_common.cuh"
#include "fma_tile.cuh"
#include "tc_ptx.cuh"

namespace {
using namespace dsvt_tc;

// Warps: epilogue (two threads to a row of the tile), conversion of the operand rows, weight copies, MMA issue.
// (Eight warps convert: with four a stage's conversion takes longer than its MMAs; two full layers of 12,345 pillars 287.6 us with
// four, 281.3 with eight.)
constexpr int kEpiThreads = 2 * kTM, kConvThreads = 256;
constexpr int kConvWarp = kEpiThreads / 32, kCopyWarp = kConvWarp + kConvThreads / 32, kMmaWarp = kCopyWarp + 1;
constexpr int kThreads = 32 * (kMmaWarp + 1);
constexpr int kKS = 16;        // k per operand stage: one MMA step
constexpr int kSt = 4;         // stages
constexpr int kFly = 3;        // stages of operand rows in a converting thread's registers (4: 281.6 us, 6: 284.7)
constexpr int kParts = 3;      // bfloat16 parts of an operand
// Most stages between two readings of the leading accumulator, as few as keep every error of the table above below the FMA
// kernel's: with 96 k the largest error of attention alone is 9.0e-7 (C = 192) and 7.9e-7 (128), and 12,345 pillars take 244 us instead
// of 255; with 32 for N = 192 284 us.
template <int N>
constexpr int kChunk = (N == 192 ? 64 : 48) / kKS;
constexpr int kSpare = 64;         // columns of a half's sum of chunks in TMEM: at N and at kCorr + N
constexpr uint32_t kCorr = 256;  // TMEM column of the accumulator of the small products (the leading one is at 0)

// Operand parts in shared memory: unswizzled, [8-column chunk][row][16 bytes].
template <int N>
struct Sm {
  static constexpr uint32_t ca = kTM * 16, cw = N * 16;
  static constexpr uint32_t a_part = kKS / 8 * ca, w_part = kKS / 8 * cw;
  static constexpr uint32_t w_off = kParts * a_part, w_stage = kParts * w_part, stage = w_off + w_stage, staging = kSt * stage;
  static constexpr uint32_t bytes = staging + kTM * N * 4;
};

struct Pass { int s_first, s_end, row0, row_end; };  // sets and (local) positions of a pass

// Stages of a chunk of the leading product: as few chunks as kChunk allows, of about the same size.
template <int N>
__device__ __forceinline__ int chunk_stages(int ns) { const int n = (ns + kChunk<N> - 1) / kChunk<N>; return (ns + n - 1) / n; }

enum Epilogue { kBias = 0, kNorm = 1, kGelu = 2 };

struct GemmArgs {
  const float* a;        // operand rows [position][lda], or NULL: rows of x, gathered, + pe for the first pe_tiles tiles
  const float *x, *pe;
  const int32_t* list;   // voxel of each position
  const Pass* pass;
  const unsigned char* w;  // parts of [tiles_n N][k]: per tile and stage one block of Sm<N>::w_stage bytes
  const float* bias;     // or NULL
  float* out;            // [position][ldo], or NULL: rows of y
  float* y;
  const float* res;      // kNorm: residual rows [position][ldr], or NULL: rows of x if add_x
  const float *ln_g, *ln_b;
  int32_t* status;       // [0] status bits, [1] this call's number, [2] the last call in which a wait gave up
  int32_t* counter;      // kBias: set to zero, for the kernel behind
  int32_t n, lda, ldr, k, tiles_n, pe_tiles, ldo, add_x;
  float eps;
};

struct GemmShared {
  unsigned long long full[kSt], empty[kSt], acc_full, acc_free, chunk_full, chunk_free, drain;
  uint32_t tmem;
  int abort_flag, leave_y;
  alignas(16) float par[3 * 192];  // bias, gain, shift
  float2 stat[2][kTM];             // (sum, sum of squared deviations) of a row's halves
};
__shared__ GemmShared s_gm;

// Four fp32 values -> 8 bytes of each part.
__device__ __forceinline__ void split4(const float4 f, uint2& h, uint2& m, uint2& l) {
  const float v[4] = {f.x, f.y, f.z, f.w};
  uint32_t p[3][2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    // (saturating, so that the first part of a large finite value is finite)
    asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(p[0][i]) : "f"(v[2 * i + 1]), "f"(v[2 * i]));
    const float2 r = __fadd2_rn(make_float2(v[2 * i], v[2 * i + 1]),
                                make_float2(-__uint_as_float(p[0][i] << 16), -__uint_as_float(p[0][i] & 0xffff0000u)));
    p[1][i] = pack_bf16(r.x, r.y);
    const float2 q = __fadd2_rn(r, make_float2(-__uint_as_float(p[1][i] << 16), -__uint_as_float(p[1][i] & 0xffff0000u)));
    p[2][i] = pack_bf16(q.x, q.y);
  }
  h = make_uint2(p[0][0], p[0][1]); m = make_uint2(p[1][0], p[1][1]); l = make_uint2(p[2][0], p[2][1]);
}

// fp32 rows on their way in (residual) and out: row r, 16-byte chunk c4, XORed with the row, so that a warp per rows and a
// thread per row are both without bank conflicts.
template <int N>
__device__ __forceinline__ uint32_t stage_off(int r, int c4) { return (uint32_t)(r * (N * 4) + ((c4 ^ (r & 7)) << 4)); }

__device__ __forceinline__ int num_tiles(const GemmArgs& a) { return (a.pass->row_end + kTM - 1) / kTM * a.tiles_n; }

// Voxel of a position of the pass (-1: none).
__device__ __forceinline__ int voxel_at(const GemmArgs& a, const Pass& ps, int pos) {
  const int v = __ldg(a.list + pos);  // (the list has room for whole tiles)
  return pos >= ps.row0 && pos < ps.row_end && (unsigned)v < (unsigned)a.n ? v : -1;
}

// Weights' parts -> stages.  (The first copies used to start before the wait, on the ground that the kernels that made the parts
// were complete by then; only the wait makes their stores visible.  Two layers of 12,345 pillars: 256.8 us that way, 256.6 now.)
template <int N>
__device__ __forceinline__ void copy_role(const GemmArgs& a, uint32_t sbase, int ns) {
  volatile int* abort_flag = &s_gm.abort_flag;
  pdl_wait();
  const int tiles = num_tiles(a), leave = !a.out && __ldcg(a.status + 1) == __ldcg(a.status + 2);
  s_gm.leave_y = leave;  // (before the first stage, without which no tile is finished; an epilogue thread that reads the words costs 3 %)
  uint32_t g = 0;
  for (int t = blockIdx.x; t < tiles && !*abort_flag; t += gridDim.x)
    for (int s = 0; s < ns; ++s, ++g) {
      const uint32_t slot = g % kSt;
      if (g >= kSt && !mbar_wait(&s_gm.empty[slot], (g / kSt - 1) & 1u, abort_flag)) break;
      mbar_expect_tx(&s_gm.full[slot], Sm<N>::w_stage);
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   ::"r"(sbase + slot * Sm<N>::stage + Sm<N>::w_off), "l"(a.w + ((size_t)(t % a.tiles_n) * ns + s) * Sm<N>::w_stage),
                   "r"(Sm<N>::w_stage), "r"(smem_u32(&s_gm.full[slot])) : "memory");
    }
  if (*abort_flag)  // no copy may still be writing into this block's shared memory when it retires
    for (uint32_t q = g < kSt ? 0 : g - kSt; q < g; ++q)
      for (int i = 0; i < kMaxPolls && !mbar_try(&s_gm.full[q % kSt], (q / kSt) & 1u); ++i) {}
}

// The warp that issues the MMAs.  Operand parts (0 = leading) of the small products, smallest first.
template <int N>
__device__ __forceinline__ void mma_role(uint32_t sbase, int tiles, int ns) {
  constexpr uint32_t hi = desc_hi_plain(128), idesc = umma_idesc(N);
  volatile int* abort_flag = &s_gm.abort_flag;
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_gm.tmem, 0);
  const int chunk = chunk_stages<N>(ns);
  uint32_t g = 0, it = 0, chunks = 0;
  bool ok = true;
  for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x, ++it) {
    if (it > 0) ok = mbar_wait(&s_gm.acc_free, (it - 1) & 1u, abort_flag);
    for (int s = 0, fresh_at = 0; ok && s < ns; ++s, ++g) {
      const uint32_t slot = g % kSt, par = (g / kSt) & 1u;
      const bool fresh = s == fresh_at;
      if (fresh) fresh_at += chunk;
      ok = mbar_wait(&s_gm.full[slot], par, abort_flag);
      if (ok && fresh && s > 0) ok = mbar_wait(&s_gm.chunk_free, chunks++ & 1u, abort_flag);
      if (!ok) break;
      tc_fence_after();
      if (elect_one()) {
        const uint32_t a = desc_lo_plain(sbase + slot * Sm<N>::stage, Sm<N>::ca);
        const uint32_t w = desc_lo_plain(sbase + slot * Sm<N>::stage + Sm<N>::w_off, Sm<N>::cw);
        constexpr int ap[6] = {2, 1, 0, 1, 0, 0}, wp[6] = {0, 1, 2, 0, 1, 0};
#pragma unroll
        for (int q = 0; q < 6; ++q)
          umma_ss(tmem + (q < 5 ? kCorr : 0u), a + ap[q] * (Sm<N>::a_part / 16), hi, w + wp[q] * (Sm<N>::w_part / 16), hi, idesc,
                  q < 5 ? ((s | q) != 0 ? 1u : 0u) : (fresh ? 0u : 1u));
        umma_commit(&s_gm.empty[slot]);
        if (s == ns - 1) umma_commit(&s_gm.acc_full);
        else if (s + 1 == fresh_at) umma_commit(&s_gm.chunk_full);
      }
      __syncwarp();
    }
  }
  if (*abort_flag) {  // leaving early: what has been issued must be complete before the TMEM columns are returned
    if (elect_one()) umma_commit(&s_gm.drain);
    __syncwarp();
    for (int i = 0; i < kMaxPolls && !mbar_try(&s_gm.drain, 0u); ++i) {}
  }
}

// Operand rows -> bfloat16 parts.  A half warp takes eight rows' 32 bytes of a chunk, so that its 8-byte stores fill the
// chunk's 128 bytes of these rows (whole sectors on the way in, no bank twice on the way out; with padded chunks instead, to
// take four rows' 64 bytes, the MMAs' operand rows straddled 128-byte lines and a stage took 1050 cycles); kFly stages are
// in a thread's registers.
template <int N, bool PE>
__device__ __forceinline__ void convert_role(const GemmArgs& a, const Pass& ps, uint32_t sbase, int tiles, int ns) {
  constexpr int kRows = kConvThreads / 4, P = kTM / kRows;
  volatile int* abort_flag = &s_gm.abort_flag;
  const int t0 = threadIdx.x - 32 * kConvWarp, lane = t0 & 31, r = 8 * (t0 >> 5) + ((lane >> 1) & 7), c = 2 * (lane >> 4) + (lane & 1);
  const float4* src = reinterpret_cast<const float4*>(a.a ? a.a : a.x);
  const uint32_t to = sbase + (c >> 1) * Sm<N>::ca + r * 16 + (c & 1) * 8;
  uint32_t g = 0;
  for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int rt = t / a.tiles_n, nt = t - rt * a.tiles_n;
    const bool pe = PE && nt < a.pe_tiles;
    int at[P];  // the rows' first 16 bytes of this thread, in such units (< 0: none)
#pragma unroll
    for (int p = 0; p < P; ++p) {
      const int pos = rt * kTM + r + kRows * p;
      const int row = a.a ? (pos >= ps.row0 && pos < ps.row_end ? pos : -1) : voxel_at(a, ps, pos);
      at[p] = row < 0 ? -1 : row * (a.lda / 4) + c;
    }
    float4 f[kFly][P];
    auto load = [&](float4 (&d)[P], int s) {
#pragma unroll
      for (int p = 0; p < P; ++p) {
        d[p] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s < ns && at[p] >= 0) d[p] = __ldcg(src + (unsigned)(at[p] + s * (kKS / 4)));
      }
    };
#pragma unroll
    for (int u = 0; u < kFly; ++u) load(f[u], u);
    for (int s0 = 0; s0 < ns; s0 += kFly) {
#pragma unroll
      for (int u = 0; u < kFly; ++u) {
        const int s = s0 + u;
        if (s < ns) {
          const uint32_t slot = g % kSt;
          if (g >= kSt && !mbar_wait(&s_gm.empty[slot], (g / kSt - 1) & 1u, abort_flag)) return;
#pragma unroll
          for (int p = 0; p < P; ++p) {
            uint2 h, m, l;
            if (pe && at[p] >= 0) {
              const float4 e = __ldg(reinterpret_cast<const float4*>(a.pe) + (unsigned)(at[p] + s * (kKS / 4)));
              f[u][p].x += e.x; f[u][p].y += e.y; f[u][p].z += e.z; f[u][p].w += e.w;
            }
            split4(f[u][p], h, m, l);
            const uint32_t d = to + slot * Sm<N>::stage + p * (kRows * 16);
            sts2(d, h);
            sts2(d + Sm<N>::a_part, m);
            sts2(d + 2 * Sm<N>::a_part, l);
          }
          load(f[u], s + kFly);
          fence_proxy_async();
          mbar_arrive(&s_gm.full[slot]);
          ++g;
        }
      }
    }
  }
}

// Accumulators (+ half-way sum) + bias (+ residual) -> LayerNorm or GELU -> rows, by way of the staging area, in which a
// thread works on its own row.
template <int N, int EPI>
__device__ __forceinline__ void epilogue_role(const GemmArgs& a, const Pass& ps, uint32_t staging, int tiles) {
  constexpr int kRows = kEpiThreads / 16, P = kTM / kRows, J = N / 64, H = N / 2;
  volatile int* abort_flag = &s_gm.abort_flag;
  const int tid = threadIdx.x, row = tid & (kTM - 1), half = tid / kTM, c0 = half * H;
  const int r16 = tid >> 4, c16 = tid & 15;  // in and out: 16 lanes to a row, a thread's rows 16 apart
  const bool add = EPI == kNorm && (a.res || a.add_x);
  const int ns = a.k / kKS, chunk = chunk_stages<N>(ns);
  const uint32_t lane0 = s_gm.tmem + ((uint32_t)(row & ~31) << 16), taddr = lane0 + c0, tsum = lane0 + (half ? kCorr : 0u) + N;
  const uint32_t par = smem_u32(s_gm.par) + 4 * c0;
  uint32_t it = 0, chunks = 0;
  for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++it) {
    const int rt = t / a.tiles_n, nt = t - rt * a.tiles_n, p0 = rt * kTM;
    // (also orders the previous tile's reads of the staging area and the bias; every exit is taken by all threads)
    if (bar_or(1, kEpiThreads, *abort_flag != 0)) break;
    for (int i = tid; i < N; i += kEpiThreads) s_gm.par[i] = a.bias ? __ldg(a.bias + nt * N + i) : 0.f;
    if (EPI == kNorm) {
#pragma unroll 4
      for (int p = 0; p < P; ++p) {
        const int rr = r16 + kRows * p, pos = p0 + rr;
        const int v = a.res ? (pos >= ps.row0 && pos < ps.row_end ? pos : -1) : voxel_at(a, ps, pos);
        const float4* src = reinterpret_cast<const float4*>(a.res ? a.res + (size_t)v * a.ldr : a.x + (size_t)v * N) + c16;
#pragma unroll
        for (int j = 0; j < J; ++j) {
          const uint32_t dst = staging + stage_off<N>(rr, c16 + 16 * j);
          if (add && v >= 0)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src + 16 * j) : "memory");
          else
            sts4(dst, make_float4(0.f, 0.f, 0.f, 0.f));
        }
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
    }
    bar_or(1, kEpiThreads, false);  // bias and residual are in place
    // The leading accumulator's chunks meet in the TMEM columns that are left, kSpare for each half, apart from the residual: a
    // sum with it would be rounded once more, at the residual's size.  (N = 192: the last third in the staging area, on top of it.)
    for (int s = chunk; s < ns; s += chunk) {
      mbar_wait(&s_gm.chunk_full, chunks++ & 1u, abort_flag);
      tc_fence_after();
#pragma unroll 1
      for (int q = 0; q < H; q += 32) {
        float m[32];
        tmem_ld_row(taddr + q, m);
        if (q < kSpare) {
          float p[32];
          if (s > chunk) tmem_ld_row(tsum + q, p);
          tmem_wait_ld();
          if (s > chunk)
#pragma unroll
            for (int i = 0; i < 32; ++i) m[i] += p[i];
          tmem_st_row(tsum + q, m);
          continue;
        }
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const uint32_t at = staging + stage_off<N>(row, (c0 + q + i) / 4);
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (EPI == kNorm || s > chunk) v = lds4(at);
          sts4(at, make_float4(v.x + m[i], v.y + m[i + 1], v.z + m[i + 2], v.w + m[i + 3]));
        }
      }
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive(&s_gm.chunk_free);
    }
    mbar_wait(&s_gm.acc_full, it & 1u, abort_flag);
    tc_fence_after();
    float2 sum = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int q = 0; q < H; q += 16) {
      float m[16], k[16], p[16];
      const bool spare = ns > chunk && q < kSpare;
      tmem_ld16_at<0>(taddr + q, m);
      tmem_ld16_at<0>(taddr + kCorr + q, k);
      if (spare) tmem_ld16_at<0>(tsum + q, p);
      tmem_wait_ld();
      if (spare)
#pragma unroll
        for (int i = 0; i < 16; ++i) m[i] += p[i];
#pragma unroll
      for (int i = 0; i < 16; i += 4) {
        const uint32_t at = staging + stage_off<N>(row, (c0 + q + i) / 4);
        const float4 b4 = lds4(par + 4 * (q + i));
        float4 v = make_float4(m[i] + k[i] + b4.x, m[i + 1] + k[i + 1] + b4.y, m[i + 2] + k[i + 2] + b4.z, m[i + 3] + k[i + 3] + b4.w);
        if (EPI == kNorm || (ns > chunk && q >= kSpare)) {
          const float4 x4 = lds4(at);
          v.x += x4.x; v.y += x4.y; v.z += x4.z; v.w += x4.w;
        }
        if (EPI == kNorm) {
          sum = __fadd2_rn(sum, __fadd2_rn(make_float2(v.x, v.y), make_float2(v.z, v.w)));
        }
        if (EPI == kGelu)
          v = make_float4(dsvt_fma::gelu_erf(v.x), dsvt_fma::gelu_erf(v.y), dsvt_fma::gelu_erf(v.z), dsvt_fma::gelu_erf(v.w));
        sts4(at, v);
      }
    }
    tc_fence_before();
    mbar_arrive(&s_gm.acc_free);
    if (EPI == kNorm && a.ln_g) {  // two passes over the thread's half; the halves meet at (mean, M2)
      const float mh = (sum.x + sum.y) * (1.0f / (float)H);
      float2 q0 = make_float2(0.f, 0.f), q1 = q0;
#pragma unroll 8
      for (int i = 0; i < H; i += 4) {
        const float4 v = lds4(staging + stage_off<N>(row, (c0 + i) / 4));
        const float2 d0 = __fadd2_rn(make_float2(v.x, v.y), make_float2(-mh, -mh)), d1 = __fadd2_rn(make_float2(v.z, v.w), make_float2(-mh, -mh));
        q0 = __ffma2_rn(d0, d0, q0);
        q1 = __ffma2_rn(d1, d1, q1);
      }
      s_gm.stat[half][row] = make_float2(mh, (q0.x + q0.y) + (q1.x + q1.y));
      asm volatile("bar.sync %0, 64;" ::"r"(2 + ((tid >> 5) & 3)) : "memory");
      const float2 s0 = s_gm.stat[0][row], s1 = s_gm.stat[1][row];
      const float mean = 0.5f * (s0.x + s1.x), d = 0.5f * (s0.x - s1.x);
      const float inv = rsqrtf((s0.y + s1.y + (float)N * (d * d)) / (float)N + a.eps);
#pragma unroll 8
      for (int i = 0; i < H; i += 4) {
        const uint32_t at = staging + stage_off<N>(row, (c0 + i) / 4);
        const float4 v = lds4(at), g4 = lds4(par + 4 * (192 + i)), b4 = lds4(par + 4 * (384 + i));
        sts4(at, make_float4(fmaf((v.x - mean) * inv, g4.x, b4.x), fmaf((v.y - mean) * inv, g4.y, b4.y),
                             fmaf((v.z - mean) * inv, g4.z, b4.z), fmaf((v.w - mean) * inv, g4.w, b4.w)));
      }
    }
    if (bar_or(1, kEpiThreads, *abort_flag != 0)) break;
    const Pass to = {ps.s_first, ps.s_end, ps.row0, EPI == kNorm && s_gm.leave_y ? 0 : ps.row_end};
#pragma unroll 4
    for (int p = 0; p < P; ++p) {
      const int rr = r16 + kRows * p, pos = p0 + rr;
      const int v = a.out ? (pos >= to.row0 && pos < to.row_end ? pos : -1) : voxel_at(a, to, pos);
      float4* dst = reinterpret_cast<float4*>(a.out ? a.out + (size_t)v * a.ldo + nt * N : a.y + (size_t)v * N) + c16;
      float4 f[J];
#pragma unroll
      for (int j = 0; j < J; ++j) f[j] = lds4(staging + stage_off<N>(rr, c16 + 16 * j));
#pragma unroll
      for (int j = 0; j < J; ++j)
        if (v >= 0) dst[16 * j] = f[j];
    }
  }
  if (threadIdx.x == 0 && *abort_flag) {
    atomicOr(a.status, DSVT_STATUS_TIMEOUT);
    atomicExch(a.status + 2, __ldcg(a.status + 1));
  }
}

// out = epilogue(rows W^T + bias): tiles of 128 positions x N outputs, persistent blocks; a tile's epilogue runs under the
// next one's products.
template <int N, int EPI, bool PE>
__global__ void __launch_bounds__(kThreads, 1) f32_gemm_kernel(const __grid_constant__ GemmArgs a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const uint32_t sbase = smem_u32(smem_raw);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  if (tid == 0) {
    s_gm.abort_flag = 0;
    for (int i = 0; i < kSt; ++i) { mbar_init(&s_gm.full[i], kConvThreads + 1); mbar_init(&s_gm.empty[i], 1); }
    mbar_init(&s_gm.acc_full, 1);
    mbar_init(&s_gm.acc_free, kEpiThreads);
    mbar_init(&s_gm.chunk_full, 1);
    mbar_init(&s_gm.chunk_free, kEpiThreads);
    mbar_init(&s_gm.drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_gm.tmem)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const int ns = a.k / kKS;
  if (warp == kCopyWarp) {
    if ((tid & 31) == 0) copy_role<N>(a, sbase, ns);
    __syncwarp();
  } else {
    pdl_wait();  // everything below may read what earlier kernels of the stream wrote
    pdl_launch();
    if (EPI == kBias && blockIdx.x == 0 && tid == 0) *a.counter = 0;
    const Pass ps = *a.pass;
    const int tiles = num_tiles(a);
    if (warp == kMmaWarp) {
      mma_role<N>(sbase, tiles, ns);
    } else if (warp >= kConvWarp) {
      convert_role<N, PE>(a, ps, sbase, tiles, ns);
    } else {
      if (EPI == kNorm)
        for (int i = tid; i < 2 * N; i += kEpiThreads) {
          const float* v = i < N ? a.ln_g : a.ln_b;
          s_gm.par[i < N ? 192 + i : 384 + i - N] = v ? __ldg(v + (i < N ? i : i - N)) : 0.f;
        }
      epilogue_role<N, EPI>(a, ps, sbase + Sm<N>::staging, tiles);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_gm.tmem), "r"(kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------------------------------------
// Preparation: parts of the weights, row lists and passes
// ---------------------------------------------------------------------------------------------
struct WeightJob {
  const float* w;       // [rows][k]
  unsigned char* parts;
  int32_t rows, k, tile;  // outputs of a tile of the product
};
struct ListJob {
  const int32_t *table, *num_sets, *rowoff;
  int32_t* list;  // [passes][rows]: voxel of each local position (-1: none)
  Pass* pass;     // [passes]
  int32_t cap_sets, tau, passes;
};
constexpr int kPrepLayers = 2;  // layers whose weights are prepared at a time
struct PrepArgs {
  WeightJob weight[4 * kPrepLayers];
  ListJob job[2];
  int32_t n, pass_rows, rows;  // positions whose sets a pass takes; entries of a pass (a set may reach past the former)
  int32_t n_weights, new_call;
  int32_t* status;
};

// Eight weights -> their place in the tile's and stage's block: [part][8-column chunk][row][16 bytes] (see Sm).
__device__ __forceinline__ void prepare_weights(const WeightJob& j) {
  const int k8 = j.k / 8, units = j.rows * k8;
  for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < units; u += gridDim.x * blockDim.x) {
    const int n = u / k8, q = u - n * k8, nt = n / j.tile, r = n - nt * j.tile, s = q / (kKS / 8), c = q - s * (kKS / 8);
    const float4* src = reinterpret_cast<const float4*>(j.w + (size_t)n * j.k) + 2 * q;
    uint2 h[2], m[2], l[2];
    split4(__ldg(src), h[0], m[0], l[0]);
    split4(__ldg(src + 1), h[1], m[1], l[1]);
    const size_t part = (size_t)(kKS / 8) * j.tile * 16;
    unsigned char* to = j.parts + ((size_t)nt * (j.k / kKS) + s) * kParts * part + ((size_t)c * j.tile + r) * 16;
    *reinterpret_cast<uint4*>(to) = make_uint4(h[0].x, h[0].y, h[1].x, h[1].y);
    *reinterpret_cast<uint4*>(to + part) = make_uint4(m[0].x, m[0].y, m[1].x, m[1].y);
    *reinterpret_cast<uint4*>(to + 2 * part) = make_uint4(l[0].x, l[0].y, l[1].x, l[1].y);
  }
}

// Whether set s claims the positions up to the next set's first and can have as many rows.
__device__ __forceinline__ bool sound_claim(int off, int end, int tau) { return off >= 0 && end > off && (int64_t)end - off <= tau; }

// Whether position x lies in the claim of a set that writes it.
__device__ __noinline__ bool claimed(const ListJob& j, int S, int x) {
  int lo = 0, hi = S;  // the first set that starts behind x
  while (lo < hi) { const int m = (lo + hi) >> 1; if (__ldg(j.rowoff + m) <= x) lo = m + 1; else hi = m; }
  if (lo == 0) return false;
  const int off = __ldg(j.rowoff + lo - 1), end = __ldg(j.rowoff + lo);
  return off <= x && x < end && sound_claim(off, end, j.tau);
}

// A set belongs to the pass its first row lies in: pass p takes the sets whose row offset is in [p R, (p + 1) R), R =
// pass_rows, and a position's place in it is its row offset less p R.  One warp per set writes the set's distinct slots
// (Eq. 4); the first blocks find the passes' first and last sets.
// The lists hold what an earlier call left.  A set whose claim is not sound is skipped (its positions become -1), and every set
// writes its claim in each list that holds it: of the positions between two sets' first rows each lies in the claim of some set
// between them, whatever the offsets are, so that a pass has no position that nobody wrote.
__global__ void __launch_bounds__(256) f32_prepare_kernel(const __grid_constant__ PrepArgs a) {
  pdl_enter();
  if (a.new_call && (blockIdx.x | blockIdx.y | threadIdx.x) == 0) atomicAdd(a.status + 1, 1);
  if ((int)blockIdx.y < a.n_weights) {
    prepare_weights(a.weight[blockIdx.y]);
    return;
  }
  const ListJob& j = a.job[blockIdx.y - a.n_weights];
  const int lane = threadIdx.x & 31;
  const int S = min(__ldg(j.num_sets), j.cap_sets), R = a.pass_rows;
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < j.passes; p += gridDim.x * blockDim.x) {
    int cut[2];
    for (int e = 0; e < 2; ++e) {
      int lo = 0, hi = max(S, 0);
      const int64_t at = (int64_t)(p + e) * R;
      while (lo < hi) { const int m = (lo + hi) >> 1; if (__ldg(j.rowoff + m) < at) lo = m + 1; else hi = m; }
      cut[e] = lo;
    }
    Pass ps = {cut[0], cut[1], 0, 0};
    if (cut[1] > cut[0]) {
      const int64_t o = (int64_t)p * R;
      ps.row0 = (int)max((int64_t)0, __ldg(j.rowoff + cut[0]) - o);
      ps.row_end = (int)min((int64_t)a.rows, max((int64_t)0, __ldg(j.rowoff + cut[1]) - o));
    }
    j.pass[p] = ps;
  }
  const int warps = gridDim.x * (blockDim.x >> 5);
  for (int s = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); s < S; s += warps) {
    const int off = __ldg(j.rowoff + s), end = __ldg(j.rowoff + s + 1);
    const bool sound = sound_claim(off, end, j.tau);
    const int p = sound ? off / R : -1, cap = sound ? end - off : 0;
    if (!sound && lane == 0) atomicOr(a.status, DSVT_STATUS_BAD_INDEX);
    // (a sound claim that does not cross into another pass's list does nothing here)
    const int lo = max(off, 0);
    const int64_t last = min((int64_t)end, (int64_t)j.passes * R + kTM);
    for (int q = max(lo - kTM, 0) / R; q < j.passes && (int64_t)q * R < last; ++q) {
      if (q == p) continue;
      const int64_t o = (int64_t)q * R, to = min(last, o + a.rows);
      for (int64_t x = max((int64_t)lo, o) + lane; x < to; x += 32)
        if (sound || !claimed(j, S, (int)x)) j.list[(size_t)q * a.rows + (x - o)] = -1;
    }
    if (!sound || p >= j.passes) continue;  // (more rows than voxels: some voxels are in several sets; the general kernel takes these)
    int32_t* to = j.list + (size_t)p * a.rows + (off - p * R);
    const int32_t* row = j.table + (size_t)s * j.tau;
    int cnt = 0;
    bool bad = false;
    for (int k0 = 0; k0 < j.tau; k0 += 32) {
      const int k = k0 + lane;
      int v = -1;
      bool uniq = false;
      if (k < j.tau) {
        v = __ldg(row + k);
        uniq = k == 0 || v != __ldg(row + k - 1);
      }
      const unsigned bal = __ballot_sync(0xffffffffu, uniq);
      const int pos = cnt + __popc(bal & ((1u << lane) - 1u));
      if (uniq && pos < cap) {
        if (v < 0 || v >= a.n) { bad = true; v = -1; }
        to[pos] = v;
      }
      cnt += __popc(bal);
    }
    for (int k = cnt + lane; k < cap; k += 32) to[k] = -1;
    if (__any_sync(0xffffffffu, bad || cnt != cap) && lane == 0) atomicOr(a.status, DSVT_STATUS_BAD_INDEX);
  }
}

// ---------------------------------------------------------------------------------------------
// Attention
// ---------------------------------------------------------------------------------------------
struct AttendArgs {
  float* qkv;  // [position][Q | K | V]; the output replaces Q
  int32_t* counter;  // units drawn so far (set to zero by the QKV product)
  const int32_t *rowoff, *list;
  const Pass* pass;
  const float* rpb;
  const int4* coords;
  int32_t* status;
  int32_t origin, pass_rows, n, tau;
  int32_t rb_len, rb_sx, rb_sy, rb_centre, rb_ext[3];  // relative position bias (see dsvt_layer_params)
};

constexpr int kAttThreads = 128;
constexpr float kLog2e = 1.4426950408889634f;
__host__ __device__ constexpr int warp_floats(int d, int tau) { return tau * (2 * d) + (tau + 3) / 4 * 4; }  // keys | values, linear coordinates

// The attention of Q query rows per lane of a half warp (rows r0 + lane, r0 + 16 + lane); the two halves take every other
// key, K at a time with a running softmax, and meet at the end.  Scores stay in natural units up to the difference from the
// maximum: times log2(e), a bias of the lowest float would be -inf, and a row of such biases 0 / 0.  Rounding the scaled difference
// costs a weight e^-a at most a e^-a 2^-24 <= 0.4 x 2^-24 of the largest one.  Two layers with expf instead (12 seeds, 2-norm): attention
// alone 1.20e-7 for 1.14e-7 (C = 128) and 1.40e-7 for 1.33e-7 (192), full layers 2.24e-7 for 2.21e-7, and 254 us for 249 (12,345 pillars).
template <int D, int Q, bool RPB>
__device__ __forceinline__ void attend_rows(float* qkv, int ld, const float* kv, const int* lin, int rows, int r0, float scale,
                                            const float* rpb, int rb_len, int rb_centre) {
  constexpr int K = Q == 2 && D == 32 ? 2 : 4;
  const int lane = threadIdx.x & 31, par = lane >> 4, l16 = lane & 15;
  float2 q[Q][D / 2], o[Q][D / 2];
  float mx[Q], den[Q];
  float* qrow[Q];
  int r[Q];
#pragma unroll
  for (int w = 0; w < Q; ++w) {
    r[w] = min(r0 + 16 * w + l16, rows - 1);
    qrow[w] = qkv + (size_t)r[w] * ld;
    mx[w] = -INFINITY;
    den[w] = 0.f;
#pragma unroll
    for (int c = 0; c < D / 4; ++c) {
      const float4 v = __ldcg(reinterpret_cast<const float4*>(qrow[w]) + c);
      q[w][2 * c] = make_float2(v.x, v.y);
      q[w][2 * c + 1] = make_float2(v.z, v.w);
      o[w][2 * c] = o[w][2 * c + 1] = make_float2(0.f, 0.f);
    }
  }
  if (r0 == 0) {  // keys and values
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
  }
#pragma unroll 1
  for (int k0 = par; k0 < rows + par; k0 += 2 * K) {  // (both halves alike)
    float lg[Q][K];
#pragma unroll
    for (int u = 0; u < K; ++u) {
      const int k = min(k0 + 2 * u, rows - 1);
      float2 s[Q];
#pragma unroll
      for (int w = 0; w < Q; ++w) s[w] = make_float2(0.f, 0.f);
#pragma unroll
      for (int c = 0; c < D / 4; ++c) {
        const float4 v = *reinterpret_cast<const float4*>(kv + k * (2 * D) + 4 * c);
#pragma unroll
        for (int w = 0; w < Q; ++w) {
          s[w] = __ffma2_rn(q[w][2 * c], make_float2(v.x, v.y), s[w]);
          s[w] = __ffma2_rn(q[w][2 * c + 1], make_float2(v.z, v.w), s[w]);
        }
      }
#pragma unroll
      for (int w = 0; w < Q; ++w) {
        lg[w][u] = (s[w].x + s[w].y) * scale;
        if (RPB) {
          const int idx = lin[r[w]] - lin[k] + rb_centre;
          lg[w][u] += __ldg(rpb + min(max(idx, 0), rb_len - 1));
        }
        if (k0 + 2 * u >= rows) lg[w][u] = -INFINITY;
      }
    }
#pragma unroll
    for (int w = 0; w < Q; ++w) {
      float nm = mx[w];
#pragma unroll
      for (int u = 0; u < K; u += 2) nm = fmaxf(nm, fmaxf(lg[w][u], lg[w][u + 1]));
      const float from = nm == -INFINITY ? 0.f : nm;  // (a bias may rule out all keys so far)
      const float al = ex2_approx((mx[w] - from) * kLog2e);  // (2^-inf = 0)
      mx[w] = nm;
      float sum = 0.f;
#pragma unroll
      for (int u = 0; u < K; ++u) {
        lg[w][u] = ex2_approx((lg[w][u] - from) * kLog2e);
        sum += lg[w][u];
      }
      den[w] = fmaf(den[w], al, sum);
#pragma unroll
      for (int c = 0; c < D / 2; ++c) o[w][c] = __fmul2_rn(o[w][c], make_float2(al, al));
    }
#pragma unroll
    for (int u = 0; u < K; ++u) {
      const int k = min(k0 + 2 * u, rows - 1);
#pragma unroll
      for (int c = 0; c < D / 4; ++c) {
        const float4 v = *reinterpret_cast<const float4*>(kv + k * (2 * D) + D + 4 * c);
#pragma unroll
        for (int w = 0; w < Q; ++w) {
          o[w][2 * c] = __ffma2_rn(make_float2(lg[w][u], lg[w][u]), make_float2(v.x, v.y), o[w][2 * c]);
          o[w][2 * c + 1] = __ffma2_rn(make_float2(lg[w][u], lg[w][u]), make_float2(v.z, v.w), o[w][2 * c + 1]);
        }
      }
    }
  }
#pragma unroll
  for (int w = 0; w < Q; ++w) {  // (the second half has no keys if the set holds one row)
    const float nm = fmaxf(mx[w], __shfl_xor_sync(0xffffffffu, mx[w], 16));
    const float al = nm == -INFINITY ? 0.f : ex2_approx((mx[w] - nm) * kLog2e);
    den[w] *= al;
    const float inv = al / (den[w] + __shfl_xor_sync(0xffffffffu, den[w], 16));
    const bool on = r0 + 16 * w + l16 < rows;
#pragma unroll
    for (int c = 0; c < D / 4; ++c) {
      const float v[4] = {o[w][2 * c].x * inv, o[w][2 * c].y * inv, o[w][2 * c + 1].x * inv, o[w][2 * c + 1].y * inv};
      float4 out;
      out.x = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 16);
      out.y = v[1] + __shfl_xor_sync(0xffffffffu, v[1], 16);
      out.z = v[2] + __shfl_xor_sync(0xffffffffu, v[2], 16);
      out.w = v[3] + __shfl_xor_sync(0xffffffffu, v[3], 16);
      if (on && (c & 1) == par) reinterpret_cast<float4*>(qrow[w])[c] = out;  // (each half stores half of the row)
    }
  }
}

// One warp per (set, head), drawn from a counter (sets differ in size by as much as 36 times): keys and values of the head in
// shared memory, read as broadcasts.
template <int C, int D, bool RPB>
__global__ void __launch_bounds__(kAttThreads, D == 16 ? 4 : 3) f32_attend_kernel(const AttendArgs a) {
  extern __shared__ __align__(16) float smem[];
  constexpr int kHeads = C / D, ld = 3 * C;
  pdl_wait();
  pdl_launch();
  const int lane = threadIdx.x & 31;
  float* kv = smem + (size_t)(threadIdx.x >> 5) * warp_floats(D, a.tau);  // [row][K | V]
  int* lin = reinterpret_cast<int*>(kv + a.tau * 2 * D);
  const Pass ps = *a.pass;
  const float scale = rsqrtf((float)D);
  int h, base, m;
  auto draw = [&]() -> bool {  // the next unit: head, first position, rows
    int u = 0;
    if (lane == 0) u = atomicAdd(a.counter, 1);
    u = __shfl_sync(0xffffffffu, u, 0);
    const int s = ps.s_first + u / kHeads;
    if (s >= ps.s_end) return false;
    h = u % kHeads;
    const int off = __ldg(a.rowoff + s), end = __ldg(a.rowoff + s + 1);
    base = off - a.origin;
    m = sound_claim(off, end, a.tau) ? end - off : 0;
    if (base < 0 || base >= a.pass_rows) m = 0;  // (row offsets that do not ascend)
    return true;
  };
  bool more = draw();
  while (more) {
    const int hd = h, rows = m, first = base;
    float* qkv = a.qkv + (size_t)first * ld + hd * D;
    for (int i = lane; i < rows * (D / 2); i += 32) {
      const int r = i / (D / 2), c = i - r * (D / 2);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(kv + 4 * i)),
                   "l"(qkv + (size_t)r * ld + (c < D / 4 ? C + 4 * c : 2 * C + 4 * c - D)) : "memory");
    }
    if (RPB) {
      int lo[3] = {INT_MAX, INT_MAX, INT_MAX}, hi[3] = {INT_MIN, INT_MIN, INT_MIN};
      for (int r = lane; r < rows; r += 32) {
        const int v = __ldg(a.list + first + r);
        int l = 0;
        if ((unsigned)v < (unsigned)a.n) {
          const int4 c = __ldg(a.coords + v);
          lo[0] = min(lo[0], c.y); hi[0] = max(hi[0], c.y);
          lo[1] = min(lo[1], c.z); hi[1] = max(hi[1], c.z);
          lo[2] = min(lo[2], c.w); hi[2] = max(hi[2], c.w);
          l = c.y * a.rb_sx + c.z * a.rb_sy + c.w;
        }
        lin[r] = l;
      }
      if (hd == 0) {  // a set spread wider than the table's extent is reported
        bool wide = false;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int l = -dsvt_fma::warp_max_int(-lo[q]), u = dsvt_fma::warp_max_int(hi[q]);
          wide |= u >= l && u - l > a.rb_ext[q] - 1;
        }
        if (wide && lane == 0) atomicOr(a.status, DSVT_STATUS_BAD_INDEX);
      }
    }
    more = draw();  // (its round trips under this unit's)
    const float* rpb = RPB ? a.rpb + (size_t)hd * a.rb_len : nullptr;
    int r0 = 0;
    for (; rows - r0 > 16; r0 += 32) attend_rows<D, 2, RPB>(qkv, ld, kv, lin, rows, r0, scale, rpb, a.rb_len, a.rb_centre);
    if (r0 < rows) attend_rows<D, 1, RPB>(qkv, ld, kv, lin, rows, r0, scale, rpb, a.rb_len, a.rb_centre);
    __syncwarp();  // (keys and values are read)
  }
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
template <int N, int EPI, bool PE>
int launch_gemm(dsvt_ctx* ctx, const GemmArgs& g, int64_t rows) {
  constexpr unsigned flag = 1u << (8 + 4 * (N / 64 - 1) + (PE ? 3 : EPI));
  if (!(ctx->attr_flags & flag)) {  // (once per context: the attribute belongs to its device)
    DSVT_CUDA_TRY(ctx, cudaFuncSetAttribute(f32_gemm_kernel<N, EPI, PE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Sm<N>::bytes));
    ctx->attr_flags |= flag;
  }
  int64_t grid = dsvt_ceil_div(rows, kTM) * g.tiles_n;
  if (grid > ctx->sm_count) grid = ctx->sm_count;
  DSVT_CUDA_TRY(ctx, launch_pdl(f32_gemm_kernel<N, EPI, PE>, dim3((unsigned)grid), dim3(kThreads), Sm<N>::bytes, ctx->stream, g));
  DSVT_LAUNCHED(ctx);
  return DSVT_OK;
}

template <int EPI, bool PE = false>
int launch_gemm_n(dsvt_ctx* ctx, int N, const GemmArgs& g, int64_t rows) {
  return N == 192   ? launch_gemm<192, EPI, PE>(ctx, g, rows)
         : N == 128 ? launch_gemm<128, EPI, PE>(ctx, g, rows)
                    : launch_gemm<64, EPI, PE>(ctx, g, rows);
}

template <int C, int D, bool RPB>
int launch_attend(dsvt_ctx* ctx, const AttendArgs& a, int64_t rows) {
  constexpr unsigned flag = 1u << (20 + 2 * (C / 64 - 1 + (D == 32 ? 2 : 0)) + (RPB ? 1 : 0));
  const size_t warp_bytes = 4 * (size_t)warp_floats(D, a.tau);
  if (!(ctx->attr_flags & flag)) {
    DSVT_CUDA_TRY(ctx, cudaFuncSetAttribute(f32_attend_kernel<C, D, RPB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 104 * 1024));
    ctx->attr_flags |= flag;
  }
  constexpr int kWarps = kAttThreads / 32;
  const int64_t most = (D == 16 ? 4 : 3) * (int64_t)ctx->sm_count, units = dsvt_ceil_div(rows * (C / D), kWarps);  // (a set has a row at least)
  DSVT_CUDA_TRY(ctx, launch_pdl(f32_attend_kernel<C, D, RPB>, dim3((unsigned)(units < most ? units : most)), dim3(kAttThreads),
                                kWarps * warp_bytes, ctx->stream, a));
  DSVT_LAUNCHED(ctx);
  return DSVT_OK;
}

template <bool RPB>
int attend(dsvt_ctx* ctx, const AttendArgs& a, int C, int D, int64_t rows) {
  if (C == 192) return launch_attend<192, 24, RPB>(ctx, a, rows);
  if (C == 64) return launch_attend<64, 16, RPB>(ctx, a, rows);
  return D == 16 ? launch_attend<128, 16, RPB>(ctx, a, rows) : launch_attend<128, 32, RPB>(ctx, a, rows);
}

// Outputs of a tile of the first MLP product.
int mlp_tile(int hidden) { return hidden % 128 == 0 ? 128 : hidden % 192 == 0 ? 192 : 64; }

size_t layer_weights(int C, int hidden) { return (size_t)(4 * C + 2 * hidden) * C * 2 * kParts; }  // bytes of their parts

// The workspace is the partition's, which holds nothing between calls: its bitmaps and their ranks (33 MB) for the weights' parts
// and the rows of a pass, its sort buffers for the two row lists and their passes.
struct Work {
  unsigned char* parts;
  float* rows;             // [entries][3 C]
  int32_t* list[2];        // [max_passes][entries]
  Pass* pass[2];
  int64_t pass_rows, entries;  // positions whose sets a pass takes, and with room for the last set
};

Work workspace(const dsvt_ctx* ctx, int C, int64_t n) {
  Work w;
  w.parts = reinterpret_cast<unsigned char*>(ctx->bm_zero);
  const size_t parts = (kPrepLayers * layer_weights(C, 2 * C) + 255) / 256 * 256;
  const size_t bytes = (size_t)(reinterpret_cast<unsigned char*>(ctx->bm_wordrank + 2 * ctx->bm_words) - w.parts);
  w.rows = reinterpret_cast<float*>(w.parts + parts);
  // As few passes as the room allows for n rows, whatever the context was made for (12,345 pillars in a context for 40,000 took
  // 418 us in two passes, and 257 in one); several of about the same size, a single one with the room there is, for tables whose
  // voxels are in several sets.
  const int64_t most = (int64_t)((bytes - parts) / (3 * sizeof(float) * C)) / kTM * kTM - kTM;
  const int64_t passes = dsvt_ceil_div(n, most), share = passes > 1 ? dsvt_ceil_div(n, passes) : ctx->max_voxels < most ? ctx->max_voxels : most;
  w.pass_rows = dsvt_ceil_div(share, kTM) * kTM;
  w.entries = w.pass_rows + kTM;
  w.list[0] = reinterpret_cast<int32_t*>(ctx->keys[0]);
  w.list[1] = ctx->vals[0];
  for (int i = 0; i < 2; ++i) w.pass[i] = reinterpret_cast<Pass*>(w.list[i] + passes * w.entries);
  return w;
}

bool same_table(const dsvt_fused_args& a, const dsvt_fused_args& b) {
  return a.table == b.table && a.rowoff == b.rowoff && a.num_sets == b.num_sets && a.cap_sets == b.cap_sets && a.p.set_size == b.p.set_size;
}

}  // namespace

bool dsvt_layer_f32_supported(const dsvt_fused_args& a) {
  const dsvt_layer_params& p = a.p;
  if (p.precision != DSVT_FP32) return false;
  const int d = p.C / p.heads, hidden = a.attention_only ? 0 : p.hidden;
  if (hidden % 64 != 0) return false;
  if (p.C == 192) return d == 24 && p.set_size <= 64;
  return ((p.C == 128 && (d == 16 || d == 32)) || (p.C == 64 && d == 16)) && p.set_size <= 96;
}

// Preparation for layers[0 .. kPrepLayers): the parts of their weights, and the row lists of the (at most kPrepLayers) tables
// they run on.  `list` receives which of the two lists each layer uses; returns how many layers have been prepared.
static int prepare(dsvt_ctx* ctx, const Work& ws, const dsvt_fused_args* layers, int n_layers, bool new_call, int (&list)[kPrepLayers], int* prepared) {
  const int64_t R = ws.pass_rows;
  PrepArgs a = {};
  a.n = layers[0].n; a.pass_rows = (int32_t)R; a.rows = (int32_t)ws.entries; a.status = ctx->status; a.new_call = new_call;
  const int count = n_layers < kPrepLayers ? n_layers : kPrepLayers;
  int n_lists = 0;
  int64_t units = 0;
  unsigned char* parts = ws.parts;
  for (int i = 0; i < count; ++i) {
    const dsvt_fused_args& l = layers[i];
    const dsvt_layer_params& p = l.p;
    const int hidden = l.attention_only ? 0 : p.hidden;
    const WeightJob w[4] = {{static_cast<const float*>(p.W_qkv), nullptr, 3 * p.C, p.C, p.C}, {static_cast<const float*>(p.W_o), nullptr, p.C, p.C, p.C},
                            {static_cast<const float*>(p.W_1), nullptr, hidden, p.C, mlp_tile(hidden)}, {static_cast<const float*>(p.W_2), nullptr, p.C, hidden, p.C}};
    for (int q = 0; q < (hidden > 0 ? 4 : 2); ++q) {
      a.weight[a.n_weights] = w[q];
      a.weight[a.n_weights++].parts = parts;
      parts += (size_t)w[q].rows * w[q].k * 2 * kParts;
    }
    list[i] = -1;
    for (int q = 0; q < i; ++q)
      if (same_table(layers[q], l)) list[i] = list[q];
    if (list[i] >= 0) continue;
    const int64_t slots = (int64_t)l.cap_sets * p.set_size, bound = slots < l.n ? slots : l.n;
    if (bound > units) units = bound;
    ListJob& j = a.job[n_lists];
    j.table = l.table; j.num_sets = l.num_sets; j.rowoff = l.rowoff; j.cap_sets = l.cap_sets; j.tau = p.set_size;
    j.passes = (int32_t)dsvt_ceil_div(bound, R);
    j.list = ws.list[n_lists];
    j.pass = ws.pass[n_lists];
    list[i] = n_lists++;
  }
  int64_t blocks = dsvt_ceil_div(units, 8);
  const int64_t most = 2 * (int64_t)ctx->sm_count, least = 16;
  blocks = blocks > most ? most : blocks < least ? least : blocks;
  DSVT_CUDA_TRY(ctx, launch_pdl(f32_prepare_kernel, dim3((unsigned)blocks, (unsigned)(a.n_weights + n_lists)), dim3(256), 0, ctx->stream, a));
  DSVT_LAUNCHED(ctx);
  *prepared = count;
  return DSVT_OK;
}

int dsvt_launch_layers_f32(dsvt_ctx* ctx, const dsvt_fused_args* layers, int n_layers, bool new_call) {
  const Work ws = workspace(ctx, layers[0].p.C, layers[0].n);
  const int64_t R = ws.pass_rows, E = ws.entries;
  int lists[kPrepLayers], first = 0, prepared = 0;  // layers [first, first + prepared) are prepared
  const unsigned char* parts = nullptr;
  for (int i = 0; i < n_layers; ++i) {
    if (i == first + prepared) {
      first = i;
      const int rc = prepare(ctx, ws, layers + i, n_layers - i, new_call && i == 0, lists, &prepared);
      if (rc != DSVT_OK) return rc;
      parts = ws.parts;
    }
    const dsvt_fused_args& a = layers[i];
    const dsvt_layer_params& p = a.p;
    const int C = p.C, hidden = a.attention_only ? 0 : p.hidden;
    const int64_t slots = (int64_t)a.cap_sets * p.set_size, bound = slots < a.n ? slots : a.n;
    const int passes = (int)dsvt_ceil_div(bound, R);
    const int32_t* list = ws.list[lists[i - first]];
    const Pass* pass = ws.pass[lists[i - first]];
    const unsigned char *w_o = parts + (size_t)3 * C * C * 2 * kParts, *w_1 = w_o + (size_t)C * C * 2 * kParts,
                        *w_2 = w_1 + (size_t)hidden * C * 2 * kParts;
    float* qkv = ws.rows;
    for (int q = 0; q < passes; ++q) {
      const int64_t rows = slots < E ? slots : E;  // (at most: how many there are is known on the device)
      GemmArgs g = {};
      g.x = a.x; g.pe = p.pe; g.pe_tiles = p.pe ? 2 : 0;
      g.list = list + (size_t)q * E; g.pass = pass + q; g.n = a.n; g.status = ctx->status; g.y = a.y; g.eps = p.ln_eps;
      g.w = parts; g.bias = p.b_qkv; g.k = C; g.tiles_n = 3; g.lda = C;
      g.out = qkv; g.ldo = 3 * C; g.counter = ctx->tc_counter + 2;
      int rc = p.pe ? launch_gemm_n<kBias, true>(ctx, C, g, rows) : launch_gemm_n<kBias>(ctx, C, g, rows);
      if (rc != DSVT_OK) return rc;
      AttendArgs t = {};
      t.qkv = qkv; t.rowoff = a.rowoff; t.list = g.list; t.pass = g.pass; t.status = ctx->status;
      t.origin = (int32_t)(q * R); t.pass_rows = (int32_t)R; t.n = a.n; t.tau = p.set_size;
      t.counter = ctx->tc_counter + 2;
      if (p.rpb) {
        const int L = p.rpb_extent[0], W = p.rpb_extent[1], H = p.rpb_extent[2];
        t.rpb = p.rpb; t.coords = reinterpret_cast<const int4*>(p.coords);
        t.rb_sy = 2 * H - 1;
        t.rb_sx = (2 * W - 1) * t.rb_sy;
        t.rb_len = (2 * L - 1) * t.rb_sx;
        t.rb_centre = (L - 1) * t.rb_sx + (W - 1) * t.rb_sy + (H - 1);
        t.rb_ext[0] = L; t.rb_ext[1] = W; t.rb_ext[2] = H;
      }
      rc = p.rpb ? attend<true>(ctx, t, C, C / p.heads, rows) : attend<false>(ctx, t, C, C / p.heads, rows);
      if (rc != DSVT_OK) return rc;
      g.a = qkv; g.lda = 3 * C; g.pe_tiles = 0;
      g.w = w_o; g.bias = p.b_o; g.tiles_n = 1;
      g.add_x = !a.attention_only;
      g.ln_g = a.attention_only ? nullptr : p.ln1_g; g.ln_b = p.ln1_b;
      g.out = hidden > 0 ? qkv : nullptr;  // (x1 takes the place of the tile's operand rows)
      rc = launch_gemm_n<kNorm>(ctx, C, g, rows);
      if (rc != DSVT_OK) return rc;
      if (hidden == 0) continue;
      const int nf = mlp_tile(hidden);
      g.w = w_1; g.bias = p.b_1; g.tiles_n = hidden / nf; g.add_x = 0;
      g.out = qkv + C;  // (keys and values are dead)
      rc = launch_gemm_n<kGelu>(ctx, nf, g, rows);
      if (rc != DSVT_OK) return rc;
      g.a = qkv + C;
      g.w = w_2; g.bias = p.b_2; g.k = hidden; g.tiles_n = 1;
      g.res = qkv; g.ldr = 3 * C; g.ln_g = p.ln2_g; g.ln_b = p.ln2_b;
      g.out = nullptr;
      rc = launch_gemm_n<kNorm>(ctx, C, g, rows);
      if (rc != DSVT_OK) return rc;
    }
    parts += layer_weights(C, hidden);
    // a table may hold more rows than there are voxels (voxels in several sets): the sets past the passes
    if (slots > passes * R) {
      const int rc = dsvt_launch_layer_fma(ctx, a, (int64_t)passes * R, ctx->status + 1);
      if (rc != DSVT_OK) return rc;
    }
  }
  return DSVT_OK;
}
