// Fused DSVT layers on the 5th-generation tensor cores (tcgen05 + TMEM), bfloat16 operands, fp32
// accumulation: gather (Eq. 4) -> QKV projection -> per-set multi-head attention (Eq. 5) -> output
// projection -> residual + LayerNorm -> MLP with GELU -> residual + LayerNorm -> scatter (App. B.1.1).
//
// One launch runs a chain of layers (one layer, the two layers of a block, or every block of a stage): layer 0
// reads x and writes y, the later layers run in place on y.  Whole sets are packed into tiles of at most 128
// distinct rows (the UMMA M) by the partition's tile plan.  The persistent CTAs (one per SM) draw tiles from a
// global counter, all tiles of layer 0 first, then layer 1, ...; a tile of layer l may be gathered as soon as
// each of its rows carries layer l - 1's completion stamp (one int per voxel, written after the row's store), so
// no CTA ever waits for a whole layer to end, and a launch pays its start-up and its tail once per chain rather
// than once per layer.  Tiles are taken in counter order and a tile only ever waits for tiles with a smaller
// number, so the tile with the smallest unfinished number can always run: no CTA has to be resident for another
// to make progress.
//
// Roles (640 threads): warps 0-15 compute (gather, TMEM epilogues, attention); warp 16 is the scheduler
// and TMA producer: it draws tiles, publishes them through a two-entry ring, two ahead, and streams the layer's
// weight matrices through a three-stage shared-memory ring with plain (single-CTA) TMA loads; warp 17
// allocates TMEM and issues the tcgen05.mma instructions; warp 18 builds the next tile's row list
// while the current tile is computed and waits for its rows' stamps; warp 19 stamps a finished tile's rows.
// The compute warps gather the next tile's rows as soon as the current tile's MMAs have stopped reading the A
// operand (if its rows are ready by then), so that its first projections overlap the current tile's tail.
//
// The projections of a layer are chunks of at most 192 output columns (K, V, Q, O, MLP-1 in pieces of
// 128 or 64 hidden columns, MLP-2), accumulated in TMEM (map at Tm) so the
// tensor pipe works on one chunk while the compute warps drain another.  The fp32 residual stream never
// leaves the chip inside a layer: x is staged in shared memory for the first residual, and
// x1 + b_2 = LN1(x + attention) + b_2 is parked in TMEM, where MLP-2 accumulates on top of it.  x1 and the MLP hidden
// are A operands in TMEM, the hidden one piece at a time: MLP-2 of a piece runs under the GELU of the next, and the
// tensor pipe reads half the shared memory it would need for both operands.
//
// Attention runs on the tensor cores too: per head, S = Q K^T over the whole tile (128 x 128) in TMEM, softmax with a
// row per thread, P back to TMEM as a bf16 A operand, O = P V.  Sets are kept apart inside the product: spare K
// columns carry a code of the row's set (see write_codes), which adds exactly zero to a score inside a set and -2^100
// to one across sets.  The products beyond a set cost the tensor pipe 3 k cycles per tile; in exchange the softmax has
// no shuffles, no per-element mask and 16 independent elements per step.
//
// Operand layouts in shared memory: the gathered rows and the weights use the K-major 128-byte-swizzled layout
// (64 bf16 columns per 128-byte row, 8-row groups of 1024 bytes, 16-byte chunk index XORed with (row & 7)).  Q, K, V
// and the attention output are unswizzled and chunk-major, [8-column chunk][128 rows][16 bytes]: a row per thread
// writes it without bank conflicts, heads of 24 columns start on a chunk, and V needs no transposition (it is read
// N-major).
//
// Every wait (on an mbarrier, on a row stamp) is bounded; a wait that gives up raises DSVT_STATUS_TIMEOUT and
// all roles leave their loops.
#include <cuda.h>
#include <limits.h>

#include <mutex>
#include <new>
#include <type_traits>
#include <vector>

#include "dsvt_common.cuh"
#include "tc_ptx.cuh"

namespace {
using namespace dsvt_tc;

constexpr int kComputeWarps = 16;
constexpr int kComputeThreads = 32 * kComputeWarps;
constexpr int kTmaWarp = kComputeWarps, kMmaWarp = kComputeWarps + 1;
constexpr int kLoadWarp0 = kComputeWarps + 2, kLoadWarps = 1;  // row-list warp, one tile ahead
constexpr int kLoadThreads = 32 * kLoadWarps;
constexpr int kStampWarp = kLoadWarp0 + kLoadWarps;  // writes the completion stamps of a finished tile's rows
constexpr int kThreads = kComputeThreads + 64 + kLoadThreads + 32;
constexpr int kStages = 3;             // weight ring depth
constexpr int kStampPolls = 1 << 18;  // polls of a row's stamp, about a microsecond each
constexpr int kMaxIdle = 1 << 24;     // rounds of looks at the attention's barriers that find nothing to do
constexpr uint32_t kChunkBytes = kTM * 16;  // an 8-column chunk of an unswizzled operand
constexpr int kMaxLayers = DSVT_MAX_CHAIN_LAYERS;  // layers one launch can chain

// TMEM map (512 columns): K, then Q accumulate at 0, V at C; in the attention every group of four warps has 128 columns
// for S, P and O; then R = the last C columns: output projection, x1 + b_2 parked,
// MLP-2 on top of it; x1 as a bf16 A operand at 0; an MLP-1 accumulator piece (128 columns); an MLP hidden piece as a
// bf16 A operand (64).  The next tile's K starts once x1 and the last MLP-1 piece are dead, its V (which overlaps the
// hidden piece and, for C = 192, R) once R has been read.
template <int C>
struct Tm {
  static constexpr uint32_t k = 0, v = C, x1 = 0, acc = C / 2, h = C / 2 + 128, r = kTmemCols - C;
  static_assert(2 * C <= kTmemCols && h + 64 <= r, "TMEM");
};

struct TcGeom {
  int hidden, heads, tau;
  int NF;       // MLP piece: hidden columns (128 or 64)
  int n_f1;     // hidden / NF
  int mode;     // 0: attention only, 1: attention + residual + LN1, 2: full layer
  uint32_t off_a, off_kv, off_code, off_stage;  // byte offsets in the dynamic shared memory
  // relative position bias (rb_len == 0: none): entries per head, strides of the x and y offsets in the table,
  // index of the zero offset, extent of the table
  int rb_len, rb_sx, rb_sy, rb_centre, rb_ext[3];
};

// One layer of a launch's chain: weight tensor maps, per-layer vectors, and the set table the layer runs on.
struct alignas(64) TcLayer {
  CUtensorMap qkv, o, w1, w2;
  const float *b_qkv, *b_o, *b_1, *b_2, *ln1_g, *ln1_b, *ln2_g, *ln2_b, *rpb;
  const float* pe;  // positional term added to the input of the query and key maps, [n][C], or NULL
  const int32_t *table, *num_sets, *rowoff;
  int32_t cap_sets;
  float eps;
};

struct TcArgs {
  const float* x;        // input of layer 0
  float* y;              // output of every layer; input of the layers after the first
  const int4* coords;    // (b, x, y, z) per voxel: read only with a position bias
  int32_t n, n_layers;
  int32_t* counter;      // [0] next tile of the launch, [1] CTAs that have left; both zero between launches
  int32_t* row_stamp;    // [n] completion stamps (n_layers > 1)
  int32_t stamp_base;    // layer l's stamp is stamp_base + l + 1
  int32_t* status;
  TcGeom g;
  TcLayer layer[kMaxLayers];
};

// Vectors of the layer that stay in shared memory (float offsets; for b_o, b_1 and b_2 see LateOff).
template <int C>
struct ParOff {
  static constexpr int b_q = 0, b_v = C, ln1_g = 2 * C, ln1_b = 3 * C, ln2_g = 4 * C, ln2_b = 5 * C;  // no key bias
  static constexpr int vectors = 6;
};
// b_o, b_2 and b_1 lie where the set codes are during the attention, from the end of the attention to the last MLP-1
// piece (float offsets; copied with the x rows).
template <int C>
struct LateOff { static constexpr int b_o = 0, b_2 = C, b_1 = 2 * C; };

// Small shared state beside the big regions.  It fills whole kilobytes, so that the dynamic shared memory behind it
// starts on a 1024-byte boundary (with C = 192 there is no byte to spare for padding).
struct alignas(1024) Misc {
  // weight ring; accumulators K / Q / MLP-1, V, R (see Tm); operand hand-offs
  unsigned long long full[kStages], empty[kStages], acc_full[3], acc_free[3];
  unsigned long long o_full;           // output projection done
  unsigned long long s_full[4], p_ready[4], ov_full[4], o_read[4];  // attention, one set per group of four warps
  unsigned long long h_ready, h_free;  // MLP hidden piece in TMEM: written / read by MLP-2
  unsigned long long a_ready;   // compute warps -> MMA: Q / attention output / x1 is in place
  unsigned long long x_ready;   // compute warps -> MMA: the gathered rows of a tile are in the A operand
  unsigned long long rl_ready[2];   // loader warp -> compute: row-list buffer b describes its next tile
  unsigned long long dep_ready[2];  // loader warp -> compute: the rows listed in buffer b carry the previous layer's stamp
  unsigned long long rl_free[2];    // compute + stamp warp -> loader warp: row-list buffer b is no longer read
  unsigned long long stored[2];     // compute -> stamp warp: the tile listed in buffer b has been stored
  unsigned long long drain;         // MMA issuer: every MMA issued before an abort has completed
  unsigned long long sched_full[2], sched_empty[2];
  uint32_t tmem_base;
  int abort_flag;
  int exit_at;   // tile iteration at which the compute warps left their loop (-1: still running; read by the stamp warp)
  int tile[2][5];  // ring of tiles: first set, number of sets (< 0: no more tiles), first row, rows, layer
  // the scheduler's view of the chain: tiles before the end of each layer, plan or not
  int tile_end[kMaxLayers];
  unsigned char lay_plan[kMaxLayers];
  // launch constants, written once before the roles start: the phase functions read them from here
  // instead of taking them as arguments, so that nothing has to stay in registers across their calls
  const float* x;   // input rows of the tile the compute warps are working on
  const float* pe;  // the layer's positional term (kernels with one)
  float* y;
  int32_t* status;
  uint32_t sbase;      // base of the dynamic shared memory as a shared-space address
  uint32_t off_a, off_kv, off_code;
  int n, tau, heads, mode, NF, n_f1, ln1, ln2;
  float eps;
  const float *b_o, *b_1, *b_2;  // see LateOff (16-byte aligned, or NULL)
  // the tile the compute warps are working on, and which row-list buffer describes it
  int rows, buf;
  int next_rows[2];        // rows of the tile listed in buffer b (< 0: there is no such tile), valid after rl_ready[b]
  const float* next_x[2];  // where that tile's input rows are read from
  int st_rows[2], st_stamp[2];  // for the stamp warp: rows of the stored tile in buffer b, the stamp they get (0: none)
  // row lists, double buffered: the loader warp fills buffer (k + 1) & 1 while the compute warps work on tile k;
  // the compute warps gather tile k + 1 as soon as tile k's MMAs no longer read the A operand
  int rowvox[2][kTM];              // tile row -> voxel (-1: none)
  unsigned char row_lo[2][kTM], row_n[2][kTM];  // per tile row: first row and row count of its set (0: see drop_wild)
  uint32_t starts[2][4];           // bit r: row r is the first of its set
  // relative position bias.  The table index is linear in the coordinate offset, so one integer per row,
  // x * rb_sx + y * rb_sy + z, serves every (query, key) pair: index = lin[query] - lin[key] + rb_centre.  Offsets
  // inside a covered set are at most (table length - 1) / 2 < 2^15 in magnitude (tables of up to 65,535 entries
  // per head), so the low 16 bits are kept and differences are taken modulo 2^16.
  // Written by the gather of a tile (after the previous tile's attention), read by the tile's attention.
  const float* rpb;
  const int4* coords;
  int rb_len, rb_sx, rb_sy, rb_centre, rb_ext[3];
  alignas(16) short rowlin[kTM];
  alignas(16) float par[6 * 192];
};
static_assert(sizeof(Misc) == 7 * 1024, "shared memory");
__shared__ Misc s_mi;

__device__ __forceinline__ void compute_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kComputeThreads) : "memory"); }

// gelu(t) = t Phi(t) with Phi(t) = 1 - h for t >= 0 and h for t < 0, h = erfc(|t| / sqrt 2) / 2; hence
// gelu(t) = max(t, 0) - |t| h.  h is evaluated as 2^p(|t|), p a degree-5 polynomial: a weighted least-squares
// fit of log2 erfc(|t| / sqrt 2) on |t| <= 8.4 (beyond that h < 1e-17), with the factor 1/2 folded into its
// constant term.  The polynomial runs on m = -min(|t|, 8.4) (odd coefficients negated), so that the last step
// is one fused multiply-add max(t, 0) + m h.  Two values at a time: the polynomial, the bias add and the last
// step are packed fp32x2 operations.  Absolute error of gelu below 2e-6 for all t, far under the bfloat16
// rounding applied to the result.
__device__ __forceinline__ float2 gelu_fast2(float2 t) {
  const float2 m = make_float2(fmaxf(-fabsf(t.x), -8.4f), fmaxf(-fabsf(t.y), -8.4f));
  float2 q = __ffma2_rn(make_float2(5.189499352e-04f, 5.189499352e-04f), m, make_float2(7.387642749e-03f, 7.387642749e-03f));
  q = __ffma2_rn(q, m, make_float2(5.253871530e-02f, 5.253871530e-02f));
  q = __ffma2_rn(q, m, make_float2(-4.592762589e-01f, -4.592762589e-01f));
  q = __ffma2_rn(q, m, make_float2(1.151083231e+00f, 1.151083231e+00f));
  q = __ffma2_rn(q, m, make_float2(-1.0f - 8.382420447e-07f, -1.0f - 8.382420447e-07f));
  const float2 h = make_float2(ex2_approx(q.x), ex2_approx(q.y));  // erfc(|t| / sqrt 2) / 2
  return __ffma2_rn(m, h, make_float2(fmaxf(t.x, 0.f), fmaxf(t.y, 0.f)));
}

// A block of 16 keys' relative position biases onto a row's scores, from the rows' linear coordinates; `tab` is the head's table,
// `root` the square root of the head dimension (the scores are still unscaled dot products when the bias is added).  An index is
// formed in the upper half of a word (`from`: (the row's coordinate + centre) 2^16 + 65535, so that the lower half never borrows),
// two keys to a word of shared memory (hybrid windows, 20,011 pillars: 309.4 us with a 16-bit read and a sign extension per key,
// 304.2 now).  A negative index is large there and takes the last entry like one past the table.
__device__ __forceinline__ void add_rpb(float (&s)[16], const float* __restrict__ tab, uint32_t from, int b, float root) {
  const uint32_t last = (uint32_t)(s_mi.rb_len - 1) << 16 | 0xffffu;
  const uint4* lin = reinterpret_cast<const uint4*>(&s_mi.rowlin[16 * b]);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const uint4 v = lin[i];
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      s[8 * i + 2 * j] += __ldg(tab + (min(from - (w[j] << 16), last) >> 16)) * root;
      s[8 * i + 2 * j + 1] += __ldg(tab + (min(from - w[j], last) >> 16)) * root;
    }
  }
}

// A compute thread's wait (out of line: one copy of the polling loop).  A wait that gives up raises the abort flag,
// which the tile loop looks at.
__device__ __noinline__ void wait_phase(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < kMaxPolls; ++i) {
    if (mbar_try(bar, parity)) { tc_fence_after(); return; }
    if ((i & 255) == 255 && *(volatile int*)&s_mi.abort_flag) return;
  }
  *(volatile int*)&s_mi.abort_flag = 1;
}
#define WAIT_PHASE(bar, parity) wait_phase(smem_u32(&s_mi.bar), (uint32_t)(parity) & 1u)

// ---------------------------------------------------------------------------------------------
// Attention
// ---------------------------------------------------------------------------------------------
// Set codes: sets of a tile are numbered 0, 1, 2, ... modulo kCodes.  A query row carries 2^100 at its set's place and
// zeros elsewhere, a key row 0 at its set's place and -1 elsewhere, so that their product is exactly 0 inside a set and
// -2^100 across sets of different numbers; key rows past the tile hold -1 throughout.  A warp whose keys span more than
// kCodes sets masks by comparing instead (softmax_rows).  Head dim 24 leaves 8 of the 32 columns of its two K steps to
// the code, the other head dims take a K step of 16 for it.
template <int D>
constexpr int kCodes = D == 24 ? 8 : 16;

template <int D>
__device__ __forceinline__ void write_codes(int b, int rows) {
  const int row = threadIdx.x;
  if (row >= kTM) return;
  const int w = row >> 5, lane = row & 31;
  int ord = __popc(s_mi.starts[b][w] & (0xffffffffu >> (31 - lane)));
  for (int j = 0; j < w; ++j) ord += __popc(s_mi.starts[b][j]);
  const int code = row < rows ? ord & (kCodes<D> - 1) : -1;
  const uint32_t base = s_mi.sbase + s_mi.off_code + row * 16;
#pragma unroll
  for (int c = 0; c < kCodes<D> / 8; ++c) {
    uint32_t q[4], k[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = code - 8 * c - 2 * i;  // 0: the low element of the pair, 1: the high one
      const bool low = code >= 0 && e == 0, high = code >= 0 && e == 1;
      q[i] = low ? 0x00007180u : high ? 0x71800000u : 0u;
      k[i] = low ? 0xbf800000u : high ? 0x0000bf80u : 0xbf80bf80u;
    }
    sts4(base + c * kChunkBytes, make_uint4(q[0], q[1], q[2], q[3]));
    sts4(base + (kCodes<D> / 8 + c) * kChunkBytes, make_uint4(k[0], k[1], k[2], k[3]));
  }
}

// The keys of a warp's 32 rows: blocks of 16 tile rows [kb0, kb1), and whether the codes keep their sets apart.
struct KeyRange { int kb0, kb1; bool coded; };
template <int D>
__device__ __forceinline__ KeyRange key_range(int r0, int rows) {
  const unsigned char* row_lo = s_mi.row_lo[s_mi.buf];
  const int rl = min(r0 + 31, rows - 1);
  KeyRange k;
  k.kb0 = row_lo[r0] >> 4;
  k.kb1 = min((row_lo[rl] + s_mi.row_n[s_mi.buf][rl] + 15) >> 4, (rows + 15) >> 4);
  const int from = 16 * k.kb0 + 1, to = min(16 * k.kb1, rows);  // set starts in here, and the set at the front
  int sets = 1;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int lo = min(max(from - 32 * j, 0), 32), hi = min(max(to - 32 * j, 0), 32);
    if (hi > lo) sets += __popc(s_mi.starts[s_mi.buf][j] & (0xffffffffu >> (32 - hi)) & (0xffffffffu << lo));
  }
  k.coded = sets <= kCodes<D>;
  return k;
}

// Softmax of one head for the 32 rows of a warp, a row per thread: S (fp32, TMEM columns [t_s, t_s + 128)) -> P (bf16
// pairs, columns [t_s, t_s + 64), zeros outside the warp's key blocks).  Returns the row's sum.  P overwrites S: block
// b's 8 columns lie in S blocks up to b, which have been read by then.
// [lo, lo + n): the rows of this row's set, by which keys are masked where the codes do not do it (!coded).
template <int D, bool RPB>
__device__ __forceinline__ float softmax_rows(uint32_t t_s, const KeyRange& k, int n_blocks, int row, int lo, int n, int h) {
  const float sc = 1.4426950408889634f * rsqrtf((float)D);  // log2(e) / sqrt(d)
  auto mask = [&](float (&s)[16], int b) {
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if ((unsigned)(16 * b + i - lo) >= (unsigned)n) s[i] = -INFINITY;
  };
  float mx = -INFINITY;
#pragma unroll 1
  for (int b = k.kb0; b < k.kb1; ++b) {
    float s[16];
    tmem_ld16_at<0>(t_s + 16 * b, s);
    tmem_wait_ld();
    if (RPB) {
      const uint32_t from = (uint32_t)(s_mi.rowlin[row] + s_mi.rb_centre) << 16 | 0xffffu;
      add_rpb(s, s_mi.rpb + (size_t)h * s_mi.rb_len, from, b, sqrtf((float)D));
      tmem_st16_at<0>(t_s + 16 * b, s);
    }
    if (!k.coded) mask(s, b);
    float m0 = fmaxf(s[0], s[1]), m1 = fmaxf(s[2], s[3]);
#pragma unroll
    for (int i = 4; i < 16; i += 4) { m0 = fmaxf(m0, fmaxf(s[i], s[i + 1])); m1 = fmaxf(m1, fmaxf(s[i + 2], s[i + 3])); }
    mx = fmaxf(mx, fmaxf(m0, m1));
  }
  if (RPB) tmem_wait_st();
  const float off = mx == -INFINITY ? 0.f : -mx * sc;  // (rows past the tile may have no key)
  const uint32_t zero[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
  for (int b = 0; b < k.kb0; ++b) tmem_st8_u32(t_s + 8 * b, zero);
  float2 sum = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int b = k.kb0; b < k.kb1; ++b) {
    float s[16];
    tmem_ld16_at<0>(t_s + 16 * b, s);
    tmem_wait_ld();
    if (!k.coded) mask(s, b);
    uint32_t p[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float2 u = __ffma2_rn(make_float2(s[2 * i], s[2 * i + 1]), make_float2(sc, sc), make_float2(off, off));
      const float2 e = make_float2(ex2_approx(u.x), ex2_approx(u.y));
      sum = __fadd2_rn(sum, e);
      p[i] = pack_bf16(e.x, e.y);
    }
    tmem_st8_u32(t_s + 8 * b, p);
  }
  for (int b = k.kb1; b < n_blocks; ++b) tmem_st8_u32(t_s + 8 * b, zero);
  tmem_wait_st();
  return sum.x + sum.y;
}

// Attention of tile k: warps 4 q + (0..3) take heads q, q + 4, ... ; their S, then P, then O live in TMEM columns
// [128 q, 128 q + 128).  The output of a head replaces its (dead) query columns.
template <int C, int D, bool RPB>
__device__ __forceinline__ void attend(int k) {
  constexpr int DC = D / 8;  // 16-byte chunks per head
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = warp >> 2;
  const int rows = s_mi.rows, row = 32 * (warp & 3) + lane;
  const bool on = 32 * (warp & 3) < rows;  // (the whole warp)
  const uint32_t t_s = s_mi.tmem_base + ((uint32_t)(32 * (warp & 3)) << 16) + 128 * q;
  KeyRange kr = {0, 0, true};
  if (on) kr = key_range<D>(32 * (warp & 3), rows);
  const int lo = s_mi.row_lo[s_mi.buf][row], n = s_mi.row_n[s_mi.buf][row];
#pragma unroll 1
  for (int h = q; h < s_mi.heads; h += 4) {
    const uint32_t par = (uint32_t)(k * (s_mi.heads >> 2) + (h >> 2)) & 1u;  // (heads so far of this group)
    wait_phase(smem_u32(&s_mi.s_full[0]) + 8 * q, par);
    float l = 1.f;
    if (on) l = softmax_rows<D, RPB>(t_s, kr, (rows + 15) >> 4, row, lo, n, h);
    tc_fence_before();
    mbar_arrive(&s_mi.p_ready[q]);
    wait_phase(smem_u32(&s_mi.ov_full[0]) + 8 * q, par);
    if (on) {
      float o[D];
      tmem_ld_row(t_s + 64, o);
      tmem_wait_ld();
      const float inv = __fdividef(1.0f, l);
      const uint32_t out = s_mi.sbase + s_mi.off_a + h * DC * kChunkBytes + row * 16;
#pragma unroll
      for (int c = 0; c < DC; ++c)
        sts4(out + c * kChunkBytes,
             make_uint4(pack_bf16(o[8 * c] * inv, o[8 * c + 1] * inv), pack_bf16(o[8 * c + 2] * inv, o[8 * c + 3] * inv),
                        pack_bf16(o[8 * c + 4] * inv, o[8 * c + 5] * inv), pack_bf16(o[8 * c + 6] * inv, o[8 * c + 7] * inv)));
    }
    tc_fence_before();
    mbar_arrive(&s_mi.o_read[q]);
  }
}

// fp32 row staging in the K/V region: row r, 16-byte chunk c4 of C/4, XORed with the row so that both
// the warp-per-row pattern (global side) and the thread-per-row pattern (TMEM side) are conflict-free.
template <int C>
__device__ __forceinline__ uint32_t stage_off(int r, int c4) {
  return (uint32_t)(r * (C * 4) + ((c4 ^ (r & 7)) << 4));
}

// ---------------------------------------------------------------------------------------------
// Roles
// ---------------------------------------------------------------------------------------------
struct RoleCtx {
  uint32_t sbase;     // 1024-aligned shared-memory base as a shared-space address
  uint32_t tmem;      // TMEM base address of the CTA's allocation
  // copies of the kernel parameters the two single-thread roles use (registers instead of parameter-space loads)
  int mode, n_f1, NF, tau, n_layers, heads;
  int pe;  // the value projection comes first and the A operand is rewritten (x + pe) before the key and query ones
  uint32_t off_a, off_kv, off_code, off_stage;
};

__device__ __forceinline__ int ld_acquire_gpu(const int32_t* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_gpu(int32_t* p, int v) {
  asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Order of the MLP pieces: M1(0), M1(1), M2(0), M1(2), M2(1), ..., M1(n-1), M2(n-2), M2(n-1), so that the next
// piece's first product runs while the compute warps apply GELU to the current one.  q in [0, 2n): piece and kind.
__device__ __forceinline__ bool mlp_step(int q, int n, int& piece) {  // true: M1
  if (q == 0) { piece = 0; return true; }
  if (q == 2 * n - 1) { piece = n - 1; return false; }
  piece = (q & 1) ? (q + 1) >> 1 : (q >> 1) - 1;
  return (q & 1) != 0;
}

// The scheduler and the MMA issuer are separate (not inlined) functions so that their polling loops get
// their own, spill-free register allocation; the compute role and its phases are inlined into the kernel, where the
// kernel parameters are constant-bank operands.

// ================= scheduler + TMA producer (one thread) ===============================================
// Tiles are numbered over the whole chain, layer after layer; a tile's number comes from the launch's counter.
// Inside a layer, tile t is entry t of the layer's plan (whole sets, at most 128 distinct rows); a layer without
// a plan is cut by row ranges instead: tile t holds the sets whose first row lies in [t R, (t + 1) R),
// R = 128 - tau + 1, found by binary search in the row offsets (slower to schedule, same results).
template <int C>
__device__ __noinline__ void producer_role(const TcArgs& a, const RoleCtx rc) {
  constexpr int NKB = C / 64;        // K blocks of a C-deep contraction
  constexpr uint32_t STAGE_BYTES = C * 128;
  Misc* mi = &s_mi;
  const uint32_t st_base = rc.sbase + rc.off_stage;
  volatile int* abort_flag = &mi->abort_flag;
  int32_t* status = a.status;
  const bool mlp = rc.mode == 2;
  const int n_chunks = 4 + (mlp ? 2 * rc.n_f1 : 0);
  const int L = rc.n_layers;
  const int Rv = kTM - rc.tau + 1;
  // the chain's tile counts
  int total = 0;
  for (int l = 0; l < L; ++l) {
    const TcLayer& ly = a.layer[l];
    const int S = min(__ldg(ly.num_sets), ly.cap_sets);
    int T = __ldg(ly.rowoff + ly.cap_sets + 1);
    mi->lay_plan[l] = T < 0 ? 0 : (T & DSVT_PLAN_PACKED) ? 2 : 1;  // none / in table order / over a reordering
    if (T < 0) T = S > 0 ? (__ldg(ly.rowoff + S) + Rv - 1) / Rv : 0;
    else T = min(T & ~DSVT_PLAN_PACKED, S);
    total += max(T, 0);
    mi->tile_end[l] = total;
  }
  // next tile: layer, first set s0, ns sets (< 0: none left), first row, rows
  auto next_tile = [&](int& lay, int& s0, int& ns, int& base, int& rows) {
    for (;;) {
      lay = 0; s0 = 0; ns = -1; base = 0; rows = 0;
      if (*abort_flag) return;
      const int g = atomicAdd(a.counter, 1);
      if (g < 0 || g >= total) return;
      int l = 0;
      while (l + 1 < L && g >= mi->tile_end[l]) ++l;
      const int t = g - (l ? mi->tile_end[l - 1] : 0);
      const TcLayer& ly = a.layer[l];
      const int S = min(__ldg(ly.num_sets), ly.cap_sets);
      int f, e;
      if (mi->lay_plan[l]) {
        const int32_t* plan = ly.rowoff + ly.cap_sets + 1;
        f = __ldg(plan + 1 + t);
        e = __ldg(plan + 2 + t);
        if (f < 0 || e <= f || e > S) { atomicOr(status, DSVT_STATUS_BAD_INDEX); continue; }
      } else {
        const int r0 = t * Rv, r1 = r0 + Rv;
        int lo = 0, hi = S;
        while (lo < hi) { const int m = (lo + hi) >> 1; if (__ldg(ly.rowoff + m) < r0) lo = m + 1; else hi = m; }
        f = lo;
        hi = S;
        while (lo < hi) { const int m = (lo + hi) >> 1; if (__ldg(ly.rowoff + m) < r1) lo = m + 1; else hi = m; }
        e = lo;
        if (e <= f) continue;  // no set starts in this row range
      }
      // rows before a position: of the table's own order, or of the packed plan's
      const int32_t* ro = mi->lay_plan[l] == 2 ? ly.rowoff + 3 * (size_t)ly.cap_sets + 3 : ly.rowoff;
      base = __ldg(ro + f);
      rows = __ldg(ro + e) - base;
      if (rows <= 0 || rows > kTM || e - f > kTM) { atomicOr(status, DSVT_STATUS_BAD_INDEX); continue; }
      lay = l; s0 = f; ns = e - f;
      return;
    }
  };
  int stage = 0, slot = 0;
  uint32_t phase = 0, sphase = 0;
  int issued[kStages];  // loads issued into each stage so far
#pragma unroll
  for (int i = 0; i < kStages; ++i) issued[i] = 0;
  int lay, s, ns, base, rows;
  int wl[2] = {0, 0}, wcount = 0, wread = 0;  // layers of the published tiles whose weights are still to be streamed
  bool all_out = false;    // the end marker has been published
  // Tiles are published two ahead of the weights (the ring has two entries), so that the loader
  // warp can prepare tile k + 1 while tile k is being computed.
  auto publish = [&]() -> bool {
    next_tile(lay, s, ns, base, rows);
    if (!mbar_wait(&mi->sched_empty[slot], sphase ^ 1u, abort_flag)) return false;
    mi->tile[slot][0] = s; mi->tile[slot][1] = ns; mi->tile[slot][2] = base; mi->tile[slot][3] = rows;
    mi->tile[slot][4] = lay;
    mbar_arrive(&mi->sched_full[slot]);
    if (++slot == 2) { slot = 0; sphase ^= 1u; }
    if (ns < 0) { all_out = true; return true; }
    wl[(wread + wcount) & 1] = lay;
    ++wcount;
    return true;
  };
  if (!publish()) goto producer_done;
  if (!all_out && !publish()) goto producer_done;
  while (wcount > 0) {
    // the layer's weights for one tile, chunk by chunk, K block by K block
    const TcLayer& ly = a.layer[wl[wread & 1]];
    for (int c = 0; c < n_chunks; ++c) {
      const CUtensorMap* map;
      int row0 = 0, col0 = 0, nkb = NKB;
      uint32_t bytes = STAGE_BYTES;
      if (c < 3) {  // K, V, Q; with a positional term V, K, Q
        map = &ly.qkv;
        row0 = (rc.pe ? (c == 0 ? 2 : c == 1 ? 1 : 0) : (c == 0 ? 1 : c == 1 ? 2 : 0)) * C;
      } else if (c == 3) {
        map = &ly.o;
      } else {
        int piece;
        if (mlp_step(c - 4, rc.n_f1, piece)) { map = &ly.w1; row0 = piece * rc.NF; bytes = (uint32_t)rc.NF * 128u; }
        else { map = &ly.w2; col0 = piece * rc.NF; nkb = rc.NF / 64; }
      }
      for (int kb = 0; kb < nkb; ++kb) {
        if (!mbar_wait(&mi->empty[stage], phase ^ 1u, abort_flag)) goto producer_done;
        mbar_expect_tx(&mi->full[stage], bytes);
        tma_load_2d(st_base + stage * STAGE_BYTES, map, col0 + kb * 64, row0, &mi->full[stage]);
        ++issued[stage];
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
    }
    ++wread;
    --wcount;
    if (!all_out && !publish()) goto producer_done;
  }
producer_done:
  if (*abort_flag) {
    // leaving early: no load may still be writing into this CTA's shared memory when it retires
#pragma unroll
    for (int i = 0; i < kStages; ++i)
      if (issued[i] > 0) {
        const uint32_t par = (uint32_t)(issued[i] - 1) & 1u;
        for (int it = 0; it < kMaxPolls && !mbar_try(&mi->full[i], par); ++it) {}
      }
  }
}

// ================= MMA issuer (one warp) ===============================================================
// The whole warp runs this code with warp-uniform values and one elected lane issues: operands then stay in uniform
// registers.  Issued by a single thread from divergent code every MMA took 46 to 65 cycles of issue (measured: eight
// N = 32 MMAs done after 788 cycles, against 249 this way), which is more than the tensor pipe needs for N <= 128 (N / 2
// cycles).  Descriptors are kept as 32-bit low words (address and leading offset, to which byte offsets / 16 are added)
// and constant high words.
template <int C, int D>
__device__ __forceinline__ void mma_role(const RoleCtx& rc) {
  constexpr int NKB = C / 64;        // K blocks of a C-deep contraction
  constexpr uint32_t STAGE16 = C * 128 / 16;
  constexpr uint32_t kChunk16 = kChunkBytes / 16, kRows16 = kTM * 128 / 16;  // a chunk; a K block of the swizzled operand
  constexpr uint32_t kHeadStep = (D / 8) * kChunk16;  // from a head's Q, K or V columns to the next head's
  constexpr uint32_t SW = kDescHiSwizzled, KM = desc_hi_plain(128), NM = desc_hi_plain(kChunkBytes);
  const uint32_t tmem = rc.tmem;
  Misc* mi = &s_mi;
  const uint32_t a_addr = rc.sbase + rc.off_a, k_addr = rc.sbase + rc.off_kv, v_addr = k_addr + (C / 8) * kChunkBytes;
  const uint32_t q_code = rc.sbase + rc.off_code, k_code = q_code + kCodes<D> / 8 * kChunkBytes;
  const uint32_t x_lo = desc_lo_swizzled(a_addr), w_lo = desc_lo_swizzled(rc.sbase + rc.off_stage);
  const uint32_t q_lo = desc_lo_plain(a_addr, kChunkBytes), k_lo = desc_lo_plain(k_addr, kChunkBytes);
  const uint32_t v_lo = desc_lo_plain(v_addr, 128);
  volatile int* abort_flag = &mi->abort_flag;
  const bool mlp = rc.mode == 2;
  const int c_v = rc.pe ? 0 : 1;  // the V chunk
  int stage = 0, slot = 0;
  uint32_t phase = 0, a_phase = 0, x_phase = 0, sphase = 0, tile = 0;
  uint32_t uses = 0, m2 = 0, heads_done = 0;  // of the K / Q / MLP-1 accumulator; MLP-2 pieces; heads of a group
  // n_kb K blocks of 64 from the weight ring; issue(kb, k4, low word of B) issues one MMA
  auto blocks = [&](int n_kb, auto issue) -> bool {
    for (int kb = 0; kb < n_kb; ++kb) {
      if (!mbar_wait(&mi->full[stage], phase, abort_flag)) return false;
      tc_fence_after();
      const uint32_t b = w_lo + stage * STAGE16;
      if (elect_one()) {
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4) issue(kb, k4, b + 2 * k4);
        umma_commit(&mi->empty[stage]);  // frees the weight stage once these MMAs have read it
      }
      __syncwarp();
      if (++stage == kStages) { stage = 0; phase ^= 1u; }
    }
    return true;
  };
  auto commit = [&](unsigned long long* bar) {
    if (elect_one()) umma_commit(bar);
    __syncwarp();
  };
  for (;; ++tile) {
    if (!mbar_wait(&mi->sched_full[slot], sphase, abort_flag)) break;
    const int ns = __shfl_sync(0xffffffffu, mi->tile[slot][1], 0), rows = __shfl_sync(0xffffffffu, mi->tile[slot][3], 0);
    if (elect_one()) mbar_arrive(&mi->sched_empty[slot]);
    if (++slot == 2) { slot = 0; sphase ^= 1u; }
    if (ns < 0) break;
    // ---- K, V, Q ----
    for (int c = 0; c < 3; ++c) {
      if (c == 0 || (c == 1 && rc.pe)) {  // (with a positional term the operand is rewritten after the V chunk)
        if (!mbar_wait(&mi->x_ready, x_phase, abort_flag)) goto mma_done;
        x_phase ^= 1u;
      }
      if (c == c_v) {
        // the columns may overlap R and the MLP hidden: the previous tile's result must have been read
        if (!mbar_wait(&mi->acc_free[2], (tile & 1u) ^ 1u, abort_flag)) goto mma_done;
        if (!mbar_wait(&mi->acc_free[1], (tile & 1u) ^ 1u, abort_flag)) goto mma_done;
      } else {
        if (!mbar_wait(&mi->acc_free[0], (uses & 1u) ^ 1u, abort_flag)) goto mma_done;
        ++uses;
      }
      tc_fence_after();
      const uint32_t d = tmem + (c == c_v ? Tm<C>::v : Tm<C>::k);
      if (!blocks(NKB, [&](int kb, int k4, uint32_t b) {
            umma_ss(d, x_lo + kb * kRows16 + 2 * k4, SW, b, SW, umma_idesc(C), (kb | k4) != 0 ? 1u : 0u);
          })) goto mma_done;
      commit(&mi->acc_full[c == c_v ? 1 : 0]);
    }
    // ---- attention: S = Q K^T, O = P V, four heads at a time ----
    if (!mbar_wait(&mi->a_ready, a_phase, abort_flag)) goto mma_done;
    a_phase ^= 1u;
    tc_fence_after();
    {
      const int n_blocks = (rows + 15) >> 4;  // of 16 keys
      const uint32_t id_s = umma_idesc(16 * n_blocks), id_o = umma_idesc(D == 24 ? 32 : D) | (1u << 16);  // V: N-major
      const int rounds = rc.heads >> 2;
      auto scores = [&](int q, int i) {
        const uint32_t d = tmem + 128 * q, step = (uint32_t)(4 * i + q) * kHeadStep;
        umma_ss(d, q_lo + step, KM, k_lo + step, KM, id_s, 0u);
        if (D == 24) {  // the last 8 columns and the code: the leading offset leads from one to the other
          const uint32_t qa = (a_addr >> 4) + 2 * kChunk16 + step, ka = (k_addr >> 4) + 2 * kChunk16 + step;
          umma_ss(d, qa | ((q_code >> 4) - qa) << 16, KM, ka | ((k_code >> 4) - ka) << 16, KM, id_s, 1u);
        } else {
          if (D == 32) umma_ss(d, q_lo + step + 2 * kChunk16, KM, k_lo + step + 2 * kChunk16, KM, id_s, 1u);
          umma_ss(d, desc_lo_plain(q_code, kChunkBytes), KM, desc_lo_plain(k_code, kChunkBytes), KM, id_s, 1u);
        }
        umma_commit(&mi->s_full[q]);
      };
      if (elect_one()) {
#pragma unroll
        for (int q = 0; q < 4; ++q) scores(q, 0);
      }
      __syncwarp();
      // the four groups advance on their own: step 2 i of a group waits for P of its head i, step 2 i + 1 for O having
      // been read (not needed after the last head: a_ready follows it)
      int left = 4 * (2 * rounds - 1);
      uint32_t step = 0;  // 8 bits per group
      for (int idle = 0; left > 0; ++idle) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int st = (int)(step >> (8 * q)) & 255, i = st >> 1;
          if (st >= 2 * rounds - 1) continue;
          if (!__all_sync(0xffffffffu, mbar_test((st & 1) ? &mi->o_read[q] : &mi->p_ready[q], (heads_done + (uint32_t)i) & 1u)))
            continue;
          tc_fence_after();
          if (elect_one()) {
            if (st & 1) {
              scores(q, i + 1);
            } else {
              const uint32_t v = v_lo + (uint32_t)(4 * i + q) * kHeadStep;
#pragma unroll
              for (int s = 0; s < 8; ++s)  // (16 keys: 8 columns of P, 256 bytes of each chunk of V)
                if (s < n_blocks)
                  umma_ts(tmem + 128 * q + 64, tmem + 128 * q + 8 * s, v + 16 * s, NM, id_o, s != 0 ? 1u : 0u);
              umma_commit(&mi->ov_full[q]);
            }
          }
          __syncwarp();
          step += 1u << (8 * q);
          --left;
          idle = 0;
        }
        if ((idle & 255) == 255 && *abort_flag) goto mma_done;
        if (idle > kMaxIdle) { *abort_flag = 1; goto mma_done; }
      }
      heads_done += (uint32_t)rounds;
    }
    // ---- output projection ----
    if (!mbar_wait(&mi->a_ready, a_phase, abort_flag)) goto mma_done;
    a_phase ^= 1u;
    tc_fence_after();
    if (!blocks(NKB, [&](int kb, int k4, uint32_t b) {
          umma_ss(tmem + Tm<C>::r, q_lo + (8 * kb + 2 * k4) * kChunk16, KM, b, SW, umma_idesc(C), (kb | k4) != 0 ? 1u : 0u);
        })) goto mma_done;
    commit(&mi->o_full);
    if (!mlp) continue;
    // ---- MLP, piece by piece, on top of the residual parked in R ----
    if (!mbar_wait(&mi->a_ready, a_phase, abort_flag)) goto mma_done;
    a_phase ^= 1u;
    for (int c = 0; c < 2 * rc.n_f1; ++c) {
      int piece;
      if (mlp_step(c, rc.n_f1, piece)) {
        if (!mbar_wait(&mi->acc_free[0], (uses & 1u) ^ 1u, abort_flag)) goto mma_done;
        ++uses;
        tc_fence_after();
        const uint32_t idesc = umma_idesc(rc.NF);
        if (!blocks(NKB, [&](int kb, int k4, uint32_t b) {  // (16 bf16 operand columns are 8 TMEM columns)
              umma_ts(tmem + Tm<C>::acc, tmem + Tm<C>::x1 + kb * 32 + k4 * 8, b, SW, idesc, (kb | k4) != 0 ? 1u : 0u);
            })) goto mma_done;
        commit(&mi->acc_full[0]);
      } else {
        if (!mbar_wait(&mi->h_ready, m2 & 1u, abort_flag)) goto mma_done;
        ++m2;
        tc_fence_after();
        if (!blocks(rc.NF / 64, [&](int kb, int k4, uint32_t b) {
              umma_ts(tmem + Tm<C>::r, tmem + Tm<C>::h + kb * 32 + k4 * 8, b, SW, umma_idesc(C), 1u);
            })) goto mma_done;
        commit(&mi->h_free);
      }
    }
    commit(&mi->acc_full[2]);
  }
mma_done:
  if (*abort_flag) {
    // leaving early: the MMAs already issued must have completed before the TMEM columns are returned
    commit(&mi->drain);
    for (int it = 0; it < kMaxPolls && !mbar_try(&mi->drain, 0u); ++it) {}
  }
}

// ================= loader warp: row list, one tile ahead of the compute warps =============================
__device__ __forceinline__ void loader_sync() { asm volatile("bar.sync 6, %0;" ::"n"(kLoadThreads) : "memory"); }

// Distinct slots of each set -> tile rows (Eq. 4) and per-row set ranges: one thread per
// set (a tile of a sparse region holds dozens of tiny sets), walking the set's table row.
// `order` (or NULL: the identity) maps the positions [s_lo, s_lo + nsets) of the tile to sets, `rowoff` holds the
// rows before each position.
template <bool RPB>
__device__ __forceinline__ void loader_row_list(const int32_t* __restrict__ table, const int32_t* __restrict__ rowoff,
                                                const int32_t* __restrict__ order, int cap_sets, int b, int lt,
                                                int s_lo, int nsets, int base) {
  const int n = s_mi.n, tau = s_mi.tau;
  for (int si = lt; si < nsets; si += kLoadThreads) {
    const int p = s_lo + si;
    const int s = order ? __ldg(order + p) : p;
    if ((unsigned)s >= (unsigned)cap_sets) {  // (only a plan that this library did not write can do that)
      atomicOr(s_mi.status, DSVT_STATUS_BAD_INDEX);
      continue;
    }
    const int32_t* trow = table + (size_t)s * tau;
    const int lb = __ldg(rowoff + p) - base, cap = __ldg(rowoff + p + 1) - __ldg(rowoff + p);
    const bool inside = lb >= 0 && lb < kTM;
    const int cnt_max = inside ? min(cap, kTM - lb) : 0;  // tile rows this set may fill
    int pos = 0, prev = 0;
    bool bad = false;
    constexpr bool rpb = RPB;
    int lo3[3] = {INT_MAX, INT_MAX, INT_MAX}, hi3[3] = {INT_MIN, INT_MIN, INT_MIN};
    for (int k0 = 0; k0 < tau; k0 += 8) {
      int v4[8];  // eight independent loads per round trip to L2 (the loader warp runs a whole tile ahead)
#pragma unroll
      for (int u = 0; u < 8; ++u) v4[u] = k0 + u < tau ? __ldg(trow + k0 + u) : 0;
      if (rpb) {  // a set spread wider than the bias table's extent is reported
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (k0 + u < tau && v4[u] >= 0 && v4[u] < n) {
            const int4 c = __ldg(s_mi.coords + v4[u]);
            lo3[0] = min(lo3[0], c.y); hi3[0] = max(hi3[0], c.y);
            lo3[1] = min(lo3[1], c.z); hi3[1] = max(hi3[1], c.z);
            lo3[2] = min(lo3[2], c.w); hi3[2] = max(hi3[2], c.w);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        if (k0 + u < tau) {
          int v = v4[u];
          const bool uniq = (k0 + u == 0) || (v != prev);
          prev = v;
          if (uniq) {
            if (pos < cnt_max) {
              if (v < 0 || v >= n) { bad = true; v = -1; }
              s_mi.rowvox[b][lb + pos] = v;
              s_mi.row_lo[b][lb + pos] = (unsigned char)lb;
              s_mi.row_n[b][lb + pos] = (unsigned char)cnt_max;
            }
            ++pos;
          }
        }
      }
    }
    if (rpb)
      for (int q = 0; q < 3; ++q) bad |= hi3[q] >= lo3[q] && hi3[q] - lo3[q] > s_mi.rb_ext[q] - 1;
    if (bad || pos != cap) atomicOr(s_mi.status, DSVT_STATUS_BAD_INDEX);
  }
}

template <int C, bool RPB>
__device__ __noinline__ void loader_role(const TcArgs& a) {
  const int lt = threadIdx.x - 32 * kLoadWarp0, lane = lt & 31;
  volatile int* abort_flag = &s_mi.abort_flag;
  int slot = 0;
  uint32_t sphase = 0;
  bool ok = true;
  for (int k = 0;; ++k) {
    ok = mbar_wait(&s_mi.sched_full[slot], sphase, abort_flag) && ok;
    // every exit from this loop is taken by all loader threads together
    if (bar_or(6, kLoadThreads, !ok || *abort_flag != 0)) break;
    const int s_lo = s_mi.tile[slot][0], nsets = s_mi.tile[slot][1], base = s_mi.tile[slot][2], rows = s_mi.tile[slot][3];
    const int lay = s_mi.tile[slot][4];
    __syncwarp();
    if (lane == 0) mbar_arrive(&s_mi.sched_empty[slot]);
    if (++slot == 2) { slot = 0; sphase ^= 1u; }
    const int b = k & 1;
    // buffer b was last used by tile k - 2: the compute warps and the stamp warp release it when they are done with it
    if (k >= 2) ok = mbar_wait(&s_mi.rl_free[b], (uint32_t)((k >> 1) - 1) & 1u, abort_flag) && ok;
    if (nsets >= 0) {
      for (int i = lt; i < kTM; i += kLoadThreads) {
        s_mi.rowvox[b][i] = -1;
        s_mi.row_lo[b][i] = (unsigned char)i;
        s_mi.row_n[b][i] = 1;
      }
      loader_sync();
      const TcLayer& ly = a.layer[lay];
      const bool packed = s_mi.lay_plan[lay] == 2;
      loader_row_list<RPB>(ly.table, packed ? ly.rowoff + 3 * (size_t)ly.cap_sets + 3 : ly.rowoff,
                           packed ? ly.rowoff + 2 * (size_t)ly.cap_sets + 3 : nullptr, ly.cap_sets, b, lt, s_lo, nsets, base);
      if (lt == 0) s_mi.next_x[b] = lay == 0 ? a.x : a.y;
    }
    if (nsets >= 0) {
      loader_sync();  // the row list is complete
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t m = __ballot_sync(0xffffffffu, s_mi.row_lo[b][32 * j + lane] == 32 * j + lane);
        if (lane == 0) s_mi.starts[b][j] = m;
      }
    }
    if (lt == 0) s_mi.next_rows[b] = nsets < 0 ? -1 : rows;
    mbar_arrive(&s_mi.rl_ready[b]);
    if (nsets < 0) break;
    // a tile of a later layer reads rows the previous layer wrote, possibly on other SMs: each row must carry that
    // layer's stamp (written after the row's store) before the tile is gathered
    if (lay > 0) {
      const int want = a.stamp_base + lay;
      for (int r = lt; r < rows && ok; r += kLoadThreads) {
        const int v = s_mi.rowvox[b][r];
        if (v < 0) continue;
        int it = 0;
        while (ld_acquire_gpu(a.row_stamp + v) != want) {
          if (++it >= kStampPolls || *abort_flag) { *abort_flag = 1; ok = false; break; }
          __nanosleep(256);
        }
      }
    }
    mbar_arrive(&s_mi.dep_ready[b]);
  }
}

// ================= stamp warp: completion stamps of a stored tile's rows ==================================
__device__ __noinline__ void stamp_role(int32_t* __restrict__ row_stamp) {
  const int lane = threadIdx.x & 31;
  volatile int* abort_flag = &s_mi.abort_flag;
  for (int k = 0;; ++k) {
    const int b = k & 1;
    // (a failed wait has raised the abort flag: the compute warps leave their loop, and so does this warp)
    if (!mbar_wait(&s_mi.stored[b], (uint32_t)(k >> 1) & 1u, abort_flag)) break;
    if (s_mi.exit_at == k) break;
    const int rows = s_mi.st_rows[b], stamp = s_mi.st_stamp[b];
    if (stamp != 0) {
      __threadfence();  // the rows' stores (ordered before this warp by the barrier) are visible before the stamps
      for (int r = lane; r < rows; r += 32) {
        const int v = s_mi.rowvox[b][r];
        if (v >= 0) st_relaxed_gpu(row_stamp + v, stamp);
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&s_mi.rl_free[b]);
  }
}

// ================= compute warps ========================================================================
// Each phase of a tile is a function that takes at most a few scalars and reads the rest from s_mi, so that the tile
// loop keeps almost nothing alive across the phases.  They are inlined: as calls they cost 3 % (the registers a callee
// may use depend on what the widest phase leaves to the caller).

// Gather (Eq. 4): the fp32 rows listed in buffer b -> bf16 A operand; all 128 rows are written (rows past the tile as
// zeros).  16 lanes to a row (256 bytes), all of a thread's rows in flight at once (C = 192: 12 loads; in two rounds the
// gather cost one L2 round trip more).  A thread's rows are 32 apart and its chunks 16, so that every address is one base
// plus constants (in lane-linear units, with a division, a row lookup and a swizzled address per 16 bytes, gather, x
// staging and row stores took 1 % more of a 32,000-pillar frame and 4 % more of two layers on 2531 rows).  ADD_PE: the
// current tile's rows once more, with the positional term added (the operand of the key and query projections).
//
// The products of the attention run over the whole tile, and zero weights or codes do not stop what is not finite: such a
// row would reach the other sets of its tile, and one of 2^60 or more could outweigh the codes.  Those values become zeros
// in the operand and their sets are marked (drop_wild); the query epilogue makes the rows of a marked set NaN.  The look is
// hidden under the loads: 32,000-pillar frame 397.5 us without and 395.8 with it, 120,000 voxels 1403.9 and 1405.4.  (A
// branch in the attention, to mask a flagged tile's scores and repair its value operand there, cost 0.5 %.)
__device__ __forceinline__ float max_abs3(float a, float b, float c) {  // (NaN if one of them is)
  float m;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c));
  return m;
}
constexpr int kUnitRows = kComputeThreads / 16;
// A thread that has gathered values that are not finite or of 2^60 or more: zeros in their place, no rows for their sets.
//   to   the thread's first 8 bytes in the operand
template <int C>
__device__ __noinline__ void drop_wild(int b, uint32_t to) {
  unsigned char *row_lo = s_mi.row_lo[b], *row_n = s_mi.row_n[b];
  for (int r = threadIdx.x / 16; r < kTM; r += kUnitRows, to += kUnitRows * 128) {
    bool bad = false;
    for (int i = 0; i < C / 32; ++i) {
      const uint32_t a = to + (i >> 1) * (kTM * 128) + 4 * (i & 1);
      uint32_t w;
      asm volatile("ld.shared.b32 %0, [%1];" : "=r"(w) : "r"(a));
      constexpr uint32_t k2p60 = (127 + 60) << 7;
      if ((w & 0x7fffu) >= k2p60) { w &= 0xffff0000u; bad = true; }
      if ((w >> 16 & 0x7fffu) >= k2p60) { w &= 0xffffu; bad = true; }
      asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(w));
    }
    if (bad) {  // (if another thread has begun to mark the set it marks all of it)
      const int lo = row_lo[r], n = row_n[r];
      for (int k = lo; k < lo + n; ++k) row_n[k] = 0;
    }
  }
}
template <int C, int D, bool RPB, bool ADD_PE>
__device__ __forceinline__ void phase_gather(int b, int rows) {
  constexpr int P = kTM / kUnitRows, J = C / 64, kFly = ADD_PE ? P / 2 : P;  // a thread's rows, chunks, rows in flight
  const int r0 = threadIdx.x / 16, c0 = threadIdx.x % 16;
  const float* x = ADD_PE ? s_mi.x : s_mi.next_x[b];
  const uint32_t to = s_mi.sbase + s_mi.off_a + swz(r0, c0 >> 1) + 8 * (c0 & 1);
  const int* rowvox = s_mi.rowvox[b];
  if (!ADD_PE) write_codes<D>(b, rows);  // (the previous tile's attention is over)
  float m0 = 0.f, m1 = 0.f;
#pragma unroll
  for (int p0 = 0; p0 < P; p0 += kFly) {
    float4 f[kFly][J];
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
      const int r = r0 + kUnitRows * (p0 + u), v = r < rows ? rowvox[r] : -1;
#pragma unroll
      for (int j = 0; j < J; ++j) {
        f[u][j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (v >= 0) {
          // (L2: the rows of a later layer were written during this launch, by any SM)
          f[u][j] = __ldcg(reinterpret_cast<const float4*>(x + (size_t)v * C) + c0 + 16 * j);
          if (ADD_PE) {
            const float4 p = __ldg(reinterpret_cast<const float4*>(s_mi.pe + (size_t)v * C) + c0 + 16 * j);
            f[u][j].x += p.x; f[u][j].y += p.y; f[u][j].z += p.z; f[u][j].w += p.w;
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kFly; ++u) {
#pragma unroll
      for (int j = 0; j < J; ++j) {
        m0 = max_abs3(m0, f[u][j].x, f[u][j].y);
        m1 = max_abs3(m1, f[u][j].z, f[u][j].w);
        sts2(to + (p0 + u) * (kUnitRows * 128) + j * (kTM * 128),
             make_uint2(pack_bf16(f[u][j].x, f[u][j].y), pack_bf16(f[u][j].z, f[u][j].w)));
      }
    }
  }
  if (!(max_abs3(m0, m1, 0.f) < 0x1p60f)) drop_wild<C>(b, to);
  if (RPB && !ADD_PE) {
    for (int r = threadIdx.x; r < kTM; r += kComputeThreads) {
      const int v = r < rows ? rowvox[r] : -1;
      int lin = 0;
      if (v >= 0) {
        const int4 c = __ldg(s_mi.coords + v);
        lin = c.y * s_mi.rb_sx + c.z * s_mi.rb_sy + c.w;
      }
      s_mi.rowlin[r] = (short)lin;
    }
  }
}

// Epilogue of a K, V or Q chunk: QC accumulator columns per thread + bias -> bf16 into an unswizzled operand tile.
// Four threads per tile row: warp w owns TMEM lanes 32 (w % 4) .. + 31 and column quarter w / 4.  Warps without rows
// only release the accumulator.
//   tcol      first TMEM column of the chunk's accumulator
//   bar       accumulator barrier pair to release
//   bias_off  float offset of the chunk's bias in the parameter block
//   dst_off   byte offset of the destination operand from the shared-memory base
// BIAS = false skips the bias (the key projection: a key bias adds
// the same amount q . b_k to every score of a query, which the softmax cancels).
// QUERY: the first query column of a row whose set is marked becomes NaN (see drop_wild), and with it the row.
template <int QC, bool BIAS, bool QUERY>
__device__ __forceinline__ void phase_epi_bf16(uint32_t tcol, int bar, int bias_off, uint32_t dst_off) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = 32 * (warp & 3) + lane, hq = warp >> 2;
  if (32 * (warp & 3) >= s_mi.rows) {
    tc_fence_before();
    mbar_arrive(&s_mi.acc_free[bar]);
    return;
  }
  const uint32_t taddr = s_mi.tmem_base + ((uint32_t)(32 * (warp & 3)) << 16) + tcol + hq * QC;
  const uint32_t bias = smem_u32(s_mi.par) + 4u * (uint32_t)(bias_off + hq * QC);
  const uint32_t dst = s_mi.sbase + dst_off + (uint32_t)(hq * (QC / 8)) * kChunkBytes + row * 16;
  float rr[QC];
  tmem_ld_row(taddr, rr);
  tmem_wait_ld();
  tc_fence_before();
  mbar_arrive(&s_mi.acc_free[bar]);  // the accumulator is in registers now
  if (QUERY && s_mi.row_n[s_mi.buf][row] == 0) rr[0] = __int_as_float(0x7fffffff);
#pragma unroll
  for (int q = 0; q < QC / 8; ++q) {
    float2 v[4] = {make_float2(rr[8 * q], rr[8 * q + 1]), make_float2(rr[8 * q + 2], rr[8 * q + 3]),
                   make_float2(rr[8 * q + 4], rr[8 * q + 5]), make_float2(rr[8 * q + 6], rr[8 * q + 7])};
    if (BIAS) {
      const float4 b0 = lds4(bias + 32 * q), b1 = lds4(bias + 32 * q + 16);
      v[0] = __fadd2_rn(v[0], make_float2(b0.x, b0.y));
      v[1] = __fadd2_rn(v[1], make_float2(b0.z, b0.w));
      v[2] = __fadd2_rn(v[2], make_float2(b1.x, b1.y));
      v[3] = __fadd2_rn(v[3], make_float2(b1.z, b1.w));
    }
    sts4(dst + q * kChunkBytes,
         make_uint4(pack_bf16(v[0].x, v[0].y), pack_bf16(v[1].x, v[1].y), pack_bf16(v[2].x, v[2].y), pack_bf16(v[3].x, v[3].y)));
  }
}

// MLP-1 piece: HC = NF / 4 hidden columns per thread, H = gelu(x1 W_1^T + b_1) into TMEM as the A operand of MLP-2.
//   bias_off  float offset of the piece's bias among the late vectors
//   h_phase   parity of h_free that says that the MLP-2 of the piece before has read its hidden columns
template <int C, int HC>
__device__ __forceinline__ void phase_mlp1(int bias_off, uint32_t h_phase) {
  const int warp = threadIdx.x >> 5, hq = warp >> 2;
  const uint32_t lane_base = s_mi.tmem_base + ((uint32_t)(32 * (warp & 3)) << 16);
  if (32 * (warp & 3) >= s_mi.rows) {  // a warp without rows keeps step with the others
    tc_fence_before();
    mbar_arrive(&s_mi.acc_free[0]);
    mbar_wait(&s_mi.h_free, h_phase, &s_mi.abort_flag);
    mbar_arrive(&s_mi.h_ready);
    return;
  }
  const uint32_t bias = s_mi.sbase + s_mi.off_code + 4u * (uint32_t)(bias_off + hq * HC);
  float rr[HC];
  tmem_ld_row(lane_base + Tm<C>::acc + hq * HC, rr);
  tmem_wait_ld();
  tc_fence_before();
  mbar_arrive(&s_mi.acc_free[0]);  // the next piece may be accumulated
  uint32_t p[HC / 2];
#pragma unroll
  for (int q = 0; q < HC / 4; ++q) {
    const float4 b4 = lds4(bias + 16 * q);
    const float2 g0 = gelu_fast2(__fadd2_rn(make_float2(rr[4 * q], rr[4 * q + 1]), make_float2(b4.x, b4.y)));
    const float2 g1 = gelu_fast2(__fadd2_rn(make_float2(rr[4 * q + 2], rr[4 * q + 3]), make_float2(b4.z, b4.w)));
    p[2 * q] = pack_bf16(g0.x, g0.y);
    p[2 * q + 1] = pack_bf16(g1.x, g1.y);
  }
  mbar_wait(&s_mi.h_free, h_phase, &s_mi.abort_flag);  // (a wait that gives up raises the abort flag)
  tc_fence_after();
  tmem_st_row_u32(lane_base + Tm<C>::h + hq * (HC / 2), p);
  tmem_wait_st();
  tc_fence_before();
  mbar_arrive(&s_mi.h_ready);
}

template <int C>
__device__ __forceinline__ void stage_late_vectors() {
  const int i = 4 * threadIdx.x;
  if (i >= 2 * C + s_mi.NF * s_mi.n_f1) return;
  const float* v = i < C ? s_mi.b_o : i < 2 * C ? s_mi.b_2 : s_mi.b_1;
  const int j = i < C ? i : i < 2 * C ? i - C : i - 2 * C;
  const uint32_t dst = s_mi.sbase + s_mi.off_code + 4u * (uint32_t)i;
  if (v) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(v + j) : "memory");
  else sts4(dst, make_float4(0.f, 0.f, 0.f, 0.f));
}

// x rows (fp32) for the first residual: asynchronous 16-byte copies global -> shared staging.
template <int C>
__device__ __forceinline__ void phase_stage_x() {
  constexpr int P = kTM / kUnitRows, J = C / 64;  // as in phase_gather
  const int r0 = threadIdx.x / 16, c0 = threadIdx.x % 16;
  const float* __restrict__ x = s_mi.x;
  const uint32_t to = s_mi.sbase + s_mi.off_kv + stage_off<C>(r0, c0);
  const int rows = s_mi.rows;
  const int* rowvox = s_mi.rowvox[s_mi.buf];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int r = r0 + kUnitRows * p;
    if (r < rows) {
      const int v = rowvox[r];
#pragma unroll
      for (int j = 0; j < J; ++j) {
        const uint32_t dst = to + p * (kUnitRows * C * 4) + j * 256;
        if (v >= 0)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst),
                       "l"(reinterpret_cast<const float4*>(x + (size_t)v * C) + c0 + 16 * j) : "memory");
        else
          sts4(dst, make_float4(0.f, 0.f, 0.f, 0.f));
      }
    }
  }
  stage_late_vectors<C>();
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// fp32 rows staged in shared memory -> coalesced global rows.
template <int C>
__device__ __forceinline__ void phase_store_rows() {
  constexpr int P = kTM / kUnitRows, J = C / 64;  // as in phase_gather
  const int r0 = threadIdx.x / 16, c0 = threadIdx.x % 16;
  float* __restrict__ y = s_mi.y;
  const uint32_t from = s_mi.sbase + s_mi.off_kv + stage_off<C>(r0, c0);
  const int rows = s_mi.rows;
  const int* rowvox = s_mi.rowvox[s_mi.buf];
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int r = r0 + kUnitRows * p, v = r < rows ? rowvox[r] : -1;
    float4 f[J];
#pragma unroll
    for (int j = 0; j < J; ++j) f[j] = lds4(from + p * (kUnitRows * C * 4) + j * 256);
#pragma unroll
    for (int j = 0; j < J; ++j)
      if (v >= 0) reinterpret_cast<float4*>(y + (size_t)v * C)[c0 + 16 * j] = f[j];
  }
}

// LayerNorm over the row that four threads share: t holds this thread's QC values, sum their sum.  Each
// thread reduces its own quarter to (mean, sum of squared deviations), the four pairs are exchanged once
// through 8-byte slots that the caller picks (slot(quarter)) and combined exactly (pairwise update of
// Chan et al.).  The four threads of a row sit in warps q, q + 4, q + 8, q + 12 and meet at a barrier of
// their own.  Leaves t normalised; a caller whose slots are overwritten by the results calls quarter_sync()
// before it stores them.
__device__ __forceinline__ void quarter_sync() {
  asm volatile("bar.sync %0, 128;" ::"r"(2 + ((threadIdx.x >> 5) & 3)) : "memory");
}
template <int C, int QC, class Slot>
__device__ __forceinline__ void layer_norm_rows(float (&t)[QC], float sum, uint32_t gain, uint32_t shift, float eps,
                                                int hq, Slot slot) {
  const float mq = sum * (1.0f / (float)QC);
  float2 sq = make_float2(0.f, 0.f);
#pragma unroll
  for (int i = 0; i < QC; i += 2) {
    const float2 d = __fadd2_rn(make_float2(t[i], t[i + 1]), make_float2(-mq, -mq));
    sq = __ffma2_rn(d, d, sq);
  }
  const float m2 = sq.x + sq.y;
  sts2(slot(hq), make_float2(mq, m2));
  quarter_sync();
  const float2 s0 = lds2(slot(0)), s1 = lds2(slot(1)), s2 = lds2(slot(2)), s3 = lds2(slot(3));
  const float mean = 0.25f * ((s0.x + s1.x) + (s2.x + s3.x));
  const float d0 = s0.x - mean, d1 = s1.x - mean, d2 = s2.x - mean, d3 = s3.x - mean;
  const float ssq = ((s0.y + s1.y) + (s2.y + s3.y)) + (float)QC * ((d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3));
  const float inv = rsqrtf(ssq * (1.0f / (float)C) + eps);
#pragma unroll
  for (int i4 = 0; i4 < QC / 4; ++i4) {
    const float4 g4 = lds4(gain + 4u * (uint32_t)(hq * QC + 4 * i4)), b4 = lds4(shift + 4u * (uint32_t)(hq * QC + 4 * i4));
    const float2 u = __fmul2_rn(__fadd2_rn(make_float2(t[4 * i4], t[4 * i4 + 1]), make_float2(-mean, -mean)), make_float2(inv, inv));
    const float2 w = __fmul2_rn(__fadd2_rn(make_float2(t[4 * i4 + 2], t[4 * i4 + 3]), make_float2(-mean, -mean)), make_float2(inv, inv));
    const float2 y0 = __ffma2_rn(u, make_float2(g4.x, g4.y), make_float2(b4.x, b4.y));
    const float2 y1 = __ffma2_rn(w, make_float2(g4.z, g4.w), make_float2(b4.z, b4.w));
    t[4 * i4] = y0.x; t[4 * i4 + 1] = y0.y; t[4 * i4 + 2] = y1.x; t[4 * i4 + 3] = y1.y;
  }
}

// Output-projection epilogue: t = Z + b_o (+ staged x); LayerNorm 1; then either the fp32 rows go to the
// staging area (mode 0 / 1: final result of the call) or, in TMEM, x1 to the A operand (bf16) and x1 + b_2 back to
// R (fp32), where the MLP-2 MMAs accumulate on top of it.
template <int C, int QC>
__device__ __forceinline__ void phase_epi_o() {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = 32 * (warp & 3) + lane, hq = warp >> 2;
  const uint32_t lane_base = s_mi.tmem_base + ((uint32_t)(32 * (warp & 3)) << 16), taddr = lane_base + Tm<C>::r + hq * QC;
  const uint32_t par = smem_u32(s_mi.par), stage = s_mi.sbase + s_mi.off_kv;
  const int mode = s_mi.mode;
  const uint32_t late = s_mi.sbase + s_mi.off_code;
  const bool add_x = mode != 0 && row < s_mi.rows;
  float t[QC];
  float sum = 0.f;
  tmem_ld_row(taddr, t);
  tmem_wait_ld();
  tc_fence_before();
  if (mode != 2) mbar_arrive(&s_mi.acc_free[2]);  // (R is not used any more)
#pragma unroll
  for (int q = 0; q < QC / 4; ++q) {
    float4 x4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (add_x) x4 = lds4(stage + stage_off<C>(row, hq * (QC / 4) + q));
    const float4 b4 = lds4(late + 4u * (uint32_t)(LateOff<C>::b_o + hq * QC + 4 * q));
    t[4 * q] += x4.x + b4.x;
    t[4 * q + 1] += x4.y + b4.y;
    t[4 * q + 2] += x4.z + b4.z;
    t[4 * q + 3] += x4.w + b4.w;
    sum += (t[4 * q] + t[4 * q + 1]) + (t[4 * q + 2] + t[4 * q + 3]);
  }
  if (mode != 0 && s_mi.ln1) {
    // exchange slots: the first eight bytes of each thread's own (already consumed) x staging chunk
    auto slot = [&](int quarter) { return stage + stage_off<C>(row, quarter * (QC / 4)); };
    layer_norm_rows<C, QC>(t, sum, par + 4 * ParOff<C>::ln1_g, par + 4 * ParOff<C>::ln1_b, s_mi.eps, hq, slot);
  }
  if (mode != 2) {
    compute_sync();  // the x staging (and the exchange slots in it) is dead once every thread has its t
#pragma unroll
    for (int i4 = 0; i4 < QC / 4; ++i4)
      sts4(stage + stage_off<C>(row, hq * (QC / 4) + i4), make_float4(t[4 * i4], t[4 * i4 + 1], t[4 * i4 + 2], t[4 * i4 + 3]));
    return;
  }
#pragma unroll
  for (int c = 0; c < QC / 16; ++c) {
    uint32_t p[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) p[i] = pack_bf16(t[16 * c + 2 * i], t[16 * c + 2 * i + 1]);
    tmem_st8_u32(lane_base + Tm<C>::x1 + hq * (QC / 2) + 8 * c, p);
  }
#pragma unroll
  for (int q = 0; q < QC / 4; ++q) {
    const float4 b4 = lds4(late + 4u * (uint32_t)(LateOff<C>::b_2 + hq * QC + 4 * q));
    t[4 * q] += b4.x;
    t[4 * q + 1] += b4.y;
    t[4 * q + 2] += b4.z;
    t[4 * q + 3] += b4.w;
  }
  tmem_st_row(taddr, t);
  tmem_wait_st();
  tc_fence_before();
}

// MLP-2 epilogue: R holds x1 + b_2 + M; LayerNorm 2; fp32 rows to the staging area.  The exchange slots are the first eight bytes of each
// thread's own output chunk, which is therefore stored last, after one more meeting of the row's threads.
template <int C, int QC>
__device__ __forceinline__ void phase_epi_f2() {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = 32 * (warp & 3) + lane, hq = warp >> 2;
  const uint32_t taddr = s_mi.tmem_base + ((uint32_t)(32 * (warp & 3)) << 16) + Tm<C>::r + hq * QC;
  const uint32_t par = smem_u32(s_mi.par), stage = s_mi.sbase + s_mi.off_kv;
  float t[QC];
  tmem_ld_row(taddr, t);
  tmem_wait_ld();
  tc_fence_before();
  mbar_arrive(&s_mi.acc_free[2]);
  const bool ln = s_mi.ln2 != 0;
  if (ln) {
    float2 sums = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < QC / 2; ++q) sums = __fadd2_rn(sums, make_float2(t[2 * q], t[2 * q + 1]));
    auto slot = [&](int quarter) { return stage + stage_off<C>(row, quarter * (QC / 4)); };
    layer_norm_rows<C, QC>(t, sums.x + sums.y, par + 4 * ParOff<C>::ln2_g, par + 4 * ParOff<C>::ln2_b, s_mi.eps, hq, slot);
  }
#pragma unroll
  for (int i4 = 1; i4 < QC / 4; ++i4)
    sts4(stage + stage_off<C>(row, hq * (QC / 4) + i4), make_float4(t[4 * i4], t[4 * i4 + 1], t[4 * i4 + 2], t[4 * i4 + 3]));
  if (ln) quarter_sync();  // the row's other threads have read this thread's slot
  sts4(stage + stage_off<C>(row, hq * (QC / 4)), make_float4(t[0], t[1], t[2], t[3]));
}

// The layer's vectors of the parameter block (absent ones as zeros; order of ParOff: b_q, b_v, ln1_g, ln1_b, ln2_g,
// ln2_b; the key bias is not needed), its scalars and the pointers to the other vectors.
template <int C>
__device__ __forceinline__ void load_layer_params(const TcLayer& ly) {
  const uint32_t par = smem_u32(s_mi.par);
  // asynchronous 4-byte copies, all in flight at once: the first reader is the V epilogue, which waits for them
  // (wait_layer_params) after the K epilogue
  for (int i = threadIdx.x; i < ParOff<C>::vectors * C; i += kComputeThreads) {
    const int which = i / C;
    const float* v = which == 0 ? ly.b_qkv : which == 1 ? (ly.b_qkv ? ly.b_qkv + 2 * C : nullptr) : which == 2 ? ly.ln1_g
                   : which == 3 ? ly.ln1_b : which == 4 ? ly.ln2_g : ly.ln2_b;
    if (v) asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(par + 4u * (uint32_t)i), "l"(v + i % C) : "memory");
    else s_mi.par[i] = 0.f;
  }
  if (threadIdx.x == 0) {
    s_mi.ln1 = ly.ln1_g != nullptr;
    s_mi.ln2 = ly.ln2_g != nullptr;
    s_mi.eps = ly.eps;
    s_mi.b_o = ly.b_o; s_mi.b_1 = ly.b_1; s_mi.b_2 = ly.b_2;
    s_mi.rpb = ly.rpb;
    s_mi.pe = ly.pe;
  }
}

__device__ __forceinline__ void wait_layer_params() {
  asm volatile("cp.async.wait_all;" ::: "memory");
  compute_sync();
}

// Barrier over the compute threads that also ANDs a predicate.
__device__ __forceinline__ bool compute_all(bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %2, 0;\n\t"
      "bar.red.and.pred p, 1, %1, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "n"(kComputeThreads), "r"((uint32_t)pred)
      : "memory");
  return r != 0;
}

// The tile loop keeps as little as possible alive across the phase calls (the tile's index k, and two flags): what it
// holds, every phase has fewer registers, and with 227 KB of shared memory taken there is no L1 left for spills.
template <int C, int D, int VAR>
__device__ __forceinline__ void compute_role(const TcArgs& a) {
  constexpr bool RPB = VAR == 1, PE = VAR == 2;
  constexpr int QC = C / 4;          // epilogue columns per thread for a C-wide chunk (four threads per row)
  volatile int* abort_flag = &s_mi.abort_flag;
  bool gathered = false;  // the tile about to start was gathered under the previous tile's MLP
  int cur_layer = -1;     // layer whose vectors are in the parameter block
  // The next tile's rows are gathered as soon as the current tile's MMAs have stopped reading the A operand (the
  // output projection is the last), so that its first projections run on the tensor pipe while the compute warps finish
  // the current tile; unless its rows are not all stamped yet: then the gather waits until this tile is done (the row
  // that is missing may be one of this tile's own).
  auto gather_next = [&](int k) {
    const int b = (k + 1) & 1;
    WAIT_PHASE(rl_ready[b], (k + 1) >> 1);
    const int nr = s_mi.next_rows[b];
    if (compute_all(nr >= 0 && *abort_flag == 0 && mbar_try(&s_mi.dep_ready[b], (uint32_t)((k + 1) >> 1) & 1u))) {
      phase_gather<C, D, RPB, false>(b, nr);
      fence_proxy_async();
      mbar_arrive(&s_mi.x_ready);
      gathered = true;
    }
  };
  int k = 0;
  for (;; ++k) {
    WAIT_PHASE(sched_full[k & 1], k >> 1);
    // also orders the previous tile's last shared-memory reads before this tile's writes; every exit from
    // this loop is taken by all compute threads together
    if (bar_or(1, kComputeThreads, *abort_flag != 0)) break;
    const int nsets = s_mi.tile[k & 1][1], layer = s_mi.tile[k & 1][4];
    if (threadIdx.x == 0) {
      s_mi.rows = s_mi.tile[k & 1][3];
      s_mi.buf = k & 1;
      s_mi.x = layer == 0 ? a.x : a.y;
      s_mi.st_stamp[k & 1] = a.n_layers > 1 ? a.stamp_base + layer + 1 : 0;
      if (k >= 1) mbar_arrive(&s_mi.rl_free[(k - 1) & 1]);  // the previous tile's row list is dead
    }
    mbar_arrive(&s_mi.sched_empty[k & 1]);
    if (nsets < 0) break;
    const bool new_params = layer != cur_layer;
    if (new_params) {  // (the previous tile's last use of the block lies before the barrier above)
      load_layer_params<C>(a.layer[layer]);
      cur_layer = layer;
    }
    if (!gathered) {  // a CTA's first tile, or a tile whose rows were not ready in time
      WAIT_PHASE(rl_ready[k & 1], k >> 1);
      WAIT_PHASE(dep_ready[k & 1], k >> 1);
      if (compute_all(*abort_flag == 0)) {
        phase_gather<C, D, RPB, false>(k & 1, s_mi.next_rows[k & 1]);
        fence_proxy_async();
      }
      mbar_arrive(&s_mi.x_ready);  // X is in place
    }
    gathered = false;
    compute_sync();  // the tile's fields are visible to the phase functions

    // (uses of the accumulators before this tile: V and R one each per tile, the first one K, Q and the MLP-1 pieces)
    // ---- chunks 0..2: K, V, Q epilogues: (+ bias,) to bf16, into the operand layout ----
    if (PE) {
      // the values come from the bare rows; the operand is then rewritten with the positional term added, for
      // the keys and the queries (the V chunk's accumulator being complete, nothing reads the operand any more)
      WAIT_PHASE(acc_full[1], k);
      if (new_params) wait_layer_params();
      phase_epi_bf16<QC, true, false>(Tm<C>::v, 1, ParOff<C>::b_v, s_mi.off_kv + (C / 8) * kChunkBytes);
      phase_gather<C, D, false, true>(k & 1, s_mi.rows);
      fence_proxy_async();
      mbar_arrive(&s_mi.x_ready);
      WAIT_PHASE(acc_full[0], k * (2 + s_mi.n_f1));
      phase_epi_bf16<QC, false, false>(Tm<C>::k, 0, 0, s_mi.off_kv);
    } else {
      WAIT_PHASE(acc_full[0], k * (2 + s_mi.n_f1));
      phase_epi_bf16<QC, false, false>(Tm<C>::k, 0, 0, s_mi.off_kv);
      WAIT_PHASE(acc_full[1], k);
      if (new_params) wait_layer_params();  // (the key epilogue adds no bias: it needs none of the vectors)
      phase_epi_bf16<QC, true, false>(Tm<C>::v, 1, ParOff<C>::b_v, s_mi.off_kv + (C / 8) * kChunkBytes);
    }
    WAIT_PHASE(acc_full[0], k * (2 + s_mi.n_f1) + 1);
    if (PE) compute_sync();  // (every thread has marked the sets of its rows with the positional term)
    phase_epi_bf16<QC, true, true>(Tm<C>::k, 0, ParOff<C>::b_q, s_mi.off_a);
    fence_proxy_async();
    mbar_arrive(&s_mi.a_ready);  // Q, K and V are in place
    // ---- attention inside each set ----
    attend<C, D, RPB>(k);
    fence_proxy_async();
    mbar_arrive(&s_mi.a_ready);  // attention output is the A operand of the output projection
    compute_sync();              // every warp is done with K and V: their region becomes fp32 staging
    if (s_mi.mode != 0) {
      phase_stage_x<C>();
    } else {
      stage_late_vectors<C>();
      asm volatile("cp.async.wait_all;" ::: "memory");
    }
    compute_sync();
    // ---- output projection epilogue: Z + b_o (+ x, LayerNorm) ----
    WAIT_PHASE(o_full, k);
    phase_epi_o<C, QC>();
    if (s_mi.mode != 2) {  // final result of this layer
      gather_next(k);
    } else {
      mbar_arrive(&s_mi.a_ready);  // x1 (bf16) is the A operand of MLP-1
      // ---- MLP-1 pieces ----
      for (int c = 0; c < s_mi.n_f1; ++c) {
        WAIT_PHASE(acc_full[0], k * (2 + s_mi.n_f1) + 2 + c);
        const uint32_t h_phase = (uint32_t)(k * s_mi.n_f1 + c + 1) & 1u;
        if (s_mi.NF == 128) phase_mlp1<C, 32>(LateOff<C>::b_1 + c * 128, h_phase);
        else phase_mlp1<C, 16>(LateOff<C>::b_1 + c * 64, h_phase);
      }
      gather_next(k);  // (the operand has been free since the output projection; under the first MLP-1 product it is slower)
      // ---- MLP-2 epilogue: y = LN2(x1 + M) ----
      WAIT_PHASE(acc_full[2], k);
      phase_epi_f2<C, QC>();
    }
    compute_sync();
    phase_store_rows<C>();
    if (threadIdx.x == 0) s_mi.st_rows[k & 1] = s_mi.rows;
    mbar_arrive(&s_mi.stored[k & 1]);  // the stamp warp takes it from here
  }
  // tell the stamp warp to leave at iteration k, once it is done with tile k - 2 (which signalled on the same barrier)
  if (k >= 2) WAIT_PHASE(rl_free[k & 1], (k >> 1) - 1);
  if (threadIdx.x == 0) s_mi.exit_at = k;
  mbar_arrive(&s_mi.stored[k & 1]);
  if (threadIdx.x == 0 && *abort_flag) atomicOr(s_mi.status, DSVT_STATUS_TIMEOUT);
}

// ---------------------------------------------------------------------------------------------
// The kernel
// ---------------------------------------------------------------------------------------------
// VAR: 0 plain, 1 relative position bias on the logits, 2 additive positional term on the query / key inputs
template <int C, int D, int VAR>
__global__ void __launch_bounds__(kThreads, 1) layer_tc_kernel(const __grid_constant__ TcArgs a) {
  constexpr bool RPB = VAR == 1;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sm = smem_raw;  // 1024-aligned: the static block before it fills whole kilobytes
  Misc* mi = &s_mi;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (warp-uniform)
  const TcGeom& g = a.g;
  if (tid == 0) {  // launch constants for the phase functions
    mi->abort_flag = (smem_u32(smem_raw) & 1023u) != 0;  // (never: checked because the layouts rest on it)
    mi->exit_at = -1;
    mi->x = a.x; mi->y = a.y; mi->status = a.status;
    mi->sbase = smem_u32(sm);
    mi->off_a = g.off_a; mi->off_kv = g.off_kv; mi->off_code = g.off_code;
    mi->n = a.n; mi->tau = g.tau; mi->heads = g.heads; mi->mode = g.mode; mi->NF = g.NF; mi->n_f1 = g.n_f1;
    mi->ln1 = mi->ln2 = 0;
    mi->eps = 0.f;
    mi->b_o = mi->b_1 = mi->b_2 = nullptr;
    mi->rpb = nullptr; mi->pe = nullptr; mi->coords = a.coords;
    mi->rb_len = g.rb_len; mi->rb_sx = g.rb_sx; mi->rb_sy = g.rb_sy; mi->rb_centre = g.rb_centre;
    mi->rb_ext[0] = g.rb_ext[0]; mi->rb_ext[1] = g.rb_ext[1]; mi->rb_ext[2] = g.rb_ext[2];
    mi->rows = mi->buf = 0;
    mi->next_rows[0] = mi->next_rows[1] = -1;
    mi->next_x[0] = mi->next_x[1] = a.x;
    mi->st_rows[0] = mi->st_rows[1] = mi->st_stamp[0] = mi->st_stamp[1] = 0;
  }
  if (tid == 32 * kLoadWarp0) {  // barriers
    for (int i = 0; i < kStages; ++i) { mbar_init(&mi->full[i], 1); mbar_init(&mi->empty[i], 1); }
    for (int i = 0; i < 3; ++i) {
      mbar_init(&mi->acc_full[i], 1);
      mbar_init(&mi->acc_free[i], kComputeThreads);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&mi->sched_full[i], 1);
      mbar_init(&mi->sched_empty[i], kComputeThreads + 1 + kLoadWarps);  // compute threads, MMA issuer, loader warp
      mbar_init(&mi->rl_free[i], 2);  // the compute warps' first thread and the stamp warp
      mbar_init(&mi->rl_ready[i], kLoadThreads);
      mbar_init(&mi->dep_ready[i], kLoadThreads);
      mbar_init(&mi->stored[i], kComputeThreads);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(&mi->s_full[i], 1);
      mbar_init(&mi->p_ready[i], kComputeThreads / 4);
      mbar_init(&mi->ov_full[i], 1);
      mbar_init(&mi->o_read[i], kComputeThreads / 4);
    }
    mbar_init(&mi->o_full, 1);
    mbar_init(&mi->h_ready, kComputeThreads);
    mbar_init(&mi->h_free, 1);
    mbar_init(&mi->a_ready, kComputeThreads);
    mbar_init(&mi->x_ready, kComputeThreads);
    mbar_init(&mi->drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&mi->tmem_base)),
                 "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // keys past a tile's rows meet zero probabilities: never let K, V or the chunks behind V hold uninitialised bit
  // patterns there (0 x NaN)
  for (uint32_t i = tid; i < (g.off_stage - g.off_kv + kStages * (uint32_t)C * 128u) / 16; i += kThreads)
    reinterpret_cast<uint4*>(sm + g.off_kv)[i] = make_uint4(0u, 0u, 0u, 0u);
  fence_proxy_async();  // the TMA writes that follow must not be overtaken by these generic stores
  // everything above touched only this CTA's own state; from here on the kernel reads what earlier kernels in the
  // stream wrote (tables, features, the launch counters): wait for them if this launch was allowed to start early
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  RoleCtx rc;
  rc.sbase = smem_u32(sm);
  rc.tmem = __shfl_sync(0xffffffffu, mi->tmem_base, 0);
  rc.mode = g.mode; rc.n_f1 = g.n_f1; rc.NF = g.NF; rc.tau = g.tau; rc.n_layers = a.n_layers; rc.heads = g.heads;
  rc.off_a = g.off_a; rc.off_kv = g.off_kv; rc.off_code = g.off_code; rc.off_stage = g.off_stage;
  rc.pe = VAR == 2;

  if (warp == kTmaWarp) {
    if ((tid & 31) == 0) producer_role<C>(a, rc);
    __syncwarp();
  } else if (warp == kMmaWarp) {
    mma_role<C, D>(rc);
    __syncwarp();
  } else if (warp == kStampWarp) {
    stamp_role(a.row_stamp);
  } else if (warp >= kLoadWarp0) {
    loader_role<C, RPB>(a);
  } else {
    compute_role<C, D, VAR>(a);
  }
  // ---- teardown: everyone meets here, then the allocating warp returns the TMEM columns ----
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(rc.tmem), "r"(kTmemCols) : "memory");
  }
  // the last CTA to leave puts the launch's counters back to zero for the next launch on this context
  if (tid == 0) {
    const int left = atomicAdd(a.counter + 1, 1);
    if (left == (int)gridDim.x - 1) {
      a.counter[0] = 0;
      a.counter[1] = 0;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static std::once_flag once;
  static EncodeTiledFn fn = nullptr;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  });
  return fn;
}

// bf16 matrix [rows][cols] row-major; box = 64 columns x box_rows rows, 128-byte swizzle.
bool make_weight_map(CUtensorMap* m, const void* w, int rows, int cols, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1u, 1u};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(w), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Tensor maps are encoded once per (matrix, shape, box) and context and kept: a backbone calls the same layers
// frame after frame.
struct dsvt_map_cache {
  struct Entry {
    const void* w;
    int rows, cols, box_rows;
    CUtensorMap map;
  };
  std::vector<Entry> entries;
  unsigned attr_done = 0;  // kernel instantiations whose shared-memory attribute is set on this context's device
};

void dsvt_map_cache_destroy(dsvt_map_cache* c) { delete c; }

namespace {

bool cached_weight_map(dsvt_ctx* ctx, CUtensorMap* out, const void* w, int rows, int cols, int box_rows) {
  if (!ctx->maps) ctx->maps = new (std::nothrow) dsvt_map_cache();
  if (!ctx->maps) return false;
  auto& v = ctx->maps->entries;
  for (const auto& e : v)
    if (e.w == w && e.rows == rows && e.cols == cols && e.box_rows == box_rows) { *out = e.map; return true; }
  dsvt_map_cache::Entry e;
  e.w = w; e.rows = rows; e.cols = cols; e.box_rows = box_rows;
  if (!make_weight_map(&e.map, w, rows, cols, box_rows)) return false;
  if (v.size() >= 256) v.erase(v.begin(), v.begin() + 128);  // (a caller that keeps changing its weights)
  v.push_back(e);
  *out = e.map;
  return true;
}

template <int C, int D, int VAR>
int launch_tc_one(dsvt_ctx* ctx, const TcArgs& a, int grid, size_t smem, int inst) {
  if (!(ctx->maps->attr_done & (1u << inst))) {  // once per instantiation and context (the attribute is per device)
    cudaError_t e = cudaFuncSetAttribute(layer_tc_kernel<C, D, VAR>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) { ctx->last_cuda_error = (int)e; return DSVT_ERR_CUDA; }
    ctx->maps->attr_done |= 1u << inst;
  }
  // launched so that it may be set up under the tail of the kernel before it in the stream (the partition, an
  // earlier chain): the kernel waits for that kernel's completion before it reads anything but its parameters
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = smem; cfg.stream = ctx->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  cudaError_t le = cudaLaunchKernelEx(&cfg, layer_tc_kernel<C, D, VAR>, a);
  if (le != cudaSuccess) { ctx->last_cuda_error = (int)le; cudaGetLastError(); return DSVT_ERR_CUDA; }
  DSVT_LAUNCHED(ctx);
  return DSVT_OK;
}

// The position bias and the positional term are compile-time variants: a layer without them runs a kernel that
// holds none of their code.
template <int C, int D>
int launch_tc(dsvt_ctx* ctx, const TcArgs& a, int grid, size_t smem, int inst) {
  if (a.g.rb_len != 0) return launch_tc_one<C, D, 1>(ctx, a, grid, smem, 3 * inst + 1);
  if (a.layer[0].pe) {
    // (the variant with a positional term is built for the paper's shape only: C = 192)
    if constexpr (C == 192) return launch_tc_one<C, D, 2>(ctx, a, grid, smem, 3 * inst + 2);
    return DSVT_ERR_UNSUPPORTED;
  }
  return launch_tc_one<C, D, 0>(ctx, a, grid, smem, 3 * inst);
}

int tc_hidden(const dsvt_fused_args& a) { return a.attention_only ? 0 : a.p.hidden; }

}  // namespace

// Shapes the tensor-core kernel covers; everything else goes to the FMA kernel.
bool dsvt_layer_tc_supported(const dsvt_fused_args& a) {
  const dsvt_layer_params& p = a.p;
  if (p.precision != DSVT_BF16_FP32ACC) return false;
  if (p.pe && (p.rpb || p.C != 192 || p.set_size > 48)) return false;  // (see launch_tc)
  if (p.rpb) {
    // row coordinates are kept as linear indices modulo 2^16 and differences are taken modulo 2^16: exact while every
    // offset inside a covered set, at most (len - 1) / 2 in magnitude, is below 2^15
    const int64_t len = (int64_t)(2 * p.rpb_extent[0] - 1) * (2 * p.rpb_extent[1] - 1) * (2 * p.rpb_extent[2] - 1);
    if (len > 65535) return false;
  }
  const int d = p.C / p.heads;
  const bool shape = (p.C == 192 && d == 24) || (p.C == 128 && (d == 16 || d == 32)) || (p.C == 64 && d == 16);
  if (!shape || p.set_size > 96) return false;
  const int hidden = tc_hidden(a);
  if (hidden != 0 && hidden != p.C && hidden != 2 * p.C) return false;
  return encode_fn() != nullptr;
}

// Two layers can share a launch if they have the same shape (one kernel instantiation, one geometry).
bool dsvt_layer_tc_chainable(const dsvt_fused_args& a, const dsvt_fused_args& b) {
  const dsvt_layer_params &p = a.p, &q = b.p;
  if (a.attention_only || b.attention_only || a.n != b.n || a.y != b.y) return false;
  if (p.C != q.C || p.heads != q.heads || tc_hidden(a) != tc_hidden(b) || p.set_size != q.set_size) return false;
  if ((p.rpb != nullptr) != (q.rpb != nullptr) || (p.pe != nullptr) != (q.pe != nullptr)) return false;
  if (p.rpb && (p.coords != q.coords || p.rpb_extent[0] != q.rpb_extent[0] || p.rpb_extent[1] != q.rpb_extent[1] ||
                p.rpb_extent[2] != q.rpb_extent[2]))
    return false;
  return true;
}

// One launch for layers[0 .. n_layers): layers[0] reads its x and writes y, every later layer runs in place on y
// (its x must be that y).  All layers pass dsvt_layer_tc_supported and are chainable with layers[0].
int dsvt_launch_layers_tc(dsvt_ctx* ctx, const dsvt_fused_args* layers, int n_layers) {
  if (n_layers < 1 || n_layers > kMaxLayers) return DSVT_ERR_INVALID_ARG;
  if (!ctx->maps) ctx->maps = new (std::nothrow) dsvt_map_cache();
  if (!ctx->maps) return DSVT_ERR_CUDA;
  const dsvt_fused_args& a0 = layers[0];
  const dsvt_layer_params& p = a0.p;
  const int C = p.C;
  TcArgs ta = {};
  TcGeom& g = ta.g;
  g.hidden = tc_hidden(a0);
  g.heads = p.heads;
  g.tau = p.set_size;
  g.mode = a0.attention_only ? 0 : (g.hidden > 0 ? 2 : 1);
  g.NF = (g.hidden % 128 == 0 && C >= 128) ? 128 : 64;
  g.n_f1 = g.hidden / g.NF;
  g.rb_len = g.rb_sx = g.rb_sy = g.rb_centre = 0;
  g.rb_ext[0] = g.rb_ext[1] = g.rb_ext[2] = 0;
  if (p.rpb) {
    const int L = p.rpb_extent[0], W = p.rpb_extent[1], H = p.rpb_extent[2];
    g.rb_sy = 2 * H - 1;
    g.rb_sx = (2 * W - 1) * g.rb_sy;
    g.rb_len = (2 * L - 1) * g.rb_sx;
    g.rb_centre = (L - 1) * g.rb_sx + (W - 1) * g.rb_sy + (H - 1);
    g.rb_ext[0] = L; g.rb_ext[1] = W; g.rb_ext[2] = H;
  }
  const int d = C / p.heads;
  g.off_a = 0;
  g.off_kv = (uint32_t)kTM * C * 2;
  g.off_code = g.off_kv + (uint32_t)kTM * 2 * C * 2;  // K + V (bf16) = fp32 staging bytes
  g.off_stage = g.off_code + 2 * (d == 24 ? 1 : 2) * kChunkBytes;
  const size_t smem = (size_t)g.off_stage + kStages * (size_t)C * 128;
  if (smem + sizeof(Misc) > 227 * 1024) return DSVT_ERR_UNSUPPORTED;  // s_mi is static shared memory
  int64_t grid = 1;
  for (int l = 0; l < n_layers; ++l) {
    const dsvt_fused_args& a = layers[l];
    const dsvt_layer_params& q = a.p;
    TcLayer& ly = ta.layer[l];
    bool okm = cached_weight_map(ctx, &ly.qkv, q.W_qkv, 3 * C, C, C) && cached_weight_map(ctx, &ly.o, q.W_o, C, C, C);
    if (g.hidden > 0)
      okm = okm && cached_weight_map(ctx, &ly.w1, q.W_1, g.hidden, C, g.NF) &&
            cached_weight_map(ctx, &ly.w2, q.W_2, C, g.hidden, C);
    else {
      ly.w1 = ly.o;
      ly.w2 = ly.o;
    }
    if (!okm) return DSVT_ERR_CUDA;
    ly.b_qkv = q.b_qkv; ly.b_o = q.b_o; ly.rpb = q.rpb; ly.pe = q.pe;
    const bool full = !a.attention_only;
    ly.b_1 = full ? q.b_1 : nullptr; ly.b_2 = full ? q.b_2 : nullptr;
    ly.ln1_g = full ? q.ln1_g : nullptr; ly.ln1_b = full ? q.ln1_b : nullptr;
    ly.ln2_g = full ? q.ln2_g : nullptr; ly.ln2_b = full ? q.ln2_b : nullptr;
    ly.table = a.table; ly.num_sets = a.num_sets; ly.rowoff = a.rowoff; ly.cap_sets = a.cap_sets;
    ly.eps = q.ln_eps;
    const int64_t cap = a.cap_sets < a.n ? a.cap_sets : a.n;
    if (cap > grid) grid = cap;
  }
  ta.x = a0.x; ta.y = a0.y; ta.n = a0.n; ta.n_layers = n_layers;
  ta.coords = reinterpret_cast<const int4*>(p.coords);
  ta.counter = ctx->tc_counter;
  ta.row_stamp = ctx->row_stamp;
  ctx->stamp_serial = (ctx->stamp_serial + 1) & 0x3ffffff;  // (stamps of launches 2^26 apart never meet)
  if (ctx->stamp_serial == 0) ctx->stamp_serial = 1;
  ta.stamp_base = (int32_t)(ctx->stamp_serial * 32u);
  ta.status = ctx->status;
  // one CTA per SM, but no more CTAs than there can be sets
  if (grid > ctx->sm_count) grid = ctx->sm_count;
  if (ctx->layer_ctas > 0 && grid > ctx->layer_ctas) grid = ctx->layer_ctas;
  if (grid < 1) grid = 1;
  if (C == 192) return launch_tc<192, 24>(ctx, ta, (int)grid, smem, 0);
  if (C == 128 && d == 16) return launch_tc<128, 16>(ctx, ta, (int)grid, smem, 1);
  if (C == 128) return launch_tc<128, 32>(ctx, ta, (int)grid, smem, 2);
  return launch_tc<64, 16>(ctx, ta, (int)grid, smem, 3);
}

int dsvt_launch_layer_tc(dsvt_ctx* ctx, const dsvt_fused_args& a) { return dsvt_launch_layers_tc(ctx, &a, 1); }

// Tensor map of a row-major bf16 matrix [rows][cols] for boxes of 64 columns x box_rows rows with the 128-byte swizzle (the
// layout every operand tile here uses), from the context's cache; false if the driver entry point is missing or refuses.
bool dsvt_cached_weight_map(dsvt_ctx* ctx, void* tensor_map, const void* w, int rows, int cols, int box_rows) {
  return cached_weight_map(ctx, reinterpret_cast<CUtensorMap*>(tensor_map), w, rows, cols, box_rows);
}
