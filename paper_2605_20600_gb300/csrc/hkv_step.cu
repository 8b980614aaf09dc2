// One decode step of one layer in a single launch: attention of every head's
// new query over the head's retained tokens and the step's new token (Eq. 1),
// fused with the append of that token to the cache (Sec. 3, KV Cache); with
// the head types decided in the same pass (Sec. 4, Step 2); or the attention
// alone.
//
// What bounds it: the K/V rows, read once (91 MB a layer on Lumina-mGPT 1024
// at rho = 1/4, 8 sequences: 13.4 us at the measured copy bandwidth), plus a
// part that does not grow with them: the last tiles, the merges, the next
// launch's start, prologue and first loads, during which DRAM is mostly idle.
// Timings below are per layer step, whole period, before -> after.
//
//  * split: a head takes one slot per 16 rows (8 of 512 bytes) and one more
//    (StepShape::cost); the layer's slots are cut into gridDim.x equal
//    contiguous ranges, one per CTA, and a cut within a quarter of a range of
//    a head's first or last row moves there (HKV_STEP_SNAP_DIV: cuts cost a
//    merge and two partial tiles; 1/64 of a range 16.87 us, 1/16 16.65, 1/4
//    16.44 on Lumina-mGPT 1024). Slots of whole tiles, as before, left CTAs
//    with up to 9 of LlamaGen-XL's heads where 8.4 is the mean: 16.4 -> 14.9
//    us there with the prologue below;
//  * a layer of short heads, no more than CTAs, gets a CTA per head
//    (kAlignedGrains), and a small layer a grid no larger than its ranges:
//    nothing is merged and every CTA of the next launch is resident before
//    this one ends (Janus-Pro-7B, 2 sequences: 6.6 -> 3.4 us);
//  * a layer of many short heads is not cut at all: CTAs take heads from a
//    counter (kHeadSlots; Janus-Pro-7B, 256 sequences: 94.5 -> 89.0 us of 87.8
//    at the measured bandwidth);
//  * a warp-specialised TMA pipeline: a producer warp, consumer warps, an
//    epilogue warp and a merge warp;
//  * bf16 consumers take q.k on the tensor cores (8 rows a warp and tile: 4
//    mma.sync of D = 128 in place of 64 mixed FMAs and 32 shuffles) and p.V in
//    fp32 FMAs. The products are exact; in which order and with which rounding
//    mma.sync adds them is not specified. The outputs' error against 64 bits
//    was 7.5e-7 at most over the timed calls before and is 6.5e-7, mostly since
//    the exponent is rounded once. The chain of a tile is what a CTA waits for:
//    0.8 us less of Lumina-mGPT 1024's step than with FMAs and shuffles. p.V on the tensor cores too, with the
//    weights cut into three bf16 parts and the rows skewed against the banks,
//    measured 1.7 us slower: the eight small copies a tile then needs;
//  * tile order: a CTA streams the start of the head that continues into a
//    later range first, then the piece of the head that began in an earlier
//    range, then the heads wholly inside its range. The piece a CTA streams
//    first is never the one that CTA combines, so a head in two pieces
//    never waits for a piece that finishes last in its CTA (measured: 0.3
//    us per step less than the other order at rho = 1/8);
//  * merges: a split head is combined by its first middle CTA (whose whole
//    range lies inside the head), else (and always in the attention alone and
//    in the step that decides the head types) by the CTA holding its last
//    row. The other pieces write their partial result to the workspace as
//    64-bit (value, launch epoch) pairs, which are single-copy atomic, so no fence
//    or flag is needed: the combining CTA's merge warp reads the pieces until
//    every pair carries this launch's epoch, while its consumers stream.
//    Pieces are combined in index order and the CTA's own piece last, so the
//    result does not depend on timing;
//  * prologue: see there;
//  * appends and counters: every CTA arrives on a per-layer barrier word
//    once it is done reading the layer's counters (a CTA that found a bad
//    head marks its arrival); once the whole grid has arrived, and unless
//    one was marked, the merge warp advances len, ntok and nbuf of the heads
//    whose last row is in the CTA's range, while the consumers stream. Their
//    new tokens go into the cache then too, or at once where every CTA has
//    checked every head (nothing in the launch reads those rows). The next
//    launch of the same layer starts after this one completes, so the
//    barrier word is free again by then;
//  * programmatic dependent launch: with the prefetch flag the prologue, the
//    arrival and the first tiles of old K/V rows go ahead of the wait for the
//    previous kernel; the step's inputs (q, the new k and v) are read after
//    it;
//  * every wait is bounded (HKV_ERR_TIMEOUT in the error word). A plain step's
//    waits on other CTAs need the whole grid resident: it is at most what
//    fits. In the attention alone and in the step that decides the head types
//    a CTA waits for lower-numbered ones only, which start before it; what
//    the latter's barrier holds up is left to the last CTA to arrive (see the
//    merge warp).
#include <math.h>
#include <stdlib.h>

#include "hkv_attn_common.cuh"
#include "hkv_device.cuh"
#include "hkv_kernels.h"

namespace hkv {
namespace {

#ifdef HKV_ATTN_TRACE
__device__ unsigned long long *g_step_trace = nullptr;  // [layer][kAttnMaxGrid][32]
#define STEP_TRACE_AT(slot) \
  g_step_trace[((size_t)(p.layer_base / p.nheads) * kAttnMaxGrid + blockIdx.x) * 32 + (slot)]
#define STEP_TRACE(slot)                                    \
  do {                                                      \
    if (g_step_trace) STEP_TRACE_AT(slot) = globaltimer(); \
  } while (0)
#define STEP_TRACE_SET(slot, v)                 \
  do {                                          \
    if (g_step_trace) STEP_TRACE_AT(slot) = (v); \
  } while (0)
#define STEP_CLK() clock64()
#else
#define STEP_CLK() 0ll
#define STEP_TRACE(slot) \
  do {                   \
  } while (0)
#define STEP_TRACE_SET(slot, v) \
  do {                          \
    (void)(v);                  \
  } while (0)
#endif

// Tuning knobs (compile time) of the one-launch step, per head dimension:
// consumer warps, bytes of K per stage, stages, tiles loaded before the wait,
// and the CTAs per SM the kernel is built to be resident with (the grid uses
// kStepActivePerSm). Rows of 256 B: 64-row tiles in 3 stages and 48-row ones
// with 6 warps are within 0.3 % of each other on large layers, 64 rows 2 %
// faster on small ones (4 stages of 48 rows +0.1 to +1.7 us, 2 stages +0.7).
// Rows of 512 B: 32-row tiles in 3 stages leave 0 bytes of an SM beside two
// CTAs; kLoneSlots says where one has the SM.
// Rows of 128 B (LlamaGen-XL's short heads, many to a CTA): 128-row tiles in
// 2 stages, 64-row ones in 3 +0.8 us. A third resident CTA per SM, so that
// the next launch's CTAs start early, leaves some SMs with three CTAs of one
// launch and others with one: +1.4 to +2.3 us.
#ifndef HKV_STEP_TILE_BYTES_D128
#define HKV_STEP_TILE_BYTES_D128 16384
#endif
#ifndef HKV_STEP_STAGES_D128
#define HKV_STEP_STAGES_D128 3
#endif
#ifndef HKV_STEP_PRE_D128
#define HKV_STEP_PRE_D128 3
#endif
#ifndef HKV_STEP_TILE_BYTES_D64
#define HKV_STEP_TILE_BYTES_D64 16384
#endif
#ifndef HKV_STEP_STAGES_D64
#define HKV_STEP_STAGES_D64 2
#endif
#ifndef HKV_STEP_PRE_D64
#define HKV_STEP_PRE_D64 2
#endif
#ifndef HKV_STEP_RESIDENT_PER_SM
#define HKV_STEP_RESIDENT_PER_SM 2
#endif
#ifndef HKV_STEP_CW_D128
#define HKV_STEP_CW_D128 8
#endif
#ifndef HKV_STEP_CW_D64
#define HKV_STEP_CW_D64 8
#endif
// consumer warps: a bf16 tile is a number of 8-row blocks for each of them
constexpr int step_cw(int D, int es) {
  return es == 4 ? 8 : D == 64 ? HKV_STEP_CW_D64 : HKV_STEP_CW_D128;
}

// Heads of at most this many grains (96 KB of K and V) are not split when
// every head can have a CTA of its own: the exchange of partial results
// costs more than the tiles it saves.
constexpr int kAlignedGrains = 12;

constexpr int step_grain(int row_bytes) { return row_bytes == 512 ? 8 : 16; }  // rows

// SHORT: the shape for layers whose every head fits kAlignedGrains: one stage
// that holds a whole head, so that the consumers pass over it once.
template <int D, typename T, bool SHORT>
using StepTile = TileShape<
    D, T, step_cw(D, sizeof(T)),
    SHORT     ? kAlignedGrains * step_grain(D * sizeof(T)) * D * (int)sizeof(T)
    : D == 64 ? HKV_STEP_TILE_BYTES_D64
              : HKV_STEP_TILE_BYTES_D128,
    SHORT ? 1 : D == 64 ? HKV_STEP_STAGES_D64 : HKV_STEP_STAGES_D128,
    SHORT ? 1 : D == 64 ? HKV_STEP_PRE_D64 : HKV_STEP_PRE_D128>;

template <int D, typename T, bool SHORT = false>
struct StepShape : StepTile<D, T, SHORT> {
  using Tile = StepTile<D, T, SHORT>;
  // states a segment hands over: one per consumer warp, or (fp32) per row group
  static constexpr int kNST = sizeof(T) == 2 ? Tile::kCW : Tile::kCW * Tile::kRPW;
  // The split counts in grains of kGR rows (4 or 8 KB of K and V). A head of
  // g grains takes g + 1 slots, at least kMinCost: the extra one stands for
  // what a head costs beyond its rows (a hand-over, a partial tile), and the
  // minimum bounds the heads of a range (step_max_heads).
  static constexpr int kGR = step_grain(Tile::kRB);
  static constexpr int kMinCost = Tile::kRB == 128 ? 5 : 3;
  // Fewest slots of a CTA's range: on small layers a longer range costs less
  // than one more piece to combine. Periods of steps over 12 layers of
  // Lumina-mGPT 1024 at rho = 1/6, ms with 2, 3, 4, 5, 6 and 8 tiles: one
  // sequence 5.85, 5.29, 5.05, 5.34, 5.55, 6.27, two sequences 6.66, 6.26,
  // 6.00, 6.33, 6.45, 6.94. Other shapes, us per layer step with 3, 4 and 6:
  // Lumina-mGPT 768 in fp32, one sequence 6.69, 6.25, 6.86, two 7.45, 7.45, 7.51;
  // LlamaGen-XL with 32 sequences 7.19, 6.97, 7.99, but with 16 5.18, 5.75, 7.50
  // (fp32 5.69, 6.55, 6.98). The kernels that stop after the attention or the
  // grouping are best with 3: attention over one dense sequence 214, 208, 209.
  static constexpr __host__ __device__ int min_chunk(bool step) {
    return SHORT ? kAlignedGrains : (step ? 4 : 3) * Tile::kTT / kGR;
  }
  __host__ __device__ static constexpr int grains(int rows) {
    return (int)(((unsigned)rows + kGR - 1) / kGR);
  }
  __host__ __device__ static constexpr int cost(int g) { return g + 1 > kMinCost ? g + 1 : kMinCost; }
};

// Layers of at least kHeadSlots slots for every CTA, no head above kHeadGrains
// grains, are not cut beforehand (StepCut): taken head by head a launch costs
// some 1.5 us more (lengths and claims are fetched on the way, the counters
// advance at the end) and its CTAs end within 2 us of each other instead of
// 5. Per layer step, cut -> head by head: Janus-Pro-7B at rho = 1/8 with 96
// sequences (121 slots) 36.8 -> 37.1 us, with 128 (162) 45.6 -> 44.9, with 160
// (202) 59.5 -> 58.5, with 256 (323) 94.5 -> 89.0; LlamaGen-XL with 250 (131)
// 24.1 -> 24.4, with 280 (166) 25.5 -> 24.6, with 400 35.5 -> 33.8; the same in
// fp32 with 140 (83) 21.0 -> 21.7, with 200 (118) 29.6 -> 29.2, with 280 40.7
// -> 40.2, with 400 58.2 -> 56.9.
#ifndef HKV_STEP_HEAD_SLOTS
#define HKV_STEP_HEAD_SLOTS 160
#endif
constexpr int kHeadSlots = HKV_STEP_HEAD_SLOTS, kHeadGrains = 16;
// Rows of 512 bytes (grains of 8) are better cut as long as the table holds
// every range's heads: heads of up to 112 rows, 3600 of them (177 slots) 44.0
// us cut and 46.6 head by head, 6000 73.8 and 76.2, 9000 (444) 111.1 and 113.4.
constexpr int kHeadSlots512 = 3 * (kStepTable - 2);  // of ranges, at 3 slots a head at least

// Rows of 512 bytes: a small layer gets one CTA an SM, which shared memory
// then keeps to itself, else two. Two halve a range; that loses where a
// head falls into more than three ranges (fewer heads than a third of the
// CTAs) or a range is short anyway (fewer than kLoneSlots slots an SM). Per
// layer step, one -> two: Lumina-mGPT 768 with 1 sequence 6.24 -> 6.78 us, 3
// (96 heads) 9.08 -> 9.24, 4 11.0 -> 10.3, 12 28.7 -> 23.4; Lumina-mGPT 1024
// with 1 8.85 -> 9.98, 3 13.9 -> 14.0, 4 17.4 -> 16.7, 10 41.7 -> 35.2;
// Janus-Pro-7B with 4 (19 slots) 6.08 -> 6.31, 8 (37) 8.3 -> 8.3, 10 (46)
// 10.7 -> 9.3, 40 30.3 -> 28.2. One CTA an SM beside one of the next launch's
// is slower than either (Lumina-mGPT 768 with 3: 9.85).
constexpr int kLoneSlots = 40;
constexpr size_t kLoneSmem = 104 * 1024;  // dynamic; twice that is more than an SM has

// A boundary between ranges that falls within 1/kSnapDiv of a range of a
// head's first or last row moves there.
#ifndef HKV_STEP_SNAP_DIV
#define HKV_STEP_SNAP_DIV 4
#endif

// ONE: a head's status and label share a byte, without which rows of 512 bytes
// had room for one CTA an SM only; elsewhere a byte each is 0.8 % faster on
// small layers (Janus-Pro-7B, 2 sequences: 2489 and 2512 us a period).
template <int N, bool ONE>
struct StepTable {  // entry h - wl: head h
  long long off[N];  // arena offset
  int vlen[N];       // rows, the new token included
  int ntok[N];
  unsigned char bad[N];  // status of the head's counters (ONE: doubled, 1 for a compressed head)
  unsigned char label[ONE ? 1 : N];
  __device__ __forceinline__ void set_label(int j, int lab) {
    if (ONE) bad[j] = lab != HKV_DENSE;
    else label[j] = (unsigned char)lab;
  }
  __device__ __forceinline__ void set(int j, int status, int lab) {
    bad[j] = (unsigned char)(ONE ? status << 1 | (lab != HKV_DENSE) : status);
    if (!ONE) label[j] = (unsigned char)lab;
  }
  __device__ __forceinline__ int status(int j) const { return ONE ? bad[j] >> 1 : bad[j]; }
  __device__ __forceinline__ bool dense(int j) const {
    return ONE ? !(bad[j] & 1) : label[j] == HKV_DENSE;
  }
};

// kWhole: the piece is its whole head; kTailPiece: the head began in an
// earlier range
constexpr int kFirst = 1, kLast = 2, kDone = 4, kWhole = 8, kTailPiece = 16;

struct TileMeta {  // producer -> consumers, one per stage
  int h, n, flags;
  int recent0;  // identification: rows from here on are among the head's newest w_loc - 1
};

constexpr int kNewRow = 32;  // flag: the tile's last row is the step's token

struct SegMeta {  // consumers -> epilogue; h < 0: no more segments
  int h, flags;
};

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t atom_add_acq_rel(uint32_t *p, uint32_t v) {
  uint32_t old;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ unsigned long long atom_exch_acq_rel(unsigned long long *p,
                                                               unsigned long long v) {
  unsigned long long old;
  asm volatile("atom.acq_rel.gpu.global.exch.b64 %0, [%1], %2;"
               : "=l"(old)
               : "l"(p), "l"(v)
               : "memory");
  return old;
}
__device__ __forceinline__ void st_release(uint32_t *p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// A float and the epoch of the launch that wrote it, as one 64-bit word:
// single-copy atomic, so a reader that sees the epoch sees the value.
__device__ __forceinline__ void st_pair(unsigned long long *p, float v, uint32_t ep) {
  const unsigned long long w = ((unsigned long long)ep << 32) | __float_as_uint(v);
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ bool ld_pair(const unsigned long long *p, uint32_t ep, float &v) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  v = __uint_as_float((uint32_t)w);
  return (uint32_t)(w >> 32) == ep;
}

// One bf16 m16n8k16 product added to c in fp32: exact products; the order and
// rounding of their sums are the hardware's.
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint4 &a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// the largest x of the warp, in every lane
__device__ __forceinline__ float warp_max(float x) {
  float y;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(x));
  return y;
}

// Combines a split head's own piece (m1, l1, r1, A1) with its other pieces,
// already combined (m2, l2, r2, A2), and stores the output row: the same
// instructions wherever it runs, so the result does not depend on which
// warp does it. Returns the head's sum and, for identification, its mass of
// newest rows.
template <int CPL, bool IDENT>
__device__ __forceinline__ void combine_store(float m1, float l1, float r1, const float *A1,
                                              float m2, float l2, float r2, const float *A2,
                                              float *out, float &Lt, float &Rt) {
  const float mx = fmaxf(m1, m2);
  const float w1 = m1 == -INFINITY ? 0.f : exp2f(m1 - mx);
  const float w2 = m2 == -INFINITY ? 0.f : exp2f(m2 - mx);
  Lt = l1 * w1 + l2 * w2;
  if (IDENT) Rt = r1 * w1 + r2 * w2;
  float A[CPL];
#pragma unroll
  for (int c = 0; c < CPL; ++c) A[c] = fmaf(A1[c], w1, A2[c] * w2) / Lt;
  Vec<CPL>::st(out, A);
}

// threads: a producer warp, the consumer warps, the epilogue warp and the
// merge warp
template <int D, typename T>
__host__ __device__ constexpr int step_threads() {
  return StepShape<D, T>::kThreads + 32;
}

// What a launch does: a decode step, the same with the head types decided in
// the pass (Sec. 4, Step 2), or attention alone (no append, no counters).
enum StepMode { kModeStep = 0, kModeIdentify = 1, kModeAttend = 2 };

// How a launch cuts the layer: into equal ranges of slots, one per CTA; the
// same with the shape for short heads; or head by head, taken as CTAs get
// free (many short heads).
enum StepCut { kCutRanges = 0, kCutShort = 1, kCutHeads = 2 };

template <int D, typename T, int MODE, int CUT>
__global__ void __launch_bounds__(step_threads<D, T>(), HKV_STEP_RESIDENT_PER_SM)
    step_kernel(const AttnArgs p) {
  using S = StepShape<D, T, CUT == kCutShort>;
  constexpr bool DYN = CUT == kCutHeads;
  static_assert(!DYN || MODE == kModeStep, "heads are taken one by one in plain steps only");
  constexpr bool FUSED = MODE != kModeAttend, IDENT = MODE == kModeIdentify;
  constexpr int kCW = S::kCW, kThr = step_threads<D, T>(), NW = kThr / 32;
  constexpr int LPR = S::kLPR, EPL = S::kEPL, RPW = S::kRPW, TT = S::kTT;
  constexpr int RB = S::kRB, NS = S::kNS, GR = S::kGR;
  constexpr int NST = S::kNST;
  constexpr int CPL = D / 32;     // output channels per epilogue lane
  constexpr int NV = IDENT ? 3 : 2;  // scalars of a partial result: maximum, sum, newest rows' sum
  constexpr int PS = step_piece_words(D);
  static_assert(NST <= 32, "a lane of the epilogue per state");
  static_assert(kStepTable <= kThr, "the table holds a range's heads");
  static_assert(TT % GR == 0, "tiles of whole grains");
  using V = Vec<CPL>;

  extern __shared__ __align__(128) unsigned char stages[];
  __shared__ uint64_t full[NS], empty[NS];
  __shared__ uint64_t epi_full[2], epi_free[2];  // two hand-over buffers
  __shared__ __align__(16) float red_acc[2][NST][D];
  __shared__ __align__(16) float red_m[2][NST], red_l[2][NST], red_r[IDENT ? 2 : 1][IDENT ? NST : 1];
  __shared__ TileMeta meta[NS];
  __shared__ SegMeta seg[2];
  __shared__ StepTable<DYN ? 1 : kThr, RB == 512> tab;
  __shared__ int2 s_w[NW];  // each warp's slots; its longest head, or a status
  // the range's ends: {first slot, first head, that head's first slot, its
  // rows} and {end slot, last head, that head's first slot, whether the range
  // ends inside its rows}
  __shared__ int4 s_lo, s_hi;
  __shared__ int s_bad;
  __shared__ int s_mg_h, s_mg_k0, s_mg_j, s_mg_np;  // the split head this CTA combines
  __shared__ uint32_t s_ep;                         // the launch's epoch
  // hand-overs between the epilogue and the merge warp: the epoch and the
  // merge head (ep_bar), the other pieces combined (oth_bar), and this CTA's
  // own piece or the news that the epilogue combined it already (own_bar)
  __shared__ uint64_t ep_bar, oth_bar, own_bar;
  __shared__ __align__(16) float own_acc[D], oth_acc[D];
  __shared__ float own_s[NV], oth_s[NV];
  __shared__ int s_own_state;  // 1: combined by the epilogue, 2: own piece handed over
  __shared__ volatile int s_abort;
  __shared__ volatile int s_streamed;  // (identification) the epilogue is done

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nheads = p.nheads;
  const int G = gridDim.x;
  const int bx = blockIdx.x;

  if (tid == 0) {
    STEP_TRACE(0);
#ifdef HKV_ATTN_TRACE
    if (g_step_trace) {
      unsigned smid;
      asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
      STEP_TRACE_AT(16) = smid;
    }
#endif
  }
  if (!p.prefetch) pdl_wait();

  // A layer of many short heads (DYN) is not cut beforehand: CTA k starts with
  // the heads k and k + G and takes further ones from a counter, so there is
  // no prologue over the layer's lengths, and CTAs that start late, as the
  // previous launch's end, take fewer. Its merge warp checks a share of the
  // heads of its own, appends their tokens and advances their counters.
  //
  // ---- prologue: the layer's lengths, one round of loads -------------------
  // Warp w takes `rows` rows of 32 consecutive heads and sums each row's
  // slots; the warps' sums give every CTA the same ranges, and only the warps
  // whose heads meet the range's ends look at their rows again. (One thread
  // per run of consecutive heads took 2.5 us to place a range of LlamaGen-XL's
  // 2560 heads, whose rows this takes one or two of.)
  // The same round fills a table of kThr heads: the whole layer, if it has no
  // more (every CTA then checks every head, and a bad one stops all of them
  // here), else those around the range's expected place (heads of equal
  // length); a range outside it reads its heads once it is known. A CTA that
  // finds a bad head in its range then streams nothing and flags the step on
  // the layer's barrier word, and no CTA appends or advances a counter.
  constexpr int kNew = FUSED ? 1 : 0;   // the step's token is one more row
  int wl = 0;  // the table's first head
  // the range: slots [a, b), heads h0 .. h0 + n - 1, the first starting at
  // slot s0 with v0 rows, the last at s1
  int a = 0, b = 0, h0 = bx, n = 1, s0 = 0, s1 = 0, v0 = 0, chunk = 1, tol = 0, own_bad = 0;
  bool has_s = false, has_e = false, in_regs = false, active = true;
  auto init_barriers = [&]() {  // one thread
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kCW);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&epi_full[s], kCW);
      mbar_init(&epi_free[s], 1);
    }
    mbar_init(&ep_bar, 32);
    mbar_init(&oth_bar, 32);
    mbar_init(&own_bar, 32);
    fence_barrier_init();
    s_abort = 0;
    s_streamed = 0;
    s_bad = 0;
    s_mg_h = -1;
  };
  // the status of a head's counters
  auto verify = [&](int l, long long o, int cp, int lab, int nb) {
    if (FUSED) {
      if (l < 0 || o < 0 || o + cp > p.arena_tokens) return (int)HKV_ERR_BOUNDS;
      if (IDENT && lab != HKV_DENSE) return (int)HKV_ERR_STATE;  // the rows' order is needed
      if (l + 1 > cp) return (int)HKV_ERR_CAPACITY;
      if (lab != HKV_DENSE && nb >= p.period) return (int)HKV_ERR_STATE;  // the update is due first
      return 0;
    }
    return l < 0 || o < 0 || o + l > p.arena_tokens ? (int)HKV_ERR_BOUNDS : 0;
  };
  // DYN: the producer's next two heads, their lengths and offsets on their
  // way, and the one after them, claimed meanwhile
  int na = bx, nb = bx + G, nc = 0, na_l = -1, nb_l = -1;
  long long na_o = 0, nb_o = 0;
  auto fetch = [&](int h, int &l, long long &o) {
    l = p.len[h];
    o = p.off[h];
  };
  auto claim = [&]() { return 2 * G + (int)atomicAdd(p.bar + 3, 1u); };
  if constexpr (DYN) {
    if (tid == 0) {
      if (na < nheads) fetch(na, na_l, na_o);
      if (nb < nheads) {
        fetch(nb, nb_l, nb_o);
        nc = claim();
      }
    }
    if (tid == kThr - 32) init_barriers();
    __syncthreads();
  } else {
    const int rows = (nheads + kThr - 1) / kThr;
    const int row0 = warp * rows;  // this warp's first row
    in_regs = rows <= 1;
    constexpr int kMost = 1 << 26;        // grains of a head, slots of a warp: beyond any arena
    constexpr int kIsBad = 0x70000000;    // a status in place of the longest head
    constexpr int kPre = 8;               // rows loaded at once
    if (!in_regs) {
      wl = (int)((float)bx * ((float)nheads / (float)G)) - kThr / 2;
      wl = wl < nheads - kThr ? wl : nheads - kThr;
      wl = wl > 0 ? wl : 0;
    }
    int key = 0;
    unsigned c0 = 0;  // in_regs: the slots of this thread's head
    int lv[kPre];
    {
      // every load issued before any use
      const int h = wl + tid;
      int l = 0, cp = 0, lab = 0, nb = 0, nt = 0;
      long long o = 0;
      if (h < nheads) {
        l = p.len[h];
        o = p.off[h];
        if (FUSED) {
          cp = p.cap[h];
          lab = p.label[p.layer_base + h];
          nb = p.nbuf[p.layer_base + h];
          nt = p.ntok[p.layer_base + h];
        }
      }
      if (!in_regs) {
#pragma unroll
        for (int i = 0; i < kPre; ++i) {
          const int r = (row0 + i) * 32 + lane;
          lv[i] = i < rows && r < nheads ? p.len[r] : -1;
        }
      }
      // the barriers, while the loads are on their way (the merge warp's lane)
      if (tid == kThr - 32) init_barriers();
      if (h < nheads) {
        const int e = verify(l, o, cp, lab, nb);
        tab.vlen[tid] = l + kNew;
        tab.off[tid] = o;
        tab.set(tid, e, lab);
        if (FUSED) tab.ntok[tid] = nt;
        if (in_regs) {
          const int g = S::grains(l + kNew);
          const int st = e ? e : g > kMost ? (int)HKV_ERR_BOUNDS : 0;
          key = st ? kIsBad + st : g;
          c0 = st ? 0u : (unsigned)S::cost(g);
        }
      }
    }
    // the slots of a head of length l of row i (a bad one: 0, and the status)
    auto slots = [&](int h, int l) {
      if (h >= nheads) return 0u;
      const int g = S::grains(l + kNew);
      const bool ok = FUSED ? l >= 0 && g <= kMost : g <= kMost && !verify(l, p.off[h], 0, 0, 0);
      if (!ok) key = kIsBad + HKV_ERR_BOUNDS;
      return ok ? (unsigned)S::cost(g) : 0u;
    };
    unsigned rowsum = 0;  // lane i: the slots of row i (up to 32 rows)
    long long wsum = 0;
    if (in_regs) {
      rowsum = __reduce_add_sync(0xFFFFFFFFu, c0);
      wsum = rowsum;
    } else {
#pragma unroll
      for (int i = 0; i < kPre; ++i) {
        if (i < rows) {
          const unsigned r = __reduce_add_sync(0xFFFFFFFFu, slots((row0 + i) * 32 + lane, lv[i]));
          if (lane == i) rowsum = r;
          wsum += r;
        }
      }
#pragma unroll 1
      for (int i = kPre; i < rows; ++i) {
        const int h = (row0 + i) * 32 + lane;
        const unsigned r = __reduce_add_sync(0xFFFFFFFFu, slots(h, h < nheads ? p.len[h] : 0));
        if (lane == i) rowsum = r;
        wsum += r;
      }
    }
    if (wsum > kMost) key = kIsBad + HKV_ERR_BOUNDS;
    key = __reduce_max_sync(0xFFFFFFFFu, key);
    if (lane == 0) s_w[warp] = make_int2((int)wsum, key);
    __syncthreads();
    if (tid == 0) STEP_TRACE(10);
    const int2 sw = lane < NW ? s_w[lane] : make_int2(0, 0);
    const int total = (int)__reduce_add_sync(0xFFFFFFFFu, (unsigned)sw.x);
    const int longest = __reduce_max_sync(0xFFFFFFFFu, sw.y);
    if (longest >= kIsBad) {  // every CTA sees it: none reads further or arrives
      pdl_wait();
      if (bx == 0 && tid == 0) {
        set_err(p.err, (uint32_t)(longest - kIsBad));
        p.ctl->valid = 0;
      }
      return;
    }
    // a CTA per head where every head is short (see kAlignedGrains), else G
    // ranges of `chunk` slots
    const bool aligned = in_regs && nheads <= G && longest <= kAlignedGrains;
    // total / G rounded up, from the grid's reciprocal (rounded up, so the
    // quotient is exact or one too large)
    chunk = G == 1 ? total : (int)__umulhi((unsigned)(total + G - 1), p.grid_recip);
    if ((long long)chunk * G > total + G - 1) --chunk;
    if (chunk < S::min_chunk(MODE == kModeStep)) chunk = S::min_chunk(MODE == kModeStep);
    tol = chunk / HKV_STEP_SNAP_DIV;
    const long long a64 = (long long)bx * chunk, b64 = a64 + chunk;
    const int a_raw = a64 < total ? (int)a64 : total, b_raw = b64 < total ? (int)b64 : total;
    active = aligned ? bx < nheads : a_raw < total;
    // boundary x inside the slots [s, s + cost) of a head of g grains
    auto snap = [&](int x, int s, int g) {
      if (x - s <= tol) return s;
      return x >= s + g - tol ? s + S::cost(g) : x;
    };
    // places head h (slots from s, v rows): whether it is in the range, and
    // the range's ends when they fall into it
    auto place = [&](int h, int s, int v) {
      const int g = S::grains(v), e = s + S::cost(g);
      if (a_raw >= e || b_raw <= s) return false;
      bool in = true;
      if (a_raw >= s) {
        const int x = snap(a_raw, s, g);
        const bool next = x == e;
        s_lo = make_int4(x, next ? h + 1 : h, next ? e : s, v);
        in = !next;
      }
      if (b_raw <= e) {
        const int x = b_raw == e ? e : snap(b_raw, s, g);
        s_hi = make_int4(x, x == s ? h - 1 : h, s, x > s && x < e);
        in = in && x != s;
      }
      return in;
    };
    if (!aligned && active) {
      const int before = (int)__reduce_add_sync(0xFFFFFFFFu, lane < warp ? (unsigned)sw.x : 0u);
      if (before < b_raw && before + (int)wsum > a_raw) {  // warp-uniform
        // one row: its heads in order
        auto place_row = [&](int i, int at) {
          const int h = (row0 + i) * 32 + lane;
          const bool in = h < nheads;
          const int j = h - wl;
          const bool here = j >= 0 && j < kThr;
          const int v = !in ? 0 : here ? tab.vlen[j] : p.len[h] + kNew;
          const int c = in ? S::cost(S::grains(v)) : 0;
          const int incl = warp_incl_scan(c);
          if (in && place(h, at + incl - c, v) && FUSED && !in_regs && here && tab.status(j))
            atomicMax(&s_bad, tab.status(j));
          return __shfl_sync(0xFFFFFFFFu, incl, 31);
        };
        if (in_regs) {
          place_row(0, before);
        } else if (rows <= 32) {
          const int incl = warp_incl_scan((int)rowsum);
          const int rs = before + incl - (int)rowsum;
          unsigned hit = __ballot_sync(0xFFFFFFFFu, lane < rows && rs < b_raw && before + incl > a_raw);
          while (hit) {
            const int i = __ffs(hit) - 1;
            hit &= hit - 1;
            place_row(i, __shfl_sync(0xFFFFFFFFu, rs, i));
          }
        } else {
          int at = before;
#pragma unroll 1
          for (int i = 0; i < rows && at < b_raw; ++i) at += place_row(i, at);
        }
      }
    }
    __syncthreads();
    if (!aligned && active) {
      const int4 lo = s_lo, hi = s_hi;
      a = lo.x;
      b = hi.x;
      h0 = lo.y;
      n = hi.y - lo.y + 1;
      s0 = lo.z;
      v0 = lo.w;
      s1 = hi.z;
      active = a < b && n > 0;
      has_s = active && s0 < a;
      has_e = active && hi.w;
    }
    if (!in_regs) {
      if (FUSED && active && n > kStepTable) {  // excluded by the host; the step is not taken
        own_bad = HKV_ERR_CAPACITY;
        active = false;
      }
      if (active && (h0 < wl || h0 + n > wl + kThr)) {  // CTA-uniform
        wl = h0;
        const int h = h0 + tid, i = p.layer_base + h;
        if (tid < n) {
          const int l = p.len[h];
          const long long o = p.off[h];
          tab.vlen[tid] = l + kNew;
          tab.off[tid] = o;
          if (FUSED) {
            const int cp = p.cap[h], lab = p.label[i], nb = p.nbuf[i], nt = p.ntok[i];
            const int e = verify(l, o, cp, lab, nb);
            if (e) atomicMax(&s_bad, e);
            tab.ntok[tid] = nt;
            tab.set_label(tid, lab);
          }
        }
        __syncthreads();
      }
      if (FUSED && s_bad) {  // a bad head in this range: stream nothing
        own_bad = own_bad > s_bad ? own_bad : s_bad;
        active = false;
      }
    }
  }
  const int h1 = h0 + n - 1;
  if (!active) has_s = has_e = false;
  // From here on nothing reads the layer's counters in global memory: the
  // merge warp arrives on the layer's barrier word below. (Attention alone
  // over more heads than the table holds looks them up; nothing writes them.)
  if (tid == 0) STEP_TRACE(1);

  // ---- producer state (warp 0, lane 0) ------------------------------------
  // Pieces in streaming order: the start of the head that continues past the
  // range, the piece of the head that began before it, the heads in between.
  const bool producer = tid == 0;
  const bool in_tab = FUSED || n <= kThr;
  auto vlen_of = [&](int h) { return in_tab ? tab.vlen[h - wl] : p.len[h] + kNew; };
  auto off_of = [&](int h) { return in_tab ? tab.off[h - wl] : (long long)p.off[h]; };
  int ph = 0, ch = h0 + (has_s ? 1 : 0);    // next piece; next whole head
  const int ch_end = has_e ? h1 - 1 : h1;   // last whole head
  int ph_h = 0, ph_r = 0, ph_end = 0, ph_v = 0, ph_flags = 0;  // the piece: head, rows, length
  long long ph_off = 0;
  bool have = false, at_start = false;
  auto open_piece = [&](int h, int from, long long to, int flags) {
    ph_h = h;
    ph_v = vlen_of(h);
    ph_off = off_of(h);
    ph_r = from;
    ph_end = to < ph_v ? (int)to : ph_v;
    ph_flags = flags;
    at_start = true;
    have = true;
  };
  // This CTA reads no further lengths: the last of the grid to say so resets
  // the head counter and lets the merge warps advance the lengths (not before
  // this CTA's has noted the generation).
  auto no_more = [&]() {
    mbar_wait(&ep_bar, 0u);
    if (atom_add_acq_rel(p.bar + 4, 1u) == (uint32_t)G - 1) {
      p.bar[3] = 0;
      p.bar[4] = 0;
      st_release(p.bar + 5, ld_acquire(p.bar + 5) + 1u);
    }
  };
  auto next_piece = [&]() {
    have = false;
    if constexpr (DYN) {
      while (na < nheads && !have) {
        const int h = na, l = na_l;
        const long long o = na_o;
        na = nb;
        na_l = nb_l;
        na_o = nb_o;
        if (nb < nheads) {
          nb = nc;
          if (nb < nheads) {
            fetch(nb, nb_l, nb_o);
            nc = claim();
          }
        }
        // (a bad head is not read; the CTA that checks it stops the step)
        if (l >= 0 && o >= 0 && o + l <= p.arena_tokens) {
          ph_h = h;
          ph_v = ph_end = l + 1;
          ph_off = o;
          ph_r = 0;
          ph_flags = kWhole;
          at_start = have = true;
        }
        if (na >= nheads) no_more();  // (after its last length, l, has arrived)
      }
      return;
    }
    if (ph == 0) {
      ph = 1;
      if (has_e && !(has_s && n == 1)) {
        open_piece(h1, 0, (long long)(b - s1) * GR, 0);
        return;
      }
    }
    if (ph == 1) {
      ph = 2;
      if (has_s) {
        open_piece(h0, (a - s0) * GR, (long long)(b - s0) * GR, kTailPiece);
        return;
      }
    }
    if (active && ch <= ch_end) {
      open_piece(ch, 0, 0x7FFFFFFF, kWhole);
      ++ch;
    }
  };
  int st_i = 0;                // stage of the next tile
  uint32_t st_ph = 1;          // its empty barrier's parity (1: not used yet)
  // the arena rows are read once per step: evict them from L2 first (measured:
  // 0.4-0.55 us per step slower without the hint)
  const uint64_t stream_pol = producer ? l2_evict_first_policy() : 0;
  auto issue_old = [&](int stage, bool open_next) {  // describe, expect and copy the arena rows
    const int left = ph_end - ph_r;
    const int rows = left < TT ? left : TT;
    const int real = ph_v - kNew;  // rows in the arena
    const int n_old = (ph_r + rows < real ? ph_r + rows : real) - ph_r;
    unsigned char *dk = stages + stage * S::kStageBytes;
    if (n_old > 0) {
      const uint32_t bytes = (uint32_t)n_old * RB;
      const long long row = ph_off + ph_r;
      mbar_expect_tx(&full[stage], 2 * bytes);
      bulk_g2s_hint(dk, static_cast<const unsigned char *>(p.K) + row * RB, bytes, &full[stage],
                    stream_pol);
      bulk_g2s_hint(dk + TT * RB, static_cast<const unsigned char *>(p.V) + row * RB, bytes,
                    &full[stage], stream_pol);
    }
    const bool last = left <= TT;
    TileMeta mt;
    mt.h = ph_h;
    mt.n = rows;
    mt.flags = ph_flags | (at_start ? kFirst : 0) | (last ? kLast : 0) |
               (FUSED && ph_r + rows == ph_v ? kNewRow : 0);
    const int rc = ph_v - (p.w_loc - 1) - ph_r;
    mt.recent0 = IDENT ? (rc < 0 ? 0 : rc < TT ? rc : TT) : 0;
    meta[stage] = mt;
    at_start = false;
    ph_r += TT;
    // (DYN: the tile before the wait for the previous kernel does not wait for
    // the next head's length)
    if (last && open_next) next_piece();
    else if (last) have = false;
  };
  auto issue_extra = [&](int stage) {  // the step's inputs, then arrive
    unsigned char *dk = stages + stage * S::kStageBytes;
    unsigned char *dv = dk + TT * RB;
    const int h = meta[stage].h, flags = meta[stage].flags;
    const size_t src = (size_t)h * RB;
    mbar_arrive_expect_tx(&full[stage], (flags & kNewRow ? 2 * RB : 0) + (flags & kFirst ? RB : 0));
    if (flags & kFirst)
      bulk_g2s(dv + TT * RB, static_cast<const unsigned char *>(p.q) + src, RB, &full[stage]);
    if (flags & kNewRow) {
      const int at = (meta[stage].n - 1) * RB;
      bulk_g2s(dk + at, static_cast<const unsigned char *>(p.k_new) + src, RB, &full[stage]);
      bulk_g2s(dv + at, static_cast<const unsigned char *>(p.v_new) + src, RB, &full[stage]);
    }
  };
  int n_pre = 0;
  if (producer) {
    if (DYN && na >= nheads) no_more();
    next_piece();
    const int lim = p.prefetch ? S::kPre : NS;
#pragma unroll 1
    while (n_pre < lim && have) {
      ++n_pre;
      issue_old(n_pre - 1, !DYN || n_pre < lim);
    }
  }
  if (tid == 0) STEP_TRACE(7);

  // ---- merge warp: the launch's epoch and the split head this CTA combines --
  // The split head: the first of the range when this CTA is that head's
  // first middle CTA (its whole range inside the head) or, for a head in two
  // pieces and in all but the plain step, holds its last row: CTAs then wait
  // for lower-numbered ones only, which start before them, so that launches
  // that share the GPU never hold each other's places. The epoch,
  // from the generation of the barrier word, is unique per (layer, launch of
  // that layer), or among the attentions alone, which have words and slots of
  // their own (p.n_layers is 1 there, whatever the layer); the
  // epilogue waits for both only when it meets a split head.
  //
  // Then this CTA arrives on the layer's barrier words {arrivals,
  // generation, worst status}: it is done reading counters. The last of the
  // grid to arrive resets the count and publishes the next generation, which
  // the others watch. A CTA with a bad head arrives after the wait for the
  // previous kernel, raises the worst status and adds 1 << 16 more; the last
  // arriver then marks the generation (the step is not taken) and reports
  // the worst status, the same whichever CTAs found bad heads first. The
  // words belong to this layer, whose previous launch is complete, so the
  // others arrive ahead of that wait.
  constexpr uint32_t kBadStep = 0x80000000u;  // in the generation: step not taken
  uint32_t gen0 = 0, gen1 = 0;
  int bar_done = 0;
  int hinted = 0;  // identification: the last CTA to arrive found the hint (see the merge warp)
  auto arrive = [&]() {  // lane 0 of the merge warp
    const uint32_t inc = own_bad ? 0x10001u : 1u;
    if (own_bad) {
      atomicMax(p.bar + 2, (uint32_t)own_bad);
      __threadfence();  // the status before the arrival
    }
    const uint32_t old = atomicAdd(p.bar, inc);
    if ((old & 0xFFFFu) == (uint32_t)G - 1) {
      const bool bad_step = ((old + inc) >> 16) != 0;
      if (bad_step) {
        __threadfence();  // the bad CTAs' statuses after their arrivals
        set_err(p.err, atomicExch(p.bar + 2, 0u));
      }
      p.bar[0] = 0;
      gen1 = (((gen0 & ~kBadStep) + 1u) & ~kBadStep) | (bad_step ? kBadStep : 0u);
      st_release(p.bar + 1, gen1);
      bar_done = 1;
    }
  };
  // DYN: this CTA's share of the heads for checks, appends and counters
  const int share = DYN ? (nheads + G - 1) / G : 0;
  const int sh0 = DYN && bx * share < nheads ? bx * share : nheads;
  const int sh1 = sh0 + share < nheads ? sh0 + share : nheads;
  uint32_t taken0 = 0;  // generation of the second barrier: every head is taken
  int k_len = 0, k_nb = -1, k_nt = 0;  // the counters of the share's first 32 heads
  if (warp == kCW + 2) {
    if constexpr (DYN) {
      int e = 0;
      for (int h = sh0 + lane; h < sh1; h += 32) {
        const int i = p.layer_base + h;
        const int l = p.len[h], lab = p.label[i], nbv = p.nbuf[i], ntv = p.ntok[i];
        e = max(e, verify(l, p.off[h], p.cap[h], lab, nbv));
        if (h < sh0 + 32) {  // kept for the advance
          k_len = l;
          k_nb = lab == HKV_DENSE ? -1 : nbv;
          k_nt = ntv;
        }
      }
      own_bad = __reduce_max_sync(0xFFFFFFFFu, e);
      if (lane == 0) taken0 = ld_acquire(p.bar + 5);
    }
    if (lane == 0) {
      if (has_s) {
        const int er = s0 + S::grains(v0);
        int k0 = (int)((unsigned)s0 / (unsigned)chunk);
        if ((long long)(k0 + 1) * chunk - s0 <= tol) ++k0;  // that boundary moved to the head's start
        int k1 = (int)((unsigned)(er - 1) / (unsigned)chunk);
        const long long x1 = (long long)k1 * chunk;
        if (x1 > s0 && x1 >= er - tol) --k1;  // that one to its end
        const int np = k1 - k0 + 1;
        if ((MODE == kModeStep && np >= 3 ? k0 + 1 : k1) == bx) {
          s_mg_k0 = k0;
          s_mg_np = np;
          s_mg_j = bx - k0;
          s_mg_h = h0;
        }
      }
      gen0 = ld_acquire(p.bar + 1);
      s_ep = ((gen0 & ~kBadStep) + 1u) * (uint32_t)p.n_layers + (uint32_t)p.layer;
      if (!own_bad) arrive();
    }
    __syncwarp();
    mbar_arrive(&ep_bar);  // all 32 lanes: the epilogue may read s_ep, s_mg_*
    if (IDENT && lane == 0 && bar_done) {
      __threadfence();  // the generation before the hint
      hinted = ld_acquire(p.bar + 6) == s_ep;
    }
  }

  if (p.prefetch) pdl_wait();  // the step's inputs are visible from here on
  if (tid == 0) STEP_TRACE(2);
  pdl_launch_dependents();

  if (warp == 0) {
    // ---- producer ----------------------------------------------------------
    if (producer) {
      long long w_empty = 0;  // cycles waiting for free stages (tracer)
#pragma unroll 1
      for (int j = 0; j < n_pre; ++j) issue_extra(j);
      if (DYN && !have) next_piece();
      st_i = n_pre < NS ? n_pre : 0;
      st_ph = n_pre < NS ? 1u : 0u;
      int armed = n_pre;  // tiles armed in all
      auto stage_free = [&]() {  // (the parity of a stage not used yet reads as complete)
        if (!s_abort && mbar_wait(&empty[st_i], st_ph)) return true;
        s_abort = 1;
        set_err(p.err, HKV_ERR_TIMEOUT);
        return false;
      };
      while (have) {
        const long long c0 = STEP_CLK();
        if (!stage_free()) break;
        w_empty += STEP_CLK() - c0;
        issue_old(st_i, true);
        issue_extra(st_i);
        ++armed;
        if (NS == 1 || ++st_i == NS) {
          st_i = 0;
          st_ph ^= 1u;
        }
      }
      if (stage_free()) {  // no more tiles: a closing record for the consumers
        meta[st_i].flags = kDone;
        mbar_arrive(&full[st_i]);
      }
      STEP_TRACE_SET(20, w_empty);
      if (!FUSED && bx == 0) p.ctl->valid = 1;  // the launch passed its checks
      if (s_abort) {
        // No bulk copy may land in shared memory after the CTA exits: wait
        // (bounded) for every armed stage that may still be in flight. A
        // stage reused after an empty-barrier wait is complete already.
        const int first = armed - NS > 0 ? armed - NS : 0;
        for (int t = first; t < armed; ++t) mbar_wait(&full[t % NS], (uint32_t)(t / NS) & 1u);
      }
    }
  } else if (warp <= kCW) {
    // ---- consumers ---------------------------------------------------------
    const int cw = warp - 1;
    const int grp = lane / LPR, col = lane % LPR;
    using M = LaneMath<T>;
    static_assert(M::kEPL == EPL, "lane mapping");
    constexpr bool MMA = sizeof(T) == 2;
    float2 acc[EPL / 2];
    float m = -INFINITY, l = 0.f, lr = 0.f;  // lr: identification's newest-row mass
    int nseg = 0;
#pragma unroll
    for (int e = 0; e < EPL / 2; ++e) acc[e] = make_float2(0.f, 0.f);
    int n_tiles = 0;
    long long w_full = 0, w_hand = 0;  // cycles waiting for tiles, for the epilogue (tracer)
    // hands one segment's state (or the closing record) to the epilogue
    auto hand_over = [&](int h, int flags) {
      const int bb = nseg & 1;
      const long long c0 = STEP_CLK();
      if (nseg >= 2 && !s_abort &&
          !mbar_wait(&epi_free[bb], (uint32_t)((nseg >> 1) - 1) & 1u)) {
        s_abort = 1;
        set_err(p.err, HKV_ERR_TIMEOUT);
      }
      w_hand += STEP_CLK() - c0;
      if (h >= 0 && MMA) {
        // The row groups share the maximum; their sums are halved between
        // the lanes of two groups at a time, so that each lane ends with its
        // own channels. l and lr are split over the quads.
        float *dst = &red_acc[bb][cw][col * EPL];
        float2 x0 = acc[0], x1 = acc[1];
        {
          const bool hi = lane & 16;
          const float2 s0v = hi ? acc[0] : acc[2], s1v = hi ? acc[1] : acc[3];
          x0 = hi ? acc[2] : acc[0];
          x1 = hi ? acc[3] : acc[1];
          x0.x += __shfl_xor_sync(0xFFFFFFFFu, s0v.x, 16);
          x0.y += __shfl_xor_sync(0xFFFFFFFFu, s0v.y, 16);
          x1.x += __shfl_xor_sync(0xFFFFFFFFu, s1v.x, 16);
          x1.y += __shfl_xor_sync(0xFFFFFFFFu, s1v.y, 16);
        }
        if (RPW == 2) {
          *reinterpret_cast<float4 *>(dst + (lane & 16 ? 4 : 0)) = make_float4(x0.x, x0.y, x1.x, x1.y);
        } else {
          const bool hi = lane & 8;
          const float2 sv = hi ? x0 : x1;
          float2 x = hi ? x1 : x0;
          x.x += __shfl_xor_sync(0xFFFFFFFFu, sv.x, 8);
          x.y += __shfl_xor_sync(0xFFFFFFFFu, sv.y, 8);
          *reinterpret_cast<float2 *>(dst + (lane & 16 ? 4 : 0) + (hi ? 2 : 0)) = x;
        }
        float ls = l, rs = lr;
#pragma unroll
        for (int o = 4; o <= 16; o <<= 1) {
          ls += __shfl_xor_sync(0xFFFFFFFFu, ls, o);
          if (IDENT) rs += __shfl_xor_sync(0xFFFFFFFFu, rs, o);
        }
        if (lane == 0) {
          red_m[bb][cw] = m;
          red_l[bb][cw] = ls;
          if (IDENT) red_r[bb][cw] = rs;
        }
      } else if (h >= 0) {
        const int si = cw * RPW + grp;
        float2 *dst = reinterpret_cast<float2 *>(&red_acc[bb][si % NST][col * EPL]);
#pragma unroll
        for (int e = 0; e < EPL / 2; ++e) dst[e] = acc[e];
        if (col == 0) {
          red_m[bb][si % NST] = m;
          red_l[bb][si % NST] = l;
          if (IDENT) red_r[bb][si % NST] = lr;
        }
      }
      if (cw == 0 && lane == 0) {
        seg[bb].h = h;
        seg[bb].flags = flags;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&epi_full[bb]);
      ++nseg;
    };
    constexpr int NJ = MMA ? D / 32 : 1;          // 16-byte pieces of a row per lane
    constexpr int NB = MMA ? TT / (kCW * 8) : 1;  // 8-row blocks per warp and tile
    constexpr int VS = MMA ? 8 / RPW : 1;         // row steps of a block's V
    constexpr bool kEarlyV = NB * VS <= 8;        // V is loaded with K while registers last
    static_assert(!MMA || TT % (kCW * 8) == 0, "blocks of 8 rows");
    uint32_t qb[NJ][2];
    typename M::Q q;
    int stage = 0;
    uint32_t fph = 0;  // parity of the stage's full barrier
    for (;;) {
      const long long c0 = STEP_CLK();
      if (!mbar_wait_unless(&full[stage], fph, &s_abort)) {
        s_abort = 1;
        set_err(p.err, HKV_ERR_TIMEOUT);
        break;
      }
      if (n_tiles > 0) w_full += STEP_CLK() - c0;
      const TileMeta mt4 = meta[stage];
      const int flags = mt4.flags;
      if (flags & kDone) break;
      if (n_tiles == 0 && tid == 32) STEP_TRACE(3);
      ++n_tiles;
      const int nr = mt4.n;
      const unsigned char *Ks = stages + stage * S::kStageBytes;
      const unsigned char *Vs = Ks + TT * RB;
      if (flags & kFirst) {  // first tile of this head in this piece
        if constexpr (MMA) {
#pragma unroll
          for (int j = 0; j < NJ; ++j) {
            const uint4 u = *reinterpret_cast<const uint4 *>(Vs + TT * RB + ((lane & 3) + 4 * j) * 16);
            qb[j][0] = lane & 4 ? u.y : u.x;
            qb[j][1] = lane & 4 ? u.w : u.z;
          }
        } else {
          M::load_q(q, *reinterpret_cast<const uint4 *>(Vs + TT * RB + col * 16), p.qscale);
        }
#pragma unroll
        for (int e = 0; e < EPL / 2; ++e) acc[e] = make_float2(0.f, 0.f);
        m = -INFINITY;
        l = 0.f;
        lr = 0.f;
      }
      if constexpr (MMA) {
        if (cw * 8 < nr) {  // the warp has rows in this tile
          // q.k of 8 rows on the tensor cores. Lane (g, t) = (lane / 4,
          // lane % 4) reads pieces t + 4j of row g, four registers x y z w of
          // two channels each, and passes them as the A fragment as they
          // are: x and z are then row g of A (k 0..7 and 8..15), y and w row
          // g + 8. The even columns of B hold the query's channels of x and
          // z, the odd ones those of y and w, so the row's dot product is
          // C[g][even] + C[g + 8][odd]: c[0] + c[3] in all lanes of quad g.
          uint4 vf[kEarlyV ? NB : 1][VS];
          // V: whole rows by groups of lanes, RPW rows a step; rows past the
          // tile's are not read (they may hold anything)
          auto load_v = [&](int rb, int st) {
            return rb + st * RPW + grp < nr
                       ? *reinterpret_cast<const uint4 *>(Vs + (rb + st * RPW + grp) * RB + col * 16)
                       : make_uint4(0u, 0u, 0u, 0u);
          };
          float dots[NB];
          float mt = -INFINITY;
#pragma unroll
          for (int b8 = 0; b8 < NB; ++b8) {
            const int rb = (b8 * kCW + cw) * 8;
            dots[b8] = -INFINITY;
            if (rb < nr) {  // warp-uniform
              const unsigned char *kr = Ks + (rb + (lane >> 2)) * RB + (lane & 3) * 16;
              uint4 kf[NJ];
#pragma unroll
              for (int j = 0; j < NJ; ++j) kf[j] = *reinterpret_cast<const uint4 *>(kr + j * 64);
              if (kEarlyV) {
#pragma unroll
                for (int st = 0; st < VS; ++st) vf[kEarlyV ? b8 : 0][st] = load_v(rb, st);
              }
              float c[2][4] = {};
#pragma unroll
              for (int j = 0; j < NJ; ++j) mma_bf16(c[j & 1], kf[j], qb[j][0], qb[j][1]);
              if (rb + (lane >> 2) < nr) dots[b8] = (c[0][0] + c[1][0]) + (c[0][3] + c[1][3]);
              mt = fmaxf(mt, dots[b8]);
            }
          }
          const float mn = fmaxf(m, warp_max(mt) * p.qscale);
          if (mn != -INFINITY) {  // warp-uniform
            if (mn != m) {
              const float corr = ex2_approx(m - mn);  // measured: 0.11 us per step less than exp2f
              l *= corr;
              if (IDENT) lr *= corr;
#pragma unroll
              for (int e = 0; e < EPL / 2; ++e) acc[e] = __fmul2_rn(acc[e], make_float2(corr, corr));
              m = mn;
            }
#pragma unroll
            for (int b8 = 0; b8 < NB; ++b8) {
              const int rb = (b8 * kCW + cw) * 8;
              if (rb < nr) {
                // of row rb + lane / 4; one rounding of the exponent
                const float pr = ex2_approx(fmaf(dots[b8], p.qscale, -mn));
                l += pr;
                if (IDENT && rb + (lane >> 2) >= mt4.recent0) lr += pr;
#pragma unroll
                for (int st = 0; st < VS; ++st)
                  M::add_v(acc, kEarlyV ? vf[kEarlyV ? b8 : 0][st] : load_v(rb, st),
                           __shfl_sync(0xFFFFFFFFu, pr, (st * RPW + grp) * 4));
              }
            }
          }
        }
      } else {
        float sc[S::kSteps];
#pragma unroll
        for (int st = 0; st < S::kSteps; ++st) {
          const int r = st * (kCW * RPW) + cw * RPW + grp;
          float dot = 0.f;
          if (r < nr) dot = M::dot(q, *reinterpret_cast<const uint4 *>(Ks + r * RB + col * 16));
#pragma unroll
          for (int o = LPR / 2; o >= 1; o >>= 1) dot += __shfl_xor_sync(0xFFFFFFFFu, dot, o);
          sc[st] = r < nr ? M::score(dot, p.qscale) : -INFINITY;
        }
        float mt = sc[0];
#pragma unroll
        for (int st = 1; st < S::kSteps; ++st) mt = fmaxf(mt, sc[st]);
        const float mn = fmaxf(m, mt);
        if (mn != -INFINITY) {
          const float corr = ex2_approx(m - mn);
          l *= corr;
          if (IDENT) lr *= corr;
#pragma unroll
          for (int e = 0; e < EPL / 2; ++e) acc[e] = __fmul2_rn(acc[e], make_float2(corr, corr));
#pragma unroll
          for (int st = 0; st < S::kSteps; ++st) {
            const int r = st * (kCW * RPW) + cw * RPW + grp;
            if (r < nr) {
              const float pr = ex2_approx(sc[st] - mn);
              l += pr;
              if (IDENT && r >= mt4.recent0) lr += pr;
              M::add_v(acc, *reinterpret_cast<const uint4 *>(Vs + r * RB + col * 16), pr);
            }
          }
          m = mn;
        }
      }
      __syncwarp();
      mbar_arrive_if(&empty[stage], lane == 0);
      if (flags & kLast) hand_over(mt4.h, flags);  // last tile of this head in this piece
      if (NS == 1 || ++stage == NS) {
        stage = 0;
        fph ^= 1u;
      }
    }
    if (tid == 32) STEP_TRACE(4);
    if (tid == 32) STEP_TRACE_SET(17, n_tiles);
    hand_over(-1, 0);  // nothing more
    if (tid == 32) STEP_TRACE_SET(21, w_full);
    if (tid == 32) STEP_TRACE_SET(22, w_hand);
  } else if (warp == kCW + 1) {
    // ---- epilogue: combine each segment's row-group states ----------------
    bool have_ep = false;  // the epoch and the merge head (merge warp)
    long long w_epi = 0;   // cycles waiting for segments (tracer)
    int k = 0;
    for (;; ++k) {
      const int bb = k & 1;
      const long long c0 = STEP_CLK();
      if (!s_abort && !mbar_wait(&epi_full[bb], (uint32_t)(k >> 1) & 1u)) {
        s_abort = 1;
        set_err(p.err, HKV_ERR_TIMEOUT);
      }
      if (k > 0) w_epi += STEP_CLK() - c0;
      if (s_abort) break;
      const SegMeta sg = seg[bb];
      if (sg.h < 0) break;
      const int h = sg.h;
      // every lane weighs every state itself: no exchange between lanes
      float ws[NST];
#pragma unroll
      for (int si = 0; si < NST; ++si) ws[si] = red_m[bb][si];
      float mx = ws[0];
#pragma unroll
      for (int si = 1; si < NST; ++si) mx = fmaxf(mx, ws[si]);
      float L = 0.f, LR = 0.f, A[CPL];
#pragma unroll
      for (int c = 0; c < CPL; ++c) A[c] = 0.f;
#pragma unroll
      for (int si = 0; si < NST; ++si) {
        ws[si] = ws[si] == -INFINITY ? 0.f : exp2f(ws[si] - mx);
        L = fmaf(red_l[bb][si], ws[si], L);
        if (IDENT) LR = fmaf(red_r[bb][si], ws[si], LR);
        float r[CPL];
        V::lds(&red_acc[bb][si][CPL * lane], r);
#pragma unroll
        for (int c = 0; c < CPL; ++c) A[c] = fmaf(r[c], ws[si], A[c]);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&epi_free[bb]);  // the consumers may reuse the buffer
      const bool whole = sg.flags & kWhole;
      if (!whole && !have_ep) {
        if (!mbar_wait(&ep_bar, 0u)) {
          s_abort = 1;
          set_err(p.err, HKV_ERR_TIMEOUT);
          break;
        }
        have_ep = true;
      }
      if (whole) {  // the whole head is in this CTA's range
        // (attention alone: a head without rows gives zeros)
        const bool none = !FUSED && L == 0.f;
#pragma unroll
        for (int c = 0; c < CPL; ++c) A[c] = none ? 0.f : A[c] / L;
        V::st(p.out + (size_t)h * D + CPL * lane, A);
        // Sec. 4 Step 2: local iff the newest w_loc - 1 tokens hold a share
        // tau of the attention
        if (IDENT && lane == 0)
          p.label_out[p.layer_base + h] = LR >= p.tau * L ? HKV_LOCAL : HKV_GLOBAL;
      } else if (h == s_mg_h) {  // this CTA combines the head
        // the other pieces already combined by the merge warp: finish here;
        // else hand this piece to the merge warp
        int ready = mbar_test_wait(&oth_bar, 0u) ? 1 : 0;
        ready = __shfl_sync(0xFFFFFFFFu, ready, 0);
        if (ready) {
          mbar_wait(&oth_bar, 0u);  // complete: every lane acquires oth_*
          float A2[CPL], Lt, Rt = 0.f;
          V::lds(&oth_acc[CPL * lane], A2);
          combine_store<CPL, IDENT>(mx, L, LR, A, oth_s[0], oth_s[1], IDENT ? oth_s[NV - 1] : 0.f,
                                    A2, p.out + (size_t)h * D + CPL * lane, Lt, Rt);
          if (IDENT && lane == 0)
            p.label_out[p.layer_base + h] = Rt >= p.tau * Lt ? HKV_LOCAL : HKV_GLOBAL;
          STEP_TRACE_SET(18, globaltimer());
        } else {
          V::st(&own_acc[CPL * lane], A);
          if (lane == 0) {
            own_s[0] = mx;
            own_s[1] = L;
            if (IDENT) own_s[NV - 1] = LR;
          }
        }
        if (lane == 0) s_own_state = ready ? 1 : 2;
        __syncwarp();
        mbar_arrive(&own_bar);  // all 32 lanes
      } else {  // a piece for the combining CTA: epoch-tagged, no fence needed
        unsigned long long *ps = p.pslot + ((size_t)bx * 2 + (sg.flags & kTailPiece ? 1 : 0)) * PS;
#pragma unroll
        for (int c = 0; c < CPL; ++c) st_pair(ps + CPL * lane + c, A[c], s_ep);
        if (lane == 0) {
          st_pair(ps + D, mx, s_ep);
          st_pair(ps + D + 1, L, s_ep);
          if (IDENT) st_pair(ps + D + 2, LR, s_ep);
        }
      }
    }
    if (IDENT && lane == 0) s_streamed = 1;
    if (lane == 0) STEP_TRACE(5);
    STEP_TRACE_SET(9, k);
    if (lane == 0) STEP_TRACE_SET(23, w_epi);
  } else {
    // ---- merge warp: appends, counters, the combined split head -------------
    if (lane == 0 && own_bad) arrive();
    gen0 = __shfl_sync(0xFFFFFFFFu, gen0, 0);
    bar_done = __shfl_sync(0xFFFFFFFFu, bar_done, 0);
    const uint64_t t0 = globaltimer();
    auto timed_out = [&]() {
      if (globaltimer() - t0 <= kWaitTimeoutNs) return false;
      if (lane == 0) {
        s_abort = 1;
        set_err(p.err, HKV_ERR_TIMEOUT);
      }
      return true;
    };
    if (own_bad) {
      // empty pieces in both of this CTA's slots, so that no combining CTA
      // waits for them (the step is not taken; the outputs are not defined)
      for (int sl = 0; sl < 2; ++sl) {
        unsigned long long *ps = p.pslot + ((size_t)bx * 2 + sl) * PS;
        for (int c = lane; c < D; c += 32) st_pair(ps + c, 0.f, s_ep);
        if (lane == 0) {
          st_pair(ps + D, -INFINITY, s_ep);
          st_pair(ps + D + 1, 0.f, s_ep);
          if (IDENT) st_pair(ps + D + 2, 0.f, s_ep);
        }
      }
    }
    auto poll = [&]() {  // whether the whole grid has arrived
      if (bar_done) return true;
      if (lane == 0) {
        gen1 = ld_acquire(p.bar + 1);
        bar_done = gen1 != gen0;
      }
      bar_done = __shfl_sync(0xFFFFFFFFu, bar_done, 0);
      return bar_done != 0;
    };
    // The heads whose last row is in the range (a range's first head always
    // reaches past its start; only its last one can continue past its end).
    const int napp = DYN ? sh1 - sh0 : active ? (has_e ? n - 1 : n) : 0;
    const int app0 = DYN ? sh0 : h0;
    // a head's last row (the step's token) in the arena, and its image tokens
    // (known: the head is in the table)
    auto last_row = [&](int h, bool known) {
      return DYN || !known ? p.off[h] + p.len[h] : tab.off[h - wl] + tab.vlen[h - wl] - 1;
    };
    auto tokens_of = [&](int h, bool known) {
      return DYN || !known ? p.ntok[p.layer_base + h] : tab.ntok[h - wl];
    };
    // Appends of `count` heads: the K/V row at index len, its position, q into
    // the ring of the periodic update. Nothing in this launch reads them.
    auto append = [&](int first, int count, bool known) {
      // the K, V and q rows of every appended head as 16-byte chunks, a
      // lane per chunk, every load of a round issued before its stores
      constexpr int CH = RB / 16;  // chunks of a row
      constexpr int NU = IDENT ? 4 : 8;  // chunks per lane and round (registers)
      const int units = count * 3 * CH;
      for (int u0 = 0; u0 < units; u0 += 32 * NU) {
        uint4 x[NU];
        unsigned char *dst[NU];
#pragma unroll
        for (int v = 0; v < NU; ++v) {
          const int u = u0 + v * 32 + lane;
          dst[v] = nullptr;
          if (u < units) {
            const int w3 = (u / CH) % 3, cc = u % CH;
            const int h = first + u / (3 * CH), i = p.layer_base + h;
            const unsigned char *src = w3 == 0 ? static_cast<const unsigned char *>(p.k_new)
                                     : w3 == 1 ? static_cast<const unsigned char *>(p.v_new)
                                               : static_cast<const unsigned char *>(p.q);
            x[v] = reinterpret_cast<const uint4 *>(src + (size_t)h * RB)[cc];
            const long long row = last_row(h, known);
            unsigned char *d = w3 == 0 ? static_cast<unsigned char *>(p.K) + row * RB
                             : w3 == 1 ? static_cast<unsigned char *>(p.V) + row * RB
                                       : static_cast<unsigned char *>(p.qbuf) +
                                             ((size_t)i * p.period + tokens_of(h, known) % p.period) * RB;
            dst[v] = d + (size_t)cc * 16;
          }
        }
#pragma unroll
        for (int v = 0; v < NU; ++v)
          if (dst[v]) *reinterpret_cast<uint4 *>(dst[v]) = x[v];
      }
      for (int h = first + lane; h < first + count; h += 32)
        p.pos[last_row(h, known)] = p.n_cond + tokens_of(h, known);
    };
    // the counters of `count` heads whose tokens are appended
    auto advance = [&](int first, int count, bool known) {
      for (int h = first + lane; h < first + count; h += 32) {
        const int i = p.layer_base + h;
        if (DYN && h < sh0 + 32) {
          p.len[h] = k_len + 1;
          p.ntok[i] = k_nt + 1;
          if (k_nb >= 0) p.nbuf[i] = k_nb + 1;
        } else if (DYN || !known) {
          ++p.len[h];
          ++p.ntok[i];
          if (p.label[i] != HKV_DENSE) ++p.nbuf[i];
        } else {
          const int j = h - wl;
          p.len[h] = tab.vlen[j];
          p.ntok[i] = tab.ntok[j] + 1;
          if (!tab.dense(j)) ++p.nbuf[i];
        }
      }
    };
    // Counters advance once the whole grid has arrived (every CTA has read
    // them). With in_regs every CTA has checked every head, so the step is
    // known to be taken and the appends need not wait for that; otherwise the
    // barrier also tells whether some CTA found a bad head.
    //
    // Identification holds no CTA back for that for long: one that has streamed
    // its range and sees no end of the arrivals for kHoldNs more leaves the rest
    // of its share (appends unless in_regs, counters) to the last CTA to arrive
    // and ends, which may be what lets that one start (launches on other
    // streams can hold its place). A launch that has the GPU to itself has
    // arrived by then; without the hold its first CTAs left their shares to one
    // warp (12 sequences of Janus-Pro-7B: 9.2 us a layer, 17 without). A CTA
    // that leaves says so in the layer's hint word and looks for the arrivals
    // once more, and the last CTA publishes them before it reads the hint, so
    // one of the two sees the other. Where both do, they settle it on a word of
    // the CTA's: whoever exchanges it second sees the other's mark, tagged with
    // the epoch, and does the share. (Without the hint, the last CTA's walk over
    // all words cost 3.8 us of a layer step of 9.7.)
    bool advanced = !FUSED || (IDENT && napp == 0);
    const unsigned long long tag = (unsigned long long)s_ep << 32;
    constexpr unsigned kLeft = 1, kArrived = 2;
    constexpr uint64_t kHoldNs = 20000;
    auto hand_word = [&](int k, int sl) { return p.pslot + ((size_t)k * 2 + sl) * PS + D + 3; };
    auto settle = [&](int first, int count, bool known) {  // once the grid has arrived
      if (IDENT && (__shfl_sync(0xFFFFFFFFu, gen1, 0) & kBadStep)) return;
      if (IDENT && !in_regs) append(first, count, known);
      advance(first, count, known);
    };
    if (FUSED && in_regs) {
      append(app0, napp, true);
      if (poll()) {
        advance(app0, napp, true);
        advanced = true;
      }
    } else if (IDENT) {
      if (!advanced && poll()) {
        settle(app0, napp, true);
        advanced = true;
      }
    } else if (FUSED) {
      while (!s_abort && !poll())
        if (timed_out()) break;
      gen1 = __shfl_sync(0xFFFFFFFFu, gen1, 0);
      STEP_TRACE_SET(19, globaltimer());
      if (!s_abort && bar_done && !(gen1 & kBadStep)) {
        append(app0, napp, true);
        if (DYN) {  // the lengths advance once no CTA reads another
          bool all = false;
          while (!s_abort && !all) {
            all = __shfl_sync(0xFFFFFFFFu, lane == 0 ? ld_acquire(p.bar + 5) != taken0 : 0, 0);
            if (!all && timed_out()) break;
          }
          __syncwarp();
          if (all) advance(app0, napp, true);
        } else {
          advance(app0, napp, true);
        }
      }
      advanced = true;
    }
    if constexpr (IDENT) {
      if (__shfl_sync(0xFFFFFFFFu, hinted, 0)) {
        for (int k0 = 0; k0 < G; k0 += 32) {
          const int k = k0 + lane;
          unsigned long long share = 0;
          if (k < G && k != bx &&
              atom_exch_acq_rel(hand_word(k, 0), tag | kArrived) == (tag | kLeft))
            share = *hand_word(k, 1);
          unsigned left = __ballot_sync(0xFFFFFFFFu, share != 0);
          while (left) {
            const unsigned long long w = __shfl_sync(0xFFFFFFFFu, share, __ffs(left) - 1);
            left &= left - 1;
            settle((int)(w >> 32), (int)(uint32_t)w, false);
          }
        }
      }
    }
    STEP_TRACE_SET(8, globaltimer());

    // The split head this CTA combines: the other pieces, combined in index
    // order once all of them carry this launch's epoch, then this CTA's own
    // piece (from the epilogue), so the result does not depend on timing.
    const int mh = s_mg_h;
    if (mh >= 0 && !s_abort) {
      const int np = s_mg_np, mj = s_mg_j, k0 = s_mg_k0;
#ifdef HKV_STEP_TEST_STALL
      // test builds only: wait for an epoch no launch writes, so that the
      // bounded wait runs out (HKV_ERR_TIMEOUT) with no bulk copy involved
      const uint32_t want = s_ep + 1u;
#else
      const uint32_t want = s_ep;
#endif
      float om = -INFINITY, ol = 0.f, orr = 0.f, oA[CPL];
      for (;;) {
        bool ready = true;
        om = -INFINITY;
        ol = orr = 0.f;
#pragma unroll
        for (int c = 0; c < CPL; ++c) oA[c] = 0.f;
        for (int t = 0; t < np && ready; ++t) {
          if (t == mj) continue;
          // piece t: the end piece of CTA k0, the start piece of the others
          const unsigned long long *ps = p.pslot + ((size_t)(k0 + t) * 2 + (t > 0 ? 1 : 0)) * PS;
          float At[CPL], mt, lt, rt = 0.f;
          bool ok = true;
#pragma unroll
          for (int c = 0; c < CPL; ++c) ok &= ld_pair(ps + CPL * lane + c, want, At[c]);
          ok &= ld_pair(ps + D, want, mt);
          ok &= ld_pair(ps + D + 1, want, lt);
          if (IDENT) ok &= ld_pair(ps + D + 2, want, rt);
          ready = __all_sync(0xFFFFFFFFu, ok);
          if (!ready) break;
          const float mn = fmaxf(om, mt);
          const float co = om == -INFINITY ? 0.f : exp2f(om - mn);
          const float ct = mt == -INFINITY ? 0.f : exp2f(mt - mn);
          ol = ol * co + lt * ct;
          orr = orr * co + rt * ct;
#pragma unroll
          for (int c = 0; c < CPL; ++c) oA[c] = fmaf(At[c], ct, oA[c] * co);
          om = mn;
        }
        if (ready || timed_out()) break;
        if (!advanced && poll()) {
          settle(app0, napp, true);
          advanced = true;
        }
      }
      // hand the combined other pieces to the epilogue (not after a wait
      // that ran out: the head's output is then not written)
      if (!s_abort) {
        V::st(&oth_acc[CPL * lane], oA);
        if (lane == 0) {
          oth_s[0] = om;
          oth_s[1] = ol;
          if (IDENT) oth_s[NV - 1] = orr;
        }
        __syncwarp();
        mbar_arrive(&oth_bar);  // all 32 lanes
      }
      // this CTA's own piece, unless the epilogue combined it already
      while (!s_abort && !mbar_try_wait(&own_bar, 0u))
        if (timed_out()) break;
      __syncwarp();
      if (!s_abort && s_own_state == 2) {
        mbar_wait(&own_bar, 0u);  // complete: every lane acquires own_*
        float A1[CPL], Lt, Rt = 0.f;
        V::lds(&own_acc[CPL * lane], A1);
        combine_store<CPL, IDENT>(own_s[0], own_s[1], IDENT ? own_s[NV - 1] : 0.f, A1, om, ol, orr,
                                  oA, p.out + (size_t)mh * D + CPL * lane, Lt, Rt);
        if (IDENT && lane == 0)
          p.label_out[p.layer_base + mh] = Rt >= p.tau * Lt ? HKV_LOCAL : HKV_GLOBAL;
        STEP_TRACE_SET(18, globaltimer());
      }
    }
    if (!advanced) {
      uint64_t hold = 0;  // lane 0: the end of the hold
      while (!s_abort && !poll()) {
        if constexpr (IDENT) {
          bool leave = false;
          if (lane == 0 && s_streamed) {
            const uint64_t now = globaltimer();
            if (hold == 0) hold = now + kHoldNs;
            leave = now >= hold;
          }
          if (__shfl_sync(0xFFFFFFFFu, leave, 0)) break;
        }
        if (timed_out()) break;
      }
      STEP_TRACE_SET(19, globaltimer());
      if (!s_abort && bar_done) {
        settle(app0, napp, true);
      } else if (IDENT && !s_abort) {
        if (lane == 0) {
          st_release(p.bar + 6, s_ep);
          __threadfence();  // the hint before the generation
        }
        if (!poll()) {
          if (lane == 0) {
            *hand_word(bx, 1) = (unsigned long long)app0 << 32 | (uint32_t)napp;
            if (atom_exch_acq_rel(hand_word(bx, 0), tag | kLeft) == (tag | kArrived)) {
              gen1 = ld_acquire(p.bar + 1);
              bar_done = 1;
            }
          }
          bar_done = __shfl_sync(0xFFFFFFFFu, bar_done, 0);
        }
        if (bar_done) settle(app0, napp, true);  // the grid has arrived meanwhile
      }
    }
    if (lane == 0) STEP_TRACE(6);
  }
}

template <class S>
constexpr size_t step_smem_of() {
  return (size_t)S::kNS * S::kStageBytes;
}
template <int D, typename T, int CUT>
constexpr size_t step_smem() {
  return step_smem_of<StepShape<D, T, CUT == kCutShort>>();
}

template <int D, typename T, int MODE, int CUT>
cudaError_t step_prepare_m(int *ctas) {
  const size_t smem = step_smem<D, T, CUT>();
  const size_t most = smem > kLoneSmem ? smem : kLoneSmem;
  cudaError_t e = cudaFuncSetAttribute(step_kernel<D, T, MODE, CUT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e != cudaSuccess) return e;
  int n = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, step_kernel<D, T, MODE, CUT>,
                                                    step_threads<D, T>(), smem);
  if (n < *ctas) *ctas = n;
  return e;
}

template <int D, typename T>
cudaError_t step_prepare_t(int *ctas) {
  *ctas = kStepActivePerSm;
  cudaError_t e = step_prepare_m<D, T, kModeStep, kCutRanges>(ctas);
  if (e == cudaSuccess) e = step_prepare_m<D, T, kModeStep, kCutShort>(ctas);
  if (e == cudaSuccess) e = step_prepare_m<D, T, kModeStep, kCutHeads>(ctas);
  if (e == cudaSuccess) e = step_prepare_m<D, T, kModeIdentify, kCutRanges>(ctas);
  if (e == cudaSuccess) e = step_prepare_m<D, T, kModeAttend, kCutRanges>(ctas);
  return e;
}

template <int D, typename T, int MODE, int CUT>
cudaError_t step_launch_m(const AttnArgs &a, StepPlan plan, cudaStream_t s) {
  static const bool pdl = getenv("HKV_NO_PDL") == nullptr;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(plan.grid);
  cfg.blockDim = dim3(step_threads<D, T>());
  cfg.dynamicSmemBytes = plan.lone ? kLoneSmem : step_smem<D, T, CUT>();
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  int na = 0;
  if (pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, step_kernel<D, T, MODE, CUT>, a);
}

template <int D, typename T>
cudaError_t step_launch_t(AttnArgs a, StepPlan plan, bool fused, cudaStream_t s) {
  // (not used for a grid of one)
  a.grid_recip = (uint32_t)(((1ull << 32) + plan.grid - 1) / plan.grid);
  if (!fused) return step_launch_m<D, T, kModeAttend, kCutRanges>(a, plan, s);
  if (a.label_out) return step_launch_m<D, T, kModeIdentify, kCutRanges>(a, plan, s);
  return plan.cut == kCutShort   ? step_launch_m<D, T, kModeStep, kCutShort>(a, plan, s)
         : plan.cut == kCutHeads ? step_launch_m<D, T, kModeStep, kCutHeads>(a, plan, s)
                                 : step_launch_m<D, T, kModeStep, kCutRanges>(a, plan, s);
}

// The CTAs a layer of n heads gets out of a full grid: see step_plan.
template <int D, typename T>
StepPlan step_plan_t(long long n, long long max_rows, int full, bool fused, bool identify) {
  using S = StepShape<D, T>;
  static_assert(step_smem_of<S>() <= kLoneSmem, "a lone CTA's shared memory holds its stages");
  const long long g = (max_rows + S::kGR - 1) / S::kGR;
  const long long total = n * (g + 1 > S::kMinCost ? g + 1 : S::kMinCost);
  const int sms = full / kStepActivePerSm > 1 ? full / kStepActivePerSm : 1;
  const bool lone = S::kRB == 512 && (total < (long long)kLoneSlots * sms || 3 * n < full);
  if (lone) full = sms;
  const int head_slots = S::kRB == 512 ? kHeadSlots512 : kHeadSlots;
  if (fused && !identify && total >= (long long)head_slots * full && g <= kHeadGrains)
    return {full, kCutHeads, 0};
  long long chunk = (total + full - 1) / full;
  const int least = S::min_chunk(fused && !identify);
  if (chunk < least) chunk = least;
  if (n > kStepTable && chunk / S::kMinCost + 2 > kStepTable) return {0, kCutRanges, 0};
  if (!fused) return {full, kCutRanges, lone};
  if (!identify && n <= full && n <= kStepTable && g <= kAlignedGrains) return {(int)n, kCutShort, 0};
  const long long need = (total + least - 1) / least;
  return {need < full ? (int)need : full, kCutRanges, lone};
}

}  // namespace

#ifdef HKV_ATTN_TRACE
extern "C" int hkv_debug_set_step_trace(unsigned long long *buf) {
  return cudaMemcpyToSymbol(g_step_trace, &buf, sizeof(buf)) == cudaSuccess ? 0 : 7;
}
#endif

StepPlan step_plan(int D, int dtype, int nheads, int max_rows, int full, bool fused, bool identify) {
  if (dtype == HKV_BF16)
    return D == 64 ? step_plan_t<64, __nv_bfloat16>(nheads, max_rows, full, fused, identify)
                   : step_plan_t<128, __nv_bfloat16>(nheads, max_rows, full, fused, identify);
  return D == 64 ? step_plan_t<64, float>(nheads, max_rows, full, fused, identify)
                 : step_plan_t<128, float>(nheads, max_rows, full, fused, identify);
}

cudaError_t step_prepare(int D, int dtype, int *ctas) {
  if (dtype == HKV_BF16)
    return D == 64 ? step_prepare_t<64, __nv_bfloat16>(ctas) : step_prepare_t<128, __nv_bfloat16>(ctas);
  return D == 64 ? step_prepare_t<64, float>(ctas) : step_prepare_t<128, float>(ctas);
}

cudaError_t launch_step(const AttnArgs &a, int D, int dtype, StepPlan plan, bool fused,
                        cudaStream_t s) {
  if (plan.grid < 1 || plan.grid > kAttnMaxGrid) return cudaErrorInvalidValue;
  if (dtype == HKV_BF16)
    return D == 64 ? step_launch_t<64, __nv_bfloat16>(a, plan, fused, s)
                   : step_launch_t<128, __nv_bfloat16>(a, plan, fused, s);
  return D == 64 ? step_launch_t<64, float>(a, plan, fused, s)
                 : step_launch_t<128, float>(a, plan, fused, s);
}

}  // namespace hkv
