// Per-head cache maintenance of HeadKV, one CTA per head:
//  * evict / append_evict: the periodic head-aware update when a head's
//    buffer holds P tokens (Sec. 4: local heads drop their history, Eq. 3;
//    global heads trim it by Stratified Token Eviction, Eqs. 4-6), and for
//    append_evict the append of the new token after it (Sec. 3, KV Cache);
//  * repack: the first update at grouping, out of place from the dense
//    cache into the ragged one (Step 3);
//  * prefill / init_dense: the uncompressed cache of Step 1;
//  * identify: threshold-based attention accumulation (Step 2);
//  * budgets: per-head budgets and the arena layout (Sec. 5.1).
//
// The update works on token POSITIONS, not on storage order, so a segment
// may hold its live tokens in any order:
//  * conditioning tokens have positions < C; the recent window is the newest
//    w image tokens, positions >= C + ntok - w; everything else is history;
//  * Eq. 5's long-range subset is the floor(T * r_s) history tokens with the
//    smallest positions (a rank select on positions);
//  * scores q-bar . k in a fixed fp32 order, keys (order-preserving score
//    bits, position) unique and ascending in eviction priority, one 8-pass
//    MSD radix select finds the quota-th key of both subsets at once;
//  * in place, the holes below the new length are refilled with the
//    surviving rows above it: at most M rows move and no move depends on
//    another, instead of shifting every row after the first eviction.
#include <math.h>
#include <stdlib.h>

#include "hkv_device.cuh"
#include "hkv_kernels.h"

namespace hkv {
namespace {

constexpr int IT = kCacheThreads;  // of the identification kernels (their sums' order goes with it)

// Threads of an update CTA (NT below: 128, 256 or 512; the results do not
// depend on it) and how many CTAs the register budget allows on an SM (48
// registers a thread, 64 with 512; no spills). An update is a chain of
// latency-bound phases between block barriers. With many heads for every SM
// what counts is how many run at once: CTAs of four warps, up to ten on an SM,
// rather than eight warps staging whole rows of keys in 70 KB, two or three on
// an SM. Lumina-mGPT 1024, 8 sequences, all layers: 475 -> 327 us (of 264 at
// the measured bandwidth); with 256 threads and four CTAs 339. LlamaGen-XL's
// 92160 heads of up to 121 rows: 1.34 -> 0.9 ms a period. With few heads a head
// has an SM nearly to itself and more warps pass over its rows at once. One
// launch, us with 128, 256 and 512 threads: segments of 1233 rows, 128 heads
// 52, 40, 34 (fp32 70, 49, 41), 512 64, 60, 48 (88, 77, 66), 1024 81, 72, 76
// (112, 100, 104), 2048 116, 110, 122 (187, 160, 174), 8192 319, 321, 399;
// of 3193 rows, 128 heads 96, 62, 49 (151, 91, 64), 2048 241, 210, 264; of 160
// rows, 256 heads 27.3, 27.0, 27.4 (30.7, 28.6, 29.6), 1024 29, 34, 44 (34,
// 37, 49). update_threads draws the lines from these.
constexpr int upd_ctas(int NT) { return NT == 128 ? 10 : NT == 256 ? 5 : 2; }

// Phase timestamps per head of the update for latency studies; compiled out
// by default.
#ifdef HKV_UPD_TRACE
__device__ unsigned long long *g_utrace = nullptr;  // [head of the layer][8], set by the tracer
#define HKV_UTRACE(slot)                                                   \
  do {                                                                     \
    if (g_utrace && threadIdx.x == 0)                                      \
      g_utrace[(size_t)blockIdx.x * 8 + (slot)] = globaltimer();           \
  } while (0)
#else
#define HKV_UTRACE(slot) \
  do {                   \
  } while (0)
#endif

__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

struct SegRef {
  const unsigned char *sk, *sv;  // source rows, row 0 = segment start
  const int32_t *spos;
  unsigned char *dk, *dv;        // destination rows
  int32_t *dpos;
  int len;                       // live source rows
  int dst_cap;                   // destination capacity (rows)
  bool in_place;
  uint32_t *err;                 // the cache's error word
};

struct UpdShared {
  unsigned long long prefix[2];
  int rem[2];
  int iscan[33];
  long long lscan[33];
  uint64_t ring_bar;  // completion of the bulk copy of the query ring
};

// Shared-memory work area of one update (dynamic).
struct UpdSmem {
  unsigned char *ring;  // [P][D] the buffered queries (<= 4 B each); then the score stages
  uint32_t *kh;         // [max_len] high words of the selection keys (the low ones: positions)
  int *ps;              // [max_len] positions of the source rows
  int16_t *aux;         // [max_len] class, then keep flag, then rank
  float *qbar;          // [D]
  int *hist;            // [512]
  int stage_rows;       // rows a warp stages at a time in the score phase
};

// Rows a warp stages at a time in the score phase: 32, or fewer when every
// warp's share of the longest segment is smaller (short segments then leave
// room for more CTAs per SM).
__host__ __device__ constexpr int stage_rows(int NT, int max_len) {
  const int share = (max_len + NT / 32 - 1) / (NT / 32);
  return max_len >= NT ? 32 : share < 1 ? 1 : share;
}

// The score phase stages 64 bytes of each row at a time, two such pieces in
// flight per warp, at a row stride of 80 bytes (lanes that read the same
// 16-byte column of consecutive rows hit distinct banks).
constexpr int kChunk = 64, kChunkStride = kChunk + 16, kChunkStages = 2;
__host__ __device__ constexpr size_t stage_bytes_of(int rows) {
  return (size_t)rows * kChunkStride * kChunkStages;
}

// the query ring (P rows of es-byte elements); after q-bar the score stages,
// and at the end the list of the rows that fill holes
__host__ __device__ constexpr size_t ring_bytes(int NT, int P, int D, int es, int max_len) {
  const size_t stages = (size_t)(NT / 32) * stage_bytes_of(stage_rows(NT, max_len));
  size_t b = (size_t)P * D * es;
  if (b < stages) b = stages;
  if (b < (size_t)max_len * 4) b = (size_t)max_len * 4;
  return (b + 15) / 16 * 16;
}

template <int NT>
__device__ __forceinline__ UpdSmem carve(unsigned char *dyn, int max_len, int D, int P, int es) {
  UpdSmem u;
  u.ring = dyn;
  u.stage_rows = stage_rows(NT, max_len);
  u.qbar = reinterpret_cast<float *>(dyn + ring_bytes(NT, P, D, es, max_len));
  u.hist = reinterpret_cast<int *>(u.qbar + D);
  u.kh = reinterpret_cast<uint32_t *>(u.hist + 512);
  u.ps = reinterpret_cast<int *>(u.kh + max_len);
  u.aux = reinterpret_cast<int16_t *>(u.ps + max_len);
  return u;
}

// The k0-th smallest key among rows of class 0 and the k1-th among rows of
// class 1 (1-based; 0 = not needed; other classes ignored), by MSD radix
// select on bytes from `top_shift` down. A key is (kh[j], ps[j]), or ps[j]
// alone. Keys are unique within a class, so each result bounds exactly k keys
// of its class from above.
template <int NT, bool HIGH>
__device__ void radix_select2(const uint32_t *kh, const int *ps, const int16_t *cls, int n, int k0,
                              int k1, int top_shift, int *hist, UpdShared &sh) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    sh.prefix[0] = sh.prefix[1] = 0ull;
    sh.rem[0] = k0;
    sh.rem[1] = k1;
  }
  __syncthreads();
  for (int shift = top_shift; shift >= 0; shift -= 8) {
    for (int i = tid; i < 512; i += NT) hist[i] = 0;
    __syncthreads();
    const unsigned long long hi = shift >= 56 ? 0ull : (~0ull << (shift + 8));
    const unsigned long long p0 = sh.prefix[0], p1 = sh.prefix[1];
    const int r0 = sh.rem[0], r1 = sh.rem[1];
    for (int j = tid; j < n; j += NT) {
      const int s = cls[j];
      if (s != 0 && s != 1) continue;
      const unsigned long long key = (HIGH ? (unsigned long long)kh[j] << 32 : 0ull) | (uint32_t)ps[j];
      if ((s ? r1 : r0) > 0 && (key & hi) == (s ? p1 : p0))
        atomicAdd(&hist[s * 256 + (int)((key >> shift) & 255ull)], 1);
    }
    __syncthreads();
    if (warp < 2) {
      const int s = warp;
      const int target = sh.rem[s];
      if (target > 0) {  // warp-uniform
        int c[8], sum = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          c[e] = hist[s * 256 + lane * 8 + e];
          sum += c[e];
        }
        const int incl = warp_incl_scan(sum);
        const int excl = incl - sum;
        if (excl < target && target <= incl) {
          int run = excl, digit = -1, rem = 0, in_bin = 0;
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            if (digit < 0 && run + c[e] >= target) {
              digit = lane * 8 + e;
              rem = target - run;
              in_bin = c[e];
            }
            run += c[e];
          }
          sh.prefix[s] |= (unsigned long long)digit << shift;
          if (rem == in_bin) {
            // every key of this bin is among the k: the bin's upper end
            // bounds exactly k keys (keys are unique), no further digit
            sh.prefix[s] |= shift > 0 ? (1ull << shift) - 1ull : 0ull;
            sh.rem[s] = 0;
          } else {
            sh.rem[s] = rem;
          }
        }
      }
    }
    __syncthreads();
    if (sh.rem[0] == 0 && sh.rem[1] == 0) break;
  }
}

__device__ __forceinline__ int block_sum(int x, UpdShared &sh) {
  int tot;
  block_excl_scan<int>(x, sh.iscan, &tot);
  return tot;
}

// Decides which rows of a segment the update evicts (Eqs. 2-6). On return
// u.aux[r] is 1 for a kept row and 0 for an evicted one (r < len), u.ps
// holds the rows' positions, and the number of evicted rows is returned.
// Block-uniform.
template <int NT, int D, typename T>
__device__ int select_evictions(const SegRef &sg, int label, const MethodArgs &m,
                                const unsigned char *qring, int ntok, const UpdSmem &u,
                                UpdShared &sh) {
  constexpr int RB = D * (int)sizeof(T);
  constexpr int EPL = Elem<T>::kPerPiece;
  const int tid = threadIdx.x;
  const int C = m.C, P = m.P;
  // the head's history budget, B_g - w with the paper's budgets, from the
  // capacity its segment was given (C + budget + P)
  const int hist_budget = sg.dst_cap - C - P - m.w > 0 ? sg.dst_cap - C - P - m.w : 0;
  // The queries of a head that will score its history come in with one bulk
  // copy, on its way while the history is counted and split.
  auto fetch_ring = [&]() {
    mbar_init(&sh.ring_bar, 1);
    fence_barrier_init();
    const uint32_t bytes = (uint32_t)P * RB;
    mbar_arrive_expect_tx(&sh.ring_bar, bytes);
    bulk_g2s(u.ring, qring, bytes, &sh.ring_bar);
  };
  const bool early = label == HKV_GLOBAL && sg.len - C - (ntok < m.w ? ntok : m.w) > hist_budget;
  if (early && tid == 0) fetch_ring();
  const int recent_from = C + (ntok > m.w ? ntok - m.w : 0);   // newest w image tokens
  int nh = 0;
  for (int r = tid; r < sg.len; r += NT) {
    const int ps = sg.spos[r];
    u.ps[r] = ps;
    const bool hist = ps >= C && ps < recent_from;
    u.aux[r] = hist ? 0 : -1;   // class: history (0) or always kept (-1)
    nh += hist ? 1 : 0;
  }
  const int NH = block_sum(nh, sh);  // history candidates (Eq. 2)
  HKV_UTRACE(1);
  int M = 0;
  if (label == HKV_LOCAL) M = NH;    // Eq. 3: no history
  else if (NH > hist_budget) M = NH - hist_budget;

  if (label == HKV_GLOBAL && M > 0) {
    auto key_of = [&](int r) { return ((unsigned long long)u.kh[r] << 32) | (uint32_t)u.ps[r]; };
    // Eq. 5: the floor(NH r_s) oldest history tokens are long-range (or,
    // in the grid-distance variant, the farthest from the newest image
    // token, equal distances older first)
    const int n_long = (int)floor((double)NH * m.r_s);
    if (n_long > 0 && n_long < NH && m.grid2d) {
      const int ref = ntok - 1;
      for (int r = tid; r < sg.len; r += NT) {
        const int i = u.ps[r] - C;
        const long long dr = i / m.row_len - ref / m.row_len, dc = i % m.row_len - ref % m.row_len;
        u.kh[r] = 0x7FFFFFFFu - (uint32_t)(dr * dr + dc * dc);
      }
      radix_select2<NT, true>(u.kh, u.ps, u.aux, sg.len, n_long, 0, 56, u.hist, sh);
      const unsigned long long k_long = sh.prefix[0];
      for (int r = tid; r < sg.len; r += NT)
        if (u.aux[r] == 0) u.aux[r] = key_of(r) <= k_long ? 0 : 1;
    } else if (n_long > 0 && n_long < NH) {
      const int maxp = C + ntok;  // positions are below it: start at its top byte
      const int top = maxp < (1 << 8) ? 0 : maxp < (1 << 16) ? 8 : maxp < (1 << 24) ? 16 : 24;
      radix_select2<NT, false>(u.kh, u.ps, u.aux, sg.len, n_long, 0, top, u.hist, sh);
      const int p_long = (int)sh.prefix[0];
      for (int r = tid; r < sg.len; r += NT)
        if (u.aux[r] == 0) u.aux[r] = u.ps[r] <= p_long ? 0 : 1;
    } else {
      for (int r = tid; r < sg.len; r += NT)
        if (u.aux[r] == 0) u.aux[r] = n_long == NH ? 0 : 1;
    }
    HKV_UTRACE(2);
    // Eq. 6 scores: q-bar = the P buffered queries, oldest first (image token
    // t in slot t mod P); the sums keep their order.
    if (!early && tid == 0) fetch_ring();
    __syncthreads();
    if (!mbar_wait(&sh.ring_bar, 0) && tid == 0) set_err(sg.err, HKV_ERR_TIMEOUT);
    for (int d = tid; d < D; d += NT) {
      float acc = 0.f;
      const int oldest = ntok % P;
#pragma unroll 8
      for (int slot = oldest; slot < P; ++slot)
        acc = __fadd_rn(acc, Elem<T>::load1(u.ring, (size_t)slot * D + d));
#pragma unroll 8
      for (int slot = 0; slot < oldest; ++slot)
        acc = __fadd_rn(acc, Elem<T>::load1(u.ring, (size_t)slot * D + d));
      u.qbar[d] = acc;
    }
    __syncthreads();
    HKV_UTRACE(3);
    // Each warp takes blocks of stage_rows rows and stages 64 bytes of every
    // candidate row at a time in the (now free) ring area with 16-byte async
    // copies, the next piece on its way while lane l sums row l's in the fixed
    // order of channels.
    const int warp = tid >> 5, lane = tid & 31;
    const int SR = u.stage_rows;
    constexpr int NCH = RB / kChunk, PPC = kChunk / 16;  // pieces of a row, 16-byte columns of one
    static_assert(RB % kChunk == 0, "whole pieces");
    unsigned char *stage = u.ring + (size_t)warp * stage_bytes_of(SR);
    const int blocks = (sg.len + SR - 1) / SR;
    const int mine = blocks > warp ? (blocks - warp + NT / 32 - 1) / (NT / 32) : 0;
    auto issue = [&](int step) {
      const int base = (warp + step / NCH * (NT / 32)) * SR;
      unsigned char *dst = stage + (step & 1) * SR * kChunkStride;
      const unsigned char *src = sg.sk + (size_t)base * RB + (step % NCH) * kChunk;
#pragma unroll 4
      for (int w = lane; w < SR * PPC; w += 32) {
        const int rr = w / PPC, pc = w % PPC;
        if (base + rr < sg.len && u.aux[base + rr] >= 0)
          cp_async16(dst + rr * kChunkStride + pc * 16, src + (size_t)rr * RB + pc * 16);
      }
    };
    if (mine > 0) issue(0);
    cp_async_commit();
    float s = 0.f;
    for (int step = 0; step < mine * NCH; ++step) {
      if (step + 1 < mine * NCH) issue(step + 1);
      cp_async_commit();
      cp_async_wait<1>();
      __syncwarp();
      const int r = (warp + step / NCH * (NT / 32)) * SR + lane;
      if (lane < SR && r < sg.len && u.aux[r] >= 0) {
        if (step % NCH == 0) s = 0.f;
        const unsigned char *krow = stage + (step & 1) * SR * kChunkStride + lane * kChunkStride;
        const float *qb = u.qbar + (step % NCH) * PPC * EPL;
#pragma unroll
        for (int pc = 0; pc < PPC; ++pc) {
          float kf[EPL];
          Elem<T>::unpack(*reinterpret_cast<const uint4 *>(krow + pc * 16), kf);
#pragma unroll
          for (int e = 0; e < EPL; ++e) s = __fadd_rn(s, __fmul_rn(qb[pc * EPL + e], kf[e]));
        }
        if (step % NCH == NCH - 1) {
          const float z = __fadd_rn(s, 0.f);  // -0 reads as +0
          const uint32_t bits = __float_as_uint(z);
          u.kh[r] = (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);  // order-preserving
        }
      }
      __syncwarp();  // the stage is rewritten by the next piece but one
    }
    __syncthreads();
    HKV_UTRACE(4);
    // M/2 from each subset; a short subset hands its excess to the other
    int m_long = M / 2, m_near = M - M / 2;
    if (m_long > n_long) {
      m_near += m_long - n_long;
      m_long = n_long;
    }
    if (m_near > NH - n_long) {
      m_long += m_near - (NH - n_long);
      m_near = NH - n_long;
    }
    radix_select2<NT, true>(u.kh, u.ps, u.aux, sg.len, m_long, m_near, 56, u.hist, sh);
    const unsigned long long thr0 = sh.prefix[0], thr1 = sh.prefix[1];
    for (int r = tid; r < sg.len; r += NT) {
      const int c = u.aux[r];
      const bool ev = c == 0 ? (m_long > 0 && key_of(r) <= thr0)
                             : c == 1 ? (m_near > 0 && key_of(r) <= thr1) : false;
      u.aux[r] = ev ? 0 : 1;
    }
    HKV_UTRACE(5);
  } else {
    if (early) {  // fetched for nothing: it must have landed before the CTA ends
      __syncthreads();
      if (!mbar_wait(&sh.ring_bar, 0) && tid == 0) set_err(sg.err, HKV_ERR_TIMEOUT);
    }
    for (int r = tid; r < sg.len; r += NT) u.aux[r] = (u.aux[r] == 0 && M > 0) ? 0 : 1;
  }
  __syncthreads();
  return M;
}

// In place: the new length is len - M; every evicted row below it takes a
// surviving row from above it (the i-th hole the i-th survivor). Sources
// are all >= new_len and destinations < new_len, so the moves are
// independent. Each thread ranks a contiguous run of rows (one block scan
// for holes and fills together), and each copy batch issues all of its
// loads before its stores. Returns the new length.
template <int NT, int D, typename T>
__device__ int fill_holes(const SegRef &sg, int M, const UpdSmem &u, UpdShared &sh) {
  constexpr int RB = D * (int)sizeof(T);
  constexpr int LPR = RB / 16;
  constexpr int B = 4;  // pieces per thread in flight
  const int tid = threadIdx.x;
  const int len = sg.len, new_len = len - M;
  if (M == 0) return len;
  // the key and stage areas are free now and hold the two index lists
  int *hole = reinterpret_cast<int *>(u.kh);    // [M]
  int *fill = reinterpret_cast<int *>(u.ring);  // [M]
  const int per = (len + NT - 1) / NT;
  const int r0 = tid * per < len ? tid * per : len;
  const int r1 = r0 + per < len ? r0 + per : len;
  long long nh = 0, nf = 0;
  for (int r = r0; r < r1; ++r) {
    const int keep = u.aux[r];
    nh += (r < new_len && !keep) ? 1 : 0;
    nf += (r >= new_len && keep) ? 1 : 0;
  }
  long long tot;
  const long long ex = block_excl_scan<long long>((nh << 32) | nf, sh.lscan, &tot);
  int hp = (int)(ex >> 32), fp = (int)(ex & 0xFFFFFFFFll);
  for (int r = r0; r < r1; ++r) {
    const int keep = u.aux[r];
    if (r < new_len && !keep) hole[hp++] = r;
    if (r >= new_len && keep) fill[fp++] = r;
  }
  __syncthreads();
  const int k = (int)(tot >> 32);  // = M: holes and fills pair up
  const int total = k * LPR;
  for (int w0 = 0; w0 < total; w0 += NT * B) {
    uint4 kb[B], vb[B];
#pragma unroll
    for (int j = 0; j < B; ++j) {
      const int w = w0 + j * NT + tid;
      if (w < total) {
        const size_t src = (size_t)fill[w / LPR] * RB + (w % LPR) * 16;
        kb[j] = __ldcg(reinterpret_cast<const uint4 *>(sg.sk + src));
        vb[j] = __ldcg(reinterpret_cast<const uint4 *>(sg.sv + src));
      }
    }
#pragma unroll
    for (int j = 0; j < B; ++j) {
      const int w = w0 + j * NT + tid;
      if (w < total) {
        const size_t dst = (size_t)hole[w / LPR] * RB + (w % LPR) * 16;
        *reinterpret_cast<uint4 *>(sg.dk + dst) = kb[j];
        *reinterpret_cast<uint4 *>(sg.dv + dst) = vb[j];
      }
    }
  }
  for (int j = tid; j < k; j += NT) sg.dpos[hole[j]] = u.ps[fill[j]];
  __syncthreads();
  return new_len;
}

// Out of place, keeping the source order: survivors are packed by a prefix
// sum of the keep flags. Returns the new length.
template <int NT, int D, typename T>
__device__ int copy_kept(const SegRef &sg, const UpdSmem &u, UpdShared &sh) {
  constexpr int RB = D * (int)sizeof(T);
  constexpr int LPR = RB / 16;
  const int tid = threadIdx.x;
  int run = 0;
  for (int base = 0; base < sg.len; base += NT) {
    const int r = base + tid;
    const int keep = r < sg.len ? u.aux[r] : 0;
    int tot;
    const int ex = block_excl_scan<int>(keep, sh.iscan, &tot);
    if (r < sg.len) u.aux[r] = keep ? run + ex : -1;
    run += tot;
  }
  __syncthreads();
  // each batch issues all of its loads before its stores
  constexpr int B = 4;
  for (int w0 = 0; w0 < sg.len * LPR; w0 += NT * B) {
    uint4 kb[B], vb[B];
    int d[B];
#pragma unroll
    for (int x = 0; x < B; ++x) {
      const int w = w0 + x * NT + tid;
      d[x] = w < sg.len * LPR ? u.aux[w / LPR] : -1;
      if (d[x] >= 0) {
        kb[x] = __ldcg(reinterpret_cast<const uint4 *>(sg.sk + (size_t)w * 16));
        vb[x] = __ldcg(reinterpret_cast<const uint4 *>(sg.sv + (size_t)w * 16));
      }
    }
#pragma unroll
    for (int x = 0; x < B; ++x)
      if (d[x] >= 0) {
        const size_t at = (size_t)d[x] * RB + (w0 + x * NT + tid) % LPR * 16;
        *reinterpret_cast<uint4 *>(sg.dk + at) = kb[x];
        *reinterpret_cast<uint4 *>(sg.dv + at) = vb[x];
      }
  }
  for (int r = tid; r < sg.len; r += NT)
    if (u.aux[r] >= 0) sg.dpos[u.aux[r]] = u.ps[r];
  __syncthreads();
  return run;
}

// The update of one head in place (local: window slide; global: STE).
template <int NT, int D, typename T>
__device__ int update_in_place(const SegRef &sg, int label, const MethodArgs &m,
                               const unsigned char *qring, int ntok, const UpdSmem &u,
                               UpdShared &sh) {
  const int M = select_evictions<NT, D, T>(sg, label, m, qring, ntok, u, sh);
  return fill_holes<NT, D, T>(sg, M, u, sh);
}

template <int NT, int D, typename T>
__global__ void __launch_bounds__(NT, upd_ctas(NT))
    evict_kernel(const CacheArgs c, const MethodArgs m, int layer_base, int max_len) {
  constexpr int RB = D * (int)sizeof(T);
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ UpdShared sh;
  // no early launch of the next kernel: a decode step that prefetches this
  // layer's cache before its own wait must start after the update is done
  pdl_wait();
  const int tid = threadIdx.x, i = layer_base + blockIdx.x;
  const uint8_t lab = c.label[i];
  const int nbuf = c.nbuf[i];
  if (lab == HKV_DENSE || nbuf < m.P) return;  // not due
  const int len = c.len[i], cp = c.cap[i];
  const long long off = c.off[i];
  if (off < 0 || cp < 0 || off + cp > c.arena_tokens || len < 0 || len > cp) {
    if (tid == 0) set_err(c.err, HKV_ERR_BOUNDS);
    return;
  }
  if (len > max_len) {
    if (tid == 0) set_err(c.err, HKV_ERR_CAPACITY);
    return;
  }
  unsigned char *K = static_cast<unsigned char *>(c.K) + off * RB;
  unsigned char *V = static_cast<unsigned char *>(c.V) + off * RB;
  int32_t *pos = c.pos + off;
  const unsigned char *qring = static_cast<const unsigned char *>(c.qbuf) + (size_t)i * m.P * RB;
  SegRef sg{K, V, pos, K, V, pos, len, cp, true, c.err};
  HKV_UTRACE(0);
  const int nl =
      update_in_place<NT, D, T>(sg, lab, m, qring, c.ntok[i],
                                carve<NT>(dyn, max_len, D, m.P, (int)sizeof(T)), sh);
  HKV_UTRACE(6);
  if (tid == 0) {
    c.len[i] = nl;
    c.nbuf[i] = 0;
  }
}

template <int NT, int D, typename T>
__global__ void __launch_bounds__(NT, upd_ctas(NT))
    append_evict_kernel(const CacheArgs c, const MethodArgs m, int layer_base, const void *q,
                        const void *k, const void *v, int max_len) {
  constexpr int RB = D * (int)sizeof(T);
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ UpdShared sh;
  pdl_wait();
  pdl_launch_dependents();
  const int tid = threadIdx.x, hl = blockIdx.x, i = layer_base + hl;
  int len = c.len[i];
  const int cp = c.cap[i];
  const long long off = c.off[i];
  const uint8_t lab = c.label[i];
  const int ntok = c.ntok[i];
  int nbuf = c.nbuf[i];
  if (off < 0 || cp < 0 || off + cp > c.arena_tokens || len < 0 || len > cp) {
    if (tid == 0) set_err(c.err, HKV_ERR_BOUNDS);
    return;
  }
  unsigned char *K = static_cast<unsigned char *>(c.K) + off * RB;
  unsigned char *V = static_cast<unsigned char *>(c.V) + off * RB;
  int32_t *pos = c.pos + off;
  const unsigned char *qring = static_cast<const unsigned char *>(c.qbuf) + (size_t)i * m.P * RB;

  if (lab != HKV_DENSE && nbuf >= m.P) {  // buffer full: head-aware update
    if (len > max_len) {
      if (tid == 0) set_err(c.err, HKV_ERR_CAPACITY);
      return;
    }
    SegRef sg{K, V, pos, K, V, pos, len, cp, true, c.err};
    len = update_in_place<NT, D, T>(sg, lab, m, qring, ntok,
                                    carve<NT>(dyn, max_len, D, m.P, (int)sizeof(T)), sh);
    nbuf = 0;
  }
  if (len >= cp) {
    if (tid == 0) {
      set_err(c.err, HKV_ERR_CAPACITY);
      c.len[i] = len;
      c.nbuf[i] = nbuf;
    }
    return;
  }
  // append the new token (K <- [K, k_t], V <- [V, v_t]) and its query
  const size_t row = (size_t)len;
  unsigned char *qdst = static_cast<unsigned char *>(c.qbuf) + ((size_t)i * m.P + ntok % m.P) * RB;
  for (int pc = tid; pc < RB / 16; pc += NT) {
    const size_t src = (size_t)hl * RB + pc * 16;
    *reinterpret_cast<uint4 *>(K + row * RB + pc * 16) =
        *reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(k) + src);
    *reinterpret_cast<uint4 *>(V + row * RB + pc * 16) =
        *reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(v) + src);
    *reinterpret_cast<uint4 *>(qdst + pc * 16) =
        *reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(q) + src);
  }
  if (tid == 0) {
    pos[row] = m.C + ntok;
    c.len[i] = len + 1;
    c.ntok[i] = ntok + 1;
    if (lab != HKV_DENSE) c.nbuf[i] = nbuf + 1;
  }
}

template <int NT, int D, typename T>
__global__ void __launch_bounds__(NT, upd_ctas(NT))
    repack_kernel(const CacheArgs dn, const CacheArgs rg, const MethodArgs m, int layer_base,
                  int max_len) {
  constexpr int RB = D * (int)sizeof(T);
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ UpdShared sh;
  // no early launch of the next kernel (as in evict_kernel): this one writes
  // every layer's cache, which a prefetching decode step reads before its wait
  pdl_wait();
  const int tid = threadIdx.x, i = layer_base + blockIdx.x;
  const int slen = dn.len[i];
  const long long soff = dn.off[i];
  const long long doff = rg.off[i];
  const int dcap = rg.cap[i];
  const uint8_t lab = rg.label[i];
  if (lab != HKV_LOCAL && lab != HKV_GLOBAL) {
    if (tid == 0) set_err(rg.err, HKV_ERR_STATE);
    return;
  }
  if (soff < 0 || slen < 0 || soff + slen > dn.arena_tokens || doff < 0 || dcap < 0 ||
      doff + dcap > rg.arena_tokens) {
    if (tid == 0) set_err(rg.err, HKV_ERR_BOUNDS);
    return;
  }
  if (slen > max_len) {
    if (tid == 0) set_err(rg.err, HKV_ERR_CAPACITY);
    return;
  }
  SegRef sg{static_cast<const unsigned char *>(dn.K) + soff * RB,
            static_cast<const unsigned char *>(dn.V) + soff * RB,
            dn.pos + soff,
            static_cast<unsigned char *>(rg.K) + doff * RB,
            static_cast<unsigned char *>(rg.V) + doff * RB,
            rg.pos + doff,
            slen,
            dcap,
            false,
            rg.err};
  const unsigned char *qring = static_cast<const unsigned char *>(dn.qbuf) + (size_t)i * m.P * RB;
  const UpdSmem u = carve<NT>(dyn, max_len, D, m.P, (int)sizeof(T));
  const int M = select_evictions<NT, D, T>(sg, lab, m, qring, dn.ntok[i], u, sh);
  if (slen - M > dcap) {
    if (tid == 0) set_err(rg.err, HKV_ERR_CAPACITY);
    return;
  }
  const int nl = copy_kept<NT, D, T>(sg, u, sh);
  if (tid == 0) {
    rg.len[i] = nl;
    rg.nbuf[i] = 0;
    rg.ntok[i] = dn.ntok[i];
  }
}

// One CTA per head, with enough threads that a prompt of 128 tokens is one
// round of loads and one of stores (each batch issues its loads first): a
// plain copy, bound by the loads in flight. 128 threads that copied 16 bytes
// of K and V at a time took 20 us for 256 heads of 128 tokens, which 5 us of
// bandwidth move.
constexpr int kPrefillBatch = 4;  // 16-byte pieces of K and of V per thread and batch

template <int D, typename T>
__global__ void __launch_bounds__(512)
    prefill_kernel(const CacheArgs c, int layer_base, int C, const void *kc, const void *vc) {
  constexpr int RB = D * (int)sizeof(T);
  // no early launch of the next kernel: a decode step of this layer may be it,
  // and prefetch (48 layers of 256 heads of 128 tokens: 235 us with, 234 without)
  pdl_wait();
  const int hl = blockIdx.x, i = layer_base + hl, tid = threadIdx.x;
  const long long off = c.off[i];
  const int cp = c.cap[i];
  const bool fresh = c.label[i] == HKV_DENSE && c.len[i] == 0;
  __syncthreads();  // every thread has read len before the first one sets it
  if (!fresh) {
    if (tid == 0) set_err(c.err, HKV_ERR_STATE);
    return;
  }
  if (off < 0 || cp < C || off + cp > c.arena_tokens) {
    if (tid == 0) set_err(c.err, cp < C ? HKV_ERR_CAPACITY : HKV_ERR_BOUNDS);
    return;
  }
  const int pieces = C * (RB / 16);
  const size_t src = (size_t)hl * C * RB;
  const uint4 *sk = reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(kc) + src);
  const uint4 *sv = reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(vc) + src);
  uint4 *dk = reinterpret_cast<uint4 *>(static_cast<unsigned char *>(c.K) + (size_t)off * RB);
  uint4 *dv = reinterpret_cast<uint4 *>(static_cast<unsigned char *>(c.V) + (size_t)off * RB);
  for (int p0 = 0; p0 < pieces; p0 += blockDim.x * kPrefillBatch) {
    uint4 kb[kPrefillBatch], vb[kPrefillBatch];
#pragma unroll
    for (int x = 0; x < kPrefillBatch; ++x) {
      const int pc = p0 + x * blockDim.x + tid;
      if (pc < pieces) {
        kb[x] = sk[pc];
        vb[x] = sv[pc];
      }
    }
#pragma unroll
    for (int x = 0; x < kPrefillBatch; ++x) {
      const int pc = p0 + x * blockDim.x + tid;
      if (pc < pieces) {
        dk[pc] = kb[x];
        dv[pc] = vb[x];
      }
    }
  }
  for (int j = tid; j < C; j += blockDim.x) c.pos[off + j] = j;
  if (tid == 0) {
    c.len[i] = C;
    c.nbuf[i] = 0;
    c.ntok[i] = 0;
  }
}

__global__ void init_dense_kernel(const CacheArgs c, int n, int seg) {
  pdl_wait();  // and no early launch: every layer's counters are written here
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const_cast<int64_t *>(c.off)[i] = (int64_t)i * seg;
    const_cast<int32_t *>(c.cap)[i] = seg;
    c.len[i] = 0;
    c.nbuf[i] = 0;
    c.ntok[i] = 0;
    const_cast<uint8_t *>(c.label)[i] = HKV_DENSE;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *c.err = 0u;
}

// Row steps of the identification kernels' logit loops whose key loads are
// issued before the first is used (one step at a time costs a memory round
// trip per step). Measured on a GB300 (one call per layer): dense segments
// of 628 tokens or more go faster with 8 (single query; 26 -> 14 us per
// layer at 628) or 4 (multi-query: -19 % at 628, -35 % at 2128 tokens) than
// with one; segments of 101-164 tokens go best with 2, where more loads in
// flight cost registers and resident CTAs.
constexpr int kIdLongSegment = 512;
// stages of the single-query kernel's keys for such segments
constexpr int kIdStageBytes = 32768, kIdStages = 3;
__host__ __device__ constexpr int id_rows_in_flight(int max_len, bool multi) {
  return max_len >= kIdLongSegment ? (multi ? 4 : 8) : 2;
}

// Shared memory of the identification kernels beyond their weights: in the
// grid-distance variant, the order keys ([max_len] 64-bit, 8-byte aligned
// after `floats` floats) and the count order ([max_len] int).
__host__ __device__ constexpr size_t id_order_offset(size_t floats) {
  return (floats * 4 + 7) / 8 * 8;
}
__host__ __device__ constexpr size_t id_smem(size_t floats, int max_len, bool grid2d) {
  return grid2d ? id_order_offset(floats) + (size_t)max_len * 12 : floats * 4;
}
__host__ __device__ constexpr size_t id_stage_at(size_t smem) { return (smem + 127) / 128 * 128; }
// dynamic, beside the kernels' static part: of one CTA of an SM, of two
constexpr size_t kIdMostSmem = 226 * 1024, kIdTwoSmem = 112 * 1024;

// The count order of the grid-distance variant of Step 2: perm[j] = the row
// of the j-th token counted. Image tokens by squared grid distance from image
// token ref, nearest first, equal distances newer first; then the
// conditioning tokens, newest first. Keys are unique (positions are); each
// row's rank is the number of smaller keys (len^2 / IT comparisons per
// thread, once per head and generation). Block-uniform.
__device__ void grid_count_order(const int32_t *pos, int len, int C, int row_len, int ref,
                                 unsigned long long *keys, int *perm) {
  for (int r = threadIdx.x; r < len; r += blockDim.x) {
    const int p = pos[r];
    const unsigned long long newer = 0xFFFFFFFFull - (uint32_t)p;
    unsigned long long key = (1ull << 63) | newer;  // conditioning: after every image token
    if (p >= C) {
      const int i = p - C;
      const long long dr = i / row_len - ref / row_len, dc = i % row_len - ref % row_len;
      key = ((unsigned long long)(dr * dr + dc * dc) << 32) | newer;
    }
    keys[r] = key;
    perm[r] = r;  // a valid row for every slot even if positions repeat
  }
  __syncthreads();
  for (int r = threadIdx.x; r < len; r += blockDim.x) {
    const unsigned long long k = keys[r];
    int rank = 0;
    for (int j = 0; j < len; ++j) rank += keys[j] < k ? 1 : 0;
    perm[rank] = r;
  }
  __syncthreads();
}

// Step 2: attention of the current query over the key cache, accumulated
// backward from the newest token until tau (or outward on the grid in the
// grid-distance variant); local iff fewer than w_loc tokens were needed.
// The dense cache holds its tokens in position order.
// One CTA per head, one and a half on an SM for 256 heads: beside the keys'
// bytes it is a chain of phases, so each phase is one block barrier: every
// warp combines the warps' maxima, sums and scan totals itself, in the order
// in which one warp did (the counts depend on it). 256 heads of 628 tokens
// (6.1 us at the measured bandwidth): 12.1 us; with those barriers 11.8, with
// the staged keys below 10.4 (512 threads without them 12.3).
//
// Two things go by the instantiation, with the same results. Short segments
// keep the block scan, which leaves the compiler a faster loop over the rows
// than the scan within the warps: LlamaGen-XL, 2560 heads of 110 tokens, 12.3
// us, 14.1 with the latter. The query is loaded beside the lengths, but after
// the checks where bf16 rows of 256 bytes are loaded straight (kLateQ):
// Lumina-mGPT 768, 256 heads of 428 tokens, 13.5 us, 17.3 when it is early;
// rows of 128 bytes and fp32 the other way round (14.0 early, 14.9 late;
// Janus-Pro-7B in fp32, 16 sequences, 10.2 and 10.6).
//
// The logits: short segments (STAGED = false) load U row steps at a time into
// registers; longer ones come through kIdStages stages of 32 KB filled by
// bulk copies, so that a head's keys are on their way before the first
// product, and a warp takes eight row steps of a stage at once: pairs of rows
// share FMAs, and the eight sums are exchanged by halves (8 shuffles instead
// of 32). Products and sums are the same operations in the same order.
template <int D, typename T, int U, bool STAGED>
__global__ void __launch_bounds__(IT)
    identify_kernel(const CacheArgs c, const MethodArgs m, int layer_base, const void *q,
                    uint8_t *label_out, int32_t *nh_out, float qscale, int max_len,
                    int stage_at) {
  constexpr int RB = D * (int)sizeof(T);
  constexpr int EPL = Elem<T>::kPerPiece;
  constexpr int LPR = RB / 16;
  constexpr int RPW = 32 / LPR;
  constexpr int NW = IT / 32;
  constexpr bool kLateQ = !STAGED && sizeof(T) == 2 && D == 128;
  extern __shared__ float e[];
  __shared__ __align__(16) float s_max[NW], s_sum[NW];
  __shared__ float s_tot[2][NW], s_scan[33];
  __shared__ int s_nh;
  __shared__ uint64_t s_full[kIdStages], s_empty[kIdStages];
  pdl_wait();
  pdl_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int hl = blockIdx.x, i = layer_base + hl;
  const int grp = lane / LPR, col = lane % LPR;
  auto load_q = [&]() {
    return *reinterpret_cast<const uint4 *>(static_cast<const unsigned char *>(q) +
                                            (size_t)hl * RB + col * 16);
  };
  uint4 qraw;
  if (!kLateQ) qraw = load_q();
  const int len = c.len[i];
  const long long off = c.off[i];
  if (tid == 0) s_nh = len;
  if (c.label[i] != HKV_DENSE) {  // only the uncompressed cache is in order
    if (tid == 0) set_err(c.err, HKV_ERR_STATE);
    return;
  }
  if (off < 0 || len <= 0 || off + len > c.arena_tokens) {
    if (tid == 0) set_err(c.err, HKV_ERR_BOUNDS);
    return;
  }
  if (len > max_len) {  // the attention row must fit in shared memory
    if (tid == 0) set_err(c.err, HKV_ERR_CAPACITY);
    return;
  }
  if (kLateQ) qraw = load_q();
  float qf[EPL];
  Elem<T>::unpack(qraw, qf);
#pragma unroll
  for (int x = 0; x < EPL; ++x) qf[x] *= qscale;
  const unsigned char *K = static_cast<const unsigned char *>(c.K) + off * RB;
  // logits (log2 units)
  float mx = -INFINITY;
  if constexpr (STAGED) {
    constexpr int ROWS = kIdStageBytes / RB;  // of a stage: eight row steps of every warp
    static_assert(ROWS == 8 * NW * RPW, "a stage is eight row steps");
    unsigned char *stage = reinterpret_cast<unsigned char *>(e) + stage_at;
    const int fills = (len + ROWS - 1) / ROWS;
    auto fill = [&](int f) {  // thread 0
      const int rows = len - f * ROWS < ROWS ? len - f * ROWS : ROWS;
      const uint32_t bytes = (uint32_t)rows * RB;
      mbar_arrive_expect_tx(&s_full[f % kIdStages], bytes);
      bulk_g2s(stage + (f % kIdStages) * kIdStageBytes, K + (size_t)f * ROWS * RB, bytes,
               &s_full[f % kIdStages]);
    };
    if (tid == 0) {
      for (int x = 0; x < kIdStages; ++x) {
        mbar_init(&s_full[x], 1);
        mbar_init(&s_empty[x], NW);
      }
      fence_barrier_init();
      for (int f = 0; f < fills && f < kIdStages; ++f) fill(f);
    }
    __syncthreads();
    float2 q2[EPL];
#pragma unroll
    for (int x = 0; x < EPL; ++x) q2[x] = make_float2(qf[x], qf[x]);
#pragma unroll 1
    for (int f = 0; f < fills; ++f) {
      const int sg = f % kIdStages;
      if (!mbar_wait(&s_full[sg], (uint32_t)(f / kIdStages) & 1u) && tid == 0)
        set_err(c.err, HKV_ERR_TIMEOUT);
      const unsigned char *src = stage + sg * kIdStageBytes + (warp * RPW + grp) * RB + col * 16;
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        float ka[EPL], kb[EPL];
        Elem<T>::unpack(*reinterpret_cast<const uint4 *>(src + u * NW * RPW * RB), ka);
        Elem<T>::unpack(*reinterpret_cast<const uint4 *>(src + (u + 1) * NW * RPW * RB), kb);
        float2 dot = make_float2(0.f, 0.f);
#pragma unroll
        for (int x = 0; x < EPL; ++x) dot = __ffma2_rn(q2[x], make_float2(ka[x], kb[x]), dot);
        v[u] = dot.x;
        v[u + 1] = dot.y;
      }
      __syncwarp();
      mbar_arrive_if(&s_empty[sg], lane == 0);
      // the sum over a row's lanes: halves of the values change hands at the
      // first three levels, so lane bits choose the row step that is left
      int step = 0;
      int o = LPR / 2;
#pragma unroll
      for (int n = 4; n >= 1; n >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int x = 0; x < n; ++x) {
          const float give = up ? v[x] : v[x + n], keep = up ? v[x + n] : v[x];
          v[x] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
        }
        step += up ? n : 0;
      }
#pragma unroll
      for (int l = LPR / 16; l >= 1; l >>= 1)
        v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], l);
      const int r = f * ROWS + step * NW * RPW + warp * RPW + grp;
      if (r < len) e[r] = v[0];  // (the lanes that share a row step store the same value)
      if (tid == 0 && f + kIdStages < fills) {
        if (!mbar_wait(&s_empty[sg], (uint32_t)(f / kIdStages) & 1u))
          set_err(c.err, HKV_ERR_TIMEOUT);
        fill(f + kIdStages);
      }
    }
  } else {
    // U row steps load before any is used
    for (int r0 = warp * RPW; r0 < len; r0 += U * NW * RPW) {
      uint4 kr[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int r = r0 + u * NW * RPW + grp;
        kr[u] = r < len ? *reinterpret_cast<const uint4 *>(K + (size_t)r * RB + col * 16)
                        : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int r = r0 + u * NW * RPW + grp;
        float kf[EPL];
        Elem<T>::unpack(kr[u], kf);
        float dot = 0.f;
#pragma unroll
        for (int x = 0; x < EPL; ++x) dot = fmaf(qf[x], kf[x], dot);
#pragma unroll
        for (int o = LPR / 2; o >= 1; o >>= 1) dot += __shfl_xor_sync(0xFFFFFFFFu, dot, o);
        if (r < len && col == 0) e[r] = dot;
      }
    }
  }
  __syncthreads();
  for (int r = tid; r < len; r += IT) mx = fmaxf(mx, e[r]);
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
  if (lane == 0) s_max[warp] = mx;
  __syncthreads();
  float all[NW];
#pragma unroll
  for (int w = 0; w < NW; w += 4)
    *reinterpret_cast<float4 *>(all + w) = *reinterpret_cast<const float4 *>(s_max + w);
#pragma unroll
  for (int w = 0; w < NW; ++w) mx = fmaxf(mx, all[w]);
  float sum = 0.f;
  for (int r = tid; r < len; r += IT) {
    const float x = exp2f(e[r] - mx);
    e[r] = x;
    sum += x;
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
  if (lane == 0) s_sum[warp] = sum;
  __syncthreads();
  float thr = 0.f;
#pragma unroll
  for (int w = 0; w < NW; w += 4)
    *reinterpret_cast<float4 *>(all + w) = *reinterpret_cast<const float4 *>(s_sum + w);
#pragma unroll
  for (int w = 0; w < NW; ++w) thr += all[w];
  thr *= m.tau;
  int *perm = nullptr;
  if (m.grid2d) {
    unsigned char *base = reinterpret_cast<unsigned char *>(e) + id_order_offset(max_len);
    perm = reinterpret_cast<int *>(base + (size_t)max_len * 8);
    grid_count_order(c.pos + off, len, m.C, m.row_len, c.ntok[i] - 1,
                     reinterpret_cast<unsigned long long *>(base), perm);
  }
  float running = 0.f;  // cumulative mass from the newest token
#pragma unroll 1
  for (int base = 0, half = 0; base < len; base += IT, half ^= 1) {
    const int jb = base + tid;  // jb-th token counted (0 = current)
    const float x = jb < len ? e[perm ? perm[jb] : len - 1 - jb] : 0.f;
    float before, tot;  // the masses before x and of the round
    if constexpr (STAGED) {
      const float incl = warp_incl_scan(x);
      if (lane == 31) s_tot[half][warp] = incl;
      __syncthreads();
      const float wv = lane < NW ? s_tot[half][lane] : 0.f;
      float wi = wv;
#pragma unroll
      for (int o = 1; o < NW; o <<= 1) {
        const float y = __shfl_up_sync(0xFFFFFFFFu, wi, o);
        if (lane >= o) wi += y;
      }
      before = __shfl_sync(0xFFFFFFFFu, wi - wv, warp) + incl - x;
      tot = __shfl_sync(0xFFFFFFFFu, wi, NW - 1);
    } else {
      before = block_excl_scan<float>(x, s_scan, &tot);
    }
    const float cum = running + before + x;
    if (jb < len && cum >= thr) atomicMin(&s_nh, jb + 1);
    running += tot;
  }
  __syncthreads();
  if (tid == 0) {
    label_out[i] = s_nh < m.w_loc ? HKV_LOCAL : HKV_GLOBAL;
    if (nh_out) nh_out[i] = s_nh;
  }
}

// Block-wide max (MAX) or sum of N floats per thread, returned to every
// thread in place; red holds N values per warp, bc the N results.
// Consecutive calls are safe: each reads its operands before the next call
// writes them.
template <bool MAX, int N>
__device__ __forceinline__ void block_all(float (&v)[N], float *red, float *bc) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int b = 0; b < N; ++b) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      const float u = __shfl_xor_sync(0xFFFFFFFFu, v[b], o);
      v[b] = MAX ? fmaxf(v[b], u) : v[b] + u;
    }
    if (lane == 0) red[b * nw + warp] = v[b];
  }
  __syncthreads();
  if (threadIdx.x < N) {
    const int b = threadIdx.x;
    float a = red[b * nw];
    for (int w = 1; w < nw; ++w) a = MAX ? fmaxf(a, red[b * nw + w]) : a + red[b * nw + w];
    bc[b] = a;
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < N; ++b) v[b] = bc[b];
}

// queries of the multi-query identification handled per pass over the keys:
// 8 for rings of at least kIdQB8From queries, else 4 (measured on a GB300:
// 8 is 17 % faster on 65-query rings over 628 keys, 4 is 26-33 % faster on
// 24-query rings over 101-164 keys, where the fewer registers of 4 give
// more CTAs per SM)
#ifndef HKV_ID_QB8_FROM
#define HKV_ID_QB8_FROM 48
#endif
constexpr int kIdQB8From = HKV_ID_QB8_FROM;
__host__ __device__ constexpr int id_qb(int P) { return P >= kIdQB8From ? 8 : 4; }

// Multi-query variant of Step 2 (not in the paper): the newest Pe = min(P,
// ntok) queries of the ring each attend over the keys that existed at their
// own step (the p-th oldest of them over the oldest len - (Pe - 1 - p)
// keys), their normalised attention rows are averaged, and the average is
// accumulated backward from the newest token until tau, as in
// identify_kernel. One CTA per head; each pass over the keys serves QB
// queries (every key row loaded once per pass, dotted with all of them).
template <int D, typename T, int QB, int U>
__global__ void __launch_bounds__(IT)
    identify_multi_kernel(const CacheArgs c, const MethodArgs m, int layer_base,
                          uint8_t *label_out, int32_t *nh_out, float qscale, int max_len) {
  constexpr int RB = D * (int)sizeof(T);
  constexpr int EPL = Elem<T>::kPerPiece;
  constexpr int LPR = RB / 16;
  constexpr int RPW = 32 / LPR;
  constexpr int NW = IT / 32;
  extern __shared__ float e[];      // [QB][max_len] the pass's logits, then weights
  float *pbar = e + QB * max_len;  // [max_len] summed weights of all queries
  __shared__ float red[QB * NW];
  __shared__ float s_b[QB];
  __shared__ float fscan[33];
  __shared__ int s_nh;
  pdl_wait();
  pdl_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int hl = blockIdx.x, i = layer_base + hl;
  const int len = c.len[i];
  const int ntok = c.ntok[i];
  const long long off = c.off[i];
  if (c.label[i] != HKV_DENSE || ntok <= 0) {  // in position order, with buffered queries
    if (tid == 0) set_err(c.err, HKV_ERR_STATE);
    return;
  }
  if (off < 0 || len <= 0 || off + len > c.arena_tokens) {
    if (tid == 0) set_err(c.err, HKV_ERR_BOUNDS);
    return;
  }
  if (len > max_len) {
    if (tid == 0) set_err(c.err, HKV_ERR_CAPACITY);
    return;
  }
  const int Pe = min(m.P, min(ntok, len));
  const int grp = lane / LPR, col = lane % LPR;
  const unsigned char *K = static_cast<const unsigned char *>(c.K) + off * RB;
  const unsigned char *ring = static_cast<const unsigned char *>(c.qbuf) + (size_t)i * m.P * RB;
  for (int r = tid; r < len; r += IT) pbar[r] = 0.f;
  for (int p0 = 0; p0 < Pe; p0 += QB) {
    // query p0 + b sees mq[b] keys (0 past the newest query)
    int mq[QB];
    float qf[QB][EPL];
#pragma unroll
    for (int b = 0; b < QB; ++b) {
      const int p = p0 + b;
      mq[b] = p < Pe ? len - (Pe - 1 - p) : 0;
#pragma unroll
      for (int x = 0; x < EPL; ++x) qf[b][x] = 0.f;
      if (p < Pe) {
        const int slot = (ntok - Pe + p) % m.P;
        Elem<T>::unpack(*reinterpret_cast<const uint4 *>(ring + (size_t)slot * RB + col * 16),
                        qf[b]);
#pragma unroll
        for (int x = 0; x < EPL; ++x) qf[b][x] *= qscale;
      }
    }
    const int mmax = len - max(0, Pe - 1 - (p0 + QB - 1));  // keys of the pass's newest query
    // logits (log2 units); U row steps load before any is used
    for (int r0 = warp * RPW; r0 < mmax; r0 += U * NW * RPW) {
      uint4 kr[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int r = r0 + u * NW * RPW + grp;
        kr[u] = r < mmax ? *reinterpret_cast<const uint4 *>(K + (size_t)r * RB + col * 16)
                         : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int r = r0 + u * NW * RPW + grp;
        float kf[EPL];
        Elem<T>::unpack(kr[u], kf);
        float dot[QB];
#pragma unroll
        for (int b = 0; b < QB; ++b) {
          dot[b] = 0.f;
#pragma unroll
          for (int x = 0; x < EPL; ++x) dot[b] = fmaf(qf[b][x], kf[x], dot[b]);
        }
#pragma unroll
        for (int b = 0; b < QB; ++b) {
#pragma unroll
          for (int o = LPR / 2; o >= 1; o >>= 1) dot[b] += __shfl_xor_sync(0xFFFFFFFFu, dot[b], o);
          if (col == 0 && r < mq[b]) e[b * max_len + r] = dot[b];
        }
      }
    }
    __syncthreads();
    float acc[QB];
#pragma unroll
    for (int b = 0; b < QB; ++b) acc[b] = -INFINITY;
    for (int r = tid; r < mmax; r += IT)
#pragma unroll
      for (int b = 0; b < QB; ++b)
        if (r < mq[b]) acc[b] = fmaxf(acc[b], e[b * max_len + r]);
    block_all<true, QB>(acc, red, s_b);
    float mx[QB];
#pragma unroll
    for (int b = 0; b < QB; ++b) {
      mx[b] = acc[b];
      acc[b] = 0.f;
    }
    for (int r = tid; r < mmax; r += IT)
#pragma unroll
      for (int b = 0; b < QB; ++b)
        if (r < mq[b]) {
          const float x = exp2f(e[b * max_len + r] - mx[b]);
          e[b * max_len + r] = x;
          acc[b] += x;
        }
    block_all<false, QB>(acc, red, s_b);
#pragma unroll
    for (int b = 0; b < QB; ++b) acc[b] = 1.f / acc[b];  // unused past the newest query
    for (int r = tid; r < mmax; r += IT) {
      float s = pbar[r];
#pragma unroll
      for (int b = 0; b < QB; ++b)
        if (r < mq[b]) s = fmaf(e[b * max_len + r], acc[b], s);
      pbar[r] = s;
    }
    __syncthreads();  // e is rewritten by the next pass
  }
  float tot[1] = {0.f};
  for (int r = tid; r < len; r += IT) tot[0] += pbar[r];
  block_all<false, 1>(tot, red, s_b);
  const float thr = tot[0] * m.tau;
  if (tid == 0) s_nh = len;
  __syncthreads();
  int *perm = nullptr;
  if (m.grid2d) {
    unsigned char *base =
        reinterpret_cast<unsigned char *>(e) + id_order_offset((size_t)(QB + 1) * max_len);
    perm = reinterpret_cast<int *>(base + (size_t)max_len * 8);
    grid_count_order(c.pos + off, len, m.C, m.row_len, ntok - 1,
                     reinterpret_cast<unsigned long long *>(base), perm);
  }
  float running = 0.f;  // cumulative mass from the newest token
  for (int base = 0; base < len; base += IT) {
    const int jb = base + tid;  // jb-th token counted (0 = current)
    const float x = jb < len ? pbar[perm ? perm[jb] : len - 1 - jb] : 0.f;
    float t;
    const float cum = running + block_excl_scan<float>(x, fscan, &t) + x;
    if (jb < len && cum >= thr) atomicMin(&s_nh, jb + 1);
    running += t;
  }
  __syncthreads();
  if (tid == 0) {
    label_out[i] = s_nh < m.w_loc ? HKV_LOCAL : HKV_GLOBAL;
    if (nh_out) nh_out[i] = s_nh;
  }
}

// Sec. 5.1 budgets (group = 0), or the aggregate-preserving variant over
// consecutive groups of `group` heads, one (sequence, layer) each: the
// (group - n_g)(B_g - w) tokens the local heads leave go to the group's n_g
// global heads in equal shares, the remainder one each to the global heads
// of lowest index.
__global__ void budgets_kernel(const uint8_t *label, int32_t *budget, int32_t *cap, int64_t *off,
                               int n, int C, int B_g, int w, int P, int group) {
  __shared__ long long scratch[33];
  pdl_wait();
  pdl_launch_dependents();
  long long running = 0;
  int bad = 0;
  for (int base = 0; base < n; base += blockDim.x) {
    const int i = base + threadIdx.x;
    long long cp = 0;
    if (i < n) {
      const uint8_t lb = label[i];
      int bg = 0;
      if (lb == HKV_GLOBAL) bg = B_g;
      else if (lb == HKV_LOCAL) bg = w;
      else bad = 1;
      if (group > 0 && lb == HKV_GLOBAL) {
        const int g0 = i / group * group;
        int ng = 0, rank = 0;
        for (int j = g0; j < g0 + group && j < n; ++j) {
          const bool gl = label[j] == HKV_GLOBAL;
          ng += gl;
          rank += gl && j < i;
        }
        const long long extra = (long long)(group - ng) * (B_g - w);
        bg += (int)(extra / ng) + (rank < extra % ng ? 1 : 0);
      }
      cp = (long long)C + bg + P;
      budget[i] = bg;
      cap[i] = (int32_t)cp;
    }
    long long tot;
    const long long ex = block_excl_scan<long long>(cp, scratch, &tot);
    if (i < n) off[i] = running + ex;
    running += tot;
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) off[n - 1] = -1;  // reported as a state error
}

// The same without groups, over several CTAs of kBudgetHeads heads each: a
// CTA counts the global heads before its own from the labels (n bytes out of
// L2, at most 1 MB, see launch_budgets), so that none waits for another. One
// CTA looping over blocks of heads took a load and a scan of 1.3 us for every
// 1024 heads.
constexpr int kBudgetHeads = 4096, kBudgetThreads = 256;
constexpr int kBudgetMost = 1 << 20;
__global__ void __launch_bounds__(kBudgetThreads)
    budgets_plain_kernel(const uint8_t *label, int32_t *budget, int32_t *cap, int64_t *off, int n,
                         int C, int B_g, int w, int P) {
  constexpr int NW = kBudgetThreads / 32, PER = kBudgetHeads / NW;
  __shared__ int s_before[NW], s_own[NW];
  pdl_wait();
  pdl_launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int first = blockIdx.x * kBudgetHeads;
  int bad = 0, count = 0;
  auto tally = [&](int i) {
    const int lb = label[i];
    bad |= lb != HKV_GLOBAL && lb != HKV_LOCAL;
    return lb == HKV_GLOBAL ? 1 : 0;
  };
#pragma unroll 16
  for (int i = tid; i < first; i += kBudgetThreads) count += tally(i);
  count = __reduce_add_sync(0xFFFFFFFFu, (unsigned)count);
  const int w0 = first + warp * PER;  // this warp's heads
  int own = 0;
#pragma unroll 16
  for (int i = w0 + lane; i < w0 + PER; i += 32) own += i < n ? tally(i) : 0;
  own = __reduce_add_sync(0xFFFFFFFFu, (unsigned)own);
  if (lane == 0) {
    s_before[warp] = count;
    s_own[warp] = own;
  }
  const bool any_bad = __syncthreads_or(bad);
  int g = 0;  // global heads before this warp's
  for (int x = 0; x < NW; ++x) g += s_before[x] + (x < warp ? s_own[x] : 0);
  const long long cl = (long long)C + w + P, cg = (long long)C + B_g + P;
#pragma unroll 4
  for (int i0 = w0; i0 < w0 + PER && i0 < n; i0 += 32) {
    const int i = i0 + lane;
    const bool gl = i < n && label[i] == HKV_GLOBAL;
    const unsigned m = __ballot_sync(0xFFFFFFFFu, gl);
    if (i < n) {
      const int rank = g + __popc(m & ((1u << lane) - 1u));
      budget[i] = gl ? B_g : w;
      cap[i] = (int32_t)(gl ? cg : cl);
      // (the CTA of the last head has seen every label: a bad one is
      // reported as a state error)
      off[i] = i == n - 1 && any_bad ? -1 : rank * cg + (i - rank) * cl;
    }
    g += __popc(m);
  }
}

}  // namespace

#ifdef HKV_UPD_TRACE
// tracer builds only: where the update's phase timestamps go
extern "C" int hkv_debug_set_utrace(unsigned long long *buf) {
  return cudaMemcpyToSymbol(g_utrace, &buf, sizeof(buf)) == cudaSuccess ? 0 : 7;
}
#endif

namespace {

// all of an SM's L1 as shared memory, so that every head of a layer (one CTA
// each) is resident at once
template <int NT, int D, typename T>
cudaError_t prepare_update_t(size_t smem) {
  const void *kernels[] = {(const void *)append_evict_kernel<NT, D, T>,
                           (const void *)evict_kernel<NT, D, T>,
                           (const void *)repack_kernel<NT, D, T>};
  cudaError_t e = cudaSuccess;
  for (const void *f : kernels) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  }
  return e;
}

template <int D, typename T>
cudaError_t prepare_t(size_t smem) {
  cudaError_t e = prepare_update_t<128, D, T>(smem);
  if (e == cudaSuccess) e = prepare_update_t<256, D, T>(smem);
  if (e == cudaSuccess) e = prepare_update_t<512, D, T>(smem);
  const void *ident[] = {(const void *)identify_kernel<D, T, 2, false>,
                         (const void *)identify_kernel<D, T, 8, false>,
                         (const void *)identify_kernel<D, T, 8, true>,
                         (const void *)identify_multi_kernel<D, T, 4, 2>,
                         (const void *)identify_multi_kernel<D, T, 4, 4>,
                         (const void *)identify_multi_kernel<D, T, 8, 2>,
                         (const void *)identify_multi_kernel<D, T, 8, 4>};
  for (const void *f : ident)
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  return e;
}

#define HKV_DISPATCH(D_, DT_, ...)                  \
  do {                                              \
    if ((DT_) == HKV_BF16) {                        \
      if ((D_) == 64) {                             \
        constexpr int kD = 64;                      \
        using kT = __nv_bfloat16;                   \
        __VA_ARGS__;                                \
      } else {                                      \
        constexpr int kD = 128;                     \
        using kT = __nv_bfloat16;                   \
        __VA_ARGS__;                                \
      }                                             \
    } else {                                        \
      if ((D_) == 64) {                             \
        constexpr int kD = 64;                      \
        using kT = float;                           \
        __VA_ARGS__;                                \
      } else {                                      \
        constexpr int kD = 128;                     \
        using kT = float;                           \
        __VA_ARGS__;                                \
      }                                             \
    }                                               \
  } while (0)

// launch with programmatic stream serialisation (the kernels wait for their
// predecessor with griddepcontrol.wait before touching memory)
template <typename... KArgs, typename... Args>
cudaError_t pdl_launch(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t s,
                       Args... args) {
  static const bool pdl = getenv("HKV_NO_PDL") == nullptr;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

size_t smem_of(int NT, int max_len, int D, int P, int es) {
  // the query ring / score stages; key words, positions (4 B each) and
  // class/flag/rank (2 B) per row; q-bar; two 256-bin histograms
  return ring_bytes(NT, P, D, es, max_len) + (size_t)D * 4 + 512 * 4 + (size_t)max_len * 10 + 16;
}

}  // namespace

size_t update_smem_bytes(int threads, int max_len, int D, int P, int dtype) {
  return smem_of(threads, max_len, D, P, dtype == HKV_BF16 ? 2 : 4);
}

// (every segment that update_limit_bytes accepts fits with 512)
int update_threads(int nheads, int max_len, int sms) {
  if (max_len < 512) return nheads <= 2 * sms ? 256 : 128;
  return nheads <= 4 * sms ? 512 : nheads <= 16 * sms ? 256 : 128;
}

size_t update_limit_bytes(int max_len, int D, int P, int dtype) {
  // the interface's own sizes, whatever the kernels' threads and stages are
  constexpr size_t kRows = 256;
  const size_t es = dtype == HKV_BF16 ? 2 : 4;
  const size_t ring = (size_t)P * D * es, rows = kRows * (D * es + 16);
  return (ring > rows ? ring : rows) + (size_t)max_len * 16 + (size_t)D * 4 + 512 * 4 + 64;
}

cudaError_t update_prepare(int D, int dtype, size_t smem) {
  HKV_DISPATCH(D, dtype, return prepare_t<kD, kT>(smem));
  return cudaErrorInvalidValue;
}

// runs the statement with NT = `threads`
#define HKV_THREADS(threads_, ...)     \
  do {                                 \
    if ((threads_) == 512) {           \
      constexpr int NT = 512;          \
      __VA_ARGS__;                     \
    } else if ((threads_) == 256) {    \
      constexpr int NT = 256;          \
      __VA_ARGS__;                     \
    } else {                           \
      constexpr int NT = 128;          \
      __VA_ARGS__;                     \
    }                                  \
  } while (0)

cudaError_t launch_append_evict(const CacheArgs &c, const MethodArgs &m, int layer_base,
                                int nheads, const void *q, const void *k, const void *v, int D,
                                int dtype, int max_len, int threads, size_t smem,
                                cudaStream_t s) {
  HKV_DISPATCH(D, dtype,
               HKV_THREADS(threads, return pdl_launch(append_evict_kernel<NT, kD, kT>, nheads, NT,
                                                      smem, s, c, m, layer_base, q, k, v,
                                                      max_len)));
  return cudaErrorInvalidValue;
}

cudaError_t launch_evict(const CacheArgs &c, const MethodArgs &m, int layer_base, int nheads,
                         int D, int dtype, int max_len, int threads, size_t smem,
                         cudaStream_t s) {
  HKV_DISPATCH(D, dtype,
               HKV_THREADS(threads, return pdl_launch(evict_kernel<NT, kD, kT>, nheads, NT, smem,
                                                      s, c, m, layer_base, max_len)));
  return cudaErrorInvalidValue;
}

cudaError_t launch_repack(const CacheArgs &dense, const CacheArgs &ragged, const MethodArgs &m,
                          int layer_base, int nheads, int D, int dtype, int max_len, int threads,
                          size_t smem, cudaStream_t s) {
  HKV_DISPATCH(D, dtype,
               HKV_THREADS(threads, return pdl_launch(repack_kernel<NT, kD, kT>, nheads, NT, smem,
                                                      s, dense, ragged, m, layer_base, max_len)));
  return cudaErrorInvalidValue;
}

cudaError_t launch_prefill(const CacheArgs &c, int layer_base, int nheads, int C, const void *kc,
                           const void *vc, int D, int dtype, cudaStream_t s) {
  // a thread for every kPrefillBatch pieces, 64 to 512 of them
  const int pieces = C * (D * (dtype == HKV_BF16 ? 2 : 4) / 16);
  int threads = (pieces / kPrefillBatch + 31) / 32 * 32;
  threads = threads < 64 ? 64 : threads > 512 ? 512 : threads;
  HKV_DISPATCH(D, dtype,
               return pdl_launch(prefill_kernel<kD, kT>, nheads, threads, 0, s, c, layer_base, C,
                                 kc, vc));
  return cudaErrorInvalidValue;
}

cudaError_t launch_init_dense(const CacheArgs &c, int n, int seg, cudaStream_t s) {
  int grid = (n + 255) / 256;
  if (grid > 4096) grid = 4096;
  if (grid < 1) grid = 1;
  return pdl_launch(init_dense_kernel, grid, 256, 0, s, c, n, seg);
}

cudaError_t launch_identify(const CacheArgs &c, const MethodArgs &m, int layer_base, int nheads,
                            const void *q, uint8_t *label_out, int32_t *nh_out, int D, int dtype,
                            int max_len, int sms, cudaStream_t s) {
  const float qscale = (float)(1.4426950408889634 / sqrt((double)D));
  const size_t smem = identify_smem_bytes(max_len, m.P, m.grid2d != 0, false);
  // the stages lie behind the rest, where both fit (identify_stage_bytes)
  const size_t staged = identify_stage_bytes(nheads, max_len, m.grid2d != 0,
                                             D * (dtype == HKV_BF16 ? 2 : 4), sms);
  if (staged > 0) {
    HKV_DISPATCH(D, dtype,
                 return pdl_launch(identify_kernel<kD, kT, 8, true>, nheads, IT, staged, s, c, m,
                                   layer_base, q, label_out, nh_out, qscale, max_len,
                                   (int)id_stage_at(smem)));
  }
  if (id_rows_in_flight(max_len, false) == 8) {
    HKV_DISPATCH(D, dtype,
                 return pdl_launch(identify_kernel<kD, kT, 8, false>, nheads, IT, smem, s, c, m,
                                   layer_base, q, label_out, nh_out, qscale, max_len, 0));
  }
  HKV_DISPATCH(D, dtype,
               return pdl_launch(identify_kernel<kD, kT, 2, false>, nheads, IT, smem, s, c, m,
                                 layer_base, q, label_out, nh_out, qscale, max_len, 0));
  return cudaErrorInvalidValue;
}

cudaError_t launch_identify_multi(const CacheArgs &c, const MethodArgs &m, int layer_base,
                                  int nheads, uint8_t *label_out, int32_t *nh_out, int D,
                                  int dtype, int max_len, cudaStream_t s) {
  const float qscale = (float)(1.4426950408889634 / sqrt((double)D));
  const size_t smem = identify_smem_bytes(max_len, m.P, m.grid2d != 0, true);
  const bool q8 = id_qb(m.P) == 8, u4 = id_rows_in_flight(max_len, true) == 4;
#define HKV_ID_MULTI(QB_, U_)                                                                  \
  HKV_DISPATCH(D, dtype,                                                                       \
               return pdl_launch(identify_multi_kernel<kD, kT, QB_, U_>, nheads, IT, smem, s, c, \
                                 m, layer_base, label_out, nh_out, qscale, max_len))
  if (q8 && u4) HKV_ID_MULTI(8, 4);
  if (q8) HKV_ID_MULTI(8, 2);
  if (u4) HKV_ID_MULTI(4, 4);
  HKV_ID_MULTI(4, 2);
#undef HKV_ID_MULTI
  return cudaErrorInvalidValue;
}

// The stages pay while the heads have an SM, or half of one, each (their keys
// are on the way before the first product, but they leave room for two CTAs an
// SM at most), and where a head's keys take 256 KB and more. us without and
// with, bf16 rows of 256 bytes: 628 tokens, 32 heads 7.8, 6.6, 256 13.3, 11.3,
// 512 18.2, 20.0, 1216 37.7, 40.8, 2560 73.7, 72.8; 1128 tokens, 512 28.1, 29.4,
// 704 47.0, 42.0, 2560 122, 113; of 128 bytes, 601 tokens, 512 12.9, 14.9, 4096
// 67, 75, 2001 tokens 173, 168; fp32 rows of 512, 628 tokens, 1024 58.3, 55.4.
// The count on the grid ranks every row and wants the other CTAs' warps: 2000
// tokens, 128 heads 175, 157, 256 (one CTA an SM with the stages) 265, 305.
size_t identify_stage_bytes(int nheads, int max_len, bool grid2d, int row_bytes, int sms) {
  if (max_len < kIdLongSegment) return 0;
  if (nheads > 2 * sms && (grid2d || (size_t)max_len * row_bytes < 256 * 1024)) return 0;
  const size_t b = id_stage_at(identify_smem_bytes(max_len, 1, grid2d, false)) +
                   (size_t)kIdStages * kIdStageBytes;
  return b <= (grid2d && nheads > sms ? kIdTwoSmem : kIdMostSmem) ? b : 0;
}

size_t identify_smem_bytes(int max_len, int P, bool grid2d, bool multi) {
  const size_t floats = multi ? (size_t)(id_qb(P) + 1) * max_len : (size_t)max_len;
  return id_smem(floats, max_len, grid2d);
}

cudaError_t launch_budgets(const uint8_t *label, int32_t *budget, int32_t *cap, int64_t *off,
                           int n, int C, int B_g, int w, int P, int group, cudaStream_t s) {
  if (group == 0 && n <= kBudgetMost)
    return pdl_launch(budgets_plain_kernel, (n + kBudgetHeads - 1) / kBudgetHeads, kBudgetThreads, 0,
                      s, label, budget, cap, off, n, C, B_g, w, P);
  return pdl_launch(budgets_kernel, 1, 1024, 0, s, label, budget, cap, off, n, C, B_g, w, P, group);
}

}  // namespace hkv
