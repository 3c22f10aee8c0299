// sp_scan_binned.cu -- the per-pair scan with the LDCA updates moved from L2
// atomics to shared-memory atomics (Sec. 3.3 update, Sec. 4.1 scan).
//
// Every pair sets the same bit b = H3(oip) in its LR LDCs LH_i(hip).  Call
// "plane b" the set of bit b of every LDC: LR x LC bits (32 KiB at k = 1024,
// LR = 4, LC = 2^16).  A pair touches exactly one plane, so:
//
//  k_bin    (persistent, one or two blocks per SM, shapes below) streams tiles
//           with 16-byte loads held in registers (the next tile's loads are
//           issued before the current tile's work), does the SEAV update of
//           Sec. 3.1-3.2 for sampled pairs (L2 RED, 1 pair in 2^tau), and
//           stages each hip in a shared-memory row of its bin b; a row's whole
//           8-hip chunks go to the block's private list for that row with one
//           32-byte store each (no global atomics; lists[row][block][0 .. cap)).
//           Hips that find their row full wait for the end of the round; only
//           skewed inputs (a full list, a row that stays full) send hips to L2
//           REDs instead (any input is correct).
//  k_apply  (one block per plane) starts the plane in shared memory from
//           zero (or from the router's pending plane when earlier updates of
//           the window have not been folded yet), sets bit (i, LH_i(hip)) for
//           every listed hip and row i with shared atomic OR, and stores the
//           plane back by TMA (the block owns it).  Bounds: the load-store pipe,
//           94% busy at 2^26 pairs, by the LR random atomics per hip.
//  k_fold   (before the next detect, copy or export of the router, or in a
//           merge, over all sources at once) ORs the plane accumulators into
//           the LDCA's logical layout [LR][LC][k / 32]: word J of 32 consecutive
//           planes is a 32 x 32 bit block whose transpose holds the words of LDCs
//           32 J .. 32 J + 31.
//
// Applicable when the bins are the LDC's k bit positions (k <= 1024) and one
// plane fits in shared memory as whole words (LC >= 32, LR x LC <= 2^20 bits).
//
// Staging shapes (the autotuner picks one per context; every shape gives the
// same bits):  k_bin block size, staging row length, tiles per flush round
// and blocks per SM -- a 1024-thread block with 44-hip rows, or two 512-thread
// blocks per SM with 20-hip rows, so that one block's flush overlaps the other's
// hashing; both flush every two of their tiles -- and the k_apply block size.
#include <cuda.h>
#include <math.h>

#include <atomic>

#include "sp_internal.h"

namespace sp {

namespace {

constexpr int kVec = 4;                            // 16-byte loads (2 pairs) per thread and tile
constexpr int kGroup = 4;                          // pairs hashed and staged together
constexpr int kChunk = 8;                          // hips per list store (32 bytes)
constexpr int kOver = 128;                         // pairs per round that found their row full
constexpr uint32_t kFull = 0xFFFFFFFFu;

__device__ __forceinline__ void seav_set(const DevParams& d, uint8_t* seav, uint32_t hip, uint32_t h1) {
  const uint32_t bit = h1 >> 29;
  const uint32_t rp = d.r ? (hip & ((1u << d.r) - 1u)) : 0u;
  const uint32_t lp = (uint32_t)((uint64_t)hip >> d.r);
  const uint64_t base = (uint64_t)rp * d.sea_bytes;
  for (uint32_t i = 0; i < d.sr; ++i) {
    const uint64_t off = base + d.row_off[i] + gather_idx(lp, d.isb[i], d.ibn[i], d.L);
    atomicOr(reinterpret_cast<uint32_t*>(seav + (off & ~3ull)), (1u << bit) << (8u * (uint32_t)(off & 3u)));
  }
}

// One L2 RED per LDCA row: the rare overflow path of k_bin (a full staging
// row or list), so the row count is read at run time.
__device__ __forceinline__ void ldca_red(const DevParams& d, uint32_t* ldca, uint32_t hip, uint32_t h3) {
  const uint32_t cshift = 32u - d.lc_log2;
  const uint32_t wshift = d.k_log2 - 5u;
#pragma unroll
  for (uint32_t i = 0; i < 8; ++i) {               // constant indices into the parameter block
    if (i < d.lr) {
      const uint32_t col = (uint32_t)((uint64_t)mas(d.ha[2 + i], d.hb[2 + i], hip) >> cshift);
      atomicOr(ldca + (((uint64_t)((i << d.lc_log2) | col) << wshift) | (h3 >> 5)), 1u << (h3 & 31u));
    }
  }
}

// 256-bit store of 8 hips (a 32-byte aligned list chunk, one full sector).
__device__ __forceinline__ void st_chunk(uint32_t* dst, uint4 a, uint4 b) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               :: "l"(dst), "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
               : "memory");
}

// k_bin: tiles of TILE = THREADS * 2 kVec pairs, tile (slot + i G) in iteration i.  Each
// thread holds kVec 16-byte loads (2 pairs each) of a tile in registers and
// issues the loads of tile i + 1 before it works on tile i, so the copy from
// HBM overlaps the work.  What is left after whole rounds over the blocks is
// cut into one small tile for each block.  H3's hash selects one of 1,024
// rows by its top 10 bits, so that rows fill alike for every k: with k < 1024 a
// bin (the hash's top log2 k bits) has several rows and lists, consecutive ones
// (k = 256 with a row per bin: 64 arrivals per 44-hip row and round, and 2^23
// pairs took 136 us, so 61).  Every row is a staging
// row of STAGE hips in shared memory that persists across tiles (a
// write-combining buffer for the bin's list).  Per tile:
//   1. every thread hashes its pairs, queues the sampled pairs (Sec. 3.1) for
//      a converged SEAV pass, takes a place in its pair's bin row with one
//      shared atomic and stores the hip there (a pair that finds its row full
//      waits for the end of the round -- by chance fewer than one in a million
//      with 44-hip rows, 16 arrivals a round on average, two in a thousand with
//      20-hip rows and 8 arrivals: a single LDCA bit set past the lists would
//      make the fold read 32 MiB of LDCA, the merge 128 MiB per router of profile
//      D3 and the reset zero them);
//   2. (after every TPR = 2 tiles) each thread takes bins tid, tid + THREADS, ...:
//      it moves the row's whole 8-hip chunks to the bin's list with 32-byte
//      stores and keeps the remainder (< 8 hips) at the front of the row; the
//      queued pairs set their SEAV bits, taken by consecutive threads.
// At the end the remainders go to the lists with plain stores; an appending
// launch first takes the tail of a list that is not a whole chunk back into
// the row, so lists stay dense and chunk stores stay 32-byte aligned.
template <int THREADS, int STAGE, int TPR, int PER_SM>
__global__ void __launch_bounds__(THREADS, PER_SM)
k_bin(DevParams d, uint8_t* __restrict__ seav, uint32_t* __restrict__ ldca,
      BinSrc src, uint32_t* __restrict__ lists, uint32_t* __restrict__ counts, uint32_t cap,
      bool append, uint32_t rot, RouterFlags* __restrict__ flags, uint32_t* __restrict__ prior) {
  static_assert(TPR == 2, "one flush round after the tiles of both register buffers");
  constexpr int QUADS = THREADS * kVec;               // 16-byte loads of a whole tile
  constexpr int TILE = QUADS * 2;
  constexpr int QUEUE = TPR * TILE / 32;              // sampled pairs per round: 4x the expected 2^-7
  extern __shared__ __align__(128) uint8_t smem_raw[];
  constexpr uint32_t bins = kBinRows;                                  // rows; bin b has kBinRows / k of them
  uint32_t* stage = reinterpret_cast<uint32_t*>(smem_raw);             // [bins][STAGE], then a 32-word sink
  uint32_t* sink = stage + bins * STAGE;                                // stores of pairs a full row refused
  uint2* s_queue = reinterpret_cast<uint2*>(sink + 32);               // [QUEUE] sampled (hip, h1)
  uint2* s_over = s_queue + QUEUE;                                      // [2][kOver] (hip, bin) of full rows, by round parity
  uint32_t* s_fill = reinterpret_cast<uint32_t*>(s_over + 2 * kOver);  // [bins] hips in the row
  uint32_t* s_cursor = s_fill + bins;                                   // [bins] list fill (whole chunks)
  __shared__ uint32_t s_qn[2], s_on[2];                                 // queue and s_over fill, by round parity
  __shared__ uint32_t s_full[kBinMaxSrc + 1], s_small[kBinMaxSrc + 1];   // tiles before stream b (fewer than 2^32 a round)
  const uint32_t tid = threadIdx.x;
  const uint32_t G = gridDim.x, cta = blockIdx.x;
  const uint32_t slot = (cta + rot) % G;          // which tiles this block takes
  const uint32_t tau_mask = (1u << d.tau) - 1u;
  constexpr uint32_t h3_shift = 32u - kBinRowsLog2;
  const uint32_t row_shift = kBinRowsLog2 - d.k_log2;                   // bin of a row
  const uint32_t lane = tid & 31u;
  uint32_t lt_mask;                                // lanes below this one
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(lt_mask));
  // a hip whose row or list was full: its LDCA bits go straight to L2, and
  // the router's flag tells the fold that the LDCA is no longer all zero
  auto spill = [&](uint32_t hip, uint32_t b) {     // b: the row
    ldca_red(d, ldca, hip, b >> row_shift);
    flags->spilled = 1u;
  };
  // A stream is a body of 16-byte quads (two pairs) and up to two single
  // pairs: its first one when it starts 8 bytes off a 16-byte boundary, its last
  // one when one is left over.  The body is cut into whole tiles (at most
  // src.full_max of a stream) and small ones of src.small_quads for the rest;
  // whole tiles of stream b are [s_full[b], s_full[b + 1]), small ones likewise.
  auto head_of = [&](uint32_t b) { return ((uintptr_t)src.ptr[b] & 15u) != 0u ? 1u : 0u; };
  auto quads_of = [&](uint32_t b) { return src.n[b] != 0 ? (src.n[b] - head_of(b)) >> 1 : (uint64_t)0; };
  if (tid < 64) {                                  // warp 0: whole tiles, warp 1: small ones
    uint32_t* pref = tid < 32 ? s_full : s_small;
    uint32_t sum[kBinMaxSrc / 32], acc = 0;
#pragma unroll
    for (int e = 0; e < kBinMaxSrc / 32; ++e) {
      const uint32_t b = lane * (kBinMaxSrc / 32) + (uint32_t)e;
      if (b < src.count) {
        const uint64_t quads = quads_of(b);
        const uint32_t full = (uint32_t)min(quads / QUADS, (uint64_t)src.full_max);
        acc += tid < 32 ? full
                        : (uint32_t)((quads - (uint64_t)full * QUADS + src.small_quads - 1) / src.small_quads);
      }
      sum[e] = acc;
    }
    uint32_t incl = acc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
#pragma unroll
    for (int e = 0; e < kBinMaxSrc / 32; ++e) pref[lane * (kBinMaxSrc / 32) + (uint32_t)e + 1] = incl - acc + sum[e];
    if (lane == 0) pref[0] = 0;
    if (tid == 0) s_qn[0] = s_qn[1] = s_on[0] = s_on[1] = 0;
    if (tid == 0 && cta == 0 && !append) {         // the round's first launch: its k_apply makes the planes pending
      if (prior != nullptr) *prior = flags->pending;
      flags->pending = 1u;
    }
  }
  auto list_of = [&](uint32_t b) { return lists + ((uint64_t)b * G + cta) * cap; };
  for (uint32_t b = tid; b < bins; b += THREADS) {
    // an appending launch continues the list: its partial chunk returns to the row
    const uint32_t have = append ? counts[(uint64_t)b * G + cta] : 0u;
    const uint32_t tail = have & (kChunk - 1u);
    for (uint32_t e = 0; e < tail; ++e) stage[b * STAGE + e] = list_of(b)[have - tail + e];
    s_fill[b] = tail;
    s_cursor[b] = have - tail;
  }
  __syncthreads();
  const uint32_t n_tiles = s_full[src.count], n_small = s_small[src.count];
  // 16-byte streaming loads of this thread's share of a whole tile; volatile,
  // so they are issued where they stand (before the work on the previous tile)
  uint32_t stream_hint = 0;                      // this block's tiles come in stream order
  auto load_tile = [&](uint4 (&r)[kVec], uint32_t tile) {
    uint32_t b = stream_hint;
    while (s_full[b + 1] <= tile) ++b;
    stream_hint = b;
    const uint4* p4 = reinterpret_cast<const uint4*>(src.ptr[b] + 2u * head_of(b)) +
                      (uint64_t)(tile - s_full[b]) * QUADS + tid;
#pragma unroll
    for (int u = 0; u < kVec; ++u)
      asm volatile("ld.global.cs.v4.u32 {%0, %1, %2, %3}, [%4];"
                   : "=r"(r[u].x), "=r"(r[u].y), "=r"(r[u].z), "=r"(r[u].w) : "l"(p4 + u * THREADS));
  };
  // step 1 for a group of kGroup pairs (valid: bit q = pair q exists):
  // hashes, the sampled-pair queue (one warp-aggregated push per pair
  // position), the row places (independent shared atomics), the staging
  // stores; a pair whose row is full is marked in the returned mask
  auto stage_group = [&](const uint32_t (&hip)[kGroup], const uint32_t (&oip)[kGroup], uint32_t valid,
                         uint32_t par, uint32_t (&bin)[kGroup]) {
    uint32_t at[kGroup], over = 0;
#pragma unroll
    for (int q = 0; q < kGroup; ++q) {
      const uint32_t h1 = mas(d.ha[0], d.hb[0], oip[q]);
      const uint32_t ballot = __ballot_sync(kFull, ((valid >> q) & 1u) && (h1 & tau_mask) == 0u);
      if (ballot) {
        uint32_t first = 0;
        if (lane == 0) first = atomicAdd(&s_qn[par], (uint32_t)__popc(ballot));
        first = __shfl_sync(kFull, first, 0) + (uint32_t)__popc(ballot & lt_mask);
        if (((ballot >> lane) & 1u) && first < (uint32_t)QUEUE) s_queue[first] = make_uint2(hip[q], h1);
        else if ((ballot >> lane) & 1u) over |= 1u << (kGroup + q);   // queue full: SEAV bits directly
      }
      bin[q] = mas(d.ha[1], d.hb[1], oip[q]) >> h3_shift;
    }
#pragma unroll
    for (int q = 0; q < kGroup; ++q)
      at[q] = ((valid >> q) & 1u) ? atomicAdd(&s_fill[bin[q]], 1u) : 0xFFFFu;
#pragma unroll
    for (int q = 0; q < kGroup; ++q) {
      // no branch: a pair that finds its row full (or no pair) stores to
      // this lane's sink word instead
      uint32_t* dst = at[q] < (uint32_t)STAGE ? stage + bin[q] * STAGE + at[q] : sink + lane;
      *dst = hip[q];
      over |= (at[q] >= (uint32_t)STAGE && at[q] != 0xFFFFu ? 1u : 0u) << q;
    }
    return over;
  };
  // the rare leftovers of a group: pairs whose row was full wait in s_over for
  // the end of the round (LDCA bits with L2 REDs only when that is full too),
  // sampled pairs the full queue did not take set their SEAV bits
  auto group_leftovers = [&](const uint32_t (&hip)[kGroup], const uint32_t (&oip)[kGroup],
                             const uint32_t (&bin)[kGroup], uint32_t over, uint32_t par) {
    if (__any_sync(kFull, over != 0u)) {
#pragma unroll
      for (int q = 0; q < kGroup; ++q) {
        if ((over >> q) & 1u) {
          const uint32_t at = atomicAdd(&s_on[par], 1u);
          if (at < (uint32_t)kOver) s_over[par * kOver + at] = make_uint2(hip[q], bin[q]);
          else spill(hip[q], bin[q]);
        }
        if ((over >> (kGroup + q)) & 1u) seav_set(d, seav, hip[q], mas(d.ha[0], d.hb[0], oip[q]));
      }
    }
  };
  // whole chunks of bin b's row (fill f <= STAGE) to its list, remainder to the front
  auto flush_row = [&](uint32_t b, uint32_t f) {
    uint32_t* row = stage + b * STAGE;
    uint32_t* list = list_of(b);
    uint32_t cur = s_cursor[b];
    const uint32_t nch = f / kChunk;
    for (uint32_t c = 0; c < nch; ++c) {
      const uint4 x = *reinterpret_cast<const uint4*>(row + c * kChunk);
      const uint4 y = *reinterpret_cast<const uint4*>(row + c * kChunk + 4);
      if (cur + kChunk <= cap) {
        st_chunk(list + cur, x, y);
        cur += kChunk;
      } else {                                      // list full: straight to L2
        const uint32_t h[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
        for (int e = 0; e < 8; ++e) spill(h[e], b);
      }
    }
    const uint32_t rem = f - nch * kChunk;
    for (uint32_t e = 0; e < rem; e += 4)           // within the row: nch * 8 + rem <= STAGE
      *reinterpret_cast<uint4*>(row + e) = *reinterpret_cast<const uint4*>(row + nch * kChunk + e);
    s_fill[b] = rem;
    s_cursor[b] = cur;
  };
  // 1. hash, queue the sampled pairs, stage the hips of one whole tile in their bins' rows
  auto stage_tile = [&](const uint4 (&r)[kVec], uint32_t par) {
#pragma unroll
    for (int g = 0; g < kVec / (kGroup / 2); ++g) {
      uint32_t hip[kGroup], oip[kGroup], bin[kGroup];
#pragma unroll
      for (int u = 0; u < kGroup / 2; ++u) {
        const uint4 v = r[g * (kGroup / 2) + u];
        hip[2 * u] = v.x; oip[2 * u] = v.y;
        hip[2 * u + 1] = v.z; oip[2 * u + 1] = v.w;
      }
      const uint32_t over = stage_group(hip, oip, (1u << kGroup) - 1u, par, bin);
      group_leftovers(hip, oip, bin, over, par);
    }
  };
  // the flush round: whole chunks to the lists; the queued SEAV updates,
  // spread over the warps
  auto flush_round = [&](uint32_t par) {
    __syncthreads();
    const uint32_t qn = s_qn[par] < (uint32_t)QUEUE ? s_qn[par] : (uint32_t)QUEUE;
    const uint32_t on = s_on[par] < (uint32_t)kOver ? s_on[par] : (uint32_t)kOver;
    if (tid == 0) s_qn[par ^ 1u] = s_on[par ^ 1u] = 0;   // read by every thread before the last barrier
    for (uint32_t b = tid; b < bins; b += THREADS) {
      const uint32_t f = s_fill[b];
      if (f >= (uint32_t)kChunk) flush_row(b, f < (uint32_t)STAGE ? f : (uint32_t)STAGE);
    }
    for (uint32_t e = tid; e < qn; e += THREADS) {   // consecutive threads: the fewest warps
      const uint2 x = s_queue[e];
      seav_set(d, seav, x.x, x.y);
    }
    __syncthreads();
    // the round's leftovers take places in the rows, which have room again
    if (tid < on) {
      const uint2 x = s_over[par * kOver + tid];
      const uint32_t at = atomicAdd(&s_fill[x.y], 1u);
      if (at < (uint32_t)STAGE) stage[x.y * STAGE + at] = x.x;
      else spill(x.x, x.y);
    }
  };
  // Tiles in pairs (i, i + 1) in the two register buffers.  A buffer's loads
  // for tile t + 2 go out as soon as tile t is staged, so the flush round
  // runs with both next tiles in flight (the flush's stores and the stream's
  // loads overlap).
  uint32_t par = 0;
  if (slot < n_tiles) {
    uint4 ra[kVec], rb[kVec];
    load_tile(ra, slot);
    if (slot + G < n_tiles) load_tile(rb, slot + G);
    for (uint32_t t = slot; t < n_tiles; t += 2 * G) {
      stage_tile(ra, par);
      if (t + 2 * G < n_tiles) load_tile(ra, t + 2 * G);
      if (t + G < n_tiles) {
        stage_tile(rb, par);
        if (t + 3 * G < n_tiles) load_tile(rb, t + 3 * G);
      }
      flush_round(par);
      par ^= 1u;
    }
  }
  // small tiles, first to the blocks that had a whole tile less, and the
  // streams' single pairs with them: all of a thread's loads, then the work
  for (uint32_t t = (slot + G - n_tiles % G) % G; t < n_small || t < src.count; t += G) {
    uint32_t b = 0, n = 0;
    uint4 r[kVec];
    if (t < n_small) {
      while (s_small[b + 1] <= t) ++b;
      const uint64_t base = (uint64_t)(s_full[b + 1] - s_full[b]) * QUADS + (uint64_t)(t - s_small[b]) * src.small_quads;
      n = (uint32_t)min(quads_of(b) - base, (uint64_t)src.small_quads);
      const uint4* p4 = reinterpret_cast<const uint4*>(src.ptr[b] + 2u * head_of(b)) + base;
#pragma unroll
      for (int u = 0; u < kVec; ++u)
        if (tid + u * THREADS < n) r[u] = __ldcs(p4 + tid + u * THREADS);
    }
#pragma unroll
    for (int g = 0; g <= kVec / (kGroup / 2); ++g) {
      uint32_t hip[kGroup] = {}, oip[kGroup] = {}, bin[kGroup], valid = 0;
      if (g < kVec / (kGroup / 2)) {
#pragma unroll
        for (int u = 0; u < kGroup / 2; ++u) {
          const int q = g * (kGroup / 2) + u;
          if (tid + (uint32_t)q * THREADS < n) {
            hip[2 * u] = r[q].x; oip[2 * u] = r[q].y;
            hip[2 * u + 1] = r[q].z; oip[2 * u + 1] = r[q].w;
            valid |= 3u << (2 * u);
          }
        }
      } else if (t < src.count && tid < 2) {          // stream t: thread 0 its first pair, thread 1 its last one
        const uint32_t head = head_of(t);
        if (src.n[t] != 0 && (tid == 0 ? head != 0u : ((src.n[t] - head) & 1u) != 0u)) {
          const uint2 v = reinterpret_cast<const uint2*>(src.ptr[t])[tid == 0 ? 0 : src.n[t] - 1];
          hip[0] = v.x; oip[0] = v.y;
          valid = 1u;
        }
      }
      if (__any_sync(kFull, valid != 0u)) {
        const uint32_t over = stage_group(hip, oip, valid, par, bin);
        group_leftovers(hip, oip, bin, over, par);
      }
    }
    flush_round(par);
    par ^= 1u;
  }
  // the last round's leftovers are in the rows: whole chunks once more
  __syncthreads();
  for (uint32_t b = tid; b < bins; b += THREADS) {
    const uint32_t f = s_fill[b];
    if (f >= (uint32_t)kChunk) flush_row(b, f < (uint32_t)STAGE ? f : (uint32_t)STAGE);
  }
  // remainders (< 8 hips per row): one more chunk, filled up with copies of a
  // hip of its own, so that k_apply reads whole 16-byte quads of a list (a bit
  // set twice is the same bit); counts[] has the real number
  for (uint32_t b = tid; b < bins; b += THREADS) {
    const uint32_t f = s_fill[b], c = s_cursor[b];
    const uint32_t* row = stage + b * STAGE;
    uint32_t kept = 0;
    if (f != 0u && c + kChunk <= cap) {
      const uint4 x = *reinterpret_cast<const uint4*>(row), y = *reinterpret_cast<const uint4*>(row + 4);
      st_chunk(list_of(b) + c,
               make_uint4(x.x, f > 1 ? x.y : x.x, f > 2 ? x.z : x.x, f > 3 ? x.w : x.x),
               make_uint4(f > 4 ? y.x : x.x, f > 5 ? y.y : x.x, f > 6 ? y.z : x.x, x.x));
      kept = f;
    } else {
      for (uint32_t e = 0; e < f; ++e) spill(row[e], b);
    }
    counts[(uint64_t)b * G + cta] = c + kept;
  }
}

// A list read once streams past L2 (evict first); a list that SPLIT > 1
// blocks read, close together in time, stays there for the second read.
template <int SPLIT>
__device__ __forceinline__ uint4 load_hips(const uint32_t* p) {
  const uint4* q = reinterpret_cast<const uint4*>(p);
  return SPLIT == 1 ? __ldcs(q) : __ldg(q);
}

// k_apply, LCL = log2 LC when it is fixed at compile time (profiles D, D3
// and S: constant shifts and row offsets), 0 for any LC.  SPLIT blocks share
// a plane, each holding LR / SPLIT of its LDCA rows in shared memory and
// reading the whole hip list: wide planes (LC = 2^18: 128 KiB for four rows)
// would otherwise leave one block per SM.
// Groups of 8 lanes walk the plane's lists on their own (list c, c + NG, ...),
// 2 x 32 hips a step, two 16-byte loads per lane, issued a step ahead and the
// first step before the plane is zeroed: short lists -- a launch of 5 M pairs
// leaves 32 hips in each, one of 2^24 108 -- are bound by the loads' latency.
// The lists' counts are in shared memory before the walk starts.  A group takes
// whole lists: sharing one among 2 or 4 groups balances the warps better and
// measured 3% slower (more ragged ends).  Two loads a step at three blocks per
// SM (40 registers): 16 routers x 2^24 pairs scan in 2.33 ms against 2.49 with
// one load, and 2^26 pairs in 333 against 336 us; at four blocks (32
// registers, spills) 2.33 ms and 344 us.
// Lists are filled up to whole 8-hip chunks (k_bin), so a lane's 4 hips are
// all there or none is.
constexpr int kQuads = 2;
template <int LR, int THREADS, int LCL, int SPLIT>
__global__ void __launch_bounds__(THREADS, 1536 / THREADS)
k_apply(DevParams d, const uint32_t* __restrict__ lists, const uint32_t* __restrict__ counts,
        uint32_t G, uint32_t cap, const uint32_t* planes, const __grid_constant__ CUtensorMap map, uint32_t box,
        bool accumulate, const uint32_t* prior) {
  extern __shared__ __align__(128) uint32_t s_plane[];
  constexpr int LRP = LR / SPLIT;                                  // rows of this block
  constexpr uint32_t NG = THREADS / 8;
  const uint32_t b = blockIdx.x / SPLIT;
  const uint32_t row0 = (blockIdx.x % SPLIT) * (uint32_t)LRP;
  const uint32_t lc_log2 = LCL ? (uint32_t)LCL : d.lc_log2;
  const uint32_t chunks = ((((uint32_t)LRP << lc_log2) >> 5) + 7u) / 8u;  // 8-word chunks of the block's rows
  uint32_t* s_count = s_plane + chunks * 8u;                       // [G]
  const uint32_t tid = threadIdx.x, lane = tid & 31u;
  const uint32_t first = 4u * (lane & 7u);                          // this lane's hips of a step
  uint32_t c = tid >> 3, at = first;
  counts += (uint64_t)b * G;
  uint32_t n = c < G ? counts[c] : 0u;
  const uint32_t* list = lists + ((uint64_t)b * G + c) * cap;
  struct Step { uint4 h[kQuads]; uint32_t have; };                 // have: valid 16-byte loads
  auto load = [&](Step& s) {
    s.have = at < n ? min((n - at + 31u) / 32u, (uint32_t)kQuads) : 0u;
#pragma unroll
    for (int u = 0; u < kQuads; ++u)
      if ((uint32_t)u < s.have) s.h[u] = load_hips<SPLIT>(list + at + 32 * u);
  };
  Step s0, s1;
  load(s0);
  // LH_i(hip) = h >> cshift (5 <= lc_log2 <= 20): LDC h >> cshift of row i is
  // bit (h >> cshift) mod 32 of plane word (i << (lc_log2 - 5)) + (h >> (cshift + 5))
  const uint32_t cshift = 32u - lc_log2;
  const uint32_t row_words_log2 = lc_log2 - 5u;
  // accumulator layout [ceil(words / 8)][k][8]: word w of plane b at
  // (w / 8) k 8 + 8 b + w mod 8, so that a 32-byte chunk holds 8 words of one
  // plane (with SPLIT > 1 a row is a multiple of 8 words)
  const uint64_t chunk_stride = (uint64_t)(1u << d.k_log2) * 8u;
  const uint32_t chunk0 = (row0 << row_words_log2) / 8u;            // the block's first chunk
  const uint32_t* src = planes + (uint64_t)b * 8u + (uint64_t)chunk0 * chunk_stride;
  // the rows' hash words, held in registers
  uint32_t a_lo[LRP], a_hi[LRP];
  uint64_t bw[LRP];
#pragma unroll
  for (int r = 0; r < LRP; ++r) {
    a_lo[r] = (uint32_t)d.ha[2 + row0 + r];
    a_hi[r] = (uint32_t)(d.ha[2 + row0 + r] >> 32);
    bw[r] = d.hb[2 + row0 + r];
  }
  for (uint32_t i = tid; i < G; i += THREADS) s_count[i] = counts[i];
  if (prior != nullptr) accumulate = *prior != 0u;
  for (uint32_t u = tid; u < chunks * 2u; u += THREADS)             // 16-byte units, consecutive lanes
    *reinterpret_cast<uint4*>(s_plane + u * 4u) =
        accumulate ? *reinterpret_cast<const uint4*>(src + (u >> 1) * chunk_stride + (u & 1u) * 4u)
                   : make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  auto set_bits = [&](uint32_t hip) {
#pragma unroll
    for (int r = 0; r < LRP; ++r) {
      const uint64_t lo = (uint64_t)a_lo[r] * hip + bw[r];
      const uint32_t h = (uint32_t)(lo >> 32) + a_hi[r] * hip;      // MAS (Sec. 3.3 LH_r)
      if (LCL) {
        atomicOr(&s_plane[((uint32_t)r << row_words_log2) + (h >> (cshift + 5u))], 1u << ((h >> cshift) & 31u));
      } else {
        // the clamping funnel shift gives 0 for the shift of 32 at lc_log2 = 5;
        // the wrapping one takes the bit position mod 32
        atomicOr(&s_plane[((uint32_t)r << row_words_log2) + __funnelshift_rc(h, 0u, cshift + 5u)],
                 __funnelshift_l(0u, 1u, h >> cshift));
      }
    }
  };
  // loads the next step, then sets the bits of the current one; false when no
  // group of the warp has a list left
  auto turn = [&](Step& cur, Step& next) {
    if (!__any_sync(kFull, c < G)) return false;
    at += 32u * kQuads;
    if (at - first >= n) {                                          // the group's next list
      c += NG;
      at = first;
      n = c < G ? s_count[c] : 0u;
      list += (uint64_t)NG * cap;
    }
    load(next);
#pragma unroll
    for (int u = 0; u < kQuads; ++u)
      if ((uint32_t)u < cur.have) {
        set_bits(cur.h[u].x);
        set_bits(cur.h[u].y);
        set_bits(cur.h[u].z);
        set_bits(cur.h[u].w);
      }
    return true;
  };
  while (turn(s0, s1) && turn(s1, s0)) {}
  // the plane's chunks go out by TMA, `box` chunks a copy: 1,024 sectors 32 KiB
  // apart (profile D), which as 32-byte stores took one wavefront of the
  // load-store pipe each, the pipe that bounds the kernel
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncthreads();
  if (tid == 0) {
    for (uint32_t ch = 0; ch < chunks; ch += box)
      asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
                   :: "l"(&map), "r"(0), "r"(b), "r"(chunk0 + ch),
                      "r"((uint32_t)__cvta_generic_to_shared(s_plane + ch * 8u)) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // shared memory is read before the block ends
  }
}

// 32 x 32 bit transpose across a warp: lane l holds row l (bit j = column j);
// afterwards lane l holds column l (bit p = row p's bit l).  Stage s = 16, 8,
// 4, 2, 1 swaps s x s blocks between lanes l and l ^ s.  With m the columns
// whose bit s is clear, the lane whose bit s is clear keeps its m columns and
// takes the partner's m columns moved up by s; the other lane keeps its ~m
// columns and takes the partner's ~m columns moved down by s.  Either move is
// a rotation of the partner's word (left by s, or by 32 - s) whose other bits
// land in the columns the lane keeps, so a stage is one shuffle, one
// funnel-shift rotation and one bitwise select.
__device__ __forceinline__ uint32_t transpose32(uint32_t x, uint32_t lane) {
  const uint32_t masks[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
  for (int st = 0; st < 5; ++st) {
    const uint32_t s = 16u >> st;
    const bool high = (lane & s) != 0u;
    const uint32_t keep = high ? ~masks[st] : masks[st];
    const uint32_t y = __shfl_xor_sync(kFull, x, s);
    const uint32_t t = __funnelshift_l(y, y, high ? 32u - s : s);
    x = (x & keep) | (t & ~keep);
  }
  return x;
}

// 256-bit load of 8 words (a 32-byte aligned plane chunk, one full sector).
__device__ __forceinline__ void ld_chunk(const uint32_t* src, uint32_t (&v)[8]) {
  asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "l"(src));
}

// 32 x 32 bit transposes of 8 blocks, one per q = lane / 4: lane (q, s) holds
// rows p = 4 i + s of block q in x[i] (bit c = column c) and afterwards columns
// c = 4 i + s (bit p = row p's bit c).  Row bits 2 - 4 are register indices, so
// three of the five butterfly stages stay in the lane (two byte permutes, one
// shift and select); row bits 0 and 1 are lane bits: one shuffle, one
// rotation and one select per word.
__device__ __forceinline__ void transpose8x4(uint32_t (&x)[8], uint32_t lane) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {                      // rows p and p + 16
    const uint32_t a = x[i], b = x[i + 4];
    x[i] = __byte_perm(a, b, 0x5410);
    x[i + 4] = __byte_perm(a, b, 0x7632);
  }
#pragma unroll
  for (int h = 0; h < 8; h += 4) {
#pragma unroll
    for (int i = h; i < h + 2; ++i) {                // rows p and p + 8
      const uint32_t a = x[i], b = x[i + 2];
      x[i] = __byte_perm(a, b, 0x6240);
      x[i + 2] = __byte_perm(a, b, 0x7351);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; i += 2) {                   // rows p and p + 4
    const uint32_t a = x[i], b = x[i + 1];
    x[i] = (a & 0x0F0F0F0Fu) | ((b << 4) & 0xF0F0F0F0u);
    x[i + 1] = ((a >> 4) & 0x0F0F0F0Fu) | (b & 0xF0F0F0F0u);
  }
  const bool hi2 = (lane & 2u) != 0u, hi1 = (lane & 1u) != 0u;
  const uint32_t keep2 = hi2 ? 0xCCCCCCCCu : 0x33333333u, rot2 = hi2 ? 30u : 2u;
  const uint32_t keep1 = hi1 ? 0xAAAAAAAAu : 0x55555555u, rot1 = hi1 ? 31u : 1u;
#pragma unroll
  for (int i = 0; i < 8; ++i) {                      // rows p and p + 2, then p and p + 1: across lanes
    const uint32_t y = __shfl_xor_sync(kFull, x[i], 2);
    x[i] = (x[i] & keep2) | (__funnelshift_l(y, y, rot2) & ~keep2);
    const uint32_t z = __shfl_xor_sync(kFull, x[i], 1);
    x[i] = (x[i] & keep1) | (__funnelshift_l(z, z, rot1) & ~keep1);
  }
}

// The folds: ldca (= dst's) |= transpose(OR of the sources' planes) | OR of the
// sources' LDCAs.  One source, the router itself, before a detect, export or
// copy; the merge of Sec. 4.2 folds all watch points' pending planes at once
// (16 routers of profile D3: one pass over 16 x 128 MiB of planes instead of 16
// folds and a merge of 16 LDCAs, 1,686 -> 443 us).
// planes: [ceil(W / 8)][k][8] words (W = LR * LC / 32 words per plane, 8-word
// chunks of the k planes side by side); ldca: [LR * LC][k / 32] words.
// A source's LDCA is read unless it is null or a flag beside it says that it is
// still all zero (FoldSrc).
__device__ __forceinline__ const uint32_t* live_ldca(const FoldSrc& s) {
  return (s.ldca == nullptr || (s.spilled != nullptr && *s.spilled == 0u)) ? nullptr : s.ldca;
}

// k < 256.  A warp task is 8 consecutive plane words J0 .. J0 + 7 (one 32-byte
// chunk of each plane it reads; 32 planes' chunks are 1 KiB of contiguous
// memory) times 4 consecutive LDC words: it transposes 32 planes x 32 LDCs per
// word and ORs the result into the lanes' LDC lines.
__global__ void __launch_bounds__(256, 2)
k_fold(FoldSrcs src, uint32_t* ldca, uint32_t W, uint32_t k_log2, const uint32_t* __restrict__ fresh,
       const uint32_t* __restrict__ pending) {
  if (pending != nullptr && *pending == 0u) return;
  const bool write_only = fresh != nullptr && *fresh == 0u;       // the LDCA is all zero: no read
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t wpl = 1u << (k_log2 - 5u);                       // words per LDC
  const uint64_t gwarp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarp = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint64_t n_groups = (W + 7) / 8;
  const uint32_t n_q = (wpl + 3) / 4;                              // groups of 4 LDC words
  for (uint64_t t = gwarp; t < n_groups * n_q; t += nwarp) {
    const uint64_t g = t / n_q;
    const uint32_t J0 = (uint32_t)(g * 8);
    const uint32_t nj = (W - J0) < 8u ? (W - J0) : 8u;
    const uint32_t q0 = (uint32_t)(t % n_q) * 4u;
    uint32_t x[4][8];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int j = 0; j < 8; ++j) x[u][j] = 0u;
    for (uint32_t s = 0; s < src.count; ++s) {
      const uint32_t* planes = src.s[s].planes;
      if (planes == nullptr) continue;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t q = q0 + u;
        const uint32_t keep = q < wpl ? kFull : 0u;     // planes past k (k < 128 only) read as zero
        uint32_t v[8];
        ld_chunk(planes + g * ((uint64_t)wpl * 256u) + (uint64_t)((q < wpl ? q : 0u) * 32u + lane) * 8u, v);
#pragma unroll
        for (int j = 0; j < 8; ++j) x[u][j] |= v[j] & keep;
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if ((uint32_t)j >= nj) break;
      uint32_t acc[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] = transpose32(x[u][j], lane);
      const uint64_t at = ((uint64_t)(J0 + j) * 32u + lane) * wpl;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (q0 + u >= wpl) break;
        uint32_t o = acc[u] | (write_only ? 0u : ldca[at + q0 + u]);
        for (uint32_t s = 0; s < src.count; ++s) {
          const uint32_t* l = live_ldca(src.s[s]);
          if (l != nullptr) o |= l[at + q0 + u];
        }
        ldca[at + q0 + u] = o;
      }
    }
  }
}

// k_fold8 (k >= 256): a warp task is 8 plane words J0 .. J0 + 7 times 8
// consecutive LDC words q0 .. q0 + 7 (256 planes).  Lane (q, s) = (lane / 4,
// lane mod 4) holds the chunks of planes 32 (q0 + q) + 4 i + s, i < 8: each of
// its 8 loads takes a whole 32-byte sector per lane and whole 128-byte lines
// per 4 lanes, and transpose8x4 leaves it word q0 + q of LDCs 32 J + 4 i + s,
// so a store covers 4 whole sectors.  Bounds: the 2 x 32 MiB it moves at
// profile D; with the 5-shuffle transpose per word and 16-byte accesses it
// took 22 us there, this way 12.5 us.
constexpr int kFold8Threads = 128;
template <bool kMulti>
__global__ void __launch_bounds__(kFold8Threads, kMulti ? 3 : 4)
k_fold8(FoldSrcs src, uint32_t* ldca, uint32_t W, uint32_t k_log2, const uint32_t* __restrict__ fresh,
        const uint32_t* __restrict__ pending) {
  if (pending != nullptr && *pending == 0u) return;
  const bool write_only = fresh != nullptr && *fresh == 0u;       // the LDCA is all zero: no read
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t wpl = 1u << (k_log2 - 5u);                       // words per LDC, >= 8
  const uint64_t gwarp = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint64_t nwarp = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint64_t n_groups = (W + 7) / 8;
  const uint32_t n_q = wpl / 8;                                    // groups of 8 LDC words
  const uint32_t q = lane >> 2, sub = lane & 3u;
  bool any_ldca = false;                                          // some source's LDCA holds bits
  if (kMulti)
    for (uint32_t s = 0; s < src.count; ++s) any_ldca |= live_ldca(src.s[s]) != nullptr;
  for (uint64_t t = gwarp; t < n_groups * n_q; t += nwarp) {
    const uint64_t g = t / n_q;
    const uint32_t J0 = (uint32_t)(g * 8);
    const uint32_t nj = (W - J0) < 8u ? (W - J0) : 8u;
    const uint32_t q0 = (uint32_t)(t % n_q) * 8u;
    const uint64_t chunk = g * ((uint64_t)wpl * 256u) + (uint64_t)((q0 + q) * 32u + sub) * 8u;
    uint32_t x[8][8];                                              // [i][j]
    if (!kMulti) {
#pragma unroll
      for (int i = 0; i < 8; ++i) ld_chunk(src.s[0].planes + chunk + i * 32, x[i]);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) x[i][j] = 0u;
      for (uint32_t s = 0; s < src.count; ++s) {
        const uint32_t* planes = src.s[s].planes;
        if (planes == nullptr) continue;
        uint32_t v[8][8];                                          // 8 loads in flight beside the 64 sums
#pragma unroll
        for (int i = 0; i < 8; ++i) ld_chunk(planes + chunk + i * 32, v[i]);
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) x[i][j] |= v[i][j];
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if ((uint32_t)j >= nj) break;
      uint32_t w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) w[i] = x[i][j];
      transpose8x4(w, lane);
      const uint64_t at = ((uint64_t)(J0 + j) * 32u + sub) * wpl + q0 + q;     // + 4 i LDCs
      if (!write_only) {
#pragma unroll
        for (int i = 0; i < 8; ++i) w[i] |= ldca[at + (uint64_t)(4 * i) * wpl];
      }
      if (kMulti && any_ldca) {
        for (uint32_t s = 0; s < src.count; ++s) {
          const uint32_t* l = live_ldca(src.s[s]);
          if (l == nullptr) continue;
#pragma unroll
          for (int i = 0; i < 8; ++i) w[i] |= l[at + (uint64_t)(4 * i) * wpl];
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) ldca[at + (uint64_t)(4 * i) * wpl] = w[i];
    }
  }
}

template <int THREADS, int STAGE, int TPR, int PER_SM>
cudaError_t bin_chunk(const DevParams& d, uint8_t* seav, uint32_t* ldca, const BinSrc& src,
                      const BinnedScratch& s, uint32_t cap, bool append, uint32_t rot, cudaStream_t st) {
  constexpr uint32_t bins = kBinRows;
  // the staging rows, the sampled-pair queue, the full rows' pairs, 2 counters per row
  const size_t bin_smem = (size_t)bins * STAGE * 4 + 32 * 4 + (size_t)(TPR * THREADS * kVec * 2 / 32 + 2 * kOver) * 8 +
                          (size_t)bins * 8;
  auto kern = k_bin<THREADS, STAGE, TPR, PER_SM>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bin_smem);
  if (e != cudaSuccess) return e;
  kern<<<s.ctas, THREADS, bin_smem, st>>>(d, seav, ldca, src, s.lists, s.counts, cap, append, rot, s.flags,
                                           s.prior);
  return cudaGetLastError();
}

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// The accumulator as a tensor [chunks][bins][8] of words; copies take `box`
// chunks of one plane.
cudaError_t plane_map(uint32_t* planes, uint32_t bins, uint32_t chunks, uint32_t box, CUtensorMap* map) {
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static std::atomic<void*> entry{nullptr};
  void* fn = entry.load(std::memory_order_acquire);
  if (fn == nullptr) {
    cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
    const cudaError_t e =
        cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found);
    if (e != cudaSuccess) return e;
    if (found != cudaDriverEntryPointSuccess || fn == nullptr) return cudaErrorSymbolNotFound;
    entry.store(fn, std::memory_order_release);
  }
  const cuuint64_t dims[3] = {8, bins, chunks}, strides[2] = {32, (cuuint64_t)bins * 32};
  const cuuint32_t boxes[3] = {8, 1, box}, steps[3] = {1, 1, 1};
  const CUresult r = reinterpret_cast<Encode>(fn)(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, planes, dims, strides, boxes,
                                                  steps, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                                  CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Dynamic shared memory of the largest k_apply: a plane of 2^20 bits, and the
// counts of k = 32's lists with the most binning blocks (167 KiB in all on 152
// SMs).  Every call sets the same limit, so that none lowers it under another
// thread's launch of the same kernel (what a launch needs follows k, LC and the
// staging shape).
int apply_smem_most() { return (1 << 17) + 2 * sm_count() * (int)sizeof(uint32_t) * (1 << (kBinRowsLog2 - 5u)); }

template <int LR, int THREADS, int LCL, int SPLIT = 1>
cudaError_t apply_round_t(const DevParams& d, const BinnedScratch& s, uint32_t cap, bool accumulate, cudaStream_t st) {
  const uint32_t bins = 1u << d.k_log2;
  const uint32_t chunks = ((((uint32_t)(LR / SPLIT) << d.lc_log2) >> 5) + 7u) / 8u;
  const uint32_t n_lists = s.ctas << (kBinRowsLog2 - d.k_log2);                    // of a plane
  const size_t apply_smem = ((size_t)chunks * 8u + n_lists) * sizeof(uint32_t);    // the rows, the lists' counts
  auto kern = k_apply<LR, THREADS, LCL, SPLIT>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, apply_smem_most());
  if (e != cudaSuccess) return e;
  // chunks of a copy: a block's chunks in equal boxes of at most 256
  uint32_t box = chunks < 256u ? chunks : 256u;
  while (chunks % box != 0u) --box;
  CUtensorMap map;
  if ((e = plane_map(s.planes, bins, chunks * (uint32_t)SPLIT, box, &map)) != cudaSuccess) return e;
  kern<<<bins * SPLIT, THREADS, apply_smem, st>>>(d, s.lists, s.counts, n_lists, cap, s.planes, map, box, accumulate,
                                             s.prior);
  return cudaGetLastError();
}

template <int LR, int THREADS>
cudaError_t apply_round_lc(const DevParams& d, const BinnedScratch& s, uint32_t cap, bool accumulate,
                           cudaStream_t st) {
  if constexpr (LR == 4) {            // the profiles' LDCA widths get constant shifts
    if (d.lc_log2 == 16) return apply_round_t<LR, THREADS, 16>(d, s, cap, accumulate, st);
    if (d.lc_log2 == 18) return apply_round_t<LR, THREADS, 18, 2>(d, s, cap, accumulate, st);
    if (d.lc_log2 == 14) return apply_round_t<LR, THREADS, 14>(d, s, cap, accumulate, st);
  }
  return apply_round_t<LR, THREADS, 0>(d, s, cap, accumulate, st);
}

template <int LR>
cudaError_t apply_round(const DevParams& d, const BinnedScratch& s, uint32_t cap, bool accumulate, cudaStream_t st) {
  return s.shape.apply_threads == 256 ? apply_round_lc<LR, 256>(d, s, cap, accumulate, st)
                                      : apply_round_lc<LR, 512>(d, s, cap, accumulate, st);
}

}  // namespace

bool binned_applicable(const DevParams& d) {
  const uint64_t plane_bits = (uint64_t)d.lr << d.lc_log2;
  return d.k_log2 >= 5 && d.k_log2 <= 10 && d.lc_log2 >= 5 && plane_bits <= (1ull << 20);
}

// The compiled staging shapes: {k_bin threads, row hips, tiles per flush
// round, blocks per SM, k_apply threads}.  Rows hold 4 x odd hips, so the
// flush's 16-byte row reads of 8 consecutive bins hit all 32 banks; a row
// holds the < 8 hips a flush leaves plus a round's arrivals with headroom
// (one block per SM: 2 tiles of 8K pairs, 16 per bin on average, 44-hip rows;
// two per SM: 2 tiles of 4K pairs, 20-hip rows).
constexpr BinShape kShapes[] = {
  {1024, 44, 2, 1, 512}, {1024, 44, 2, 1, 256},
  {512, 20, 2, 2, 512},  {512, 20, 2, 2, 256},
};

int binned_shape_count() { return (int)(sizeof(kShapes) / sizeof(kShapes[0])); }
BinShape binned_shape(int i) { return kShapes[(i >= 0 && i < binned_shape_count()) ? i : 0]; }

// List capacity for a round of n_pairs split into `chunks` binning launches:
// a block takes at most ceil(tiles / ctas) + 1 tiles per launch (the tile to
// block mapping rotates between launches), spread over the rows; 8 standard
// deviations plus 32 of headroom, so that only skewed inputs overflow.
uint32_t binned_list_cap(uint64_t n_pairs, const BinShape& shape, uint32_t ctas, uint32_t chunks) {
  const uint64_t tile = binned_tile_pairs(shape);
  const uint64_t tiles = (n_pairs + tile - 1) / tile;
  const uint64_t per_cta = (tiles + ctas - 1) / ctas + (chunks > 1 ? chunks : 1);
  const double m = (double)(per_cta * tile < n_pairs ? per_cta * tile : n_pairs) / kBinRows;
  uint64_t cap = (uint64_t)(m + 8.0 * sqrt(m + 1.0) + 32.0);
  cap = (cap + 7) & ~7ull;                                   // 32-byte list starts
  return (uint32_t)cap;
}

int binned_ctas(const BinShape& shape) { return sm_count() * (int)shape.per_sm; }

int binned_fold_grid() { return sm_count() * 8; }

cudaError_t launch_fold_multi(const DevParams& d, const FoldSrcs& src, uint32_t* ldca, int grid, cudaStream_t st,
                              const uint32_t* fresh, const uint32_t* pending) {
  const uint32_t words = (uint32_t)(((uint64_t)d.lr << d.lc_log2) >> 5);
  if (d.k_log2 < 8) k_fold<<<grid, 256, 0, st>>>(src, ldca, words, d.k_log2, fresh, pending);
  else if (src.count == 1 && src.s[0].planes && !src.s[0].ldca)
    k_fold8<false><<<2 * grid, kFold8Threads, 0, st>>>(src, ldca, words, d.k_log2, fresh, pending);
  else k_fold8<true><<<2 * grid, kFold8Threads, 0, st>>>(src, ldca, words, d.k_log2, fresh, pending);
  return cudaGetLastError();
}

cudaError_t launch_fold(const DevParams& d, const uint32_t* planes, uint32_t* ldca, int grid, cudaStream_t st,
                        const uint32_t* fresh, const uint32_t* pending) {
  FoldSrcs src{};
  src.s[0].planes = planes;
  src.count = 1;
  return launch_fold_multi(d, src, ldca, grid, st, fresh, pending);
}

BinSrc bin_src_one(const uint32_t* pairs, uint64_t n_pairs) {
  BinSrc src{};
  src.ptr[0] = pairs;
  src.n[0] = n_pairs;
  src.count = 1;
  return src;
}

cudaError_t binned_bin_chunk(const DevParams& d, uint8_t* seav, uint32_t* ldca, BinSrc& src,
                             const BinnedScratch& s, uint32_t cap, bool append, uint64_t* rot, cudaStream_t st) {
  if (src.count == 0) return cudaSuccess;
  // the list stride never exceeds what was allocated (hips past a full list go
  // to L2 REDs, so a smaller cap only costs speed)
  if (cap > s.cap_alloc) cap = s.cap_alloc;
  const BinShape& h = s.shape;
  // Whole tiles as long as they make whole rounds over the blocks; the rest in
  // small tiles, one for each block (whole warps of quads).  Streams of a
  // batched launch keep all their whole tiles.
  const uint64_t most = binned_tile_pairs(h) / 2;
  uint64_t quads = 0, full = 0;
  for (uint32_t b = 0; b < src.count; ++b) {
    // as k_bin counts them: a first pair off a 16-byte boundary is none of them
    const uint64_t head = src.n[b] != 0 && ((uintptr_t)src.ptr[b] & 15u) != 0u ? 1u : 0u, q = (src.n[b] - head) / 2;
    quads += q;
    full += q / most;
  }
  if (src.count == 1) full = full / s.ctas * s.ctas;
  src.full_max = src.count == 1 ? (uint32_t)full : 0xFFFFFFFFu;
  uint64_t small = (quads - full * most + s.ctas - 1) / s.ctas;
  small = (small + 31) & ~31ull;
  src.small_quads = (uint32_t)(small < 32 ? 32 : small > most ? most : small);
  const uint32_t r = (uint32_t)(*rot % s.ctas);
  *rot += full + s.ctas - 1;
  if (h.threads == 512) return bin_chunk<512, 20, 2, 2>(d, seav, ldca, src, s, cap, append, r, st);
  return bin_chunk<1024, 44, 2, 1>(d, seav, ldca, src, s, cap, append, r, st);
}

cudaError_t binned_apply_round(const DevParams& d, const BinnedScratch& s, uint32_t cap, bool accumulate,
                               cudaStream_t st) {
  if (cap > s.cap_alloc) cap = s.cap_alloc;          // the same clamp as the round's binning launches
  switch (d.lr) {
    case 1: return apply_round<1>(d, s, cap, accumulate, st);
    case 2: return apply_round<2>(d, s, cap, accumulate, st);
    case 3: return apply_round<3>(d, s, cap, accumulate, st);
    case 4: return apply_round<4>(d, s, cap, accumulate, st);
    case 5: return apply_round<5>(d, s, cap, accumulate, st);
    case 6: return apply_round<6>(d, s, cap, accumulate, st);
    case 7: return apply_round<7>(d, s, cap, accumulate, st);
    default: return apply_round<8>(d, s, cap, accumulate, st);
  }
}

uint32_t binned_tile_pairs(const BinShape& shape) { return shape.threads * (uint32_t)kVec * 2u; }

uint64_t binned_planes_bytes(const DevParams& d) {
  const uint64_t words = ((uint64_t)d.lr << d.lc_log2) >> 5;          // per plane
  return ((words + 7) / 8) * 8 * ((uint64_t)1 << d.k_log2) * sizeof(uint32_t);
}

cudaError_t launch_scan_binned(const DevParams& d, uint8_t* seav, uint32_t* ldca, const uint32_t* pairs,
                               uint64_t n_pairs, const BinnedScratch& s, cudaStream_t st) {
  uint64_t done = 0;
  bool accumulate = s.accumulate;
  while (done < n_pairs) {
    const uint64_t n = (n_pairs - done) < s.max_pairs ? (n_pairs - done) : s.max_pairs;
    const uint32_t cap = binned_list_cap(n, s.shape, s.ctas, 1);
    BinSrc src = bin_src_one(pairs + 2 * done, n);
    uint64_t rot = 0;
    cudaError_t e = binned_bin_chunk(d, seav, ldca, src, s, cap, false, &rot, st);
    if (e == cudaSuccess) e = binned_apply_round(d, s, cap, accumulate, st);
    if (e != cudaSuccess) return e;
    accumulate = true;
    done += n;
  }
  return cudaSuccess;
}

}  // namespace sp
