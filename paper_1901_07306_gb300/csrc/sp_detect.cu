// sp_detect.cu -- end-of-window restore and filter (Sec. 3.2-3.3, Sec. 4.2).
//
// k_detect: one warp per SEA (a block's warps share its part of the 2^r SEAs).
//   1. HSE(i): lanes test the SEs of a row for weight >= 3 (4 per lane per
//      32-bit load on rows of 128+ SEs) and a ballot/popc prefix compacts the
//      hot columns into a per-warp list in shared memory (Sec. 3.2, "hot SE").
//   2. CIS: lanes split the product HSE(0) x HSE(1); each lane then walks
//      rows 2 .. SR-1 depth first.  A partial tuple is dropped as soon as two
//      rows disagree on a shared LP bit (it then matches no LP) or the AND of
//      its SEs falls below weight 3 -- AND only clears bits, so the pruning
//      loses nothing against testing complete tuples (Sec. 3.2, SEU test).
//   3. A complete tuple fixes every LP bit (Eq. 3, coverage constraint);
//      ip = LP << r | RP goes to a per-warp queue.  Once enough are queued after
//      a turn of 32 pairs, or the warp has no SEA left, it tests the queued hosts
//      together: the LDC union (AND over the LR rows, Sec. 3.3) of one host is
//      read as LR lines of k bits spread over the lanes (one coalesced load per row and lane), z0 = k - popc by a
//      warp reduction.  The host survives when z0 <= Z_theta, the integer
//      form of Est >= threshold (Eq. 4).  A full queue falls back to the
//      same test in one lane.  For a sliding router (Sec. 5.2) a line word
//      is the union of the slice bits not yet committed and the 32 stamps of
//      the word that are active at the router's slice clock.
//   Survivors are collected per warp and appended as (ip << 32 | z0) keys, up
//   to 32 and more per atomic on the one result counter.
// k_sort_emit: sorts the keys by ip (ascending; ips are unique) and writes
//   sp_candidate records with est taken from a table of -k ln(z0 / k).  Up to
//   2,048 keys one block sorts them in shared memory (bitonic).  Above that,
//   the cooperative grid sorts runs of 2,048 keys in shared memory, one block
//   per run, then merges groups of up to 8 runs per round between grid-wide
//   barriers: each key's place in the merged run is its index in its own run
//   plus the number of keys of the group's other runs below it (binary searches
//   side by side).  The rounds alternate between the key buffer and the record
//   buffer (which holds at least as many bytes); the last one reads the key
//   buffer and writes the records.
#include <cooperative_groups.h>

#include <atomic>

#include "sp_internal.h"

namespace cg = cooperative_groups;

namespace sp {

namespace {

constexpr int kDetectWarps = 8;
constexpr int kDetectThreads = kDetectWarps * 32;
constexpr int kHostQueue = 256;                  // complete tuples queued per warp
constexpr uint32_t kFull = 0xFFFFFFFFu;
constexpr uint32_t kTestAt = 32;                  // queued hosts a warp tests together (fewer at its end)
constexpr int kPending = 64;                     // found keys a warp holds back before it appends them
// SEAs of a multiple of 16 bytes, up to 1 KiB, are staged in shared memory:
// two per warp, the next one copied while the current one is worked on
constexpr uint32_t kStagedSea = 1024;

// 16-byte asynchronous copy from global to shared memory (one per lane)
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory"); }

// How k_detect reads an SEA: rows from global memory, rows of a staged SEA, or
// a staged SEA of four rows of 128 SEs whose LP has at most 24 bits (profiles D,
// D3, S and K12).
enum class Form { kDirect, kStaged, kFour };
__host__ __device__ constexpr uint32_t list_bytes(Form form) { return form == Form::kFour ? 4u : 2u; }   // per SE

struct Found {
  uint64_t* keys;
  uint32_t cap;
  uint64_t max_join;
  DetectStatus* status;
};

// Where the LDCA test reads the bits of an LDC line.  Discrete window: the
// LDCA itself.  Sliding window (Sec. 5.2): word w of the window LDCA is the
// union of the bits of the slice sketch not yet committed (bits[w]) and the
// stamps of word w (32 bytes at stamps + 32 w) active at the router's clock.
// Only the lines of tested hosts are read, so a detect touches a few MB of
// stamps instead of streaming the whole counter pool.
struct LdcaRead {
  const uint32_t* bits;
  const uint4* stamps;
  uint32_t cur4, k4;
};

template <bool kSliding>
__device__ __forceinline__ uint32_t ldc_word(const LdcaRead& a, uint64_t w) {
  if (!kSliding) return a.bits[w];
  return a.bits[w] | active32(a.stamps[2 * w], a.stamps[2 * w + 1], a.cur4, a.k4);
}

// word index of the first word of host ip's LDC line in LDCA row i
__device__ __forceinline__ uint64_t ldc_line(const DevParams& d, uint32_t ip, uint32_t i) {
  const uint32_t col = (uint32_t)((uint64_t)mas(d.ha[2 + i], d.hb[2 + i], ip) >> (32u - d.lc_log2));
  return (uint64_t)((i << d.lc_log2) | col) << (d.k_log2 - 5u);
}

// z0 of one host in one lane: the rare fallback of a full queue, kept small
// (it is inlined into the join, whose registers count)
template <bool kSliding>
__device__ __forceinline__ uint32_t ldc_zeros(const DevParams& d, const LdcaRead& a, uint32_t ip) {
  const uint32_t wpl = 1u << (d.k_log2 - 5u);
  uint32_t ones = 0;
  if (!kSliding && wpl >= 4u) {
#pragma unroll 1
    for (uint32_t w = 0; w < wpl; w += 4) {
      uint4 u = make_uint4(kFull, kFull, kFull, kFull);
#pragma unroll 1
      for (uint32_t i = 0; i < d.lr; ++i) {
        const uint4 v = *reinterpret_cast<const uint4*>(a.bits + ldc_line(d, ip, i) + w);
        u.x &= v.x; u.y &= v.y; u.z &= v.z; u.w &= v.w;
      }
      ones += __popc(u.x) + __popc(u.y) + __popc(u.z) + __popc(u.w);
    }
    return (1u << d.k_log2) - ones;
  }
#pragma unroll 1
  for (uint32_t w = 0; w < wpl; ++w) {
    uint32_t u = kFull;
#pragma unroll 1
    for (uint32_t i = 0; i < d.lr; ++i) u &= ldc_word<kSliding>(a, ldc_line(d, ip, i) + w);
    ones += __popc(u);
  }
  return (1u << d.k_log2) - ones;
}

__device__ __forceinline__ void keep_host(uint32_t ip, uint32_t z0, uint32_t z_theta, const Found& f) {
  if (z0 <= z_theta) {
    const uint32_t slot = atomicAdd(&f.status->count, 1u);
    if (slot < f.cap) f.keys[slot] = ((uint64_t)ip << 32) | z0;
    else atomicOr(&f.status->overflow, 1u);
  }
}

// One complete, consistent tuple: count it against the join bound and queue
// its IP for the warp's LDCA test (tested here when the queue is full).
// Returns false when the detect must stop (a bound was hit).
template <bool kSliding>
__device__ __forceinline__ bool emit_lp(const DevParams& d, const LdcaRead& ldca,
                                        uint32_t rp, uint32_t lp, uint32_t z_theta,
                                        const Found& f, uint32_t& join_local,
                                        uint32_t* queue, uint32_t* queue_n) {
  if (++join_local == 64u) {
    const unsigned long long prev = atomicAdd(reinterpret_cast<unsigned long long*>(&f.status->join), 64ull);
    join_local = 0;
    if (prev + 64ull > f.max_join) { atomicOr(&f.status->overflow, 2u); return false; }
  }
  const uint32_t ip = (uint32_t)(((uint64_t)lp << d.r) | rp);
  const uint32_t at = atomicAdd(queue_n, 1u);
  if (at < (uint32_t)kHostQueue) queue[at] = ip;
  else keep_host(ip, ldc_zeros<kSliding>(d, ldca, ip), z_theta, f);
  return true;
}

// Found keys of one warp, held back in shared memory (n is warp-uniform).  One
// atomic per found host on the one result counter serialises in its L2 slice:
// 150,000 results took 378 us that way; appended 32 and more at a time the
// counter is out of the way.
struct Pending {
  uint64_t* keys;                                  // [kPending], shared memory
  uint32_t n;
};

// appends the warp's pending keys (all lanes call it)
__device__ __forceinline__ void flush_pending(Pending& p, const Found& f, uint32_t lane) {
  if (p.n == 0) return;
  __syncwarp();                                    // the keys are written
  uint32_t at = 0;
  if (lane == 0) at = atomicAdd(&f.status->count, p.n);
  at = __shfl_sync(kFull, at, 0);
  for (uint32_t i = lane; i < p.n; i += 32) {
    if (at + i < f.cap) f.keys[at + i] = p.keys[i];
    else atomicOr(&f.status->overflow, 1u);
  }
  p.n = 0;
  __syncwarp();                                    // the keys are read
}

// The warp's LDCA test of n queued hosts (all lanes call it).  A host's LR
// lines of wpl words are split over the lanes: with wpl >= 32 each lane
// takes every 32nd word of each line and two hosts go per pass; with
// wpl < 32 a pass takes 32 / wpl hosts, one word per lane.
template <bool kSliding>
__device__ void test_queue(const DevParams& d, const LdcaRead& ldca, const uint32_t* queue,
                           uint32_t n, uint32_t z_theta, const Found& f, Pending& pend, uint32_t lane) {
  const uint32_t wpl = 1u << (d.k_log2 - 5u);
  const uint32_t k = 1u << d.k_log2;
  if (wpl >= 32) {
    for (uint32_t q = 0; q < n; q += 2) {
      const bool two = q + 1 < n;
      const uint32_t ip0 = queue[q], ip1 = two ? queue[q + 1] : ip0;
      uint32_t ones0 = 0, ones1 = 0;
      for (uint32_t w = lane; w < wpl; w += 32) {
        uint32_t u0 = kFull, u1 = kFull;
        for (uint32_t i = 0; i < d.lr; ++i) {
          u0 &= ldc_word<kSliding>(ldca, ldc_line(d, ip0, i) + w);
          u1 &= ldc_word<kSliding>(ldca, ldc_line(d, ip1, i) + w);
        }
        ones0 += __popc(u0);
        ones1 += __popc(u1);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        ones0 += __shfl_xor_sync(kFull, ones0, o);
        ones1 += __shfl_xor_sync(kFull, ones1, o);
      }
      const bool keep0 = k - ones0 <= z_theta, keep1 = two && k - ones1 <= z_theta;   // warp-uniform
      if (lane == 0) {
        if (keep0) pend.keys[pend.n] = ((uint64_t)ip0 << 32) | (k - ones0);
        if (keep1) pend.keys[pend.n + (keep0 ? 1u : 0u)] = ((uint64_t)ip1 << 32) | (k - ones1);
      }
      pend.n += (keep0 ? 1u : 0u) + (keep1 ? 1u : 0u);
      if (pend.n > (uint32_t)kPending - 32u) flush_pending(pend, f, lane);
    }
  } else {
    const uint32_t per = 32u / wpl;                 // hosts per pass
    const uint32_t sub = lane / wpl, w = lane % wpl;
    for (uint32_t q0 = 0; q0 < n; q0 += per) {
      const uint32_t q = q0 + sub;
      uint32_t ones = 0;
      if (q < n) {
        const uint32_t ip = queue[q];
        uint32_t u = kFull;
        for (uint32_t i = 0; i < d.lr; ++i) u &= ldc_word<kSliding>(ldca, ldc_line(d, ip, i) + w);
        ones = __popc(u);
      }
      for (uint32_t o = wpl >> 1; o > 0; o >>= 1) ones += __shfl_xor_sync(kFull, ones, o);
      const bool keep = w == 0 && q < n && k - ones <= z_theta;      // at most 32 hosts a pass
      const uint32_t bal = __ballot_sync(kFull, keep);
      if (keep) pend.keys[pend.n + __popc(bal & ((1u << lane) - 1u))] = ((uint64_t)queue[q] << 32) | (k - ones);
      pend.n += __popc(bal);
      if (pend.n > (uint32_t)kPending - 32u) flush_pending(pend, f, lane);
    }
  }
}

// A warp's time goes to latencies (a core-link SEA has 1.4 hot SEs per row and
// one or two hosts to test): its SEA's copy, the join's dependent reads, one
// round trip to the LDC lines per test pass.  The next SEA is copied
// meanwhile; hosts are tested two a pass once kTestAt are queued or the warp
// is done, not one or two after every SEA; and the warps of a block take its
// SEAs from one counter, since SEAs differ.  Detect of 16 merged routers (65,536
// SEAs): 139 us with a test after every SEA and SEAs in a fixed stride, 121 this
// way, 106 with the four-row form and without spills (five blocks per SM there,
// 48 registers; six, at 40, gain nothing).
template <bool kSliding, Form kForm>
__global__ void __launch_bounds__(kDetectThreads, kForm == Form::kFour ? 5 : 4)
k_detect(DevParams d, const uint8_t* __restrict__ seav, LdcaRead ldca, const uint64_t* __restrict__ clock,
         uint32_t k_slices, uint32_t z_theta, Found f) {
  constexpr bool kStaged = kForm != Form::kDirect;
  extern __shared__ __align__(16) uint32_t s_dyn[];
  if (kSliding) {                                   // the window of the router's current slice
    ldca.cur4 = ((uint32_t)(*clock % 255u) + 1u) * 0x01010101u;
    ldca.k4 = k_slices * 0x01010101u;
  }
  __shared__ uint32_t s_queue_n[kDetectWarps], s_next;
  __shared__ uint64_t s_pending[kDetectWarps][kPending];
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
  uint32_t* queue = s_dyn + warp * kHostQueue;           // [kDetectWarps][kHostQueue] IPs
  uint32_t* queue_n = &s_queue_n[warp];
  // the warp's hot SEs, row by row: columns (uint16), with kFour whole entries (uint32)
  uint16_t* lists = reinterpret_cast<uint16_t*>(s_dyn + kDetectWarps * kHostQueue) + warp * d.sea_bytes;
  uint32_t* entries = s_dyn + kDetectWarps * kHostQueue + warp * 512u;
  Pending pend{s_pending[warp], 0u};
  if (lane == 0) *queue_n = 0;
  if (threadIdx.x == 0) s_next = 0;
  __syncthreads();
  const uint32_t n_sea = 1u << d.r;
  // the block's SEAs are blockIdx.x, blockIdx.x + gridDim.x, ...; a warp takes the next one
  auto next_sea = [&]() {
    uint32_t k = 0;
    if (lane == 0) k = atomicAdd(&s_next, 1u);
    k = __shfl_sync(kFull, k, 0);
    const uint64_t rp = (uint64_t)blockIdx.x + (uint64_t)k * gridDim.x;
    return rp < n_sea ? (uint32_t)rp : n_sea;
  };
  // staged SEAs (16-byte aligned SEAV and SEA size): the warp's two buffers
  // after the lists; 16 bytes per lane and copy by cp.async, one commit group
  // per SEA (empty past the last SEA, so that the count of groups in flight
  // stays fixed)
  uint8_t* buffers = reinterpret_cast<uint8_t*>(s_dyn + kDetectWarps * kHostQueue) +
                     (size_t)kDetectWarps * d.sea_bytes * list_bytes(kForm) + (size_t)warp * 2u * d.sea_bytes;
  auto stage_sea = [&](uint32_t rp, uint32_t slot) {
    if (rp < n_sea)
      for (uint32_t o = 16u * lane; o < d.sea_bytes; o += 512u)
        cp_async16(buffers + slot * d.sea_bytes + o, seav + (uint64_t)rp * d.sea_bytes + o);
    cp_async_commit();
  };
  // kFour: this lane's 16 SEs of an SEA are in row lane / 8; LP bits that row i
  // shares with the rows before it
  const uint32_t my_isb = kForm == Form::kFour ? d.isb[lane >> 3] : 0u;
  const uint32_t shared1 = d.cover[1] & d.cover[0], shared2 = d.cover[2] & (d.cover[0] | d.cover[1]);
  const uint32_t shared3 = d.cover[3] & (d.cover[0] | d.cover[1] | d.cover[2]);
  uint32_t rp = next_sea(), slot = 0;
  if (kStaged) stage_sea(rp, 0u);
  uint32_t join_local = 0;
  bool stop = false;
  // The pairs of HSE(0) x HSE(1) in turns of one per lane (body: a lane's join
  // from its pair on).  A turn that leaves kTestAt hosts queued is followed by
  // their test, so that an SEA with hundreds of tuples does not fill the queue:
  // a host that finds it full is tested in one lane, 32 round trips at k = 1,024
  // (profile S, five hosts an SEA: 742 us with the test after each SEA, 248 so;
  // ten an SEA 4,849 and 887).
  auto join_turns = [&](uint32_t total, auto body) {
    for (uint32_t first = 0; first < total && !stop; first += 32u) {
      if (first + lane < total) body(first + lane);
      __syncwarp();
      const uint32_t nq = __shfl_sync(kFull, lane == 0 ? *queue_n : 0u, 0);   // one value for all lanes
      if (nq >= kTestAt) {
        test_queue<kSliding>(d, ldca, queue, min(nq, (uint32_t)kHostQueue), z_theta, f, pend, lane);
        __syncwarp();
        if (lane == 0) *queue_n = 0;
        __syncwarp();
      }
      stop = __any_sync(kFull, stop);
    }
  };
  while (rp < n_sea && !stop) {
    // the join-bound flag (warp-uniform: lane 0 reads it, every lane sees its
    // value) is read here and tested after this SEA, so the read overlaps the
    // work; a warp stops at most one SEA later than the bound was hit
    const uint32_t ov = lane == 0 ? *reinterpret_cast<volatile uint32_t*>(&f.status->overflow) : 0u;
    const uint8_t* sea = seav + (uint64_t)rp * d.sea_bytes;
    uint32_t rp_next = n_sea;
    if (kStaged) {
      // the next SEA goes to the buffer this warp read last (every lane passed
      // the __syncwarp at the end of that turn); then wait for this SEA's copy
      // and make every lane's bytes visible
      rp_next = next_sea();
      stage_sea(rp_next, slot ^ 1u);
      cp_async_wait<1>();
      __syncwarp();
      sea = buffers + slot * d.sea_bytes;
      slot ^= 1u;
    }
    if (kForm == Form::kFour) {
      // 1. hot SEs: a lane looks at 16 SEs at once (weights side by side in a
      // word), a scan over the row's 8 lanes gives the places; an entry is the
      // column's LP bits (Eq. 3) with the SE above them
      const uint4 x = *reinterpret_cast<const uint4*>(sea + 16u * lane);
      const uint32_t w[4] = {x.x, x.y, x.z, x.w};
      uint32_t hot = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t y = w[j] - ((w[j] >> 1) & 0x55555555u);
        y = (y & 0x33333333u) + ((y >> 2) & 0x33333333u);
        y = (y + (y >> 4)) & 0x0F0F0F0Fu;
        y = ((y + 0x7D7D7D7Du) >> 7) & 0x01010101u;                // weight >= 3, a bit per byte
        hot |= (((y * 0x00204081u) >> 21) & 0xFu) << (4 * j);
      }
      uint32_t at = __popc(hot);
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, at, o, 8);
        if ((lane & 7u) >= (uint32_t)o) at += y;
      }
      const uint32_t row_n = __shfl_sync(kFull, at, 7, 8);
      if (!__any_sync(kFull, row_n == 0u)) {                       // a row without a hot SE: no tuple
        at -= __popc(hot);
        while (hot != 0u) {
          const uint32_t j = __ffs(hot) - 1u;
          hot &= hot - 1u;
          entries[(lane & 24u) * 16u + at++] =
              spread_idx(16u * (lane & 7u) + j, my_isb, d.L) | (uint32_t)sea[16u * lane + j] << 24;
        }
        const uint32_t n0 = __shfl_sync(kFull, row_n, 0), n1 = __shfl_sync(kFull, row_n, 8);
        const uint32_t n2 = __shfl_sync(kFull, row_n, 16), n3 = __shfl_sync(kFull, row_n, 24);
        __syncwarp();
        // 2. lanes split HSE(0) x HSE(1); a partial tuple is its LP bits with its
        // SEU above them, dropped as soon as shared bits differ or the SEU is light
        constexpr uint32_t kLp = 0x00FFFFFFu;
        const uint32_t total = n0 * n1;                            // <= 2^14: the float quotient is exact
        const float inv1 = 1.0f / (float)n1;
        join_turns(total, [&](uint32_t t) {
          const uint32_t t0 = (uint32_t)(((float)t + 0.5f) * inv1);
          const uint32_t e0 = entries[t0], e1 = entries[128u + t - t0 * n1];
          if (((e0 ^ e1) & shared1) != 0u) return;
          const uint32_t p = ((e0 | e1) & kLp) | (e0 & e1 & ~kLp);
          if (__popc(p >> 24) < 3) return;
          for (uint32_t i = 0; i < n2 && !stop; ++i) {
            const uint32_t e2 = entries[256u + i];
            const uint32_t q = ((p | e2) & kLp) | (p & e2 & ~kLp);
            if (((p ^ e2) & shared2) != 0u || __popc(q >> 24) < 3) continue;
            for (uint32_t k = 0; k < n3 && !stop; ++k) {
              const uint32_t e3 = entries[384u + k];
              if (((q ^ e3) & shared3) != 0u || __popc((q & e3) >> 24) < 3) continue;
              if (!emit_lp<kSliding>(d, ldca, rp, (q | e3) & kLp, z_theta, f, join_local, queue, queue_n)) stop = true;
            }
          }
        });
      }
    } else {
      // 1. hot SEs per row
      uint32_t cnt[8];
      bool empty = false;
      for (uint32_t i = 0; i < d.sr; ++i) {
        const uint32_t sc = 1u << d.ibn[i];
        const uint8_t* row = sea + d.row_off[i];
        uint32_t n = 0;
        if (sc >= 128 && ((uintptr_t)row & 3u) == 0) {
          // rows of 128+ SEs, word aligned: 4 SEs per lane per load; the list
          // is ordered by (byte of the word, lane), which only changes the order
          // in which candidates are tried
          for (uint32_t c0 = 0; c0 < sc; c0 += 128) {
            const uint32_t w = *reinterpret_cast<const uint32_t*>(row + c0 + 4 * lane);
  #pragma unroll
            for (uint32_t j = 0; j < 4; ++j) {
              const bool hot = __popc((w >> (8 * j)) & 0xFFu) >= 3;
              const uint32_t bal = __ballot_sync(kFull, hot);
              if (hot) lists[d.row_off[i] + n + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(c0 + 4 * lane + j);
              n += __popc(bal);
            }
          }
        } else {
          for (uint32_t c0 = 0; c0 < sc; c0 += 32) {
            const uint32_t c = c0 + lane;
            const bool hot = c < sc && __popc((uint32_t)row[c]) >= 3;
            const uint32_t bal = __ballot_sync(kFull, hot);
            if (hot) lists[d.row_off[i] + n + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)c;
            n += __popc(bal);
          }
        }
        cnt[i] = n;
        if (n == 0) {                                  // no tuple can cover this row: the SEA yields nothing
          empty = true;
          break;
        }
      }
      __syncwarp();
      if (!empty) {
        // 2. lanes split HSE(0) x HSE(1); depth-first over the remaining rows
        const uint32_t n1 = d.sr > 1 ? cnt[1] : 1u;
        const uint32_t total = cnt[0] * n1;                       // <= 2^24: exact as a float
        const float inv1 = 1.0f / (float)n1;
        join_turns(total, [&](uint32_t t) {
          // t / n1 and t mod n1: a float quotient is off by one at most
          uint32_t t0 = (uint32_t)((float)t * inv1);
          int t1 = (int)(t - t0 * n1);
          if (t1 < 0) { --t0; t1 += (int)n1; }
          if (t1 >= (int)n1) { ++t0; t1 -= (int)n1; }
          const uint32_t c0 = lists[d.row_off[0] + t0];
          uint32_t km = d.cover[0];
          uint32_t kv = spread_idx(c0, d.isb[0], d.L);
          uint32_t seu = sea[d.row_off[0] + c0];
          uint32_t start = 1;
          if (d.sr > 1) {
            const uint32_t c1 = lists[d.row_off[1] + (uint32_t)t1];
            const uint32_t v1 = spread_idx(c1, d.isb[1], d.L);
            if (((v1 ^ kv) & d.cover[1] & km) != 0u) return;
            seu &= sea[d.row_off[1] + c1];
            if (__popc(seu) < 3) return;
            km |= d.cover[1];
            kv |= v1;
            start = 2;
          }
          if (start == d.sr) {
            if (!emit_lp<kSliding>(d, ldca, rp, kv, z_theta, f, join_local, queue, queue_n)) stop = true;
            return;
          }
          uint32_t pos[8], skm[8], skv[8], sseu[8];
          int dd = (int)start;
          pos[dd] = 0; skm[dd] = km; skv[dd] = kv; sseu[dd] = seu;
          while (dd >= (int)start && !stop) {
            if (pos[dd] >= cnt[dd]) {
              if (--dd >= (int)start) ++pos[dd];
              continue;
            }
            const uint32_t c = lists[d.row_off[dd] + pos[dd]];
            const uint32_t v = spread_idx(c, d.isb[dd], d.L);
            const uint32_t s2 = sseu[dd] & sea[d.row_off[dd] + c];
            if (((v ^ skv[dd]) & d.cover[dd] & skm[dd]) == 0u && __popc(s2) >= 3) {
              if (dd == (int)d.sr - 1) {
                if (!emit_lp<kSliding>(d, ldca, rp, skv[dd] | v, z_theta, f, join_local, queue, queue_n)) stop = true;
                ++pos[dd];
              } else {
                const int nx = dd + 1;
                pos[nx] = 0; skm[nx] = skm[dd] | d.cover[dd]; skv[nx] = skv[dd] | v; sseu[nx] = s2;
                dd = nx;
              }
            } else {
              ++pos[dd];
            }
          }
        });
      }
    }
    __syncwarp();                                      // the lists and the SEA are read
    const bool bound = (__shfl_sync(kFull, ov, 0) & 2u) != 0u;
    stop = __any_sync(kFull, stop) || bound;
    rp = kStaged ? rp_next : next_sea();
  }
  if (*queue_n != 0u) test_queue<kSliding>(d, ldca, queue, min(*queue_n, (uint32_t)kHostQueue), z_theta, f, pend, lane);
  flush_pending(pend, f, lane);
  if (kStaged) cp_async_wait<0>();                 // no copy in flight at exit
  join_local = __reduce_add_sync(kFull, join_local);           // one atomic per warp
  if (lane == 0 && join_local) atomicAdd(reinterpret_cast<unsigned long long*>(&f.status->join), (unsigned long long)join_local);
}

// ---- sort + emit ----------------------------------------------------------
constexpr int kSortThreads = 1024;
constexpr uint32_t kRun = 2048;           // keys one block sorts in shared memory (16 KiB, two per thread)
constexpr int kWays = 8;                  // runs merged per round, at most

__device__ __forceinline__ void emit_record(uint64_t key, const double* est_table, sp_candidate* out) {
  sp_candidate c;
  c.ip = (uint32_t)(key >> 32);
  c.z0 = (uint32_t)key;
  c.est = est_table[c.z0];
  c.flags = c.z0 == 0u ? SP_FLAG_SATURATED : 0u;
  c.pad = 0u;
  *out = c;
}

// bitonic sort of m (a power of two, 2 <= m <= kRun) keys in shared memory,
// ascending; one compare-exchange per thread and stage.  A warp's 32
// compare-exchanges of a stage with stride <= 32 stay within its own 64 keys,
// so those stages need only the warp's own barrier.
__device__ void smem_bitonic(uint64_t* a, uint32_t m) {
  const uint32_t i = threadIdx.x;
  for (uint32_t size = 2; size <= m; size <<= 1) {
    for (uint32_t stride = size >> 1; stride > 0; stride >>= 1) {
      if (i < m / 2) {
        const uint32_t lo = 2 * i - (i & (stride - 1));
        const uint32_t hi = lo + stride;
        const bool up = (lo & size) == 0;
        const uint64_t x = a[lo], y = a[hi];
        if ((x > y) == up) { a[lo] = y; a[hi] = x; }
      }
      // the next stage's stride: stride / 2, or `size` at the start of the next size
      const uint32_t next = stride > 1 ? stride >> 1 : size;
      if (stride > 32u || next > 32u) __syncthreads();
      else __syncwarp();
    }
  }
  __syncthreads();
}

// Place of a key within its group of WAYS runs of w keys (a power of two;
// group = [base, end) of src, only its last run may be shorter): the keys of
// every run below it (its index, in its own).  The searches of the
// runs advance together, so a step costs one memory round trip for all; ips are
// unique, so a step compares the keys' upper words.
template <int WAYS>
__device__ __forceinline__ uint32_t merged_place(const uint64_t* src, uint32_t base, uint32_t end, uint32_t w,
                                                 uint64_t key) {
  const uint32_t ip = (uint32_t)(key >> 32);
  const uint32_t* ips = reinterpret_cast<const uint32_t*>(src) + 1;       // ips[2 g] = ip of key g
  uint32_t pos[WAYS];
#pragma unroll
  for (int q = 0; q < WAYS; ++q) pos[q] = 0;
  // after steps w, w / 2, ..., 1: pos[q] = keys of run q below key
  for (uint32_t step = w; step > 0; step >>= 1) {
#pragma unroll
    for (int q = 0; q < WAYS; ++q) {
      const uint32_t at = pos[q] + step;                           // 1-based rank tried
      const uint64_t g = (uint64_t)base + (uint64_t)q * w + at - 1;
      if (at <= w && g < end && ips[2 * g] < ip) pos[q] = at;
    }
  }
  uint32_t place = base;                                           // the own run counts the key's index in it
#pragma unroll
  for (int q = 0; q < WAYS; ++q) place += pos[q];
  return place;
}

// one merge round: groups of WAYS runs of w keys, to dst or (out != null) to the records
template <int WAYS>
__device__ __forceinline__ void merge_round(const uint64_t* src, uint64_t* dst, sp_candidate* out,
                                            const double* est_table, uint64_t n, uint64_t w) {
  const uint64_t group = w * WAYS;
  for (uint64_t i = (uint64_t)blockIdx.x * kSortThreads + threadIdx.x; i < n; i += (uint64_t)gridDim.x * kSortThreads) {
    const uint64_t base = i / group * group;
    const uint64_t end = base + group < n ? base + group : n;
    const uint64_t key = src[i];
    const uint32_t place = merged_place<WAYS>(src, (uint32_t)base, (uint32_t)end, (uint32_t)w, key);
    if (out) emit_record(key, est_table, out + place);
    else dst[place] = key;
  }
}

// Bounds: latency.  Up to kRun keys: 66 stages in one block (4.4 us at ~500
// keys).  Above: one run per block, then ceil(log8(runs)) merge rounds; 8 ways
// because a key's searches are then bound by their round trips, not by their
// instructions (a detect with 150,000 results: 234 us with 16 ways, 195 with 8).
// publish (may be null): receives the finished status, and the working status
// is zeroed for the next detect -- by one thread, once no block needs the
// count any more (with at most kRun keys the other blocks return whether they
// read the count or the zero).
__global__ void __launch_bounds__(kSortThreads)
k_sort_emit(uint64_t* keys, uint32_t cap, DetectStatus* status, const double* est_table,
            sp_candidate* out, DetectStatus* publish) {
  __shared__ uint64_t s_keys[kRun];
  const uint32_t n = min(status->count, cap);        // the same for every block (above kRun)
  const uint32_t tid = threadIdx.x;
  auto hand_over = [&]() {
    if (publish != nullptr && blockIdx.x == 0 && tid == 0) {
      *publish = *status;
      *status = DetectStatus{0u, 0u, 0ull};
    }
  };
  if (n <= kRun) {                                  // one block, in shared memory
    if (blockIdx.x != 0) return;
    __syncthreads();                                // every thread of the block has the count
    hand_over();
    if (n == 0) return;
    uint32_t m = 2;
    while (m < n) m <<= 1;
    for (uint32_t i = tid; i < m; i += kSortThreads) s_keys[i] = i < n ? keys[i] : ~0ull;
    __syncthreads();
    smem_bitonic(s_keys, m);
    for (uint32_t i = tid; i < n; i += kSortThreads) emit_record(s_keys[i], est_table, out + i);
    return;
  }
  cg::grid_group grid = cg::this_grid();
  uint64_t* tmp = reinterpret_cast<uint64_t*>(out);  // cap records of 24 bytes hold n keys
  uint32_t rounds = 0;
  for (uint64_t w = kRun; w < n; w *= kWays) ++rounds;   // >= 1
  // 1. sorted runs, written where an odd number of rounds ends up reading the key buffer
  uint64_t* src = (rounds & 1u) ? keys : tmp;
  uint64_t* dst = (rounds & 1u) ? tmp : keys;
  const uint32_t runs = (n + kRun - 1) / kRun;
  for (uint32_t r = blockIdx.x; r < runs; r += gridDim.x) {
    const uint32_t base = r * kRun;
    const uint32_t len = min(kRun, n - base);
    for (uint32_t i = tid; i < kRun; i += kSortThreads) s_keys[i] = i < len ? keys[base + i] : ~0ull;
    __syncthreads();
    smem_bitonic(s_keys, kRun);
    for (uint32_t i = tid; i < len; i += kSortThreads) src[base + i] = s_keys[i];
    __syncthreads();
  }
  // 2. merge rounds; the last one reads the key buffer and writes the records
  for (uint64_t w = kRun; w < n; w *= kWays) {
    grid.sync();
    if (w == kRun) hand_over();                                    // every block has the count
    const uint64_t left = (n + w - 1) / w;                         // runs
    sp_candidate* to = left <= kWays ? out : nullptr;
    if (left <= 2) merge_round<2>(src, dst, to, est_table, n, w);
    else if (left <= 4) merge_round<4>(src, dst, to, est_table, n, w);
    else merge_round<kWays>(src, dst, to, est_table, n, w);
    uint64_t* t = src;
    src = dst;
    dst = t;
  }
}

}  // namespace

namespace {

// Blocks of a kernel that a device holds at a given dynamic shared memory
// size, asked once: the last answer is kept per kernel, packed into one word
// (device + 1, shared memory, blocks), so that any thread may ask.
template <typename Kernel>
cudaError_t resident_blocks(Kernel kern, int threads, uint32_t smem, std::atomic<uint64_t>& last, int* blocks) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t key = ((uint64_t)(dev + 1) << 48) | ((uint64_t)smem << 24);
  const uint64_t was = last.load(std::memory_order_acquire);
  if ((was & ~0xFFFFFFull) == key) {
    *blocks = (int)(was & 0xFFFFFFull);
    return cudaSuccess;
  }
  int sms = 0, per_sm = 0;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem)) != cudaSuccess) return e;
  *blocks = sms * per_sm;
  last.store(key | (uint64_t)*blocks, std::memory_order_release);
  return cudaSuccess;
}

// dynamic shared memory of k_detect for the largest SEA (4,096 bytes, unstaged); staged ones need less
constexpr int kDetectSmemMost = kDetectWarps * (kHostQueue * 4 + 4096 * 2);

template <bool kSliding, Form kForm>
cudaError_t detect_launch_form(const DevParams& d, const uint8_t* seav, const LdcaRead& ldca, const uint64_t* clock,
                                 uint32_t k_slices, uint32_t z_theta, const Found& f, cudaStream_t s) {
  const size_t smem = (size_t)kDetectWarps * kHostQueue * sizeof(uint32_t) +
                      (size_t)kDetectWarps * d.sea_bytes * list_bytes(kForm) +
                      (kForm != Form::kDirect ? (size_t)kDetectWarps * 2u * d.sea_bytes : 0u);
  auto kern = k_detect<kSliding, kForm>;
  // the limit is set to the same constant once per device: no call lowers it under another's launch
  static std::atomic<uint64_t> limit_set{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 64 || !((limit_set.load(std::memory_order_acquire) >> dev) & 1u)) {
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kDetectSmemMost)) != cudaSuccess)
      return e;
    if (dev < 64) limit_set.fetch_or(1ull << dev, std::memory_order_release);
  }
  static std::atomic<uint64_t> resident{0};
  int most = 0;
  if ((e = resident_blocks(kern, kDetectThreads, (uint32_t)smem, resident, &most)) != cudaSuccess) return e;
  if (most < 1) return cudaErrorInvalidConfiguration;
  const uint64_t n_sea = 1ull << d.r;
  uint64_t grid = (n_sea + kDetectWarps - 1) / kDetectWarps;
  if (grid > (uint64_t)most) grid = (uint64_t)most;
  kern<<<(unsigned)grid, kDetectThreads, smem, s>>>(d, seav, ldca, clock, k_slices, z_theta, f);
  return cudaGetLastError();
}

template <bool kSliding>
cudaError_t detect_launch(const DevParams& d, const uint8_t* seav, const LdcaRead& ldca, const uint64_t* clock,
                          uint32_t k_slices, uint32_t z_theta, uint64_t* keys, uint32_t cap, uint64_t max_join,
                          DetectStatus* status, cudaStream_t s) {
  const Found f{keys, cap, max_join, status};
  // staged SEAs need 16-byte copies; above kStagedSea the buffers would cost blocks
  if ((d.sea_bytes & 15u) != 0u || d.sea_bytes > kStagedSea || ((uintptr_t)seav & 15u) != 0u)
    return detect_launch_form<kSliding, Form::kDirect>(d, seav, ldca, clock, k_slices, z_theta, f, s);
  const bool four = d.sr == 4 && d.L <= 24 && d.ibn[0] == 7 && d.ibn[1] == 7 && d.ibn[2] == 7 && d.ibn[3] == 7;
  return four ? detect_launch_form<kSliding, Form::kFour>(d, seav, ldca, clock, k_slices, z_theta, f, s)
              : detect_launch_form<kSliding, Form::kStaged>(d, seav, ldca, clock, k_slices, z_theta, f, s);
}

}  // namespace

cudaError_t launch_detect(const DevParams& d, const uint8_t* seav, const uint32_t* ldca,
                          uint32_t z_theta, uint64_t* keys, uint32_t cap, uint64_t max_join,
                          DetectStatus* status, cudaStream_t s) {
  return detect_launch<false>(d, seav, LdcaRead{ldca, nullptr, 0u, 0u}, nullptr, 0u, z_theta, keys, cap, max_join,
                              status, s);
}

cudaError_t launch_detect_sliding(const DevParams& d, const uint8_t* seav, const uint32_t* ldca,
                                  const uint8_t* st_ldca, const uint64_t* clock, uint32_t k, uint32_t z_theta,
                                  uint64_t* keys, uint32_t cap, uint64_t max_join, DetectStatus* status,
                                  cudaStream_t s) {
  const LdcaRead a{ldca, reinterpret_cast<const uint4*>(st_ldca), 0u, 0u};
  return detect_launch<true>(d, seav, a, clock, k, z_theta, keys, cap, max_join, status, s);
}

cudaError_t launch_sort_emit(uint64_t* keys, uint32_t cap, DetectStatus* status,
                             const double* est_table, uint32_t /*k_log2*/,
                             sp_candidate* out, DetectStatus* publish, cudaStream_t s) {
  // a cooperative grid (every block resident) of at most one block per SM,
  // and no more blocks than runs of the largest count
  static std::atomic<uint64_t> resident{0};
  int most = 0;
  cudaError_t e = resident_blocks(k_sort_emit, kSortThreads, 0u, resident, &most);
  if (e != cudaSuccess) return e;
  if (most < 1) return cudaErrorInvalidConfiguration;
  const uint32_t max_runs = (cap + kRun - 1) / kRun;
  const unsigned grid = max_runs < (uint32_t)most ? (max_runs ? max_runs : 1u) : (unsigned)most;
  void* args[] = {&keys, &cap, &status, &est_table, &out, &publish};
  e = cudaLaunchCooperativeKernel((const void*)k_sort_emit, dim3(grid), dim3(kSortThreads), args, 0, s);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace sp
