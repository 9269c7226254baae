// Execution of a batch of literals and copies by a thread block: what the
// Snappy and Zstandard decoders share once they know a batch's elements.
//
// Copies name earlier output, possibly of the same batch, so executing
// elements one after another makes every batch a chain.  Here the unit is
// the output byte: every byte of a chunk finds its element (a bit per
// element start, counted by the warp that holds the word), takes its value
// from the literals or from output before the chunk, or notes which earlier
// byte of the chunk it repeats; the few that do (5-12% on the eight-column
// table's pages) then follow those notes to a byte that has a value (their
// depth is the number of copies stacked on one another, not the number of
// elements).  The chunk is assembled in a shared-memory ring of recent
// output and leaves it as 16-byte stores.  Bound by instruction issue (about
// 45 per byte and lane) and, where copies reach past the ring, by L2 latency:
// four words are in flight per warp.
//
// Positions are "virtual": output offset + (output address mod 32), so that
// words of 32 positions are aligned in memory and in the ring alike.
#pragma once
#include <stdint.h>

#include "dev_util.cuh"

namespace pqi {

constexpr uint32_t LZ_LIT = 0x80000000u;  // LzRec::src of a literal: LZ_LIT | index of its first byte
constexpr uint16_t LZ_ROOT = 0xffffu;     // the byte has its value

struct LzRec {
  uint32_t start;  // virtual position of the element's first byte
  uint32_t src;    // literal: LZ_LIT | literal index; copy: back offset
};

// The last of elements [0, n), n <= 1024, that starts at or before `v` (one
// warp: two 32-way steps).
__device__ __forceinline__ int lz_find(const LzRec* rec, int n, uint32_t v, int lane) {
  const uint32_t hi = __ballot_sync(0xffffffffu, 32 * lane < n && rec[32 * lane].start <= v);
  const int b = hi ? 32 * (__popc(hi) - 1) : 0;
  const uint32_t lo = __ballot_sync(0xffffffffu, b + lane < n && rec[b + lane].start <= v);
  return b + (lo ? __popc(lo) - 1 : 0);
}

// (Not inlined: inlined, the division is computed for every byte.)
static __device__ __noinline__ uint32_t lz_mod(uint32_t a, uint32_t b) { return a % b; }

// Output [vb, ve) of one batch of n elements (n <= 1024, in order, the first
// at vb, none empty).  mask: bit i of word w set where an element starts at
// position 32 (vb / 32 + w) + i.  kChunk: positions resolved at a time, 32
// words per warp at most; kRing >= 2 kChunk, a power of two.  `notes` holds
// kChunk entries.  lit(i) is the address of literal byte i (shared or
// global memory).  The ring holds no position
// below vfloor.  Block-collective; ends without a barrier (the caller's next
// one orders it before mask or rec are written again).
template <int kThreads, uint32_t kChunk, uint32_t kRing, typename Lit>
__device__ void lz_run(const LzRec* rec, int n, const uint32_t* mask, uint8_t* ring, uint16_t* notes, uint8_t* vout,
                       uint32_t vb, uint32_t ve, uint32_t vfloor, Lit lit) {
  constexpr uint32_t RM = kRing - 1;
  constexpr int kWarps = kThreads / 32;
  constexpr int U = 4;  // words in flight
  static_assert(kRing >= 2 * kChunk && (kRing & RM) == 0 && kChunk / 32 <= 32 * kWarps, "chunk and ring sizes");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t le = 0xffffffffu >> (31 - lane);  // lanes up to this one
  for (uint32_t c0 = vb; c0 < ve;) {
    const uint32_t ca = c0 & ~31u;
    const uint32_t c1 = ve - ca < kChunk ? ve : ca + kChunk;
    uint32_t rlo = c1 > kRing ? c1 - kRing : 0u;  // older positions may have lost their ring slot
    rlo = rlo > vfloor ? rlo : vfloor;
    // the warp's words [wa, wa + nw): lane k holds word k's start bits and
    // the element that its first position belongs to (the one before the
    // batch, -1, when the batch starts inside the word)
    const uint32_t words = (c1 - ca + 31) >> 5, per = (words + kWarps - 1) / kWarps;
    const uint32_t wa = per * warp;
    const int nw = wa < words ? static_cast<int>(words - wa < per ? words - wa : per) : 0;
    const uint32_t w0 = (ca >> 5) - (vb >> 5) + wa;
    uint32_t mym = 0;
    int mye = 0;
    if (nw > 0) {
      if (lane < nw) mym = mask[w0 + lane];
      const uint32_t v0 = ca + 32 * wa;
      const int first = v0 < vb ? -1 : lz_find(rec, n, v0, lane);
      // (a start at the word's own bit 0 is the element found)
      const int cnt = __popc(lane == 0 ? mym & ~1u : mym);
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      mye = first + incl - cnt + ((mym & 1u) && lane > 0 ? 1 : 0);
      mym &= ~1u;
    }
    uint32_t pend = 0;  // bit k: word k holds unresolved bytes
    for (int k0 = 0; k0 < nw; k0 += U) {
      uint32_t note[U];
      const uint8_t* from[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = k0 + u;
        const uint32_t m = __shfl_sync(0xffffffffu, mym, k & 31);
        const int e = __shfl_sync(0xffffffffu, mye, k & 31) + __popc(m & le);
        const uint32_t v = ca + 32 * (wa + k) + lane;
        note[u] = LZ_ROOT;
        from[u] = ring;
        if (k < nw && v >= c0 && v < c1) {
          const LzRec r = rec[e];
          const uint32_t d = v - r.start;
          if (r.src & LZ_LIT) {
            from[u] = lit((r.src & ~LZ_LIT) + d);
          } else {
            // a copy longer than its offset repeats the bytes before its start
            const uint32_t s = d < r.src ? v - r.src : r.start - r.src + lz_mod(d, r.src);
            if (s >= c0)
              note[u] = s - ca;
            else
              from[u] = s >= rlo ? ring + (s & RM) : vout + s;
          }
        }
      }
      uint32_t byte[U];
#pragma unroll
      for (int u = 0; u < U; ++u) byte[u] = *from[u];  // shared or global memory, all in flight together
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = k0 + u;
        const uint32_t v = ca + 32 * (wa + k) + lane;
        if (k < nw && v >= c0 && v < c1) {
          if (note[u] == LZ_ROOT) ring[v & RM] = static_cast<uint8_t>(byte[u]);
          notes[v - ca] = static_cast<uint16_t>(note[u]);
        }
        if (__any_sync(0xffffffffu, note[u] != LZ_ROOT)) pend |= 1u << (k & 31);
      }
    }
    __syncthreads();
    // each pass follows up to 8 notes per byte and shortens them (notes of
    // other bytes shorten meanwhile), so chains of any depth inside the
    // chunk end within kChunk / 8 passes, in practice in the first
    for (uint32_t pass = 0; pass <= kChunk / 8; ++pass) {
      uint32_t left = 0;
      for (int k0 = 0; k0 < nw; k0 += U) {
        if (!((pend >> k0) & ((1u << U) - 1u))) continue;
        uint32_t q[U], nx[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const uint32_t v = ca + 32 * (wa + k0 + u) + lane;
          q[u] = k0 + u < nw && v >= c0 && v < c1 ? notes[v - ca] : LZ_ROOT;
        }
        uint32_t first[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          first[u] = q[u];
          nx[u] = q[u] != LZ_ROOT ? notes[q[u]] : LZ_ROOT;
        }
        for (int s = 0; s < 8; ++s) {
          bool open = false;
#pragma unroll
          for (int u = 0; u < U; ++u) open |= nx[u] != LZ_ROOT;
          if (!__any_sync(0xffffffffu, open)) break;
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (nx[u] != LZ_ROOT) {
              q[u] = nx[u];
              nx[u] = notes[q[u]];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const uint32_t v = ca + 32 * (wa + k0 + u) + lane;
          if (first[u] != LZ_ROOT) {
            if (nx[u] == LZ_ROOT) ring[v & RM] = ring[(ca + q[u]) & RM];
            if (q[u] != first[u]) notes[v - ca] = static_cast<uint16_t>(q[u]);
          }
          if (__any_sync(0xffffffffu, nx[u] != LZ_ROOT)) left |= 1u << (k0 + u);
        }
      }
      pend = left;
      if (!__syncthreads_or(pend != 0)) break;
    }
    for (uint32_t x = (c0 & ~15u) + 16 * threadIdx.x; x < c1; x += 16 * kThreads) {
      if (x >= c0 && x + 16 <= c1) {
        *reinterpret_cast<uint4*>(vout + x) = *reinterpret_cast<const uint4*>(ring + (x & RM));
      } else {
        for (uint32_t k = x < c0 ? c0 : x; k < x + 16 && k < c1; ++k) vout[k] = ring[k & RM];
      }
    }
    c0 = c1;
  }
}

// src[0, n) to dst by all warps of the block, a slice each.  (Not inlined:
// a dozen 16-byte values in flight would cost the decoders registers.)
// kReadOnly: the source is not written by the running kernel.
template <int kThreads, bool kReadOnly = true>
__device__ __noinline__ void lz_block_copy(uint8_t* dst, const uint8_t* src, uint32_t n) {
  constexpr uint32_t kWarps = kThreads / 32;
  const uint64_t per = ((static_cast<uint64_t>(n) + kWarps * 16 - 1) / (kWarps * 16)) * 16;
  const uint64_t b = per * (threadIdx.x >> 5), e = b + per < n ? b + per : n;
  if (b < e) warp_copy<kReadOnly>(dst + b, src + b, e - b, threadIdx.x & 31);
}

// ------------------------------------------------------------------ groups of element pairs

// Workspace of lz_pairs: kThreads <= 512 threads, kChunk and kRing as for
// lz_run; a batch writes up to 4 kChunk bytes.
template <int kThreads_, uint32_t kChunk_, uint32_t kRing_>
struct __align__(16) LzPairs {
  static constexpr int kThreads = kThreads_;
  static constexpr uint32_t kChunk = kChunk_, kRing = kRing_, kOut = 4 * kChunk_;
  uint8_t ring[kRing];
  LzRec rec[2 * kThreads];
  uint16_t notes[kChunk];
  uint32_t mask[kOut / 32 + 2];
  uint32_t out_at[kThreads + 1], cnt_at[kThreads + 1];  // sums before each thread's pair
  uint32_t len[2][kThreads], src[2][kThreads];
  uint64_t tmp64[32];
  uint32_t tmp[32];
};
constexpr uint32_t LZ_LONG = 4096;  // pairs with an element of this length are written on their own

// One element of n bytes at output position v; v moves past it.  A long
// literal is copied straight to the output when plain(i, n, v) gives the
// address of its bytes (null: they overlap their place, or repeat), others
// go through lz_run in pieces.  kReadOnly: the literals are not written by the
// running kernel.
template <bool kReadOnly, typename W, typename Lit, typename Plain>
__device__ void lz_one(W& S, uint8_t* vout, uint32_t& v, uint32_t& vfloor, uint32_t src, uint32_t n, Lit lit,
                       Plain plain) {
  if (n >= LZ_LONG && (src & LZ_LIT)) {
    const uint8_t* from = plain(src & ~LZ_LIT, n, v);
    if (from) {
      lz_block_copy<W::kThreads, kReadOnly>(vout + v, from, n);
      v += n;
      vfloor = v;
      __syncthreads();
      return;
    }
  }
  while (n) {
    const uint32_t c = n < LZ_LONG ? n : LZ_LONG;
    for (uint32_t w = threadIdx.x; w < LZ_LONG / 32 + 2; w += W::kThreads) S.mask[w] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
      S.rec[0] = LzRec{v, src};
      S.mask[0] = 1u << (v & 31);
    }
    __syncthreads();
    lz_run<W::kThreads, W::kChunk, W::kRing>(S.rec, 1, S.mask, S.ring, S.notes, vout, v, v + c, vfloor, lit);
    __syncthreads();
    v += c;
    n -= c;
    if (src & LZ_LIT) src += c;
  }
}

// The pairs of threads [0, nb), one after another: element a (len_a bytes
// from src_a, an LzRec source), then element b; empty ones have length 0.
// Returns with v past the output.  Block-collective.
template <bool kReadOnly, typename W, typename Lit, typename Plain>
__device__ void lz_pairs(W& S, int nb, uint8_t* vout, uint32_t& v, uint32_t& vfloor, uint32_t len_a, uint32_t src_a,
                         uint32_t len_b, uint32_t src_b, Lit lit, Plain plain) {
  const int tid = threadIdx.x;
  if (tid >= nb) len_a = len_b = 0;
  const bool alone = len_a >= LZ_LONG || len_b >= LZ_LONG;
  uint32_t total, count;
  const uint32_t o_at = block_exclusive_sum<uint32_t>(len_a + len_b, S.tmp, &total);
  const uint32_t c_at = block_exclusive_sum<uint32_t>((len_a ? 1u : 0u) + (len_b ? 1u : 0u) + (alone ? 1u << 16 : 0u),
                                                      S.tmp, &count);
  S.out_at[tid] = o_at;
  S.cnt_at[tid] = c_at;
  S.len[0][tid] = len_a;
  S.len[1][tid] = len_b;
  S.src[0][tid] = src_a;
  S.src[1][tid] = src_b;
  if (tid == 0) {
    S.out_at[W::kThreads] = total;
    S.cnt_at[W::kThreads] = count;
  }
  __syncthreads();
  for (int i0 = 0; i0 < nb;) {
    // as many pairs as fit a batch, up to one that is written on its own
    const bool fits = tid >= i0 && tid < nb && S.out_at[tid + 1] - S.out_at[i0] <= W::kOut - 64 &&
                      (S.cnt_at[tid + 1] >> 16) == (S.cnt_at[i0] >> 16);
    const int k = __syncthreads_count(fits);
    if (k == 0) {
      lz_one<kReadOnly>(S, vout, v, vfloor, S.src[0][i0], S.len[0][i0], lit, plain);
      lz_one<kReadOnly>(S, vout, v, vfloor, S.src[1][i0], S.len[1][i0], lit, plain);
      i0 += 1;
      continue;
    }
    const int i1 = i0 + k;
    const uint32_t bytes = S.out_at[i1] - S.out_at[i0];
    if (bytes) {
      for (uint32_t w = tid; w < (bytes + 31) / 32 + 2 && w < W::kOut / 32 + 2; w += W::kThreads) S.mask[w] = 0;
      __syncthreads();
      if (tid >= i0 && tid < i1) {
        uint32_t a = v + o_at - S.out_at[i0];
        uint32_t e = (c_at - S.cnt_at[i0]) & 0xffffu;
        if (len_a) {
          S.rec[e++] = LzRec{a, src_a};
          atomicOr(S.mask + ((a >> 5) - (v >> 5)), 1u << (a & 31));
          a += len_a;
        }
        if (len_b) {
          S.rec[e] = LzRec{a, src_b};
          atomicOr(S.mask + ((a >> 5) - (v >> 5)), 1u << (a & 31));
        }
      }
      __syncthreads();
      lz_run<W::kThreads, W::kChunk, W::kRing>(S.rec, static_cast<int>((S.cnt_at[i1] - S.cnt_at[i0]) & 0xffffu), S.mask,
                                               S.ring, S.notes, vout, v, v + bytes, vfloor, lit);
      v += bytes;
      __syncthreads();
    }
    i0 = i1;
  }
}

}  // namespace pqi
