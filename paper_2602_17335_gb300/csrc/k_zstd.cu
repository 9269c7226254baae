// Zstandard page decompression (the codec the paper's Section 2 lists beside
// Snappy), one thread block per page.  The page jobs have the Snappy jobs'
// layout (verbatim V2 level prefix, then the frames); jobs of another codec
// are skipped (the Snappy kernel runs over the same job list).
//
// Of a compressed block, what one thread used to do end to end (265 ms for a
// 2^20-row eight-column table, all of it latency) is divided as follows:
//
//  Huffman literals  every thread decodes its share of a stream's bits from
//      a guessed code boundary; Huffman codes fall into step within a few
//      dozen symbols, so after two to four rounds of handing each share's true
//      end to the next thread every start is right (at worst one more share
//      per round, a serial decode).  A second pass writes the symbols.
//  tables            Huffman and FSE tables are filled by the block: symbol
//      ranks by ballots instead of a running index.
//  sequences         the FSE chain stays serial, but only the chain: one
//      thread follows the three states and the bit position from staged bits
//      (three table words, whose bit counts add up in one sum, and one bit
//      window a sequence) and notes where each sequence starts.  A thread
//      per sequence then reads its values; repeat offsets are resolved by a
//      scan over the maps that sequences apply to the last three offsets.
//      (With all of it on one thread a sequence took 1240 cycles.)
//  execution         literal runs and matches are written by lz_run
//      (lz_exec.cuh), all bytes of a batch in parallel.
//
// Bound by the latency of a page's blocks, one after another: of the 530,000
// cycles of a 128 KB block of 112,000 literals and 800 sequences, 195,000 are
// byte writing, 130,000 Huffman literals, 85,000 the sequence chain, 77,000
// tables.  Pages run side by side, two a multiprocessor (2^20-row eight-column
// table: 2.5 ms a read).
//
// Huffman and RLE literals are kept in the page's own output tail until the
// sequences use them (the output never passes the unread ones: what is still
// to be written is at least what is unread); raw literals stay in the input.
#include <stddef.h>

#include "dev_util.cuh"
#include "lz_exec.cuh"
#include "snappy_job.h"
#include "zstd_dec.cuh"

namespace pqi {
namespace {

constexpr int ZT = 512;                 // threads
constexpr int Z_HW = 3;                 // the Huffman weights' slot among the FSE builds
constexpr int Z_SEQ = ZT;               // sequences decoded at a time, one a thread
constexpr int Z_UNROLL = 8;             // sequences the chain follows between checks of the bit position
constexpr int Z_PAD = 28;               // words of zeros before the staged bytes: the chain reads up to
                                        // 8 * 89 + 128 bits below the stream's start before such a check
constexpr uint32_t Z_BITS = (Z_SEQ * 89 + 7) / 8 + 64;  // staged bytes: a sequence takes 89 bits at most

struct __align__(16) ZBlock {
  LzPairs<ZT, 8192, 32768> lz;
  // sequence tables (literal lengths, offsets, match lengths), by state
  uint32_t step[3][512];       // extra bits | state bits << 8 | next state base << 16, a state
                               // being the byte offset of its row in `step`
  uint32_t base[3][512];       // value without its extra bits
  __align__(16) uint32_t bits[Z_PAD + (Z_BITS + 16) / 4];  // staged input: words of zeros, then 16-byte aligned
  uint16_t huf[2048];          // code bits << 8 | symbol, by the next huf_bits bits
  __align__(4) uint8_t weights[256];
  ZFse hw[64];                 // table of the Huffman weights
  // FSE builds: the three sequence tables, and the Huffman weights' (Z_HW)
  uint8_t sym[4][512];         // symbol of each state
  uint8_t rank_sym[4][512];    // symbols in the order they are spread
  int16_t norm[4][64];
  uint16_t next[4][64];
  int32_t mode[3], nsym[4], al[4];
  int32_t huf_bits, n_weights;
  uint32_t wcount[16], wstart[16], wrank[16];
  uint8_t order[256];          // Huffman: symbols by weight, then value
  int32_t end[ZT];             // Huffman: where each thread's share ends
  uint32_t tmp[32];
  int32_t err;
  uint32_t used;
  // a group of sequences
  uint32_t at[Z_SEQ], states[Z_SEQ];   // bit position and states each starts with
  uint32_t map[ZT / 32][3];            // the warps' maps of the repeat offsets
  uint32_t rep[3];
  int32_t bad;
  uint32_t sl, so, sm, pos;            // the chain between groups
};

// The error any thread has noted in S.err by now, the same for all threads.
// Block-collective, with a barrier: the word is read on one side of it and
// decided on by all threads at once.  (Read by each thread after a plain
// barrier, a slow warp could see a later error than the others, return where
// they went on, and leave the block's barriers out of step for its next pages.)
__device__ __forceinline__ int z_error(const ZBlock& S) { return __syncthreads_or(S.err) ? S.err : 0; }

__device__ __forceinline__ uint64_t z_load8(const uint8_t* p) { return ld_unaligned_g(p, 8); }

// A backward bit stream read through 64-bit windows: p's bits [0, pos) are
// unread, the next ones are the highest.  The loads touch aligned 8-byte
// words around the stream (the page is followed by readable slack).
struct ZRead {
  const uint8_t* p;
  int32_t pos;
};
// The 64 bits below pos with the next bit at the top (at least 57 of them
// valid unless fewer are left; zeros below the stream's start).
__device__ __forceinline__ uint64_t z_top(const ZRead& r) {
  if (r.pos <= 0) return 0;
  const int32_t b1 = (r.pos + 7) >> 3;
  if (b1 >= 8) return z_load8(r.p + b1 - 8) << (8 * b1 - r.pos);
  uint64_t v = 0;
  for (int i = 0; i < b1; ++i) v |= static_cast<uint64_t>(__ldg(r.p + i)) << (8 * i);
  return v << (64 - r.pos);
}
__device__ __forceinline__ uint32_t z_take(uint64_t& w, uint32_t n) {  // n <= 32 top bits
  const uint32_t v = static_cast<uint32_t>((w >> 1) >> (63 - n));
  w <<= n;
  return v;
}
__device__ __forceinline__ uint32_t z_bits(ZRead& r, uint32_t n) {
  uint64_t w = z_top(r);
  r.pos -= static_cast<int32_t>(n);
  return z_take(w, n);
}
__device__ __forceinline__ bool z_open(ZRead& r, const uint8_t* p, uint32_t len) {
  if (len == 0) return false;
  const uint32_t last = __ldg(p + len - 1);
  if (last == 0) return false;
  r.p = p;
  r.pos = static_cast<int32_t>((len - 1) * 8) + z_hb(last);
  return true;
}

// Stages bytes [from, to) of the input into S.bits, 16-byte aligned; returns
// the bit index of byte `from` there.  Block-collective, without barriers.
// Reads up to 15 bytes before and 16 after the range.
__device__ __forceinline__ uint32_t z_stage(ZBlock& S, const uint8_t* from, const uint8_t* to) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(from) & ~uintptr_t(15);
  const uint32_t n = static_cast<uint32_t>(((reinterpret_cast<uintptr_t>(to) + 15) & ~uintptr_t(15)) - a) / 16;
  uint4* d = reinterpret_cast<uint4*>(S.bits + Z_PAD);
  for (uint32_t i = threadIdx.x; i < n && 16 * i + 16 <= sizeof(S.bits) - 4 * Z_PAD; i += ZT)
    d[i] = __ldg(reinterpret_cast<const uint4*>(a) + i);
  return 32 * Z_PAD + 8 * static_cast<uint32_t>(reinterpret_cast<uintptr_t>(from) - a);
}
// The 32 staged bits from bit index b on, and those below bit index b (b >= 32).
__device__ __forceinline__ uint32_t z_from(const ZBlock& S, uint32_t b) {
  return __funnelshift_r(S.bits[b >> 5], S.bits[(b >> 5) + 1], b & 31);
}
__device__ __forceinline__ uint32_t z_below(const ZBlock& S, uint32_t b) { return z_from(S, b - 32); }
__device__ __forceinline__ uint32_t z_high(uint32_t w, uint32_t n) { return __funnelshift_l(w, 0u, n); }  // n < 32 top bits

// Normalized counts of a table description at staged bit index b0, `len`
// bytes long (z_read_norm from shared memory, in words).  Returns 0 or an
// error; *used = bytes consumed.
__device__ int z_norm(const ZBlock& S, uint32_t b0, uint32_t len, int max_al, int max_sym, int16_t* norm, int32_t* nsym,
                      int32_t* al, uint32_t* used) {
  if (len == 0) return ZE_FSE;
  const uint32_t end = b0 + 8 * len;
  uint32_t b = b0;
  const int a = static_cast<int>(z_from(S, b) & 15u) + 5;
  b += 4;
  if (a > max_al) return ZE_FSE;
  int32_t remaining = 1 << a;
  int s = 0;
  while (remaining > 0) {
    if (s >= max_sym) return ZE_FSE;
    const uint32_t nv = static_cast<uint32_t>(remaining) + 2;  // values 0 .. remaining + 1
    const int nbits = z_hb(nv - 1) + 1;                        // 2^nbits >= nv
    const uint32_t spare = (1u << nbits) - nv, half = 1u << (nbits - 1);
    const uint32_t w = z_from(S, b);
    uint32_t value = w & (half - 1);
    if (value < spare) {
      b += nbits - 1;
    } else {
      value = w & (2 * half - 1);
      if (value >= half) value -= spare;
      b += nbits;
    }
    if (b > end) return ZE_FSE;
    const int prob = static_cast<int>(value) - 1;
    norm[s++] = static_cast<int16_t>(prob);
    remaining -= prob == -1 ? 1 : prob;
    if (prob == 0) {
      for (;;) {
        const uint32_t rep = z_from(S, b) & 3u;
        b += 2;
        if (b > end) return ZE_FSE;
        for (uint32_t r = 0; r < rep; ++r) {
          if (s >= max_sym) return ZE_FSE;
          norm[s++] = 0;
        }
        if (rep != 3) break;
      }
    }
  }
  if (remaining < 0) return ZE_FSE;
  *nsym = s;
  *al = a;
  *used = (b - b0 + 7) / 8;
  return ZE_OK;
}

// ------------------------------------------------------------------ tables

// Decoding table of distribution `which` (S.norm, S.nsym, S.al), one warp:
// S.sym per state, then its bits and base.  emit(state, symbol, bits, base).
template <typename Emit>
__device__ int z_fse_table(ZBlock& S, int which, int max_log, Emit emit) {
  const int lane = threadIdx.x & 31;
  const int al = S.al[which], size = 1 << al, nsym = S.nsym[which];
  if (al > max_log || nsym > 64) return ZE_FSE;
  const int16_t* norm = S.norm[which];
  uint8_t* sym = S.sym[which];
  uint8_t* rs = S.rank_sym[which];
  uint16_t* next = S.next[which];
  // symbols in spreading order; those of probability "below one" take the
  // last states instead
  int n_low = 0, spread = 0;
  for (int s0 = 0; s0 < nsym; s0 += 32) {
    const int s = s0 + lane;
    const int c = s < nsym ? norm[s] : 0;
    const uint32_t low = __ballot_sync(0xffffffffu, c == -1);
    if (c == -1) {
      const int st = size - 1 - (n_low + __popc(low & ((1u << lane) - 1u)));
      if (st >= 0) sym[st] = static_cast<uint8_t>(s);
    }
    n_low += __popc(low);
    if (s < nsym) next[s] = static_cast<uint16_t>(c == -1 ? 1 : c);
    int incl = c > 0 ? c : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const int from = spread + incl - (c > 0 ? c : 0);
    for (uint32_t m = __ballot_sync(0xffffffffu, c > 0); m; m &= m - 1) {
      const int k = __ffs(m) - 1;
      const int f = __shfl_sync(0xffffffffu, from, k), cc = __shfl_sync(0xffffffffu, c, k);
      for (int i = lane; i < cc; i += 32)
        if (f + i < size) rs[f + i] = static_cast<uint8_t>(s0 + k);
    }
    spread += __shfl_sync(0xffffffffu, incl, 31);
  }
  __syncwarp();
  if (n_low + spread != size) return ZE_FSE;
  const int high = size - 1 - n_low;
  const uint32_t step = (size >> 1) + (size >> 3) + 3, msk = size - 1;
  int done = 0;
  for (int i0 = 0; i0 < size; i0 += 32) {
    const uint32_t p = (static_cast<uint32_t>(i0 + lane) * step) & msk;
    const bool ok = i0 + lane < size && static_cast<int>(p) <= high;
    const uint32_t m = __ballot_sync(0xffffffffu, ok);
    if (ok) sym[p] = rs[done + __popc(m & ((1u << lane) - 1u))];
    done += __popc(m);
  }
  __syncwarp();
  // state st is the k-th of its symbol: x = count + k
  for (int s0 = 0; s0 < size; s0 += 32) {
    const int st = s0 + lane;
    const bool on = st < size;
    const int s = on ? sym[st] : 64 + lane;
    const uint32_t same = __match_any_sync(0xffffffffu, s);
    uint32_t x = 0;
    if (on) x = next[s] + __popc(same & ((1u << lane) - 1u));
    __syncwarp();
    if (on && lane == 31 - __clz(same)) next[s] = static_cast<uint16_t>(next[s] + __popc(same));
    __syncwarp();
    if (on) {
      const int nb = al - z_hb(x);
      emit(st, s, nb, (x << nb) - size);
    }
  }
  __syncwarp();
  return ZE_OK;
}

// The sequence table row of `state`: symbol s, nb state bits, next base.
__device__ __forceinline__ void z_entry(ZBlock& S, int which, int state, uint32_t s, uint32_t nb, uint32_t next) {
  uint32_t base;
  int extra;
  if (which == 1) {
    base = 1u << s;
    extra = static_cast<int>(s);
  } else if (which == 0) {
    z_ll(s, &base, &extra);
  } else {
    z_ml(s, &base, &extra);
  }
  S.base[which][state] = base;
  S.step[which][state] = static_cast<uint32_t>(extra) | (nb << 8) | ((4 * next + 2048 * which) << 16);
}

// The Huffman tree description at p[0, len): S.huf, S.huf_bits; S.used bytes.
// Returns 0 or an error.  Block-collective.
__device__ int z_huffman_tree(ZBlock& S, const uint8_t* p, uint32_t len) {
  const int tid = threadIdx.x;
  if (tid < 16) S.wcount[tid] = 0;
  for (int i = tid; i < 256; i += ZT) S.weights[i] = 0;
  const uint32_t head = len ? __ldg(p) : 0u;
  const uint32_t b0 = z_stage(S, p, p + (len < 130 ? len : 130));
  __syncthreads();
  if (head >= 128) {
    const int n = static_cast<int>(head) - 127;
    const uint32_t nbytes = (n + 1) / 2;
    if (1 + nbytes <= len) {
      for (int i = tid; i < n; i += ZT) {
        const uint32_t b = __ldg(p + 1 + i / 2);
        S.weights[i] = static_cast<uint8_t>((i & 1) ? (b & 15) : (b >> 4));
      }
    }
    if (tid == 0) {
      S.n_weights = n;
      S.used = 1 + nbytes;
      if (1 + nbytes > len) S.err = ZE_HUF;
    }
  } else if (tid < 32) {
    // weights under an FSE table of their own
    int bad = len == 0 || head == 0 || 1 + head > len;
    uint32_t u = 0;
    if (!bad) {
      if (tid == 0) {
        bad = z_norm(S, b0 + 8, head, 6, 16, S.norm[Z_HW], &S.nsym[Z_HW], &S.al[Z_HW], &u);
      }
      bad = __shfl_sync(0xffffffffu, bad, 0);
      __syncwarp();
    }
    if (!bad)
      bad = z_fse_table(S, Z_HW, 6, [&](int st, int s, int nb, uint32_t base) {
        S.hw[st] = ZFse{static_cast<uint8_t>(s), static_cast<uint8_t>(nb), static_cast<uint16_t>(base)};
      });
    if (!bad && tid == 0) {
      int n = 0;
      const uint32_t first = b0 + 8 * (1 + u), stop = b0 + 8 * (1 + head);  // the backward stream's bits
      const uint32_t last = u < head ? z_from(S, stop - 8) & 0xffu : 0u;
      if (last == 0) {
        bad = 1;
      } else {
        // (bits below the stream's start are read as whatever is staged
        // there: a stream that takes such bits ends right there)
        uint32_t b = stop - 8 + z_hb(last);
        const uint32_t al = S.al[Z_HW];
        uint32_t s1 = z_high(z_below(S, b), al), s2 = z_high(z_below(S, b - al), al);
        b -= 2 * al;
        const auto short_of = [&](uint32_t take) { return b < first + take; };
        if (short_of(0)) bad = 1;
        while (!bad) {
          if (n > 253) {
            bad = 1;
            break;
          }
          ZFse e = S.hw[s1];
          S.weights[n++] = e.sym;
          if (short_of(e.nbits)) {
            S.weights[n++] = S.hw[s2].sym;
            break;
          }
          s1 = e.base + z_high(z_below(S, b), e.nbits);
          b -= e.nbits;
          e = S.hw[s2];
          S.weights[n++] = e.sym;
          if (short_of(e.nbits)) {
            S.weights[n++] = S.hw[s1].sym;
            break;
          }
          s2 = e.base + z_high(z_below(S, b), e.nbits);
          b -= e.nbits;
        }
      }
      S.n_weights = n;
      S.used = 1 + head;
    }
    if (bad) S.err = ZE_HUF;
  }
  if (const int e = z_error(S)) return e;
  // the last symbol's weight is what is left to the next power of two
  const int n = S.n_weights;
  if (tid < 32) {
    uint32_t total = 0;
    bool bad = n >= 256 || n < 1;
    for (int i = tid; i < n && i < 256; i += 32) {
      const uint32_t w = S.weights[i];
      if (w > 11) bad = true;
      else if (w) total += 1u << (w - 1);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    bad = __any_sync(0xffffffffu, bad) || total == 0;
    if (tid == 0) {
      if (!bad) {
        const int mb = z_hb(total) + 1;
        const uint32_t rest = (1u << mb) - total;
        if (mb > 11 || (rest & (rest - 1))) {
          bad = true;
        } else {
          S.weights[n] = static_cast<uint8_t>(z_hb(rest) + 1);
          S.huf_bits = mb;
        }
      }
      if (bad) S.err = ZE_HUF;
    }
  }
  if (const int e = z_error(S)) return e;
  const int ns = n + 1, mb = S.huf_bits;
  if (tid < ns && S.weights[tid]) atomicAdd(&S.wcount[S.weights[tid]], 1u);
  __syncthreads();
  if (tid == 0) {
    uint32_t at = 0, rank = 0;
    for (int w = 1; w <= 12; ++w) {
      S.wstart[w] = at;
      S.wrank[w] = rank;
      at += w <= mb ? S.wcount[w] << (w - 1) : 0u;
      rank += S.wcount[w];
    }
    if (at != (1u << mb)) S.err = ZE_HUF;  // (a weight above mb would be left out)
  }
  if (const int e = z_error(S)) return e;
  if (tid < ns && S.weights[tid]) {
    // its place among the symbols of its weight
    const uint32_t w = S.weights[tid], same = w * 0x01010101u;
    const uint32_t* w4 = reinterpret_cast<const uint32_t*>(S.weights);
    uint32_t before = 0;
    for (int i = 0; i < tid / 4; ++i) before += __popc(__vcmpeq4(w4[i], same)) >> 3;
    before += __popc(__vcmpeq4(w4[tid / 4], same) & ((1u << (8 * (tid & 3))) - 1u)) >> 3;
    S.order[S.wrank[w] + before] = static_cast<uint8_t>(tid);
  }
  __syncthreads();
  for (uint32_t i = tid; i < (1u << mb); i += ZT) {
    int w = 1;
    while (w < mb && S.wstart[w + 1] <= i) ++w;
    const uint32_t sym = S.order[S.wrank[w] + ((i - S.wstart[w]) >> (w - 1))];
    S.huf[i] = static_cast<uint16_t>(((mb + 1 - w) << 8) | sym);
  }
  __syncthreads();
  return ZE_OK;
}

// ------------------------------------------------------------------ Huffman literals

// Symbols of one stream whose codes start at staged bits (lim, pos]: each is
// given to put(symbol, true); returns the position after the last.  A window
// holds 64 bits, enough for five codes of at most 12, and is reloaded by all
// lanes of a warp at once (where each lane ran dry, every symbol waited for
// some lane's load: 570 cycles a symbol); past lim a lane decodes on without
// moving, as a branch a symbol cost more than that.
template <typename Put>
__device__ __forceinline__ int32_t z_huf_share(const uint16_t* huf, int mb, const uint32_t* words, int32_t pos,
                                               int32_t lim, Put put) {
  const int drop = 32 - mb;
  while (pos > lim) {
    const uint32_t* q = words + (pos >> 5);
    const uint32_t q0 = q[0], q1 = q[-1], q2 = q[-2];
    uint32_t hi = __funnelshift_r(q1, q0, pos), lo = __funnelshift_r(q2, q1, pos);
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const uint32_t e = huf[hi >> drop];
      const bool live = pos > lim;
      const uint32_t n = live ? e >> 8 : 0u;
      put(e & 0xffu, live);
      hi = __funnelshift_l(lo, hi, n);
      lo <<= n;
      pos -= static_cast<int32_t>(n);
    }
  }
  return pos;
}

// The same, only counted: (position after the last, symbols).  (Not inlined:
// three copies of it cost the kernel registers.)
__device__ __noinline__ int2 z_huf_count(const uint16_t* huf, int mb, const uint32_t* words, int32_t pos, int32_t lim) {
  int32_t m = 0;
  const int32_t end = z_huf_share(huf, mb, words, pos, lim, [&](uint32_t, bool live) { m += live; });
  return make_int2(end, m);
}

// The literal streams into out.  The streams are decoded from the top, a part
// at a time that fits the idle workspace of lz_pairs (gathered from the input
// by 32 lanes in 32 lines, a window of a warp took 64 L1 wavefronts: 205,000
// cycles a block of 112,000 literals, now 130,000, a third of them the
// scattered stores), every thread a share of a part.
// A share is decoded in three pieces, so that a thread whose start moves need
// only decode until it meets a piece's end that it had reached before.
// Returns 0 or an error.  Block-collective.
__device__ int z_huffman_literals(ZBlock& S, const ZHufStreams& hs, uint8_t* out) {
  const int tid = threadIdx.x;
  const int per = ZT / hs.n, k = tid / per, i = tid % per;
  const int mb = S.huf_bits;
  constexpr uint32_t kPad = 4;  // words of padding below a stream's bytes
  uint32_t* const work = reinterpret_cast<uint32_t*>(S.lz.rec);
  constexpr uint32_t kWork = (sizeof(S.lz) - offsetof(decltype(S.lz), rec)) / 64 * 16;  // words
  const uint32_t room = kWork / hs.n / 4 * 4;  // words of a stream (16-byte aligned)
  uint32_t* const words = work + room * k;
  const int32_t most = static_cast<int32_t>((room - kPad - 16) * 32 / per);  // bits of a share
  ZRead r{nullptr, 0};
  const bool ok = z_open(r, hs.p[k], hs.len[k]);
  if (!ok && i == 0) S.err = ZE_STREAM;
  int32_t top = ok ? r.pos : 0;  // bits left
  uint32_t written = 0;          // symbols of the stream before the part
  const uint32_t want = hs.cnt[k];
  const int lane = tid & 31, warp = tid >> 5;
  for (;;) {
    int32_t share = (top + per - 1) / per > 128 ? (top + per - 1) / per : 128;
    share = share < most ? share : most;
    const int32_t low = top - share * per > 0 ? top - share * per : 0;
    // bytes [from, (top + 7) / 8): the part's and, below it, those its last codes reach into
    const int32_t from = low / 8 > 16 ? low / 8 - 16 : 0;
    const uintptr_t a = reinterpret_cast<uintptr_t>(r.p + from) & ~uintptr_t(15);
    if (top > 0) {
      const uint32_t n16 = static_cast<uint32_t>((reinterpret_cast<uintptr_t>(r.p) + (top + 7) / 8 + 15 - a) / 16);
      uint4* d = reinterpret_cast<uint4*>(words + kPad);
      for (uint32_t q = i; q < n16; q += per) d[q] = __ldg(reinterpret_cast<const uint4*>(a) + q);
    }
    // stream bit b is staged bit b + base
    const int32_t base = static_cast<int32_t>(8 * (reinterpret_cast<intptr_t>(r.p) - static_cast<intptr_t>(a))) + 32 * kPad;
    __syncthreads();
    const int32_t hi = top - i * share > 0 ? top - i * share : 0;
    int32_t start = hi;
    const int32_t lim = hi - share > low ? hi - share : low;
    int32_t met[3] = {-1, -1, -1};  // where each piece ended, and its symbols
    uint32_t cnt[3] = {0, 0, 0};
    const int32_t cut[3] = {hi - (hi - lim) / 4, hi - (hi - lim) / 2, lim};
    int32_t end = start;
    bool todo = true;
    // a round fixes at least one more share of every stream
    for (int round = 0; round <= per; ++round) {
      if (todo) {
        int32_t q = start;
        bool same = false;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          if (!same) {
            const int2 r2 = z_huf_count(S.huf, mb, words, q + base, cut[c] + base);
            q = r2.x - base;
            cnt[c] = static_cast<uint32_t>(r2.y);
            same = q == met[c];
            met[c] = q;
          }
        }
        end = met[2];
        S.end[tid] = end;
      }
      __syncthreads();
      const int32_t s = i == 0 ? start : S.end[tid - 1];
      todo = s != start;
      start = s;
      if (!__syncthreads_or(todo)) break;
    }
    const uint32_t count = cnt[0] + cnt[1] + cnt[2];
    // each share's place among its stream's symbols
    uint32_t incl = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) S.tmp[warp] = incl;
    __syncthreads();
    uint32_t before = written + incl - count, total = 0;
    for (int w = k * per / 32; w < (k + 1) * per / 32; ++w) {
      before += w < warp ? S.tmp[w] : 0u;
      total += S.tmp[w];
    }
    const int32_t next = S.end[k * per + per - 1];  // where the part's codes end
    if (i == 0 && (total > want - written || (low == 0 && (next != 0 || written + total != want)))) S.err = ZE_STREAM;
    if (const int e = z_error(S)) return e;
    // bytes up to the first 4-byte boundary, words, bytes
    uint8_t* o = out + hs.out[k] + before;
    uint32_t skip = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(o) & 3), fill = skip, word = 0;
    o -= skip;
    z_huf_share(S.huf, mb, words, start + base, lim + base, [&](uint32_t b, bool live) {
      word |= (live ? b : 0u) << (8 * fill);
      fill += live;
      if (fill == 4) {
        if (skip) {
          for (uint32_t q = skip; q < 4; ++q) o[q] = static_cast<uint8_t>(word >> (8 * q));
          skip = 0;
        } else {
          *reinterpret_cast<uint32_t*>(o) = word;
        }
        o += 4;
        word = fill = 0;
      }
    });
    for (uint32_t q = skip; q < fill; ++q) o[q] = static_cast<uint8_t>(word >> (8 * q));
    written += total;
    top = low > 0 && next > 0 ? next : 0;
    if (i == 0 && low > 0 && next <= 0 && (next != 0 || written != want)) S.err = ZE_STREAM;
    if (!__syncthreads_or(top > 0)) break;
  }
  return z_error(S);
}

// ------------------------------------------------------------------ a compressed block

// Compressed block src[0, len): its output from `out` on (frame output starts
// at out0) into dst[0, dst_len).  The ring holds nothing below vfloor.
// Moves out past the block's output; returns 0 or an error.  Block-collective.
__device__ __forceinline__ int z_block(ZBlock& S, const uint8_t* src, uint32_t len, uint8_t* dst, uint64_t& out,
                                       uint64_t out0, uint64_t dst_len, uint32_t& vfloor) {
  const int tid = threadIdx.x;
  // literals section
  if (len == 0) return ZE_LIT;
  const uint32_t b0 = __ldg(src), type = b0 & 3, sf = (b0 >> 2) & 3;
  uint32_t hlen, regen, csize = 0;
  if (type < 2) {
    hlen = (sf & 1) == 0 ? 1 : (sf == 1 ? 2 : 3);
    if (len < hlen) return ZE_LIT;
    const uint32_t h = z_le(src, static_cast<int>(hlen));
    regen = hlen == 1 ? b0 >> 3 : h >> 4;
  } else {
    const uint32_t bits = sf < 2 ? 10 : sf == 2 ? 14 : 18;
    hlen = sf < 2 ? 3 : sf == 2 ? 4 : 5;
    if (len < hlen) return ZE_LIT;
    uint64_t h = 0;
    for (int i = static_cast<int>(hlen) - 1; i >= 0; --i) h = (h << 8) | __ldg(src + i);
    regen = static_cast<uint32_t>((h >> 4) & ((1u << bits) - 1));
    csize = static_cast<uint32_t>((h >> (4 + bits)) & ((1u << bits) - 1));
  }
  if (regen > dst_len - out) return ZE_SIZE;
  const uint8_t* lit = dst + (dst_len - regen);  // Huffman literals: in the output's tail
  uint32_t lit_step = 1, used = hlen;
  bool lit_ro = false;
  if (type == 0) {
    if (hlen + regen > len) return ZE_LIT;
    lit = src + hlen;
    lit_ro = true;
    used += regen;
  } else if (type == 1) {
    if (hlen + 1 > len) return ZE_LIT;
    lit = src + hlen;
    lit_step = 0;
    used += 1;
  } else {
    if (hlen + csize > len) return ZE_LIT;
    const uint8_t* q = src + hlen;
    uint32_t qlen = csize;
    if (type == 2) {
      if (const int e = z_huffman_tree(S, q, qlen)) return e;
      q += S.used;
      qlen -= S.used;
    } else if (S.huf_bits == 0) {
      return ZE_HUF;
    }
    ZHufStreams hs;
    const int e = z_huf_split(q, qlen, regen, sf == 0 ? 1 : 4, &hs);
    if (e) return e;
    if (const int e = z_huffman_literals(S, hs, dst + (dst_len - regen))) return e;
    used += csize;
  }
  // sequences section: header and tables
  const uint8_t* p = src + used;
  const uint32_t plen = len - used;
  if (plen == 0) return ZE_SEQ;
  uint32_t nseq = __ldg(p), q = 1;
  if (nseq == 0 && plen != 1) return ZE_SEQ;
  if (nseq >= 128) {
    const bool big = nseq == 255;
    if (plen < (big ? 3u : 2u)) return ZE_SEQ;
    nseq = big ? __ldg(p + 1) + (static_cast<uint32_t>(__ldg(p + 2)) << 8) + 0x7F00 : ((nseq - 128) << 8) + __ldg(p + 1);
    q = big ? 3 : 2;
  }
  if (nseq) {
    // modes and descriptions: at most 1 + 3 * 53 * 2 bytes are read
    const uint32_t b0 = z_stage(S, p, p + (plen < 400 ? plen : 400));
    __syncthreads();
    if (tid == 0) {
      int e = ZE_OK;
      const uint32_t modes = q < plen ? z_from(S, b0 + 8 * q) & 0xffu : 3u;
      if (modes & 3) e = ZE_SEQ;
      uint32_t at = q + 1;
      for (int w = 0; w < 3 && !e; ++w) {
        const int mode = static_cast<int>((modes >> (6 - 2 * w)) & 3);
        const int max_sym = w == 0 ? 36 : w == 1 ? 32 : 53;
        S.mode[w] = mode;
        if (mode == 0) {
          int nsym, al;
          z_default_norm(w, S.norm[w], &nsym, &al);
          S.nsym[w] = nsym;
          S.al[w] = al;
        } else if (mode == 1) {
          const uint32_t s = at < plen ? z_from(S, b0 + 8 * at) & 0xffu : 255u;
          if (s >= static_cast<uint32_t>(max_sym)) e = ZE_SEQ;
          else z_entry(S, w, 0, s, 0, 0);
          S.al[w] = 0;
          at += 1;
        } else if (mode == 2) {
          uint32_t u = 0;
          const uint32_t have = at < plen ? (plen - at < 128 ? plen - at : 128) : 0;
          e = z_norm(S, b0 + 8 * at, have, w == 1 ? 8 : 9, max_sym, S.norm[w], &S.nsym[w], &S.al[w], &u);
          at += u;
        } else if (S.al[w] < 0) {
          e = ZE_SEQ;
        }
      }
      S.used = at;
      S.err = e;
    }
    if (const int e = z_error(S)) return e;
    const int w = tid >> 5;
    if (w < 3 && (S.mode[w] == 0 || S.mode[w] == 2)) {
      const int e = z_fse_table(S, w, 9, [&](int st, int s, int nb, uint32_t base) {
        z_entry(S, w, st, static_cast<uint32_t>(s), static_cast<uint32_t>(nb), base);
      });
      if (e) S.err = e;
    }
    if (const int e = z_error(S)) return e;
    if (tid == 0) {
      ZRead r{nullptr, 0};
      const uint32_t at = S.used;
      if (at > plen || !z_open(r, p + at, plen - at)) {
        S.err = ZE_SEQ;
      } else {
        S.sl = 4 * z_bits(r, S.al[0]);
        S.so = 4 * z_bits(r, S.al[1]) + 2048;
        S.sm = 4 * z_bits(r, S.al[2]) + 4096;
        if (r.pos < 0) S.err = ZE_STREAM;
        S.pos = static_cast<uint32_t>(r.pos);
      }
    }
    if (const int e = z_error(S)) return e;
  }
  const uint8_t* bs = p + (nseq ? S.used : 0u);  // the sequence bits
  const uint32_t va = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(dst) & 31);
  uint8_t* vout = dst - va;
  const auto lit_byte = [=](uint32_t i) { return lit + i * lit_step; };
  uint32_t lits = 0;  // literals used
  // where n literals from the i-th on can be copied from at once
  const auto plain = [=](uint32_t i, uint32_t n, uint32_t v) -> const uint8_t* {
    return lit_step && (lit_ro || lit + i >= vout + v + n) ? lit + i : nullptr;
  };
  uint32_t v = va + static_cast<uint32_t>(out);
  for (uint32_t done = 0; done < nseq;) {
    const int nb = nseq - done < Z_SEQ ? static_cast<int>(nseq - done) : Z_SEQ;
    const bool final = done + nb == nseq;
    // the chain: states and bit position of each sequence of the group
    const uint32_t pos = S.pos, low = pos > Z_SEQ * 89u ? (pos - Z_SEQ * 89u) / 8 : 0u;
    const uint32_t b0 = z_stage(S, bs + low, bs + (pos + 7) / 8);
    if (tid < Z_PAD) S.bits[tid] = 0;
    __syncthreads();
    if (tid == 0) {
      uint32_t sl = S.sl, so = S.so, sm = S.sm;
      const uint32_t first = b0;  // no sequence of a sound stream starts below it
      uint32_t b = b0 + pos - 8 * low;
      int e = ZE_OK;
      const int linked = final ? nb - 1 : nb;  // the stream's last sequence has no state bits
      // The 96 bits below b are loaded beside the table words, so that once
      // these give the bit count of the values the state bits are two shifts
      // away (loading them from there: 185 cycles a sequence, so: 104).
      const auto row = [&](uint32_t at) {
        return *reinterpret_cast<const uint32_t*>(reinterpret_cast<const uint8_t*>(S.step) + at);
      };
      const auto follow = [&](int i) {
        const uint32_t cl = row(sl), co = row(so), cm = row(sm);
        const uint32_t* const q = S.bits + (b >> 5);
        const uint32_t q0 = q[0], q1 = q[-1], q2 = q[-2], q3 = q[-3];
        const uint32_t t0 = __funnelshift_r(q1, q0, b), t1 = __funnelshift_r(q2, q1, b), t2 = __funnelshift_r(q3, q2, b);
        S.at[i] = b;
        S.states[i] = (sl >> 2) | (so << 7) | (sm << 17);
        // (sums of the two bit counts, at most 63 and 26; the rest overflows
        // upwards; shifts take the low five bits)
        const uint32_t sum = cl + co + cm;
        const uint32_t w = (sum & 32u) ? __funnelshift_l(t2, t1, sum) : __funnelshift_l(t1, t0, sum);
        sl = (cl >> 16) + 4 * z_high(w, cl >> 8);
        sm = (cm >> 16) + 4 * z_high(__funnelshift_l(0u, w, cl >> 8), cm >> 8);
        so = (co >> 16) + 4 * z_high(__funnelshift_l(0u, w, (cl + cm) >> 8), co >> 8);
        b -= (sum & 0xffu) + ((sum >> 8) & 0xffu);
      };
      int i = 0;
      for (; i + Z_UNROLL <= linked && b >= first; i += Z_UNROLL) {
#pragma unroll
        for (int u = 0; u < Z_UNROLL; ++u) follow(i + u);
      }
      for (; i < linked && b >= first; ++i) follow(i);
      if (final && b >= first) {
        S.at[i] = b;
        S.states[i] = (sl >> 2) | (so << 7) | (sm << 17);
        b -= (row(sl) + row(so) + row(sm)) & 0xffu;
      }
      if (b < first) e = ZE_STREAM;
      S.sl = sl;
      S.so = so;
      S.sm = sm;
      S.pos = b - b0 + 8 * low;
      if (!e && final && b - b0 + 8 * low != 0) e = ZE_STREAM;
      S.err = e;
      S.bad = ZE_OK;
    }
    if (const int e = z_error(S)) return e;
    // a sequence a thread: its values, and what it does to the last three offsets
    const int lane = tid & 31, warp = tid >> 5;
    uint32_t ll = 0, ml = 0, ov = 0;
    if (tid < nb) {
      const uint32_t st = S.states[tid], sl = st & 511u, so = ((st >> 9) & 1023u) - 512, sm = (st >> 19) - 1024;
      uint32_t b = S.at[tid];
      const uint32_t xo = S.step[1][so] & 0xffu, xm = S.step[2][sm] & 0xffu, xl = S.step[0][sl] & 0xffu;
      ov = S.base[1][so] + z_high(z_below(S, b), xo);
      b -= xo;
      ml = S.base[2][sm] + z_high(z_below(S, b), xm);
      b -= xm;
      ll = S.base[0][sl] + z_high(z_below(S, b), xl);
      if (ov >> 31) atomicMax(&S.bad, static_cast<int>(ZE_OFFSET));  // (past any output, and not a map's offset)
    }
    // a map's slot: an offset, or Z_SLOT | which earlier one << 24 | how much is taken from it
    constexpr uint32_t Z_SLOT = 0x80000000u;
    uint32_t m0 = Z_SLOT, m1 = Z_SLOT | 1u << 24, m2 = Z_SLOT | 2u << 24;  // after the sequence, from before it
    if (tid < nb) {
      const uint32_t i0 = m0, i1 = m1, i2 = m2;
      const uint32_t idx = ov > 3 ? 4 : (ll > 0 ? ov - 1 : ov);
      if (idx) {
        m0 = idx == 4 ? ov - 3 : idx == 1 ? i1 : idx == 2 ? i2 : i0 + 1;
        m1 = i0;
        m2 = idx == 1 ? i2 : i1;
      }
    }
    const auto through = [&](uint32_t slot, uint32_t a0, uint32_t a1, uint32_t a2) {
      // slot of a later map applied to an earlier map's result
      if (!(slot & Z_SLOT)) return slot;
      const uint32_t k = (slot >> 24) & 3u, less = slot & 0xffffffu;
      const uint32_t a = k == 0 ? a0 : k == 1 ? a1 : a2;
      return (a & Z_SLOT) ? a + less : (a > less ? a - less : 0u);
    };
    const auto apply = [&](uint32_t a0, uint32_t a1, uint32_t a2) {
      const uint32_t r0 = through(m0, a0, a1, a2), r1 = through(m1, a0, a1, a2), r2 = through(m2, a0, a1, a2);
      m0 = r0;
      m1 = r1;
      m2 = r2;
    };
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t a0 = __shfl_up_sync(0xffffffffu, m0, o), a1 = __shfl_up_sync(0xffffffffu, m1, o),
                     a2 = __shfl_up_sync(0xffffffffu, m2, o);
      if (lane >= o) apply(a0, a1, a2);
    }
    if (lane == 31) {
      S.map[warp][0] = m0;
      S.map[warp][1] = m1;
      S.map[warp][2] = m2;
    }
    __syncthreads();
    if (tid == 0) {
      uint32_t r0 = S.rep[0], r1 = S.rep[1], r2 = S.rep[2];
      for (int w = 0; w < ZT / 32; ++w) {  // each warp's map becomes what precedes it
        const uint32_t a0 = S.map[w][0], a1 = S.map[w][1], a2 = S.map[w][2];
        S.map[w][0] = r0;
        S.map[w][1] = r1;
        S.map[w][2] = r2;
        const uint32_t n0 = through(a0, r0, r1, r2), n1 = through(a1, r0, r1, r2), n2 = through(a2, r0, r1, r2);
        r0 = n0;
        r1 = n1;
        r2 = n2;
      }
      S.rep[0] = r0;
      S.rep[1] = r1;
      S.rep[2] = r2;
    }
    __syncthreads();
    apply(S.map[warp][0], S.map[warp][1], S.map[warp][2]);
    // the sequence's offset is the first of the three after it
    const uint32_t off = m0;
    // output and literals before the sequence
    uint64_t tot;
    const uint64_t ol = block_exclusive_sum<uint64_t>(static_cast<uint64_t>(ll + ml) | (static_cast<uint64_t>(ll) << 32),
                                                      S.lz.tmp64, &tot);
    const uint32_t l_at = static_cast<uint32_t>(ol >> 32);
    if (tid < nb) {
      const uint64_t at = static_cast<uint64_t>(v - va) + static_cast<uint32_t>(ol);
      const uint32_t rest = regen - lits;  // literals before the group
      int e = ZE_OK;
      if (l_at > rest || ll > rest - l_at) e = ZE_SEQ;
      else if (off == 0 || off > at + ll - out0) e = ZE_OFFSET;
      else if (at + ml + (rest - l_at) > dst_len) e = ZE_SIZE;  // (unread literals included)
      if (e) atomicMax(&S.bad, e);
    }
    __syncthreads();
    if (const int e = S.bad) return e;
    if (lit_ro)
      lz_pairs<true>(S.lz, nb, vout, v, vfloor, ll, LZ_LIT | (lits + l_at), ml, off, lit_byte, plain);
    else
      lz_pairs<false>(S.lz, nb, vout, v, vfloor, ll, LZ_LIT | (lits + l_at), ml, off, lit_byte, plain);
    lits += static_cast<uint32_t>(tot >> 32);
    done += static_cast<uint32_t>(nb);
  }
  // the literals after the last sequence
  if (lit_ro) lz_one<true>(S.lz, vout, v, vfloor, LZ_LIT | lits, regen - lits, lit_byte, plain);
  else lz_one<false>(S.lz, vout, v, vfloor, LZ_LIT | lits, regen - lits, lit_byte, plain);
  out = v - va;
  return ZE_OK;
}

// Every frame of src[0, src_len) into dst[0, dst_len); returns 0 or an error.
// Block-collective.
__device__ __forceinline__ int z_frames(ZBlock& S, const uint8_t* src, uint32_t src_len, uint8_t* dst, uint64_t dst_len) {
  const int tid = threadIdx.x;
  uint32_t pos = 0;
  uint64_t out = 0;
  const uint32_t va = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(dst) & 31);
  uint32_t vfloor = va;
  if (tid == 0) S.err = 0;
  while (pos < src_len) {
    if (src_len - pos < 4) return ZE_TRUNC;
    const uint32_t magic = z_le(src + pos, 4);
    if ((magic & 0xFFFFFFF0u) == 0x184D2A50u) {  // a skippable frame
      if (src_len - pos < 8) return ZE_TRUNC;
      const uint32_t sz = z_le(src + pos + 4, 4);
      if (static_cast<uint64_t>(pos) + 8 + sz > src_len) return ZE_TRUNC;
      pos += 8 + sz;
      continue;
    }
    if (magic != 0xFD2FB528u) return ZE_MAGIC;
    pos += 4;
    if (pos >= src_len) return ZE_TRUNC;
    const uint32_t fhd = __ldg(src + pos++);
    if (fhd & 8) return ZE_HEADER;
    const uint32_t fcs_flag = fhd >> 6, single = (fhd >> 5) & 1, checksum = (fhd >> 2) & 1, dflag = fhd & 3;
    if (!single) ++pos;  // window descriptor
    const uint32_t dlen = dflag == 3 ? 4 : dflag;
    const uint32_t flen = fcs_flag == 0 ? single : fcs_flag == 1 ? 2 : fcs_flag == 2 ? 4 : 8;
    if (static_cast<uint64_t>(pos) + dlen + flen > src_len) return ZE_TRUNC;
    if (dlen && z_le(src + pos, static_cast<int>(dlen)) != 0) return ZE_DICT;
    pos += dlen;
    int64_t fcs = -1;
    if (flen) {
      uint64_t v = 0;
      for (int i = static_cast<int>(flen) - 1; i >= 0; --i) v = (v << 8) | __ldg(src + pos + i);
      fcs = static_cast<int64_t>(v + (flen == 2 ? 256 : 0));
      pos += flen;
    }
    __syncthreads();
    if (tid == 0) {
      S.huf_bits = 0;
      S.al[0] = S.al[1] = S.al[2] = -1;
      S.rep[0] = 1;
      S.rep[1] = 4;
      S.rep[2] = 8;
    }
    __syncthreads();
    const uint64_t out0 = out;
    for (;;) {
      if (src_len - pos < 3) return ZE_TRUNC;
      const uint32_t h = z_le(src + pos, 3);
      pos += 3;
      const uint32_t last = h & 1, type = (h >> 1) & 3, bsize = h >> 3;
      if (type == 0) {
        if (bsize > src_len - pos) return ZE_TRUNC;
        if (bsize > dst_len - out) return ZE_SIZE;
        lz_block_copy<ZT, true>(dst + out, src + pos, bsize);
        out += bsize;
        pos += bsize;
        vfloor = va + static_cast<uint32_t>(out);
        __syncthreads();
      } else if (type == 1) {
        if (pos >= src_len) return ZE_TRUNC;
        if (bsize > dst_len - out) return ZE_SIZE;
        const uint8_t b = __ldg(src + pos);
        for (uint32_t i = tid; i < bsize; i += ZT) dst[out + i] = b;
        out += bsize;
        pos += 1;
        vfloor = va + static_cast<uint32_t>(out);
        __syncthreads();
      } else if (type == 2) {
        if (bsize > (128u << 10) || bsize > src_len - pos) return ZE_BLOCK;
        if (const int e = z_block(S, src + pos, bsize, dst, out, out0, dst_len, vfloor)) return e;
        pos += bsize;
      } else {
        return ZE_BLOCK;
      }
      if (last) break;
    }
    if (checksum) {
      if (src_len - pos < 4) return ZE_TRUNC;
      pos += 4;
    }
    if (fcs >= 0 && static_cast<uint64_t>(fcs) != out - out0) return ZE_SIZE;
  }
  return out == dst_len ? ZE_OK : ZE_SIZE;
}

__global__ void __launch_bounds__(ZT, 2) k_zstd(const SnappyJob* __restrict__ jobs, int n_jobs, DevStatus* st) {
  extern __shared__ __align__(16) uint8_t z_smem[];
  ZBlock& S = *reinterpret_cast<ZBlock*>(z_smem);
  for (int j = blockIdx.x; j < n_jobs; j += gridDim.x) {
    const SnappyJob jb = jobs[j];
    if (jb.codec != CODEC_ZSTD) continue;
    int rc = 0;
    if (jb.prefix > jb.src_len || jb.prefix > jb.dst_len) {
      rc = ZE_TRUNC;
    } else if (jb.raw && jb.src_len != jb.dst_len) {
      rc = ZE_SIZE;
    } else {
      lz_block_copy<ZT, true>(jb.dst, jb.src, jb.raw ? jb.src_len : jb.prefix);
      if (!jb.raw)
        rc = z_frames(S, jb.src + jb.prefix, jb.src_len - jb.prefix, jb.dst + jb.prefix, jb.dst_len - jb.prefix);
    }
    if (rc && threadIdx.x == 0) report(st, DERR_CORRUPT, jb.page, WHERE_SNAPPY, 100 + rc);
    __syncthreads();
  }
}

}  // namespace

void launch_zstd(const SnappyJob* jobs, int n_jobs, int n_sms, DevStatus* st, cudaStream_t s) {
  if (n_jobs <= 0) return;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_zstd, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(ZBlock));
    attr = true;
  }
  const int grid = n_jobs < 2 * n_sms ? n_jobs : 2 * n_sms;
  k_zstd<<<grid, ZT, sizeof(ZBlock), s>>>(jobs, n_jobs, st);
}

}  // namespace pqi
