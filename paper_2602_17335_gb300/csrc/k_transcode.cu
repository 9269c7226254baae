// V2 page encodings made readable as PLAIN pages before the walk.
//
// The paper's Section 3 ("Encoding Flexibility", Insight 3) counts the V2
// encodings among the GPU-friendly ones.  Three of them are read here:
//
//   BYTE_STREAM_SPLIT        K streams of N bytes (stream b = byte b of every
//                            value)  ->  N little-endian K-byte values
//   DELTA_LENGTH_BYTE_ARRAY  DELTA_BINARY_PACKED INT32 lengths, then the bytes
//   DELTA_BYTE_ARRAY         DELTA_BINARY_PACKED INT32 prefix lengths, then the
//                            suffixes as DELTA_LENGTH_BYTE_ARRAY; value i is
//                            the first prefix[i] bytes of value i-1 followed by
//                            suffix i
//
// Strings get a table with one (offset << 32) | length entry per value
// (PlanPage::vtab), offsets into the page's value bytes, which the expansion
// reads like dictionary entries.  The bytes of DELTA_LENGTH_BYTE_ARRAY values
// stay where the page has them.  Of a DELTA_BYTE_ARRAY page, the suffix bytes
// are copied to a piece of the plan's pool; a value without a prefix is its
// suffix there, and a value without a suffix is the beginning of its
// predecessor and points where that one does (sorted columns are mostly such
// values).  Only values with both are put together, behind the suffixes, as
// a copy of the predecessor's beginning and a literal each: lz_pairs does
// it, however the prefixes stack up.
//
// BYTE_STREAM_SPLIT is a transpose of bytes, many blocks a page (k_bss, HBM
// bound).  The string encodings take one block per page (k_transcode): one
// thread follows the DELTA block headers in staged bytes (about 100 cycles a
// block of 128 lengths, the latency of a page), all threads decode the
// lengths, 2048 at a time.  The page's level bytes stay in front of its
// values, so that the walk parses the body like a PLAIN page's.  On an error
// the plan page keeps its level bytes only, so that later stages read nothing
// past them.
#include "decode_job.h"
#include "dev_util.cuh"
#include "lz_exec.cuh"

namespace pqi {
namespace {

constexpr int TC_THREADS = 512;
constexpr int TC_PER_THREAD = 4;
constexpr uint32_t TC_MAX_BLOCK = TC_THREADS * TC_PER_THREAD;  // DELTA block values a cursor holds
constexpr uint32_t TC_MAX_LIST = TC_MAX_BLOCK / 128;           // blocks have 128 values or more
constexpr uint32_t TC_WIN = 9216;  // staged stream bytes: a block takes 10 + 64 + 8192 at most

// Block-shared state of one DELTA_BINARY_PACKED INT32 stream.
struct DCursor {
  uint32_t hdr_end;   // first block header
  uint32_t pos;       // next block header
  uint32_t end;       // end of the readable bytes
  uint32_t left;      // values still to decode after the buffered ones
  uint32_t nbuf;      // values in buf
  uint32_t cnt;       // values in the blocks being decoded
  uint32_t bs, mbc, vpm, total;
  int32_t first;
  int32_t last;       // last decoded value
  int32_t started;
  uint32_t w0, wn;    // the window: source offset of its first byte (up to 15 before the stream), bytes
  uint32_t shift;     // byte `w0` sits at win[shift]
  int64_t minv[TC_MAX_LIST];   // listed blocks: min delta,
  uint32_t wid[TC_MAX_LIST];   // window offset of the width bytes
  uint32_t data[TC_MAX_LIST];  // and of the packed deltas
  int32_t buf[TC_MAX_BLOCK];
  __align__(16) uint8_t win[TC_WIN + 64];
};

struct TcSmem {
  LzPairs<TC_THREADS, 4096, 16384> lz;
  DCursor c[2];
  int64_t tmp[32];
  int32_t err;
  int32_t flag;             // DERR_* of the first error
  int32_t detail;
  uint32_t v0;
  uint32_t more;            // the window has to move
  uint64_t dst_off;
  int32_t wlast[TC_THREADS / 32];  // length of each warp's last value with a suffix, -1 none
  uint32_t wlast_at[TC_THREADS / 32];  // and where it lies
};

__device__ __forceinline__ void tc_fail(TcSmem& sm, uint32_t flag, int detail) {
  if (atomicCAS(&sm.err, 0, 1) == 0) {
    sm.flag = static_cast<int32_t>(flag);
    sm.detail = detail;
  }
}

// Whether any thread has failed by now, the same answer for all threads.
// Block-collective, with a barrier: the word is read on one side of it and
// decided on by all threads at once (a warp that read it by itself could see a
// later failure than the others and leave their next barriers to them).
__device__ __forceinline__ bool tc_error(const TcSmem& sm) { return __syncthreads_or(sm.err) != 0; }

// Moves the cursor's window to source offset `from` (block-collective, a
// barrier on each side).  Reads up to 15 bytes on either side of the source.
__device__ void tc_stage(const uint8_t* b, DCursor& c, uint32_t from) {
  __syncthreads();
  const uintptr_t a = reinterpret_cast<uintptr_t>(b + from) & ~uintptr_t(15);
  const uintptr_t lim = (reinterpret_cast<uintptr_t>(b + c.end) + 15) & ~uintptr_t(15);
  const uint32_t n = lim - a < TC_WIN ? static_cast<uint32_t>(lim - a) : TC_WIN;
  for (uint32_t i = threadIdx.x; 16 * i < n; i += TC_THREADS)
    reinterpret_cast<uint4*>(c.win)[i] = __ldg(reinterpret_cast<const uint4*>(a) + i);
  if (threadIdx.x == 0) {
    c.shift = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(b + from) - a);
    c.w0 = from;
    c.wn = n - c.shift;
  }
  __syncthreads();
}

// The block header at source offset q, of a block whose first `need`
// miniblocks hold values.  1: header and packed deltas lie in the window, 0:
// they do not (data end unknown or past it), -1: malformed.  *hdr: bytes
// before the widths; *size: the whole block's bytes; header_only: the deltas
// need not be in the window.
__device__ int tc_block(const DCursor& c, uint32_t q, uint32_t need, bool header_only, uint32_t* hdr, uint32_t* size,
                        int64_t* minv) {
  const uint32_t have = q >= c.w0 && q - c.w0 < c.wn ? c.wn - (q - c.w0) : 0u;
  const bool all = c.w0 + c.wn >= c.end;  // nothing follows the window
  if (!all && have < 10 + c.mbc) return 0;
  const uint8_t* w = c.win + c.shift + (q - c.w0);
  const uint32_t left = c.end - q;
  uint64_t z = 0;
  uint32_t vl = 0, bits = 0;
  if (c.mbc == 4 && left >= 20) {
    uint32_t w4;
    vl = static_cast<uint32_t>(delta_header16<true>(w, &z, &w4));
    if (!vl) return -1;
    for (uint32_t m = 0; m < need; ++m) {
      const uint32_t wd = (w4 >> (8 * m)) & 0xffu;
      if (wd > 32) return -1;
      bits += wd;
    }
  } else {
    const int n = uleb([&](uint32_t i) { return static_cast<uint32_t>(w[i]); }, 0, left, &z);
    if (!n || left - n < c.mbc) return -1;
    vl = static_cast<uint32_t>(n);
    for (uint32_t m = 0; m < need; ++m) {
      if (w[vl + m] > 32) return -1;
      bits += w[vl + m];
    }
  }
  *hdr = vl;
  *size = vl + c.mbc + bits * c.vpm / 8;
  *minv = unzigzag(z);
  if (*size > left) return -1;
  return header_only || *size <= have ? 1 : 0;
}

// Parses the stream header at `p` and walks the block headers to the stream
// end (after the last miniblock that holds values).  Records the result in
// `c`; false, with the error in sm, when it is malformed.  Block-collective.
__device__ bool dstream_open(const uint8_t* b, uint32_t p, uint32_t end, DCursor& c, TcSmem& sm) {
  if (threadIdx.x == 0) {
    auto get = [b](uint32_t i) { return ld_u8(b + i); };
    uint64_t v[4];
    uint32_t q = p;
    int bad = 0;
    for (int k = 0; k < 4 && !bad; ++k) {
      const int n = uleb(get, q, end, &v[k]);
      if (!n) bad = 1;
      q += static_cast<uint32_t>(n);
    }
    if (!bad && (v[0] == 0 || v[0] % 128 || v[1] == 0 || v[0] % v[1] || (v[0] / v[1]) % 32)) bad = 2;
    if (bad) {
      tc_fail(sm, DERR_CORRUPT, bad);
    } else if (v[0] > TC_MAX_BLOCK || v[2] > 0x7fffffffull) {
      tc_fail(sm, DERR_UNSUPPORTED, 3);
    } else {
      c.bs = static_cast<uint32_t>(v[0]);
      c.mbc = static_cast<uint32_t>(v[1]);
      c.vpm = c.bs / c.mbc;
      c.total = static_cast<uint32_t>(v[2]);
      c.first = static_cast<int32_t>(static_cast<uint32_t>(static_cast<uint64_t>(unzigzag(v[3]))));
      c.hdr_end = c.pos = q;
      c.end = end;
      c.left = c.total ? c.total - 1 : 0;
      c.w0 = q;
      c.wn = 0;
    }
  }
  if (tc_error(sm)) return false;
  while (c.left) {  // each window holds one header at least
    tc_stage(b, c, c.pos);
    if (threadIdx.x == 0) {
      uint32_t q = c.pos, left = c.left;
      const uint32_t q0 = q, wend = c.w0 + c.wn, end = c.end;
      const uint8_t* w = c.win + c.shift - c.w0;  // window byte of source offset x: w + x
      const bool common = c.mbc == 4 && c.vpm == 32;
      while (left) {
        while (common && left >= 128 && q + 20 <= wend) {
          uint32_t z, w4;
          const uint32_t size = delta_common(w + q, 32, &z, &w4);
          if (size == 0 || size > end - q) break;
          q += size;
          left -= 128;
        }
        if (!left || (q != q0 && q >= wend && q < end)) break;  // (the next window starts there)
        const uint32_t bc = left < c.bs ? left : c.bs;
        uint32_t hdr, size;
        int64_t mn;
        const int k = q < c.end ? tc_block(c, q, (bc + c.vpm - 1) / c.vpm, true, &hdr, &size, &mn) : -1;
        if (k < 0 || (k == 0 && q == q0)) {
          tc_fail(sm, DERR_CORRUPT, 4);
          left = 0;
          break;
        }
        if (k == 0) break;
        q += size;
        left -= bc;
      }
      c.pos = q;  // stream end, until dstream_rewind
      c.left = left;
    }
    __syncthreads();
  }
  return !tc_error(sm);
}

__device__ __forceinline__ void dstream_rewind(DCursor& c) {
  c.pos = c.hdr_end;
  c.started = 0;
  c.nbuf = 0;
  c.wn = 0;
}

// All threads: decodes the next buffer of values (the header's first value,
// then the whole blocks that the buffer holds and the window has: thread 0
// lists them, every thread decodes TC_PER_THREAD values).  Returns false on
// an error.
__device__ bool dstream_refill(const uint8_t* b, DCursor& c, TcSmem& sm) {
  for (int attempt = 0; attempt < 2; ++attempt) {
    if (threadIdx.x == 0) {
      sm.more = 0;
      c.cnt = 0;
      if (!c.started) {
        c.started = 1;
        c.left = c.total ? c.total - 1 : 0;
        c.nbuf = c.total ? 1 : 0;
        c.buf[0] = c.first;
        c.last = c.first;
      } else if (c.left) {
        uint32_t q = c.pos, cnt = 0, n = 0, left = c.left;
        const uint32_t wend = c.w0 + c.wn, wbase = c.shift - c.w0;
        const bool common = c.mbc == 4 && c.vpm == 32;
        while (left && n < TC_MAX_LIST) {
          if (common && left >= 128 && q >= c.w0 && q + 20 <= wend) {
            uint32_t z, w4;
            const uint32_t size = delta_common(c.win + (wbase + q), 32, &z, &w4);
            if (size && size <= wend - q && size <= c.end - q) {
              c.minv[n] = unzigzag(z);
              c.wid[n] = wbase + q + 1;
              c.data[n] = wbase + q + 5;
              ++n;
              q += size;
              cnt += 128;
              left -= 128;
              continue;
            }
          }
          const uint32_t bc = left < c.bs ? left : c.bs;
          if (cnt + c.bs > TC_MAX_BLOCK) break;
          uint32_t hdr, size;
          int64_t mn;
          const int k = q < c.end ? tc_block(c, q, (bc + c.vpm - 1) / c.vpm, false, &hdr, &size, &mn) : -1;
          if (k < 0) {
            tc_fail(sm, DERR_CORRUPT, 7);
            break;
          }
          if (k == 0) {
            if (n == 0) {
              if (attempt) tc_fail(sm, DERR_CORRUPT, 8);
              sm.more = 1;
            }
            break;
          }
          c.minv[n] = mn;
          c.wid[n] = c.shift + (q - c.w0) + hdr;
          c.data[n] = c.wid[n] + c.mbc;
          ++n;
          q += size;
          cnt += bc;
          left -= bc;
        }
        c.pos = q;
        c.cnt = cnt;
      } else {
        tc_fail(sm, DERR_CORRUPT, 9);  // more values asked for than the stream holds
      }
    }
    if (tc_error(sm)) return false;
    if (!sm.more) break;
    tc_stage(b, c, c.pos);
  }
  const uint32_t cnt = c.cnt;
  if (cnt) {
    const uint32_t k0 = threadIdx.x * TC_PER_THREAD;
    int64_t d[TC_PER_THREAD];
    int64_t s = 0;
    // (a thread's values lie in one miniblock: those have 32 values or more)
    const uint32_t blk = k0 / c.bs, r0 = k0 - blk * c.bs, m = r0 / c.vpm;
    uint32_t bit = 0;
    int w = 0;
    if (k0 < cnt) {
      const uint8_t* wd = c.win + c.wid[blk];
      uint32_t before = 0;
      for (uint32_t i = 0; i < m; ++i) before += wd[i];
      w = wd[m];
      bit = 8 * c.data[blk] + before * c.vpm + (r0 - m * c.vpm) * static_cast<uint32_t>(w);
    }
    const uint32_t* w32 = reinterpret_cast<const uint32_t*>(c.win);
#pragma unroll
    for (int u = 0; u < TC_PER_THREAD; ++u) {
      if (k0 + u < cnt) {
        const uint32_t x = __funnelshift_r(w32[bit >> 5], w32[(bit >> 5) + 1], bit & 31);
        s += c.minv[blk] + static_cast<int64_t>(w >= 32 ? x : x & ((1u << w) - 1u));
        bit += static_cast<uint32_t>(w);
      }
      d[u] = s;
    }
    int64_t tot;
    const int64_t ex = block_exclusive_sum<int64_t>(s, sm.tmp, &tot);
    const int64_t base = static_cast<int64_t>(c.last) + ex;
#pragma unroll
    for (int u = 0; u < TC_PER_THREAD; ++u)
      if (k0 + u < cnt) c.buf[k0 + u] = static_cast<int32_t>(static_cast<uint32_t>(static_cast<uint64_t>(base + d[u])));
    __syncthreads();
    if (threadIdx.x == 0) {
      c.last = c.buf[cnt - 1];
      c.nbuf = cnt;
      c.left -= cnt;
    }
    __syncthreads();
  }
  return true;
}

// DELTA_LENGTH_BYTE_ARRAY values at src[v0, src_len): their entries, with
// offsets from v0, into tab.  Returns the values, or -1 on an error.
__device__ int64_t tc_dlba(const TranscodeJob& j, TcSmem& sm, uint32_t v0, uint64_t* tab) {
  DCursor& c = sm.c[0];
  if (!dstream_open(j.src, v0, j.src_len, c, sm)) return -1;
  const uint32_t M = c.total;
  const uint32_t cstart = c.pos;
  if (M > static_cast<uint32_t>(j.num_values) || (j.required && M != static_cast<uint32_t>(j.num_values))) {
    if (threadIdx.x == 0) tc_fail(sm, DERR_CORRUPT, 20);
    return -1;
  }
  __syncthreads();
  if (threadIdx.x == 0) dstream_rewind(c);
  __syncthreads();
  const int64_t room = static_cast<int64_t>(j.src_len) - cstart;
  int64_t K = 0, C = 0;
  while (K < M) {
    if (!dstream_refill(j.src, c, sm)) return -1;
    const uint32_t n = c.nbuf, k0 = threadIdx.x * TC_PER_THREAD;
    int64_t len[TC_PER_THREAD], mine = 0;
#pragma unroll
    for (int u = 0; u < TC_PER_THREAD; ++u) {
      len[u] = k0 + u < n ? c.buf[k0 + u] : 0;
      if (len[u] < 0) tc_fail(sm, DERR_CORRUPT, 21);
      mine += len[u];
    }
    int64_t tot;
    int64_t at = C + block_exclusive_sum<int64_t>(mine, sm.tmp, &tot);
    if (tc_error(sm)) return -1;
    if (C + tot > room) {
      if (threadIdx.x == 0) tc_fail(sm, DERR_CORRUPT, 22);
      return -1;
    }
#pragma unroll
    for (int u = 0; u < TC_PER_THREAD; ++u) {
      if (k0 + u < n)
        tab[K + k0 + u] = (static_cast<uint64_t>(cstart - v0 + at) << 32) | static_cast<uint64_t>(len[u]);
      at += len[u];
    }
    K += n;
    C += tot;
    __syncthreads();
  }
  return M;
}

// DELTA_BYTE_ARRAY values at src[v0, src_len): first a pass over both length
// streams that checks them, totals the value bytes and leaves (prefix << 32)
// | suffix in tab; then the suffixes, and the values that have a prefix too,
// are written at dst + v0 of a piece of the pool (sm.dst_off) and the entries
// replace the lengths.  Returns the value bytes written, or -1 on an error;
// *values: the count.
__device__ int64_t tc_dba(const TranscodeJob& j, TcSmem& sm, uint32_t v0, uint8_t* pool, uint64_t pool_cap,
                          unsigned long long* pool_used, uint64_t* tab, int64_t* values) {
  DCursor& cp = sm.c[0];
  DCursor& cs = sm.c[1];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (!dstream_open(j.src, v0, j.src_len, cp, sm)) return -1;
  if (!dstream_open(j.src, cp.pos, j.src_len, cs, sm)) return -1;
  const uint32_t M = cp.total;
  const uint32_t cstart = cs.pos;
  if (cs.total != M || M > static_cast<uint32_t>(j.num_values) ||
      (j.required && M != static_cast<uint32_t>(j.num_values))) {
    if (t == 0) tc_fail(sm, DERR_CORRUPT, 33);
    return -1;
  }
  __syncthreads();
  if (t == 0) {
    dstream_rewind(cp);
    dstream_rewind(cs);
  }
  __syncthreads();
  const int64_t room = static_cast<int64_t>(j.src_len) - cstart;
  int64_t T = 0, S = 0, prevL = 0;
  uint32_t up = 0, np = 0, us = 0, ns = 0;
  for (int64_t K = 0; K < M;) {
    if (up == np) {
      if (!dstream_refill(j.src, cp, sm)) return -1;
      np = cp.nbuf;
      up = 0;
    }
    if (us == ns) {
      if (!dstream_refill(j.src, cs, sm)) return -1;
      ns = cs.nbuf;
      us = 0;
    }
    const uint32_t n = min(np - up, ns - us), k0 = t * TC_PER_THREAD;
    int64_t sumL = 0, sumS = 0;
#pragma unroll
    for (int u = 0; u < TC_PER_THREAD; ++u) {
      const uint32_t k = k0 + u;
      if (k < n) {
        const int64_t p = cp.buf[up + k], s = cs.buf[us + k];
        // a prefix may not be longer than the value before it (none before value 0)
        const int64_t before = k ? static_cast<int64_t>(cp.buf[up + k - 1]) + cs.buf[us + k - 1] : prevL;
        if (p < 0 || s < 0) tc_fail(sm, DERR_CORRUPT, 30);
        else if (p > before) tc_fail(sm, DERR_CORRUPT, 31);
        tab[K + k] = (static_cast<uint64_t>(p) << 32) | static_cast<uint32_t>(s);
        sumL += p + s;
        sumS += s;
      }
    }
    int64_t totL, totS;
    block_exclusive_sum<int64_t>(sumL, sm.tmp, &totL);
    block_exclusive_sum<int64_t>(sumS, sm.tmp, &totS);
    if (tc_error(sm)) return -1;
    if (S + totS > room) {
      if (t == 0) tc_fail(sm, DERR_CORRUPT, 32);
      return -1;
    }
    prevL = static_cast<int64_t>(cp.buf[up + n - 1]) + cs.buf[us + n - 1];
    K += n;
    T += totL;
    S += totS;
    up += n;
    us += n;
    __syncthreads();
  }
  if (t == 0) {
    const uint64_t need = (static_cast<uint64_t>(v0) + static_cast<uint64_t>(S + T) + 32 + 15) & ~uint64_t(15);
    if (static_cast<uint64_t>(v0) + 4ull * M + static_cast<uint64_t>(T) > 0x7fffffffull) {
      tc_fail(sm, DERR_UNSUPPORTED, 34);
    } else if (need > pool_cap) {
      tc_fail(sm, DERR_CAPACITY, 35);
    } else {
      const unsigned long long off = atomicAdd(pool_used, static_cast<unsigned long long>(need));
      if (off + need > pool_cap) tc_fail(sm, DERR_CAPACITY, 36);
      else sm.dst_off = off;
    }
  }
  if (tc_error(sm)) return -1;
  // body: levels, the S suffix bytes, the values put together (offsets below
  // count from behind the levels)
  uint8_t* body = pool + sm.dst_off + v0;
  const uint32_t sufs = static_cast<uint32_t>(S);
  lz_block_copy<TC_THREADS>(body, j.src + cstart, sufs);
  uint8_t* out = body + sufs;
  const uint32_t va = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(out) & 31);
  uint32_t v = va, vfloor = va;
  const uint8_t* src = j.src;
  const auto lit = [src](uint32_t i) { return src + i; };
  const auto plain = [src](uint32_t i, uint32_t, uint32_t) { return src + i; };
  uint32_t lastO = 0, lastL = 0, s_at = 0;  // where the last value with a suffix lies, its length; suffix bytes used
  for (int64_t K = 0; K < M; K += TC_THREADS) {
    const int nb = M - K < TC_THREADS ? static_cast<int>(M - K) : TC_THREADS;
    const uint64_t e = t < nb ? tab[K + t] : 0ull;
    const uint32_t p = static_cast<uint32_t>(e >> 32), s = static_cast<uint32_t>(e);
    const bool own = t < nb && s > 0, built = own && p > 0;
    // suffix bytes and built bytes before this value (both below 2^31)
    uint64_t tot;
    const uint64_t ex = block_exclusive_sum<uint64_t>(
        static_cast<uint64_t>(s) | (static_cast<uint64_t>(built ? p + s : 0u) << 32),
        reinterpret_cast<uint64_t*>(sm.tmp), &tot);
    const uint32_t my_s = s_at + static_cast<uint32_t>(ex), my_v = v - va + static_cast<uint32_t>(ex >> 32);
    const uint32_t my_o = built ? sufs + my_v : my_s;
    // the last value with a suffix before this one
    const uint32_t m = __ballot_sync(0xffffffffu, own), below = m & ((1u << lane) - 1u);
    const int from = below ? 31 - __clz(below) : 0;
    uint32_t prevO = __shfl_sync(0xffffffffu, my_o, from), prevL = __shfl_sync(0xffffffffu, p + s, from);
    if (lane == (m ? 31 - __clz(m) : 0)) {
      sm.wlast[warp] = m ? static_cast<int32_t>(p + s) : -1;
      sm.wlast_at[warp] = my_o;
    }
    __syncthreads();
    int w = warp - 1;
    while (w >= 0 && sm.wlast[w] < 0) --w;
    if (!below) {
      prevO = w >= 0 ? sm.wlast_at[w] : lastO;
      prevL = w >= 0 ? static_cast<uint32_t>(sm.wlast[w]) : lastL;
    }
    w = TC_THREADS / 32 - 1;
    while (w >= 0 && sm.wlast[w] < 0) --w;
    if (w >= 0) {
      lastO = sm.wlast_at[w];
      lastL = static_cast<uint32_t>(sm.wlast[w]);
    }
    if (t < nb) tab[K + t] = (static_cast<uint64_t>(own ? my_o : prevO) << 32) | (p + s);
    if (tot >> 32)  // (the predecessor's beginning: suffix bytes in the page, or what was just built)
      lz_pairs<true>(sm.lz, nb, out - va, v, vfloor, built ? p : 0u, prevO < sufs ? LZ_LIT | (cstart + prevO) : prevL,
                     built ? s : 0u, LZ_LIT | (cstart + my_s), lit, plain);
    s_at += static_cast<uint32_t>(tot);
    __syncthreads();
  }
  *values = M;
  return static_cast<int64_t>(sufs) + (v - va);
}

// Level bytes in front of the values of page j, and whether they are sound.
__device__ __forceinline__ bool tc_levels(const TranscodeJob& j, uint32_t* v0, int* detail) {
  *v0 = 0;
  if (j.levels < 0) {
    const uint32_t L = j.src_len >= 4 ? ld_le32_g(j.src) : 0xffffffffu;
    *detail = 10;
    if (j.src_len < 4 || L > j.src_len - 4) return false;
    *v0 = 4 + L;
  } else {
    *detail = 11;
    if (static_cast<uint32_t>(j.levels) > j.src_len) return false;
    *v0 = static_cast<uint32_t>(j.levels);
  }
  return true;
}

__global__ void __launch_bounds__(TC_THREADS, 2) k_transcode(const TranscodeJob* jobs, PlanPage* pps, uint8_t* pool,
                                                            uint64_t pool_cap, unsigned long long* pool_used,
                                                            uint64_t* vpos, DevStatus* st) {
  extern __shared__ __align__(16) uint8_t tc_smem[];
  TcSmem& sm = *reinterpret_cast<TcSmem*>(tc_smem);
  const TranscodeJob j = jobs[blockIdx.x];
  if (j.enc == ENC_BSS) return;
  const uint32_t vtab = pps[j.pp].vtab;
  uint64_t* tab = vtab && vpos ? vpos + (vtab - 1) : nullptr;
  {
    // the page's bytes into L2 first (a hint)
    const uintptr_t e = reinterpret_cast<uintptr_t>(j.src) + j.src_len;
    for (uintptr_t q = (reinterpret_cast<uintptr_t>(j.src) & ~uintptr_t(127)) + 128u * threadIdx.x; q < e;
         q += 128u * blockDim.x)
      asm volatile("prefetch.global.L2 [%0];" ::"l"(q));
  }
  if (threadIdx.x == 0) {
    sm.err = 0;
    sm.flag = 0;
    sm.detail = 0;
    sm.dst_off = 0;
    sm.c[0].started = sm.c[1].started = 0;
    uint32_t v0;
    int detail;
    if (!tc_levels(j, &v0, &detail)) tc_fail(sm, DERR_CORRUPT, detail);
    else if (!tab) tc_fail(sm, DERR_CORRUPT, 13);  // an earlier scan of the plan failed here
    sm.v0 = v0;
  }
  __syncthreads();
  const bool failed = tc_error(sm);
  const uint32_t v0 = sm.v0;
  int64_t values = -1, bytes = -1;
  if (!failed) {
    if (j.enc == ENC_DELTA_LBA) {
      values = tc_dlba(j, sm, v0, tab);
    } else if (j.enc == ENC_DELTA_BA) {
      bytes = tc_dba(j, sm, v0, pool, pool_cap, pool_used, tab, &values);
    } else if (threadIdx.x == 0) {
      tc_fail(sm, DERR_UNSUPPORTED, 12);
    }
  }
  __syncthreads();
  const bool ok = values >= 0 && !sm.err;
  const bool moved = j.enc == ENC_DELTA_BA;
  uint8_t* dst = pool + sm.dst_off;
  if (ok && moved)
    for (uint32_t i = threadIdx.x; i < v0; i += blockDim.x) dst[i] = ld_u8(j.src + i);
  if (threadIdx.x == 0) {
    PlanPage* pp = pps + j.pp;
    if (ok) {
      pp->body = moved ? dst : j.src;
      pp->body_len = moved ? static_cast<int32_t>(v0 + bytes) : static_cast<int32_t>(j.src_len);
      pp->dblocks = static_cast<int32_t>(values);
    } else {
      // the page keeps its level bytes only: later stages find no values
      // (and the walk does not read the value table, which this page did not
      // fill)
      pp->body = j.src;
      pp->body_len = static_cast<int32_t>(v0);
      pp->vtab = 0;
      report(st, static_cast<uint32_t>(sm.flag), j.page, WHERE_TRANSCODE, sm.detail);
    }
  }
}

// Bytes b of values [k, k + 4) in the low to high bytes of a word, from the
// stream that starts at s + b * n (aligned loads of the words around them).
__device__ __forceinline__ uint32_t bss_word(const uint8_t* s, uint64_t n, uint32_t b, uint64_t k) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(s) + static_cast<uint64_t>(b) * n + k;
  const uint32_t* q = reinterpret_cast<const uint32_t*>(a & ~uintptr_t(3));
  const uint32_t sh = static_cast<uint32_t>(a & 3) * 8;
  const uint32_t lo = __ldg(q);
  return sh ? __funnelshift_r(lo, __ldg(q + 1), sh) : lo;
}

// Four words of four bytes each, transposed.
__device__ __forceinline__ void bss_transpose(uint32_t (&w)[4]) {
  const uint32_t a = __byte_perm(w[0], w[1], 0x5140), b = __byte_perm(w[0], w[1], 0x7362);
  const uint32_t c = __byte_perm(w[2], w[3], 0x5140), d = __byte_perm(w[2], w[3], 0x7362);
  w[0] = __byte_perm(a, c, 0x5410);
  w[1] = __byte_perm(a, c, 0x7632);
  w[2] = __byte_perm(b, d, 0x5410);
  w[3] = __byte_perm(b, d, 0x7632);
}

// BYTE_STREAM_SPLIT pages, blockIdx.y the job: four values a thread and step,
// one aligned word of each stream, 16-byte stores.  The new body starts where
// its values fall on a 16-byte boundary.  Every whole value of the streams is
// written.
// A block for every 8 KiB of the largest page (a step of its threads, at 8-byte
// values), at most 32: with 32 for any page, 8192 pages of 2 KiB took 974 us a
// read, so 714 (and 64 KiB pages, 2^23 rows, 319 instead of 356).
constexpr uint32_t BSS_BLOCK_BYTES = 8 << 10;
__global__ void __launch_bounds__(256) k_bss(const TranscodeJob* jobs, PlanPage* pps, DevStatus* st) {
  const TranscodeJob j = jobs[blockIdx.y];
  if (j.enc != ENC_BSS) return;
  uint32_t v0;
  int detail;
  const uint32_t w = static_cast<uint32_t>(j.width);
  bool ok = tc_levels(j, &v0, &detail);
  if (ok && (w == 0 || (j.src_len - v0) % w)) {
    ok = false;
    detail = 40;
  }
  uint8_t* body = j.dst + ((16 - (v0 & 15)) & 15);  // (the scratch holds 32 bytes more than the page)
  const uint32_t bytes = j.src_len - v0;
  const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x, step = gridDim.x * blockDim.x;
  if (ok) {
    const uint64_t n = bytes / w;
    const uint8_t* s = j.src + v0;
    uint8_t* d = body + v0;
    const uint64_t n4 = w == 4 || w == 8 ? n / 4 : 0;
    for (uint64_t g = tid; g < n4; g += step) {
      uint32_t lo[4], hi[4];
#pragma unroll
      for (uint32_t b = 0; b < 4; ++b) {
        lo[b] = bss_word(s, n, b, 4 * g);
        hi[b] = w == 8 ? bss_word(s, n, b + 4, 4 * g) : 0u;
      }
      bss_transpose(lo);
      if (w == 4) {
        reinterpret_cast<uint4*>(d)[g] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      } else {
        bss_transpose(hi);
        reinterpret_cast<uint4*>(d)[2 * g] = make_uint4(lo[0], hi[0], lo[1], hi[1]);
        reinterpret_cast<uint4*>(d)[2 * g + 1] = make_uint4(lo[2], hi[2], lo[3], hi[3]);
      }
    }
    for (uint64_t k = 4 * n4 + tid; k < n; k += step)
      for (uint32_t b = 0; b < w; ++b) d[k * w + b] = static_cast<uint8_t>(ld_u8(s + static_cast<uint64_t>(b) * n + k));
    for (uint32_t i = tid; i < v0; i += step) body[i] = static_cast<uint8_t>(ld_u8(j.src + i));
  }
  if (tid == 0) {
    PlanPage* pp = pps + j.pp;
    pp->body = ok ? body : j.src;
    pp->body_len = static_cast<int32_t>(ok ? v0 + bytes : v0);
    if (!ok) {
      pp->vtab = 0;
      report(st, DERR_CORRUPT, j.page, WHERE_TRANSCODE, detail);
    }
  }
}

}  // namespace

void launch_transcode(const TranscodeJob* jobs, int n, int n_bss, uint32_t max_bss, PlanPage* pps, uint8_t* pool,
                      uint64_t pool_cap, uint32_t* counters, uint64_t* vpos, DevStatus* st, cudaStream_t s) {
  if (n <= 0) return;
  if (n_bss > 0) {
    const unsigned want = max_bss / BSS_BLOCK_BYTES + 1, blocks = want < 32 ? want : 32;
    launch_slices(n, [&](int at, int m) { k_bss<<<dim3(blocks, m), 256, 0, s>>>(jobs + at, pps, st); });
  }
  if (n_bss == n) return;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_transcode, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(TcSmem));
    attr = true;
  }
  k_transcode<<<n, TC_THREADS, sizeof(TcSmem), s>>>(jobs, pps, pool, pool_cap,
                                                    reinterpret_cast<unsigned long long*>(counters + TC_POOL_COUNTER),
                                                    vpos, st);
}

}  // namespace pqi
