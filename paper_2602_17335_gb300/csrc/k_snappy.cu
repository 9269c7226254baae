// K1 — Snappy page decompression, one thread block per page.
//
// Parquet compresses every page body separately with its chunk's codec
// (paper Section 2; Section 3 "No Unnecessary Compression" weighs its cost).
// A raw Snappy block is a ULEB128 length followed by elements chosen by the
// low two tag bits: a literal (length in the tag, or in 1-4 following
// bytes) or a copy of `length` bytes from `offset` bytes back in the output
// (1-, 2- or 4-byte offsets).  Copies are defined byte by byte, so an offset
// smaller than the length repeats a pattern.
//
// Element headers form a chain: one thread stepping along it takes 250-300
// cycles an element (64-80 dependent instructions), which used to be the
// whole cost of element-dense pages.  Here the block computes, for every
// byte of the staged input window, where the next header would be if a
// header started there (independent, a dozen instructions a byte), and
// doubles that map four times; thread 0 then steps 16 elements at a time
// (one shared load) and the block fills in the rest.  All headers of the
// batch are decoded together, output positions come from a block scan, and
// the bytes are produced by lz_run (lz_exec.cuh), which has no order between
// elements either.  Windows with few elements (literal-heavy pages) are
// stepped through serially instead: the tables would cost more.  Literals
// that leave the window go straight from input to output, all warps copying.
//
// The compressed page streams through two shared-memory windows filled by
// the bulk-copy engine (the next window is in flight while the current one
// is decoded).
#include "dev_util.cuh"
#include "lz_exec.cuh"
#include "snappy_job.h"

namespace pqi {

// Lane 0's input windows, all scalars (they stay in registers): the current
// window (*0) and the other one (*1), swapped when the parse moves on.
// Window offsets are input offsets modulo 2^32 (a window may start up to 15
// bytes before the input).
struct SnIn {
  const uint8_t* in;
  uint32_t in_len;
  uint8_t* b0;
  uint8_t* b1;
  uint64_t* m0;
  uint64_t* m1;
  uint32_t w0, w1, n0, n1, p0, p1;
  uint32_t e1;  // a copy into window 1 is in flight
  uint32_t cap; // window bytes
};

__device__ __forceinline__ void sn_swap(SnIn& s) {
  uint8_t* tb = s.b0; s.b0 = s.b1; s.b1 = tb;
  uint64_t* tm = s.m0; s.m0 = s.m1; s.m1 = tm;
  uint32_t t = s.w0; s.w0 = s.w1; s.w1 = t;
  t = s.n0; s.n0 = s.n1; s.n1 = t;
  t = s.p0; s.p0 = s.p1; s.p1 = t;
}

// Copy of input [from, from + s.cap) (16-byte aligned start, at most 16
// bytes past the input) into buffer `buf`.
__device__ __forceinline__ void sn_issue(const SnIn& s, uint8_t* buf, uint64_t* bar, uint32_t from, uint32_t* w,
                                         uint32_t* n) {
  const uintptr_t base = reinterpret_cast<uintptr_t>(s.in);
  const uintptr_t a = (base + from) & ~uintptr_t(15);
  const uintptr_t lim = (base + s.in_len + 16) & ~uintptr_t(15);
  uint32_t bytes = static_cast<uint32_t>(lim > a ? lim - a : 16);
  if (bytes > s.cap) bytes = s.cap;
  if (bytes < 16) bytes = 16;
  *w = static_cast<uint32_t>(a - base);
  *n = bytes;
  fence_proxy_async_smem();
  mbar_arrive_expect_tx(bar, bytes);
  bulk_g2s(buf, reinterpret_cast<const void*>(a), bytes, bar);
}

__device__ __forceinline__ void sn_prefetch(SnIn& s) {
  const uint32_t end = s.w0 + s.n0;  // input offset just past window 0
  if (end < s.in_len) {  // input left beyond window 0
    sn_issue(s, s.b1, s.m1, end - 16, &s.w1, &s.n1);
    s.e1 = 1;
  } else {
    s.n1 = 0;
  }
}

// 32-bit load from a shared-memory address (the windows are read this way
// on the serial header chains: fewer and cheaper loads than bytes through
// generic pointers).
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}

// Makes input bytes [p, p + 5) readable in window 0 (bytes past the input
// end are slack).  False if a copy never arrived.
__device__ __forceinline__ bool sn_ensure(SnIn& s, uint32_t p) {
  if (p - s.w0 < s.n0 && (p - s.w0 + 5 <= s.n0 || s.w0 + s.n0 >= s.in_len)) return true;
  if (s.e1) {
    const bool ok = mbar_wait(s.m1, s.p1);
    s.p1 ^= 1u;
    s.e1 = 0;
    if (!ok) return false;
    if (p - s.w1 < s.n1 && (p - s.w1 + 5 <= s.n1 || s.w1 + s.n1 >= s.in_len)) {
      sn_swap(s);
      sn_prefetch(s);
      return true;
    }
  }
  // a jump past the prefetched window (a long literal): load at p
  sn_issue(s, s.b1, s.m1, p, &s.w1, &s.n1);
  const bool ok = mbar_wait(s.m1, s.p1);
  s.p1 ^= 1u;
  if (!ok) return false;
  sn_swap(s);
  sn_prefetch(s);
  return true;
}

// The element whose header sits at input offset pa, from its bytes h[0..4]
// (bytes past the input are never used): kind, length, argument (literal:
// input offset of its bytes; copy: back offset) and the next header's input
// offset.  False when the header or the literal runs past the input.
__device__ __forceinline__ bool sn_hdr(uint32_t tag, uint32_t x, uint32_t pa, uint32_t in_len, uint32_t* kind,
                                       uint32_t* len, uint32_t* arg, uint32_t* next) {
  const uint32_t k = tag & 3, t6 = tag >> 2, left = in_len - pa - 1;  // bytes after the tag
  uint32_t l, a, hl;
  if (k == 0) {
    const uint32_t nb = t6 < 60 ? 0u : t6 - 59;
    const uint32_t vm = nb == 0 ? t6 : (nb == 4 ? x : (x & ((1u << (8 * nb)) - 1u)));
    if (nb > left || vm == 0xffffffffu) return false;
    l = vm + 1;
    hl = 1 + nb;
    if (l > left - nb) return false;
    a = pa + hl;
  } else {
    hl = k == 1 ? 2u : (k == 2 ? 3u : 5u);
    if (hl - 1 > left) return false;
    l = k == 1 ? 4 + (t6 & 7) : t6 + 1;
    a = k == 1 ? (((tag >> 5) << 8) | (x & 0xffu)) : (k == 2 ? (x & 0xffffu) : x);
  }
  *kind = k;
  *len = l;
  *arg = a;
  *next = pa + hl + (k == 0 ? l : 0u);
  return true;
}

// Bytes [q, q + 5) of a window as (tag, the 4 bytes after it), from two
// 32-bit shared loads (the window buffer is readable for 16 bytes past its
// end).
__device__ __forceinline__ void sn_bytes5(uint32_t sa, uint32_t* tag, uint32_t* x) {
  const uint32_t a = sa & ~3u, sh = (sa & 3u) * 8;
  const uint32_t lo = lds32(a), hi = lds32(a + 4);
  *tag = __funnelshift_r(lo, hi, sh) & 0xffu;
  *x = __funnelshift_rc(lo, hi, sh + 8);  // (a shift of 32 gives hi)
}

// A page's block: kThreads threads, kWin bytes per input window.  Two
// shapes: pages of at least the block threshold take 16 warps and 8 KB
// windows (a page's latency counts), the many small pages of other files 4
// warps and 2 KB windows (more of them resident).
template <int kThreads, uint32_t kWin>
struct SnShape {
  static constexpr int kEl = 4 * kThreads < 1024 ? 4 * kThreads : 1024;  // elements of a batch
  static constexpr int kPer = kEl / kThreads;       // elements a thread decodes
  static constexpr uint32_t kChunk = kWin > 4096 ? 8192 : 2 * kWin;  // output resolved at a time
  static constexpr uint32_t kRing = 4 * kChunk;
  static constexpr uint32_t kOut = 4 * kChunk;      // output of a batch (less its long literal)
};
// Headers found in a window of kWin bytes, at most kEl of them.
template <uint32_t kWin, int kEl>
struct SnHeaders {
  static constexpr uint32_t kTab = kWin + 16;
  uint16_t j1[kTab];       // next header after the one at each window byte
  uint16_t jab[2 * kTab];  // doubled maps
  uint16_t pos[kEl];       // window offsets of the headers
  uint16_t hop[kEl / 16];
  int32_t n, nh;           // headers, hops
};
template <int kThreads, uint32_t kWin>
struct __align__(16) SnBlock {
  using Sh = SnShape<kThreads, kWin>;
  uint8_t ring[Sh::kRing];
  uint8_t win[2][kWin + 32];
  LzRec rec[Sh::kEl];
  SnHeaders<kWin, Sh::kEl> h;  // (its doubled maps are lz_run's notes afterwards)
  uint32_t mask[Sh::kOut / 32 + 2];
  uint64_t bar[2];
  uint32_t tmp[32];
  uint32_t w0, n0, wsel, bad;       // the window of the batch
  int32_t cut, act;                 // first element not in the batch and why
  uint32_t total, next;             // output of the batch's elements; input offset after it
  uint32_t larg, llen;              // the long literal that ends the batch
  SnIn in;                          // thread 0's window state
};
constexpr uint16_t SN_NONE = 0xffffu;  // the next header lies outside the tables
constexpr uint32_t kAhead = 128 * 1024; // input bytes asked into L2 ahead of a page's position
constexpr int SN_SERIAL = 64;          // headers per batch on the serial path
constexpr int SN_DENSE = 24;           // windows with at least this many elements take the tables

// Bytes from a header at a window byte to the next header (its tag and the
// four bytes after it; nothing is checked: only true headers are, later).
__device__ __forceinline__ uint32_t sn_advance(uint32_t tag, uint32_t x) {
  const uint32_t kind = tag & 3;
  uint32_t adv = kind ? (0x5320u >> (4 * kind)) & 15u : (tag >> 2) + 2;
  if (kind == 0 && tag >= 240) {  // literal lengths of 1-4 bytes
    const uint32_t nb = (tag >> 2) - 59;
    const uint32_t lv = x & (0xffffffffu >> (32 - 8 * nb));
    adv = (lv < 0xfffffu ? lv : 0xfffffu) + nb + 2;
  }
  return adv;
}

// Headers of window bytes [q0, L) from the one at q0 on, into S.pos (at most
// kEl; the last one found may lead past L).  Block-collective; ends with a
// barrier.
template <int kThreads, uint32_t kWin, int kEl>
__device__ void sn_find_headers(SnHeaders<kWin, kEl>& S, const uint8_t* wb, uint32_t q0, uint32_t L, bool dense) {
  using H = SnHeaders<kWin, kEl>;
  if (!dense) {
    if (threadIdx.x == 0) {
      int nb = 0;
      uint32_t q = q0;
      const uint32_t sb = smem_u32(wb);
      while (nb < SN_SERIAL) {
        S.pos[nb++] = static_cast<uint16_t>(q);
        uint32_t tag, x;
        sn_bytes5(sb + q, &tag, &x);
        q += sn_advance(tag, x);
        if (q >= L) break;
      }
      S.n = nb;
    }
    __syncthreads();
    return;
  }
  const uint32_t* w32 = reinterpret_cast<const uint32_t*>(wb);
  constexpr int G = (kWin / 4 + kThreads - 1) / kThreads;  // groups of four window bytes per thread
  const uint32_t g0 = (q0 >> 2) + threadIdx.x;
  {
    uint32_t a[G], b[G];
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const uint32_t g = g0 + i * kThreads;
      a[i] = 4 * g < L ? w32[g] : 0u;
      b[i] = 4 * g < L ? w32[g + 1] : 0u;
    }
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const uint32_t g = g0 + i * kThreads;
      uint32_t v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t tag = (a[i] >> (8 * k)) & 0xffu;
        const uint32_t x = k == 3 ? b[i] : __funnelshift_r(a[i], b[i], 8 * (k + 1));
        const uint32_t nx = 4 * g + k + sn_advance(tag, x);
        v[k] = nx < L ? nx : SN_NONE;
      }
      if (4 * g < L) *reinterpret_cast<uint2*>(S.j1 + 4 * g) = make_uint2(v[0] | (v[1] << 16), v[2] | (v[3] << 16));
    }
  }
  __syncthreads();
  const uint16_t* src = S.j1;
#pragma unroll 1
  for (int r = 0; r < 4; ++r) {  // 2, 4, 8, 16 elements
    uint16_t* dst = S.jab + ((r & 1) ? H::kTab : 0u);
    uint2 m[G];
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const uint32_t g = g0 + i * kThreads;
      m[i] = 4 * g < L ? *reinterpret_cast<const uint2*>(src + 4 * g) : make_uint2(0xffffffffu, 0xffffffffu);
    }
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const uint32_t h[4] = {m[i].x & 0xffffu, m[i].x >> 16, m[i].y & 0xffffu, m[i].y >> 16};
      uint32_t v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = h[k] == SN_NONE ? SN_NONE : src[h[k]];
      m[i] = make_uint2(v[0] | (v[1] << 16), v[2] | (v[3] << 16));
    }
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const uint32_t g = g0 + i * kThreads;
      if (4 * g < L) *reinterpret_cast<uint2*>(dst + 4 * g) = m[i];
    }
    __syncthreads();
    src = dst;
  }
  if (threadIdx.x == 0) {
    int nb = 0, nh = 0;
    uint32_t q = q0, nx = src[q];
    while (nb + 16 <= kEl && nx != SN_NONE) {
      S.hop[nh++] = static_cast<uint16_t>(q);
      nb += 16;
      q = nx;
      nx = src[q];
    }
    while (nb < kEl) {
      nx = S.j1[q];
      S.pos[nb++] = static_cast<uint16_t>(q);
      if (nx == SN_NONE) break;
      q = nx;
    }
    S.n = nb;
    S.nh = nh;
  }
  __syncthreads();
  for (int h = threadIdx.x; h < S.nh; h += kThreads) {
    uint32_t q = S.hop[h];
#pragma unroll 4
    for (int k = 0; k < 16; ++k) {
      const uint32_t nx = S.j1[q];
      S.pos[16 * h + k] = static_cast<uint16_t>(q);
      q = nx;
    }
  }
  __syncthreads();
}

// One Snappy element stream: in[ip, in_len) into out[0, out_len), which no
// copy reaches out of.  par: thread 0's phase parities of the window barriers.
template <int kThreads, uint32_t kWin>
__device__ __forceinline__ void sn_decode(SnBlock<kThreads, kWin>& S, const uint8_t* in, uint32_t ip, uint32_t in_len, uint8_t* out,
                          uint32_t out_len, uint32_t* par, int page, DevStatus* st) {
  using Sh = SnShape<kThreads, kWin>;
  const int tid = threadIdx.x;
      const uint32_t va = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(out) & 31);
      uint8_t* vout = out - va;
      // thread 0's window state
      SnIn& sin = S.in;
      if (tid == 0) sin = SnIn{in, in_len, S.win[0], S.win[1], &S.bar[0], &S.bar[1], 0, 0, 0, 0, par[0], par[1], 0, kWin};
      bool loaded = false, lost = false;  // thread 0's: the first window was asked for; a copy never arrived
      uint32_t op = 0;
      int bad = 0;         // 1 malformed, 2 a copy never arrived
      bool dense = false;  // the last window held many elements
      uint32_t vfloor = 0; // the ring holds nothing below this position
      uint32_t fetched = 0;  // input asked into L2 ahead of the windows
      // each element consumes >= 2 input bytes, so in_len bounds the batches
      for (uint32_t guard = 0; guard <= in_len && ip < in_len; ++guard) {
        if (tid == 0) {
          bool ok = true;
          if (!loaded) {
            sn_issue(sin, sin.b0, sin.m0, ip, &sin.w0, &sin.n0);
            ok = mbar_wait(sin.m0, sin.p0);
            sin.p0 ^= 1u;
            if (ok) sn_prefetch(sin);
            loaded = true;
          } else {
            ok = !lost && sn_ensure(sin, ip);
          }
          S.bad = ok ? 0u : 2u;
          S.w0 = sin.w0;
          S.n0 = sin.n0;
          S.wsel = sin.b0 == S.win[1] ? 1u : 0u;
          S.cut = Sh::kEl;
          S.act = 0;
          S.total = 0;
        }
        for (uint32_t w = tid; w < Sh::kOut / 32 + 2; w += kThreads) S.mask[w] = 0;
        while (fetched < in_len && fetched < ip + kAhead) {
          if (fetched + 128 * tid < in_len)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(in + fetched + 128 * tid));
          fetched += 128 * kThreads;
        }
        __syncthreads();
        if (S.bad) {
          bad = 2;
          break;
        }
        const uint32_t w0 = S.w0, n0 = S.n0;
        const uint8_t* wb = S.win[S.wsel];
        const uint32_t q0 = ip - w0;
        const uint32_t L = w0 + n0 >= in_len ? in_len - w0 : n0 - 4;  // headers below L have all their bytes here
        sn_find_headers<kThreads>(S.h, wb, q0, L, dense);
        const int n = S.h.n;
        dense = n >= SN_DENSE;
        // the warp's elements: `seg` in a row, lane l the (32 u + l)-th (src: a
        // literal's input offset | LZ_LIT, or a copy's back offset; len 0:
        // malformed)
        constexpr int kWarps = kThreads / 32;
        const int lane = tid & 31, warp = tid >> 5;
        const int seg = 32 * ((n + 32 * kWarps - 1) / (32 * kWarps));
        uint32_t len[Sh::kPer], src[Sh::kPer], at[Sh::kPer];
        uint32_t run = 0;
  #pragma unroll
        for (int u = 0; u < Sh::kPer; ++u) {
          const int e = warp * seg + 32 * u + lane;
          len[u] = src[u] = 0;
          if (32 * u < seg && e < n) {
            uint32_t tag, x, kind, nx;
            sn_bytes5(smem_u32(wb) + S.h.pos[e], &tag, &x);
            if (!sn_hdr(tag, x, w0 + S.h.pos[e], in_len, &kind, &len[u], &src[u], &nx)) len[u] = 0;
            else if (kind == 0) src[u] |= LZ_LIT;
            else if (src[u] & LZ_LIT) len[u] = 0;  // an offset of 2 GB or more is past any output
          }
        }
  #pragma unroll
        for (int u = 0; u < Sh::kPer; ++u) {
          uint32_t incl = len[u];
  #pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
          }
          at[u] = run + incl - len[u];
          run += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) S.tmp[warp] = run;
        __syncthreads();
        {
          const uint32_t tv = lane < kWarps ? S.tmp[lane] : 0u;
          uint32_t incl = tv;
  #pragma unroll
          for (int o = 1; o < kWarps; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
          }
          const uint32_t base = __shfl_sync(0xffffffffu, incl - tv, warp);
  #pragma unroll
          for (int u = 0; u < Sh::kPer; ++u) at[u] += base;
        }
        // the batch ends before its first element that is malformed, is a
        // literal reaching past the window, or exceeds the batch's output
        auto valid = [&](uint32_t o, uint32_t l, uint32_t sr) {
          const uint32_t p = op + o;
          return l != 0 && p <= out_len && l <= out_len - p && ((sr & LZ_LIT) || (sr != 0 && sr <= p));
        };
        auto longlit = [&](uint32_t l, uint32_t sr) { return (sr & LZ_LIT) && ((sr & ~LZ_LIT) - w0) + l > n0; };
  #pragma unroll
        for (int u = 0; u < Sh::kPer; ++u) {
          const int e = warp * seg + 32 * u + lane;
          const bool in_list = 32 * u < seg && e < n;
          const bool stop = in_list && (!valid(at[u], len[u], src[u]) || longlit(len[u], src[u]) ||
                                        at[u] + len[u] > Sh::kOut - 32);
          const uint32_t b = __ballot_sync(0xffffffffu, stop);
          if (b && lane == 0) atomicMin(&S.cut, warp * seg + 32 * u + __ffs(b) - 1);
        }
        __syncthreads();
        const int ne = S.cut < n ? S.cut : n;
        const uint32_t vb = va + op;
  #pragma unroll
        for (int u = 0; u < Sh::kPer; ++u) {
          const int e = warp * seg + 32 * u + lane;
          if (32 * u < seg && e < n) {
            if (e < ne) {
              const uint32_t a = vb + at[u];
              S.rec[e] = LzRec{a, (src[u] & LZ_LIT) ? LZ_LIT | ((src[u] & ~LZ_LIT) - w0) : src[u]};
              atomicOr(S.mask + ((a >> 5) - (vb >> 5)), 1u << (a & 31));
              if (e == ne - 1) S.total = at[u] + len[u];
              if (e == n - 1) {
                uint32_t tag, x;
                sn_bytes5(smem_u32(wb) + S.h.pos[e], &tag, &x);
                S.next = w0 + S.h.pos[e] + sn_advance(tag, x);
              }
            } else if (e == ne) {  // the element after the batch
              const bool lit = longlit(len[u], src[u]);
              S.act = !valid(at[u], len[u], src[u]) ? 1 : (lit ? 2 : 0);
              S.larg = src[u] & ~LZ_LIT;
              S.llen = len[u];
              S.next = lit ? (src[u] & ~LZ_LIT) + len[u] : w0 + S.h.pos[e];
            }
          }
        }
        __syncthreads();
        const uint32_t total = S.total, next = S.next;
        const int act = S.act;
        if (act == 1) {
          bad = 1;
          break;
        }
        if (act == 2 && tid == 0 && next < in_len) {
          // the window behind the long literal, on its way while the batch
          // and the literal are written
          if (sin.e1) {
            lost = !mbar_wait(sin.m1, sin.p1);
            sin.p1 ^= 1u;
            sin.e1 = 0;
          }
          if (!lost && (next - sin.w1 >= sin.n1 || (next - sin.w1 + 5 > sin.n1 && sin.w1 + sin.n1 < in_len))) {
            sn_issue(sin, sin.b1, sin.m1, next, &sin.w1, &sin.n1);
            sin.e1 = 1;
          }
        }
        if (total)
          lz_run<kThreads, Sh::kChunk, Sh::kRing>(S.rec, ne, S.mask, S.ring, S.h.jab, vout, vb, vb + total, vfloor,
                                                  [wb](uint32_t i) { return wb + i; });
        op += total;
        if (act == 2) {  // straight to the output; the ring starts anew behind it
          lz_block_copy<kThreads>(out + op, in + S.larg, S.llen);
          op += S.llen;
          vfloor = va + op;
        }
        ip = next;
        __syncthreads();
      }
      __syncthreads();
  if (tid == 0) {
    // settle the window copy still in flight before the buffers are reused
    if (sin.e1) {
      mbar_wait(sin.m1, sin.p1);
      sin.p1 ^= 1u;
      sin.e1 = 0;
    }
    if (bad == 2) report(st, DERR_TIMEOUT, page, WHERE_SNAPPY, 5);
    else if (bad || op != out_len || ip != in_len) report(st, DERR_CORRUPT, page, WHERE_SNAPPY, 4);
    // carry the physical buffers' parities to the next stream
    const bool sw0 = sin.b0 == S.win[0];
    par[0] = sw0 ? sin.p0 : sin.p1;
    par[1] = sw0 ? sin.p1 : sin.p0;
  }
}

// Length preamble of a page's stream: its bytes, 0 when it does not parse or
// does not declare out_len bytes.
__device__ __forceinline__ uint32_t sn_preamble(const uint8_t* in, uint32_t in_len, uint32_t out_len) {
  uint64_t declared = 0;
  const int pl = uleb([&](uint32_t k) { return static_cast<uint32_t>(__ldg(in + k)); }, 0, in_len, &declared);
  return declared == out_len ? static_cast<uint32_t>(pl) : 0u;
}

// kFragments: the work list is the fragments [first, first + n_work) of split
// pages, else jobs [0, n_work) (split pages skipped: their fragments are work
// of their own).
template <int kThreads, uint32_t kWin, bool kFragments>
__global__ void __launch_bounds__(kThreads, kThreads == 512 ? 2 : 5)
    k_snappy(const SnappyJob* __restrict__ jobs, int first, int n_work, SnapState ss, DevStatus* st) {
  extern __shared__ __align__(16) uint8_t sn_smem[];
  SnBlock<kThreads, kWin>& S = *reinterpret_cast<SnBlock<kThreads, kWin>*>(sn_smem);
  const int tid = threadIdx.x;
  if (tid == 0) {
    mbar_init(&S.bar[0], 1);
    mbar_init(&S.bar[1], 1);
  }
  fence_mbar_init();
  __syncthreads();
  uint32_t par[2] = {0, 0};
  for (int w = blockIdx.x; w < n_work; w += gridDim.x) {
    const SnappyJob jb = jobs[kFragments ? ss.owner[first + w] : w];
    if (jb.codec != CODEC_SNAPPY) continue;  // another codec's kernel takes it
    const uint8_t* in = jb.src + jb.prefix;
    uint32_t in_len = jb.src_len - jb.prefix;
    uint8_t* out = jb.dst + jb.prefix;
    uint32_t out_len = jb.dst_len - jb.prefix;
    uint32_t ip = 0;
    if (kFragments) {
      const uint32_t k = first + w - jb.sub;
      if (!ss.bad[jb.sub]) {
        const uint32_t a = ss.start[jb.sub + k];
        const uint32_t b = k + 1 < jb.nsub ? ss.start[jb.sub + k + 1] : in_len;
        in += a;
        in_len = b - a;
        out += static_cast<uint64_t>(k) * SNAPPY_FRAGMENT;
        out_len = k + 1 < jb.nsub ? SNAPPY_FRAGMENT : out_len - k * SNAPPY_FRAGMENT;
      } else if (k == 0) {  // not framed: the whole page here
        ip = sn_preamble(in, in_len, out_len);
        if (ip == 0) {
          if (tid == 0) report(st, DERR_CORRUPT, jb.page, WHERE_SNAPPY, 3);
          continue;
        }
      } else {
        continue;
      }
    } else {
      if (jb.nsub > 1) continue;
      if (jb.prefix > jb.src_len || jb.prefix > jb.dst_len || (jb.raw && jb.src_len != jb.dst_len)) {
        if (tid == 0) report(st, DERR_CORRUPT, jb.page, WHERE_SNAPPY, jb.raw ? 2 : 1);
        continue;
      }
      lz_block_copy<kThreads>(jb.dst, jb.src, jb.raw ? jb.src_len : jb.prefix);  // V2 levels are never compressed
      if (jb.raw) continue;
      ip = sn_preamble(in, in_len, out_len);
      if (ip == 0) {
        if (tid == 0) report(st, DERR_CORRUPT, jb.page, WHERE_SNAPPY, 3);
        continue;
      }
    }
    sn_decode(S, in, ip, in_len, out, out_len, par, jb.page, st);
  }
}

// ------------------------------------------------------------------ split pages

// Element scan of the split pages, a thread block per segment of
// SNAPPY_SEGMENT input bytes (cut at multiples of it from the input's first
// 16-byte boundary on).  Which bytes of a segment are headers depends on
// where the last element before it ends, so the page is one chain; but where
// the chain leaves the segment can be computed for every possible entry at
// once, right to left: the exit from each byte's 32 bytes (a thread each,
// its bytes in registers), from its 1 KB (a warp each), 4 KB and the segment,
// one lookup per byte and level.  A block then waits only for its
// predecessor's exit, looks up its own and passes that on (about a
// microsecond a segment), while all segments' maps are built in parallel.
// With its entry known, one thread hops over the 1 KB blocks, each warp over
// the 32-byte runs of its block, each lane over the elements of its run: the
// lanes' outputs are added up, and with the output of the segments before
// they record which elements start a 64 KiB fragment.  An element that spans
// two fragments, a copy that reaches out of its fragment, or anything the
// decoder would reject marks the page: it is then decompressed whole, by one
// block, which reports what is wrong.
//
// Bound by the maps' lookups (issue and shared-memory latency) and, for dense
// segments, by the lanes' elements (about 80 cycles each, 16 at most).  With
// the elements listed by the decoder's windowed tables instead of the maps' own
// levels, and one 32-bit map whose levels replaced one another (a barrier per
// KB), the scan of an INT64 dictionary column (2^23 rows, 1 MiB pages, 3600
// elements a segment) took 210 us, now 120, its 1 MiB dictionary pages' 140,
// now 100.
//
// The list's pages are cut into up to SNAPPY_RUNS runs of whole pages,
// each with a ticket counter from which blocks take its segments in order
// (and go on to the next run when one is used up): the segment a block waits
// for has always been taken by a block that is running, and the waits of
// different runs overlap (in one run, 64 pages of 32 segments took 560 us, the
// chain's 2048 hops).  Waits are bounded all the same.
constexpr int SC_THREADS = 1024;
constexpr uint32_t SC_POLLS = 1u << 22;
constexpr uint32_t SC_NONE = 0xffffffffu;
// Maps by segment byte (at sc_slot): where the chain from a header there
// leaves the byte's 32 bytes / 1 KB / (4 KB, then) segment: a byte of the
// segment, or SC_LAST | the header of the element that leads out of the segment.
constexpr uint32_t SC_LAST = 0x8000u;
struct __align__(16) SnScan {
  uint16_t run[SNAPPY_SEGMENT], blk[SNAPPY_SEGMENT], seg[SNAPPY_SEGMENT];
  uint8_t stage[SNAPPY_SEGMENT + 32];
  uint64_t bar, tmp[32];
  uint32_t block_entry[32];  // the first header of each 1 KB
  uint32_t ticket, entry, next, from, to, done;
  int32_t job;
};

// Map slot of a segment byte: its place in its 32 bytes is permuted by the
// number of the 64 bytes, so that the same place of 32 successive runs falls
// on 32 banks.
__device__ __forceinline__ uint32_t sc_slot(uint32_t p) { return p ^ ((p >> 5) & 30u); }

// One 64-bit word written by another block of this launch: polled until its
// flag is set.  0 when it never is.
__device__ __forceinline__ unsigned long long sn_await(const unsigned long long* p) {
  for (uint32_t i = 0; i < SC_POLLS; ++i) {
    const unsigned long long v = *reinterpret_cast<const volatile unsigned long long*>(p);
    if (v & SN_SET) return v;
  }
  return 0;
}

// The job that holds segment g (one warp, 32 ways a step): the last one that
// starts at or before it.
__device__ __forceinline__ int sc_job(const SnappyJob* jobs, int n, uint32_t g, int lane) {
  int lo = 0;
  while (n > 1) {
    const int step = (n + 31) / 32;
    const uint32_t m = __ballot_sync(0xffffffffu, lane * step < n && jobs[lo + lane * step].seg <= g);
    const int k = 31 - __clz(m | 1u);
    lo += k * step;
    n = n - k * step < step ? n - k * step : step;
  }
  return lo;
}

// Split pages whose elements are long (incompressible values: a literal per
// fragment and a few copies): one thread steps along the page, straight from
// the input, and records its fragments; the scan then leaves the page out.  It
// gives up, and leaves the page to the scan, once elements are shorter than
// SC_LONG bytes on average, or at anything the scan would mark the page for.
// Bound by the latency of a load an element: 64 1 MiB pages of doubles (5
// elements per 32 KB) 89 us and the scan 35, where the scan's maps took 300.
// Data pages only: dictionary pages are few, mostly dense, and waited for
// (giving up on four of them took 24 us of their column's 250).
constexpr uint32_t SC_LONG = 1024;
__global__ void __launch_bounds__(32) k_snappy_long(const SnappyJob* __restrict__ jobs, SnapState ss) {
  if (threadIdx.x != 0) return;
  const SnappyJob jb = jobs[blockIdx.x];
  if (jb.nsub <= 1) return;
  const uint8_t* in = jb.src + jb.prefix;
  const uint32_t in_len = jb.src_len - jb.prefix, out_len = jb.dst_len - jb.prefix;
  uint32_t q = sn_preamble(in, in_len, out_len), o = 0;
  if (q == 0) return;
  for (uint32_t n = 0; q < in_len; ++n) {
    if (n > 16 + q / SC_LONG) return;
    const uint64_t h = ld_unaligned_g(in + q, 8);
    uint32_t kind, len, arg, nx;
    if (!sn_hdr(static_cast<uint32_t>(h) & 0xffu, static_cast<uint32_t>(h >> 8), q, in_len, &kind, &len, &arg, &nx)) return;
    const uint32_t in_frag = o & (SNAPPY_FRAGMENT - 1);
    if (len > SNAPPY_FRAGMENT - in_frag || len > out_len - o || (kind != 0 && (arg == 0 || arg > in_frag))) return;
    if (in_frag == 0) ss.start[jb.sub + o / SNAPPY_FRAGMENT] = q;
    o += len;
    q = nx;
  }
  if (q == in_len && o == out_len) ss.bad[jb.sub + 1] = 1;  // (a split page has three fragments or more)
}

__global__ void __launch_bounds__(SC_THREADS, 1) k_snappy_scan(const SnappyJob* __restrict__ jobs, int n_jobs,
                                                               uint32_t seg_begin, uint32_t n_segs, SnapState ss,
                                                               uint32_t* tickets, DevStatus* st) {
  extern __shared__ __align__(16) uint8_t sn_smem[];
  SnScan& S = *reinterpret_cast<SnScan*>(sn_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) mbar_init(&S.bar, 1);
  fence_mbar_init();
  uint32_t parity = 0;
  // warp 0: the run it takes segments from, whether its bounds are in S, and
  // how many runs it has found used up (a used-up run stays so)
  int run = blockIdx.x % SNAPPY_RUNS, used = 0;
  bool bounded = false;
  for (;;) {
    if (warp == 0) {
      uint32_t t = 0xffffffffu;
      while (used < SNAPPY_RUNS) {
        if (!bounded) {
          // a run starts after the page that holds the segment before its share
          uint32_t bound[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const uint32_t x = static_cast<uint32_t>(static_cast<uint64_t>(n_segs) * (run + i) / SNAPPY_RUNS);
            bound[i] = seg_begin;
            if (x > 0) {
              const SnappyJob& jb = jobs[sc_job(jobs, n_jobs, seg_begin + x - 1, lane)];
              bound[i] = jb.seg + jb.nseg;
            }
          }
          if (lane == 0) {
            S.from = bound[0];
            S.to = bound[1];
          }
          __syncwarp();
          bounded = true;
        }
        if (lane == 0 && S.from < S.to) t = S.from + atomicAdd(tickets + run, 1u);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t < S.to) {
          const int j = sc_job(jobs, n_jobs, t, lane);
          // of a page that k_snappy_long has done, the first segment only
          if (t != jobs[j].seg && ss.bad[jobs[j].sub + 1]) continue;
          if (lane == 0) S.job = j;
          break;
        }
        t = 0xffffffffu;
        run = (run + 1) % SNAPPY_RUNS;
        bounded = false;
        ++used;
        __syncwarp();
      }
      if (lane == 0) S.ticket = t;
    }
    __syncthreads();
    const uint32_t g = S.ticket;
    if (g == 0xffffffffu) break;
    const SnappyJob jb = jobs[S.job];
    const uint32_t k = g - jb.seg;  // segment of the page
    const uint8_t* in = jb.src + jb.prefix;
    const uint32_t in_len = jb.src_len - jb.prefix, out_len = jb.dst_len - jb.prefix;
    if (k == 0) {
      lz_block_copy<SC_THREADS>(jb.dst, jb.src, jb.prefix);  // V2 level bytes, never compressed
      for (uint32_t f = tid; f < jb.nsub; f += SC_THREADS) ss.owner[jb.sub + f] = static_cast<uint32_t>(S.job);
    }
    if (ss.bad[jb.sub + 1]) {
      __syncthreads();
      continue;
    }
    // segment byte p is input byte org + p (the first segment starts at the
    // 16-byte boundary before the input)
    const uint32_t lead = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(in) & 15);
    const uint32_t org = k * SNAPPY_SEGMENT - lead;  // (modulo 2^32)
    const uint32_t left = in_len - org, L = left < SNAPPY_SEGMENT ? left : SNAPPY_SEGMENT;
    // stage the segment and the header bytes after it, at most 16 bytes past
    // the input
    if (tid == 0) {
      const uintptr_t a0 = reinterpret_cast<uintptr_t>(in) - lead + static_cast<uint64_t>(k) * SNAPPY_SEGMENT;
      const uintptr_t lim = (reinterpret_cast<uintptr_t>(in) + in_len + 16) & ~uintptr_t(15);
      uint64_t bytes = lim - a0;
      if (bytes > SNAPPY_SEGMENT + 32) bytes = SNAPPY_SEGMENT + 32;
      fence_proxy_async_smem();
      mbar_arrive_expect_tx(&S.bar, static_cast<uint32_t>(bytes));
      bulk_g2s(S.stage, reinterpret_cast<const void*>(a0), static_cast<uint32_t>(bytes), &S.bar);
    }
    bool staged = mbar_wait(&S.bar, parity);
    if (!staged) staged = mbar_wait(&S.bar, parity) && false;  // (the copy may not outlive its buffer)
    parity ^= 1u;
    const bool all_staged = !__syncthreads_or(!staged);
    if (tid == 0) {
      // the predecessor's exit is there already, and the chain leaves the
      // segment within a few elements (literal-heavy pages): no map needed
      S.done = 0;
      unsigned long long v = 0;
      if (k == 0) {
        const uint32_t pl = all_staged ? sn_preamble(in, in_len, out_len) : 0u;
        v = SN_SET | (pl ? pl : 0xffffffffu);  // (0xffffffff, passed on: the page is decompressed whole)
        S.entry = static_cast<uint32_t>(v);
      } else {
        v = *reinterpret_cast<const volatile unsigned long long*>(ss.exit + g - 1);
      }
      if (v) {
        const uint32_t e = static_cast<uint32_t>(v);
        uint32_t x = e;
        int n = 0;
        for (; n < SN_SERIAL && all_staged && x - org < L; ++n) {
          uint32_t tag, by;
          sn_bytes5(smem_u32(S.stage) + (x - org), &tag, &by);
          x += sn_advance(tag, by);
        }
        if (x - org >= L) {
          *reinterpret_cast<volatile unsigned long long*>(ss.exit + g) = SN_SET | x;
          S.entry = e;
          S.next = x;
          S.done = 1;
        }
      }
    }
    if (tid < 32) S.block_entry[tid] = SC_NONE;
    __syncthreads();
    static_assert(SNAPPY_SEGMENT == 32 * SC_THREADS && SC_THREADS == 32 * 32 && SNAPPY_SEGMENT == SC_LAST,
                  "a run a thread, a block a warp");
    const bool listed = S.done != 0;  // (few elements: thread 0 steps along them, without maps)
    if (!listed) {
      // (bytes past L lead past L: every position a level reads is set)
      {
        const uint4* s4 = reinterpret_cast<const uint4*>(S.stage) + 2 * tid;
        const uint4 lo = s4[0], hi = s4[1];
        const uint32_t w[9] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w,
                               reinterpret_cast<const uint32_t*>(S.stage)[8 * tid + 8]};
        const uint32_t p0 = 32 * tid;
#pragma unroll
        for (int r = 31; r >= 0; --r) {
          const uint32_t a = w[r / 4], b = w[r / 4 + 1];
          const uint32_t tag = (a >> (8 * (r & 3))) & 0xffu;
          const uint32_t by = (r & 3) == 3 ? b : __funnelshift_r(a, b, 8 * ((r & 3) + 1));
          const uint32_t nx = p0 + r + sn_advance(tag, by);
          uint32_t v = nx < L ? nx : SC_LAST | (p0 + r);
          if (v < p0 + 32) v = S.run[sc_slot(v)];
          S.run[sc_slot(p0 + r)] = static_cast<uint16_t>(v);
        }
        __syncwarp();
      }
      for (int i = 31; i >= 0; --i) {
        const uint32_t p = 1024 * warp + 32 * i + lane;
        if (p < L) {
          uint32_t v = S.run[sc_slot(p)];
          if (v < 1024u * warp + 1024u) v = S.blk[sc_slot(v)];
          S.blk[sc_slot(p)] = static_cast<uint16_t>(v);
        }
        __syncwarp();
      }
      __syncthreads();
      for (int j = 3; j >= 0; --j) {  // block j of every 4 KB
#pragma unroll
        for (uint32_t q = 0; q < 8; ++q) {
          const uint32_t p = 4096 * q + 1024 * j + tid;
          if (p < L) {
            uint32_t v = S.blk[sc_slot(p)];
            if (v < 4096 * q + 4096) v = S.seg[sc_slot(v)];
            S.seg[sc_slot(p)] = static_cast<uint16_t>(v);
          }
        }
        __syncthreads();
      }
      for (int q = 6; q >= 0; --q) {
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) {
          const uint32_t p = 4096 * q + 1024 * j + tid;
          if (p < L) {
            const uint32_t v = S.seg[sc_slot(p)];
            if (v < SC_LAST) S.seg[sc_slot(p)] = S.seg[sc_slot(v)];
          }
        }
        __syncthreads();
      }
      // the chain: entry from the segment before, exit to the one after
      if (tid == 0) {
        uint32_t e = S.entry;  // (k == 0)
        bool ok = all_staged;
        if (k > 0) {
          const unsigned long long v = sn_await(ss.exit + g - 1);
          e = static_cast<uint32_t>(v);
          if (!v) {
            ok = false;
            report(st, DERR_TIMEOUT, jb.page, WHERE_SNAPPY, 6);
          }
        }
        uint32_t x = e;
        if (!ok) x = e = 0xffffffffu;  // (passed on: the page is decompressed whole)
        else if (e - org < L) {
          const uint32_t h = S.seg[sc_slot(e - org)] & (SC_LAST - 1);
          uint32_t tag, by;
          sn_bytes5(smem_u32(S.stage) + h, &tag, &by);
          x = org + h + sn_advance(tag, by);
        }
        *reinterpret_cast<volatile unsigned long long*>(ss.exit + g) = SN_SET | x;
        S.entry = e;
        S.next = x;
        if (x <= in_len)  // (not after a failed wait, nor past a literal that overruns the input)
          for (uint32_t q = e - org; q < L;) {
            S.block_entry[q >> 10] = q;
            q = S.blk[sc_slot(q)];
          }
      }
    }
    __syncthreads();
    const uint32_t entry = S.entry, exit = S.next;
    bool good = entry <= in_len && exit <= in_len;
    // the thread's elements: those of its 32 bytes, all of the segment's for
    // thread 0 where it has stepped along them
    uint32_t first = SC_NONE, end = 32 * tid + 32;
    if (listed) {
      end = L;
      if (good && tid == 0) first = entry - org;
    } else {
      for (uint32_t q = S.block_entry[warp]; q < 1024u * warp + 1024u;) {
        if (static_cast<uint32_t>(lane) == ((q >> 5) & 31u)) first = q;
        q = S.run[sc_slot(q)];
      }
    }
    end = end < L ? end : L;
    uint64_t mine = 0;
    for (uint32_t q = first; q < end;) {
      uint32_t tag, x, kind, len, arg, nx;
      sn_bytes5(smem_u32(S.stage) + q, &tag, &x);
      if (!sn_hdr(tag, x, org + q, in_len, &kind, &len, &arg, &nx)) {
        good = false;
        break;
      }
      mine += len;
      q = nx - org;
    }
    uint64_t total;
    const uint64_t o_at = block_exclusive_sum<uint64_t>(mine, S.tmp, &total);
    if (total > out_len) good = false;
    good = !__syncthreads_or(!good);
    if (tid == 0)
      *reinterpret_cast<volatile unsigned long long*>(ss.len + g) = SN_SET | (good ? total : 0u);
    // output of the segments before this one
    uint64_t part = 0;
    for (uint32_t i = tid; i < k; i += SC_THREADS) {
      const unsigned long long v = sn_await(ss.len + jb.seg + i);
      if (!v) good = false;
      part += static_cast<uint32_t>(v);
    }
    uint64_t base;
    block_exclusive_sum<uint64_t>(part, S.tmp, &base);
    if (base > out_len || total > out_len - base) good = false;
    if (good) {
      uint32_t o = static_cast<uint32_t>(base + o_at);
      for (uint32_t q = first; q < end;) {
        uint32_t tag, x, kind, len, arg, nx;
        sn_bytes5(smem_u32(S.stage) + q, &tag, &x);
        sn_hdr(tag, x, org + q, in_len, &kind, &len, &arg, &nx);
        const uint32_t in_frag = o & (SNAPPY_FRAGMENT - 1);
        if (in_frag + len > SNAPPY_FRAGMENT || (kind != 0 && (arg == 0 || arg > in_frag))) good = false;
        if (in_frag == 0 && o / SNAPPY_FRAGMENT < jb.nsub) ss.start[jb.sub + o / SNAPPY_FRAGMENT] = org + q;
        o += len;
        q = nx - org;
      }
      if (k + 1 == jb.nseg && (exit != in_len || base + total != out_len)) good = false;
    }
    if (__syncthreads_or(!good) && tid == 0) atomicOr(ss.bad + jb.sub, 1u);
  }
}

void launch_snappy_scan(const SnappyJob* jobs, int n_jobs, uint32_t seg_begin, uint32_t n_segs, SnapState ss,
                        uint32_t* tickets, bool long_first, int n_sms, DevStatus* st, cudaStream_t s) {
  if (n_jobs <= 0 || n_segs == 0) return;
  static bool attr = false;
  if (!attr) {
    cudaFuncSetAttribute(k_snappy_scan, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(SnScan));
    attr = true;
  }
  const unsigned blocks = n_segs < static_cast<uint32_t>(n_sms) ? n_segs : n_sms;
  if (long_first) k_snappy_long<<<n_jobs, 32, 0, s>>>(jobs, ss);
  k_snappy_scan<<<blocks, SC_THREADS, sizeof(SnScan), s>>>(jobs, n_jobs, seg_begin, n_segs, ss, tickets, st);
}

template <int kThreads, uint32_t kWin, bool kFragments>
static void launch_snappy_shape(const SnappyJob* jobs, int first, int n, SnapState ss, int n_sms, DevStatus* st,
                                cudaStream_t s) {
  constexpr uint32_t smem = sizeof(SnBlock<kThreads, kWin>);
  static int bps = 0;
  if (!bps) {
    cudaFuncSetAttribute(k_snappy<kThreads, kWin, kFragments>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_snappy<kThreads, kWin, kFragments>, kThreads, smem);
    bps = b < 1 ? 1 : b;
  }
  const int blocks = n < n_sms * bps ? n : n_sms * bps;
  k_snappy<kThreads, kWin, kFragments><<<blocks, kThreads, smem, s>>>(jobs, first, n, ss, st);
}

void launch_snappy(const SnappyJob* jobs, int n_jobs, int n_sms, DevStatus* st, cudaStream_t s, bool wide) {
  if (n_jobs <= 0) return;
  // few enough pages for all of them to run at once: the wide shape too
  // (224 pages of 64 KiB: 414 us in the narrow one)
  if (wide || n_jobs <= 2 * n_sms)
    launch_snappy_shape<512, 8192, false>(jobs, 0, n_jobs, SnapState{}, n_sms, st, s);
  else
    launch_snappy_shape<128, 2048, false>(jobs, 0, n_jobs, SnapState{}, n_sms, st, s);
}

void launch_snappy_fragments(const SnappyJob* jobs, int first, int n, SnapState ss, int n_sms, DevStatus* st,
                             cudaStream_t s) {
  if (n > 0) launch_snappy_shape<512, 8192, true>(jobs, first, n, ss, n_sms, st, s);
}

}  // namespace pqi
