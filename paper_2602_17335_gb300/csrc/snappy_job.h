// One page to decompress (K1): built by the planner, read by the Snappy or
// the Zstandard kernel.
#pragma once
#include <stdint.h>

namespace pqi {

// The reference Snappy compressor works on 64 KiB fragments of its input,
// each on its own: no copy reaches into an earlier fragment and no element
// spans two.  The elements of a page whose decompressed stream is longer than
// SNAPPY_SPLIT_MIN are located first (k_snappy_scan, SNAPPY_SEGMENT input
// bytes per thread block); where the page has that structure, its fragments
// are then decompressed by a thread block each.
constexpr uint32_t SNAPPY_FRAGMENT = 65536;
constexpr uint32_t SNAPPY_SPLIT_MIN = 2 * SNAPPY_FRAGMENT;
constexpr uint32_t SNAPPY_SEGMENT = 32768;
constexpr int SNAPPY_RUNS = 16;  // ticket counters of one list's element scan

struct SnappyJob {
  const uint8_t* src;  // stored page body
  uint8_t* dst;        // decompressed page body (capacity dst_len + 16)
  uint32_t src_len;
  uint32_t dst_len;    // expected output bytes, including the verbatim prefix
  uint32_t prefix;     // bytes copied verbatim first (V2 level bytes)
  uint32_t raw;        // 1: no decompression (V2 page with is_compressed = false)
  int32_t page;        // page-table row, for error reports
  int32_t codec;       // CODEC_SNAPPY or CODEC_ZSTD: the kernel of the other codec skips the job
  uint32_t nsub;       // > 1: a split page, whose fragments are numbers [sub, sub + nsub) of the plan's
  uint32_t sub;
  uint32_t nseg;       // and its input segments [seg, seg + nseg) (unsplit pages: none, at the same count)
  uint32_t seg;
};

// Device state of the plan's split pages, zeroed before each scan: per
// fragment three words, per segment two flagged 64-bit words.
struct SnapState {
  uint32_t* owner;     // fragment: its job's index in the job list, written by the scan
  uint32_t* start;     // fragment: input offset of its first element
  uint32_t* bad;       // first fragment of a job: the page is not framed, decompress it whole;
                       // second: k_snappy_long has recorded its fragments
  unsigned long long* exit;  // segment: SN_SET | input offset of the first element past it
  unsigned long long* len;   // segment: SN_SET | output bytes of the elements that start in it
};
constexpr unsigned long long SN_SET = 1ull << 63;
constexpr uint64_t snap_state_bytes(uint64_t fragments, uint64_t segments) { return 12 * fragments + 16 * segments; }
inline SnapState snap_state(uint8_t* base, uint64_t fragments, uint64_t segments) {
  SnapState s{};
  s.exit = reinterpret_cast<unsigned long long*>(base);
  s.len = s.exit + segments;
  s.owner = reinterpret_cast<uint32_t*>(s.len + segments);
  s.start = s.owner + fragments;
  s.bad = s.start + fragments;
  return s;
}

}  // namespace pqi
