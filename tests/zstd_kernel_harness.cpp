// Test harness: the Zstandard kernel (csrc/k_zstd.cu) on the CPU.  The pages'
// bytes and output buffers are heap blocks with the slack that the engine
// gives them and no more, so that a memory checker sees any access outside.
#include "cuda_on_cpu.h"

#include "k_zstd.cu"

// Decodes n pages (page i: src[at[i], at[i + 1]) to len[i] bytes, one after another
// in `out`) in `blocks` thread blocks, warps in the seed's order.  Returns 0,
// or -1 for a fault of the block (its text in `text`); flags and the first bad
// page come back in err.
extern "C" int zstd_kernel_decode(const uint8_t* src, const uint32_t* at, const uint32_t* len, int n, int blocks,
                                  unsigned seed, uint8_t* out, int32_t* err, char* text) {
  using namespace pqi;
  emu::reset(seed);
  std::vector<SnappyJob> jobs(n);
  std::vector<uint8_t*> in(n), to(n);
  for (int i = 0; i < n; ++i) {
    const uint32_t sl = at[i + 1] - at[i];
    const uint32_t lead = (16 + 7 * i) & 31;  // any alignment, 16 readable bytes around
    in[i] = static_cast<uint8_t*>(malloc(16 + lead + sl + 16));
    memcpy(in[i] + 16 + lead, src + at[i], sl);
    to[i] = static_cast<uint8_t*>(malloc(16 + len[i] + 16));
    SnappyJob& j = jobs[i];
    j = SnappyJob{};
    j.src = in[i] + 16 + lead;
    j.dst = to[i] + 16;
    j.src_len = sl;
    j.dst_len = len[i];
    j.page = i;
    j.codec = CODEC_ZSTD;
  }
  DevStatus st{0, -1, 0, 0};
  launch_zstd(jobs.data(), n, blocks, &st, nullptr);
  uint32_t o = 0;
  for (int i = 0; i < n; ++i) {
    memcpy(out + o, to[i] + 16, len[i]);
    o += len[i];
    free(in[i]);
    free(to[i]);
  }
  err[0] = static_cast<int32_t>(st.flags);
  err[1] = st.first_page;
  err[2] = st.detail;
  if (emu::fault()) {
    strncpy(text, emu::fault(), 255);
    return -1;
  }
  return 0;
}
