// Test harness: the transcode of delta-coded string pages (csrc/k_transcode.cu)
// on the CPU.  Page bytes, pool and entry tables are heap blocks of their sizes
// and the slack that the engine gives them.
#include "cuda_on_cpu.h"

#include "k_transcode.cu"

// Pages i: src[at[i], at[i + 1]), encoding enc[i], rows[i] rows (REQUIRED, no
// level bytes), string bytes chars[i] of the chunk.  Per page, values[i] (-1: failed)
// and, for sound pages, lengths and bytes of the values one after another in
// `len` and `out`.  Returns 0, or -1 for a fault of the block.
extern "C" int transcode_pages(const uint8_t* src, const uint32_t* at, const int32_t* enc, const int32_t* rows,
                               const int64_t* chars, int n, unsigned seed, int32_t* values, uint32_t* len, uint8_t* out,
                               int32_t* err, char* text) {
  using namespace pqi;
  emu::reset(seed);
  std::vector<TranscodeJob> jobs(n);
  std::vector<PlanPage> pps(n);
  std::vector<uint8_t*> in(n);
  uint64_t table = 0, pool_cap = 0;
  for (int i = 0; i < n; ++i) {
    const uint32_t sl = at[i + 1] - at[i], lead = (5 * i) & 15;
    in[i] = static_cast<uint8_t*>(malloc(16 + lead + sl + 16));
    memcpy(in[i] + 16 + lead, src + at[i], sl);
    TranscodeJob& j = jobs[i];
    j = TranscodeJob{};
    j.src = in[i] + 16 + lead;
    j.src_len = sl;
    j.pp = static_cast<uint32_t>(i);
    j.page = i;
    j.enc = enc[i];
    j.num_values = rows[i];
    j.required = 1;
    pps[i] = PlanPage{};
    pps[i].dblocks = -1;
    pps[i].body = j.src;
    pps[i].body_len = static_cast<int32_t>(sl);
    pps[i].vtab = static_cast<uint32_t>(1 + table);
    table += static_cast<uint64_t>(rows[i]);
    pool_cap += ((sl + 63) & ~15u) + ((static_cast<uint64_t>(chars[i]) + 15) & ~uint64_t(15));
  }
  uint64_t* tab = static_cast<uint64_t*>(malloc(8 * table + 1));
  uint8_t* pool = static_cast<uint8_t*>(malloc(pool_cap + 64));
  uint32_t counters[8] = {};
  DevStatus st{0, -1, 0, 0};
  launch_transcode(jobs.data(), n, 0, 0, pps.data(), pool, pool_cap, counters, tab, &st, nullptr);
  uint64_t w = 0, o = 0;
  for (int i = 0; i < n && !emu::fault(); ++i) {
    const PlanPage& pp = pps[i];
    values[i] = pp.vtab && pp.dblocks >= 0 ? pp.dblocks : -1;
    const uint64_t* t = tab + (jobs[i].num_values && pp.vtab ? pp.vtab - 1 : 0);
    for (int32_t k = 0; k < values[i]; ++k) {
      const uint32_t l = static_cast<uint32_t>(t[k]);
      if ((t[k] >> 32) + l > static_cast<uint64_t>(pp.body_len)) {
        strcpy(text, "entry outside the page");
        return -1;
      }
      len[w++] = l;
      memcpy(out + o, pp.body + (t[k] >> 32), l);
      o += l;
    }
  }
  free(tab);
  free(pool);
  for (uint8_t* p : in) free(p);
  err[0] = static_cast<int32_t>(st.flags);
  err[1] = st.first_page;
  err[2] = st.detail;
  if (emu::fault()) {
    strncpy(text, emu::fault(), 255);
    return -1;
  }
  return 0;
}
