// The fibers behind cuda_on_cpu.h (compiled without sanitizers: they switch
// stacks).
#include "cuda_on_cpu.h"

#include <dlfcn.h>
#include <sys/mman.h>
#include <ucontext.h>

#undef threadIdx
#undef blockIdx
#undef blockDim
#undef gridDim

namespace emu {
namespace {

constexpr size_t kStack = 256 * 1024;
enum State { READY, IN_WARP, IN_BLOCK, LEFT };

struct Fiber {
  ucontext_t at;      // where it goes on
  State state = READY;
  int site = 0;
  int mode = 0;
};
struct Warp {
  uint64_t value[2][32];
  unsigned turn = 0;
  int arrived = 0;
};

std::vector<uint8_t*> stacks;
std::vector<Fiber> fibers;
std::vector<Warp> warps;
const std::function<void()>* body;
int current = -1, n_threads = 0;
ucontext_t scheduler;
dim3 block_size, grid_size, block_at;
int block_value = 0;
std::mt19937 order;
bool shuffled = false;
std::string first_fault;

void note(const std::string& what) {
  if (first_fault.empty()) first_fault = what;
}

void entry() {
  (*body)();
  fibers[current].state = LEFT;
  setcontext(&scheduler);
}

// (libc's own: a sanitizer's clears the whole stack's shadow at every switch)
using Swap = int (*)(ucontext_t*, const ucontext_t*);
Swap swap_context() {
  void* c = dlopen("libc.so.6", RTLD_LAZY);
  void* f = c ? dlsym(c, "swapcontext") : nullptr;
  return f ? reinterpret_cast<Swap>(f) : &swapcontext;
}
const Swap swap = swap_context();

void to_scheduler() { swap(&fibers[current].at, &scheduler); }

void resume(int i) {
  current = i;
  swap(&scheduler, &fibers[i].at);
}

// One warp as far as it goes; the number of its lanes that left or wait at a
// block barrier.
void run_warp(int w) {
  const int b = 32 * w, e = std::min(n_threads, b + 32);
  for (;;) {
    bool any = false;
    for (int i = b; i < e; ++i)
      if (fibers[i].state == READY) {
        any = true;
        resume(i);
      }
    if (!any) return;
  }
}

void run_block() {
  for (auto& f : fibers) f.state = READY;
  for (auto& w : warps) w = Warp{};
  for (int i = 0; i < n_threads; ++i) {
    getcontext(&fibers[i].at);
    fibers[i].at.uc_stack.ss_sp = stacks[i];
    fibers[i].at.uc_stack.ss_size = kStack;
    fibers[i].at.uc_link = nullptr;
    makecontext(&fibers[i].at, entry, 0);
  }
  std::vector<int> list;
  for (size_t w = 0; w < warps.size(); ++w) list.push_back(static_cast<int>(w));
  for (;;) {
    if (shuffled) std::shuffle(list.begin(), list.end(), order);
    for (int w : list) run_warp(w);
    int left = 0, in_block = 0, site = -1, mode = 0, sum = 0;
    for (const auto& f : fibers) {
      if (f.state == LEFT) ++left;
      if (f.state == IN_WARP) return note("lanes wait for their warp at line " + std::to_string(f.site));
      if (f.state == IN_BLOCK) {
        if (in_block++ && (f.site != site || f.mode != mode))
          return note("threads wait at different barriers, lines " + std::to_string(site) + " and " + std::to_string(f.site));
        site = f.site;
        mode = f.mode;
      }
    }
    if (left == n_threads) return;
    if (left) return note("threads left while others wait at line " + std::to_string(site));
    sum = block_value;
    block_value = mode == 1 ? sum != 0 : sum;
    for (auto& f : fibers) f.state = READY;
    // (each thread takes the value as it goes on; it is cleared by the first to arrive again)
  }
}

int arrivals = 0, taken = 0;

}  // namespace

uint8_t* smem = nullptr;

uint3 thread_index() { return uint3{static_cast<unsigned>(current), 0, 0}; }
uint3 block_index() { return uint3{block_at.x, block_at.y, block_at.z}; }
dim3 block_dim() { return block_size; }
dim3 grid_dim() { return grid_size; }

int block_sync(int value, int site, int mode) {
  static int sum = 0;
  if (arrivals == 0) sum = 0;
  sum += value;
  if (++arrivals == n_threads) {
    arrivals = 0;
    block_value = sum;
  }
  Fiber& f = fibers[current];
  f.state = IN_BLOCK;
  f.site = site;
  f.mode = mode;
  to_scheduler();
  return block_value;
}

const uint64_t* warp_exchange(uint64_t value, int site) {
  Warp& w = warps[current / 32];
  const int b = current / 32 * 32;
  const unsigned t = w.turn & 1;
  w.value[t][current - b] = value;
  Fiber& f = fibers[current];
  f.site = site;
  if (++w.arrived == 32) {
    w.arrived = 0;
    ++w.turn;
    for (int i = b; i < b + 32; ++i) {
      if (fibers[i].site != site)
        note("lanes at different warp operations, lines " + std::to_string(site) + " and " +
             std::to_string(fibers[i].site));
      fibers[i].state = READY;
    }
  } else {
    f.state = IN_WARP;
    to_scheduler();
  }
  return w.value[t];
}

void launch(const std::function<void()>& fn, dim3 grid, dim3 block, size_t shared) {
  n_threads = static_cast<int>(block.x);
  while (stacks.size() < static_cast<size_t>(n_threads))
    stacks.push_back(static_cast<uint8_t*>(
        mmap(nullptr, kStack, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0)));
  fibers.resize(n_threads);
  warps.resize((n_threads + 31) / 32);
  body = &fn;
  grid_size = grid;
  block_size = block;
  for (unsigned y = 0; y < grid.y; ++y)
    for (unsigned x = 0; x < grid.x && first_fault.empty(); ++x) {
      block_at = dim3(x, y, 1);
      arrivals = 0;
      void* p = nullptr;
      if (posix_memalign(&p, 1024, (shared + 15) & ~size_t(15))) abort();
      for (size_t i = 0; i < shared; ++i) static_cast<uint8_t*>(p)[i] = static_cast<uint8_t>(order());
      smem = static_cast<uint8_t*>(p);
      run_block();
      free(p);
      smem = nullptr;
    }
}

void reset(unsigned seed) {
  order.seed(seed);
  shuffled = seed != 0;
  first_fault.clear();
}
const char* fault() { return first_fault.empty() ? nullptr : first_fault.c_str(); }

}  // namespace emu

extern "C" cudaError_t cudaPeekAtLastError() { return cudaSuccess; }
