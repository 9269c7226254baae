// What a kernel's source needs to compile as host C++ and run a thread block at
// a time: every CUDA thread is a fiber, a barrier or a warp operation waits for
// the threads it names.  Checked on the way: all threads of a block meet at the
// same barrier, all lanes of a warp at the same operation, none leaves while
// others wait.  Warps run in a seeded order between barriers, each as far as it
// can, so that what one warp writes after a barrier is seen by another that has
// yet to read there.
//
// The sources are given to the compiler with `extern __shared__` arrays,
// launches and inline PTX replaced (cuda_on_cpu.py).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

// (all that the harnesses take from the standard library: CUDA's keywords are macros below)
#include <algorithm>
#include <functional>
#include <memory>
#include <random>
#include <string>
#include <vector>

namespace emu {
extern uint8_t* smem;                         // dynamic shared memory, of exactly the launch's size
uint3 thread_index();
uint3 block_index();
dim3 block_dim();
dim3 grid_dim();
int block_sync(int value, int site, int mode);  // mode: 0 barrier, 1 or, 2 and, 3 count
// The warp's values at this operation, by lane (valid until the lane's next one).
const uint64_t* warp_exchange(uint64_t value, int site);
void launch(const std::function<void()>& body, dim3 grid, dim3 block, size_t shared);
// Seed of the warp order (0: warp 0 always first); the first fault of the
// launches since (or null).
void reset(unsigned seed);
const char* fault();

template <typename T>
uint64_t bits(T v) {
  static_assert(sizeof(T) <= 8, "warp operand");
  uint64_t b = 0;
  memcpy(&b, &v, sizeof v);
  return b;
}
template <typename T>
T from(uint64_t b) {
  T v;
  memcpy(&v, &b, sizeof v);
  return v;
}
inline int lane() { return static_cast<int>(thread_index().x & 31); }
template <typename T>
T shfl(T v, int src, int site) {
  const uint64_t* w = warp_exchange(bits(v), site);
  return src >= 0 && src < 32 ? from<T>(w[src]) : v;
}
inline unsigned ballot(bool p, int site) {
  const uint64_t* w = warp_exchange(p, site);
  unsigned m = 0;
  for (int i = 0; i < 32; ++i) m |= static_cast<unsigned>(w[i] != 0) << i;
  return m;
}
template <typename T>
unsigned match(T v, int site) {
  const uint64_t* w = warp_exchange(bits(v), site);
  unsigned m = 0;
  for (int i = 0; i < 32; ++i) m |= static_cast<unsigned>(w[i] == bits(v)) << i;
  return m;
}
}  // namespace emu

#undef __launch_bounds__
#undef __shared__
#undef __forceinline__
#define __launch_bounds__(...)
#define __shared__ static
#undef __noinline__
#define __forceinline__ inline
#define __noinline__ __attribute__((noinline))
#define threadIdx (emu::thread_index())
#define blockIdx (emu::block_index())
#define blockDim (emu::block_dim())
#define gridDim (emu::grid_dim())

#define __syncthreads() ((void)emu::block_sync(0, __LINE__, 0))
#define __syncthreads_or(p) (emu::block_sync((p) ? 1 : 0, __LINE__, 1))
#define __syncthreads_count(p) (emu::block_sync((p) ? 1 : 0, __LINE__, 3))
#define __syncwarp() ((void)emu::warp_exchange(0, __LINE__))
#define __shfl_sync(m, v, src) (emu::shfl((v), (src) & 31, __LINE__))
#define __shfl_up_sync(m, v, d) (emu::shfl((v), emu::lane() - static_cast<int>(d), __LINE__))
#define __shfl_down_sync(m, v, d) (emu::shfl((v), emu::lane() + static_cast<int>(d), __LINE__))
#define __shfl_xor_sync(m, v, d) (emu::shfl((v), emu::lane() ^ static_cast<int>(d), __LINE__))
#define __ballot_sync(m, p) (emu::ballot((p), __LINE__))
#define __any_sync(m, p) (emu::ballot((p), __LINE__) != 0)
#define __all_sync(m, p) (emu::ballot((p), __LINE__) == 0xffffffffu)
#define __match_any_sync(m, v) (emu::match((v), __LINE__))

template <typename T>
inline T __ldg(const T* p) { return *p; }
inline int __popc(unsigned x) { return __builtin_popcount(x); }
inline int __clz(unsigned x) { return x ? __builtin_clz(x) : 32; }
inline int __ffs(int x) { return __builtin_ffs(x); }
inline int __ffsll(long long x) { return __builtin_ffsll(x); }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  return static_cast<unsigned>((((static_cast<uint64_t>(hi) << 32) | lo) << (s & 31)) >> 32);
}
inline unsigned __funnelshift_r(unsigned lo, unsigned hi, unsigned s) {
  return static_cast<unsigned>(((static_cast<uint64_t>(hi) << 32) | lo) >> (s & 31));
}
inline unsigned __funnelshift_rc(unsigned lo, unsigned hi, unsigned s) {
  return static_cast<unsigned>(((static_cast<uint64_t>(hi) << 32) | lo) >> (s < 32 ? s : 32));
}
inline unsigned __byte_perm(unsigned a, unsigned b, unsigned s) {
  const uint64_t v = (static_cast<uint64_t>(b) << 32) | a;
  unsigned r = 0;
  for (int i = 0; i < 4; ++i) r |= static_cast<unsigned>((v >> (8 * ((s >> (4 * i)) & 7))) & 0xff) << (8 * i);
  return r;
}
template <typename F>
inline unsigned emu_bytes(unsigned a, unsigned b, F f) {
  unsigned r = 0;
  for (int i = 0; i < 32; i += 8) r |= (f((a >> i) & 0xff, (b >> i) & 0xff) ? 0xffu : 0u) << i;
  return r;
}
inline unsigned __vcmpeq4(unsigned a, unsigned b) { return emu_bytes(a, b, [](unsigned x, unsigned y) { return x == y; }); }
inline unsigned __vcmpgtu4(unsigned a, unsigned b) { return emu_bytes(a, b, [](unsigned x, unsigned y) { return x > y; }); }
inline unsigned __dp4a(unsigned a, unsigned b, unsigned c) {
  for (int i = 0; i < 32; i += 8) c += ((a >> i) & 0xff) * ((b >> i) & 0xff);
  return c;
}
inline size_t __cvta_generic_to_shared(const void* p) { return static_cast<const uint8_t*>(p) - emu::smem; }

template <typename T, typename U>
inline T atomicAdd(T* p, U v) { const T o = *p; *p = static_cast<T>(o + v); return o; }
template <typename T, typename U>
inline T atomicOr(T* p, U v) { const T o = *p; *p = static_cast<T>(o | v); return o; }
template <typename T, typename U>
inline T atomicMax(T* p, U v) { const T o = *p; *p = std::max(o, static_cast<T>(v)); return o; }
template <typename T, typename U>
inline T atomicMin(T* p, U v) { const T o = *p; *p = std::min(o, static_cast<T>(v)); return o; }
template <typename T, typename U, typename V>
inline T atomicCAS(T* p, U c, V v) { const T o = *p; if (o == static_cast<T>(c)) *p = static_cast<T>(v); return o; }
template <typename... A>
inline cudaError_t cudaFuncSetAttribute(void (*)(A...), cudaFuncAttribute, int) { return cudaSuccess; }
template <typename... A>
inline cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, void (*)(A...), int, size_t) {
  return *n = 1, cudaSuccess;
}
using std::max;
using std::min;
