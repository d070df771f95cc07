// What device_source.py needs to compile device functions of csrc/ for the
// host: the CUDA names they use, a block's threads as host threads, and a block
// barrier that ends the program with status 3 when the threads' barriers do not
// pair up.
#pragma once

#include <algorithm>
#include <chrono>
#include <condition_variable>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <thread>
#include <vector>
#include <sys/mman.h>
#include <unistd.h>

#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __shared__ static
#define __launch_bounds__(...)

using std::max;
using std::min;

struct Dim {
  unsigned int x;
};
inline thread_local Dim threadIdx{0};
inline Dim blockIdx{0}, blockDim{1}, gridDim{1};
inline void (*after_barrier)() = nullptr;  // called by every thread that leaves a barrier

struct int4 {
  int x, y, z, w;
};
inline int4 make_int4(int x, int y, int z, int w) { return {x, y, z, w}; }

inline int block_barrier(int p) {
  static std::mutex mu;
  static std::condition_variable cv;
  static unsigned int arrived = 0, turn = 0;
  static int any = 0, result = 0;
  int r;
  {
    std::unique_lock<std::mutex> lk(mu);
    any |= p != 0;
    if (++arrived == blockDim.x) {
      result = any;
      any = 0;
      arrived = 0;
      ++turn;
      cv.notify_all();
    } else {
      const unsigned int mine = turn;
      if (!cv.wait_for(lk, std::chrono::seconds(10), [&] { return turn != mine; })) {
        puts("the threads' barriers do not pair up");
        fflush(stdout);
        _exit(3);
      }
    }
    r = result;
  }
  if (after_barrier) after_barrier();
  return r;
}
inline void __syncthreads() { block_barrier(0); }
inline int __syncthreads_or(int p) { return block_barrier(p); }
inline int __syncthreads_and(int p) { return !block_barrier(!p); }

template <typename T, typename U>
T atomicAdd(T* p, U x) {
  return __atomic_fetch_add(p, (T)x, __ATOMIC_SEQ_CST);
}

// Runs f as every thread of one block of `threads` threads.
template <typename F>
void run_block(unsigned int threads, F f) {
  blockDim.x = threads;
  std::vector<std::thread> t;
  for (unsigned int i = 0; i < threads; ++i)
    t.emplace_back([=] {
      threadIdx.x = i;
      f();
    });
  for (auto& x : t) x.join();
}

// `count` int32 zeros (pages of the one zero page) with 9 GB on both sides
// that end the program when they are read.
inline const int32_t* guarded_zeros(int64_t count) {
  const size_t side = size_t(9) << 30, bytes = ((size_t)count * 4 + 4095) & ~size_t(4095);
  char* p = (char*)mmap(nullptr, side * 2 + bytes, PROT_NONE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (p == MAP_FAILED || mprotect(p + side, bytes, PROT_READ) != 0) {
    puts("no address space");
    exit(4);
  }
  return (const int32_t*)(p + side);
}
