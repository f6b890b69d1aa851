// warp_host_stubs.h -- a warp of 32 lanes on the host: each lane of a function that a whole warp executes is a
// coroutine, and a warp operation (shuffle, ballot, ...) waits until all 32 lanes have come to one of the same
// kind. Lanes that come to different operations, or end while others wait in one, are an error (on a GPU:
// undefined, a hang for instance). The rest of the CUDA names are cuda_host_stubs.h's.
#pragma once
#include <ucontext.h>

#include <functional>
#include <memory>

#define __shfl_sync one_lane_shfl_sync
#define __shfl_up_sync one_lane_shfl_up_sync
#define __shfl_down_sync one_lane_shfl_down_sync
#define __shfl_xor_sync one_lane_shfl_xor_sync
#define __ballot_sync one_lane_ballot_sync
#define __any_sync one_lane_any_sync
#define __all_sync one_lane_all_sync
#define __reduce_or_sync one_lane_reduce_or_sync
#define __syncwarp one_lane_syncwarp
#include "cuda_host_stubs.h"
#undef __shfl_sync
#undef __shfl_up_sync
#undef __shfl_down_sync
#undef __shfl_xor_sync
#undef __ballot_sync
#undef __any_sync
#undef __all_sync
#undef __reduce_or_sync
#undef __syncwarp

inline unsigned long long atomicOr(unsigned long long* p, unsigned long long v) {
  const unsigned long long o = *p;
  *p |= v;
  return o;
}

class HostWarp {
 public:
  // body(lane) in 32 lanes; false: the lanes parted
  bool run(const std::function<void(int)>& body) {
    body_ = &body;
    for (int l = 0; l < 32; ++l) {
      if (!stack_[l]) stack_[l].reset(new char[kStack]);
      getcontext(&ctx_[l]);
      ctx_[l].uc_stack.ss_sp = stack_[l].get();
      ctx_[l].uc_stack.ss_size = kStack;
      ctx_[l].uc_link = &main_;
      done_[l] = false;
      turn_[l] = 0;
      makecontext(&ctx_[l], (void (*)())enter, 0);
    }
    for (;;) {
      int ended = 0;
      for (int l = 0; l < 32; ++l) {
        lane_ = l;
        host_threadIdx.x = (unsigned)l;
        if (!done_[l]) swapcontext(&main_, &ctx_[l]);
        ended += done_[l];
      }
      host_threadIdx.x = 0;
      if (ended == 32) return true;
      if (ended) return false;
      for (int l = 1; l < 32; ++l)
        if (kind_[l] != kind_[0]) return false;
    }
  }
  // every lane's v of this operation, 32 values
  template <class T>
  const uint64_t* meet(int kind, T v) {
    static_assert(sizeof(T) <= 8, "");
    uint64_t* buf = value_[turn_[lane_]++ & 1];  // (a lane may be an operation ahead of one that still reads)
    buf[lane_] = 0;
    std::memcpy(&buf[lane_], &v, sizeof(T));
    kind_[lane_] = kind;
    swapcontext(&ctx_[lane_], &main_);
    return buf;
  }
  int lane() const { return lane_; }

 private:
  static constexpr size_t kStack = 256 * 1024;
  static void enter();
  ucontext_t main_, ctx_[32];
  std::unique_ptr<char[]> stack_[32];
  const std::function<void(int)>* body_ = nullptr;
  bool done_[32];
  unsigned turn_[32];
  int kind_[32], lane_ = 0;
  uint64_t value_[2][32];
};
inline HostWarp host_warp;
inline void HostWarp::enter() {
  (*host_warp.body_)(host_warp.lane_);
  host_warp.done_[host_warp.lane_] = true;
}

template <class T>
inline T warp_value(const uint64_t* buf, int lane) {
  T v;
  std::memcpy(&v, &buf[lane], sizeof(T));
  return v;
}
template <class T>
inline T __shfl_sync(unsigned, T v, int src, int = 32) { return warp_value<T>(host_warp.meet(1, v), src & 31); }
template <class T>
inline T __shfl_up_sync(unsigned, T v, unsigned d, int = 32) {
  const uint64_t* b = host_warp.meet(2, v);
  const int l = host_warp.lane() - (int)d;
  return l >= 0 ? warp_value<T>(b, l) : v;
}
template <class T>
inline T __shfl_down_sync(unsigned, T v, unsigned d, int = 32) {
  const uint64_t* b = host_warp.meet(3, v);
  const int l = host_warp.lane() + (int)d;
  return l < 32 ? warp_value<T>(b, l) : v;
}
template <class T>
inline T __shfl_xor_sync(unsigned, T v, int m, int = 32) { return warp_value<T>(host_warp.meet(4, v), host_warp.lane() ^ m); }
inline unsigned __ballot_sync(unsigned, int p) {
  const uint64_t* b = host_warp.meet(5, p != 0);
  unsigned m = 0;
  for (int l = 0; l < 32; ++l) m |= (b[l] & 1u) << l;
  return m;
}
inline int __any_sync(unsigned m, int p) { return __ballot_sync(m, p) != 0u; }
inline int __all_sync(unsigned m, int p) { return __ballot_sync(m, p) == 0xffffffffu; }
inline unsigned __reduce_or_sync(unsigned, unsigned v) {
  const uint64_t* b = host_warp.meet(6, v);
  unsigned m = 0;
  for (int l = 0; l < 32; ++l) m |= (unsigned)b[l];
  return m;
}
inline void __syncwarp(unsigned = 0xffffffffu) { host_warp.meet(7, 0); }
