// Host bookkeeping without CUDA calls of its own (it compiles and is tested with a plain C++
// compiler): the growth of a workspace where memory may run out, and work done once per device.
#pragma once
#include <cstddef>
#include <mutex>

namespace tdmrg {

// Grows the block (p, bytes) to `want` bytes, contents lost.  get(&q, n) returns 0 or an error and
// put(q) gives a block back; is_oom(e) tells the errors after which the smaller block is kept.  The
// new block is taken before the old one is given back; where there is no room for both, the old one
// goes first, and comes back where the larger one does not fit even then.  Returns the error of the
// larger allocation (the block is then the old size, or empty if even that is gone).
template <class Err, class Get, class Put, class Oom>
Err grow_block(void*& p, std::size_t& bytes, std::size_t want, Get get, Put put, Oom is_oom) {
  void* q = nullptr;
  Err e = get(&q, want);
  if (e == Err(0)) {
    if (p) put(p);
    p = q;
    bytes = want;
    return e;
  }
  if (!p || !is_oom(e)) return e;
  const std::size_t old = bytes;
  put(p);
  p = nullptr;
  bytes = 0;
  q = nullptr;
  e = get(&q, want);
  if (e == Err(0)) {
    p = q;
    bytes = want;
    return e;
  }
  q = nullptr;
  if (is_oom(e) && get(&q, old) == Err(0)) {
    p = q;
    bytes = old;
  }
  return e;
}

// f() once for every device (its error is returned and tried again by the next call); safe with
// several threads
class OncePerDevice {
 public:
  template <class Err, class F>
  Err run(int dev, Err bad_device, F f) {
    if (dev < 0 || dev >= kDevices) return bad_device;
    std::lock_guard<std::mutex> lock(mu_);
    if (done_[dev]) return Err(0);
    const Err e = f();
    done_[dev] = e == Err(0);
    return e;
  }

 private:
  static constexpr int kDevices = 64;
  std::mutex mu_;
  bool done_[kDevices] = {};
};

}  // namespace tdmrg
