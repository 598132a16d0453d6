// Settings that the CUDA runtime keeps per device (such as a kernel's limit of
// dynamic shared memory) and that a call site makes once on each.
#pragma once
#include <atomic>
#include <cstdint>

namespace spin {

class OncePerDevice {
 public:
  // whether mark(dev) has been called (devices from 64 on: never)
  bool done(int dev) const { return dev >= 0 && dev < 64 && (seen_.load() >> dev & 1u) != 0; }
  void mark(int dev) {
    if (dev >= 0 && dev < 64) seen_.fetch_or((uint64_t)1 << dev);
  }

 private:
  std::atomic<uint64_t> seen_{0};
};

}  // namespace spin
