// Host state that belongs to a device and follows its user to another one. Api: the CUDA runtime
// calls made here (CudaApi in launch.h; a test puts a fake one in its place).
#pragma once

#include <atomic>
#include <cstdint>

namespace gipm {

// A stream with the events that fork it from the caller's stream and join it back. It belongs to the
// device that was current at create(); create() on another device makes it anew there.
template <typename Api> class SideStreamOf {
 public:
  typename Api::Stream s{};
  typename Api::Event fork{}, join{};
  SideStreamOf() = default;
  SideStreamOf(const SideStreamOf &) = delete;
  SideStreamOf &operator=(const SideStreamOf &) = delete;
  ~SideStreamOf() { destroy(); }
  // high: the highest stream priority instead of the default one. False if a call fails.
  bool create(bool high) {
    int dev = 0;
    if (!Api::current_device(dev)) return false;
    if (s && dev == device_) return true;
    destroy();
    device_ = dev;
    if (Api::create(high, s) && Api::create(fork) && Api::create(join)) return true;
    destroy();
    return false;
  }

 private:
  void destroy() {
    if (fork) Api::destroy(fork);
    if (join) Api::destroy(join);
    if (s) Api::destroy(s);
    fork = join = typename Api::Event{};
    s = typename Api::Stream{};
  }
  int device_ = -1;
};

// What is done once per device of the process (a function attribute): true for each device's first
// caller, and for later ones until done() says that it succeeded.
class DeviceOnce {
 public:
  bool needed(int dev) const { return !(mask_.load(std::memory_order_acquire) >> (dev & 63) & 1u); }
  void done(int dev) { mask_.fetch_or(uint64_t(1) << (dev & 63), std::memory_order_release); }

 private:
  std::atomic<uint64_t> mask_{0};
};

}  // namespace gipm
