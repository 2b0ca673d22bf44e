// A number that is found once per device: attributes of a kernel (the dynamic
// shared memory and the cluster sizes it may use) and what follows from them hold
// for the device that is current when they are set, not for the process.
#pragma once

#include <atomic>

#include <cuda_runtime.h>

namespace mg {

constexpr int kMaxDevices = 64;  // devices beyond are asked every time

struct PerDevice {
  std::atomic<long long> v[kMaxDevices];  // 0: not found yet (static storage)
};

// The current device's number, from find() the first time; numbers below 1 are
// not kept. Threads that find it at the same time find the same.
template <typename F> long long per_device(PerDevice &p, F find) {
  int d = -1;
  if (cudaGetDevice(&d) != cudaSuccess || d < 0 || d >= kMaxDevices) return find();
  long long x = p.v[d].load(std::memory_order_acquire);
  if (x == 0 && (x = find()) > 0) p.v[d].store(x, std::memory_order_release);
  return x;
}

}  // namespace mg
