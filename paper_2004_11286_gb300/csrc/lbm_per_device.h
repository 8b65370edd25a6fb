// lbm_per_device.h -- what a launcher finds out or sets up once for each device
// (kernel attributes, resident blocks, SM counts).  A kernel's attributes
// belong to one device's context, and a process may hold handles on several.
#pragma once

#include <atomic>

namespace lbm {

constexpr int MAX_DEVICES = 64;

// Static storage only (zero: not known yet).  Threads may find out the same
// value at the same time; find() must be safe to repeat.
struct PerDevice {
  std::atomic<int> value[MAX_DEVICES];
  // The value of device `dev`: find() the first time, > 0 on success (a
  // failure is not remembered), on every call for devices past the table.
  template <class F>
  int get(int dev, F&& find) {
    if (dev < 0 || dev >= MAX_DEVICES) return find();
    int v = value[dev].load(std::memory_order_acquire);
    if (v <= 0) {
      v = find();
      if (v > 0) value[dev].store(v, std::memory_order_release);
    }
    return v;
  }
};

}  // namespace lbm
