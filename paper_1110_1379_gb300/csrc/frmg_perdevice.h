// frmg_perdevice.h -- values that belong to one CUDA device, found once per
// device of the process: a kernel's attributes (cudaFuncSetAttribute acts on
// the current device only) and what the occupancy calculator says of it.
// Contexts on several devices and threads share them.
#pragma once

#include <map>
#include <mutex>
#include <utility>

namespace frmg {

template <typename T>
class PerDevice {
  std::mutex m;
  std::map<int, T> value;

 public:
  // The device's value; the first call for a device makes it (an exception
  // from make leaves it unmade).
  template <typename F>
  T get(int device, F &&make) {
    std::lock_guard<std::mutex> lock(m);
    auto it = value.find(device);
    if (it == value.end()) it = value.emplace(device, std::forward<F>(make)()).first;
    return it->second;
  }
};

}  // namespace frmg
