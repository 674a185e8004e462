// kernel_limits.cuh -- resident blocks per SM of kernels with dynamic shared
// memory, and the limit on that memory raised where a launch needs more than
// the default 48 KB.
//
// Both belong to a kernel on a device: a process may hold graphs on several, and
// cudaFuncSetAttribute acts on the current one.  So everything here is kept by
// (device, kernel).  Api stands for the three CUDA calls (a host test gives its
// own).
#pragma once
#include <cstddef>
#include <map>
#include <mutex>
#include <tuple>
#include <utility>

namespace dfpr {

template <class Api>
class KernelLimits {
 public:
  using Error = typename Api::Error;

  // *bps: resident blocks per SM of fn on the current device, its limit raised
  // to smem bytes first if it is lower
  Error get(const void* fn, int threads, size_t smem, int* bps) {
    int dev = 0;
    Error e = Api::device(&dev);
    if (e != Api::ok) return e;
    std::lock_guard<std::mutex> lock(mu_);
    const auto key = std::make_tuple(dev, fn, threads, smem);
    const auto it = blocks_.find(key);
    if (it != blocks_.end()) {
      *bps = it->second;
      return Api::ok;
    }
    size_t& lim = limit_[std::make_pair(dev, fn)];
    if (smem > lim) {
      if ((e = Api::raise(fn, smem)) != Api::ok) return e;
      lim = smem;
    }
    int b = 0;
    if ((e = Api::blocks(&b, fn, threads, smem)) != Api::ok) return e;
    if (b < 1) return Api::does_not_fit;
    blocks_[key] = b;
    *bps = b;
    return Api::ok;
  }

 private:
  std::mutex mu_;
  std::map<std::pair<int, const void*>, size_t> limit_;
  std::map<std::tuple<int, const void*, int, size_t>, int> blocks_;
};

}  // namespace dfpr
