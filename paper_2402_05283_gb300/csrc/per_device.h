// per_device.h - facts that are found once on each device: a kernel's opt-in
// attributes, how many of its clusters fit.  Plain C++, so that it is tested
// without a GPU.
#pragma once
#include <map>
#include <mutex>

namespace cpra {

template <class T> class PerDevice {
 public:
  // v <- the value of device dev.  make(T&) finds it the first time, and again
  // after it has failed (returned anything but the zero of its error type,
  // which is handed on); threads that ask meanwhile wait for it.
  template <class F> auto get(int dev, T& v, F&& make) -> decltype(make(v)) {
    using E = decltype(make(v));
    std::lock_guard<std::mutex> lock(mu_);
    const auto it = found_.find(dev);
    if (it != found_.end()) {
      v = it->second;
      return E{};
    }
    T t{};
    const E e = make(t);
    if (e == E{}) v = found_.emplace(dev, t).first->second;
    return e;
  }

 private:
  std::mutex mu_;
  std::map<int, T> found_;
};

}  // namespace cpra
