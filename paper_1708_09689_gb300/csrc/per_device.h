// Process-wide state that belongs to a device: a kernel's attributes, streams and events hold on
// the device they were made on, so what is kept of them is kept per device.  Host only.
#pragma once

#include <map>
#include <mutex>
#include <set>
#include <utility>

namespace pvsc {

// Work to be done once per (device, key): run(device, key, f) calls f() unless it has succeeded
// (returned 0) for that pair before, and returns its result.
template <class Key>
class OncePerDevice {
 public:
  template <class F>
  int run(int device, const Key& key, F&& f) {
    std::lock_guard<std::mutex> lk(mu_);
    if (done_.count({device, key})) return 0;
    const int rc = f();
    if (rc == 0) done_.insert({device, key});
    return rc;
  }

 private:
  std::mutex mu_;
  std::set<std::pair<int, Key>> done_;
};

// A T per device: get(device, &t, create) makes it with create(T&) on the first call for that device
// (kept only if that returns 0) and hands out the one of the device.  A T stays where it is.
template <class T>
class PerDevice {
 public:
  template <class F>
  int get(int device, T** out, F&& create) {
    std::lock_guard<std::mutex> lk(mu_);
    auto it = at_.find(device);
    if (it == at_.end()) {
      T t{};
      if (const int rc = create(t)) return rc;
      it = at_.emplace(device, std::move(t)).first;
    }
    *out = &it->second;
    return 0;
  }

 private:
  std::mutex mu_;
  std::map<int, T> at_;
};

}  // namespace pvsc
