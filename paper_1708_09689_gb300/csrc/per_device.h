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

}  // namespace pvsc
