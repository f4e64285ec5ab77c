// How much dynamic shared memory each kernel has been allowed, per device.
#pragma once

#include <cstddef>
#include <map>
#include <mutex>
#include <utility>

namespace bmg {

// The limit is an attribute of a kernel on a device, shared by all host
// threads.  It is therefore asked for once per device, not per process, and
// only ever raised: a thread that set a smaller size of its own between
// another's request and launch would have that launch refused.
class SharedOptIn {
 public:
  // Whether `kern` may use `bytes` on device `dev`; allow(bytes) asks for them
  // where no call before this one has been granted as many.
  template <class Allow>
  bool ensure(const void* kern, int dev, size_t bytes, Allow allow) {
    std::lock_guard<std::mutex> g(mu_);
    const auto it = granted_.find({kern, dev});
    if (it != granted_.end() && it->second >= bytes) return true;
    if (!allow(bytes)) return false;
    granted_[{kern, dev}] = bytes;
    return true;
  }

 private:
  std::mutex mu_;
  std::map<std::pair<const void*, int>, size_t> granted_;
};

}  // namespace bmg
