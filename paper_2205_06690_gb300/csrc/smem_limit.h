// The highest dynamic shared-memory limit set so far, per device and kernel. The limit is an attribute of
// the kernel on one device, shared by every context and host thread: lowering it for one launch could
// make another thread's larger launch of the same kernel fail in between. So it is only ever raised, under
// a lock. (No CUDA in this header: the caller passes the device and the setter.)
#pragma once

#include <stddef.h>

#include <map>
#include <mutex>
#include <utility>

namespace sbse {

class SmemLimits {
 public:
  // set(bytes): raises the attribute on `device`, true on success
  template <class Set> void raise(int device, const void *fn, size_t bytes, Set set) {
    std::lock_guard<std::mutex> lk(mx_);
    size_t &c = cur_[{device, fn}];
    if (bytes > c && set(bytes)) c = bytes;
  }

 private:
  std::mutex mx_;
  std::map<std::pair<int, const void *>, size_t> cur_;
};

}  // namespace sbse
