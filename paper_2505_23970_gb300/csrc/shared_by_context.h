// What the users of a CUDA context share, with the count of them (host code).
#pragma once
#include <mutex>

namespace gc {

using ContextId = unsigned long long;  // 0: none

// Handles (pointers), one per device and context, made for the first user and
// destroyed with the last.  A device reset makes a new context in which a new
// handle may have the value of an old one, so a user gives its handle back together
// with the context it got it in.  The handle of a context that is gone went with it
// and is only forgotten.
template <typename Handle>
class SharedByContext {
 public:
  // make() may return nullptr; so does acquire then, and there is nothing to release.
  template <typename Make>
  Handle acquire(int device, ContextId context, Make make) {
    if (context == 0) return nullptr;
    std::lock_guard<std::mutex> lock(mutex_);
    Entry* empty = nullptr;
    for (Entry& e : entries_) {
      if (e.users == 0) {
        if (!empty) empty = &e;
      } else if (e.device == device && e.context == context) {
        ++e.users;
        return e.handle;
      }
    }
    const Handle handle = empty ? make() : nullptr;
    if (handle) *empty = Entry{handle, device, context, 1};
    return handle;
  }

  // alive(): does the context still exist?  destroy(handle) is called if so.
  template <typename Alive, typename Destroy>
  void release(int device, ContextId context, Handle handle, Alive alive, Destroy destroy) {
    if (!handle) return;
    std::lock_guard<std::mutex> lock(mutex_);
    for (Entry& e : entries_) {
      if (e.users == 0 || e.device != device || e.context != context || e.handle != handle)
        continue;
      if (--e.users == 0 && alive()) destroy(e.handle);
      return;
    }
  }

 private:
  struct Entry {
    Handle handle;
    int device;
    ContextId context;
    int users;  // 0: the entry is free
  };
  std::mutex mutex_;
  Entry entries_[64] = {};
};

}  // namespace gc
