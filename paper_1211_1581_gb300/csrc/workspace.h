// workspace.h -- the library's workspace of one device: which buffer a call gets
// and when a larger one is taken.  The allocator is a parameter, so that the
// rules run on the host alone too.  An Allocator has
//   bool capturing()               the call's stream is being captured
//   bool synchronize()             wait for the device
//   bool allocate(void**, size_t)  false: not to be had
//   void release(void*)
//   bool available(size_t*)        free device memory
#pragma once
#include <cstddef>
#include <cstdint>

#include "mxm.h"
#include "mxm_internal.h"

namespace mxm {

struct Workspace {
  void* base = nullptr;
  size_t bytes = 0;
  bool owned = true;           // allocated by the library
  size_t refused = SIZE_MAX;   // the least optional size that could not be had
};

// A new buffer of at least `need` bytes: an eighth more where that is there.
template <typename Allocator>
bool workspace_allocate(Workspace& w, size_t need, Allocator& a) {
  void* p = nullptr;
  size_t got = align_up(need + need / 8, size_t(2) << 20);
  if (!a.allocate(&p, got)) {
    got = need;
    if (!a.allocate(&p, got)) return false;
  }
  w.base = p;
  w.bytes = got;
  return true;
}

// What a call cannot do without.
template <typename Allocator>
mxm_status workspace_need(Workspace& w, size_t need, Allocator& a) {
  if (need <= w.bytes) return MXM_OK;
  if (!w.owned) return MXM_ERR_WORKSPACE_TOO_SMALL;
  if (a.capturing()) return MXM_ERR_NO_WORKSPACE;
  if (w.base != nullptr) {
    if (!a.synchronize()) return MXM_ERR_CUDA;
    a.release(w.base);
    w.base = nullptr;
    w.bytes = 0;
  }
  return workspace_allocate(w, need, a) ? MXM_OK : MXM_ERR_CUDA;
}

// What a call can make use of, `least` being what it cannot do without.  false:
// not to be had, and a buffer that holds `least` is still there.  It is given up
// for a larger one only when that one is in hand, or when the two together would
// not fit but the larger alone would; and a size that was refused is not asked
// for again (every call of a product on a nearly full device would synchronise
// and allocate otherwise) until the caller sets the workspace.
template <typename Allocator>
bool workspace_want(Workspace& w, size_t want, size_t least, Allocator& a) {
  if (want <= w.bytes) return true;
  if (!w.owned || want >= w.refused || a.capturing()) return false;
  if (w.base == nullptr || w.bytes < least) {  // of no use to the call
    if (workspace_need(w, want, a) == MXM_OK) return true;
    w.refused = want;
    return false;
  }
  Workspace larger;
  if (workspace_allocate(larger, want, a)) {
    if (!a.synchronize()) {
      a.release(larger.base);
      return false;
    }
    a.release(w.base);
    w.base = larger.base;
    w.bytes = larger.bytes;
    return true;
  }
  size_t free = 0;
  if (a.available(&free) && free + w.bytes >= want && a.synchronize()) {
    const size_t had = w.bytes;
    a.release(w.base);
    w.base = nullptr;
    w.bytes = 0;
    if (workspace_allocate(w, want, a)) return true;
    if (a.allocate(&w.base, had)) w.bytes = had;
    else w.base = nullptr;
  }
  w.refused = want;
  return false;
}

}  // namespace mxm
