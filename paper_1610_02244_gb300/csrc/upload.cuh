// Where a host table waits for its copy to the device.  CUDA only says that an asynchronous
// copy from pageable memory "might" be staged before the call returns; where the GPU reads
// pageable memory in place (a Grace host), a table that dies or changes after the call could
// be read late.  Tables therefore go through a pinned buffer of two halves used in turn; a
// half is written again only after the event behind its last copy.  All copies of a half are
// on one stream, so that one event covers them.  Plain host code: tests/upload_host.cu runs it
// against copies that are made as late as its rules allow.
#pragma once
#include <cstddef>

namespace tnt {

struct UploadRing {
  size_t half = 0;             // bytes of a half
  size_t pos = 0;              // of the half in use
  int cur = 0;                 // that half
  bool busy[2] = {false, false};
  const void* stream = nullptr;

  // The stream was replaced: the next copies open the other half even if the new stream has the old
  // one's handle (the half's event was recorded on a stream that may be gone).
  void detach() { stream = this; }

  // Offset for `bytes` (at most half) on stream st; *wait = the half whose event must pass
  // before the bytes are written, or -1.  After the copy the caller records event `cur`.
  size_t place(size_t bytes, const void* st, int* wait) {
    *wait = -1;
    if (pos > 0 && (st != stream || pos + bytes > half)) {
      cur ^= 1;
      pos = 0;
      if (busy[cur]) *wait = cur;
    }
    stream = st;
    const size_t at = (size_t)cur * half + pos;
    pos += (bytes + 255) & ~(size_t)255;
    busy[cur] = true;
    return at;
  }
};

}  // namespace tnt
