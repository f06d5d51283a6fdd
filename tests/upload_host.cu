// Host check of csrc/upload.cuh: copies queued per stream and carried out only when something
// waits for them (an event, or the end), the latest that CUDA allows, must still find the bytes
// they were given.  Random sizes (empty, one byte, up to a whole half), stream changes, and streams
// replaced by new ones of the same handle.
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <vector>

#include "upload.cuh"

static uint64_t s = 0x9e3779b97f4a7c15ull;
static uint64_t next_u64() {
  uint64_t z = (s += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

struct Copy {
  int stream;
  size_t at;
  std::vector<unsigned char> want;
};

int main() {
  int bad = 0;
  long waits = 0, streams = 0;
  for (int run = 0; run < 200; ++run) {
    tnt::UploadRing r;
    r.half = run % 2 ? 4096 : 16384;
    std::vector<unsigned char> buf(2 * r.half);
    std::vector<Copy> queue;         // pending, in the order of the calls
    size_t upto[2] = {0, 0};         // event of a half: copies of its stream before this index
    int ev_stream[2] = {0, 0};
    size_t done = 0;                 // queue entries already dropped from the front
    auto carry_out = [&](int st, size_t end) {  // stream st's copies before index `end`
      for (size_t i = 0; i < queue.size(); ++i)
        if (queue[i].stream == st && done + i < end && !queue[i].want.empty()) {
          bad += memcmp(buf.data() + queue[i].at, queue[i].want.data(), queue[i].want.size()) != 0;
          queue[i].want.clear();
        }
    };
    int stream = 1, handle = 1, streams_made = 3;  // handles 1..3 at first stand for streams 1..3
    int of_handle[4] = {0, 1, 2, 3};
    for (int k = 0; k < 400; ++k) {
      if (next_u64() % 16 == 0) {
        handle = 1 + (int)(next_u64() % 3);
        if (next_u64() % 4 == 0) {
          of_handle[handle] = ++streams_made;
          r.detach();
        }
        stream = of_handle[handle];
        ++streams;
      }
      const uint64_t kind = next_u64() % 8;
      const size_t bytes = kind == 0 ? 1 : kind == 1 ? r.half : kind == 2 ? r.half - 1 : 1 + next_u64() % (r.half / 4);
      int wait;
      const size_t at = r.place(bytes, (const void*)(intptr_t)handle, &wait);
      if (wait >= 0) {
        ++waits;
        carry_out(ev_stream[wait], upto[wait]);
      }
      bad += at + bytes > buf.size();
      std::vector<unsigned char> d(bytes);
      for (auto& b : d) b = (unsigned char)next_u64();
      memcpy(buf.data() + at, d.data(), bytes);
      queue.push_back(Copy{stream, at, d});
      upto[r.cur] = done + queue.size();
      ev_stream[r.cur] = stream;
    }
    for (int st = 1; st <= streams_made; ++st) carry_out(st, (size_t)-1);
  }
  std::printf("waits %ld stream changes %ld mismatches %d\n", waits, streams, bad);
  return bad || !waits ? 1 : 0;
}
