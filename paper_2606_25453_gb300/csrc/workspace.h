// workspace.h -- when a handle's own workspace grows, and what becomes of the
// block it outgrows.  Host logic alone: the allocator is a parameter.
#pragma once
#include <cstddef>
#include <cstdint>
#include <new>

namespace emu {

struct OldBlock {
  void* p;
  OldBlock* next;
};

struct Workspace {
  void* p = nullptr;
  size_t bytes = 0;
  bool in_graph = false;    // a stream capture recorded work on p
  OldBlock* old = nullptr;  // outgrown blocks that graphs may still replay on, kept until the end
  size_t failed = 0;        // size of the last optional growth that failed
  int skip = 0;             // optional growths of that size to refuse without another attempt
};

// Optional growths refused after a failed one.  A failed allocation costs far
// more than the call it serves; memory that another owner gives back is found
// again within this many calls.
constexpr int kWsSkip = 64;

// At least `bytes` at *out; false if they cannot be had.  mem.capturing():
// the call's stream is being captured; mem.alloc(n): n bytes or null;
// mem.release(p): p may be reused once the work enqueued so far is done.
//  - Nothing grows inside a capture: the memory would belong to the graph.
//  - A block that a capture used stays until ws_close: the graph replays on it.
//  - optional: the caller can do with less.  Then the block it has is given up
//    only for a larger one in hand, or if both do not fit beside each other,
//    and a size that failed is not tried again for kWsSkip calls.
template <class Mem>
bool ws_reserve(Workspace& w, size_t bytes, bool optional, Mem& mem, uint8_t** out) {
  if (bytes == 0) bytes = 256;
  const bool grow = bytes > w.bytes;
  if (grow || !w.in_graph) {
    const bool capturing = mem.capturing();
    if (grow && capturing) return false;
    if (capturing) w.in_graph = true;
  }
  if (grow) {
    if (optional && w.skip > 0 && bytes >= w.failed) {
      --w.skip;
      return false;
    }
    const size_t want = bytes + bytes / 8;
    OldBlock* keep = nullptr;
    if (w.p && w.in_graph) {
      keep = new (std::nothrow) OldBlock{w.p, w.old};
      if (!keep) return false;
    }
    auto give_back = [&] {
      if (w.p && !keep) mem.release(w.p);
      w.p = nullptr;
      w.bytes = 0;
    };
    void* p = nullptr;
    if (optional || keep) p = mem.alloc(want);
    if (!p && !keep) {
      const bool again = !optional || w.p;  // else tried already, with nothing to give back
      give_back();
      if (again) p = mem.alloc(want);
    }
    if (!p) {
      delete keep;
      if (optional) {
        w.failed = bytes;
        w.skip = kWsSkip;
      }
      return false;
    }
    if (keep) w.old = keep;
    give_back();
    w.p = p;
    w.bytes = want;
    w.in_graph = false;
  }
  *out = static_cast<uint8_t*>(w.p);
  return true;
}

// The block goes back, or stays for the graphs that use it; false (and nothing
// done) without host memory to note it.
template <class Mem>
bool ws_drop(Workspace& w, Mem& mem) {
  if (w.p && w.in_graph) {
    OldBlock* const keep = new (std::nothrow) OldBlock{w.p, w.old};
    if (!keep) return false;
    w.old = keep;
  } else if (w.p) {
    mem.release(w.p);
  }
  w.p = nullptr;
  w.bytes = 0;
  w.in_graph = false;
  w.skip = 0;
  return true;
}

// Every block back; nothing may still run on them.
template <class Mem>
void ws_close(Workspace& w, Mem& mem) {
  if (w.p) mem.release(w.p);
  while (w.old) {
    OldBlock* const b = w.old;
    w.old = b->next;
    mem.release(b->p);
    delete b;
  }
  w = Workspace();
}

}  // namespace emu
