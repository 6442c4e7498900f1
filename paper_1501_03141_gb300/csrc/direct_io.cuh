// Whether a call can work on the caller's arrays in place of staged copies
// (host code without CUDA calls).
#pragma once

#include <cstddef>
#include <cstdint>
#include <initializer_list>

namespace pdep {

struct Span {
  const void* p;
  size_t bytes;
  bool on_gpu;   // device or managed memory
  bool managed;  // managed: any GPU may use it
  int device;    // the GPU that device memory belongs to
};

// All on the context's GPU, aligned for FP64 loads, and the written array apart
// from the read ones.  Arrays on another GPU or that overlap go through the
// copies, as host arrays do.
inline bool direct_io(int device, const Span& out, std::initializer_list<Span> in) {
  auto usable = [&](const Span& s) {
    return s.p && s.on_gpu && (s.managed || s.device == device) && !((uintptr_t)s.p & 7);
  };
  if (!usable(out)) return false;
  const char* o = (const char*)out.p;
  for (const Span& x : in) {
    const char* q = (const char*)x.p;
    if (!usable(x)) return false;
    if (q < o + out.bytes && o < q + x.bytes) return false;
  }
  return true;
}

}  // namespace pdep
