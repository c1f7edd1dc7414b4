// Which parts of a call may run side by side (host code without CUDA, tested by itself).
#pragma once
#include <cstddef>
#include <cstdint>

namespace lp {

struct Span {   // memory of the caller's; p == nullptr: not given
  const void* p;
  size_t n;
};
inline bool overlap(const Span& a, const Span& b) {
  const uintptr_t x = reinterpret_cast<uintptr_t>(a.p), y = reinterpret_cast<uintptr_t>(b.p);
  return a.p && b.p && x < y + b.n && y < x + a.n;
}

// Updates of the modules' multipliers: one after another where a buffer serves two of them.
inline bool multipliers_apart(const Span* lambda, int n) {
  for (int k = 0; k < n; ++k)
    for (int j = 0; j < k; ++j)
      if (overlap(lambda[k], lambda[j])) return false;
  return true;
}

// Distillation of n AuxNets (or stacks): AuxNet i reads the images or x[i - 1], and x[i] and dx[i], and writes x_new[i].  One
// does not depend on another, unless a corrected variable is written over what another one reads or writes (x_new = x: then
// one after another, and AuxNet i sees the corrected x[i - 1]).
inline bool corrections_apart(const Span& images, const Span* x, const Span* dx, const Span* x_new, int n) {
  for (int i = 0; i < n; ++i) {
    if (overlap(x_new[i], images)) return false;
    for (int j = 0; j < n; ++j)
      if (overlap(x_new[i], x[j]) || (j != i && (overlap(x_new[i], dx[j]) || overlap(x_new[i], x_new[j])))) return false;
  }
  return true;
}

}  // namespace lp
