// The reduced-system buffers of a workspace: one block of device memory, laid out
// for a capacity of contact vertices and replaced when n_c passes it.  Host logic
// without CUDA calls (the caller allocates and frees), so it is unit-tested on the
// CPU.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace fsim {

// One allocation handed out in 512-byte steps; with base NULL it only counts what
// it would hand out.
struct Arena {
  char* base = nullptr;
  size_t used = 0;
  void* take(size_t bytes) {
    void* p = base ? base + used : nullptr;
    used += (bytes + 511) / 512 * 512;
    return p;
  }
};

struct ReducedViews {
  double* Bc;      // (3 cap)^2
  int* bocc;       // cap^2 occupancy, cap^2 lists, cap counts, 32 barrier words
  double* red;     // elems
  float* redf;     // elems
};
inline ReducedViews reduced_views(Arena& a, int cap, int64_t elems) {
  const size_t c = (size_t)cap;
  ReducedViews v;
  v.Bc = static_cast<double*>(a.take(sizeof(double) * 9 * c * c));
  v.bocc = static_cast<int*>(a.take(sizeof(int) * (2 * c * c + c + 32)));
  v.red = static_cast<double*>(a.take(sizeof(double) * (size_t)elems));
  v.redf = static_cast<float*>(a.take(sizeof(float) * (size_t)elems));
  return v;
}
inline size_t reduced_view_bytes(int cap, int64_t elems) {
  Arena a;
  reduced_views(a, cap, elems);
  return a.used;
}

template <typename W>
void set_reduced(W& m, const ReducedViews& v, int cap, int64_t elems) {
  m.Bc = v.Bc;
  m.bocc = v.bocc;
  m.red = v.red;
  m.redf = v.redf;
  m.nc_cap = cap;
  m.red_cap = elems;
}

template <typename W>
bool reduced_fits(const W& m, int nc) {
  return m.Bc != nullptr && nc <= m.nc_cap;
}

// The capacity to grow to: by 1.5 times, at least 16, at most n2.
inline int grown_reduced_cap(int nc, int cap, int n2) {
  return std::min(std::max(nc, std::max(16, cap * 3 / 2)), std::max(n2, 1));
}

// Replaces m's buffers by ones of capacity cap, or leaves m without any (capacity 0)
// when alloc returns NULL.  The old ones are dropped first, so that both need not
// fit, and the generation goes up before they are: a captured launch sequence
// that names them is never replayed, whatever follows.  They are all in one block,
// so a workspace never holds some of them.
template <typename W, typename Alloc, typename Release>
bool grow_reduced(W& m, int cap, int64_t elems, Alloc alloc, Release release) {
  void* old = m.Bc;                 // the block begins with Bc
  ++m.red_gen;
  set_reduced(m, ReducedViews{}, 0, 0);
  if (old) release(old);
  Arena a{static_cast<char*>(alloc(reduced_view_bytes(cap, elems))), 0};
  if (!a.base) return false;
  set_reduced(m, reduced_views(a, cap, elems), cap, elems);
  return true;
}

}  // namespace fsim
