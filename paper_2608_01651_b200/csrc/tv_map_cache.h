// Tensor maps of the verify kernels, kept between calls (host code only).
//
// A map holds a base address, extents and strides, nothing of what lies there: a serving loop calls
// with the same buffers round after round, so the encodes of a launch are kept per thread.  What a
// kept set is found by is every value that it was encoded from, each compared for equality.
#pragma once
#include <cuda.h>
#include <stdint.h>

namespace tvtc {

// 4-D view of a node-indexed tensor: element (z, h, t, c) at z*sb + h*sh + t*st + c (element
// strides), c < d contiguous.  z = layer*request for dense and strided layouts, the layer for the
// planes of a packed forest (t then runs over the plane's `capacity` rows).
struct NodeView {
  uint64_t d, T, Hx, Z;
  int64_t sb, sh, st;
};
inline bool operator==(const NodeView& a, const NodeView& b) {
  return a.d == b.d && a.T == b.T && a.Hx == b.Hx && a.Z == b.Z && a.sb == b.sb && a.sh == b.sh && a.st == b.st;
}
// Tensor maps want ascending strides: the node and head dimensions go in stride order, and the
// kernel is told which of the two coordinates comes first.
inline bool node_first_of(const NodeView& v) { return v.Hx == 1 || v.st <= v.sh; }

// What a set of maps was encoded from: base addresses, the views of q and k | v | O (all zero where the
// set has no such map), the number of states, the nodes of a tree and the form of the boxes.
struct MapKey {
  const void* ptr[5];
  NodeView view[3];
  uint64_t items;
  int32_t T, kind;
};
inline bool operator==(const MapKey& a, const MapKey& b) {
  for (int i = 0; i < 5; ++i)
    if (a.ptr[i] != b.ptr[i]) return false;
  return a.items == b.items && a.T == b.T && a.kind == b.kind && a.view[0] == b.view[0] && a.view[1] == b.view[1] &&
         a.view[2] == b.view[2];
}

struct MapSet {
  MapKey key;
  alignas(64) CUtensorMap map[5];
};

template <class Make>
inline const MapSet* cached_maps(const MapKey& key, Make make) {
  constexpr int kEntries = 16;
  static thread_local MapSet cache[kEntries];
  static thread_local int used = 0, next = 0;
  for (int i = 0; i < used; ++i)
    if (cache[i].key == key) return &cache[i];
  MapSet& e = cache[next];
  e.key = key;
  if (!make(e.map)) {
    e.key = MapKey{};   // never matches: no launch has zero items
    return nullptr;
  }
  if (used < kEntries) ++used;
  next = (next + 1) % kEntries;
  return &e;
}

}  // namespace tvtc
