// Words of the order-free traversal (k2_parents.cu), one per vertex and tree.
//
// Until a vertex has reported to its parent: unreported children (high half) and
// sizes reported (low half).  After that: preorder offset (high half) and the
// ancestor that it is relative to (low half).  A child's offset is at least 1; the
// root is at offset 0 of itself.
//
// Plain C++ (constexpr, no CUDA): the same header is compiled by the host tests.
#pragma once

#include <cstdint>

namespace kc_host {

// Whether v, whose word was read as w, starts a report: it has no children.  A leaf's
// word is zero until its own report; a vertex with children holds their count, then
// their sizes, then an offset of at least 1, so never zero -- but the root, whose
// offset is 0 and whose ancestor is itself: vertex 0's word is zero again when it is
// the root of a finished tree.  The root is no leaf (n is at least 2).
constexpr bool par_is_leaf(uint64_t w, int64_t v, int64_t root) { return w == 0 && v != root; }

// What a child of size sz adds to its parent's word.
constexpr uint64_t par_report(int32_t sz) { return (uint64_t)(uint32_t)sz - (1ull << 32); }

// The parent's word before such an addition: whether the child was the last one, and
// the sizes that were there.
constexpr bool par_was_last(uint64_t old) { return (old >> 32) == 1; }
constexpr int32_t par_sizes(uint64_t old) { return (int32_t)(uint32_t)old; }

// The word of a vertex at offset `off` of ancestor a.
constexpr uint64_t par_at(uint32_t off, int32_t a) { return (uint64_t)off << 32 | (uint32_t)a; }

}  // namespace kc_host
