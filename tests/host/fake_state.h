// The state of a fake of the CUDA runtime, for running the library's host code without a GPU: device
// memory is host memory whose live blocks are known, an allocation beyond `limit` fails, streams and
// events do nothing (fake_runtime.cpp).
#pragma once

#include <cstddef>
#include <cstdint>

namespace fake {
extern size_t live, limit, total;
extern bool capturing;
extern int stale;     // accesses outside live memory
extern int unsafe;    // calls that would invalidate a stream capture, made during one
// What the projection of the next forwards counts.
extern unsigned long long visible, cells, pairs, pairs_per_cell;
// Whether the forwards to come have to write their pairs to one place, and where they do.
extern bool one_place;
extern const void* wrote_pairs;

void check(const void* p, size_t bytes, const char* what);
}  // namespace fake
