// Placement in the descriptor ring.
#pragma once

#include <cstddef>
#include <initializer_list>

namespace tlr {

// Bytes an array takes in the ring (arrays start on 256-byte boundaries).
inline size_t ring_bytes(size_t bytes) { return (bytes + 255) & ~(size_t)255; }

// Room behind `off` for arrays of these sizes one after the other: true, with
// `restart` set (and off 0) if the ring has to begin anew, its readers waited
// for; false if a ring of `cap` bytes cannot hold them together.  What one launch
// reads is placed after one call for all of it: placed one by one, a later
// array begins anew over an earlier one of the same launch when the two
// together exceed the ring.
inline bool ring_room(size_t cap, size_t &off, std::initializer_list<size_t> sizes, bool &restart) {
    size_t need = 0;
    for (size_t b : sizes) need += ring_bytes(b);
    restart = need <= cap && off + need > cap;
    if (restart) off = 0;
    return need <= cap;
}

}  // namespace tlr
