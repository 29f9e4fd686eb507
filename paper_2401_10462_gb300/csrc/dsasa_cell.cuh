// The structure of a cell as its dual triangulation: a vertex is a triangle of plane ids, counter-
// clockwise seen from outside, with its neighbours across the edges (v0 v1), (v1 v2), (v2 v0); both
// are packed as three bytes of a word.
#pragma once
#include "dsasa_math.cuh"

namespace dsasa {

// Whether the vertex v2 (neighbours adj2) across edge k of vertex t (planes v) has that edge the other
// way round and t across it.  When it holds for every edge of every vertex, the step from a face's
// vertex to its next one can be undone, so a walk around a face comes back to where it began.
DS_HD bool edge_agrees(unsigned v, unsigned v2, unsigned adj2, int t, int k) {
    const unsigned a = (v >> (8 * k)) & 255u, b = (v >> (k == 2 ? 0 : 8 * k + 8)) & 255u;
    const unsigned x = v2 & 255u, y = (v2 >> 8) & 255u, z = (v2 >> 16) & 255u;
    const unsigned back = x == b && y == a ? adj2 : (y == b && z == a ? adj2 >> 8 : (z == b && x == a ? adj2 >> 16 : 255u));
    return (back & 255u) == (unsigned)t;
}

}  // namespace dsasa
