// Host build of the cell structure's checks for CPU unit tests (tests/test_cell_structure.py).
#include "../paper_2401_10462_gb300/csrc/dsasa_cell.cuh"

using namespace dsasa;

// the number of directed edges of a cell that do not agree: n vertices of three plane bytes each
// (dead: 0x00ffffff), their packed neighbours
extern "C" int cc_disagreeing(const unsigned* v, const unsigned* adj, int n) {
    int bad = 0;
    for (int t = 0; t < n; ++t)
        for (int k = 0; k < 3; ++k) {
            const int t2 = (adj[t] >> (8 * k)) & 255u;
            if (v[t] != 0x00ffffffu && (t2 >= n || !edge_agrees(v[t], v[t2], adj[t2], t, k))) ++bad;
        }
    return bad;
}
