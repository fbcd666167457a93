// Host driver for the walks around the nodes (csrc/topology.cpp): reads
// "n_nodes n_tris", the coordinates and the triangles from stdin, prints the
// edge order, the slots and the records.
#include <cstdio>
#include <string>
#include <vector>

#include "topology.h"

int main() {
    int nn = 0, nt = 0;
    if (std::scanf("%d %d", &nn, &nt) != 2) return 2;
    std::vector<double> x(3 * (size_t)nn);
    std::vector<int32_t> t(3 * (size_t)nt);
    for (double &v : x)
        if (std::scanf("%lf", &v) != 1) return 2;
    for (int32_t &v : t)
        if (std::scanf("%d", &v) != 1) return 2;
    lbib::Topology T;
    std::string err;
    if (!lbib::build_template(x.data(), nn, t.data(), nt, nullptr, T, err)) return 3;
    lbib::ring_walks(T, 0x8000u);
    for (int e : T.quad_order) std::printf("%d %d\n", T.edges[2 * e], T.edges[2 * e + 1]);
    std::printf("%zu %zu\n", T.slots.size() / 3, T.rings.size() / 4);
    for (int v : T.slots) std::printf("%d\n", v);
    for (uint32_t v : T.rings) std::printf("%u\n", v);
    return 0;
}
