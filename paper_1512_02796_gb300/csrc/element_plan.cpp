// Host side of the element plan (see element.h): tet, edge and node
// numberings and the lists that connect them.  Depends on the mesh only;
// row and tet loops run on the host threads in fixed ranges.
#include "element.h"

#include <algorithm>

#include "host_threads.h"

namespace qpat {
namespace {

template <typename F>
void parallel(int64_t n, const F& fn) {
    parallel_ranges(n, n < 8192 ? 1 : host_threads(), [&](int, int64_t b, int64_t e) { fn(b, e); });
}

inline int64_t sell_at(const std::vector<int64_t>& ptr, int64_t row, int k) {
    return (ptr[size_t(row >> 5)] + k) * 32 + (row & 31);
}

// Edge (i, j), i < j, by a search of i's row.
inline int32_t find_edge(const HostMesh& h, const ElementPlan& p, int32_t i, int32_t j) {
    for (int k = 0; k < h.sell_len[size_t(i)]; ++k) {
        const int64_t at = sell_at(h.sell_ptr, i, k);
        if (p.ent_col[size_t(at)] == j) return p.ent_edge[size_t(at)];
    }
    return -1;
}

}  // namespace

ElementPlan build_element_plan(const HostMesh& h) {
    ElementPlan p;
    const int64_t N = h.N, E = h.E;
    // ---- tets by their lowest node, so that neighbouring rows read neighbouring tets
    {
        std::vector<int64_t> at(size_t(N + 1), 0);
        auto lowest = [&](int64_t t) {
            const int32_t* v = &h.tets[size_t(4 * t)];
            return std::min(std::min(v[0], v[1]), std::min(v[2], v[3]));
        };
        for (int64_t t = 0; t < E; ++t) ++at[size_t(lowest(t) + 1)];
        for (int64_t i = 0; i < N; ++i) at[size_t(i + 1)] += at[size_t(i)];
        p.tet.resize(size_t(4 * E));
        for (int64_t t = 0; t < E; ++t)
            std::copy_n(&h.tets[size_t(4 * t)], 4, &p.tet[size_t(4 * at[size_t(lowest(t))]++)]);
    }
    // ---- tets of each node
    p.node_ptr.assign(size_t(N + 1), 0);
    p.node_tet.resize(size_t(4 * E));
    for (int32_t v : p.tet) ++p.node_ptr[size_t(v + 1)];
    for (int64_t i = 0; i < N; ++i) p.node_ptr[size_t(i + 1)] += p.node_ptr[size_t(i)];
    {
        std::vector<int64_t> at(p.node_ptr.begin(), p.node_ptr.end() - 1);
        for (int64_t q = 0; q < 4 * E; ++q) p.node_tet[size_t(at[size_t(p.tet[size_t(q)])]++)] = int32_t(q / 4);
    }
    // ---- edges: the entries right of the diagonal, row by row
    p.ent_col.assign(h.sell_col.size(), 0);
    p.ent_edge.assign(h.sell_col.size(), -1);
    std::vector<int64_t> first(size_t(N + 1), 0);
    parallel(h.nslices, [&](int64_t b, int64_t e) {
        for (int64_t s = b; s < e; ++s) {
            const int nb = h.node_ptr[size_t(h.patch_of_slice[size_t(s)])];
            for (int64_t g = 32 * s; g < 32 * s + 32; ++g) {
                for (int64_t k = h.sell_ptr[size_t(s)]; k < h.sell_ptr[size_t(s + 1)]; ++k) {
                    const int64_t at = k * 32 + (g & 31);
                    p.ent_col[size_t(at)] = g < N ? h.nodes[size_t(nb + h.sell_col[size_t(at)])] : 0;
                }
                if (g < N)
                    for (int k = 0; k < h.sell_len[size_t(g)]; ++k)
                        first[size_t(g + 1)] += p.ent_col[size_t(sell_at(h.sell_ptr, g, k))] > g;
            }
        }
    });
    for (int64_t i = 0; i < N; ++i) first[size_t(i + 1)] += first[size_t(i)];
    p.NE = first[size_t(N)];
    p.edge.resize(size_t(2 * p.NE));
    parallel(N, [&](int64_t b, int64_t e) {
        for (int64_t g = b; g < e; ++g) {
            int64_t id = first[size_t(g)];
            for (int k = 0; k < h.sell_len[size_t(g)]; ++k) {
                const int64_t at = sell_at(h.sell_ptr, g, k);
                if (p.ent_col[size_t(at)] > g) {
                    p.edge[size_t(2 * id)] = int32_t(g);
                    p.edge[size_t(2 * id + 1)] = p.ent_col[size_t(at)];
                    p.ent_edge[size_t(at)] = int32_t(id++);
                }
            }
        }
    });
    p.in_prior.assign(size_t(p.NE), 0);
    p.pent_edge.assign(h.psell_col.size(), -1);
    parallel(N, [&](int64_t b, int64_t e) {
        for (int64_t g = b; g < e; ++g) {
            for (int k = 0; k < h.sell_len[size_t(g)]; ++k) {
                const int64_t at = sell_at(h.sell_ptr, g, k);
                if (p.ent_col[size_t(at)] < g) p.ent_edge[size_t(at)] = find_edge(h, p, p.ent_col[size_t(at)], int32_t(g));
            }
            const int nb = h.node_ptr[size_t(h.patch_of_slice[size_t(g >> 5)])];
            for (int k = 0; k < h.psell_len[size_t(g)]; ++k) {
                const int64_t at = sell_at(h.psell_ptr, g, k);
                const int32_t j = h.nodes[size_t(nb + h.psell_col[size_t(at)])];
                if (j == g) continue;
                const int32_t id = find_edge(h, p, std::min<int32_t>(j, int32_t(g)), std::max<int32_t>(j, int32_t(g)));
                p.pent_edge[size_t(at)] = id;
                if (j > g) p.in_prior[size_t(id)] = 1;
            }
        }
    });
    // ---- edges of each tet, tets around each edge
    p.tet_edge.resize(size_t(6 * E));
    parallel(E, [&](int64_t b, int64_t e) {
        for (int64_t t = b; t < e; ++t)
            for (int q = 0; q < 6; ++q) {
                const int32_t u = p.tet[size_t(4 * t + edge_a(q))], v = p.tet[size_t(4 * t + edge_b(q))];
                p.tet_edge[size_t(6 * t + q)] = find_edge(h, p, std::min(u, v), std::max(u, v));
            }
    });
    p.edge_ptr.assign(size_t(p.NE + 1), 0);
    // an edge (i, j) belongs to i's tets that hold j: the lists of row i are written by one thread
    auto each = [&](int64_t g, const auto& fn) {
        for (int64_t q = p.node_ptr[size_t(g)]; q < p.node_ptr[size_t(g + 1)]; ++q) {
            const int64_t t = p.node_tet[size_t(q)];
            for (int c = 0; c < 6; ++c) {
                const int32_t id = p.tet_edge[size_t(6 * t + c)];
                if (id >= first[size_t(g)] && id < first[size_t(g + 1)]) fn(id, uint32_t(8 * t + c));
            }
        }
    };
    parallel(N, [&](int64_t b, int64_t e) {
        for (int64_t g = b; g < e; ++g) each(g, [&](int32_t id, uint32_t) { ++p.edge_ptr[size_t(id + 1)]; });
    });
    for (int64_t i = 0; i < p.NE; ++i) p.edge_ptr[size_t(i + 1)] += p.edge_ptr[size_t(i)];
    p.edge_tet.resize(size_t(6 * E));
    parallel(N, [&](int64_t b, int64_t e) {
        std::vector<int64_t> at;
        for (int64_t g = b; g < e; ++g) {
            at.assign(p.edge_ptr.begin() + first[size_t(g)], p.edge_ptr.begin() + first[size_t(g + 1)]);
            each(g, [&](int32_t id, uint32_t code) { p.edge_tet[size_t(at[size_t(id - first[size_t(g)])]++)] = code; });
        }
    });
    // ---- Robin sums of the boundary faces (1/2 integral x v of the weak form: |F| / 24 (1 + delta_ab))
    p.edge_vr.assign(size_t(2 * p.NE), 0.0);
    p.node_vr.assign(size_t(2 * N), 0.0);
    for (int64_t f = 0; f < h.F; ++f)
        for (int a = 0; a < 3; ++a) {
            const int32_t u = h.faces_lib[size_t(3 * f + a)], v = h.faces_lib[size_t(3 * f + (a + 1) % 3)];
            p.node_vr[size_t(2 * int64_t(u) + 1)] += h.farea[size_t(f)] / 12.0;
            p.edge_vr[size_t(2 * int64_t(find_edge(h, p, std::min(u, v), std::max(u, v))) + 1)] += h.farea[size_t(f)] / 24.0;
        }
    return p;
}

std::string check_element_plan(const HostMesh& h, const ElementPlan& p) {
    const int64_t N = h.N, E = h.E;
    if (int64_t(p.tet.size()) != 4 * E || int64_t(p.node_tet.size()) != 4 * E || p.node_ptr[size_t(N)] != 4 * E)
        return "element plan: tet counts";
    if (p.edge_ptr[size_t(p.NE)] != 6 * E) return "element plan: tets around edges";
    for (int64_t i = 0; i < N; ++i)
        for (int64_t q = p.node_ptr[size_t(i)]; q < p.node_ptr[size_t(i + 1)]; ++q) {
            const int32_t* v = &p.tet[size_t(4 * int64_t(p.node_tet[size_t(q)]))];
            if (v[0] != i && v[1] != i && v[2] != i && v[3] != i) return "element plan: tet of a node";
            if (q > p.node_ptr[size_t(i)] && p.node_tet[size_t(q)] <= p.node_tet[size_t(q - 1)])
                return "element plan: tets of a node ascending";
        }
    for (int64_t t = 0; t < E; ++t)
        for (int c = 0; c < 6; ++c) {
            const int32_t id = p.tet_edge[size_t(6 * t + c)];
            const int32_t u = p.tet[size_t(4 * t + edge_a(c))], v = p.tet[size_t(4 * t + edge_b(c))];
            if (id < 0 || id >= p.NE || p.edge[size_t(2 * id)] != std::min(u, v) || p.edge[size_t(2 * id + 1)] != std::max(u, v))
                return "element plan: edge of a tet";
        }
    for (int64_t e = 0; e < p.NE; ++e) {
        if (p.edge[size_t(2 * e)] >= p.edge[size_t(2 * e + 1)] || p.edge[size_t(2 * e + 1)] >= N) return "element plan: edge nodes";
        for (int64_t q = p.edge_ptr[size_t(e)]; q < p.edge_ptr[size_t(e + 1)]; ++q) {
            const uint32_t code = p.edge_tet[size_t(q)];
            if (int64_t(code >> 3) >= E || (code & 7) > 5 || p.tet_edge[size_t(6 * int64_t(code >> 3) + (code & 7))] != e)
                return "element plan: tet of an edge";
            if (q > p.edge_ptr[size_t(e)] && code <= p.edge_tet[size_t(q - 1)]) return "element plan: tets of an edge ascending";
        }
    }
    for (int prior = 0; prior < 2; ++prior) {
        const auto& ptr = prior ? h.psell_ptr : h.sell_ptr;
        const auto& len = prior ? h.psell_len : h.sell_len;
        const auto& col = prior ? h.psell_col : h.sell_col;
        const auto& ent = prior ? p.pent_edge : p.ent_edge;
        for (int64_t g = 0; g < N; ++g) {
            const int nb = h.node_ptr[size_t(h.patch_of_slice[size_t(g >> 5)])];
            for (int k = 0; k < int(ptr[size_t((g >> 5) + 1)] - ptr[size_t(g >> 5)]); ++k) {
                const int64_t at = sell_at(ptr, g, k);
                const int32_t j = h.nodes[size_t(nb + col[size_t(at)])], id = ent[size_t(at)];
                if (!prior && p.ent_col[size_t(at)] != j) return "element plan: column of an entry";
                if (k >= len[size_t(g)] || j == g ? id != -1
                                                  : id < 0 || id >= p.NE || p.edge[size_t(2 * id)] != std::min<int64_t>(j, g) ||
                                                        p.edge[size_t(2 * id + 1)] != std::max<int64_t>(j, g) ||
                                                        (prior && !p.in_prior[size_t(id)]))
                    return "element plan: edge of an entry";
            }
        }
    }
    return "";
}

}  // namespace qpat
