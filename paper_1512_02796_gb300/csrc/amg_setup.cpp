// Host side of the smoothed-aggregation hierarchy (see amg.h): aggregates
// of the matrix graph, the patterns of P, A P, R = P^T and P^T A P on every
// level, and the index plans that let the device form their values with
// plain gathers.  Everything here depends on the pattern only, is computed
// once per mesh and pattern, and is deterministic (row loops are split over
// host threads in fixed contiguous ranges and concatenated in order).
#include "amg.h"
#include "host_threads.h"
#include "qpat_internal.h"

#include <algorithm>

namespace qpat {
namespace {

// Threads for n rows (coarse levels have few, long rows).
int threads_for(int64_t n) { return n < 256 ? 1 : host_threads(); }

struct Csr {
    int64_t n = 0;
    std::vector<int64_t> ptr;
    std::vector<int32_t> col;
    int64_t len(int64_t i) const { return ptr[i + 1] - ptr[i]; }
};

// Distinct column ids of one row, collected in O(1) each.
struct Marker {
    std::vector<int64_t> stamp;
    std::vector<int32_t> list;
    explicit Marker(int64_t ncols) : stamp(size_t(ncols), -1) {}
    void begin() { list.clear(); }
    void add(int32_t c, int64_t row) {
        if (stamp[size_t(c)] != row) {
            stamp[size_t(c)] = row;
            list.push_back(c);
        }
    }
};

// CSR of n rows over ncols columns; row i = sorted distinct ids that
// gather(i, marker) adds.
template <typename G>
Csr build_rows(int64_t n, int64_t ncols, const G& gather) {
    const int nt = threads_for(n);
    std::vector<std::vector<int32_t>> cols(static_cast<size_t>(nt));
    std::vector<std::vector<int64_t>> lens(static_cast<size_t>(nt));
    parallel_ranges(n, nt, [&](int t, int64_t b, int64_t e) {
        Marker mk(ncols);
        auto& c = cols[size_t(t)];
        auto& l = lens[size_t(t)];
        l.reserve(size_t(e - b));
        for (int64_t i = b; i < e; ++i) {
            mk.begin();
            gather(i, mk);
            std::sort(mk.list.begin(), mk.list.end());
            c.insert(c.end(), mk.list.begin(), mk.list.end());
            l.push_back(int64_t(mk.list.size()));
        }
    });
    Csr out;
    out.n = n;
    out.ptr.assign(size_t(n + 1), 0);
    int64_t row = 0;
    for (int t = 0; t < nt; ++t)
        for (int64_t L : lens[size_t(t)]) {
            out.ptr[size_t(row + 1)] = out.ptr[size_t(row)] + L;
            ++row;
        }
    out.col.reserve(size_t(out.ptr[size_t(n)]));
    for (int t = 0; t < nt; ++t) out.col.insert(out.col.end(), cols[size_t(t)].begin(), cols[size_t(t)].end());
    return out;
}

// Position of column c in the sorted row [b, e) of col (the caller knows it is there).
inline int slot_of(const int32_t* col, int64_t b, int64_t e, int32_t c) {
    return int(std::lower_bound(col + b, col + e, c) - (col + b));
}

bool sell_from_csr(const Csr& c, SellPattern& s, std::string& err) {
    if (c.n > 0 && c.ptr[size_t(c.n)] >= int64_t(kAmgRowMajorLen) * c.n) {
        // long rows: row-major, so that the lanes sharing a row read consecutive entries
        s.n = c.n;
        s.nslices = 0;
        s.rowmajor = true;
        s.ptr = c.ptr;
        s.col = c.col;
        s.len.assign(size_t(c.n), 0);
        s.maxlen = 0;
        for (int64_t i = 0; i < c.n; ++i) {
            if (c.len(i) > 65535) {
                err = "multigrid: a row of a level holds more than 65535 entries";
                return false;
            }
            s.len[size_t(i)] = uint16_t(c.len(i));
            s.maxlen = std::max(s.maxlen, int(c.len(i)));
        }
        return true;
    }
    s.n = c.n;
    s.rowmajor = false;
    s.nslices = (c.n + 31) / 32;
    s.ptr.assign(size_t(s.nslices + 1), 0);
    s.len.assign(size_t(32 * s.nslices), 0);
    s.maxlen = 0;
    for (int64_t sl = 0; sl < s.nslices; ++sl) {
        int64_t w = 0;
        for (int64_t i = 32 * sl; i < std::min(c.n, 32 * sl + 32); ++i) w = std::max(w, c.len(i));
        if (w > 65535) {
            err = "multigrid: a row of a level holds more than 65535 entries";
            return false;
        }
        s.ptr[size_t(sl + 1)] = s.ptr[size_t(sl)] + w;
        s.maxlen = std::max(s.maxlen, int(w));
    }
    s.col.assign(size_t(32 * s.ptr[size_t(s.nslices)]), 0);
    for (int64_t sl = 0; sl < s.nslices; ++sl) {
        const int64_t w = s.ptr[size_t(sl + 1)] - s.ptr[size_t(sl)];
        for (int lane = 0; lane < 32; ++lane) {
            const int64_t i = 32 * sl + lane;
            const int64_t L = i < c.n ? c.len(i) : 0;
            if (i < c.n) s.len[size_t(i)] = uint16_t(L);
            for (int64_t k = 0; k < w; ++k)
                s.col[size_t((s.ptr[size_t(sl)] + k) * 32 + lane)] =
                    k < L ? c.col[size_t(c.ptr[size_t(i)] + k)] : int32_t(i < c.n ? i : 0);
        }
    }
    return true;
}

// One round of pairwise matching on a weighted graph (w: number of fine edges
// between two nodes): nodes in the given order take the free neighbour they
// share most edges with (ties: first in the order); a node without a free
// neighbour joins the pair it shares most edges with.
std::vector<int32_t> match(const AmgGraphPlan& G, int64_t& npairs) {
    const int64_t n = int64_t(G.order.size());
    std::vector<int32_t> rank(static_cast<size_t>(n)), to(size_t(n), -1);
    for (int64_t q = 0; q < n; ++q) rank[size_t(G.order[size_t(q)])] = int32_t(q);
    auto best = [&](int32_t i, bool taken) {
        int32_t j = -1;
        int64_t at = 0;
        for (int64_t k = G.ptr[size_t(i)]; k < G.ptr[size_t(i + 1)]; ++k) {
            const int32_t c = G.col[size_t(k)];
            if ((to[size_t(c)] >= 0) != taken) continue;
            if (j < 0 || G.w[size_t(k)] > G.w[size_t(at)] ||
                (G.w[size_t(k)] == G.w[size_t(at)] && rank[size_t(c)] < rank[size_t(j)])) {
                j = c;
                at = k;
            }
        }
        return j;
    };
    int32_t np = 0;
    std::vector<int32_t> alone;
    for (int32_t i : G.order) {
        if (to[size_t(i)] >= 0) continue;
        const int32_t j = best(i, false);
        if (j < 0) {
            alone.push_back(i);
            continue;
        }
        to[size_t(i)] = to[size_t(j)] = np++;
    }
    std::vector<int32_t> joins(alone.size());
    for (size_t q = 0; q < alone.size(); ++q) {
        const int32_t j = best(alone[q], true);
        joins[q] = j < 0 ? -1 : to[size_t(j)];
    }
    for (size_t q = 0; q < alone.size(); ++q) to[size_t(alone[q])] = joins[q] >= 0 ? joins[q] : np++;
    npairs = np;
    return to;
}

// The graph of the sets `to`: edge counts between different sets, rows sorted; sets keep their numbers as order.
AmgGraphPlan merge(const AmgGraphPlan& G, const std::vector<int32_t>& to, int64_t nc) {
    const int64_t n = int64_t(to.size());
    std::vector<int64_t> mptr(size_t(nc + 1), 0);
    std::vector<int32_t> members(static_cast<size_t>(n));
    for (int32_t t : to) ++mptr[size_t(t + 1)];
    for (int64_t I = 0; I < nc; ++I) mptr[size_t(I + 1)] += mptr[size_t(I)];
    {
        std::vector<int64_t> at(mptr.begin(), mptr.end() - 1);
        for (int64_t i = 0; i < n; ++i) members[size_t(at[size_t(to[size_t(i)])]++)] = int32_t(i);
    }
    auto gather = [&](int64_t I, Marker& mk) {
        for (int64_t q = mptr[size_t(I)]; q < mptr[size_t(I + 1)]; ++q) {
            const int32_t i = members[size_t(q)];
            for (int64_t k = G.ptr[size_t(i)]; k < G.ptr[size_t(i + 1)]; ++k) {
                const int32_t J = to[size_t(G.col[size_t(k)])];
                if (J != I) mk.add(J, I);
            }
        }
    };
    const Csr c = build_rows(nc, nc, gather);
    AmgGraphPlan out;
    out.w.assign(c.col.size(), 0);
    parallel_ranges(nc, threads_for(nc), [&](int, int64_t b, int64_t e) {
        for (int64_t I = b; I < e; ++I)
            for (int64_t q = mptr[size_t(I)]; q < mptr[size_t(I + 1)]; ++q) {
                const int32_t i = members[size_t(q)];
                for (int64_t k = G.ptr[size_t(i)]; k < G.ptr[size_t(i + 1)]; ++k) {
                    const int32_t J = to[size_t(G.col[size_t(k)])];
                    if (J != I)
                        out.w[size_t(c.ptr[size_t(I)] + slot_of(c.col.data(), c.ptr[size_t(I)], c.ptr[size_t(I + 1)], J))] +=
                            G.w[size_t(k)];
                }
            }
    });
    out.ptr = c.ptr;
    out.col = c.col;
    out.order.resize(size_t(nc));
    for (int64_t I = 0; I < nc; ++I) out.order[size_t(I)] = int32_t(I);
    return out;
}

// Aggregates of 8: three rounds of pairwise matching, heaviest neighbours
// first and in the order of the grid the nodes come from, which on a
// structured grid gives its 2 x 2 x 2 blocks.  The graph becomes the next
// level's.  Aggregates are numbered by their first node.
std::vector<int32_t> aggregate(AmgGraphPlan& G, int64_t& nagg) {
    const int64_t n = int64_t(G.order.size());
    std::vector<int32_t> agg(static_cast<size_t>(n));
    for (int64_t i = 0; i < n; ++i) agg[size_t(i)] = int32_t(i);
    int64_t nc = n;
    for (int round = 0; round < 3; ++round) {
        const std::vector<int32_t> to = match(G, nc);
        G = merge(G, to, nc);
        for (int32_t& a : agg) a = to[size_t(a)];
    }
    std::vector<int32_t> name(size_t(nc), -1);
    int32_t next = 0;
    for (int32_t& a : agg) {
        if (name[size_t(a)] < 0) name[size_t(a)] = next++;
        a = name[size_t(a)];
    }
    // the graph in the new numbers, visited in the old order
    AmgGraphPlan H;
    H.order = name;
    H.ptr.assign(size_t(nc + 1), 0);
    H.col.resize(G.col.size());
    H.w.resize(G.w.size());
    for (int64_t I = 0; I < nc; ++I) H.ptr[size_t(name[size_t(I)] + 1)] = G.ptr[size_t(I + 1)] - G.ptr[size_t(I)];
    for (int64_t I = 0; I < nc; ++I) H.ptr[size_t(I + 1)] += H.ptr[size_t(I)];
    for (int64_t I = 0; I < nc; ++I)
        for (int64_t k = G.ptr[size_t(I)], o = H.ptr[size_t(name[size_t(I)])]; k < G.ptr[size_t(I + 1)]; ++k, ++o) {
            H.col[size_t(o)] = name[size_t(G.col[size_t(k)])];
            H.w[size_t(o)] = G.w[size_t(k)];
        }
    G = std::move(H);
    nagg = nc;
    return agg;
}

}  // namespace

namespace {

bool set_diag(AmgLevelPlan& L) {
    const SellPattern& A = L.A;
    L.diag.assign(size_t(A.n), -1);
    for (int64_t i = 0; i < A.n; ++i)
        for (int k = 0; k < A.len[size_t(i)]; ++k)
            if (A.col[size_t(A.pos(i, k))] == i) {
                L.diag[size_t(i)] = k;
                break;
            }
    return std::find(L.diag.begin(), L.diag.end(), -1) == L.diag.end();
}

// The transfer from level L to the next one; `coarse` receives the next
// level's pattern (rows sorted).
bool build_transfer(AmgLevelPlan& L, AmgGraphPlan& graph, Csr& coarse, std::string& err) {
    const SellPattern& A = L.A;
    const int64_t n = A.n;
    const int nt = threads_for(n);
    int64_t nc = 0;
    const AmgGraphPlan fine = graph;
    L.agg = aggregate(graph, nc);
    L.nc = nc;
    if (nc <= 0 || nc >= n) {
        err = "multigrid: aggregation made no progress";
        return false;
    }
    // P: row i holds the aggregates of i and of its graph neighbours
    const Csr Pc = build_rows(n, nc, [&](int64_t i, Marker& mk) {
        mk.add(L.agg[size_t(i)], i);
        for (int64_t k = fine.ptr[size_t(i)]; k < fine.ptr[size_t(i + 1)]; ++k) mk.add(L.agg[size_t(fine.col[size_t(k)])], i);
    });
    if (!sell_from_csr(Pc, L.P, err)) return false;
    L.a2p.assign(size_t(A.entries()), kAmgDropped);
    L.pself.assign(size_t(n), 0);
    parallel_ranges(n, nt, [&](int, int64_t b, int64_t e) {
        std::vector<int64_t> kept(size_t(n), -1);
        for (int64_t i = b; i < e; ++i) {
            const int64_t pb = Pc.ptr[size_t(i)], pe = Pc.ptr[size_t(i + 1)];
            kept[size_t(i)] = i;
            for (int64_t k = fine.ptr[size_t(i)]; k < fine.ptr[size_t(i + 1)]; ++k) kept[size_t(fine.col[size_t(k)])] = i;
            for (int k = 0; k < A.len[size_t(i)]; ++k) {
                const int64_t at = A.pos(i, k);
                const int32_t j = A.col[size_t(at)];
                if (kept[size_t(j)] == i) L.a2p[size_t(at)] = uint16_t(slot_of(Pc.col.data(), pb, pe, L.agg[size_t(j)]));
            }
            L.pself[size_t(i)] = uint16_t(slot_of(Pc.col.data(), pb, pe, L.agg[size_t(i)]));
        }
    });
    // A P: row i is the union of the P rows of i's neighbours
    Csr APc = build_rows(n, nc, [&](int64_t i, Marker& mk) {
        for (int k = 0; k < A.len[size_t(i)]; ++k) {
            const int32_t j = A.col[size_t(A.pos(i, k))];
            for (int64_t q = Pc.ptr[size_t(j)]; q < Pc.ptr[size_t(j + 1)]; ++q) mk.add(Pc.col[size_t(q)], i);
        }
    });
    for (int64_t i = 0; i < n; ++i)
        if (APc.len(i) > 65535) {
            err = "multigrid: a row of A P holds more than 65535 entries";
            return false;
        }
    L.ap_sptr.assign(size_t(n + 1), 0);
    for (int64_t i = 0; i < n; ++i) {
        int64_t s = 0;
        for (int k = 0; k < A.len[size_t(i)]; ++k) s += Pc.len(A.col[size_t(A.pos(i, k))]);
        L.ap_sptr[size_t(i + 1)] = L.ap_sptr[size_t(i)] + s;
    }
    L.ap_slot.assign(size_t(L.ap_sptr[size_t(n)]), 0);
    parallel_ranges(n, nt, [&](int, int64_t b, int64_t e) {
        std::vector<uint16_t> where(static_cast<size_t>(nc));
        for (int64_t i = b; i < e; ++i) {
            for (int64_t q = APc.ptr[size_t(i)]; q < APc.ptr[size_t(i + 1)]; ++q)
                where[size_t(APc.col[size_t(q)])] = uint16_t(q - APc.ptr[size_t(i)]);
            int64_t o = L.ap_sptr[size_t(i)];
            for (int k = 0; k < A.len[size_t(i)]; ++k) {
                const int32_t j = A.col[size_t(A.pos(i, k))];
                for (int64_t q = Pc.ptr[size_t(j)]; q < Pc.ptr[size_t(j + 1)]; ++q)
                    L.ap_slot[size_t(o++)] = where[size_t(Pc.col[size_t(q)])];
            }
        }
    });
    // R = P^T: coarse row I lists the fine rows whose P row holds I, ascending
    Csr Rc;
    Rc.n = nc;
    Rc.ptr.assign(size_t(nc + 1), 0);
    for (int32_t I : Pc.col) ++Rc.ptr[size_t(I + 1)];
    for (int64_t I = 0; I < nc; ++I) Rc.ptr[size_t(I + 1)] += Rc.ptr[size_t(I)];
    Rc.col.assign(Pc.col.size(), 0);
    std::vector<int64_t> rsrc(Pc.col.size(), -1);
    {
        std::vector<int64_t> next(Rc.ptr.begin(), Rc.ptr.end() - 1);
        for (int64_t i = 0; i < n; ++i)
            for (int64_t q = Pc.ptr[size_t(i)]; q < Pc.ptr[size_t(i + 1)]; ++q) {
                const int64_t at = next[size_t(Pc.col[size_t(q)])]++;
                Rc.col[size_t(at)] = int32_t(i);
                rsrc[size_t(at)] = L.P.pos(i, int(q - Pc.ptr[size_t(i)]));
            }
    }
    if (!sell_from_csr(Rc, L.R, err)) return false;
    L.r_src.assign(size_t(L.R.entries()), -1);
    for (int64_t I = 0; I < nc; ++I)
        for (int k = 0; k < L.R.len[size_t(I)]; ++k) L.r_src[size_t(L.R.pos(I, k))] = rsrc[size_t(Rc.ptr[size_t(I)] + k)];
    // P^T A P: coarse row I is the union of the A P rows of R's row I
    coarse = build_rows(nc, nc, [&](int64_t I, Marker& mk) {
        for (int64_t q = Rc.ptr[size_t(I)]; q < Rc.ptr[size_t(I + 1)]; ++q) {
            const int32_t i = Rc.col[size_t(q)];
            for (int64_t a = APc.ptr[size_t(i)]; a < APc.ptr[size_t(i + 1)]; ++a) mk.add(APc.col[size_t(a)], I);
        }
    });
    L.g_ptr.assign(size_t(nc + 1), 0);
    for (int64_t I = 0; I < nc; ++I) {
        int64_t s = 0;
        for (int64_t q = Rc.ptr[size_t(I)]; q < Rc.ptr[size_t(I + 1)]; ++q) s += APc.len(Rc.col[size_t(q)]);
        L.g_ptr[size_t(I + 1)] = L.g_ptr[size_t(I)] + s;
    }
    L.g_slot.assign(size_t(L.g_ptr[size_t(nc)]), 0);
    parallel_ranges(nc, threads_for(nc), [&](int, int64_t b, int64_t e) {
        std::vector<uint16_t> where(static_cast<size_t>(nc));
        for (int64_t I = b; I < e; ++I) {
            for (int64_t q = coarse.ptr[size_t(I)]; q < coarse.ptr[size_t(I + 1)]; ++q)
                where[size_t(coarse.col[size_t(q)])] = uint16_t(q - coarse.ptr[size_t(I)]);
            int64_t o = L.g_ptr[size_t(I)];
            for (int64_t q = Rc.ptr[size_t(I)]; q < Rc.ptr[size_t(I + 1)]; ++q) {
                const int32_t i = Rc.col[size_t(q)];
                for (int64_t a = APc.ptr[size_t(i)]; a < APc.ptr[size_t(i + 1)]; ++a)
                    L.g_slot[size_t(o++)] = where[size_t(APc.col[size_t(a)])];
            }
        }
    });
    L.ap_ptr = std::move(APc.ptr);
    L.ap_col = std::move(APc.col);
    return true;
}

}  // namespace

AmgPlan amg_build_plan(const SellPattern& fine, AmgGraphPlan graph) {
    AmgPlan plan;
    plan.levels.reserve(kAmgMaxLevels);
    plan.levels.emplace_back();
    plan.levels[0].A = fine;
    if (!set_diag(plan.levels[0])) {
        plan.error = "multigrid: a row of the pattern has no diagonal entry";
        return plan;
    }
    while (plan.levels.back().A.n > kAmgCoarsest) {
        if (int(plan.levels.size()) >= kAmgMaxLevels) {
            plan.error = "multigrid: no coarsest level of at most 64 rows within 12 levels";
            return plan;
        }
        Csr coarse;
        if (!build_transfer(plan.levels.back(), graph, coarse, plan.error)) return plan;
        plan.levels.emplace_back();
        if (!sell_from_csr(coarse, plan.levels.back().A, plan.error)) return plan;
        if (!set_diag(plan.levels.back())) {
            plan.error = "multigrid: a coarse row has no diagonal entry";
            return plan;
        }
    }
    return plan;
}

}  // namespace qpat

namespace qpat {

SellPattern amg_fine_pattern(const HostMesh& h) {
    SellPattern f;
    f.n = h.N;
    f.nslices = int64_t(h.psell_ptr.size()) - 1;
    f.ptr = h.psell_ptr;
    f.col.assign(size_t(32 * h.psell_ptr.back()), 0);
    f.len.assign(h.psell_len.begin(), h.psell_len.end());
    f.maxlen = 0;
    for (int64_t s = 0; s < f.nslices; ++s) {
        const int64_t w = f.ptr[size_t(s + 1)] - f.ptr[size_t(s)];
        f.maxlen = std::max(f.maxlen, int(w));
        const int nb = h.node_ptr[size_t(h.patch_of_slice[size_t(s)])];
        for (int lane = 0; lane < 32; ++lane) {
            const int64_t g = 32 * s + lane;
            for (int64_t k = 0; k < w; ++k) {
                const int64_t at = (f.ptr[size_t(s)] + k) * 32 + lane;
                f.col[size_t(at)] = g < h.N ? h.nodes[size_t(nb + h.psell_col[size_t(at)])] : 0;
            }
        }
    }
    return f;
}

AmgGraphPlan amg_fine_graph(const HostMesh& h, const SellPattern& fine) {
    AmgGraphPlan G;
    const int64_t n = fine.n;
    G.ptr.assign(size_t(n + 1), 0);
    for (int64_t i = 0; i < n; ++i) G.ptr[size_t(i + 1)] = G.ptr[size_t(i)] + fine.len[size_t(i)] - 1;  // without the diagonal
    G.col.reserve(size_t(G.ptr[size_t(n)]));
    for (int64_t i = 0; i < n; ++i)
        for (int k = 0; k < fine.len[size_t(i)]; ++k) {
            const int32_t j = fine.col[size_t(fine.pos(i, k))];
            if (j != i) G.col.push_back(j);
        }
    G.w.assign(G.col.size(), 1);
    // by z, then y, then x, on the lattice of the Morton order (which absorbs the rounding of grid coordinates)
    double lo[3] = {h.xyz[0], h.xyz[1], h.xyz[2]};
    for (int64_t i = 0; i < n; ++i)
        for (int c = 0; c < 3; ++c) lo[c] = std::min(lo[c], h.xyz[size_t(3 * i + c)]);
    std::vector<std::pair<uint64_t, int32_t>> key(static_cast<size_t>(n));
    for (int64_t i = 0; i < n; ++i) {
        uint64_t code = 0;
        for (int c = 2; c >= 0; --c) {
            const double t = (h.xyz[size_t(3 * i + c)] - lo[c]) / std::max(h.extent, 1e-300);
            code = code << 21 | uint64_t(std::min(std::max(t, 0.0), 1.0) * double((1u << 21) - 1) + 0.5);
        }
        key[size_t(i)] = {code, int32_t(i)};
    }
    std::sort(key.begin(), key.end());
    G.order.resize(size_t(n));
    for (int64_t q = 0; q < n; ++q) G.order[size_t(q)] = key[size_t(q)].second;
    return G;
}

std::string amg_check_plan(const AmgPlan& plan) {
    if (!plan.error.empty()) return plan.error;
    if (plan.levels.empty()) return "no levels";
    for (size_t l = 0; l < plan.levels.size(); ++l) {
        const AmgLevelPlan& L = plan.levels[l];
        const SellPattern& A = L.A;
        const std::string at = "level " + std::to_string(l) + ": ";
        for (int64_t i = 0; i < A.n; ++i)
            if (L.diag[size_t(i)] < 0 || A.col[size_t(A.pos(i, L.diag[size_t(i)]))] != i) return at + "diagonal slot";
        if (l + 1 == plan.levels.size()) {
            if (L.nc != 0) return at + "coarsest level with a transfer";
            if (A.n > kAmgCoarsest) return at + "coarsest level too large";
            break;
        }
        const SellPattern& C = plan.levels[l + 1].A;
        if (L.nc != C.n || L.nc >= A.n) return at + "coarse size";
        // every aggregate non-empty
        std::vector<int> members(size_t(L.nc), 0);
        for (int32_t a : L.agg) {
            if (a < 0 || a >= L.nc) return at + "aggregate id";
            ++members[size_t(a)];
        }
        if (std::find(members.begin(), members.end(), 0) != members.end()) return at + "empty aggregate";
        // P rows: the aggregates of the row's neighbours, a2p and pself point at them
        for (int64_t i = 0; i < A.n; ++i) {
            const int LP = L.P.len[size_t(i)];
            for (int k = 1; k < LP; ++k)
                if (L.P.col[size_t(L.P.pos(i, k - 1))] >= L.P.col[size_t(L.P.pos(i, k))]) return at + "P row order";
            if (L.pself[size_t(i)] >= LP || L.P.col[size_t(L.P.pos(i, L.pself[size_t(i)]))] != L.agg[size_t(i)])
                return at + "pself";
            for (int k = 0; k < A.len[size_t(i)]; ++k) {
                const int64_t e = A.pos(i, k);
                const int s = L.a2p[size_t(e)];
                if (s == kAmgDropped && A.col[size_t(e)] != i) continue;
                if (s >= LP || L.P.col[size_t(L.P.pos(i, s))] != L.agg[size_t(A.col[size_t(e)])]) return at + "a2p";
            }
        }
        // A P slots name the P entry's column
        for (int64_t i = 0; i < A.n; ++i) {
            int64_t o = L.ap_sptr[size_t(i)];
            const int64_t b = L.ap_ptr[size_t(i)], e = L.ap_ptr[size_t(i + 1)];
            for (int k = 0; k < A.len[size_t(i)]; ++k) {
                const int32_t j = A.col[size_t(A.pos(i, k))];
                for (int kk = 0; kk < L.P.len[size_t(j)]; ++kk) {
                    const int s = L.ap_slot[size_t(o++)];
                    if (s >= e - b || L.ap_col[size_t(b + s)] != L.P.col[size_t(L.P.pos(j, kk))]) return at + "ap_slot";
                }
            }
            if (o != L.ap_sptr[size_t(i + 1)]) return at + "ap_sptr";
        }
        // R = P^T: every P entry exactly once, at the right row and column
        std::vector<char> seen(size_t(L.P.entries()), 0);
        int64_t count = 0;
        for (int64_t I = 0; I < L.nc; ++I)
            for (int k = 0; k < L.R.len[size_t(I)]; ++k) {
                const int64_t e = L.R.pos(I, k);
                const int64_t src = L.r_src[size_t(e)];
                const int32_t i = L.R.col[size_t(e)];
                if (src < 0 || src >= L.P.entries() || seen[size_t(src)]) return at + "r_src";
                seen[size_t(src)] = 1;
                ++count;
                // src must lie in row i of P and hold column I
                bool ok = false;
                for (int kk = 0; kk < L.P.len[size_t(i)] && !ok; ++kk) ok = L.P.pos(i, kk) == src && L.P.col[size_t(src)] == I;
                if (!ok) return at + "R is not P^T";
            }
        int64_t pentries = 0;
        for (int64_t i = 0; i < A.n; ++i) pentries += L.P.len[size_t(i)];
        if (count != pentries) return at + "R misses P entries";
        // Galerkin slots name the A P column in the coarse row
        for (int64_t I = 0; I < L.nc; ++I) {
            int64_t o = L.g_ptr[size_t(I)];
            for (int k = 0; k < L.R.len[size_t(I)]; ++k) {
                const int32_t i = L.R.col[size_t(L.R.pos(I, k))];
                for (int64_t a = L.ap_ptr[size_t(i)]; a < L.ap_ptr[size_t(i + 1)]; ++a) {
                    const int s = L.g_slot[size_t(o++)];
                    if (s >= C.len[size_t(I)] || C.col[size_t(C.pos(I, s))] != L.ap_col[size_t(a)]) return at + "g_slot";
                }
            }
            if (o != L.g_ptr[size_t(I + 1)]) return at + "g_ptr";
        }
        // the coarse pattern is symmetric
        for (int64_t I = 0; I < C.n; ++I)
            for (int k = 0; k < C.len[size_t(I)]; ++k) {
                const int32_t J = C.col[size_t(C.pos(I, k))];
                bool found = false;
                for (int kk = 0; kk < C.len[size_t(J)] && !found; ++kk) found = C.col[size_t(C.pos(J, kk))] == I;
                if (!found) return at + "coarse pattern not symmetric";
            }
    }
    return "";
}

}  // namespace qpat
