// Host build of the nested-dissection trees and their device tables (nd.cuh).
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <exception>
#include <functional>
#include <mutex>
#include <numeric>
#include <system_error>
#include <thread>

#include "common.cuh"
#include "ndsolve.cuh"

namespace thm {

namespace {

// Cells of a leaf of the bisection.  Order 2 stops at 2x2 cells (the cells
// themselves are leaves below, for their bubbles); order 1 has no such leaves
// and stops earlier, where a node's dense block is still about as large as
// the padding of its rows.
int leaf_cells(const thm_mesh* m) { return m->dim == 3 ? 8 : m->order == 2 ? 4 : 8; }

// A node absorbs its children while their unknowns together stay below this:
// every absorbed level is two dependent steps less in a solve.
constexpr int ND_MERGE = 24;

struct Bin {                       // bisection node over cells [c0, c1) of the permuted cell list
    int l = -1, r = -1, parent = -1, depth = 0, c0 = 0, c1 = 0;
    int node = -1;                 // tree node that holds its unknowns
};
struct Node {
    int parent = -1, depth = 0, rank = 0;
    std::vector<int> ch;
    std::vector<int32_t> s, b;     // local rows
    int vpos = 0, upos = 0;        // in the CTA's vector / the level's u buffer
    int row_f = 0, row_b = 0, slt_f = 0, slt_b = 0;
    int64_t id = 0;                // global node number
    int64_t front = 0;             // its front's place in the depth's workspace
    double cost = 0;               // values under the node
};

struct SubTree {
    std::vector<Node> nodes;       // [0] is the root
    int maxdepth = 0;
};

// Bisection of the cells cs by their centres.
void bisect(const thm_mesh* m, std::vector<int32_t>& cs, int leaf, std::vector<Bin>& bins) {
    const int d = m->dim, nv = d == 2 ? 4 : 8;
    std::vector<double> X((size_t)cs.size() * d);
    std::vector<int> at(cs.size());
    std::iota(at.begin(), at.end(), 0);
    for (size_t i = 0; i < cs.size(); ++i)
        for (int k = 0; k < d; ++k) {
            double a = 0;
            for (int v = 0; v < nv; ++v) a += m->coords[m->cells[(int64_t)cs[i] * nv + v] * d + k];
            X[i * d + k] = a / nv;
        }
    bins.clear();
    bins.emplace_back();
    bins[0].c1 = (int)cs.size();
    for (size_t q = 0; q < bins.size(); ++q) {
        const int c0 = bins[q].c0, c1 = bins[q].c1, n = c1 - c0;
        if (n <= leaf) continue;
        double lo[3], hi[3];
        int axes[3] = {0, 1, 2};
        for (int k = 0; k < d; ++k) {
            lo[k] = 1e300; hi[k] = -1e300;
            for (int i = c0; i < c1; ++i) { lo[k] = std::min(lo[k], X[at[i] * d + k]); hi[k] = std::max(hi[k], X[at[i] * d + k]); }
        }
        std::stable_sort(axes, axes + d, [&](int a, int b) { return hi[a] - lo[a] > (hi[b] - lo[b]) * (1 + 1e-9); });
        int cut = -1;
        for (int t = 0; t < d && cut < 0; ++t) {          // the gap nearest the middle, along the longest axis that has one
            const int k = axes[t];
            const double tol = 1e-9 * (hi[k] - lo[k]);
            std::sort(at.begin() + c0, at.begin() + c1, [&](int a, int b) {
                return X[a * d + k] != X[b * d + k] ? X[a * d + k] < X[b * d + k] : a < b;
            });
            for (int i = c0 + 1; i < c1; ++i)
                if (X[at[i] * d + k] - X[at[i - 1] * d + k] > tol && (cut < 0 || std::abs(2 * (i - c0) - n) < std::abs(2 * (cut - c0) - n)))
                    cut = i;
        }
        if (cut < 0) cut = c0 + n / 2;                    // coincident centres
        for (int side = 0; side < 2; ++side) {
            Bin b;
            b.parent = (int)q;
            b.depth = bins[q].depth + 1;
            b.c0 = side == 0 ? c0 : cut;
            b.c1 = side == 0 ? cut : c1;
            (side == 0 ? bins[q].l : bins[q].r) = (int)bins.size();
            bins.push_back(b);
        }
    }
    std::vector<int32_t> out(cs.size());
    for (size_t i = 0; i < cs.size(); ++i) out[i] = cs[at[i]];
    cs.swap(out);
}

// The tree of subdomain s for C = 2^p CTAs, with the unknowns of `moves` in the nodes it names.
void build_tree(const thm_mesh* m, int s, std::vector<int32_t> cs, int p, const std::vector<NdMove>* moves,
                std::vector<int32_t>& cell_bin, SubTree& T) {
    const auto& S = m->subs[s];
    std::vector<Bin> bins;
    bisect(m, cs, leaf_cells(m), bins);
    for (size_t q = 0; q < bins.size(); ++q)
        if (bins[q].l < 0)
            for (int i = bins[q].c0; i < bins[q].c1; ++i) cell_bin[cs[i]] = (int32_t)q;
    // the part that holds all cells of a row: lowest common ancestor of their leaves
    const int ne = (int)S.ne;
    std::vector<std::vector<int32_t>> srow(bins.size());
    for (int i = 0; i < ne; ++i) {
        const int64_t r = S.off + i;
        int a = -1;
        for (int t = 0; t < m->maxc; ++t) {
            const int32_t c = m->row_cell[r * m->maxc + t];
            if (c < 0) break;
            int b = cell_bin[c];
            if (a < 0) { a = b; continue; }
            while (bins[a].depth > bins[b].depth) a = bins[a].parent;
            while (bins[b].depth > bins[a].depth) b = bins[b].parent;
            while (a != b) { a = bins[a].parent; b = bins[b].parent; }
        }
        srow[a].push_back((int32_t)r);
    }
    // nodes: the top p cuts are the root; a node absorbs its two children
    // while the unknowns together stay small
    T.nodes.clear();
    for (size_t q = 0; q < bins.size(); ++q) {
        const int par = bins[q].parent;
        const bool join = par >= 0 && (bins[q].depth <= p - 1 || bins[q].node == -2);
        if (join) {
            bins[q].node = bins[par].node;
        } else {
            bins[q].node = (int)T.nodes.size();
            T.nodes.emplace_back();
            if (par >= 0) {
                T.nodes.back().parent = bins[par].node;
                T.nodes[bins[par].node].ch.push_back(bins[q].node);
            }
        }
        Node& N = T.nodes[bins[q].node];
        N.s.insert(N.s.end(), srow[q].begin(), srow[q].end());
        if (bins[q].l >= 0 && bins[q].depth >= p) {
            const size_t a = srow[bins[q].l].size() + srow[bins[q].r].size();
            if (N.s.size() + a <= (size_t)ND_MERGE && bins[bins[q].l].l >= 0 && bins[bins[q].r].l >= 0)
                bins[bins[q].l].node = bins[bins[q].r].node = -2;
        }
    }
    // order 2: a leaf per cell for its bubbles
    std::vector<int> cell_node(cs.size(), -1);
    if (m->order == 2)
        for (size_t i = 0; i < cs.size(); ++i) {
            const int host = bins[cell_bin[cs[i]]].node;
            cell_node[i] = (int)T.nodes.size();
            Node N;
            N.parent = host;
            for (int k = 8; k < 12; ++k) N.s.push_back(m->cell_loc[(int64_t)cs[i] * 12 + k]);
            std::sort(N.s.begin(), N.s.end());
            T.nodes.push_back(N);
            T.nodes[host].ch.push_back(cell_node[i]);
        }
    if (moves && !moves->empty()) {
        std::vector<int32_t> to(S.n, -1);
        for (const NdMove& v : *moves) to[v.row - S.off] = v.node;
        for (auto& N : T.nodes)
            N.s.erase(std::remove_if(N.s.begin(), N.s.end(), [&](int32_t r) { return to[r - S.off] >= 0; }), N.s.end());
        for (const NdMove& v : *moves) T.nodes[v.node].s.push_back(v.row);
    }
    // depths and ancestor unknowns, children before parents (a parent's number is lower than its children's)
    T.maxdepth = 0;
    std::vector<std::vector<int32_t>> own(T.nodes.size());
    for (size_t q = 1; q < T.nodes.size(); ++q) {
        T.nodes[q].depth = T.nodes[T.nodes[q].parent].depth + 1;
        T.maxdepth = std::max(T.maxdepth, T.nodes[q].depth);
    }
    const int dpc = m->dpc;                            // (what a node eliminates itself is sorted out below)
    for (size_t i = 0; i < cs.size(); ++i)
        for (int k = 0; k < dpc; ++k) {
            const int32_t r = m->cell_loc[(int64_t)cs[i] * dpc + k];
            if (r >= 0) own[m->order == 2 ? cell_node[i] : bins[cell_bin[cs[i]]].node].push_back(r);
        }
    std::vector<int32_t> mark(S.n, -1);
    for (int q = (int)T.nodes.size() - 1; q >= 0; --q) {
        Node& N = T.nodes[q];
        std::sort(N.s.begin(), N.s.end());
        for (int32_t r : N.s) mark[r - S.off] = q;
        auto take = [&](int32_t r) {
            if (mark[r - S.off] != q) { mark[r - S.off] = q; N.b.push_back(r); }
        };
        for (int32_t r : own[q]) take(r);
        for (int c : N.ch)
            for (int32_t r : T.nodes[c].b) take(r);
        std::sort(N.b.begin(), N.b.end());
        N.cost += (double)N.s.size() * (N.s.size() + 2.0 * N.b.size()) + 64.0;
        if (N.parent >= 0) T.nodes[N.parent].cost += N.cost;
    }
    // the root's subtrees to the CTAs, largest first to the least loaded
    std::vector<int> top = T.nodes[0].ch;
    std::stable_sort(top.begin(), top.end(), [&](int a, int b) { return T.nodes[a].cost > T.nodes[b].cost; });
    std::vector<double> load(1 << p, 0.0);
    for (int c : top) {
        const int r = (int)(std::min_element(load.begin(), load.end()) - load.begin());
        T.nodes[c].rank = r;
        load[r] += T.nodes[c].cost;
    }
    for (size_t q = 1; q < T.nodes.size(); ++q)
        if (T.nodes[q].parent > 0) T.nodes[q].rank = T.nodes[T.nodes[q].parent].rank;
}

int pad4(int v) { return (v + 3) / 4 * 4; }

// Tables of one subdomain, positions within its own arrays; `nodes` in the tree's order, and childs numbered
// in it.  False: an index outgrows its 16 bits.
bool emit_tables(const thm_mesh* m, int sub, SubTree& T, int C, NdHost& H) {
    const int mw = m->maxc / 2;
    const auto& S = m->subs[sub];
    H.C = C;
    H.mw = mw;
    H.welem.assign(1, 0);
    H.nodes.resize(T.nodes.size());
    int64_t fo = 0;                                    // factor offset, in 128 entries
    bool fits = true;
    std::vector<int32_t> place(S.n, -1);               // front index of a local row of the subdomain
    size_t ss = 0, sb = 0;                             // all s, all b
    for (auto& N : T.nodes) {
        H.welem[0] += (int64_t)N.s.size() * (N.s.size() + 2 * N.b.size());
        ss += N.s.size();
        sb += N.b.size();
    }
    const size_t nrow = 2 * ss + sb + (size_t)64 * C * (T.maxdepth + 2);
    H.rowd.reserve(nrow);
    H.rowm.reserve(nrow * mw);
    H.ymap.reserve((ss + 4 * T.nodes.size()) * mw);
    H.idx.reserve(sb + 4 * T.nodes.size() + (size_t)C * (T.maxdepth + 2) * 256);
    H.perm.reserve(ss + 4 * T.nodes.size() + (size_t)C * (T.nodes[0].s.size() + 8));
    H.rows.reserve(ss + sb);
    H.cmap.reserve(sb);
    H.childs.reserve(T.nodes.size());
    const Node& root = T.nodes[0];
    const int sr = (int)root.s.size(), srp = pad4(sr);
    std::vector<std::vector<uint32_t>> rmap(sr);
    std::vector<int32_t> vrow(S.n, -1);                // vector entry of a local row in the CTA at hand
    const int share = (sr + C - 1) / C;
    for (int rk = 0; rk < C; ++rk) {
        NdPart P{};
        P.lev0 = (int32_t)H.levs.size();
        P.slt0 = (int32_t)H.slt.size();
        P.perm0 = (int64_t)H.perm.size();
        P.sroot = sr;
        P.rr0 = std::min(sr, rk * share);
        P.nrr = std::min(sr, (rk + 1) * share) - P.rr0;
        std::vector<std::vector<int>> lv(T.maxdepth + 1);
        for (size_t q = 1; q < T.nodes.size(); ++q)
            if (T.nodes[q].rank == rk) lv[T.nodes[q].depth].push_back((int)q);
        int deepest = 0;
        for (int d = 1; d <= T.maxdepth; ++d)
            if (!lv[d].empty()) deepest = d;
        P.nlev = deepest;
        // vector: root, a zero entry, the levels deepest first
        for (int i = 0; i < srp + 4; ++i) H.perm.push_back(i < sr ? root.s[i] : -1);
        for (int i = 0; i < sr; ++i) vrow[root.s[i] - S.off] = i;
        int vo = srp + 4;
        const int zero = srp;
        for (int d = deepest; d >= 1; --d) {
            std::stable_sort(lv[d].begin(), lv[d].end(), [&](int a, int b) { return T.nodes[a].s.size() > T.nodes[b].s.size(); });
            for (int q : lv[d]) {
                Node& N = T.nodes[q];
                N.vpos = vo;
                for (size_t i = 0; i < N.s.size(); ++i) { vrow[N.s[i] - S.off] = vo + (int)i; H.perm.push_back(N.s[i]); }
                vo += pad4((int)N.s.size());
                while ((int64_t)H.perm.size() - P.perm0 < vo) H.perm.push_back(-1);
            }
        }
        P.nvec = vo;
        H.z.nvec = std::max(H.z.nvec, vo);
        fits = fits && vo < (int)ND_U;
        auto new_slice = [&](int nq) {
            H.slt.push_back(make_int2((int)fo, nq));
            fo += nq;
            fits = fits && fo < (int64_t)INT32_MAX;
        };
        // slices over rows whose column quads are nqs; returns the number of slices
        auto slices = [&](const std::vector<int>& nqs) {
            int n = 0;
            for (size_t i = 0; i < nqs.size(); i += 32, ++n)
                new_slice(*std::max_element(nqs.begin() + i, nqs.begin() + std::min(nqs.size(), i + 32)));
            return n;
        };
        auto share_cols = [&](int nsl, const std::vector<int>& nqs) {
            if (nsl == 0 || nsl * 2 > ND_NW) return 1;
            const int mq = *std::max_element(nqs.begin(), nqs.end());
            return std::max(1, std::min(ND_NW / nsl, mq / 2));
        };
        auto pad_rows = [&](size_t words) {
            while (H.rowd.size() % 32) {
                H.rowd.push_back(ND_NOROW);
                for (size_t w = 0; w < words; ++w) H.rowm.push_back(0xffffffffu);
            }
        };
        // ---- up
        for (int d = deepest; d >= 1; --d) {
            NdLev L{};
            L.depth = d;
            int uo = 0;
            for (int q : lv[d]) { T.nodes[q].upos = uo; uo += (int)T.nodes[q].b.size(); }
            H.z.nu[d & 1] = std::max(H.z.nu[d & 1], uo);
            fits = fits && uo < (int)ND_U;
            L.v0 = lv[d].empty() ? vo : T.nodes[lv[d][0]].vpos;
            int nv = 0;
            for (int q : lv[d]) nv += pad4((int)T.nodes[q].s.size());
            L.nv = nv;
            L.ymap = (int32_t)(H.ymap.size() / mw);
            L.rowf = (int32_t)H.rowd.size();
            L.sltf = (int32_t)H.slt.size() - P.slt0;
            std::vector<int> nqs;
            for (int q : lv[d]) {
                Node& N = T.nodes[q];
                const int sn = (int)N.s.size(), bn = (int)N.b.size();
                std::vector<uint32_t> map((size_t)(pad4(sn) + bn) * 2 * mw, ND_NONE);   // s part padded, then b
                std::vector<int> cnt(pad4(sn) + bn, 0);
                for (int i = 0; i < sn; ++i) place[N.s[i] - S.off] = i;
                for (int i = 0; i < bn; ++i) place[N.b[i] - S.off] = pad4(sn) + i;
                for (int c : N.ch) {
                    const Node& K = T.nodes[c];
                    for (size_t i = 0; i < K.b.size(); ++i) {
                        const int at = place[K.b[i] - S.off];
                        if (cnt[at] >= 2 * mw) fail(THM_EINVAL, "internal: too many subtrees share an unknown");
                        map[(size_t)at * 2 * mw + cnt[at]++] = (uint32_t)(K.upos + i);
                    }
                }
                auto words = [&](int at, std::vector<uint32_t>& to) {
                    for (int w = 0; w < mw; ++w)
                        to.push_back((map[(size_t)at * 2 * mw + 2 * w] & 0xffffu) | map[(size_t)at * 2 * mw + 2 * w + 1] << 16);
                };
                for (int i = 0; i < pad4(sn); ++i) words(i, H.ymap);
                N.row_f = (int)H.rowd.size() - L.rowf;
                N.slt_f = P.slt0 + L.sltf;
                for (int i = 0; i < sn + bn; ++i) {
                    const uint32_t dst = i < sn ? (uint32_t)(N.vpos + i) : (ND_U | (uint32_t)(N.upos + i - sn));
                    H.rowd.push_back((uint32_t)(N.vpos - L.v0) | dst << 16);
                    words(i < sn ? i : pad4(sn) + i - sn, H.rowm);
                    nqs.push_back(pad4(sn) / 4);
                }
            }
            pad_rows(mw);
            L.nsf = slices(nqs);
            L.ksf = share_cols(L.nsf, nqs);
            int mq = 0;
            for (int v : nqs) mq = std::max(mq, v);
            H.z.ny = std::max(H.z.ny, nv + 4 * mq);
            H.levs.push_back(L);
        }
        {   // the root's rows of this CTA
            NdLev L{};
            L.nv = sr;
            L.rowf = (int32_t)H.rowd.size();
            L.sltf = (int32_t)H.slt.size() - P.slt0;
            std::vector<int> nqs(P.nrr, srp / 4);
            for (int i = 0; i < P.nrr; ++i) {
                H.rowd.push_back((uint32_t)(P.rr0 + i) << 16);
                for (int w = 0; w < mw; ++w) H.rowm.push_back(0xffffffffu);
            }
            pad_rows(mw);
            L.nsf = slices(nqs);
            L.ksf = share_cols(L.nsf, nqs);
            H.z.ny = std::max(H.z.ny, srp);
            H.levs.push_back(L);
            for (int c : root.ch)
                if (T.nodes[c].rank == rk)
                    for (size_t i = 0; i < T.nodes[c].b.size(); ++i) {
                        const int at = vrow[T.nodes[c].b[i] - S.off];
                        rmap[at].push_back((uint32_t)rk << 16 | (uint32_t)(T.nodes[c].upos + i));
                    }
        }
        // ---- down, nearest the root first (the order the solve streams them in)
        for (int d = 1; d <= deepest; ++d) {
            NdLev& L = H.levs[P.lev0 + deepest - d];
            std::vector<int> order = lv[d];
            std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return T.nodes[a].b.size() > T.nodes[b].b.size(); });
            while (H.idx.size() % 4) H.idx.push_back((uint16_t)zero);
            L.idx = (int32_t)H.idx.size();
            L.rowb = (int32_t)H.rowd.size();
            L.sltb = (int32_t)H.slt.size() - P.slt0;
            std::vector<int> nqs;
            for (int q : order) {
                Node& N = T.nodes[q];
                N.row_b = (int)H.rowd.size() - L.rowb;
                N.slt_b = P.slt0 + L.sltb;
                if (N.b.empty()) continue;
                const size_t i0 = (H.idx.size() - (size_t)L.idx) / 4;
                fits = fits && i0 < 0xffffu;
                for (int32_t r : N.b) H.idx.push_back((uint16_t)vrow[r - S.off]);
                while (H.idx.size() % 4) H.idx.push_back((uint16_t)zero);
                for (size_t i = 0; i < N.s.size(); ++i) {
                    H.rowd.push_back((uint32_t)i0 | (uint32_t)(N.vpos + i) << 16);
                    for (int w = 0; w < mw; ++w) H.rowm.push_back(0xffffffffu);
                    nqs.push_back(pad4((int)N.b.size()) / 4);
                }
            }
            pad_rows(mw);
            L.nsb = slices(nqs);
            L.ksb = share_cols(L.nsb, nqs);
            int mq = 0;
            for (int v : nqs) mq = std::max(mq, v);
            for (int i = 0; i < 4 * mq; ++i) H.idx.push_back((uint16_t)zero);   // narrower rows read on to their slice's width
        }
        P.nslt = (int32_t)H.slt.size() - P.slt0;
        while (H.slt.size() % 2) H.slt.push_back(make_int2(0, 0));
        H.z.nlev = std::max(H.z.nlev, P.nlev);
        H.z.nslt = std::max(H.z.nslt, (P.nslt + 1) / 2 * 2);
        H.parts.push_back(P);
    }
    // root: children's entries per unknown
    const int32_t rm0 = (int32_t)(H.rmap.size() / (2 * mw));
    for (int i = 0; i < sr; ++i) {
        THM_REQUIRE((int)rmap[i].size() <= 2 * mw, "internal: too many subtrees share a root unknown");
        for (int c = 0; c < 2 * mw; ++c) H.rmap.push_back(c < (int)rmap[i].size() ? rmap[i][c] : 0xffffffffu);
    }
    for (int rk = 0; rk < C; ++rk) H.parts[rk].rmap0 = rm0;
    // the factorisation's view
    for (size_t q = 0; q < T.nodes.size(); ++q) {
        Node& N = T.nodes[q];
        NdNode& D = H.nodes[q];
        D.s = (int32_t)N.s.size();
        D.b = (int32_t)N.b.size();
        D.sub = sub;
        D.slt_f = N.slt_f;
        D.slt_b = N.slt_b;
        D.row_f = N.row_f;
        D.row_b = N.row_b;
        D.root_rows = q == 0 ? std::max(1, share) : 0;
        D.rows0 = (int64_t)H.rows.size();
        H.rows.insert(H.rows.end(), N.s.begin(), N.s.end());
        H.rows.insert(H.rows.end(), N.b.begin(), N.b.end());
        D.child0 = (int32_t)H.childs.size();
        D.nchild = (int32_t)N.ch.size();
        for (size_t i = 0; i < N.s.size(); ++i) place[N.s[i] - S.off] = (int32_t)i;
        for (size_t i = 0; i < N.b.size(); ++i) place[N.b[i] - S.off] = (int32_t)(N.s.size() + i);
        for (int c : N.ch) {
            H.childs.push_back((int32_t)c);
            H.nodes[c].cmap0 = (int64_t)H.cmap.size();
            for (int32_t r : T.nodes[c].b) H.cmap.push_back(place[r - S.off]);
        }
    }
    H.fac_elems = fo * 128;
    return fits;
}

// fn(i) for i < n on at most `most` threads; the first exception comes back here.
void parallel(int n, int most, const std::function<void(int)>& fn) {
    const int nt = std::max(1, std::min<int>({most, n, (int)std::thread::hardware_concurrency()}));
    std::atomic<int> next{0};
    std::mutex mu;
    std::exception_ptr err;
    auto work = [&]() {
        try {
            for (int i; (i = next++) < n;) fn(i);
        } catch (...) {
            std::lock_guard<std::mutex> g(mu);
            if (!err) err = std::current_exception();
        }
    };
    std::vector<std::thread> th;
    th.reserve(nt);
    try {
        for (int t = 1; t < nt; ++t) th.emplace_back(work);
    } catch (const std::system_error&) {               // no more threads: those there are do it
    }
    work();
    for (auto& t : th) t.join();
    if (err) std::rethrow_exception(err);
}

}  // namespace

bool place_tables(NdHost& H, const NdPlace& at) {
    const size_t most = INT32_MAX, mw = H.mw;
    if (at.levs + H.levs.size() > most || at.slt + H.slt.size() > most || at.rowd + H.rowd.size() > most ||
        at.idx + H.idx.size() > most || (at.fac + H.fac_elems) / 128 > most)
        return false;
    THM_REQUIRE(at.slt % 2 == 0 && at.idx % 4 == 0 && at.fac % 128 == 0, "internal: tables out of alignment");
    for (NdPart& P : H.parts) {
        P.lev0 += (int32_t)at.levs;
        P.slt0 += (int32_t)at.slt;
        P.rmap0 += (int32_t)(at.rmap / (2 * mw));
        P.perm0 += (int64_t)at.perm;
    }
    for (NdLev& L : H.levs) {
        L.rowf += (int32_t)at.rowd;
        L.rowb += (int32_t)at.rowd;
        L.ymap += (int32_t)(at.ymap / mw);
        L.idx += (int32_t)at.idx;
    }
    for (int2& v : H.slt) v.x += (int)(at.fac / 128);
    for (NdNode& N : H.nodes) { N.slt_f += (int32_t)at.slt; N.slt_b += (int32_t)at.slt; }
    return true;
}

NdSizes larger(NdSizes a, const NdSizes& b) {
    a.nlev = std::max(a.nlev, b.nlev);
    a.nslt = std::max(a.nslt, b.nslt);
    a.nvec = std::max(a.nvec, b.nvec);
    a.ny = std::max(a.ny, b.ny);
    for (int k = 0; k < 2; ++k) a.nu[k] = std::max(a.nu[k], b.nu[k]);
    return a;
}

// Whether an apply, resp. a subdomain solve with m steps per cycle, fits shared
// memory in FP64 (the larger of the two precisions).
static bool apply_fits(const NdSizes& z) {
    NdMem mm{};
    return nd_fit<double2>(z, true, 0, 0, &mm) > 0;
}
static bool solve_fits(const thm_mesh* mesh, const NdSizes& z, int C, int m) {
    NdMem mm{};
    int64_t n = 0;
    for (const auto& S : mesh->subs) n = std::max(n, S.n);
    return nd_fit<double2>(z, true, sub_krylov_bytes<double2>(sub_rows(n, C), m, 1), sub_keep_bytes(m), &mm) > 0;
}

bool build_tables(const thm_mesh* m, NdHost& H, const std::vector<int>& list, int p,
                  const std::vector<std::vector<NdMove>>* moves) {
    const int ns = (int)list.size(), C = 1 << p, mw = m->maxc / 2;
    H = NdHost();
    std::vector<std::vector<int32_t>> cells(ns);
    {
        std::vector<int32_t> at(m->n_sub, -1);
        for (int i = 0; i < ns; ++i) at[list[i]] = i;
        for (int64_t c = 0; c < m->n_cell; ++c)
            if (at[m->cell_sub[c]] >= 0) cells[at[m->cell_sub[c]]].push_back((int32_t)c);
    }
    H.C = C;
    H.mw = mw;
    size_t nc = 0;
    for (const auto& c : cells) nc += c.size();
    const bool big = nc >= 8192;                          // (threads cost: 1 ms for 15 of them three times)
    std::vector<SubTree> trees(ns);
    std::vector<int32_t> cell_bin(m->n_cell, -1);         // cells belong to one subdomain each: no sharing
    std::vector<NdHost> part(ns);
    std::vector<char> ok(ns, 0);
    parallel(ns, big ? 16 : 8, [&](int i) {
        build_tree(m, list[i], std::move(cells[i]), p, moves ? &(*moves)[list[i]] : nullptr, cell_bin, trees[i]);
        ok[i] = emit_tables(m, list[i], trees[i], C, part[i]);
    });
    // node numbers: by depth, deepest first
    int maxd = 0;
    for (const auto& T : trees) maxd = std::max(maxd, T.maxdepth);
    std::vector<std::vector<std::pair<int, int>>> by(maxd + 1);
    for (int s = 0; s < ns; ++s)
        for (size_t q = 0; q < trees[s].nodes.size(); ++q) by[trees[s].nodes[q].depth].emplace_back(s, (int)q);
    int64_t id = 0;
    H.depth_node.assign(1, 0);
    for (int d = maxd; d >= 0; --d) {
        int64_t front = 0;
        int ms = 0, mn = 0;
        for (auto& e : by[d]) {
            Node& N = trees[e.first].nodes[e.second];
            N.id = id++;
            H.node_ref.push_back({list[e.first], e.second, N.parent});
            const int64_t n = (int64_t)(N.s.size() + N.b.size());
            N.front = front;
            front += n * n;
            ms = std::max(ms, (int)N.s.size());
            mn = std::max(mn, (int)n);
        }
        H.depth_node.push_back(id);
        H.depth_front.push_back(front);
        H.depth_s.push_back(ms);
        H.depth_n.push_back(mn);
    }
    // the subdomains' tables one behind the other
    std::vector<NdPlace> at(ns + 1);
    std::vector<size_t> rows0(ns + 1, 0), cmap0(ns + 1, 0), child0(ns + 1, 0);
    bool fits = true;
    NdPlace end{};
    for (int i = 0; i < ns; ++i) {
        const NdHost& P = part[i];
        at[i] = end;
        end = NdPlace{end.levs + P.levs.size(), end.slt + P.slt.size(), end.rowd + P.rowd.size(), end.ymap + P.ymap.size(),
                      end.rmap + P.rmap.size(), end.idx + P.idx.size(), end.perm + P.perm.size(), end.fac + P.fac_elems};
        rows0[i + 1] = rows0[i] + P.rows.size();
        cmap0[i + 1] = cmap0[i] + P.cmap.size();
        child0[i + 1] = child0[i] + P.childs.size();
        H.z = larger(H.z, P.z);
        fits = fits && ok[i];
    }
    if (!fits || child0[ns] > INT32_MAX || !apply_fits(H.z)) return false;
    H.parts.resize((size_t)ns * C);
    H.welem.resize(ns);
    H.levs.resize(end.levs); H.slt.resize(end.slt);
    H.rowd.resize(end.rowd); H.rowm.resize(end.rowd * mw);
    H.ymap.resize(end.ymap); H.rmap.resize(end.rmap); H.perm.resize(end.perm);
    H.idx.assign(end.idx + 64, 0);                     // (a lane reads whole quads)
    H.nodes.resize(id);
    H.rows.resize(rows0[ns]); H.cmap.resize(cmap0[ns]); H.childs.resize(child0[ns]);
    H.fac_elems = (int64_t)end.fac + 128;
    parallel(ns, big ? 16 : 1, [&](int i) {
        NdHost& P = part[i];
        ok[i] = place_tables(P, at[i]);
        std::copy(P.parts.begin(), P.parts.end(), H.parts.begin() + (size_t)i * C);
        H.welem[i] = P.welem[0];
        std::copy(P.levs.begin(), P.levs.end(), H.levs.begin() + at[i].levs);
        std::copy(P.slt.begin(), P.slt.end(), H.slt.begin() + at[i].slt);
        std::copy(P.rowd.begin(), P.rowd.end(), H.rowd.begin() + at[i].rowd);
        std::copy(P.rowm.begin(), P.rowm.end(), H.rowm.begin() + at[i].rowd * mw);
        std::copy(P.ymap.begin(), P.ymap.end(), H.ymap.begin() + at[i].ymap);
        std::copy(P.rmap.begin(), P.rmap.end(), H.rmap.begin() + at[i].rmap);
        std::copy(P.idx.begin(), P.idx.end(), H.idx.begin() + at[i].idx);
        std::copy(P.perm.begin(), P.perm.end(), H.perm.begin() + at[i].perm);
        std::copy(P.rows.begin(), P.rows.end(), H.rows.begin() + rows0[i]);
        std::copy(P.cmap.begin(), P.cmap.end(), H.cmap.begin() + cmap0[i]);
        std::transform(P.childs.begin(), P.childs.end(), H.childs.begin() + child0[i],
                       [&](int32_t q) { return (int32_t)trees[i].nodes[q].id; });
        for (size_t q = 0; q < P.nodes.size(); ++q) {
            NdNode N = P.nodes[q];
            N.rows0 += (int64_t)rows0[i];
            N.cmap0 += (int64_t)cmap0[i];
            N.child0 += (int32_t)child0[i];
            N.front = trees[i].nodes[q].front;
            H.nodes[trees[i].nodes[q].id] = N;
        }
        P = NdHost();
    });
    for (char o : ok) fits = fits && o;
    return fits;
}

void build_nd(thm_mesh* m) {
    const int ns = m->n_sub;
    std::vector<int> all(ns);
    std::iota(all.begin(), all.end(), 0);
    int dev = 0, sms = 0;
    THM_CUDA(cudaGetDevice(&dev));
    THM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    // CTAs per subdomain: as many as keep two on every SM busy, but not so
    // many that a CTA has less than a warp pass of unknowns
    int p = 0;
    while (p < 3 && (int64_t)ns * (2 << p) <= 2 * (int64_t)sms && m->n_loc / ns >= (int64_t)(64 << (p + 1))) ++p;
    // ... and more where a CTA's shared memory is too small for a solve of the
    // default restart length (40x40 order-2 cells: 246 KB with one CTA, 131 KB
    // with two, of 226)
    int applies = -1;                                      // an apply fits, at least
    for (;; ++p) {
        m->nd_ok = build_tables(m, m->nd, all, p, nullptr);
        if (m->nd_ok) applies = p;
        if (p == 3 || (m->nd_ok && solve_fits(m, m->nd.z, 1 << p, ND_RESTART))) break;
    }
    if (!m->nd_ok && applies >= 0) m->nd_ok = build_tables(m, m->nd, all, applies, nullptr);
    if (!m->nd_ok) return;                                 // reported by the first apply, as a size limit of the kernel
    auto& H = m->nd;
    auto& D = m->ndd;
    D.parts.upload(H.parts);
    D.levs.upload(H.levs);
    D.slt.upload(H.slt);
    D.rowd.upload(H.rowd);
    D.rowm.upload(H.rowm);
    D.ymap.upload(H.ymap);
    D.rmap.upload(H.rmap);
    D.idx.upload(H.idx);
    D.perm.upload(H.perm);
    D.welem.upload(H.welem);
    D.nodes.upload(H.nodes);
    D.rows.upload(H.rows);
    D.cmap.upload(H.cmap);
    D.childs.upload(H.childs);
}

}  // namespace thm
