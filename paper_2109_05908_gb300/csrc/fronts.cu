// Substructuring plan of a sparse symmetric positive definite matrix (host
// code): a nested dissection of its graph, cut into stages, so that the exact
// solve with the matrix becomes a few rounds of independent dense products.
//
// The graph's vertices carry weights (a vertex stands for that many
// unknowns, all coupled to each other and to every unknown of a neighbouring
// vertex).  Level-set separators (George 1973) give a tree of vertex sets;
// a subtree of at most T_0 unknowns is one part of stage 0; what remains of a
// subtree of at most T_1 > T_0 unknowns after its stage-0 parts is one part of
// stage 1, and so on, the last stage taking what remains of each connected
// component.  Parts of one stage are not coupled to each other once the
// earlier stages are eliminated, and a part is coupled to its boundary, the
// unknowns of later stages next to its subtree.
#include <algorithm>
#include <cmath>
#include <limits>
#include <utility>

#include "fronts.h"

namespace amdd {
namespace {

struct Node {
    std::vector<int32_t> verts;  // separator, or the whole set of a leaf
    std::vector<int> kids;
    int64_t w = 0, subw = 0;
    int parent = -1, stage = 0;
};

struct Cutter {
    const std::vector<int32_t>& ptr;
    const std::vector<int32_t>& adj;
    const std::vector<int32_t>& wt;
    int64_t leaf;
    std::vector<int> tag, level;
    std::vector<Node> nodes;
    int next_tag = 1;

    Cutter(const std::vector<int32_t>& p, const std::vector<int32_t>& a, const std::vector<int32_t>& w, int64_t lf)
        : ptr(p), adj(a), wt(w), leaf(lf), tag(w.size(), 0), level(w.size(), -1) {}

    // breadth-first order of the set tagged t from s; levels in `level`
    void bfs(int32_t s, int t, std::vector<int32_t>& q) {
        q.clear();
        q.push_back(s);
        level[s] = 0;
        for (size_t h = 0; h < q.size(); ++h) {
            const int32_t v = q[h];
            for (int32_t k = ptr[v]; k < ptr[v + 1]; ++k) {
                const int32_t u = adj[k];
                if (tag[u] == t && level[u] < 0) {
                    level[u] = level[v] + 1;
                    q.push_back(u);
                }
            }
        }
    }
    int64_t weight(const std::vector<int32_t>& vs) const {
        int64_t s = 0;
        for (int32_t v : vs) s += wt[v];
        return s;
    }
    int add(std::vector<int32_t> verts, const std::vector<int>& kids) {
        const int id = (int)nodes.size();
        Node nd;
        nd.w = weight(verts);
        nd.verts = std::move(verts);
        nd.kids = kids;
        nd.subw = nd.w;
        for (int k : kids) {
            nd.subw += nodes[k].subw;
            nodes[k].parent = id;
        }
        nodes.push_back(std::move(nd));
        return id;
    }

    // trees of the set tagged t (one for each connected component; small
    // components are taken together when `pack`)
    std::vector<int> run(const std::vector<int32_t>& set, int t, bool pack) {
        std::vector<int> roots;
        if (set.empty()) return roots;
        std::vector<std::vector<int32_t>> comps;
        for (int32_t v : set)
            if (level[v] < 0) {
                comps.emplace_back();
                bfs(v, t, comps.back());
            }
        for (int32_t v : set) level[v] = -1;
        std::vector<int32_t> bag;
        int64_t bagw = 0;
        for (auto& c : comps) {
            const int64_t w = weight(c);
            if (pack && comps.size() > 1 && 2 * w <= leaf) {
                if (bagw + w > leaf && !bag.empty()) {
                    roots.push_back(add(std::move(bag), {}));
                    bag.clear();
                    bagw = 0;
                }
                bag.insert(bag.end(), c.begin(), c.end());
                bagw += w;
                continue;
            }
            const int tc = next_tag++;
            for (int32_t v : c) tag[v] = tc;
            roots.push_back(cut(c, tc, w));
        }
        if (!bag.empty()) roots.push_back(add(std::move(bag), {}));
        return roots;
    }

    // the tree of a connected set tagged t, given in breadth-first order
    int cut(const std::vector<int32_t>& set, int t, int64_t w) {
        if (w <= leaf || set.size() < 3) return add(set, {});
        // levels from a pseudo-peripheral vertex: the last vertex of a search
        // from the last vertex of a search
        std::vector<int32_t> q;
        bfs(set.back(), t, q);
        const int32_t far = q.back();
        for (int32_t v : q) level[v] = -1;
        bfs(far, t, q);
        const int nlev = level[q.back()] + 1;
        if (nlev < 3) {
            for (int32_t v : q) level[v] = -1;
            return add(set, {});
        }
        std::vector<int64_t> lw(nlev, 0);
        for (int32_t v : q) lw[level[v]] += wt[v];
        // the lightest level that leaves at least a third of the weight on each
        // side, else the level at the middle
        int best = -1, mid = 1;
        int64_t before = lw[0];
        for (int l = 1; l + 1 < nlev; ++l) {
            const int64_t after = w - before - lw[l];
            if (before < w / 2) mid = l;
            if (3 * before >= w - lw[l] && 3 * after >= w - lw[l] && (best < 0 || lw[l] < lw[best])) best = l;
            before += lw[l];
        }
        if (best < 0) best = mid;
        std::vector<int32_t> a, b, sep;
        for (int32_t v : q) {
            if (level[v] < best)
                a.push_back(v);
            else if (level[v] > best)
                b.push_back(v);
            else {  // a vertex of the level without a neighbour beyond it needs no place in the separator
                bool far = false;
                for (int32_t k = ptr[v]; k < ptr[v + 1] && !far; ++k)
                    far = tag[adj[k]] == t && level[adj[k]] == best + 1;
                (far ? sep : a).push_back(v);
            }
        }
        for (int32_t v : q) level[v] = -1;
        const int ta = next_tag++, tb = next_tag++, ts = next_tag++;
        for (int32_t v : a) tag[v] = ta;
        for (int32_t v : b) tag[v] = tb;
        for (int32_t v : sep) tag[v] = ts;
        std::vector<int> kids = run(a, ta, true);
        const std::vector<int> kb = run(b, tb, true);
        kids.insert(kids.end(), kb.begin(), kb.end());
        return add(std::move(sep), kids);
    }
};

}  // namespace

FrontPlan plan_fronts(const std::vector<int32_t>& ptr, const std::vector<int32_t>& adj,
                      const std::vector<int32_t>& wt, const std::vector<int32_t>& base, int leaf, int ratio) {
    FrontPlan P;
    const int nv = (int)wt.size();
    Cutter C(ptr, adj, wt, leaf);
    std::vector<int32_t> all(nv);
    for (int v = 0; v < nv; ++v) all[v] = v;
    const std::vector<int> roots = C.run(all, 0, false);
    std::vector<Node>& N = C.nodes;  // children before parents

    // stage thresholds: leaf, then geometrically (ratio at most `ratio`) up to a
    // sixth of the largest component, then the components whole
    int64_t largest = 0;
    for (int r : roots) largest = std::max(largest, N[r].subw);
    std::vector<int64_t> T{leaf};
    if (largest > 12 * (int64_t)leaf) {
        const double span = (double)largest / 6.0 / leaf;
        const int q = std::max(1, (int)std::ceil(std::log(span) / std::log((double)ratio) - 1e-9));
        for (int k = 1; k <= q; ++k) T.push_back((int64_t)(leaf * std::pow(span, (double)k / q)));
    }
    T.push_back(std::numeric_limits<int64_t>::max());
    int nst = 0;
    for (Node& x : N) {
        int s = 0;
        while (x.subw > T[s]) ++s;
        x.stage = s;
        nst = std::max(nst, s + 1);
    }
    // parts: a node whose parent is of a later stage (or a root) tops a part;
    // the part holds the nodes of its own stage below it
    std::vector<int> part(N.size(), -1);
    std::vector<std::vector<int>> members;
    std::vector<int> top;
    for (int x = (int)N.size() - 1; x >= 0; --x) {
        const int par = N[x].parent;
        if (par >= 0 && N[par].stage == N[x].stage) {
            part[x] = part[par];
        } else {
            part[x] = (int)members.size();
            members.emplace_back();
            top.push_back(x);
        }
        members[part[x]].push_back(x);
    }
    std::vector<int> order(members.size());
    for (size_t k = 0; k < order.size(); ++k) order[k] = (int)k;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return N[top[a]].stage < N[top[b]].stage; });

    int64_t n = 0;
    for (int32_t w : wt) n += w;
    P.n = n;
    P.perm.reserve(n);
    P.stage_part.assign(nst + 1, 0);
    P.stage_off.assign(nst + 1, 0);
    std::vector<int> slot(members.size());
    std::vector<int64_t> vpos(nv);     // plan position of a vertex's first unknown
    std::vector<int> vpart(nv, -1);    // its part (plan numbering)
    for (size_t k = 0; k < order.size(); ++k) {
        const int q = order[k];
        slot[q] = (int)k;
        Front f;
        f.stage = N[top[q]].stage;
        f.i0 = (int64_t)P.perm.size();
        for (int x : members[q])
            for (int32_t v : N[x].verts) {
                vpos[v] = (int64_t)P.perm.size();
                vpart[v] = (int)k;
                for (int32_t u = 0; u < wt[v]; ++u) P.perm.push_back(base[v] + u);
            }
        f.m = (int)(P.perm.size() - f.i0);
        P.fronts.push_back(f);
        P.stage_part[f.stage + 1] = (int)k + 1;
        P.stage_off[f.stage + 1] = (int64_t)P.perm.size();
    }
    for (int s = 1; s <= nst; ++s) {
        P.stage_part[s] = std::max(P.stage_part[s], P.stage_part[s - 1]);
        P.stage_off[s] = std::max(P.stage_off[s], P.stage_off[s - 1]);
    }
    // boundaries: the later-stage vertices next to the part or on the boundary
    // of one of its children (fronts come in stage order, children first)
    std::vector<std::vector<int32_t>> bv(order.size());  // boundary vertices
    std::vector<int> stamp(nv, -1);
    std::vector<std::vector<int>> kids(order.size());
    for (size_t k = 0; k < order.size(); ++k) {
        const int q = order[k];
        std::vector<int32_t>& b = bv[k];
        auto reach = [&](int32_t u) {
            if (vpart[u] != (int)k && P.fronts[vpart[u]].stage > P.fronts[k].stage && stamp[u] != (int)k) {
                stamp[u] = (int)k;
                b.push_back(u);
            }
        };
        for (int x : members[q])
            for (int32_t v : N[x].verts)
                for (int32_t e = ptr[v]; e < ptr[v + 1]; ++e) reach(adj[e]);
        for (int c : kids[k])
            for (int32_t u : bv[c]) reach(u);
        std::sort(b.begin(), b.end(), [&](int32_t x, int32_t y) { return vpos[x] < vpos[y]; });
        Front& f = P.fronts[k];
        f.b0 = (int64_t)P.bnd.size();
        for (int32_t v : b)
            for (int32_t u = 0; u < wt[v]; ++u) P.bnd.push_back((int32_t)(vpos[v] + u));
        f.nb = (int)((int64_t)P.bnd.size() - f.b0);
        f.parent = f.nb > 0 ? slot[part[N[top[q]].parent]] : -1;
        if (f.parent >= 0) kids[f.parent].push_back((int)k);
    }
    return P;
}

}  // namespace amdd
