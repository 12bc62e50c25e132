// wide.cu -- 4-wide BVH of the static part of the scene, collapsed on the
// host from the binary PLOC tree (sm_103a library, host code).
//
// Each wide node holds up to four children: a cut of its binary subtree into
// at most four nodes.  A binary node over two triangles that share an edge is
// kept whole as one leaf (a quad: one box test for both, four vertices to
// fetch and transform instead of six).  The cuts minimise the surface-area
// cost of the whole wide tree (below), found bottom up by dynamic programming
// over the binary tree.  The child boxes are the binary tree's own boxes
// (already enlarged by the builder), so every triangle stays inside every box
// on its path and a traversal finds exactly the hits the binary tree finds.
//   On the 2M-triangle city 0.70M of the leaves hold two triangles; the tree
// has 0.50M wide nodes instead of 0.68M.  (With the traversal of one
// visit per leaf test: nearest hit on the 198k-triangle scene 1.65 -> 1.50
// ms, shadow rays 1.30 -> 1.20 ms; breadth-first or depth-first node order
// and other cost weights made no difference.)
//
// Node layout (7 x 16 bytes, children in slots 0..3, internal ones first):
//   [0] lo.x of the four children   [1] hi.x
//   [2] lo.y                        [3] hi.y
//   [4] lo.z                        [5] hi.z
//   [6] int32: first child node (the internal children are consecutive),
//       first leaf record (so are the leaves), number of internal children
// Leaf record (4 x 16 bytes): four vertices, see trav_leaf.
// An empty slot has the box [+inf, -inf]: whatever the ray direction, its
// entry distance is +inf, so it never reports a hit.  A traversal reads the
// near and far plane arrays of each axis by the sign of the ray direction
// (lo is near for a positive direction), so it needs no per-child min / max.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <limits>
#include <vector>

#include "bvh.cuh"

namespace adgi {

namespace {

struct Cand {
    int ref;  // >= 0 a binary node, < 0 ~(triangle slot)
    float lo[3], hi[3];
};

inline double area(const Cand& c)
{
    const double dx = (double)c.hi[0] - c.lo[0], dy = (double)c.hi[1] - c.lo[1], dz = (double)c.hi[2] - c.lo[2];
    return dx * dy + dy * dz + dz * dx;
}

inline void children_of(const BNode& n, Cand out[2])
{
    out[0].ref = n.d.x;
    out[0].lo[0] = n.a.x, out[0].lo[1] = n.a.y, out[0].lo[2] = n.a.z;
    out[0].hi[0] = n.a.w, out[0].hi[1] = n.b.x, out[0].hi[2] = n.b.y;
    out[1].ref = n.d.y;
    out[1].lo[0] = n.b.z, out[1].lo[1] = n.b.w, out[1].lo[2] = n.c.x;
    out[1].hi[0] = n.c.y, out[1].hi[1] = n.c.z, out[1].hi[2] = n.c.w;
}

// Surface-area cost of a wide tree: a ray enters a box with a chance in
// proportion to its surface area, a visit of a wide node costs kCostNode and
// a triangle test kCostTri.  A wide node made at binary node u costs
// kCostNode A(u) plus the cost of its children; a triangle child costs
// kCostTri times its own box's area.  The weights are lane operations of the
// traversal: a visit tests four boxes (13 each) and spends about 20 more on
// ordering the hits and on the stack; a watertight triangle test takes 55.
constexpr double kCostNode = 72.0, kCostTri = 55.0, kCostPair = 80.0;

// The dynamic programme.  For binary node v and a budget of k slots (1..4):
//   F(v, k) = least cost of covering v's subtree with at most k children of
//             the wide node above it;
//   F(v, 1) = cost of v as one child (a wide node of its own made at v);
//   F(v, k) = min(F(v, 1), min over a of F(l, a) + F(r, k - a)), k >= 2,
// where l, r are v's binary children (a triangle costs the same in any
// budget).  The wide node made at v takes the best cut of v into four:
//   S(v) = min over a in 1..3 of F(l, a) + F(r, 4 - a).
struct CutPlan {
    std::vector<double> F;         // [4 n]: F(v, k) at 4 v + k - 1 (k = 4 unused)
    std::vector<signed char> cut;  // [4 n]: a of the best split at budget k; 0: keep v whole
    std::vector<char> pair;        // [n]: v kept whole is one leaf of two triangles
};

inline double cost_of(const CutPlan& P, const Cand& c, int k)
{
    return c.ref < 0 ? kCostTri * area(c) : P.F[4 * (size_t)c.ref + (k - 1)];
}

// best split of binary node v (children c) into budget k >= 2
inline double best_split(const CutPlan& P, const Cand c[2], int k, int* a_out)
{
    double best = std::numeric_limits<double>::infinity();
    int arg = 1;
    for (int a = 1; a < k; ++a) {
        const double x = cost_of(P, c[0], a) + cost_of(P, c[1], k - a);
        if (x < best) {
            best = x;
            arg = a;
        }
    }
    *a_out = arg;
    return best;
}

inline bool same_vertex(const float4& a, const float4& b)
{
    return std::memcmp(&a, &b, 3 * sizeof(float)) == 0;
}

// Triangles t1 and t2 (three vertices each) share an edge in opposite
// directions: the rotations r1, r2 such that t1 = (v0, v1, v2) and
// t2 = (v0, v2, v3) when vertex j of the rotated triangle is vertex
// (j + r) % 3 of the original.
bool pair_of(const float4* t1, const float4* t2, int* r1, int* r2)
{
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)  // t1's v0 = vertex i, its v2 = vertex i + 2; t2's v0 = vertex j, v2 = vertex j + 1
            if (same_vertex(t1[i], t2[j]) && same_vertex(t1[(i + 2) % 3], t2[(j + 1) % 3])) {
                *r1 = i;
                *r2 = j;
                return true;
            }
    return false;
}

// Returns false on a malformed tree (a child index out of range or a node
// reached twice).
bool plan_cuts(const BNode* bn, int n, const float4* tri, CutPlan& P)
{
    P.F.assign(4 * (size_t)n, 0.0);
    P.cut.assign(4 * (size_t)n, 0);
    P.pair.assign((size_t)n, 0);
    // a pre-order list; walked backwards it visits children before parents
    std::vector<int> order;
    std::vector<char> seen((size_t)n, 0);
    order.reserve(n);
    std::vector<int> st{0};
    while (!st.empty()) {
        const int v = st.back();
        st.pop_back();
        if (v >= n || seen[v]) return false;
        seen[v] = 1;
        order.push_back(v);
        if (bn[v].d.x >= 0) st.push_back(bn[v].d.x);
        if (bn[v].d.y >= 0) st.push_back(bn[v].d.y);
    }
    for (size_t i = order.size(); i-- > 0;) {
        const int v = order[i];
        Cand c[2];
        children_of(bn[v], c);
        Cand u;
        for (int j = 0; j < 3; ++j) {
            u.lo[j] = std::min(c[0].lo[j], c[1].lo[j]);
            u.hi[j] = std::max(c[0].hi[j], c[1].hi[j]);
        }
        int a4 = 1;
        const double whole = kCostNode * area(u) + best_split(P, c, 4, &a4);
        double* F = &P.F[4 * (size_t)v];
        signed char* cut = &P.cut[4 * (size_t)v];
        int r1, r2;
        const double pair = kCostPair * area(u);
        const bool as_pair = c[0].ref < 0 && c[1].ref < 0 && pair < whole &&
                             pair_of(tri + 3 * (size_t)~c[0].ref, tri + 3 * (size_t)~c[1].ref, &r1, &r2);
        const double one = as_pair ? pair : whole;
        P.pair[v] = as_pair;
        F[0] = one;
        cut[0] = 0;
        for (int k = 2; k <= 3; ++k) {
            int a = 1;
            const double s = best_split(P, c, k, &a);
            F[k - 1] = s < one ? s : one;
            cut[k - 1] = s < one ? (signed char)a : 0;
        }
        F[3] = F[2];  // no child of a wide node gets four slots
        cut[3] = (signed char)a4;  // the split of v's own wide node
    }
    return true;
}

// the slots of budget k that cover c (c an internal node cut at budget k,
// or kept whole)
void emit_cut(const BNode* bn, const CutPlan& P, const Cand& c, int k, Cand* out, int& n_out)
{
    const int a = c.ref < 0 ? 0 : P.cut[4 * (size_t)c.ref + (k - 1)];
    if (a == 0) {
        out[n_out++] = c;
        return;
    }
    Cand two[2];
    children_of(bn[c.ref], two);
    emit_cut(bn, P, two[0], a, out, n_out);
    emit_cut(bn, P, two[1], k - a, out, n_out);
}

}  // namespace

int collapse_wide4(const BNode* bn, int n_bnodes, const float4* tri, std::vector<float4>& out, std::vector<float4>& rec,
                   int* depth_out)
{
    out.clear();
    rec.clear();
    *depth_out = 0;
    if (n_bnodes < 1) return 0;
    CutPlan P;
    if (!plan_cuts(bn, n_bnodes, tri, P)) return -1;
    struct Item {
        int bnode, wnode, depth;
    };
    std::vector<Item> st{{0, 0, 1}};
    int n_wide = 1;
    const float inf = std::numeric_limits<float>::infinity();
    auto bits = [](int x) {
        float f;
        std::memcpy(&f, &x, 4);
        return f;
    };
    out.resize(7);
    while (!st.empty()) {  // depth first
        const Item it = st.back();
        st.pop_back();
        Cand two[2], c[4];
        children_of(bn[it.bnode], two);
        const int a = P.cut[4 * (size_t)it.bnode + 3];
        int n = 0;
        emit_cut(bn, P, two[0], a, c, n);
        emit_cut(bn, P, two[1], 4 - a, c, n);
        // internal children first
        auto inner = [&](const Cand& x) { return x.ref >= 0 && !P.pair[x.ref]; };
        std::stable_sort(c, c + n, [&](const Cand& x, const Cand& y) { return inner(x) && !inner(y); });
        int ni = 0;
        while (ni < n && inner(c[ni])) ++ni;
        const int first = n_wide, leaf0 = (int)(rec.size() / 4);
        n_wide += ni;
        out.resize(7 * (size_t)n_wide);
        float4* box = &out[7 * (size_t)it.wnode];
        for (int k = 0; k < 4; ++k) {
            float* p[6] = {&box[0].x + k, &box[1].x + k, &box[2].x + k, &box[3].x + k, &box[4].x + k, &box[5].x + k};
            for (int j = 0; j < 3; ++j) {
                *p[2 * j] = k < n ? c[k].lo[j] : inf;
                *p[2 * j + 1] = k < n ? c[k].hi[j] : -inf;
            }
        }
        box[6] = make_float4(bits(first), bits(leaf0), bits(ni), bits(0));
        for (int k = ni; k < n; ++k) {
            float4 q[4];
            if (c[k].ref < 0) {
                const float4* t = tri + 3 * (size_t)~c[k].ref;
                for (int j = 0; j < 3; ++j) q[j] = t[j];
                q[3] = t[2];
                q[1].w = bits(0);
                q[2].w = bits(-1);
                q[3].w = bits(0);
            } else {
                const float4* t1 = tri + 3 * (size_t)~bn[c[k].ref].d.x;
                const float4* t2 = tri + 3 * (size_t)~bn[c[k].ref].d.y;
                int r1 = 0, r2 = 0;
                pair_of(t1, t2, &r1, &r2);
                for (int j = 0; j < 3; ++j) q[j] = t1[(j + r1) % 3];
                q[3] = t2[(2 + r2) % 3];
                q[0].w = t1[0].w;
                q[2].w = t2[0].w;
                // a triangle rotated by r is brought back to its own order by 3 - r more
                q[1].w = bits((3 - r1) % 3);
                q[3].w = bits((3 - r2) % 3);
            }
            rec.insert(rec.end(), q, q + 4);
        }
        for (int k = ni - 1; k >= 0; --k) st.push_back({c[k].ref, first + k, it.depth + 1});
        if (it.depth > *depth_out) *depth_out = it.depth;
    }
    return n_wide;
}

}  // namespace adgi
