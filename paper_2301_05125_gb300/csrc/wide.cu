// wide.cu -- 4-wide BVH of the static part of the scene, collapsed on the
// device from the binary PLOC tree (sm_103a).
//
// Each wide node holds up to four children: a cut of its binary subtree into
// at most four nodes.  A binary node over two triangles that share an edge is
// kept whole as one leaf (a quad: one box test for both, four vertices to
// fetch and transform instead of six).  The cuts minimise the surface-area
// cost of the whole wide tree (below), found bottom up by dynamic programming
// over the binary tree.  The child boxes are the binary tree's own boxes
// (already enlarged by the builder), so every triangle stays inside every box
// on its path and a traversal finds exactly the hits the binary tree finds.
//
// Node layout (7 x 16 bytes, children in slots 0..3, internal ones first):
//   [0] lo.x of the four children   [1] hi.x
//   [2] lo.y                        [3] hi.y
//   [4] lo.z                        [5] hi.z
//   [6] int32: first child node (the internal children are consecutive),
//       first leaf record (so are the leaves), number of internal children
// Leaf record (4 x 16 bytes): four vertices, see trav_leaf.
// An empty slot has the box [+inf, -inf]: whatever the ray direction, its
// entry distance is +inf, so it reports no hit (but see kWideSpare for rays
// that are not finite).  A traversal reads the
// near and far plane arrays of each axis by the sign of the ray direction
// (lo is near for a positive direction), so it needs no per-child min / max.
//
// Two passes: k_wide_plan walks up from the leaves (the second thread to
// reach a node plans it) and leaves each node's best cuts and the size of the
// wide subtree made at it; k_wide_emit, one launch a level, places every wide
// node from its parent's place and those sizes, so the layout (a node's
// children together, then the children's subtrees in order) does not depend
// on the order of the threads.  (On the host this took a copy of the tree
// there and back and 60 ms at 198k triangles, 0.5 s at 2M.)
#include <algorithm>

#include "adgi_internal.cuh"
#include "bvh.cuh"
#include "kernels.cuh"

namespace adgi {

// What the plan says of binary node v: the least cost of covering its subtree
// with 1, 2 or 3 slots of the wide node above it, and the wide nodes (the
// levels of wide nodes in `levels`, eight bits each) and leaf records which
// that cover makes.  own: the same for the wide node made at v, its own
// excluded.
// word: bits 0-1 the split a at budget 2 (0: v whole), 2-3 at budget 3, 4-5
// that of v's own wide node, 6: v whole is a leaf of two triangles, 8-9 and
// 10-11 the rotations of the two.
struct __align__(16) WidePlan {
    float cost[3];
    uint32_t word;
    int nodes[3];
    int leaves[3];
    uint32_t levels;
    int own_nodes, own_leaves, own_levels, pad[2];
};
static_assert(sizeof(WidePlan) == 64, "read as four float4");

namespace {

// Surface-area cost of a wide tree: a ray enters a box with a chance in
// proportion to its surface area, a visit of a wide node costs kCostNode and
// a triangle test kCostTri (kCostPair for two that share an edge).  A wide
// node made at binary node u costs kCostNode A(u) plus the cost of its
// children; a leaf costs its test times its own box's area.  The weights are
// lane operations of the traversal: a visit tests four boxes (13 each) and
// spends about 20 more on ordering the hits and on the stack; a watertight
// triangle test takes 55.
constexpr float kCostNode = 72.0f, kCostTri = 55.0f, kCostPair = 80.0f;

// The dynamic programme.  For binary node v and a budget of k slots (1..4):
//   F(v, k) = least cost of covering v's subtree with at most k children of
//             the wide node above it;
//   F(v, 1) = cost of v as one child (a wide node of its own made at v, or a
//             leaf of two triangles);
//   F(v, k) = min(F(v, 1), min over a of F(l, a) + F(r, k - a)), k >= 2,
// where l, r are v's binary children (a triangle costs the same in any
// budget).  The wide node made at v takes the best cut of v into four:
//   S(v) = min over a in 1..3 of F(l, a) + F(r, 4 - a).
__device__ __forceinline__ int split_of(uint32_t word, int k) { return k < 2 ? 0 : (int)(word >> (2 * (k - 2))) & 3; }
__device__ __forceinline__ bool pair_leaf(uint32_t word) { return (word >> 6) & 1u; }

struct Child {
    int ref;  // >= 0 a binary node, < 0 ~(triangle slot)
    float3 lo, hi;
};

__device__ __forceinline__ void children_of(const BNode* bn, int v, Child c[2])
{
    const float4 a = bn[v].a, b = bn[v].b, d = bn[v].c;
    const int4 r = bn[v].d;
    c[0] = Child{r.x, make_float3(a.x, a.y, a.z), make_float3(a.w, b.x, b.y)};
    c[1] = Child{r.y, make_float3(b.z, b.w, d.x), make_float3(d.y, d.z, d.w)};
}

__device__ __forceinline__ float area(float3 lo, float3 hi)
{
    const float x = hi.x - lo.x, y = hi.y - lo.y, z = hi.z - lo.z;
    return x * y + y * z + z * x;
}

__device__ __forceinline__ bool same_vertex(float4 a, float4 b)
{
    return __float_as_uint(a.x) == __float_as_uint(b.x) && __float_as_uint(a.y) == __float_as_uint(b.y) &&
           __float_as_uint(a.z) == __float_as_uint(b.z);
}

// The triangles at slots s1 and s2 share an edge in opposite directions: the
// rotations r1, r2 such that they are (v0, v1, v2) and (v0, v2, v3) when
// vertex j of a rotated triangle is vertex (j + r) % 3 of the original.
__device__ __forceinline__ bool pair_of(const float4* __restrict__ tri, int s1, int s2, int& r1, int& r2)
{
    const float4 A[3] = {tri[3 * (size_t)s1], tri[3 * (size_t)s1 + 1], tri[3 * (size_t)s1 + 2]};
    const float4 B[3] = {tri[3 * (size_t)s2], tri[3 * (size_t)s2 + 1], tri[3 * (size_t)s2 + 2]};
    bool found = false;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)  // v0 = vertex i = vertex j, v2 = vertex i + 2 = vertex j + 1
            if (!found && same_vertex(A[i], B[j]) && same_vertex(A[(i + 2) % 3], B[(j + 1) % 3])) {
                r1 = i;
                r2 = j;
                found = true;
            }
    return found;
}

__device__ __forceinline__ WidePlan load_plan(const WidePlan* p)  // written by other threads of the launch
{
    WidePlan r;
    float4* d = reinterpret_cast<float4*>(&r);
    const float4* s = reinterpret_cast<const float4*>(p);
#pragma unroll
    for (int k = 0; k < 4; ++k) d[k] = __ldcg(s + k);
    return r;
}

// a triangle as a slot: the same for any budget
__device__ __forceinline__ WidePlan tri_plan(const Child& c)
{
    WidePlan r{};
    for (int k = 0; k < 3; ++k) {
        r.cost[k] = kCostTri * area(c.lo, c.hi);
        r.leaves[k] = 1;
    }
    return r;
}

// thread i: up from triangle slot i
__global__ void k_wide_plan(const BNode* __restrict__ bn, const float4* __restrict__ tri, int ns,
                            const int* __restrict__ par_int, const int* __restrict__ par_leaf, WideBufs W)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ns) return;
    int v = par_leaf[i];
    for (int step = 0; step < 4096; ++step) {
        __threadfence();
        if (atomicAdd(W.flags + v, 1) == 0) return;  // the sibling's subtree is not planned yet
        __threadfence();
        Child c[2];
        children_of(bn, v, c);
        const float A = area(make_float3(fminf(c[0].lo.x, c[1].lo.x), fminf(c[0].lo.y, c[1].lo.y), fminf(c[0].lo.z, c[1].lo.z)),
                             make_float3(fmaxf(c[0].hi.x, c[1].hi.x), fmaxf(c[0].hi.y, c[1].hi.y), fmaxf(c[0].hi.z, c[1].hi.z)));
        const WidePlan l = c[0].ref < 0 ? tri_plan(c[0]) : load_plan(W.plan + c[0].ref);
        const WidePlan r = c[1].ref < 0 ? tri_plan(c[1]) : load_plan(W.plan + c[1].ref);
        WidePlan p{};
        // the wide node made here: the best cut into four
        float best = l.cost[0] + r.cost[2];
        int a4 = 1;
        if (l.cost[1] + r.cost[1] < best) best = l.cost[1] + r.cost[1], a4 = 2;
        if (l.cost[2] + r.cost[0] < best) best = l.cost[2] + r.cost[0], a4 = 3;
        auto pick = [](const int* x, int k) { return k == 1 ? x[0] : k == 2 ? x[1] : x[2]; };
        auto lev = [](uint32_t x, int k) { return (int)(x >> (8 * (k - 1))) & 255; };
        p.own_nodes = pick(l.nodes, a4) + pick(r.nodes, 4 - a4);
        p.own_leaves = pick(l.leaves, a4) + pick(r.leaves, 4 - a4);
        p.own_levels = min(255, 1 + max(lev(l.levels, a4), lev(r.levels, 4 - a4)));
        // covered by one slot: that node, or a leaf of two triangles
        int r1 = 0, r2 = 0;
        const float whole = kCostNode * A + best;
        const bool pair = c[0].ref < 0 && c[1].ref < 0 && kCostPair * A < whole && pair_of(tri, ~c[0].ref, ~c[1].ref, r1, r2);
        p.word = (uint32_t)a4 << 4 | (pair ? 64u : 0u) | (uint32_t)r1 << 8 | (uint32_t)r2 << 10;
        p.cost[0] = pair ? kCostPair * A : whole;
        p.nodes[0] = pair ? 0 : 1 + p.own_nodes;
        p.leaves[0] = pair ? 1 : p.own_leaves;
        p.levels = pair ? 0u : (uint32_t)p.own_levels;
        // by two or three
        const float c2 = l.cost[0] + r.cost[0];
        const float c3 = fminf(l.cost[0] + r.cost[1], l.cost[1] + r.cost[0]);
        const int a3 = l.cost[0] + r.cost[1] <= c3 ? 1 : 2;
#pragma unroll
        for (int k = 2; k <= 3; ++k) {
            const float s = k == 2 ? c2 : c3;
            const int a = k == 2 ? 1 : a3;
            const bool split = s < p.cost[0];
            if (split) p.word |= (uint32_t)a << (2 * (k - 2));
            p.cost[k - 1] = split ? s : p.cost[0];
            p.nodes[k - 1] = split ? pick(l.nodes, a) + pick(r.nodes, k - a) : p.nodes[0];
            p.leaves[k - 1] = split ? pick(l.leaves, a) + pick(r.leaves, k - a) : p.leaves[0];
            p.levels |= (uint32_t)(split ? max(lev(l.levels, a), lev(r.levels, k - a)) : (int)(p.levels & 255u)) << (8 * (k - 1));
        }
        float4* d = reinterpret_cast<float4*>(W.plan + v);
        const float4* q = reinterpret_cast<const float4*>(&p);
#pragma unroll
        for (int k = 0; k < 4; ++k) __stcg(d + k, q[k]);
        if (v == 0) return;
        v = par_int[v];
    }
}

// The slots of the wide node made at v, in cut order, with the plan words of
// the binary nodes among them; returns how many.
__device__ __forceinline__ int cut_of(const BNode* __restrict__ bn, const WidePlan* __restrict__ plan, int v,
                                      Child out[4], uint32_t word[4])
{
    Child st[4], two[2];
    int sk[4], sp = 0, n = 0;
    children_of(bn, v, two);
    const int a = split_of(plan[v].word, 4);
    st[sp] = two[1], sk[sp++] = 4 - a;
    st[sp] = two[0], sk[sp++] = a;
    while (sp > 0) {
        const Child c = st[--sp];
        const int k = sk[sp];
        const uint32_t w = c.ref < 0 ? 0u : plan[c.ref].word;
        const int s = c.ref < 0 ? 0 : split_of(w, k);
        if (s == 0) {
            word[n] = w;
            out[n++] = c;
            continue;
        }
        children_of(bn, c.ref, two);
        st[sp] = two[1], sk[sp++] = k - s;
        st[sp] = two[0], sk[sp++] = s;
    }
    return n;
}

// Level `level`: its wide nodes from queue[level & 1] ({binary node, wide
// node, first node and first leaf record of its subtree}), the next level's
// into the other.  Four lanes a node, one a slot.
__global__ void __launch_bounds__(128) k_wide_emit(const BNode* __restrict__ bn, const float4* __restrict__ tri, WideBufs W,
                                                   int level, float4* __restrict__ out, float4* __restrict__ rec)
{
    const int4* __restrict__ q = W.queue[level & 1];
    int4* __restrict__ q2 = W.queue[(level & 1) ^ 1];
    const int items = level == 0 ? 1 : W.count[level];
    const int lane = threadIdx.x & 31, k = lane & 3;
    const int per = gridDim.x * blockDim.x / 4, rounds = (items + per - 1) / per;  // the same for every lane
    for (int rd = 0; rd < rounds; ++rd) {
        const int t = rd * per + (int)(blockIdx.x * blockDim.x + threadIdx.x) / 4;
        const bool on = t < items;
        const int4 it = level == 0 || !on ? make_int4(0, 0, 1, 0) : q[t];
        Child c[4];
        uint32_t word[4];
        const int n = cut_of(bn, W.plan, it.x, c, word);
        // the slot order: internal children first, both kinds in cut order
        int ni = 0;
#pragma unroll
        for (int m = 0; m < 4; ++m) ni += m < n && c[m].ref >= 0 && !pair_leaf(word[m]) ? 1 : 0;
        Child x = c[0];
        uint32_t xw = word[0];
        int in = 0, lf = ni;
#pragma unroll
        for (int m = 0; m < 4; ++m)
            if (m < n) {
                const int at = c[m].ref >= 0 && !pair_leaf(word[m]) ? in++ : lf++;
                if (at == k) x = c[m], xw = word[m];
            }
        // the children's subtrees follow one another
        int nodes = 0, leaves = 0;
        if (k < ni) nodes = W.plan[x.ref].own_nodes, leaves = W.plan[x.ref].own_leaves;
        int nb = nodes, lb = leaves;
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            const int a = __shfl_up_sync(0xFFFFFFFFu, nb, o, 4), b = __shfl_up_sync(0xFFFFFFFFu, lb, o, 4);
            if (k >= o) nb += a, lb += b;
        }
        int first = 0;
        if (k == 0 && on && ni > 0) first = atomicAdd(W.count + level + 1, ni);
        first = __shfl_sync(0xFFFFFFFFu, first, 0, 4);
        if (!on) continue;
        float* box = reinterpret_cast<float*>(out + 7 * (size_t)it.y);
        const float inf = __int_as_float(0x7F800000);
        box[k] = k < n ? x.lo.x : inf;
        box[4 + k] = k < n ? x.hi.x : -inf;
        box[8 + k] = k < n ? x.lo.y : inf;
        box[12 + k] = k < n ? x.hi.y : -inf;
        box[16 + k] = k < n ? x.lo.z : inf;
        box[20 + k] = k < n ? x.hi.z : -inf;
        if (k == 0) reinterpret_cast<int4*>(out)[7 * (size_t)it.y + 6] = make_int4(it.z, it.w, ni, 0);
        if (k < ni) {
            q2[first + k] = make_int4(x.ref, it.z + k, it.z + ni + nb - nodes, it.w + (n - ni) + lb - leaves);
        } else if (k < n) {
            int s1 = ~x.ref, s2 = -1, r1 = 0, r2 = 0;
            if (x.ref >= 0) {
                const int4 ch = bn[x.ref].d;
                s1 = ~ch.x, s2 = ~ch.y;
                r1 = (int)(xw >> 8) & 3, r2 = (int)(xw >> 10) & 3;
            }
            float4 v[4];
            for (int j = 0; j < 3; ++j) v[j] = tri[3 * (size_t)s1 + (j + r1) % 3];
            if (s2 >= 0)
                v[3] = tri[3 * (size_t)s2 + (2 + r2) % 3];
            else  // no second triangle: the parallelogram's, whose test is cheap (v3 = v2 would always have a zero edge)
                v[3] = make_float4(v[0].x + (v[2].x - v[1].x), v[0].y + (v[2].y - v[1].y), v[0].z + (v[2].z - v[1].z), 0.f);
            // a triangle rotated by r is brought back to its own order by 3 - r more
            v[0].w = tri[3 * (size_t)s1].w;
            v[1].w = __int_as_float((3 - r1) % 3);
            v[2].w = s2 >= 0 ? tri[3 * (size_t)s2].w : __int_as_float(-1);
            v[3].w = __int_as_float((3 - r2) % 3);
            float4* dst = rec + 4 * (size_t)(it.w + (k - ni));
            for (int j = 0; j < 4; ++j) dst[j] = v[j];
        }
    }
}

}  // namespace

// Carve the collapse's scratch for ns triangles out of one block (base may be
// null to only compute the size).
size_t carve_wide_scratch(void* base, int ns, WideBufs& W)
{
    const size_t n = (size_t)(ns > 0 ? ns : 1);
    size_t off = 0;
    auto take = [&](size_t bytes) -> void* {
        void* p = base ? (void*)((char*)base + off) : nullptr;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    W.plan = (WidePlan*)take(sizeof(WidePlan) * n);
    W.flags = (int*)take(sizeof(int) * n);
    for (int k = 0; k < 2; ++k) W.queue[k] = (int4*)take(sizeof(int4) * n);
    W.count = (int*)take(sizeof(int) * (kWide4Stack / 3 + 2));
    return off;
}

// The cuts of the binary tree of ns triangles; *sizes: its wide nodes, leaf
// records and levels (synchronises the stream).
cudaError_t plan_wide4(const BvhBufs& B, const WideBufs& W, int ns, int sizes[3], cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(W.flags, 0, sizeof(int) * (size_t)ns, s);
    if (e != cudaSuccess) return e;
    k_wide_plan<<<(ns + 127) / 128, 128, 0, s>>>(B.nodes, B.tri_v, ns, B.par_int, B.par_leaf, W);
    count_launches(1);
    WidePlan root{};
    e = cudaMemcpyAsync(&root, W.plan, sizeof(root), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    sizes[0] = root.own_nodes + 1;
    sizes[1] = root.own_leaves;
    sizes[2] = root.own_levels;
    return e;
}

// Write the planned tree (sizes as planned, at most kWide4Stack / 3 levels)
// and the spare records after its leaves.
cudaError_t emit_wide4(const BvhBufs& B, const WideBufs& W, const int sizes[3], float4* nodes, float4* leaves, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(W.count, 0, sizeof(int) * (kWide4Stack / 3 + 2), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(leaves + 4 * (size_t)sizes[1], 0, 4 * sizeof(float4) * kWideSpare, s);
    for (int l = 0; l < sizes[2] && e == cudaSuccess; ++l) {
        // a level has at most 4^l nodes; a grid of 152 x 8 blocks covers the large ones in a loop
        const int blocks = l < 8 ? std::max(1, (1 << (2 * l)) / 32) : 152 * 8;
        k_wide_emit<<<blocks, 128, 0, s>>>(B.nodes, B.tri_v, W, l, nodes, leaves);
        count_launches(1);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace adgi
