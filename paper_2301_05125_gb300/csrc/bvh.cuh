// bvh.cuh -- device LBVH owned by a volume (see bvh.cu).
#pragma once
#include <cuda_runtime.h>

#include "adgi_internal.cuh"

namespace adgi {

// Device buffers of one build: the outputs (tri_v, nodes) and the scratch.
struct BvhBufs {
    float4* tri_v = nullptr;     // [3*n] output: BVH order, v0.w = original index
    BNode* nodes = nullptr;      // [n-1] output
    float4* tri_in = nullptr;    // [3*n] scratch: the listed triangles, v0.w = original index
    int* par_int = nullptr;
    int* par_leaf = nullptr;
    int* flags = nullptr;
    uint64_t* keys[2] = {nullptr, nullptr};
    uint32_t* vals[2] = {nullptr, nullptr};
    uint32_t* hist = nullptr;
    uint32_t* bounds = nullptr;
    int* err = nullptr;
};

// extra scratch of the PLOC build
struct PlocBufs {
    int* cid[2] = {nullptr, nullptr};
    float4* blo[2] = {nullptr, nullptr};
    float4* bhi[2] = {nullptr, nullptr};
    int* nn = nullptr;
    uint64_t* flags = nullptr;
    uint64_t* pre = nullptr;
    uint64_t* sums = nullptr;
    uint64_t* total = nullptr;
    void* state = nullptr;  // two PlocState
    int* pos = nullptr;     // position of each listed triangle in Morton order
    int* mate = nullptr;
};

// The radix sort's tile (keys a block sorts at a time), one for all sizes, so
// that scratch cut for n keys also holds any smaller sort.  Stand-alone builds
// with tiles of 1,024 / 2,048 keys, us: 65,536 triangles 186 / 204, 262,144 222
// / 238, 524,288 294 / 299, 700,000 345 / 358, 1,048,576 611 / 602, 2,000,000
// 1,060 / 1,077, 3,000,000 1,455 / 1,445.
constexpr int kRadixTile = 1024;
constexpr size_t radix_tiles(size_t n) { return ((n > 0 ? n : 1) + kRadixTile - 1) / kRadixTile; }
// counters for a sort of n keys: per tile and digit twice, and one total per digit
constexpr size_t radix_hist_entries(size_t n) { return 2 * 256 * radix_tiles(n) + 256; }

// Bytes of the scratch block carve_bvh_scratch() cuts for a linear build of
// nt triangles: the listed triangles (48 B each), parent links and flags
// (3 x 4 B), sort keys (2 x 8 B) and values (2 x 4 B), the radix sort's
// counters, the centroid bounds and the error word, every piece rounded up to
// 256 bytes.
constexpr size_t bvh_r256(size_t b) { return (b + 255) & ~(size_t)255; }
constexpr size_t bvh_scratch_layout_bytes(size_t nt)
{
    const size_t n = nt > 0 ? nt : 1;
    return bvh_r256(48 * n) + 3 * bvh_r256(4 * n) + 2 * bvh_r256(8 * n) + 2 * bvh_r256(4 * n) +
           bvh_r256(4 * radix_hist_entries(n)) + bvh_r256(4 * 8) + bvh_r256(4 * 2);
}

// scratch of the 4-wide collapse (wide.cu)
struct WidePlan;
struct WideBufs {
    WidePlan* plan = nullptr;  // [n] per binary node
    int* flags = nullptr;      // [n]
    int4* queue[2] = {nullptr, nullptr};
    int* count = nullptr;      // nodes of each level
};

// The 4-wide tree of the static part: plan the cuts of the binary tree
// B.nodes (root 0) over the triangles B.tri_v, then write it (7 float4 a node,
// 4 float4 a leaf record).
//   A ray of NaN or infinite components can hit every slot of a node, empty
// ones too, and then tests the records after the node's own, up to two beyond
// (a node has two children at least).  Those are other leaves, where a test
// more changes no hit, or kWideSpare records of zeros after the last, which no
// ray hits: the array has room for them.  (A mask in every visit would cost the
// other rays an instruction.)
constexpr int kWideSpare = 2;
size_t carve_wide_scratch(void* base, int ns, WideBufs& W);
cudaError_t plan_wide4(const BvhBufs& B, const WideBufs& W, int ns, int sizes[3], cudaStream_t s);
cudaError_t emit_wide4(const BvhBufs& B, const WideBufs& W, const int sizes[3], float4* nodes, float4* leaves, cudaStream_t s);

size_t bvh_scratch_bytes(int nt);
cudaError_t scan_exclusive_u32(uint32_t* a, int n, uint32_t* part, cudaStream_t s);
cudaError_t radix_sort_pairs(uint64_t* const keys[2], uint32_t* const vals[2], uint32_t* hist, int n, int bits,
                             cudaStream_t s, int* cur_out);
size_t carve_bvh_scratch(void* base, int nt, BvhBufs& B);
size_t ploc_scratch_bytes(int nt);
size_t carve_ploc_scratch(void* base, int nt, PlocBufs& Q);
// node_off, tri_off: the tree's place in the arrays that its references are
// made for; tri_orig (optional): the listed triangles' vertices in original
// order are written there too
cudaError_t build_lbvh(const BvhBufs& B, const float* d_verts, const int* d_idx, int nv, int nt, float eps, int* err,
                       cudaStream_t s, int* root_leaf, const int* list = nullptr, int node_off = 0, int tri_off = 0,
                       float4* tri_orig = nullptr);
cudaError_t build_ploc(const BvhBufs& B, const PlocBufs& Q, const float* d_verts, const int* d_idx, int nv, int nt,
                       float eps, int* err, cudaStream_t s, int* root_leaf, const int* list = nullptr);
cudaError_t split_static_moving(const int* d_idx, const uint8_t* vmoved, int nt, int nv, const PlocBufs& Q,
                                int* slist, int* dlist, int* ns, int* nd, cudaStream_t s);
cudaError_t fill_tri_orig(const float* d_verts, const int* d_idx, const int* list, int nv, int nt, float4* tri_orig,
                          cudaStream_t s);
// cudaMalloc for a volume's buffers (capi.cu: failures can be injected)
cudaError_t volume_malloc(void** p, size_t bytes);

// A BVH owned by a volume (static part: PLOC; moving part: linear BVH).
struct Bvh {
    int n_tris = 0;
    int root_leaf = -1;
    float4* tri_v = nullptr;  // [3*n] BVH order, v0.w = original index
    BNode* nodes = nullptr;   // [n-1]
    void* scratch = nullptr;
    void* pscratch = nullptr;
    BvhBufs bufs;
    PlocBufs pbufs;
    int cap_ = 0;
    size_t bytes_ = 0;

    cudaError_t reserve(int nt, bool ploc);
    cudaError_t build(const float* d_verts, const int* d_idx, int nv, int nt, float eps, int* err, cudaStream_t s,
                      const int* list);  // PLOC
    // a linear build of the listed triangles into tris / nodes at tri_off /
    // node_off, and their vertices into tri_orig
    cudaError_t build_moving(const float* d_verts, const int* d_idx, int nv, int nt, float eps, int* err, cudaStream_t s,
                             const int* list, float4* tris, BNode* nodes, int node_off, int tri_off, float4* tri_orig);
    void release();
    size_t bytes() const;
};

}  // namespace adgi
