// bvh.cu -- software BVH for the probe rays (the paper traces with DXR on RT
// cores, Sec. 5; here a linear BVH is built on the device every time the
// geometry moves).
//
// Build: centroid bounds -> 63-bit Morton codes -> stable LSD radix sort
// (8 passes of 8 bits) -> Karras (HPG 2012) radix-tree hierarchy
// -> bottom-up child boxes, each leaf box enlarged by eps so that box tests
// stay conservative for the watertight triangle test.
#include <algorithm>
#include <cstdio>

#include "adgi_internal.cuh"
#include "bvh.cuh"
#include "kernels.cuh"
#include "bvhbody.cuh"

namespace adgi {

namespace {

constexpr int kSortThreads = 256;


__global__ void k_init_bounds(uint32_t* __restrict__ bounds)
{
    if (threadIdx.x < 3) bounds[threadIdx.x] = 0xFFFFFFFFu;
    else if (threadIdx.x < 6) bounds[threadIdx.x] = 0u;
}


__global__ void k_tri_prep(const float* __restrict__ verts, const int* __restrict__ idx, const int* __restrict__ list,
                           int nt, int nv, float4* __restrict__ tri_in, uint32_t* __restrict__ bounds,
                           int* __restrict__ err)
{
    __shared__ uint32_t s_lo[3], s_hi[3];
    if (threadIdx.x < 3) {
        s_lo[threadIdx.x] = 0xFFFFFFFFu;
        s_hi[threadIdx.x] = 0u;
    }
    __syncthreads();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nt) tri_fetch(verts, idx, list, nv, i, tri_in, s_lo, s_hi, err);
    __syncthreads();
    if (threadIdx.x < 3) {
        atomicMin(&bounds[threadIdx.x], s_lo[threadIdx.x]);
        atomicMax(&bounds[3 + threadIdx.x], s_hi[threadIdx.x]);
    }
}




// vertices of the listed triangles into an original-order array (shading)
__global__ void k_fill_orig(const float* __restrict__ verts, const int* __restrict__ idx, const int* __restrict__ list,
                            int nt, int nv, float4* __restrict__ tri_orig)
{
    fill_orig_body(verts, idx, list, nt, nv, tri_orig, blockIdx.x * blockDim.x + threadIdx.x);
}

constexpr int kSmallThreads = 1024;

__global__ void __launch_bounds__(kSmallThreads) k_morton_small(const float* __restrict__ verts,
                                                                const int* __restrict__ idx,
                                                                const int* __restrict__ list, int nt, int nv,
                                                                float4* __restrict__ tri_in, uint64_t* __restrict__ keys,
                                                                uint32_t* __restrict__ vals,
                                                                float4* __restrict__ tri_v, int* __restrict__ err)
{
    __shared__ uint64_t sk[kSmallBuild];
    __shared__ uint32_t sv[kSmallBuild];
    morton_small_body(verts, idx, list, nt, nv, tri_in, keys, vals, tri_v, err, sk, sv);
}

__global__ void k_hierarchy(const uint64_t* __restrict__ keys, int n, BNode* __restrict__ nodes,
                            int* __restrict__ par_int, int* __restrict__ par_leaf, int node_off, int tri_off)
{
    hierarchy_body(keys, n, nodes, par_int, par_leaf, blockIdx.x * blockDim.x + threadIdx.x, node_off, tri_off);
}

__global__ void k_bounds(const float4* __restrict__ tri_v, int n, BNode* nodes, const int* __restrict__ par_int,
                         const int* __restrict__ par_leaf, int* flags, float eps, int* err, int node_off, int tri_off)
{
    bounds_body(tri_v, n, nodes, par_int, par_leaf, flags, eps, err, blockIdx.x * blockDim.x + threadIdx.x, node_off,
                tri_off);
}

// A small linear build (nt <= kSmallBuild) in one block and one launch: the
// triangles, their Morton order, the radix tree and the boxes, bottom up with
// parents, flags and node boxes in shared memory, where a step up costs some
// 0.1 us instead of the 1 us of a chain of global round trips.  The nodes are
// those of the larger build's kernels.  (A city's 240 moving triangles: five
// launches of 52 us together before, one of 18 us.)
struct SmallLayout {
    uint32_t keys, vals, lo, hi, child, par_int, par_leaf, flags, total;
};

__host__ __device__ inline SmallLayout small_layout(int nt)
{
    uint32_t n2 = 2;
    while ((int)n2 < nt) n2 <<= 1;
    SmallLayout L;
    uint32_t o = 0;
    L.lo = o, o += 16 * n2;
    L.hi = o, o += 16 * n2;
    L.keys = o, o += 8 * n2;
    L.child = o, o += 8 * n2;
    L.vals = o, o += 4 * n2;
    L.par_int = o, o += 4 * n2;
    L.par_leaf = o, o += 4 * n2;
    L.flags = o, o += 4 * n2;
    L.total = o;
    return L;
}

__global__ void __launch_bounds__(kSmallThreads)
    k_build_small(const float* __restrict__ verts, const int* __restrict__ idx, const int* __restrict__ list, int nt, int nv,
                  float4* tri_in, uint64_t* __restrict__ keys, uint32_t* __restrict__ vals, float4* tri_v, BNode* nodes,
                  int* __restrict__ par_int_out, int* __restrict__ par_leaf_out, float eps, int* err, int node_off, int tri_off,
                  float4* tri_orig)
{
    extern __shared__ __align__(16) unsigned char small_smem[];
    const SmallLayout L = small_layout(nt);
    uint64_t* sk = reinterpret_cast<uint64_t*>(small_smem + L.keys);
    uint32_t* sv = reinterpret_cast<uint32_t*>(small_smem + L.vals);
    float4* lo = reinterpret_cast<float4*>(small_smem + L.lo);  // boxes of the internal nodes
    float4* hi = reinterpret_cast<float4*>(small_smem + L.hi);
    int2* child = reinterpret_cast<int2*>(small_smem + L.child);
    int* par_int = reinterpret_cast<int*>(small_smem + L.par_int);
    int* par_leaf = reinterpret_cast<int*>(small_smem + L.par_leaf);
    int* flags = reinterpret_cast<int*>(small_smem + L.flags);
    const int tid = threadIdx.x, nthr = blockDim.x;
    if (tri_orig)
        for (int i = tid; i < nt; i += nthr) fill_orig_body(verts, idx, list, nt, nv, tri_orig, i);
    morton_small_body(verts, idx, list, nt, nv, tri_in, keys, vals, tri_v, err, sk, sv);
    if (nt < 2) return;
    for (int i = tid; i < nt; i += nthr) flags[i] = 0;
    for (int i = tid; i < nt - 1; i += nthr) {
        const int2 c = karras_children(sk, nt, i);
        child[i] = c;
        for (int ch : {c.x, c.y}) {
            if (ch < 0)
                par_leaf[~ch] = par_leaf_out[~ch] = i;
            else
                par_int[ch] = par_int_out[ch] = i;
        }
        if (i == 0) par_int[0] = par_int_out[0] = -1;
    }
    __syncthreads();  // (also the block's tri_v)
    auto box_of = [&](int ch, float3& l, float3& h) {
        if (ch < 0) {
            leaf_box(tri_v, ~ch, eps, l, h);
        } else {
            l = make_float3(lo[ch].x, lo[ch].y, lo[ch].z);
            h = make_float3(hi[ch].x, hi[ch].y, hi[ch].z);
        }
    };
    for (int i = tid; i < nt; i += nthr) {
        int par = par_leaf[i];
        for (int depth = 0; par >= 0; ++depth) {
            if (depth > 128) {  // a radix tree over 95-bit keys is at most 95 deep
                atomicOr(err, kErrBvh);
                break;
            }
            __threadfence_block();
            if (atomicAdd(&flags[par], 1) == 0) break;
            __threadfence_block();
            const int2 c = child[par];
            float3 l0, h0, l1, h1;
            box_of(c.x, l0, h0);
            box_of(c.y, l1, h1);
            BNode b;
            b.a = make_float4(l0.x, l0.y, l0.z, h0.x);
            b.b = make_float4(h0.y, h0.z, l1.x, l1.y);
            b.c = make_float4(l1.z, h1.x, h1.y, h1.z);
            b.d = relocated(c, node_off, tri_off);
            nodes[par] = b;
            lo[par] = make_float4(fminf(l0.x, l1.x), fminf(l0.y, l1.y), fminf(l0.z, l1.z), 0.f);
            hi[par] = make_float4(fmaxf(h0.x, h1.x), fmaxf(h0.y, h1.y), fmaxf(h0.z, h1.z), 0.f);
            par = par_int[par];
        }
    }
}

__global__ void k_morton(const float4* __restrict__ tri_in, int nt, const uint32_t* __restrict__ bounds,
                         uint64_t* __restrict__ keys, uint32_t* __restrict__ vals)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    keys[t] = morton_key(tri_in[3 * (size_t)t], tri_in[3 * (size_t)t + 1], tri_in[3 * (size_t)t + 2], bounds);
    vals[t] = (uint32_t)t;
}

// Radix sort, one pass of eight bits: k_radix_scan, then k_radix_scatter.
// hist[d nb + b]: keys of digit d in tile b.  The first pass's counts come
// from k_radix_hist, the later ones from the scatter before (a key's next
// digit is counted at the tile where it lands), so a pass is two launches.
//   (Tiles of 4,096 keys with a count, a one-block scan and an unstaged
// scatter a pass left most of the chip idle below a million keys: 116k keys
// in eight passes took 321 us, 3.25M in three 280 us; now 89 and 145 us.)
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const uint64_t* __restrict__ keys, int n, int shift,
                                                             uint32_t* __restrict__ hist, int nb)
{
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int base = blockIdx.x * kRadixTile;
    for (int i = base + (int)threadIdx.x; i < min(n, base + kRadixTile); i += kSortThreads)
        atomicAdd(&h[(uint32_t)(keys[i] >> shift) & 255u], 1u);
    __syncthreads();
    hist[(size_t)threadIdx.x * nb + blockIdx.x] = h[threadIdx.x];
}

// exclusive prefix of v over the block's 256 threads; *total: the sum
__device__ __forceinline__ uint64_t sort_exscan(uint64_t v, uint64_t* red, uint64_t* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) red[warp] = x;
    __syncthreads();
    uint64_t pre = x - v, all = 0;
    for (int w = 0; w < kSortThreads / 32; ++w) {
        if (w < warp) pre += red[w];
        all += red[w];
    }
    *total = all;
    return pre;
}

// digit blockIdx.x: its counts become the tiles' offsets inside the digit;
// the next pass's counts are cleared
__global__ void __launch_bounds__(kSortThreads) k_radix_scan(uint32_t* __restrict__ hist, uint32_t* __restrict__ next,
                                                             int nb, uint32_t* __restrict__ totals)
{
    __shared__ uint64_t red[kSortThreads / 32];
    uint32_t* row = hist + (size_t)blockIdx.x * nb;
    uint64_t carry = 0;
    for (int b0 = 0; b0 < nb; b0 += kSortThreads) {
        const int b = b0 + (int)threadIdx.x;
        uint64_t all;
        const uint64_t pre = sort_exscan(b < nb ? row[b] : 0u, red, &all);
        if (b < nb) {
            row[b] = (uint32_t)(carry + pre);
            next[(size_t)blockIdx.x * nb + b] = 0u;
        }
        carry += all;
    }
    if (threadIdx.x == 0) totals[blockIdx.x] = (uint32_t)carry;
}

// A warp ranks its keys 32 at a time (equal digits matched across the lanes),
// the block adds its warps' counts, and the tile is put in digit order in
// shared memory before it is written, so that writes run along the digits.
__global__ void __launch_bounds__(kSortThreads)
    k_radix_scatter(const uint64_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint64_t* __restrict__ kout,
                    uint32_t* __restrict__ vout, int n, int shift, const uint32_t* __restrict__ hist,
                    const uint32_t* __restrict__ totals, uint32_t* __restrict__ next, int nb)
{
    constexpr int kWarps = kSortThreads / 32, kTile = kRadixTile, kItems = kTile / kSortThreads;
    __shared__ uint32_t cnt[kWarps][256], at[256], dst[256];
    __shared__ uint64_t sk[kTile];
    __shared__ uint32_t sv[kTile];
    __shared__ uint64_t red[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, base = blockIdx.x * kTile;
    const int live = min(kTile, n - base);
#pragma unroll
    for (int w = 0; w < kWarps; ++w) cnt[w][tid] = 0u;
    uint64_t k[kItems];
    uint32_t v[kItems], rank[kItems];
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        const int i = (warp * kItems + r) * 32 + lane;
        k[r] = i < live ? kin[base + i] : 0ull;
        v[r] = i < live ? vin[base + i] : 0u;
    }
    __syncthreads();
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        const bool on = (warp * kItems + r) * 32 + lane < live;
        const uint32_t d = on ? (uint32_t)(k[r] >> shift) & 255u : 256u;  // the lanes past the end match each other
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
        const uint32_t before = on ? cnt[warp][d] : 0u;
        rank[r] = before + __popc(peers & lt);
        __syncwarp();
        if (on && (peers & lt) == 0u) cnt[warp][d] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {  // thread = digit: its warps' offsets, its place in the tile and in the output
        uint32_t run = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t c = cnt[w][tid];
            cnt[w][tid] = run;
            run += c;
        }
        uint64_t all;
        const uint64_t pre = sort_exscan((uint64_t)run << 32 | totals[tid], red, &all);  // totals add up to n < 2^32
        at[tid] = (uint32_t)(pre >> 32);
        dst[tid] = (uint32_t)pre + hist[(size_t)tid * nb + blockIdx.x] - at[tid];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        if ((warp * kItems + r) * 32 + lane >= live) continue;
        const uint32_t d = (uint32_t)(k[r] >> shift) & 255u, q = at[d] + cnt[warp][d] + rank[r];
        sk[q] = k[r];
        sv[q] = v[r];
    }
    __syncthreads();
    // (Counted one atomic a key, 200,000 equal keys took 640 us a build: each
    // warp's 32 counts, and those of all tiles' keys that land in one tile, went
    // to one address.  A warp whose keys all count there adds them at once.)
    for (int i0 = 0; i0 < live; i0 += kSortThreads) {
        const int i = i0 + tid;
        const bool on = i < live;
        uint32_t to = 0xFFFFFFFFu;  // the count of the key's next digit
        if (on) {
            const uint64_t key = sk[i];
            const uint32_t pos = dst[(uint32_t)(key >> shift) & 255u] + (uint32_t)i;
            kout[pos] = key;
            vout[pos] = sv[i];
            to = ((uint32_t)(key >> (shift + 8)) & 255u) * (uint32_t)nb + pos / kTile;
        }
        if (next) {
            const bool all = __all_sync(0xFFFFFFFFu, to == __shfl_sync(0xFFFFFFFFu, to, 0));
            if (all ? on && lane == 0 : on) atomicAdd(next + to, all ? 32u : 1u);
        }
    }
}

// exclusive scan of a small array in one block of 1024 threads
__global__ void k_scan_small(uint32_t* __restrict__ a, int n)
{
    __shared__ uint32_t part[1024];
    int tid = threadIdx.x;
    int per = (n + 1023) / 1024;
    int s0 = tid * per, s1 = min(n, s0 + per);
    uint32_t sum = 0;
    for (int i = s0; i < s1; ++i) sum += a[i];
    part[tid] = sum;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        uint32_t v = tid >= off ? part[tid - off] : 0u;
        __syncthreads();
        part[tid] += v;
        __syncthreads();
    }
    uint32_t run = part[tid] - sum;
    for (int i = s0; i < s1; ++i) {
        uint32_t v = a[i];
        a[i] = run;
        run += v;
    }
}

// Exclusive scan of a large array in three launches: per-chunk sums, a scan
// of the (at most 1024) sums, and a scan of each chunk from its carry.
constexpr int kScanChunks = 1024;

__global__ void __launch_bounds__(256) k_scan_reduce(const uint32_t* __restrict__ a, int n, int per,
                                                     uint32_t* __restrict__ part)
{
    __shared__ uint32_t red[8];
    const int b0 = blockIdx.x * per, b1 = min(n, b0 + per);
    uint32_t s = 0;
    for (int i = b0 + threadIdx.x; i < b1; i += blockDim.x) s += a[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(256) k_scan_apply(uint32_t* __restrict__ a, int n, int per,
                                                    const uint32_t* __restrict__ part)
{
    __shared__ uint32_t wsum[8];
    const int b0 = blockIdx.x * per, b1 = min(n, b0 + per);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t carry = part[blockIdx.x];
    for (int t0 = b0; t0 < b1; t0 += 4 * (int)blockDim.x) {  // tiles of 4 items per thread
        const int i0 = t0 + 4 * (int)threadIdx.x;
        uint32_t v[4], tot = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = i0 + k < b1 ? a[i0 + k] : 0u;
            tot += v[k];
        }
        uint32_t x = tot;  // inclusive scan of the thread totals in the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        uint32_t before = carry, all = 0;
        for (int w = 0; w < nw; ++w) {
            const uint32_t ws = wsum[w];
            if (w < warp) before += ws;
            all += ws;
        }
        before += x - tot;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i0 + k < b1) a[i0 + k] = before;
            before += v[k];
        }
        carry += all;
        __syncthreads();
    }
}

__global__ void k_tri_order(const float4* __restrict__ tri_in, const uint32_t* __restrict__ order, int nt,
                            float4* __restrict__ tri_v)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nt) return;
    uint32_t t = order[i];
    tri_v[3 * (size_t)i] = tri_in[3 * (size_t)t];
    tri_v[3 * (size_t)i + 1] = tri_in[3 * (size_t)t + 1];
    tri_v[3 * (size_t)i + 2] = tri_in[3 * (size_t)t + 2];
}






// ---------------------------------------------------------------- PLOC
// Parallel locally-ordered clustering (Meister & Bittner, TVCG 2018): clusters
// in Morton order; each finds its nearest neighbour by the surface area of the
// merged box within +-kPlocR positions; mutual nearest neighbours merge into a
// new node; the cluster array is compacted; repeat until one cluster is left.
// A wide window finds better partners (+-1,536 positions: nearest hit 1.20 ms
// on the 198k-triangle scene, against 1.29 at +-256), but after the reinsertion
// below a narrow one's tree is as good and found sooner: tunnel / scaled update
// ms and 198k static build ms at +-8: 2.28 / 6.64 / 4.26, +-16: 2.28 / 6.58 /
// 4.22, +-32: 2.26 / 6.63 / 4.35, +-64: 2.30 / 6.70 / 4.70.
constexpr int kPlocR = 16;
constexpr int kPlocT = 256;
constexpr int kPlocTail = 512;    // clusters that one block finishes on its own
constexpr int kPlocRounds = 8;    // rounds launched between two looks at the count
constexpr int kMergeItems = 1, kMergeBlock = kPlocT * kMergeItems;

// the clustering's state, kept on the device so that rounds follow one
// another without the host: round r reads st[r & 1] and writes the other
struct PlocState {
    int count;     // clusters left
    int node_top;  // nodes [node_top, n - 1) exist
    int stuck;     // a round merged nothing (cannot happen with strict ties)
    int pair_top;  // nodes [pair_top, n - 1) are the pairs merged first
};

// half the surface area; the rounded steps are fixed, so that it is the same
// at every use and grows with the extents (the neighbour search's bound)
__device__ __forceinline__ float box_area(float4 lo, float4 hi)
{
    const float dx = hi.x - lo.x, dy = hi.y - lo.y, dz = hi.z - lo.z;
    return __fmaf_rn(dx, dy, __fmaf_rn(dy, dz, __fmul_rn(dz, dx)));
}

__global__ void k_ploc_init(const float4* __restrict__ tri_v, int n, float eps, int* __restrict__ cid,
                            float4* __restrict__ blo, float4* __restrict__ bhi)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float4 A = tri_v[3 * (size_t)i], B = tri_v[3 * (size_t)i + 1], C = tri_v[3 * (size_t)i + 2];
    eps = tri_eps(eps, A, B, C);
    blo[i] = make_float4(fminf(fminf(A.x, B.x), C.x) - eps, fminf(fminf(A.y, B.y), C.y) - eps,
                         fminf(fminf(A.z, B.z), C.z) - eps, 0.f);
    bhi[i] = make_float4(fmaxf(fmaxf(A.x, B.x), C.x) + eps, fmaxf(fmaxf(A.y, B.y), C.y) + eps,
                         fmaxf(fmaxf(A.z, B.z), C.z) + eps, 0.f);
    cid[i] = ~i;
}

__global__ void k_ploc_begin(PlocState* st, int n)
{
    st[0] = PlocState{n, n - 1, 0, n - 1};
}

// ---- pairs of triangles that share an edge, merged before the first round,
// so that quads become one leaf of the 4-wide tree (wide.cu) whatever else
// lies nearby.  Looked for among the next kPairWin triangles of the list on
// either side (meshes emit the halves of a quad together).  Left to the
// clustering alone, 29 % of the 2M-triangle city's triangles ended up apart
// from their other half (boxes that tie or overlap); merged first: nearest
// hit 5.72 -> 4.10 ms, shadow rays 4.16 -> 2.74 ms per scaled update (198k
// triangles: 1.30 -> 1.29 and 1.02 -> 0.98).
constexpr int kPairWin = 4;

__global__ void k_pair_pos(const uint32_t* __restrict__ order, int n, int* __restrict__ pos)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) pos[order[i]] = i;
}

__device__ __forceinline__ bool same_vertex(float4 a, float4 b)
{
    return __float_as_uint(a.x) == __float_as_uint(b.x) && __float_as_uint(a.y) == __float_as_uint(b.y) &&
           __float_as_uint(a.z) == __float_as_uint(b.z);
}

// Two passes: mate[] of pass 0 is each triangle's best partner; pass 1 (prev
// = pass 0's) keeps the mutual pairs and lets the others choose again among
// the others.
__global__ void k_pair_mates(const float4* __restrict__ tri_v, const uint32_t* __restrict__ order,
                             const int* __restrict__ pos, int n, const float4* __restrict__ blo,
                             const float4* __restrict__ bhi, const int* __restrict__ prev, int* __restrict__ mate)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (prev && prev[i] != i && prev[prev[i]] == i) {
        mate[i] = prev[i];
        return;
    }
    const float4 A[3] = {tri_v[3 * (size_t)i], tri_v[3 * (size_t)i + 1], tri_v[3 * (size_t)i + 2]};
    const float4 lo = blo[i], hi = bhi[i];
    const float own = box_area(lo, hi);
    const int u = (int)order[i];
    float best = 0.0f;
    int bj = i;
    for (int k = -kPairWin; k <= kPairWin; ++k) {
        if (k == 0 || u + k < 0 || u + k >= n) continue;
        const int j = pos[u + k];
        if (prev && prev[j] != j && prev[prev[j]] == j) continue;  // taken
        const float4 B[3] = {tri_v[3 * (size_t)j], tri_v[3 * (size_t)j + 1], tri_v[3 * (size_t)j + 2]};
        bool edge = false;  // an edge of A, backwards in B
        for (int x = 0; x < 3; ++x)
            for (int y = 0; y < 3; ++y)
                edge = edge || (same_vertex(A[x], B[(y + 1) % 3]) && same_vertex(A[(x + 1) % 3], B[y]));
        if (!edge) continue;
        const float4 l2 = blo[j], h2 = bhi[j];
        const float both = own + box_area(l2, h2);
        const float u2 = box_area(make_float4(fminf(lo.x, l2.x), fminf(lo.y, l2.y), fminf(lo.z, l2.z), 0.f),
                                  make_float4(fmaxf(hi.x, h2.x), fmaxf(hi.y, h2.y), fmaxf(hi.z, h2.z), 0.f));
        // worth one box: a pair's test costs 80, two triangles' 55 each
        if (80.0f * u2 < 55.0f * both && u2 - both < best) {
            best = u2 - both;
            bj = j;
        }
    }
    mate[i] = bj;
}

// the merged area of a box with group g's nearest point: at most that with
// any box inside the group (areas grow with the extents, also in the rounded
// steps of box_area)
__device__ __forceinline__ float group_bound(float4 lo, float4 hi, float4 gl, float4 gh)
{
    return box_area(make_float4(fminf(lo.x, gh.x), fminf(lo.y, gh.y), fminf(lo.z, gh.z), 0.f),
                    make_float4(fmaxf(hi.x, gl.x), fmaxf(hi.y, gl.y), fmaxf(hi.z, gl.z), 0.f));
}

// the boxes [j0, j1) at blo, bhi (in shared memory, read by all lanes at once)
// against cluster i's: the least merged area, ties to the smaller index
__device__ __forceinline__ void nearest_of(const float4* blo, const float4* bhi, int j0, int j1, int i, float4 lo,
                                           float4 hi, float& best, int& bj)
{
#pragma unroll 4
    for (int j = j0; j < j1; ++j) {
        const float4 l2 = blo[j - j0], h2 = bhi[j - j0];
        const float a = box_area(make_float4(fminf(lo.x, l2.x), fminf(lo.y, l2.y), fminf(lo.z, l2.z), 0.f),
                                 make_float4(fmaxf(hi.x, h2.x), fmaxf(hi.y, h2.y), fmaxf(hi.z, h2.z), 0.f));
        if (j != i && (a < best || (a == best && j < bj))) {
            best = a;
            bj = j;
        }
    }
}

// Nearest neighbour of every cluster: the least merged area over the window,
// ties to the smaller index.  The block's boxes and kPlocR on either side are
// staged in shared memory.
__global__ void __launch_bounds__(kPlocT) k_ploc_nn(const PlocState* __restrict__ st, const float4* __restrict__ blo,
                                                    const float4* __restrict__ bhi, int* __restrict__ nn)
{
    __shared__ float4 s_lo[kPlocT + 2 * kPlocR], s_hi[kPlocT + 2 * kPlocR];
    const int count = st->count, base = blockIdx.x * kPlocT, first = base - kPlocR;
    if (base >= count) return;
    for (int k = threadIdx.x; k < kPlocT + 2 * kPlocR; k += kPlocT) {
        const int j = min(max(first + k, 0), count - 1);
        s_lo[k] = __ldg(blo + j);
        s_hi[k] = __ldg(bhi + j);
    }
    __syncthreads();
    const int i = base + (int)threadIdx.x;
    if (i >= count) return;
    float best = __int_as_float(0x7F800000);
    int bj = i;
    const int j0 = max(i - kPlocR, 0), j1 = min(i + kPlocR + 1, count);
    nearest_of(s_lo + (j0 - first), s_hi + (j0 - first), j0, j1, i, s_lo[i - first], s_hi[i - first], best, bj);
    nn[i] = bj;
}

// cluster i of a round: kept (high word), makes a node (low word)
__device__ __forceinline__ uint64_t ploc_flags(const int* __restrict__ nn, int i)
{
    const int j = nn[i];
    const bool mutual = j != i && nn[j] == i;
    return (uint64_t)!(mutual && j < i) << 32 | (uint64_t)(mutual && i < j);
}

__device__ __forceinline__ uint64_t ploc_block_sum(uint64_t v, uint64_t* red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    uint64_t t = 0;
    for (int w = 0; w < kPlocT / 32; ++w) t += red[w];
    return t;
}

__global__ void __launch_bounds__(kPlocT) k_ploc_count(const PlocState* __restrict__ st, const int* __restrict__ nn,
                                                       uint64_t* __restrict__ sums)
{
    __shared__ uint64_t red[kPlocT / 32];
    const int count = st->count, base = blockIdx.x * kMergeBlock;
    if (base >= count) return;
    uint64_t v = 0;
    for (int k = 0; k < kMergeItems; ++k) {
        const int i = base + k * kPlocT + (int)threadIdx.x;
        if (i < count) v += ploc_flags(nn, i);
    }
    v = ploc_block_sum(v, red);
    if (threadIdx.x == 0) sums[blockIdx.x] = v;
}

// The mutual pairs become nodes, numbered from the top in cluster order, and
// the clusters are compacted in order; each block adds up the counts of the
// blocks before it.  The last block writes the next round's state.
__global__ void __launch_bounds__(kPlocT)
    k_ploc_merge(const PlocState* __restrict__ st, PlocState* __restrict__ st2, int must, const int* __restrict__ nn,
                 const uint64_t* __restrict__ sums, const int* __restrict__ cid, const float4* __restrict__ blo,
                 const float4* __restrict__ bhi, int* __restrict__ cid2, float4* __restrict__ blo2,
                 float4* __restrict__ bhi2, BNode* __restrict__ nodes, int* __restrict__ par_int,
                 int* __restrict__ par_leaf)
{
    __shared__ uint64_t red[kPlocT / 32];
    const int count = st->count, node_top = st->node_top, base = blockIdx.x * kMergeBlock;
    if (base >= count) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint64_t pre = 0;
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += kPlocT) pre += sums[k];
    pre = ploc_block_sum(pre, red);
    const int i0 = base + kMergeItems * (int)threadIdx.x;
    uint64_t fl[kMergeItems], run = 0;
#pragma unroll
    for (int k = 0; k < kMergeItems; ++k) {
        fl[k] = i0 + k < count ? ploc_flags(nn, i0 + k) : 0ull;
        run += fl[k];
    }
    uint64_t x = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) red[warp] = x;
    __syncthreads();
    uint64_t all = pre;
    for (int w = 0; w < kPlocT / 32; ++w) {
        if (w < warp) pre += red[w];
        all += red[w];
    }
    pre += x - run;
    if (base + kMergeBlock >= count && threadIdx.x == 0) {
        const int merges = (int)(all & 0xFFFFFFFFu);
        *st2 = PlocState{(int)(all >> 32), node_top - merges, st->stuck | (must && count > 1 && merges == 0),
                         must ? st->pair_top : node_top - merges};
    }
    for (int k = 0; k < kMergeItems; ++k) {
        const int i = i0 + k;
        if (fl[k] >> 32) {
            const int pos = (int)(pre >> 32);
            float4 la = blo[i], ha = bhi[i];
            int c = cid[i];
            if (fl[k] & 1u) {
                const int j = nn[i], node = node_top - 1 - (int)(pre & 0xFFFFFFFFu), cj = cid[j];
                const float4 lb = blo[j], hb = bhi[j];
                BNode b;
                b.a = make_float4(la.x, la.y, la.z, ha.x);
                b.b = make_float4(ha.y, ha.z, lb.x, lb.y);
                b.c = make_float4(lb.z, hb.x, hb.y, hb.z);
                b.d = make_int4(c, cj, 0, 0);
                nodes[node] = b;
                for (int c2 : {c, cj}) {
                    if (c2 < 0)
                        par_leaf[~c2] = node;
                    else
                        par_int[c2] = node;
                }
                c = node;
                la = make_float4(fminf(la.x, lb.x), fminf(la.y, lb.y), fminf(la.z, lb.z), 0.f);
                ha = make_float4(fmaxf(ha.x, hb.x), fmaxf(ha.y, hb.y), fmaxf(ha.z, hb.z), 0.f);
            }
            cid2[pos] = c;
            blo2[pos] = la;
            bhi2[pos] = ha;
        }
        pre += fl[k];
    }
}

// The last rounds, from at most kPlocTail clusters to one, by one block: a
// round is then a few block barriers instead of three launches.
__global__ void __launch_bounds__(kPlocTail)
    k_ploc_tail(PlocState* st, const int* __restrict__ cid, const float4* __restrict__ blo,
                const float4* __restrict__ bhi, BNode* __restrict__ nodes, int* __restrict__ par_int,
                int* __restrict__ par_leaf)
{
    constexpr int kW = kPlocTail / 32;
    __shared__ float4 s_lo[kPlocTail], s_hi[kPlocTail];
    __shared__ int s_cid[kPlocTail], s_nn[kPlocTail];
    __shared__ float4 s_glo[kW], s_ghi[kW];
    __shared__ int s_keep[kW], s_merge[kW];
    const int i = threadIdx.x, lane = i & 31, warp = i >> 5;
    int count = st->count, node_top = st->node_top, stuck = st->stuck;
    const int pair_top = st->pair_top;
    if (count > kPlocTail) return;
    if (i < count) {
        s_lo[i] = blo[i];
        s_hi[i] = bhi[i];
        s_cid[i] = cid[i];
    }
    __syncthreads();
    while (count > 1) {
        const int ngroups = (count + 31) / 32;
        if (warp < ngroups) {
            const int j = min(i, count - 1);
            const float4 l = s_lo[j], h = s_hi[j];
            const float4 gl = make_float4(ord2f(__reduce_min_sync(0xFFFFFFFFu, f2ord(l.x))),
                                          ord2f(__reduce_min_sync(0xFFFFFFFFu, f2ord(l.y))),
                                          ord2f(__reduce_min_sync(0xFFFFFFFFu, f2ord(l.z))), 0.f);
            const float4 gh = make_float4(ord2f(__reduce_max_sync(0xFFFFFFFFu, f2ord(h.x))),
                                          ord2f(__reduce_max_sync(0xFFFFFFFFu, f2ord(h.y))),
                                          ord2f(__reduce_max_sync(0xFFFFFFFFu, f2ord(h.z))), 0.f);
            if (lane == 0) s_glo[warp] = gl, s_ghi[warp] = gh;
        }
        __syncthreads();
        const bool valid = i < count;
        int bj = i;
        if (warp < ngroups) {
            const float4 lo = s_lo[min(i, count - 1)], hi = s_hi[min(i, count - 1)];
            float best = __int_as_float(0x7F800000);
            for (int d = 0; d < 2 * kW; ++d) {
                const int g = warp + ((d & 1) ? (d + 1) / 2 : -(d / 2));
                if (g < 0 || g >= ngroups) continue;
                if (d > 0) {
                    const float lb = group_bound(lo, hi, s_glo[g], s_ghi[g]);
                    if (!__any_sync(0xFFFFFFFFu, valid && (lb < best || (lb == best && 32 * g < bj)))) continue;
                }
                nearest_of(s_lo + 32 * g, s_hi + 32 * g, 32 * g, min(32 * g + 32, count), i, lo, hi, best, bj);
            }
        }
        s_nn[i] = bj;
        __syncthreads();
        const bool mutual = valid && bj != i && s_nn[bj] == i;
        const bool keep = valid && !(mutual && bj < i), merge = mutual && i < bj;
        const uint32_t mk = __ballot_sync(0xFFFFFFFFu, keep), mm = __ballot_sync(0xFFFFFFFFu, merge);
        if (lane == 0) s_keep[warp] = __popc(mk), s_merge[warp] = __popc(mm);
        // the kept clusters' new boxes, read before the lists are rewritten
        float4 la = make_float4(0.f, 0.f, 0.f, 0.f), ha = la, lb = la, hb = la;
        int c = 0, cj = 0;
        if (keep) la = s_lo[i], ha = s_hi[i], c = s_cid[i];
        if (merge) lb = s_lo[bj], hb = s_hi[bj], cj = s_cid[bj];
        __syncthreads();
        const uint32_t lt = (1u << lane) - 1u;
        int pos = __popc(mk & lt), rank = __popc(mm & lt), kept = 0, merged = 0;
        for (int w = 0; w < kW; ++w) {
            if (w < warp) pos += s_keep[w], rank += s_merge[w];
            kept += s_keep[w];
            merged += s_merge[w];
        }
        if (merge) {
            const int node = node_top - 1 - rank;
            BNode b;
            b.a = make_float4(la.x, la.y, la.z, ha.x);
            b.b = make_float4(ha.y, ha.z, lb.x, lb.y);
            b.c = make_float4(lb.z, hb.x, hb.y, hb.z);
            b.d = make_int4(c, cj, 0, 0);
            nodes[node] = b;
            for (int c2 : {c, cj}) {
                if (c2 < 0)
                    par_leaf[~c2] = node;
                else
                    par_int[c2] = node;
            }
            c = node;
            la = make_float4(fminf(la.x, lb.x), fminf(la.y, lb.y), fminf(la.z, lb.z), 0.f);
            ha = make_float4(fmaxf(ha.x, hb.x), fmaxf(ha.y, hb.y), fmaxf(ha.z, hb.z), 0.f);
        }
        if (keep) s_lo[pos] = la, s_hi[pos] = ha, s_cid[pos] = c;
        __syncthreads();
        count = kept;
        node_top -= merged;
        if (merged == 0) {  // cannot happen with strict ties
            stuck = 1;
            break;
        }
    }
    if (i == 0) *st = PlocState{count, node_top, stuck, pair_top};
}

// ---------------------------------------------------------------- reinsertion
// Parallel reinsertion (Meister & Bittner, "Parallel Reinsertion for Bounding
// Volume Hierarchy Optimization", 2018): a subtree v is taken out of the tree
// and put back beside another node `out` where that shrinks the tree's summed
// box areas most.  A round looks for the best move of every kReEvery-th child
// place (at least one box area saved: p's, the parent that goes with v), from
// the parent upwards through the other subtrees on the way, branch and bound.
// Moves change the records of three nodes: v's parent p, p's parent, and the
// parent of `out`; the better of two moves that share one wins (re_key: gain,
// then place, so the result does not depend on the order of threads).
//   No move may put a subtree into itself, also not by way of others: a move
// is dropped when a winner's v lies between the node where its way turns
// downwards and `out`.  That is enough: from v upwards in the new tree one
// passes that turning point, an ancestor of v in the old tree, or is first
// led into another moved subtree's new place, whose own turning point is
// higher still; so every way up ends at the root.
//   Boxes are found again bottom up after each round.  Hits do not depend on
// the tree's shape.
__device__ __forceinline__ void child_box(const BNode& n, int k, float4& lo, float4& hi)
{
    if (k == 0) {
        lo = make_float4(n.a.x, n.a.y, n.a.z, 0.f);
        hi = make_float4(n.a.w, n.b.x, n.b.y, 0.f);
    } else {
        lo = make_float4(n.b.z, n.b.w, n.c.x, 0.f);
        hi = make_float4(n.c.y, n.c.z, n.c.w, 0.f);
    }
}

__device__ __forceinline__ BNode make_node(float4 lo0, float4 hi0, float4 lo1, float4 hi1, int c0, int c1)
{
    BNode b;
    b.a = make_float4(lo0.x, lo0.y, lo0.z, hi0.x);
    b.b = make_float4(hi0.y, hi0.z, lo1.x, lo1.y);
    b.c = make_float4(lo1.z, hi1.x, hi1.y, hi1.z);
    b.d = make_int4(c0, c1, 0, 0);
    return b;
}

__device__ __forceinline__ float4 fmin4(float4 a, float4 b)
{
    return make_float4(fminf(a.x, b.x), fminf(a.y, b.y), fminf(a.z, b.z), 0.f);
}
__device__ __forceinline__ float4 fmax4(float4 a, float4 b)
{
    return make_float4(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z), 0.f);
}

__device__ __forceinline__ void set_parent(int ref, int parent, int* par_int, int* par_leaf)
{
    if (ref >= 0)
        par_int[ref] = parent;
    else
        par_leaf[~ref] = parent;
}

// one box of a node's record: 24 bytes that no other child's share
__device__ __forceinline__ void put_box(BNode* n, int k, float4 lo, float4 hi)
{
    float* f = reinterpret_cast<float*>(n);
    if (k == 0) {
        n->a = make_float4(lo.x, lo.y, lo.z, hi.x);
        *reinterpret_cast<float2*>(f + 4) = make_float2(hi.y, hi.z);
    } else {
        *reinterpret_cast<float2*>(f + 6) = make_float2(lo.x, lo.y);
        n->c = make_float4(lo.z, hi.x, hi.y, hi.z);
    }
}

__device__ __forceinline__ void put_ref(BNode* n, int k, int ref)
{
    reinterpret_cast<int*>(&n->d)[k] = ref;
}

// Nearest hit / shadow rays for the 198k- and 2M-triangle scenes: without 1.20
// / 0.83 and 3.81 / 2.06 ms; every 3rd place, 15 rounds, 64 visits: 0.84 / 0.62
// and 2.65 / 1.60.  Tunnel and scaled update and static build of 198k (ms)
// for every 2nd place, 14 rounds: 2.10 / 6.25 / 3.59; 3rd, 15: 2.15 / 6.21 / 3.63;
// 3rd, 21: 2.11 / 6.15 / 4.30; 3rd, 30: 2.11 / 6.12 / 5.33; 4th, 24: 2.10 / 6.26 /
// 4.67.  Fewer visits cost more than they save (32: scaled nearest hit 2 %
// more).  A search is a chain of dependent reads (64 us a round of a third of
// 198k triangles' places), the refit another (41 us).
constexpr int kReEvery = 2;    // a round looks at every kReEvery-th child place
constexpr int kReRounds = 14;
constexpr int kReVisits = 64;  // nodes a search looks at, at most
constexpr int kReStack = 48;
// Internal nodes (without pairs) up to which one block makes all rounds, with
// barriers where the others have 70 launches.  adgi_set_scene, one block /
// launches, us: 100 unpaired triangles 557 / 880, 600 1,129 / 1,392, 1,000
// 1,439 / 1,590, 1,500 1,937 / 1,700, 2,000 2,286 / 1,799, 4,000 4,155 / 2,046.
constexpr int kReSmall = 1152;

// A place is 2 * node + child.  top: nodes from there on are pairs, which stay
// together.
struct ReBufs {
    BNode* nodes;
    int* par_int;
    int* par_leaf;
    int top;
    unsigned long long* lock;  // per node: the best move that changes its record
    int* moved;                // per node: the last round that moved it
    int* cnt;                  // per node: children refitted
    float* gain;               // per place of the round: its move, or gain 0
    int* out;
    int* pivot;
};

__device__ __forceinline__ unsigned long long re_key(float gain, int place)
{
    return (unsigned long long)__float_as_uint(gain) << 32 | (unsigned)place;
}

// the best move of the child at `place`, and a bid for the three records that
// it would change
__device__ __forceinline__ void re_search(const ReBufs& R, int place, int j)
{
    const int p = place >> 1, k = place & 1;
    float best = 0.0f;
    int out = -1, piv = -1;
    if (p != 0) {
        const BNode N = R.nodes[p];
        float4 vlo, vhi, rlo, rhi, olo, ohi;  // v, the rest of the pivot's side without v, the pivot's other child
        child_box(N, k, vlo, vhi);
        child_box(N, 1 - k, rlo, rhi);
        const float av = box_area(vlo, vhi);
        float d = box_area(fmin4(vlo, rlo), fmax4(vhi, rhi));  // saved so far: p's own box
        best = 1e-6f * d;
        int st_ref[kReStack];
        float st_d[kReStack];
        int sp = 0, pivot = p;
        const int sib = k ? N.d.x : N.d.y;
        if (sib >= 0 && sib < R.top) {
            const float e = box_area(rlo, rhi);
            if (e - av > best) st_ref[sp] = sib, st_d[sp++] = e;
        }
        // One node a turn, whether down the stack or, when that is empty, up to
        // the next pivot, so that the lanes of a warp take turns together (as
        // two nested loops a round took 106 us instead of 64).
        for (int visits = 0; visits < kReVisits; ++visits) {
            while (sp > 0 && !(st_d[sp - 1] - av > best)) --sp;
            const bool down = sp > 0;
            const int from = pivot;
            if (!down && pivot == 0) break;
            if (!down) pivot = R.par_int[from];
            const int x = down ? st_ref[--sp] : pivot;
            float dx = down ? st_d[sp] : d;
            const BNode M = R.nodes[x];
            float4 lo[2], hi[2];
            child_box(M, 0, lo[0], hi[0]);
            child_box(M, 1, lo[1], hi[1]);
            int side = -1;  // the pivot's child on v's side
            if (!down) {
                side = M.d.x == from ? 0 : 1;
                const float4 flo = side ? lo[1] : lo[0], fhi = side ? hi[1] : hi[0];
                if (from != p) {  // from's box shrinks to what is left
                    rlo = fmin4(rlo, olo), rhi = fmax4(rhi, ohi);
                    d += box_area(flo, fhi) - box_area(rlo, rhi);
                }
                olo = side ? lo[0] : lo[1], ohi = side ? hi[0] : hi[1];
                dx = d;
            }
            float e[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const float u = box_area(fmin4(lo[c], vlo), fmax4(hi[c], vhi));
                if (c != side && dx - u > best) best = dx - u, out = 2 * x + c, piv = pivot;
                e[c] = dx - (u - box_area(lo[c], hi[c]));
            }
            const bool in0 = side != 0 && M.d.x >= 0 && M.d.x < R.top && e[0] - av > best;
            const bool in1 = side != 1 && M.d.y >= 0 && M.d.y < R.top && e[1] - av > best;
            const bool first0 = e[0] > e[1];  // the likelier child is looked at next
            if (in1 && first0 && sp < kReStack) st_ref[sp] = M.d.y, st_d[sp++] = e[1];
            if (in0 && sp < kReStack) st_ref[sp] = M.d.x, st_d[sp++] = e[0];
            if (in1 && !first0 && sp < kReStack) st_ref[sp] = M.d.y, st_d[sp++] = e[1];
        }
    }
    R.gain[j] = out >= 0 ? best : 0.0f;
    R.out[j] = out;
    R.pivot[j] = piv;
    if (out >= 0) {
        const unsigned long long key = re_key(best, place);
        atomicMax(R.lock + p, key);
        atomicMax(R.lock + R.par_int[p], key);
        atomicMax(R.lock + (out >> 1), key);
    }
}

// a move that lost a record is off; the others' subtrees are marked
__device__ __forceinline__ void re_win(const ReBufs& R, int place, int j, int round)
{
    const float gain = R.gain[j];
    if (!(gain > 0.0f)) return;
    const unsigned long long key = re_key(gain, place);
    const int p = place >> 1;
    if (R.lock[p] != key || R.lock[R.par_int[p]] != key || R.lock[R.out[j] >> 1] != key) {
        R.gain[j] = 0.0f;
        return;
    }
    const int v = (place & 1) ? R.nodes[p].d.y : R.nodes[p].d.x;
    if (v >= 0 && v < R.top) R.moved[v] = round + 1;
}

// a move into a subtree that is itself moved is off
__device__ __forceinline__ void re_check(const ReBufs& R, int j, int round)
{
    if (!(R.gain[j] > 0.0f)) return;
    const int pivot = R.pivot[j];
    int x = R.out[j] >> 1;
    for (int step = 0; x != pivot; ++step, x = R.par_int[x])
        if (R.moved[x] == round + 1 || step > 4096) {  // (or very deep in a tree that is replaced anyway)
            R.gain[j] = 0.0f;
            return;
        }
}

__device__ __forceinline__ bool re_apply(const ReBufs& R, int place, int j)
{
    if (!(R.gain[j] > 0.0f)) return false;
    const int p = place >> 1, k = place & 1, out = R.out[j], q = out >> 1, g = R.par_int[p];
    const BNode N = R.nodes[p], Q = R.nodes[q];
    float4 vlo, vhi, slo, shi, olo, ohi;
    child_box(N, k, vlo, vhi);
    child_box(N, 1 - k, slo, shi);
    child_box(Q, out & 1, olo, ohi);
    const int v = k ? N.d.y : N.d.x, sib = k ? N.d.x : N.d.y, o = (out & 1) ? Q.d.y : Q.d.x;
    const int pg = R.nodes[g].d.x == p ? 0 : 1;
    put_box(R.nodes + g, pg, slo, shi);  // the sibling in p's place
    put_ref(R.nodes + g, pg, sib);
    set_parent(sib, g, R.par_int, R.par_leaf);
    put_box(R.nodes + q, out & 1, fmin4(olo, vlo), fmax4(ohi, vhi));  // p in out's place
    put_ref(R.nodes + q, out & 1, p);
    R.par_int[p] = q;
    R.nodes[p] = make_node(olo, ohi, vlo, vhi, o, v);
    set_parent(o, p, R.par_int, R.par_leaf);
    return true;
}

// boxes bottom up from the nodes without inner children; every bid is taken back
__device__ __forceinline__ void re_refit(const ReBufs& R, int i)
{
    R.lock[i] = 0ull;
    auto inner = [&](int c) { return c >= 0 && c < R.top; };
    const int4 d = R.nodes[i].d;
    if (inner(d.x) || inner(d.y)) return;
    int x = i;
    for (int step = 0; x != 0 && step < R.top; ++step) {
        BNode N;
        N.a = __ldcg(&R.nodes[x].a), N.b = __ldcg(&R.nodes[x].b), N.c = __ldcg(&R.nodes[x].c);
        float4 l0, h0, l1, h1;
        child_box(N, 0, l0, h0);
        child_box(N, 1, l1, h1);
        const int up = R.par_int[x];
        const int4 u = R.nodes[up].d;
        put_box(R.nodes + up, u.x == x ? 0 : 1, fmin4(l0, l1), fmax4(h0, h1));
        if (inner(u.x) && inner(u.y)) {
            if (add_acq_rel(R.cnt + up, 1) == 0) return;  // the other child follows
            R.cnt[up] = 0;
        }
        x = up;
    }
}

__device__ __forceinline__ int re_count(int top, int round)  // places of a round
{
    return (2 * top - round % kReEvery + kReEvery - 1) / kReEvery;
}

__global__ void __launch_bounds__(128) k_re_search(ReBufs R, int round)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < re_count(R.top, round)) re_search(R, kReEvery * j + round % kReEvery, j);
}
__global__ void __launch_bounds__(256) k_re_win(ReBufs R, int round)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < re_count(R.top, round)) re_win(R, kReEvery * j + round % kReEvery, j, round);
}
__global__ void __launch_bounds__(256) k_re_check(ReBufs R, int round)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < re_count(R.top, round)) re_check(R, j, round);
}
__global__ void __launch_bounds__(256) k_re_apply(ReBufs R, int round)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < re_count(R.top, round)) re_apply(R, kReEvery * j + round % kReEvery, j);
}
__global__ void __launch_bounds__(256) k_re_refit(ReBufs R)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < R.top) re_refit(R, i);
}

// all rounds of a small tree in one block; ends when kReEvery rounds in a row
// moved nothing
__global__ void __launch_bounds__(1024) k_re_small(ReBufs R)
{
    int idle = 0;
    for (int round = 0; round < kReRounds && idle < kReEvery; ++round) {
        const int n = re_count(R.top, round), r0 = round % kReEvery, t = threadIdx.x, T = blockDim.x;
        for (int j = t; j < n; j += T) re_search(R, kReEvery * j + r0, j);
        __syncthreads();
        for (int j = t; j < n; j += T) re_win(R, kReEvery * j + r0, j, round);
        __syncthreads();
        for (int j = t; j < n; j += T) re_check(R, j, round);
        __syncthreads();
        bool any = false;
        for (int j = t; j < n; j += T) any |= re_apply(R, kReEvery * j + r0, j);
        idle = __syncthreads_or(any) ? 0 : idle + 1;
        for (int i = t; i < R.top; i += T) re_refit(R, i);
        __syncthreads();
    }
}

static cudaError_t reinsert(const BvhBufs& B, const PlocBufs& Q, int nt, int top, cudaStream_t s)
{
    if (top < 3) return cudaSuccess;
    // in the clustering's lists, which are free by now (16 n bytes each)
    ReBufs R{B.nodes, B.par_int, B.par_leaf, top};
    R.lock = reinterpret_cast<unsigned long long*>(Q.blo[0]);
    R.moved = reinterpret_cast<int*>(R.lock + nt);
    R.cnt = R.moved + nt;
    R.gain = reinterpret_cast<float*>(Q.bhi[0]);
    R.out = reinterpret_cast<int*>(Q.blo[1]);
    R.pivot = reinterpret_cast<int*>(Q.bhi[1]);
    cudaError_t e = cudaMemsetAsync(Q.blo[0], 0, sizeof(float4) * (size_t)nt, s);
    if (e != cudaSuccess) return e;
    if (top <= kReSmall) {
        k_re_small<<<1, 1024, 0, s>>>(R);
        count_launches(1);
        return cudaGetLastError();
    }
    for (int round = 0; round < kReRounds; ++round) {
        const int n = (2 * top + kReEvery - 1) / kReEvery, b = (n + 255) / 256;
        k_re_search<<<(n + 127) / 128, 128, 0, s>>>(R, round);
        k_re_win<<<b, 256, 0, s>>>(R, round);
        k_re_check<<<b, 256, 0, s>>>(R, round);
        k_re_apply<<<b, 256, 0, s>>>(R, round);
        k_re_refit<<<(top + 255) / 256, 256, 0, s>>>(R);
        count_launches(5);
    }
    return cudaGetLastError();
}

// depth of every leaf below the root (node 0), bounded walk; max into *depth
__global__ void k_leaf_depth(int n, const int* __restrict__ par_int, const int* __restrict__ par_leaf,
                             int* __restrict__ depth)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int d = 1, x = par_leaf[i];
    while (x != 0 && d < 4096) {
        x = par_int[x];
        ++d;
    }
    atomicMax(depth, d);
}

// ---------------------------------------------------------------- 64-bit scan
// exclusive scan in three phases: per-block scans of 1024 values, a scan of
// the block totals (one block), and the add-back.
constexpr int kScanT = 256, kScanItems = 4, kScanBlock = kScanT * kScanItems;

__global__ void __launch_bounds__(kScanT) k_scan64_block(const uint64_t* __restrict__ in, uint64_t* __restrict__ out,
                                                         uint64_t* __restrict__ sums, int n)
{
    __shared__ uint64_t wsum[kScanT / 32];
    const int base = blockIdx.x * kScanBlock + threadIdx.x * kScanItems;
    uint64_t v[kScanItems], run = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = base + k < n ? in[base + k] : 0ull;
        run += v[k];
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint64_t x = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    uint64_t wbase = 0;
    for (int k = 0; k < w; ++k) wbase += wsum[k];
    uint64_t pre = wbase + x - run;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        if (base + k < n) out[base + k] = pre;
        pre += v[k];
    }
    if (threadIdx.x == kScanT - 1) sums[blockIdx.x] = wbase + x;
}

__global__ void k_scan64_small(uint64_t* __restrict__ a, int n, uint64_t* __restrict__ total)
{
    __shared__ uint64_t part[1024];
    int tid = threadIdx.x;
    int per = (n + 1023) / 1024;
    int s0 = tid * per, s1 = min(n, s0 + per);
    uint64_t sum = 0;
    for (int i = s0; i < s1; ++i) sum += a[i];
    part[tid] = sum;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
        uint64_t v = tid >= off ? part[tid - off] : 0ull;
        __syncthreads();
        part[tid] += v;
        __syncthreads();
    }
    uint64_t run = part[tid] - sum;
    for (int i = s0; i < s1; ++i) {
        uint64_t v = a[i];
        a[i] = run;
        run += v;
    }
    if (tid == 1023) *total = part[1023];
}

__global__ void k_scan64_add(uint64_t* __restrict__ out, const uint64_t* __restrict__ sums, int n)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] += sums[i / kScanBlock];
}

}  // namespace

size_t Bvh::bytes() const { return bytes_; }

size_t bvh_scratch_bytes(int nt)
{
    BvhBufs B;
    return carve_bvh_scratch(nullptr, nt, B);
}

// Carve the scratch buffers of a linear build for nt triangles out of one
// block (base may be null to only compute the size); every piece 256-byte
// aligned.
size_t carve_bvh_scratch(void* base, int nt, BvhBufs& B)
{
    const size_t n = (size_t)(nt > 0 ? nt : 1);
    size_t off = 0;
    auto take = [&](size_t bytes) -> void* {
        void* p = base ? (void*)((char*)base + off) : nullptr;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    B.tri_in = (float4*)take(sizeof(float4) * 3 * n);
    B.par_int = (int*)take(sizeof(int) * n);
    B.par_leaf = (int*)take(sizeof(int) * n);
    B.flags = (int*)take(sizeof(int) * n);
    B.keys[0] = (uint64_t*)take(sizeof(uint64_t) * n);
    B.keys[1] = (uint64_t*)take(sizeof(uint64_t) * n);
    B.vals[0] = (uint32_t*)take(sizeof(uint32_t) * n);
    B.vals[1] = (uint32_t*)take(sizeof(uint32_t) * n);
    B.hist = (uint32_t*)take(sizeof(uint32_t) * radix_hist_entries(n));
    B.bounds = (uint32_t*)take(sizeof(uint32_t) * 8);
    B.err = (int*)take(sizeof(int) * 2);
    return off;  // == bvh_scratch_layout_bytes(nt), the same pieces in the same order
}

// Stable LSD radix sort of n (key, value) pairs on key bits [0, bits), eight
// bits per pass; the result is in keys[*cur], vals[*cur].  hist holds
// radix_hist_entries(n) counters.
cudaError_t radix_sort_pairs(uint64_t* const keys[2], uint32_t* const vals[2], uint32_t* hist, int n, int bits,
                             cudaStream_t s, int* cur_out)
{
    int cur = 0;
    if (n > 0) {
        const int nb = (int)radix_tiles((size_t)n);
        uint32_t* h[2] = {hist, hist + (size_t)256 * nb};
        uint32_t* totals = hist + (size_t)512 * nb;
        k_radix_hist<<<nb, kSortThreads, 0, s>>>(keys[0], n, 0, h[0], nb);
        count_launches(1);
        for (int shift = 0; shift < bits; shift += 8) {
            uint32_t* next = shift + 8 < bits ? h[cur ^ 1] : nullptr;
            k_radix_scan<<<256, kSortThreads, 0, s>>>(h[cur], h[cur ^ 1], nb, totals);
            k_radix_scatter<<<nb, kSortThreads, 0, s>>>(keys[cur], vals[cur], keys[cur ^ 1], vals[cur ^ 1], n, shift,
                                                        h[cur], totals, next, nb);
            count_launches(2);
            cur ^= 1;
        }
    }
    *cur_out = cur;
    return cudaGetLastError();
}

// Exclusive scan of a[0..n) in place: one block for small arrays, the
// three-launch scan (part: 1024 partial sums) for large ones.
cudaError_t scan_exclusive_u32(uint32_t* a, int n, uint32_t* part, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    if (part != nullptr && n > 65536) {
        const int G = std::min(kScanChunks, (n + 1023) / 1024), per = (n + G - 1) / G;
        k_scan_reduce<<<G, 256, 0, s>>>(a, n, per, part);
        k_scan_small<<<1, 1024, 0, s>>>(part, G);
        k_scan_apply<<<G, 256, 0, s>>>(a, n, per, part);
        count_launches(3);
    } else {
        k_scan_small<<<1, 1024, 0, s>>>(a, n);
        count_launches(1);
    }
    return cudaGetLastError();
}

// Morton order of the listed triangles into B.tri_v (all builds start here)
static cudaError_t morton_order(const BvhBufs& B, const float* d_verts, const int* d_idx, const int* list, int nv,
                                int nt, int* err, cudaStream_t s, int* cur_out)
{
    const int T = 256;
    if (nt <= kSmallBuild) {
        k_morton_small<<<1, kSmallThreads, 0, s>>>(d_verts, d_idx, list, nt, nv, B.tri_in, B.keys[0], B.vals[0],
                                                    B.tri_v, err);
        count_launches(1);
        *cur_out = 0;
        return cudaGetLastError();
    }
    k_init_bounds<<<1, 32, 0, s>>>(B.bounds);
    count_launches(1);
    k_tri_prep<<<(nt + T - 1) / T, T, 0, s>>>(d_verts, d_idx, list, nt, nv, B.tri_in, B.bounds, err);
    count_launches(1);
    k_morton<<<(nt + T - 1) / T, T, 0, s>>>(B.tri_in, nt, B.bounds, B.keys[0], B.vals[0]);
    count_launches(1);
    int cur = 0;
    cudaError_t e = radix_sort_pairs(B.keys, B.vals, B.hist, nt, 64, s, &cur);
    if (e != cudaSuccess) return e;
    k_tri_order<<<(nt + T - 1) / T, T, 0, s>>>(B.tri_in, B.vals[cur], nt, B.tri_v);
    count_launches(1);
    *cur_out = cur;
    return cudaGetLastError();
}

// Linear BVH (Karras 2012) of the listed triangles (list = null: all).  Every
// buffer comes from B (scratch) or the outputs B.tri_v / B.nodes; all work is
// ordered on stream s; nothing is allocated.
cudaError_t build_lbvh(const BvhBufs& B, const float* d_verts, const int* d_idx, int nv, int nt, float eps, int* err,
                       cudaStream_t s, int* root_leaf, const int* list, int node_off, int tri_off, float4* tri_orig)
{
    if (nt <= 0) {
        *root_leaf = -1;
        return cudaSuccess;
    }
    *root_leaf = nt == 1 ? 0 : -1;
    if (nt <= kSmallBuild) {
        cudaError_t e = raise_smem_limit((const void*)k_build_small, small_layout(kSmallBuild).total);
        if (e != cudaSuccess) return e;
        const int t = std::min(kSmallThreads, (nt + 31) / 32 * 32);
        k_build_small<<<1, t, small_layout(nt).total, s>>>(d_verts, d_idx, list, nt, nv, B.tri_in, B.keys[0], B.vals[0], B.tri_v,
                                                           B.nodes, B.par_int, B.par_leaf, eps, err, node_off, tri_off, tri_orig);
        count_launches(1);
        return cudaGetLastError();
    }
    const int T = 256;
    int cur = 0;
    cudaError_t e = tri_orig ? fill_tri_orig(d_verts, d_idx, list, nv, nt, tri_orig, s) : cudaSuccess;
    if (e == cudaSuccess) e = morton_order(B, d_verts, d_idx, list, nv, nt, err, s, &cur);
    if (e == cudaSuccess) e = cudaMemsetAsync(B.flags, 0, sizeof(int) * (size_t)nt, s);
    if (e != cudaSuccess) return e;
    k_hierarchy<<<(nt - 1 + T - 1) / T, T, 0, s>>>(B.keys[cur], nt, B.nodes, B.par_int, B.par_leaf, node_off, tri_off);
    count_launches(1);
    k_bounds<<<(nt + T - 1) / T, T, 0, s>>>(B.tri_v, nt, B.nodes, B.par_int, B.par_leaf, B.flags, eps, err, node_off, tri_off);
    count_launches(1);
    return cudaGetLastError();
}

// PLOC build of the listed triangles: Morton order as for the linear BVH,
// then agglomerative clustering and the reinsertion rounds.  The host reads the
// cluster count every kPlocRounds rounds, to shrink the grids; meant for
// geometry that changes rarely.  Nodes are numbered from the top so that the
// final merge is node 0.  (A level of 198k triangles and a first batch of rays
// took 19.4 ms with a look at the count and six launches a round over a window
// of +-1,536; with the rounds on the device, the narrow window and the one-block
// tail, and the pairs, the reinsertion and the 4-wide tree on top, 3.5.)
cudaError_t build_ploc(const BvhBufs& B, const PlocBufs& Q, const float* d_verts, const int* d_idx, int nv, int nt,
                       float eps, int* err, cudaStream_t s, int* root_leaf, const int* list)
{
    if (nt <= 0) {
        *root_leaf = -1;
        return cudaSuccess;
    }
    int cur = 0;
    cudaError_t e = morton_order(B, d_verts, d_idx, list, nv, nt, err, s, &cur);
    if (e != cudaSuccess) return e;
    if (nt == 1) {
        *root_leaf = 0;
        return cudaGetLastError();
    }
    *root_leaf = -1;
    const int T = 256;
    k_ploc_init<<<(nt + T - 1) / T, T, 0, s>>>(B.tri_v, nt, eps, Q.cid[0], Q.blo[0], Q.bhi[0]);
    PlocState* st = reinterpret_cast<PlocState*>(Q.state);
    k_ploc_begin<<<1, 1, 0, s>>>(st, nt);
    count_launches(2);
    // one round of merges, from the neighbours in nn; c: the lists and the
    // state it reads; bound: clusters there are at most
    int c = 0, bound = nt;
    auto merge = [&](const int* nn, int must) {  // must: some pair is mutual
        const int mb = (bound + kMergeBlock - 1) / kMergeBlock;
        k_ploc_count<<<mb, kPlocT, 0, s>>>(st + c, nn, Q.sums);
        k_ploc_merge<<<mb, kPlocT, 0, s>>>(st + c, st + (c ^ 1), must, nn, Q.sums, Q.cid[c], Q.blo[c], Q.bhi[c], Q.cid[c ^ 1],
                                           Q.blo[c ^ 1], Q.bhi[c ^ 1], B.nodes, B.par_int, B.par_leaf);
        count_launches(2);
        c ^= 1;
    };
    // first the triangles that share an edge
    k_pair_pos<<<(nt + T - 1) / T, T, 0, s>>>(B.vals[cur], nt, Q.pos);
    k_pair_mates<<<(nt + T - 1) / T, T, 0, s>>>(B.tri_v, B.vals[cur], Q.pos, nt, Q.blo[0], Q.bhi[0], nullptr, Q.mate);
    k_pair_mates<<<(nt + T - 1) / T, T, 0, s>>>(B.tri_v, B.vals[cur], Q.pos, nt, Q.blo[0], Q.bhi[0], Q.mate, Q.nn);
    count_launches(3);
    merge(Q.nn, 0);
    PlocState h{};
    for (bool tail = false; !tail;) {
        if (bound <= kPlocTail) {
            k_ploc_tail<<<1, kPlocTail, 0, s>>>(st + c, Q.cid[c], Q.blo[c], Q.bhi[c], B.nodes, B.par_int, B.par_leaf);
            count_launches(1);
            tail = true;
        } else {
            for (int r = 0; r < kPlocRounds; ++r) {
                k_ploc_nn<<<(bound + kPlocT - 1) / kPlocT, kPlocT, 0, s>>>(st + c, Q.blo[c], Q.bhi[c], Q.nn);
                count_launches(1);
                merge(Q.nn, 1);
            }
        }
        e = cudaMemcpyAsync(&h, st + c, sizeof(h), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return e;
        if (h.stuck || h.count < 1 || h.count > bound) return cudaErrorUnknown;
        bound = h.count;
    }
    if (h.count != 1 || h.node_top != 0) return cudaErrorUnknown;
    e = reinsert(B, Q, nt, h.pair_top, s);
    if (e != cudaSuccess) return e;
    // the traversal stack holds at most depth-1 entries: a deeper tree is
    // replaced by the linear BVH (depth <= 95 by construction)
    e = cudaMemsetAsync(Q.total, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    k_leaf_depth<<<(nt + T - 1) / T, T, 0, s>>>(nt, B.par_int, B.par_leaf, (int*)Q.total);
    count_launches(1);
    int depth = 0;
    e = cudaMemcpyAsync(&depth, Q.total, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    if (depth >= kMaxDepth) return build_lbvh(B, d_verts, d_idx, nv, nt, eps, err, s, root_leaf, list);
    return cudaGetLastError();
}

size_t ploc_scratch_bytes(int nt)
{
    PlocBufs Q;
    return carve_ploc_scratch(nullptr, nt, Q);
}

size_t carve_ploc_scratch(void* base, int nt, PlocBufs& Q)
{
    const size_t n = (size_t)(nt > 0 ? nt : 1);
    size_t off = 0;
    auto take = [&](size_t bytes) -> void* {
        void* p = base ? (void*)((char*)base + off) : nullptr;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    for (int k = 0; k < 2; ++k) {
        Q.cid[k] = (int*)take(sizeof(int) * n);
        Q.blo[k] = (float4*)take(sizeof(float4) * n);
        Q.bhi[k] = (float4*)take(sizeof(float4) * n);
    }
    Q.nn = (int*)take(sizeof(int) * n);
    Q.flags = (uint64_t*)take(sizeof(uint64_t) * n);
    Q.pre = (uint64_t*)take(sizeof(uint64_t) * n);
    Q.sums = (uint64_t*)take(sizeof(uint64_t) * ((n + kMergeBlock - 1) / kMergeBlock + 1));
    static_assert(kMergeBlock <= kScanBlock, "one array serves both");
    Q.total = (uint64_t*)take(sizeof(uint64_t));
    Q.state = take(2 * sizeof(PlocState));
    Q.pos = (int*)Q.flags;  // the scan arrays serve split_static_moving only
    Q.mate = (int*)Q.pre;
    return off;
}

__global__ void k_classify(const int* __restrict__ idx, const uint8_t* __restrict__ vmoved, int nt, int nv,
                           uint64_t* __restrict__ fl)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    bool mv = false;
    for (int v = 0; v < 3; ++v) {
        int vi = idx[3 * (size_t)t + v];
        if (vi >= 0 && vi < nv && vmoved[vi]) mv = true;
    }
    fl[t] = mv ? 1ull : (1ull << 32);  // static count high, moving count low
}

__global__ void k_split(const uint64_t* __restrict__ fl, const uint64_t* __restrict__ pre, int nt,
                        int* __restrict__ slist, int* __restrict__ dlist)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nt) return;
    uint64_t p = pre[t];
    if (fl[t] >> 32)
        slist[p >> 32] = t;
    else
        dlist[p & 0xFFFFFFFFu] = t;
}

// Split the triangles into static (no moved vertex) and moving ones, keeping
// index order in both lists; returns the counts (synchronises the stream).
cudaError_t split_static_moving(const int* d_idx, const uint8_t* vmoved, int nt, int nv, const PlocBufs& Q,
                                int* slist, int* dlist, int* ns, int* nd, cudaStream_t s)
{
    *ns = 0;
    *nd = 0;
    if (nt <= 0) return cudaSuccess;
    const int T = 256;
    k_classify<<<(nt + T - 1) / T, T, 0, s>>>(d_idx, vmoved, nt, nv, Q.flags);
    count_launches(1);
    const int sb = (nt + kScanBlock - 1) / kScanBlock;
    k_scan64_block<<<sb, kScanT, 0, s>>>(Q.flags, Q.pre, Q.sums, nt);
    count_launches(1);
    k_scan64_small<<<1, 1024, 0, s>>>(Q.sums, sb, Q.total);
    count_launches(1);
    k_scan64_add<<<(nt + T - 1) / T, T, 0, s>>>(Q.pre, Q.sums, nt);
    count_launches(1);
    k_split<<<(nt + T - 1) / T, T, 0, s>>>(Q.flags, Q.pre, nt, slist, dlist);
    count_launches(1);
    uint64_t tot = 0;
    cudaError_t e = cudaMemcpyAsync(&tot, Q.total, sizeof(tot), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    *ns = (int)(tot >> 32);
    *nd = (int)(tot & 0xFFFFFFFFu);
    return cudaSuccess;
}

cudaError_t fill_tri_orig(const float* d_verts, const int* d_idx, const int* list, int nv, int nt, float4* tri_orig,
                          cudaStream_t s)
{
    if (nt <= 0) return cudaSuccess;
    k_fill_orig<<<(nt + 255) / 256, 256, 0, s>>>(d_verts, d_idx, list, nt, nv, tri_orig);
    count_launches(1);
    return cudaGetLastError();
}

void Bvh::release()
{
    cudaFree(scratch);
    cudaFree(pscratch);
    cudaFree(tri_v);
    cudaFree(nodes);
    *this = Bvh();
}

cudaError_t Bvh::reserve(int nt, bool ploc)
{
    if (nt <= cap_ && (!ploc || pscratch)) return cudaSuccess;
    int n = nt > cap_ ? nt : cap_;
    release();
    n = n > 0 ? n : 1;
    size_t sb = bvh_scratch_bytes(n);
    cudaError_t e = volume_malloc(&scratch, sb);
    if (e != cudaSuccess) return e;
    e = volume_malloc((void**)&tri_v, sizeof(float4) * 3 * (size_t)n);
    if (e != cudaSuccess) return e;
    e = volume_malloc((void**)&nodes, sizeof(BNode) * (size_t)n);
    if (e != cudaSuccess) return e;
    size_t pb = 0;
    if (ploc) {
        WideBufs W;
        pb = std::max(ploc_scratch_bytes(n), carve_wide_scratch(nullptr, n, W));  // one after the other
        e = volume_malloc(&pscratch, pb);
        if (e != cudaSuccess) return e;
        carve_ploc_scratch(pscratch, n, pbufs);
    }
    carve_bvh_scratch(scratch, n, bufs);
    bufs.tri_v = tri_v;
    bufs.nodes = nodes;
    cap_ = n;
    bytes_ = sb + pb + sizeof(float4) * 3 * (size_t)n + sizeof(BNode) * (size_t)n;
    return cudaSuccess;
}

cudaError_t Bvh::build(const float* d_verts, const int* d_idx, int nv, int nt, float eps, int* err, cudaStream_t s,
                       const int* list)
{
    n_tris = 0;
    if (nt == 0) return cudaSuccess;
    cudaError_t e = reserve(nt, true);  // may reset every member
    if (e != cudaSuccess) return e;
    n_tris = nt;
    return build_ploc(bufs, pbufs, d_verts, d_idx, nv, nt, eps, err, s, &root_leaf, list);
}

cudaError_t Bvh::build_moving(const float* d_verts, const int* d_idx, int nv, int nt, float eps, int* err, cudaStream_t s,
                              const int* list, float4* tris, BNode* nodes_out, int node_off, int tri_off, float4* tri_orig)
{
    n_tris = 0;
    if (nt == 0) return cudaSuccess;
    cudaError_t e = reserve(nt, false);
    if (e != cudaSuccess) return e;
    n_tris = nt;
    BvhBufs B = bufs;
    B.tri_v = tris;
    B.nodes = nodes_out;
    return build_lbvh(B, d_verts, d_idx, nv, nt, eps, err, s, &root_leaf, list, node_off, tri_off, tri_orig);
}

}  // namespace adgi
