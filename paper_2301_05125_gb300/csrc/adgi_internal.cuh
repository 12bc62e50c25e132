// adgi_internal.cuh -- device data layout and inline device code shared by the
// library's kernels (sm_103a).  Nothing here is shared with the CPU oracle.
//
// Exactness: every floating-point step whose result becomes an integer or a
// discrete decision (ray directions, the watertight hit test, shadow
// visibility, the lit test, the quantised heuristics, texel binning) is
// written with the *_rn intrinsics, which are never fused or reordered, so it
// reproduces IEEE single precision bit for bit.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_fp16.h>

#include "../../include/adgi.h"

namespace adgi {

constexpr int kPilots = 8;
constexpr int kMaxLights = 64;
constexpr uint32_t kMiss = 0xFFFFFFFFu;
constexpr uint32_t kBackBit = 0x80000000u;

// ----------------------------------------------------------------- device data
struct Light {
    int kind;
    float v[3];
    float rgb[3];
};

// BVH node: the boxes of both children (so one fetch decides both) and the
// child references; a child >= 0 is an internal node, < 0 is ~(triangle slot).
struct __align__(16) BNode {
    float4 a;  // c0.lo.xyz, c0.hi.x
    float4 b;  // c0.hi.yz, c1.lo.xy
    float4 c;  // c1.lo.z, c1.hi.xyz
    int4 d;    // left, right, -, -
};

// The scene: a static part (quality BVH, built once) and a moving part
// (linear BVH, rebuilt when vertices move), in one node array and one
// triangle array.  The static part's ns triangles occupy slots [0, ns) and
// its internal nodes [0, ns-1); the moving part's triangles follow at slot
// ns and its nodes at node max(ns-1, 0), with child references relocated
// to these global indices, so a traversal needs no per-part pointers.  Hits
// are ranked over both by (t, original triangle index).
constexpr int kWide4Stack = 160;  // entries of the 4-wide traversal's stack, three a level

struct SceneDev {
    const float4* w4;       // 4-wide tree of the static part (7 float4 a node), or null: the binary tree
    const float4* wq;       // its leaves: one or two triangles each (4 float4 a record)
    const BNode* nodes;     // internal nodes of both parts
    const float4* tri_v;    // both parts' triangles in BVH order, .w of v0 = original index
    int root[2];            // root node of each part's tree (-1: fewer than two triangles)
    int leaf[2];            // slot of a part's only triangle (-1: none, or a tree)
    int max_iter;           // traversal step limit (a correct tree needs fewer node visits)
    int n_tris;
    int n_verts;
    const float4* tri_orig; // [n_tris*3] vertices in original order (shading normal)
    const float* albedo;    // [n_tris*3]
    int* err;               // anomaly flags (kErr*), 0 when all is well
};

constexpr int kErrTraversal = 1;  // a traversal exceeded max_iter
constexpr int kErrRayRange = 2;   // a probe's ray range exceeded the buffers
constexpr int kErrBvh = 4;        // the bottom-up box pass exceeded its depth bound
constexpr int kErrIndex = 8;      // a triangle referenced a vertex outside the array

struct FrameConst {
    uint64_t pilot_key;     // sm(sm(seed) ^ pair)
    float R[9];             // main-ray rotation
    float sky[3];
    int n_lights;
    int even;               // first frame of a pair: pilots are blended
    int pair_valid;         // the previous frame was the first of this pair
    int has_camera;
    float cam[3];
    float cam_k;
    uint64_t mh_key;        // Metropolis counters of this frame: sm(sm(seed ^ 'METRO') ^ frame)
    uint64_t dyn_key;       // the dynamic chains' counters: sm(sm(seed ^ 'DYNAM') ^ frame)
    int has_clip;           // clip volumes from clip[] (with has_camera)
    float clip[16];         // row-major view-projection
};

struct VolConst {
    float origin[3], spacing[3];
    int dims[3];
    int P;
    int n_irr, n_dep, Ti, Td;
    float tmin;             // (float)(1e-4 * s)
    float depth_max;
    float qv_scale;         // (float)(256 / s)
    float qc_scale;         // (float)(64 / s)
    float var_min;          // (float)(1e-6 * s^2): the Chebyshev minimum variance
    float var_rel;          // optional further floor var_rel * mu2 (0: none)
    float hyst;
    int theta;
    int m0, rays_max, rays_avg;
    int fp16;               // atlas storage: 0 FP32, 1 FP16 (RN), 2 FP16 (SR), 3 packed 32-bit codes
    const float* ctab;      // packed code values: [512] 9-bit, [256] 8-bit, [8192] 13-bit mean, [8192] 13-bit square
    float s_f;              // (float) cage diagonal: the packed visibility normaliser
    uint32_t R_main;        // main-ray buffer length
    int* err;               // anomaly flags (kErr*)
    int dyn;                // dynamic chains on (Metropolis mode with dyn_ratio > 0)
    float hyst_dyn;         // hysteresis of the dynamic rays' batch step
    const uint8_t* cls;     // [P] clip volume of this frame: 2 V_in, 1 V_out - V_in, 0 outside
    int p_lo, p_hi;         // probes this launch works on: [0, P), or one rank's slab of a split update
};

// This frame's dynamic rays (dynamic chains over virtual proxies), grouped
// by probe: probe p sends, for every octant o whose proxy cell is traced,
// one ray through the centre of each irradiance texel listed for o.
struct DynRays {
    const uint32_t* off;      // [P+1] first dynamic ray of each probe; off[P] = rays this frame
    const uint8_t* incl;      // [Pp*8] 1: the cell (proxy, octant) is traced
    const int* ntex;          // [8] texels whose centre lies in each octant
    const int* tex_t;         // [8][n_irr^2] their tile indices
    const float4* tex_dir;    // [8][n_irr^2] their centre directions
    int dp[3];                // proxy grid
};

// ----------------------------------------------------------------- exact FP32
__device__ __forceinline__ float fa(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fs(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fm(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fd(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float fsq(float a) { return __fsqrt_rn(a); }
__device__ __forceinline__ float dot3x(float ax, float ay, float az, float bx, float by, float bz)
{
    return fa(fa(fm(ax, bx), fm(ay, by)), fm(az, bz));
}

__host__ __device__ __forceinline__ uint64_t splitmix(uint64_t x)
{
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// probe position (FP32): origin + spacing * index
__device__ __forceinline__ float3 probe_pos(const VolConst& V, int p)
{
    int ix = p % V.dims[0];
    int iy = (p / V.dims[0]) % V.dims[1];
    int iz = p / (V.dims[0] * V.dims[1]);
    return make_float3(fa(V.origin[0], fm(V.spacing[0], (float)ix)), fa(V.origin[1], fm(V.spacing[1], (float)iy)),
                       fa(V.origin[2], fm(V.spacing[2], (float)iz)));
}

// q_c of probe p (Eq. cameraD): 1023 within cam_k of the camera, else the
// LUT bin of width s/64 at the distance beyond cam_k; 1023 without a camera
__device__ __forceinline__ uint32_t qc_of_probe(const VolConst& V, const FrameConst& F,
                                                const uint16_t* __restrict__ lut_c, int p)
{
    if (!F.has_camera) return 1023u;
    float3 pp = probe_pos(V, p);
    float dx = fs(pp.x, F.cam[0]), dy = fs(pp.y, F.cam[1]), dz = fs(pp.z, F.cam[2]);
    float dist = fsq(dot3x(dx, dy, dz, dx, dy, dz));
    if (dist < F.cam_k) return 1023u;
    float q = fm(fs(dist, F.cam_k), V.qc_scale);
    uint32_t i = q < 4095.0f ? (uint32_t)floorf(q) : 4095u;
    return __ldg(lut_c + i);
}

// Pilot direction of (probe, octant) for the frame pair encoded in key:
// a uniform point of the octant's simplex from a 64-bit hash, normalised.
__device__ __forceinline__ float3 pilot_dir(uint64_t key, uint32_t probe, int o)
{
    uint64_t h = splitmix(key ^ ((uint64_t)probe * 8u + (uint64_t)o));
    const float k24 = 5.9604644775390625e-08f;
    float u1 = fm(__uint2float_rn((uint32_t)(h >> 40)), k24);
    float u2 = fm(__uint2float_rn((uint32_t)((h >> 16) & 0xFFFFFFu)), k24);
    if (fa(u1, u2) > 1.0f) {
        float a = fs(1.0f, u2), b = fs(1.0f, u1);
        u1 = a;
        u2 = b;
    }
    float x = u1, y = u2, z = fs(fs(1.0f, u1), u2);
    if (o & 1) x = -x;
    if (o & 2) y = -y;
    if (o & 4) z = -z;
    float l = fsq(dot3x(x, y, z, x, y, z));
    return make_float3(fd(x, l), fd(y, l), fd(z, l));
}

__device__ __forceinline__ float3 rotate(const float* R, float4 s)
{
    return make_float3(fa(fa(fm(R[0], s.x), fm(R[1], s.y)), fm(R[2], s.z)),
                       fa(fa(fm(R[3], s.x), fm(R[4], s.y)), fm(R[5], s.z)),
                       fa(fa(fm(R[6], s.x), fm(R[7], s.y)), fm(R[8], s.z)));
}

// ----------------------------------------------------------------- octahedral
__device__ __forceinline__ float sgnf(float v) { return v >= 0.0f ? 1.0f : -1.0f; }

__device__ __forceinline__ float2 oct_encode_x(float3 w)
{
    float l1 = fa(fa(fabsf(w.x), fabsf(w.y)), fabsf(w.z));
    float px = fd(w.x, l1), py = fd(w.y, l1);
    if (w.z < 0.0f) {
        float qx = fm(fs(1.0f, fabsf(py)), sgnf(px));
        float qy = fm(fs(1.0f, fabsf(px)), sgnf(py));
        px = qx;
        py = qy;
    }
    return make_float2(px, py);
}

// unit direction of octahedral coordinates (ux, uy), exact FP32
__device__ __forceinline__ float3 oct_decode_x(float ux, float uy)
{
    float x = ux, y = uy;
    const float z = fs(fs(1.0f, fabsf(x)), fabsf(y));
    if (z < 0.0f) {
        const float fx = fm(fs(1.0f, fabsf(uy)), sgnf(ux));
        const float fy = fm(fs(1.0f, fabsf(ux)), sgnf(uy));
        x = fx;
        y = fy;
    }
    const float l = fsq(dot3x(x, y, z, x, y, z));
    return make_float3(fd(x, l), fd(y, l), fd(z, l));
}

// direction through the centre of interior texel (cx, cy) of an n x n
// octahedral grid: u = (c + 1/2)/n * 2 - 1 per axis, FP32 in that order
__device__ __forceinline__ float3 texel_centre_dir(int cx, int cy, int n)
{
    const float fn = (float)n;
    return oct_decode_x(fs(fm(fd(fa((float)cx, 0.5f), fn), 2.0f), 1.0f), fs(fm(fd(fa((float)cy, 0.5f), fn), 2.0f), 1.0f));
}

// nearest interior texel, as row*(n+2)+col with both in 1..n
__device__ __forceinline__ int texel_of(float2 p, int n)
{
    float fn = (float)n;
    int cx = (int)floorf(fm(fm(fa(p.x, 1.0f), 0.5f), fn));
    int cy = (int)floorf(fm(fm(fa(p.y, 1.0f), 0.5f), fn));
    cx = min(max(cx, 0), n - 1);
    cy = min(max(cy, 0), n - 1);
    return (cy + 1) * (n + 2) + (cx + 1);
}

// ----------------------------------------------------------------- watertight
struct WRay {
    float ox, oy, oz;
    int kz;  // the dominant axis of the direction; the other two follow it cyclically
    bool neg;  // its component is negative
    float Sx, Sy, Sz;
};

__device__ __forceinline__ float comp(float x, float y, float z, int k) { return k == 0 ? x : (k == 1 ? y : z); }

// The test's definition swaps the two other axes when the dominant component
// is negative (so that det > 0 is a front face).  Swapping them only negates
// U, V, W, det and T exactly -- products commute and a - b = -(b - a) in IEEE
// arithmetic -- so the axes stay in cyclic order here and the sign of det is
// flipped instead.
__device__ __forceinline__ WRay wray(float3 o, float3 d)
{
    WRay r;
    r.ox = o.x;
    r.oy = o.y;
    r.oz = o.z;
    int kz = 0;
    float m = fabsf(d.x);
    if (fabsf(d.y) > m) {
        kz = 1;
        m = fabsf(d.y);
    }
    if (fabsf(d.z) > m) kz = 2;
    const float dz = comp(d.x, d.y, d.z, kz);
    r.kz = kz;
    r.neg = dz < 0.0f;
    r.Sx = fd(comp(d.y, d.z, d.x, kz), dz);
    r.Sy = fd(comp(d.z, d.x, d.y, kz), dz);
    r.Sz = fd(1.0f, dz);
    return r;
}

// a vertex in the ray's sheared frame: (x, y) where the ray is the origin,
// z along the dominant axis (not scaled by Sz)
__device__ __forceinline__ float3 wvert(const WRay& r, float4 v)
{
    const float x = fs(v.x, r.ox), y = fs(v.y, r.oy), z = fs(v.z, r.oz);
    const float kz = comp(x, y, z, r.kz);
    return make_float3(fs(comp(y, z, x, r.kz), fm(r.Sx, kz)), fs(comp(z, x, y, r.kz), fm(r.Sy, kz)), kz);
}

__device__ __forceinline__ float wedge(float3 p, float3 q) { return fs(fm(p.x, q.y), fm(p.y, q.x)); }
__device__ __forceinline__ float wedge64(float3 p, float3 q)
{
    return __double2float_rn(__dsub_rn(__dmul_rn((double)p.x, (double)q.y), __dmul_rn((double)p.y, (double)q.x)));
}

// the line misses the triangle: the edge functions have both signs
__device__ __forceinline__ bool wmiss(float U, float V, float W)
{
    return fminf(fminf(U, V), W) < 0.0f && fmaxf(fmaxf(U, V), W) > 0.0f;
}

// t and det from the edge functions and the vertices' z, in vertex order
__device__ __forceinline__ bool wdist(const WRay& r, float U, float V, float W, float az, float bz, float cz, float& t,
                                      float& det)
{
    det = fa(fa(U, V), W);
    if (det == 0.0f) return false;
    const float T = fa(fa(fm(U, fm(r.Sz, az)), fm(V, fm(r.Sz, bz))), fm(W, fm(r.Sz, cz)));
    t = fd(T, det);
    if (r.neg) det = -det;
    return true;
}

// Woop-Benthin-Wald watertight test.  Returns true when the ray's line crosses
// the triangle, with t and det; det > 0 is a front-face hit.
__device__ __forceinline__ bool wtri(const WRay& r, float4 A4, float4 B4, float4 C4, float& t, float& det)
{
    const float3 A = wvert(r, A4), B = wvert(r, B4), C = wvert(r, C4);
    float U = wedge(C, B), V = wedge(A, C), W = wedge(B, A);
    if (U == 0.0f || V == 0.0f || W == 0.0f) U = wedge64(C, B), V = wedge64(A, C), W = wedge64(B, A);
    if (wmiss(U, V, W)) return false;
    return wdist(r, U, V, W, A.z, B.z, C.z, t, det);
}

constexpr float kBoxSlack = 1.0001f;  // pruning slack on the best t (conservative)
// LBVH depth is at most 95 (63 key bits + 32 index bits); a PLOC tree can be
// deeper, so its builder checks the depth against kMaxDepth.  The near-first
// traversal stack holds at most one pending entry per level.
constexpr int kMaxDepth = 96;
constexpr int kStack = kMaxDepth;
constexpr int kTravStack = kWide4Stack + 8 > kStack + 2 ? kWide4Stack + 8 : kStack + 2;  // one array serves both traversals

// A load of data that an earlier phase of the same launch may have written.
// The ordinary kernels take the read-only (non-coherent) path; the
// persistent batched tick (tick.cu), whose phases follow one another inside
// one launch, takes a plain coherent load, which its grid barriers order.
template <bool kLive, typename T>
__device__ __forceinline__ T ldl(const T* p)
{
    if constexpr (kLive)
        return *p;
    else
        return __ldg(p);
}

// Traversal of the two-part scene as one flat loop over one stack of
// global node indices.  The loop has no early exit, so the lanes of a warp
// reconverge every iteration.

// One traversal in flight.  Closest hit: t in (tmin, tmax], ranked by
// (t, original index) -- a strict order, so the result does not depend on
// the traversal order.  Any hit: t in (tmin, tmax), stops at the first.
// The state is scalars only, so it can live in registers; the node stack is
// a separate local array.
struct Trav {
    WRay wr;
    float3 o, inv, oi;      // oi = o * inv: slab tests as one FMA per plane
    float tmin, tmax, lim;  // lim: box pruning bound
    float t_best, best_det;
    int best_orig;
    bool found;
    int sp, iter;
    int next;  // the node to visit next (-1: take the stack top); saves a push and a pop per single-child step
};

// Conservative slab test of one box against [0, lim] with the plane
// distances as fma(plane, 1/d, -o/d): the rounding of o/d moves a plane by
// about 2^-24 |o|, far inside the boxes' enlargement (>= 1e-5 of the
// largest coordinate), so no box that the ray enters is culled.  NaNs
// (0 * inf) drop out of fminf/fmaxf, which keeps the test conservative.
__device__ __forceinline__ bool slab_fma(float lox, float loy, float loz, float hix, float hiy, float hiz, float3 inv,
                                         float3 oi, float lim, float& tnear)
{
    float tx0 = fmaf(lox, inv.x, -oi.x), tx1 = fmaf(hix, inv.x, -oi.x);
    float ty0 = fmaf(loy, inv.y, -oi.y), ty1 = fmaf(hiy, inv.y, -oi.y);
    float tz0 = fmaf(loz, inv.z, -oi.z), tz1 = fmaf(hiz, inv.z, -oi.z);
    float tn = fmaxf(fmaxf(fminf(tx0, tx1), fminf(ty0, ty1)), fmaxf(fminf(tz0, tz1), 0.0f));
    float tf = fminf(fminf(fmaxf(tx0, tx1), fmaxf(ty0, ty1)), fminf(fmaxf(tz0, tz1), lim));
    tnear = tn;
    return tn <= tf;
}

// a triangle that the ray's line crosses at tt
__device__ __forceinline__ void trav_take(Trav& T, float tt, float det, int orig, bool any)
{
    if (!(tt > T.tmin)) return;
    if (any) {
        if (tt < T.tmax) T.found = true;
        return;
    }
    const bool better = T.found ? (tt < T.t_best || (tt == T.t_best && orig < T.best_orig)) : (tt <= T.tmax);
    if (better) {
        T.found = true;
        T.t_best = tt;
        T.best_orig = orig;
        T.best_det = det;
    }
}

// the triangle at slot `slot` of the BVH-ordered array (kLive: it may have
// been written earlier in the same launch, see ldl)
template <bool kLive = false>
__device__ __forceinline__ void trav_tri(Trav& T, const float4* tri_v, int slot, bool any, uint32_t* ntri)
{
    if (ntri) ++*ntri;
    const float4* tv = tri_v + 3 * (size_t)slot;
    float4 A = ldl<kLive>(tv), Bv = ldl<kLive>(tv + 1), C = ldl<kLive>(tv + 2);
    float tt, det;
    if (wtri(T.wr, A, Bv, C, tt, det)) trav_take(T, tt, det, __float_as_int(A.w), any);
}

// A leaf of the 4-wide tree: triangle (v0, v1, v2) and, where the record has
// two, triangle (v0, v2, v3), which share the edge v0 v2 (opposite
// directions).  The two tests take wtri's steps on each triangle, operation
// by operation, but transform four vertices instead of six and use the shared
// edge's function for both (its sign flipped, exactly).  .w: the two original
// indices in v0 and v2 (-1: no second triangle), in v1 and v3 the rotations
// that bring the triangles back to their own vertex order, in which det and T
// are summed.  A record of one triangle is tested with a second one all the
// same (its result is dropped), the other half of its parallelogram: with v3 = v2 an
// edge was zero in every test, and the double precision that asks for took a
// million rays through 50,000 triangles without a common edge from 1.07 to
// 2.95 ms.  (Asking for the triangle here before the zeros cost the other
// scenes 0.6 to 1.5 %.)
__device__ __forceinline__ void trav_leaf(Trav& T, const float4* wq, int rec, bool any, uint32_t* ntri)
{
    const float4* q = reinterpret_cast<const float4*>(reinterpret_cast<const char*>(wq) + 64u * (uint32_t)rec);
    const float4 q0 = __ldg(q), q1 = __ldg(q + 1), q2 = __ldg(q + 2), q3 = __ldg(q + 3);
    const float3 v0 = wvert(T.wr, q0), v1 = wvert(T.wr, q1), v2 = wvert(T.wr, q2), v3 = wvert(T.wr, q3);
    float U0 = wedge(v2, v1), V0 = wedge(v0, v2), W0 = wedge(v1, v0);  // (v0, v1, v2)
    float U1 = wedge(v3, v2), V1 = wedge(v0, v3), W1 = -V0;             // (v0, v2, v3)
    const int id1 = __float_as_int(q2.w);
    if (ntri) *ntri += id1 >= 0 ? 2u : 1u;
    // an edge through the ray: that triangle's edge functions in double
    if (U0 == 0.0f || V0 == 0.0f || W0 == 0.0f) U0 = wedge64(v2, v1), V0 = wedge64(v0, v2), W0 = wedge64(v1, v0);
    if (U1 == 0.0f || V1 == 0.0f || W1 == 0.0f) U1 = wedge64(v3, v2), V1 = wedge64(v0, v3), W1 = wedge64(v2, v0);
    // Few leaves are hit, and those mostly in one of their two triangles: the
    // rest of the test is one piece of code for either, run by the lanes with a
    // hit together (a copy for each triangle ran them one after the other:
    // nearest hit 1.29 -> 1.25 ms on the tunnel scene, 4.10 -> 4.02 on the
    // scaled one, 2 % fewer instructions).
    bool in0 = !wmiss(U0, V0, W0), in1 = id1 >= 0 && !wmiss(U1, V1, W1);
    while (in0 || in1) {
        float U = in0 ? U0 : U1, V = in0 ? V0 : V1, W = in0 ? W0 : W1;
        float az = v0.z, bz = in0 ? v1.z : v2.z, cz = in0 ? v2.z : v3.z;
        const int ro = __float_as_int(in0 ? q1.w : q3.w), id = in0 ? __float_as_int(q0.w) : id1;
        if (in0)
            in0 = false;
        else
            in1 = false;
        if (ro == 1) {  // the triangle's own order is (b, c, a)
            const float u = U, x = az;
            U = V, V = W, W = u;
            az = bz, bz = cz, cz = x;
        } else if (ro == 2) {  // (c, a, b)
            const float w = W, x = cz;
            W = V, V = U, U = w;
            cz = bz, bz = az, az = x;
        }
        float tt, det;
        if (wdist(T.wr, U, V, W, az, bz, cz, tt, det)) {
            trav_take(T, tt, det, id, any);
            if (any && T.found) return;
        }
    }
}

// set up a traversal
__device__ __forceinline__ void trav_init(Trav& T, float3 o, float3 d, float tmin, float tmax, bool any)
{
    T.wr = wray(o, d);
    T.o = o;
    // The box test uses 1/d with components below 1e-20 in magnitude raised
    // to +-1e-20: a zero component would make o * inv infinite and the FMA
    // slab form inf - inf = NaN, rejecting every box (axis-aligned rays: an
    // axis-aligned sun, texel-centre directions on the octahedral diamond).
    // The raised component moves the ray by 1e-20 t along that axis, far
    // below the boxes' enlargement, so the test stays conservative; the
    // triangle test keeps the exact direction.
    const float kTiny = 1e-20f;
    const float dx = fabsf(d.x) < kTiny ? copysignf(kTiny, d.x) : d.x;
    const float dy = fabsf(d.y) < kTiny ? copysignf(kTiny, d.y) : d.y;
    const float dz = fabsf(d.z) < kTiny ? copysignf(kTiny, d.z) : d.z;
    T.inv = make_float3(1.0f / dx, 1.0f / dy, 1.0f / dz);
    T.oi = make_float3(o.x * T.inv.x, o.y * T.inv.y, o.z * T.inv.z);
    T.next = -1;
    T.tmin = tmin;
    T.tmax = tmax;
    T.lim = any ? (isinf(tmax) ? tmax : tmax * kBoxSlack) : tmax * kBoxSlack;
    T.t_best = tmax;
    T.best_det = 0.0f;
    T.best_orig = 0x7FFFFFFF;
    T.found = false;
    T.sp = 0;
    T.iter = 0;
}

// The parts that the binary traversal walks (the static part only when it
// has no 4-wide tree): single-triangle parts are tested here, trees pushed.
// kLive: the moving part may have been rebuilt earlier in the same launch
// (its nodes and triangles are read with ldl).
template <bool kLive = false>
__device__ __forceinline__ void trav_roots(Trav& T, int* stack, const SceneDev& S, bool any, uint32_t* ntri)
{
    if (S.n_tris == 0) return;
    for (int pi = 1; pi >= (S.w4 ? 1 : 0); --pi) {
        const int root = pi ? S.root[1] : S.root[0], leaf = pi ? S.leaf[1] : S.leaf[0];
        if (root >= 0)
            stack[T.sp++] = root;
        else if (leaf >= 0)
            trav_tri<kLive>(T, S.tri_v, leaf, any, ntri);
    }
    if (any && T.found) T.sp = 0;
}

// one node visit; false once the traversal is over
template <bool kLive = false>
__device__ __forceinline__ bool trav_step(Trav& T, int* stack, const SceneDev& S, bool any,
                                          uint32_t* nbox = nullptr, uint32_t* ntri = nullptr)
{
    if (T.next < 0 && T.sp <= 0) return false;
    if (++T.iter > S.max_iter) {
        atomicOr(S.err, kErrTraversal);
        T.sp = 0;
        T.next = -1;
        return false;
    }
    if (nbox) *nbox += 2;
    const int e = T.next >= 0 ? T.next : stack[--T.sp];
    T.next = -1;
    const BNode* nd = S.nodes + e;
    float4 a = ldl<kLive>(&nd->a), b = ldl<kLive>(&nd->b), c = ldl<kLive>(&nd->c);
    int4 ch = ldl<kLive>(&nd->d);
    const float lim = any ? T.lim : T.t_best * kBoxSlack;
    float t0, t1;
    const bool h0 = slab_fma(a.x, a.y, a.z, a.w, b.x, b.y, T.inv, T.oi, lim, t0);
    const bool h1 = slab_fma(b.z, b.w, c.x, c.y, c.z, c.w, T.inv, T.oi, lim, t1);
    if (h0 && ch.x < 0) trav_tri<kLive>(T, S.tri_v, ~ch.x, any, ntri);
    if (h1 && ch.y < 0) trav_tri<kLive>(T, S.tri_v, ~ch.y, any, ntri);
    const bool i0 = h0 && ch.x >= 0, i1 = h1 && ch.y >= 0;
    if (i0 && i1) {  // the near child next, the far one on the stack
        const bool first0 = t0 <= t1;
        if (T.sp < kStack + 2) {
            stack[T.sp++] = first0 ? ch.y : ch.x;
            T.next = first0 ? ch.x : ch.y;
        } else {
            atomicOr(S.err, kErrTraversal);  // cannot happen: depths are bounded by the builders
        }
    } else if (i0 || i1) {
        T.next = i0 ? ch.x : ch.y;
    }
    if (any && T.found) {  // a blocker ends a shadow ray
        T.sp = 0;
        T.next = -1;
    }
    return T.next >= 0 || T.sp > 0;
}

__device__ __forceinline__ uint32_t trav_hit(const Trav& T)
{
    return T.found ? ((uint32_t)T.best_orig | (T.best_det < 0.0f ? kBackBit : 0u)) : kMiss;
}

__device__ __forceinline__ float4 w4_load(const float4* w4, uint32_t byte)
{
    return __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const char*>(w4) + byte));
}

// plane distances of the four children, fma(plane, 1/d, -o/d), as two-wide
// FMAs: a float4 of planes is two aligned register pairs, so the pairs need
// no moves (10 fewer instructions a visit: nearest hit -3 %)
__device__ __forceinline__ void plane4(float4 v, float inv, float noi, float* out)
{
    const float2 i2 = make_float2(inv, inv), o2 = make_float2(noi, noi);
    const float2 a = __ffma2_rn(make_float2(v.x, v.y), i2, o2), b = __ffma2_rn(make_float2(v.z, v.w), i2, o2);
    out[0] = a.x, out[1] = a.y, out[2] = b.x, out[3] = b.y;
}

// One visit of the static part's 4-wide tree without its leaf tests: node
// `node`, the traversal's group and stack (depth sp), the byte offsets of the
// near planes in a node (the far planes' follow).  The hit leaves are
// records leaf0 + k for the bits k of `leaves`.  Returns the node to visit
// next, or -1 when none is left.
//   A node's internal children fill its first slots and are consecutive
// nodes, so a child is named by its slot, and a sort key is one word: the
// distance's bits (non-negative, so they order as integers) with the slot in
// the two lowest bits.  The order of nearly equal distances is then by slot,
// which changes no hit.
__device__ __forceinline__ int trav4_inner(Trav& T, int* stack, int& sp, int node, const SceneDev& S, bool any,
                                           uint32_t ox, uint32_t oy, uint32_t oz, uint32_t* nbox, uint32_t& leaves,
                                           int& leaf0)
{
    leaves = 0;
    if (nbox) *nbox += 4;
    const uint32_t at = 112u * (uint32_t)node;
    float nx[4], ny[4], nz[4], fx[4], fy[4], fz[4];
    const float4 vnx = w4_load(S.w4, at + ox), vfx = w4_load(S.w4, at + 16u - ox);
    const float4 vny = w4_load(S.w4, at + oy), vfy = w4_load(S.w4, at + 80u - oy);
    const float4 vnz = w4_load(S.w4, at + oz), vfz = w4_load(S.w4, at + 144u - oz);
    const float4 r4 = w4_load(S.w4, at + 96u);  // first child, first leaf, child count
    const int first = __float_as_int(r4.x), ni = __float_as_int(r4.z);
    plane4(vnx, T.inv.x, -T.oi.x, nx);
    plane4(vfx, T.inv.x, -T.oi.x, fx);
    plane4(vny, T.inv.y, -T.oi.y, ny);
    plane4(vfy, T.inv.y, -T.oi.y, fy);
    plane4(vnz, T.inv.z, -T.oi.z, nz);
    plane4(vfz, T.inv.z, -T.oi.z, fz);
    const float lim = any ? T.lim : T.t_best * kBoxSlack;
    uint32_t key[4], hits = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float tn = fmaxf(fmaxf(nx[k], ny[k]), fmaxf(nz[k], 0.0f));
        const float tf = fminf(fminf(fx[k], fy[k]), fminf(fz[k], lim));
        const bool hit = tn <= tf;
        if (hit) hits |= 1u << k;
        // closest hit: nearest entry first (least key).  Any hit: only the
        // first place is sorted, and it goes to the child holding the longest
        // stretch of the ray (greatest key), the likeliest to hold a blocker
        // (measured: shadow rays 2-7 % faster than nearest first).
        key[k] = hit && k < ni ? ((__float_as_uint(any ? tf - tn : tn) & ~3u) | (uint32_t)k) : (any ? 0u : ~0u);
    }
    leaves = hits >> ni;
    leaf0 = __float_as_int(r4.y);
    hits &= (1u << ni) - 1u;
    if (hits == 0u) return sp == 0 ? -1 : stack[--sp];
    if (any) {
        const uint32_t b = max(max(key[0], key[1]), max(key[2], key[3])) & 3u;
        hits &= ~(1u << b);
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (hits & (1u << k)) stack[sp++] = first + k;
        return first + (int)b;
    }
#define ADGI_CSWAP(i, j)                         \
    {                                            \
        const uint32_t lo = min(key[i], key[j]); \
        key[j] = max(key[i], key[j]);            \
        key[i] = lo;                             \
    }
    ADGI_CSWAP(0, 1)
    ADGI_CSWAP(2, 3)
    ADGI_CSWAP(0, 2)
    ADGI_CSWAP(1, 3)
    ADGI_CSWAP(1, 2)
#undef ADGI_CSWAP
    if (key[3] != ~0u) stack[sp++] = first + (int)(key[3] & 3u);
    if (key[2] != ~0u) stack[sp++] = first + (int)(key[2] & 3u);
    if (key[1] != ~0u) stack[sp++] = first + (int)(key[1] & 3u);
    return first + (int)(key[0] & 3u);
}

// The static part's 4-wide tree (T set up by trav_init): from the root, each
// visit tests the four child boxes with the near / far planes of each axis
// read by the sign of the ray direction (so an entry distance is a max and an
// exit distance a min of three FMAs) and continues with the nearest hit
// internal child; the other hit internal children are pushed, farthest
// first (closest hit).
//   The kernels are bound by instruction issue at a third of the lanes: in
// most visits of a warp two or three lanes hit a leaf, and testing it at once
// runs the triangle test for them alone, at about the cost of the visit
// itself.  So a lane makes kLeafVisits visits, whatever leaves they hit, and
// then tests all of them: the triangle tests run a third as often with three
// times the lanes, no lane ever waits for another, and the pruning bound is
// at most two visits late.  Measured on the tunnel / scaled scenes (GB300,
// ms; visits per leaf test 2, 3, 4): nearest hit 0.86, 0.84, 0.96 / 2.67,
// 2.58, 2.76; shadow rays 0.65, 0.62, 0.65 / 1.70, 1.62, 1.64 (with leaves of
// one triangle and a deeper tree, 1 visit: 13 % above 3; 5 visits: 12 %
// above).  (As a loop over one copy of the visit, three visits were 7 %
// slower: the unrolled copies' instructions still fit.)
// The pruning bound and the (t, index) ranking are those of trav_step, and
// the hit is the least (t, index) over the same candidates, so it is the
// same in any visiting order.
constexpr int kLeafVisits = 3;

__device__ __forceinline__ void trav4(Trav& T, int* stack, const SceneDev& S, bool any, uint32_t* nbox = nullptr,
                                      uint32_t* ntri = nullptr)
{
    const uint32_t ox = T.inv.x >= 0.0f ? 0u : 16u, oy = T.inv.y >= 0.0f ? 32u : 48u, oz = T.inv.z >= 0.0f ? 64u : 80u;
    int node = 0, sp = 0;
    while (node >= 0) {
        // both bounds once for all of the round's visits, each of which pushes
        // three at most (tested in every visit, nearest hits took 6 % longer)
        T.iter += kLeafVisits;
        if (T.iter > S.max_iter || sp + 3 * kLeafVisits > kTravStack) {  // the builder bounds both: cannot happen
            atomicOr(S.err, kErrTraversal);
            break;
        }
        uint32_t m = 0;  // hit leaves: four bits a visit
        int leaf0[kLeafVisits];
#pragma unroll
        for (int v = 0; v < kLeafVisits; ++v) {
            uint32_t hit = 0;
            leaf0[v] = 0;
            if (node >= 0) node = trav4_inner(T, stack, sp, node, S, any, ox, oy, oz, nbox, hit, leaf0[v]);
            m |= hit << (4 * v);
        }
        while (m) {
            const int k = __ffs(m) - 1;
            m &= m - 1u;
            int base = leaf0[0];
#pragma unroll
            for (int v = 1; v < kLeafVisits; ++v)
                if (k >= 4 * v) base = leaf0[v] - 4 * v;
            trav_leaf(T, S.wq, base + k, any, ntri);
            if (any && T.found) return;
        }
    }
}

// nearest hit with t in (tmin, tmax] (one thread, one ray); kLive: as for
// trav_roots
template <bool kLive = false>
__device__ __forceinline__ void trace_closest(const SceneDev& S, float3 o, float3 d, float tmin, float tmax,
                                              float& t_best, uint32_t& hit_best, uint32_t* nbox = nullptr,
                                              uint32_t* ntri = nullptr)
{
    Trav T;
    int stack[kTravStack];  // of the 4-wide traversal, then of the binary one
    trav_init(T, o, d, tmin, tmax, false);
    if (S.w4) trav4(T, stack, S, false, nbox, ntri);  // the static part's 4-wide tree first, then the moving part
    trav_roots<kLive>(T, stack, S, false, ntri);
    while (trav_step<kLive>(T, stack, S, false, nbox, ntri)) {
    }
    t_best = T.t_best;
    hit_best = trav_hit(T);
}

// any hit with t in (tlo, thi): shadow visibility (one thread, one ray)
template <bool kLive = false>
__device__ __forceinline__ bool trace_any(const SceneDev& S, float3 o, float3 d, float tlo, float thi,
                                          uint32_t* nbox = nullptr, uint32_t* ntri = nullptr)
{
    Trav T;
    int stack[kTravStack];  // of the 4-wide traversal, then of the binary one
    trav_init(T, o, d, tlo, thi, true);
    if (S.w4) trav4(T, stack, S, true, nbox, ntri);
    if (!T.found) trav_roots<kLive>(T, stack, S, true, ntri);
    while (trav_step<kLive>(T, stack, S, true, nbox, ntri)) {
    }
    return T.found;
}


// ----------------------------------------------------------------- atlas access
// Packed texels (the paper's 32-bit codecs): irradiance R bits 0-8, G 9-17,
// B 18-25, count 26-31; visibility mean bits 0-12, mean square 13-25, count
// 26-31, both in units of the cage diagonal s.  A code stands for the value
// of its table entry.
constexpr int kCt9 = 0, kCt8 = 512, kCtM = 768, kCtQ = 768 + 8192, kCtSize = 768 + 2 * 8192;

__device__ __forceinline__ float4 irr_unpack(const float* __restrict__ ct, uint32_t c)
{
    return make_float4(__ldg(ct + kCt9 + (c & 511u)), __ldg(ct + kCt9 + ((c >> 9) & 511u)),
                       __ldg(ct + kCt8 + ((c >> 18) & 255u)), (float)(c >> 26));
}

// {mean, variance} in world units from a packed visibility texel
__device__ __forceinline__ float2 dep_unpack(const float* __restrict__ ct, float s, uint32_t c)
{
    const float m = __ldg(ct + kCtM + (c & 8191u)) * s;
    const float q = __ldg(ct + kCtQ + ((c >> 13) & 8191u)) * (s * s);
    return make_float2(m, fmaxf(q - m * m, 0.0f));
}

// kFmt: the storage when the kernel is made for it (0 FP32, 1 FP16, 3 packed
// codes), so that a loop's loads stay in one block of code; -1: V.fp16 decides
template <int kFmt = -1>
__device__ __forceinline__ float4 irr_load(const VolConst& V, const void* irr, size_t idx)
{
    const int fmt = kFmt >= 0 ? kFmt : V.fp16;
    if (fmt == 3) return irr_unpack(V.ctab, reinterpret_cast<const uint32_t*>(irr)[idx]);
    if (fmt) {
        const __half2* h = reinterpret_cast<const __half2*>(irr) + 2 * idx;
        float2 a = __half22float2(h[0]), b = __half22float2(h[1]);
        return make_float4(a.x, a.y, b.x, b.y);
    }
    return reinterpret_cast<const float4*>(irr)[idx];
}

// depth texel as {mean, variance}
template <int kFmt = -1>
__device__ __forceinline__ float2 dep_load(const VolConst& V, const void* dep, size_t idx)
{
    const int fmt = kFmt >= 0 ? kFmt : V.fp16;
    if (fmt == 3) return dep_unpack(V.ctab, V.s_f, reinterpret_cast<const uint32_t*>(dep)[idx]);
    if (fmt) return __half22float2(reinterpret_cast<const __half2*>(dep)[idx]);
    return reinterpret_cast<const float2*>(dep)[idx];
}

// The four texels at (x, y), (x+1, y), (x, y+1), (x+1, y+1) of a tile of width
// T: tile p of ti2 texels, first texel `at` in it.  One 64-bit product and one
// row step for all four addresses.
template <int kFmt>
__device__ __forceinline__ void irr_quad(const VolConst& V, const void* irr, int p, int ti2, int at, int T, float4 v[4])
{
    const uint64_t i = (uint64_t)(uint32_t)p * (uint32_t)ti2 + (uint32_t)at;
    if constexpr (kFmt == 0) {
        const float4* a = reinterpret_cast<const float4*>(irr) + i;
        const float4* b = a + T;
        v[0] = a[0], v[1] = a[1], v[2] = b[0], v[3] = b[1];
    } else {
        v[0] = irr_load<kFmt>(V, irr, i), v[1] = irr_load<kFmt>(V, irr, i + 1);
        v[2] = irr_load<kFmt>(V, irr, i + T), v[3] = irr_load<kFmt>(V, irr, i + T + 1);
    }
}

template <int kFmt>
__device__ __forceinline__ void dep_quad(const VolConst& V, const void* dep, int p, int td2, int at, int T, float2 v[4])
{
    const uint64_t i = (uint64_t)(uint32_t)p * (uint32_t)td2 + (uint32_t)at;
    if constexpr (kFmt == 0) {
        const float2* a = reinterpret_cast<const float2*>(dep) + i;
        const float2* b = a + T;
        v[0] = a[0], v[1] = a[1], v[2] = b[0], v[3] = b[1];
    } else {
        v[0] = dep_load<kFmt>(V, dep, i), v[1] = dep_load<kFmt>(V, dep, i + 1);
        v[2] = dep_load<kFmt>(V, dep, i + T), v[3] = dep_load<kFmt>(V, dep, i + T + 1);
    }
}

// The bilinear taps of an irradiance tile at octahedral coordinates p: the
// same texels and fractions in every probe's tile.
struct IrrTaps {
    int at;  // first texel in the tile
    float ax, ay;
};

__device__ __forceinline__ IrrTaps irr_taps(const VolConst& V, float2 p)
{
    const int n = V.n_irr;
    float fx = (1.0f + (p.x + 1.0f) * 0.5f * (float)n) - 0.5f;
    float fy = (1.0f + (p.y + 1.0f) * 0.5f * (float)n) - 0.5f;
    int x0 = min(max((int)floorf(fx), 0), n);
    int y0 = min(max((int)floorf(fy), 0), n);
    IrrTaps t;
    t.ax = fminf(fmaxf(fx - (float)x0, 0.0f), 1.0f);
    t.ay = fminf(fmaxf(fy - (float)y0, 0.0f), 1.0f);
    t.at = y0 * V.Ti + x0;
    return t;
}

template <int kFmt>
__device__ __forceinline__ void irr_bilinear(const VolConst& V, const void* base, int p, const IrrTaps& t, float* out)
{
    const float ax = t.ax, ay = t.ay;
    float4 v[4];
    irr_quad<kFmt>(V, base, p, V.Ti * V.Ti, t.at, V.Ti, v);
    const float4 v00 = v[0], v01 = v[1], v10 = v[2], v11 = v[3];
    out[0] = (1.0f - ay) * ((1.0f - ax) * v00.x + ax * v01.x) + ay * ((1.0f - ax) * v10.x + ax * v11.x);
    out[1] = (1.0f - ay) * ((1.0f - ax) * v00.y + ax * v01.y) + ay * ((1.0f - ax) * v10.y + ax * v11.y);
    out[2] = (1.0f - ay) * ((1.0f - ax) * v00.z + ax * v01.z) + ay * ((1.0f - ax) * v10.z + ax * v11.z);
}

// FP32 coordinate of probe plane j along axis k (where the probes sit)
__device__ __forceinline__ float pcoord(const VolConst& V, int k, int j)
{
    return fa(V.origin[k], fm(V.spacing[k], (float)j));
}

// (o - pb) + t*d with the rounding errors of the product and the sum carried
// (FMA residual + two-sum), so the result has a small *relative* error even
// when the hit point sits next to a probe plane far from the world origin.
__device__ __forceinline__ float local_offset(float o, float pb, float t, float d)
{
    float a = fs(o, pb);  // probe planes: exact difference
    float p = fm(t, d);
    float e = __fmaf_rn(t, d, -p);
    float s = fa(a, p);
    float bb = fs(s, a);
    float err = fa(fs(a, fs(s, bb)), fs(p, bb));
    return fa(s, fa(e, err));
}

// Bilinear filter of depth texels {mean, variance}: filtered mean, and the
// filtered variance sum w var_t + sum w (mean_t - mean)^2 -- the variance of
// the filtered {d, d^2} moments, formed without cancellation.
__device__ __forceinline__ void filter_moments(float w00, float w01, float w10, float w11, float2 v00, float2 v01,
                                               float2 v10, float2 v11, float* mom)
{
    float mu = w00 * v00.x + w01 * v01.x + w10 * v10.x + w11 * v11.x;
    float d00 = v00.x - mu, d01 = v01.x - mu, d10 = v10.x - mu, d11 = v11.x - mu;
    float var = w00 * (v00.y + d00 * d00) + w01 * (v01.y + d01 * d01) + w10 * (v10.y + d10 * d10) +
                w11 * (v11.y + d11 * d11);
    mom[0] = mu;
    mom[1] = var;
}

// Depth moments of probe tile p at the direction of dv (not normalised:
// the octahedral map is scale invariant), FP32 bilinear fractions.
template <int kFmt>
__device__ __forceinline__ void depth_moments(const VolConst& V, const void* dep, int p, float dx, float dy,
                                              float dz, float* mom, float* cond)
{
    // the fractions only weight a bilinear lookup: fast division (2 ulp)
    float l1 = fabsf(dx) + fabsf(dy) + fabsf(dz);
    float px = __fdividef(dx, l1), py = __fdividef(dy, l1);
    if (dz < 0.0f) {
        float qx = (1.0f - fabsf(py)) * sgnf(px);
        float qy = (1.0f - fabsf(px)) * sgnf(py);
        px = qx;
        py = qy;
    }
    const int n = V.n_dep, T = V.Td;
    float fx = (1.0f + (px + 1.0f) * 0.5f * (float)n) - 0.5f;
    float fy = (1.0f + (py + 1.0f) * 0.5f * (float)n) - 0.5f;
    int x0 = min(max((int)floorf(fx), 0), n);
    int y0 = min(max((int)floorf(fy), 0), n);
    float ax = fminf(fmaxf(fx - (float)x0, 0.0f), 1.0f);
    float ay = fminf(fmaxf(fy - (float)y0, 0.0f), 1.0f);
    float2 v[4];
    dep_quad<kFmt>(V, dep, p, T * T, y0 * T + x0, T, v);
    const float2 v00 = v[0], v01 = v[1], v10 = v[2], v11 = v[3];
    float w00 = (1.f - ax) * (1.f - ay), w01 = ax * (1.f - ay), w10 = (1.f - ax) * ay, w11 = ax * ay;
    filter_moments(w00, w01, w10, w11, v00, v01, v10, v11, mom);
    // conditioning of the filtered variance against the fractions: what a
    // texel adds to the variance per unit weight, over the floored variance
    float var = fmaxf(mom[1], fmaxf(V.var_rel * (mom[1] + mom[0] * mom[0]), V.var_min));
    float d00 = v00.x - mom[0], d01 = v01.x - mom[0], d10 = v10.x - mom[0], d11 = v11.x - mom[0];
    float s2 = fmaxf(fmaxf(v00.y + d00 * d00, v01.y + d01 * d01), fmaxf(v10.y + d10 * d10, v11.y + d11 * d11));
    *cond = __fdividef(s2, var);
}

// ---------------------------------------------------------------- double-float
// Unevaluated sums hi + lo of two floats (Dekker / Knuth error-free
// transformations), for the few quantities that need ~2^-44 relative precision.
struct df {
    float h, l;
};
__device__ __forceinline__ df two_sum(float a, float b)
{
    float s = fa(a, b);
    float bb = fs(s, a);
    return {s, fa(fs(a, fs(s, bb)), fs(b, bb))};
}
__device__ __forceinline__ df fast_two_sum(float a, float b)
{
    float s = fa(a, b);
    return {s, fs(b, fs(s, a))};
}
__device__ __forceinline__ df two_prod(float a, float b)
{
    float p = fm(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ df df_add(df a, df b)
{
    df s = two_sum(a.h, b.h);
    return fast_two_sum(s.h, fa(s.l, fa(a.l, b.l)));
}
__device__ __forceinline__ df df_neg(df a) { return {-a.h, -a.l}; }
__device__ __forceinline__ df df_abs(df a) { return a.h < 0.0f ? df_neg(a) : a; }
__device__ __forceinline__ df df_mul_f(df a, float b)
{
    df p = two_prod(a.h, b);
    return fast_two_sum(p.h, __fmaf_rn(a.l, b, p.l));
}
__device__ __forceinline__ df df_div(df a, df b)
{
    float q1 = fd(a.h, b.h);
    df r = df_add(a, df_neg(df_mul_f(b, q1)));
    float q2 = fd(r.h, b.h);
    return fast_two_sum(q1, q2);
}
// (o - p) + t*d as a double-float: exact inputs, error ~2^-44 relative
__device__ __forceinline__ df df_offset(float o, float p, float t, float d)
{
    return df_add(two_sum(o, -p), two_prod(t, d));
}

// The depth lookup with the direction and the bilinear fractions in
// double-float (for footprints where FP32 fractions would perturb the filtered
// variance): the offset is rebuilt exactly from (o, p, t, d).
static __device__ __noinline__ void depth_moments_precise(const VolConst& V, const void* dep, size_t tile,
                                                          const float* o, const float* p, float t, const float* d,
                                                          float* mom)
{
    df dx = df_offset(o[0], p[0], t, d[0]);
    df dy = df_offset(o[1], p[1], t, d[1]);
    df dz = df_offset(o[2], p[2], t, d[2]);
    df l1 = df_add(df_add(df_abs(dx), df_abs(dy)), df_abs(dz));
    df px = df_div(dx, l1), py = df_div(dy, l1);
    if (dz.h < 0.0f) {
        const df one = {1.0f, 0.0f};
        df qx = df_add(one, df_neg(df_abs(py)));
        df qy = df_add(one, df_neg(df_abs(px)));
        px = px.h >= 0.0f ? qx : df_neg(qx);
        py = py.h >= 0.0f ? qy : df_neg(qy);
    }
    const int n = V.n_dep, T = V.Td;
    const float hn = 0.5f * (float)n;
    df fx = df_add(df_mul_f(px, hn), {hn + 0.5f, 0.0f});
    df fy = df_add(df_mul_f(py, hn), {hn + 0.5f, 0.0f});
    float x0f = floorf(fx.h), y0f = floorf(fy.h);
    if (fx.h == x0f && fx.l < 0.0f) x0f -= 1.0f;
    if (fy.h == y0f && fy.l < 0.0f) y0f -= 1.0f;
    int x0 = min(max((int)x0f, 0), n);
    int y0 = min(max((int)y0f, 0), n);
    float ax = fminf(fmaxf(fa(fs(fx.h, (float)x0), fx.l), 0.0f), 1.0f);
    float ay = fminf(fmaxf(fa(fs(fy.h, (float)y0), fy.l), 0.0f), 1.0f);
    float bx = fminf(fmaxf(fs(fs((float)(x0 + 1), fx.h), fx.l), 0.0f), 1.0f);
    float by = fminf(fmaxf(fs(fs((float)(y0 + 1), fy.h), fy.l), 0.0f), 1.0f);
    size_t i00 = tile + (size_t)(y0 * T + x0);
    float2 v00 = dep_load(V, dep, i00), v01 = dep_load(V, dep, i00 + 1);
    float2 v10 = dep_load(V, dep, i00 + T), v11 = dep_load(V, dep, i00 + T + 1);
    float w00 = bx * by, w01 = ax * by, w10 = bx * ay, w11 = ax * ay;
    filter_moments(w00, w01, w10, w11, v00, v01, v10, v11, mom);
}

// The cage of a query point x = o + t*d: its lower probe, and per axis the
// offsets of x from the two probe planes and their layer weights.  The cage is
// the one whose FP32 probe planes bracket x; offsets are formed without
// rounding x to world coordinates.
struct Cage {
    int b[3];
    float off[2][3];  // from the lower, the upper plane
    float w[2][3];
};

// kPoint: the point is o itself (t = 0), where the offsets and their
// double-float forms come out as the plain differences, bit for bit
template <bool kPoint>
__device__ __forceinline__ Cage cage_of(const VolConst& V, const float* os, float t, const float* ds)
{
    auto offset = [&](int k, int j) { return kPoint ? fs(os[k], pcoord(V, k, j)) : local_offset(os[k], pcoord(V, k, j), t, ds[k]); };
    Cage C;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float g = floorf(((kPoint ? os[k] : fa(os[k], fm(t, ds[k]))) - V.origin[k]) / V.spacing[k]);
        int bi = (int)fminf(fmaxf(g, 0.0f), (float)(V.dims[k] - 2));
        float l = offset(k, bi);
        if (bi > 0 && l < 0.0f) {
            --bi;
            l = offset(k, bi);
        } else if (bi < V.dims[k] - 2) {
            float l2 = offset(k, bi + 1);
            if (l2 >= 0.0f) {
                ++bi;
                l = l2;
            }
        }
        C.b[k] = bi;
        C.off[0][k] = l;
        C.off[1][k] = offset(k, bi + 1);
        // both layer weights from the double-float offset l to plane b: alpha
        // = l/s and 1 - alpha = (s - l)/s, each with full relative precision
        // (1 - alpha formed in FP32 loses it next to the upper plane, where a
        // nearly empty lower-layer weight can still decide the normalised sum)
        const df lf = kPoint ? two_sum(os[k], -pcoord(V, k, bi)) : df_offset(os[k], pcoord(V, k, bi), t, ds[k]);
        const df rf = df_add({V.spacing[k], 0.0f}, df_neg(lf));
        C.w[1][k] = fminf(fmaxf(fa(lf.h, lf.l) / V.spacing[k], 0.0f), 1.0f);
        C.w[0][k] = fminf(fmaxf(fa(rf.h, rf.l) / V.spacing[k], 0.0f), 1.0f);
    }
    return C;
}

// probe corner c of the cage: its trilinear weight wt, its Chebyshev weight
// wc and its irradiance E at the taps
template <int kFmt>
__device__ __forceinline__ void query_probe(const VolConst& V, const void* irr, const void* dep, const float* os, float t,
                                            const float* ds, const Cage& C, const IrrTaps& taps, int c, float& wt,
                                            float& wc, float* E)
{
    const int o0 = c & 1, o1 = (c >> 1) & 1, o2 = (c >> 2) & 1;
    wt = (o0 ? C.w[1][0] : C.w[0][0]) * (o1 ? C.w[1][1] : C.w[0][1]) * (o2 ? C.w[1][2] : C.w[0][2]);
    const int ix = C.b[0] + o0, iy = C.b[1] + o1, iz = C.b[2] + o2;
    const int p = ix + V.dims[0] * (iy + V.dims[1] * iz);
    const float dx = o0 ? C.off[1][0] : C.off[0][0], dy = o1 ? C.off[1][1] : C.off[0][1], dz = o2 ? C.off[1][2] : C.off[0][2];
    float dist = sqrtf(dx * dx + dy * dy + dz * dz);
    float mom[2] = {0.f, 0.f};
    if (dist > 0.f) {
        float cond;
        depth_moments<kFmt>(V, dep, p, dx, dy, dz, mom, &cond);
        if (cond > 128.0f) {  // FP32 fractions would move the variance by > ~6e-5
            const float pc[3] = {pcoord(V, 0, ix), pcoord(V, 1, iy), pcoord(V, 2, iz)};
            depth_moments_precise(V, dep, (size_t)p * ((size_t)V.Td * V.Td), os, pc, t, ds, mom);
        }
    }
    wc = 1.f;
    if (dist > mom[0]) {
        // one-sided Chebyshev bound with the minimum variance 1e-6 s^2,
        // or var_rel * mu2 (mu2 = var + mean^2) where a volume asks for it
        float var = fmaxf(mom[1], fmaxf(V.var_rel * (mom[1] + mom[0] * mom[0]), V.var_min));
        float dd = dist - mom[0];
        wc = __fdividef(var, var + dd * dd);
    }
    irr_bilinear<kFmt>(V, irr, p, taps, E);
}

__device__ __forceinline__ IrrTaps normal_taps(const VolConst& V, float3 nrm)
{
    float nl = sqrtf(nrm.x * nrm.x + nrm.y * nrm.y + nrm.z * nrm.z);
    float3 nd = nl > 0.0f ? make_float3(nrm.x / nl, nrm.y / nl, nrm.z / nl) : make_float3(0.f, 0.f, 1.f);
    return irr_taps(V, oct_encode_x(nd));
}

// 8-probe trilinear x Chebyshev irradiance query at x = o + t*d (the public
// query passes t = 0).
template <int kFmt, bool kPoint>
__device__ __forceinline__ float3 query_irr_at(const VolConst& V, const void* irr, const void* dep, float3 o, float t,
                                               float3 d, float3 nrm)
{
    float os[3] = {o.x, o.y, o.z}, ds[3] = {d.x, d.y, d.z};
    const Cage C = cage_of<kPoint>(V, os, t, ds);
    const IrrTaps taps = normal_taps(V, nrm);
    float sum[3] = {0.f, 0.f, 0.f}, sumt[3] = {0.f, 0.f, 0.f}, sw = 0.f;
#pragma unroll 1
    for (int c = 0; c < 8; ++c) {
        float wt, wc, E[3];
        query_probe<kFmt>(V, irr, dep, os, t, ds, C, taps, c, wt, wc, E);
        float w = wt * wc;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            sum[k] += w * E[k];
            sumt[k] += wt * E[k];
        }
        sw += w;
    }
    if (sw >= 1e-12f) return make_float3(sum[0] / sw, sum[1] / sw, sum[2] / sw);
    return make_float3(sumt[0], sumt[1], sumt[2]);
}

// Dynamic ray r: its probe p, irradiance texel t (tile index) and direction
// d; false beyond this frame's rays.
__device__ __forceinline__ bool dyn_ray_of(const VolConst& V, const DynRays& D, uint32_t r, int& p, int& t, float3& d)
{
    if (r >= __ldg(D.off + V.P)) return false;
    int lo = 0, hi = V.P - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(D.off + mid) <= r)
            lo = mid;
        else
            hi = mid - 1;
    }
    p = lo;
    uint32_t j = r - __ldg(D.off + p);
    const int ix = p % V.dims[0], iy = (p / V.dims[0]) % V.dims[1], iz = p / (V.dims[0] * V.dims[1]);
    const int q = ix / 3 + D.dp[0] * (iy / 3 + D.dp[1] * (iz / 3));
    const int nn = V.n_irr * V.n_irr;
    for (int o = 0; o < 8; ++o) {
        if (!__ldg(D.incl + q * 8 + o)) continue;
        const uint32_t n = (uint32_t)__ldg(D.ntex + o);
        if (j < n) {
            t = __ldg(D.tex_t + o * nn + (int)j);
            const float4 w = __ldg(D.tex_dir + o * nn + (int)j);
            d = make_float3(w.x, w.y, w.z);
            return true;
        }
        j -= n;
    }
    return false;
}

}  // namespace adgi
