// wave.cuh -- device bodies of the ray wavefront (sm_103a): the pilot and
// adaptive nearest-hit traces and the three shading steps (prep, shadow
// rays, finish).  The ordinary kernels (trace.cu, shade.cu) and the
// persistent batched tick (tick.cu) run the same bodies.
#pragma once
#include "adgi_internal.cuh"
#include "kernels.cuh"

namespace adgi {

namespace {
// probe owning main ray r: the last p with off[p] <= r, searched in [lo, hi]
template <bool kLive = false>
__device__ __forceinline__ int probe_of_ray(const uint32_t* off, uint32_t r, int lo, int hi)
{
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (ldl<kLive>(off + mid) <= r)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// per block: bounds of the probe range of this block's rays, in shared memory
template <bool kLive = false>
__device__ __forceinline__ void block_probe_range(const uint32_t* off, int P, uint32_t r0, uint32_t r1, int* s_lo,
                                                  int* s_hi)
{
    if (threadIdx.x == 0) *s_lo = probe_of_ray<kLive>(off, r0, 0, P - 1);
    if (threadIdx.x == 32 % blockDim.x) *s_hi = probe_of_ray<kLive>(off, r1, 0, P - 1);
    __syncthreads();
}

// direction at position k of the SF row of m points, and its SF index *i
__device__ __forceinline__ float3 main_dir(const FrameConst& F, const float4* __restrict__ sf, uint32_t m, uint32_t k,
                                           uint32_t* i)
{
    float4 s = __ldg(sf + (size_t)m * (m - 1) / 2 + k);
    *i = (uint32_t)__float_as_int(s.w);
    return rotate(F.R, s);
}

// j: the thread's index in the pilot-ray launch (one warp: 32 consecutive j)
template <bool kLive = false>
__device__ __forceinline__ void pilot_trace_body(const VolConst& V, const FrameDev* FD, const SceneDev& S, int2* hit,
                                                 int j)
{
    const FrameConst& F = FD->F;
    // A warp traces one octant of 32 consecutive probes (the stratified
    // directions of one octant, from neighbouring origins), not 8 octants of
    // 4 probes.  Thread j of the launch: group g = j / 256 of 32 probes,
    // octant (j / 32) % 8, probe 32 g + j % 32; results stay at 8 p + o.
    const int p = V.p_lo + ((j >> 8) << 5) + (j & 31), o = (j >> 5) & 7;
    if (p >= V.p_hi) return;
    const int i = p * kPilots + o;
    if (V.cls[p] == 0) {  // outside V_out: no pilot rays
        hit[i] = make_int2((int)kMiss, 0x7F800000);
        return;
    }
    float3 org = probe_pos(V, p);
    float3 d = pilot_dir(F.pilot_key, (uint32_t)p, o);
    float t;
    uint32_t h;
    trace_closest<kLive>(S, org, d, V.tmin, __int_as_float(0x7F800000), t, h);
    hit[i] = make_int2((int)h, __float_as_int(t));
}

// Adaptive ray r (its probe searched in [lo, hi]): row position r - off[p]
// of probe p, whose SF index i names the slot off[p] + i of the result.
template <bool kLive>
__device__ __forceinline__ void main_trace_ray(const VolConst& V, const FrameConst& F, const SceneDev& S,
                                               const uint32_t* off, const float4* __restrict__ sf, int2* hit,
                                               uint32_t r, int lo, int hi)
{
    int p = probe_of_ray<kLive>(off, r, lo, hi);
    uint32_t base = ldl<kLive>(off + p);
    uint32_t m = ldl<kLive>(off + p + 1) - base;
    if (m > (uint32_t)(V.rays_max - kPilots) || r - base >= m) {
        atomicOr(V.err, kErrRayRange);
        return;
    }
    float3 org = probe_pos(V, p);
    uint32_t i;
    float3 d = main_dir(F, sf, m, r - base, &i);
    if (i >= m) {
        atomicOr(V.err, kErrRayRange);
        return;
    }
    float t;
    uint32_t h;
    trace_closest<kLive>(S, org, d, V.tmin, __int_as_float(0x7F800000), t, h);
    hit[base + i] = make_int2((int)h, __float_as_int(t));
}

// One warp: rays [rb + 32 w, rb + 32 w + 32), one lane a row position (the
// rows are in a spatial order, so a warp traces nearby directions); the probe
// range is found by two lanes and passed round the warp (no block barrier).
// chunk_p: the probe of ray rb + 32 c for every chunk c of the rays; written
// here for the shading, and in the persistent tick (all probes only) by the
// allocation, where it bounds the search here too.
template <bool kLive>
__device__ __forceinline__ void main_trace_warp_body(const VolConst& V, const FrameDev* FD, const SceneDev& S,
                                                     const uint32_t* off, const float4* __restrict__ sf, uint32_t R,
                                                     int2* hit, unsigned w, uint32_t* chunk_p)
{
    const FrameConst& F = FD->F;
    const int lane = threadIdx.x & 31;
    const uint32_t rb = ldl<kLive>(off + V.p_lo), re = min(ldl<kLive>(off + V.p_hi), R);
    const uint32_t r0 = rb + 32u * w;
    if (r0 >= re) return;  // the whole warp
    const uint32_t r1 = min(re - 1, r0 + 31u);
    int lo = 0, hi = 0;
    if (kLive) {
        lo = (int)ldl<kLive>(chunk_p + w);
        hi = r0 + 32u < re ? (int)ldl<kLive>(chunk_p + w + 1) : V.P - 1;
    } else {
        if (lane == 0) lo = probe_of_ray<kLive>(off, r0, 0, V.P - 1);
        if (lane == 1) hi = probe_of_ray<kLive>(off, r1, 0, V.P - 1);
        lo = __shfl_sync(0xFFFFFFFFu, lo, 0);
        hi = __shfl_sync(0xFFFFFFFFu, hi, 1);
        if (lane == 0) chunk_p[w] = (uint32_t)lo;
    }
    const uint32_t r = r0 + lane;
    if (r >= re) return;
    main_trace_ray<kLive>(V, F, S, off, sf, hit, r, lo, hi);
}

constexpr float kInvPi = 0.31830987f;
constexpr float kLumR = 0.2126f, kLumG = 0.7152f, kLumB = 0.0722f;


// The rays of a launch: pilot rays (ray r = probe r/8, octant r%8), adaptive
// rays (ray r of the prefix offsets off[], its probe searched between those
// of its chunk's first ray and the next one's) or Metropolis samples (ray r = sample sf[sel[r]] of the
// grouped order: the positions whose +w ray stands for itself).
struct RaySet {
    int mode;                 // 0 pilot, 1 adaptive, 2 Metropolis samples in grouped order, 3 dynamic rays
    uint32_t n;               // rays in the set (dynamic rays: the budget)
    const uint32_t* off;      // adaptive: prefix offsets
    const float4* sf;         // adaptive: spherical Fibonacci sets; samples: {w.xyz, probe bits}
    DynRays dyn;              // dynamic rays
    const uint32_t* sel;      // samples: thread r takes grouped position sel[r], r < min(n, *sel_n)
    const unsigned* sel_n;
    uint8_t* njobs;           // samples: the shadow jobs of each position taken
    const uint32_t* chunk_p;  // adaptive: the probe of ray 32 c
};

enum { kNoRay, kRay, kDropped };  // none (or an inconsistent range), a ray, one outside its clip volume

// Ray idx of the set for probes [p_lo, p_hi).  A pilot ray is stored at slot
// 8 p + octant, an adaptive ray at base + (SF index of its row position), so
// that a warp works on nearby directions.  Gives the slot, and a ray's origin
// and direction.
template <bool kLive>
__device__ __forceinline__ int ray_of(const VolConst& V, const FrameConst& F, const RaySet& Rs, uint32_t idx,
                                      uint32_t& slot, float3& o, float3& d)
{
    if (idx >= Rs.n) return kNoRay;
    if (Rs.mode == 0) {
        slot = (uint32_t)V.p_lo * kPilots + idx;
        const int p = (int)(slot >> 3);
        if (V.cls[p] == 0) return kDropped;  // outside V_out: no pilot ray
        o = probe_pos(V, p);
        d = pilot_dir(F.pilot_key, (uint32_t)p, (int)(slot & 7));
        return kRay;
    }
    if (Rs.mode == 3) {
        int p, t;
        if (!dyn_ray_of(V, Rs.dyn, idx, p, t, d)) return kNoRay;
        slot = idx;
        o = probe_pos(V, p);
        return kRay;
    }
    if (Rs.mode == 2) {
        if (idx >= *Rs.sel_n) return kNoRay;
        slot = Rs.sel[idx];
        const float4 a = __ldg(Rs.sf + slot);
        const int p = __float_as_int(a.w);
        if (p < 0 || p >= V.P) return kNoRay;
        if (V.cls[p] != 2) return kDropped;  // a sample outside V_in
        o = probe_pos(V, p);
        d = make_float3(a.x, a.y, a.z);
        return kRay;
    }
    const uint32_t first = ldl<kLive>(Rs.off + V.p_lo), r = first + idx;
    const uint32_t end = min(ldl<kLive>(Rs.off + V.p_hi), V.R_main);
    if (r >= end) return kNoRay;  // beyond the adaptive rays of the probes (unspent budget)
    const uint32_t c = idx >> 5, next = first + 32u * (c + 1u);
    const int lo = (int)ldl<kLive>(Rs.chunk_p + c), hi = next < end ? (int)ldl<kLive>(Rs.chunk_p + c + 1) : V.P - 1;
    int p = probe_of_ray<kLive>(Rs.off, r, lo, hi);
    uint32_t base = ldl<kLive>(Rs.off + p), m = ldl<kLive>(Rs.off + p + 1) - base;
    if (m > (uint32_t)(V.rays_max - kPilots) || r - base >= m) return kNoRay;
    o = probe_pos(V, p);
    float4 s = __ldg(Rs.sf + (size_t)m * (m - 1) / 2 + (r - base));
    const uint32_t i = (uint32_t)__float_as_int(s.w);
    if (i >= m) return kNoRay;
    slot = base + i;
    d = rotate(F.R, s);
    return kRay;
}

// exact FP32 geometric normal of triangle tri (original order; kLive: a
// moving triangle's row may have been written earlier in the same launch)
template <bool kLive = false>
__device__ __forceinline__ float3 tri_normal(const SceneDev& S, int tri)
{
    float4 A = ldl<kLive>(S.tri_orig + 3 * (size_t)tri), B = ldl<kLive>(S.tri_orig + 3 * (size_t)tri + 1),
           C = ldl<kLive>(S.tri_orig + 3 * (size_t)tri + 2);
    float e1x = fs(B.x, A.x), e1y = fs(B.y, A.y), e1z = fs(B.z, A.z);
    float e2x = fs(C.x, A.x), e2y = fs(C.y, A.y), e2z = fs(C.z, A.z);
    float cx = fs(fm(e1y, e2z), fm(e1z, e2y));
    float cy = fs(fm(e1z, e2x), fm(e1x, e2z));
    float cz = fs(fm(e1x, e2y), fm(e1y, e2x));
    float cl = fsq(dot3x(cx, cy, cz, cx, cy, cz));
    return cl > 0.0f ? make_float3(fd(cx, cl), fd(cy, cl), fd(cz, cl)) : make_float3(0.f, 0.f, 1.f);
}

__device__ __forceinline__ float3 shadow_dir(const Light& Li, float3 xs)
{
    return Li.kind == 0 ? make_float3(fs(Li.v[0], xs.x), fs(Li.v[1], xs.y), fs(Li.v[2], xs.z))
                        : make_float3(-Li.v[0], -Li.v[1], -Li.v[2]);
}

// Every ray's miss, back-face or dropped record; the front-face hits go to the
// list of the finish step (their idx), and their shadow jobs to the job list.
// Bound by instruction issue (850 a warp).  The probe of a ray is searched
// between those of its chunk of 32: two threads searching all offsets for a
// block held up the others at a barrier (adaptive rays of the scaled scene 203
// -> 164 us, of the tunnel 112 -> 91).
template <bool kLive>
__device__ __forceinline__ void shade_prep_body(const VolConst& V, const FrameDev* FD, const SceneDev& S,
                                                const RaySet& Rs, const int2* hit, const ShadeWork& W,
                                                unsigned* front_count, float4* rec, float* lum, unsigned bx)
{
    const FrameConst& F = FD->F;
    const LightSet& L = FD->L;
    if (Rs.mode == 2 && bx * blockDim.x >= *Rs.sel_n) return;  // the whole block
    const uint32_t idx = bx * blockDim.x + threadIdx.x;
    bool front = false;
    float3 xs = make_float3(0.f, 0.f, 0.f), n = make_float3(0.f, 0.f, 1.f);
    uint32_t slot = 0;
    float3 o, d;
    const int kind = ray_of<kLive>(V, F, Rs, idx, slot, o, d);
    if (kind == kDropped) {  // nothing gathered
        rec[slot] = make_float4(0.f, 0.f, 0.f, V.depth_max);
        if (lum) lum[slot] = 0.0f;
    } else if (kind == kRay) {
        const int2 hv = hit[slot];
        const uint32_t h = (uint32_t)hv.x;
        const float t = __int_as_float(hv.y);
        if (h == kMiss) {
            rec[slot] = make_float4(F.sky[0], F.sky[1], F.sky[2], V.depth_max);
            if (lum) lum[slot] = fa(fa(fm(kLumR, F.sky[0]), fm(kLumG, F.sky[1])), fm(kLumB, F.sky[2]));
        } else if (h & kBackBit) {
            rec[slot] = make_float4(0.f, 0.f, 0.f, fminf(t, V.depth_max));
            if (lum) lum[slot] = 0.0f;
        } else {
            W.vis[slot] = 0ull;
            n = tri_normal<kLive>(S, (int)h);
            float3 x = make_float3(fa(o.x, fm(t, d.x)), fa(o.y, fm(t, d.y)), fa(o.z, fm(t, d.z)));
            xs = make_float3(fa(x.x, fm(V.tmin, n.x)), fa(x.y, fm(V.tmin, n.y)), fa(x.z, fm(V.tmin, n.z)));
            front = true;
        }
    }
    // The block's jobs take one range of the job list: one atomic per block
    // on the shared counter (one per warp and light contended on that
    // address).  They go there light by light, and by warp for each light:
    // a round of 32 jobs in k_shadow is then mostly one light seen from
    // neighbouring hit points of the block's rays (with the warps outermost a
    // round held two or three lights: k_shadow 2.25 against 2.10 ms for the
    // 2.5 M adaptive rays of the scaled scene, 893 against 838 us for the
    // tunnel's; the longer scan costs k_shade_prep 7 us).  Pass 1
    // counts each warp's jobs for each light, the first warp scans the counts
    // and claims the range, pass 2 writes the jobs.
    const unsigned lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    auto wants = [&](int l) {
        if (!front) return false;
        const float3 D = shadow_dir(L.l[l], xs);
        return dot3x(n.x, n.y, n.z, D.x, D.y, D.z) > 0.0f;
    };
    __shared__ unsigned s_c[8 * kMaxLights], s_f[8], s_base[2];  // at most 256 threads: 8 warps
    const unsigned nw = blockDim.x >> 5, cells = nw * (unsigned)L.n, below = (1u << lane) - 1u;
    const unsigned front_mask = __ballot_sync(0xFFFFFFFFu, front);
    if (lane == 0) s_f[w] = (unsigned)__popc(front_mask);
    unsigned long long mine = 0;  // the lights this lane wants
    for (int l = 0; l < L.n; ++l) {
        const bool want = wants(l);
        const unsigned c = (unsigned)__popc(__ballot_sync(0xFFFFFFFFu, want));
        if (lane == 0) s_c[(unsigned)l * nw + w] = c;
        mine |= (unsigned long long)want << l;
    }
    if (Rs.mode == 2 && idx < min(Rs.n, *Rs.sel_n)) Rs.njobs[Rs.sel[idx]] = (uint8_t)__popcll(mine);
    __syncthreads();
    if (w == 0) {
        auto scan = [&](unsigned c) {  // inclusive
#pragma unroll
            for (int q = 1; q < 32; q <<= 1) {
                const unsigned y = __shfl_up_sync(0xFFFFFFFFu, c, q);
                if (lane >= (unsigned)q) c += y;
            }
            return c;
        };
        unsigned run = 0;
        for (unsigned k0 = 0; k0 < cells; k0 += 32) {
            const unsigned c = k0 + lane < cells ? s_c[k0 + lane] : 0u, x = scan(c);
            if (k0 + lane < cells) s_c[k0 + lane] = run + x - c;
            run += __shfl_sync(0xFFFFFFFFu, x, 31);
        }
        const unsigned c = lane < nw ? s_f[lane] : 0u, x = scan(c);
        if (lane < nw) s_f[lane] = x - c;
        const unsigned nf = __shfl_sync(0xFFFFFFFFu, x, 31), take = lane == 0 ? run : nf;
        if (lane < 2) s_base[lane] = take ? atomicAdd(lane ? front_count : W.job_count, take) : 0u;
    }
    __syncthreads();
    if (front) W.fronts[s_base[1] + s_f[w] + (unsigned)__popc(front_mask & below)] = idx;
    for (int l = 0; l < L.n; ++l) {
        const bool want = (mine >> l) & 1ull;
        const unsigned mask = __ballot_sync(0xFFFFFFFFu, want);
        if (want) {
            const unsigned js = s_base[0] + s_c[(unsigned)l * nw + w] + (unsigned)__popc(mask & below);
            if (js < W.job_cap) {
                W.jobs[js] = make_uint4(__float_as_uint(xs.x), __float_as_uint(xs.y), __float_as_uint(xs.z), slot);
                W.job_light[js] = (uint8_t)l;
            } else {
                atomicOr(V.err, kErrRayRange);
            }
        }
    }
}

// Shadow job j (one lane): light l of the job is seen from its origin when
// no triangle blocks the segment (point light) or the ray (sun); then bit l
// of the ray's visibility word is set.
template <bool kLive = false>
__device__ __forceinline__ void shadow_job(const LightSet& L, const SceneDev& S, const uint4* jobs,
                                           const uint8_t* job_light, unsigned long long* vis, unsigned j)
{
    uint4 jb = jobs[j];
    int l = job_light[j];
    const Light& Li = L.l[l];
    float3 xs = make_float3(__uint_as_float(jb.x), __uint_as_float(jb.y), __uint_as_float(jb.z));
    float3 D = shadow_dir(Li, xs);
    float thi = Li.kind == 0 ? 1.0f : __int_as_float(0x7F800000);
    if (!trace_any<kLive>(S, xs, D, 0.0f, thi)) atomicOr(vis + jb.w, 1ull << l);
}

// The shadow jobs [0, min(*job_count, job_cap)) in rounds of 32 consecutive
// jobs, one a lane, with a uniform trip count per warp and an explicit
// reconvergence per round (lanes that finish early wait instead of running
// ahead on their own).  Each warp takes the next round from the counter
// next_round (zero before the launch), so a warp that drew short rays takes
// more rounds and the warps end together.  leader: the one lane that counts
// the jobs.
template <bool kLive = false>
__device__ __forceinline__ void shadow_body(const FrameDev* FD, const SceneDev& S, const uint4* jobs,
                                            const uint8_t* job_light, const unsigned* job_count, unsigned job_cap,
                                            unsigned long long* vis, unsigned long long* shadow_ctr,
                                            unsigned* next_round, bool leader)
{
    const LightSet& L = FD->L;
    const unsigned total = min(*job_count, job_cap);
    if (leader) atomicAdd(shadow_ctr, (unsigned long long)total);
    const unsigned lane = threadIdx.x & 31u, rounds = (total + 31u) / 32u;
    for (;;) {
        unsigned g = 0;
        if (lane == 0) g = atomicAdd(next_round, 1u);
        g = __shfl_sync(0xFFFFFFFFu, g, 0);
        if (g >= rounds) break;
        const unsigned j = 32u * g + lane;
        if (j < total) shadow_job<kLive>(L, S, jobs, job_light, vis, j);
        __syncwarp();
    }
}

// Front-face hit number bx * blockDim.x + threadIdx.x of the list.  The rays
// that miss or hit a back face (two of five in the scaled scene) have their
// records from the prep step, so that every lane here has a hit to shade: 2,560
// instructions a warp, most of them the eight probes of the multi-bounce term.
// With a lane a ray 19.7 of 32 lanes worked: adaptive rays of the scaled scene
// 744 -> 473 us, of the tunnel 396 -> 276.  Bound by instruction issue and the
// gathers' latency.
template <bool kLive, int kFmt>
__device__ __forceinline__ void shade_finish_body(const VolConst& V, const FrameDev* FD, const SceneDev& S,
                                                  const RaySet& Rs, const int2* hit, const unsigned long long* vis,
                                                  const uint32_t* fronts, const unsigned* front_count,
                                                  const void* __restrict__ irr, const void* __restrict__ dep,
                                                  float4* rec, float* lum, unsigned bx)
{
    const FrameConst& F = FD->F;
    const LightSet& L = FD->L;
    // adaptive rays and samples always carry the multi-bounce term; pilot
    // records are blended (so need it) only on the first frame of a pair
    const int bounce = Rs.mode != 0 || F.even;
    const uint32_t at = bx * blockDim.x + threadIdx.x;
    if (at >= *front_count) return;
    uint32_t slot;
    float3 o, d;
    if (ray_of<kLive>(V, F, Rs, fronts[at], slot, o, d) != kRay) return;
    const int2 hv = hit[slot];
    const int tri = hv.x;
    const float t = __int_as_float(hv.y), depth = fminf(t, V.depth_max);
    const float3 n = tri_normal<kLive>(S, tri);
    const float3 x = make_float3(fa(o.x, fm(t, d.x)), fa(o.y, fm(t, d.y)), fa(o.z, fm(t, d.z)));
    unsigned long long vm = vis[slot];
    float E0 = 0.f, E1 = 0.f, E2 = 0.f;
    for (int l = 0; l < L.n; ++l) {
        if (!((vm >> l) & 1ull)) continue;
        const Light& Li = L.l[l];
        float g;
        if (Li.kind == 0) {
            float dx = fs(Li.v[0], x.x), dy = fs(Li.v[1], x.y), dz = fs(Li.v[2], x.z);
            float d2 = dot3x(dx, dy, dz, dx, dy, dz);
            float nd = dot3x(n.x, n.y, n.z, dx, dy, dz);
            g = nd > 0.0f ? fd(nd, fm(d2, fsq(d2))) : 0.0f;
        } else {
            float ndD = dot3x(n.x, n.y, n.z, -Li.v[0], -Li.v[1], -Li.v[2]);
            float l2 = dot3x(Li.v[0], Li.v[1], Li.v[2], Li.v[0], Li.v[1], Li.v[2]);
            g = fd(ndD, fsq(l2));
        }
        E0 = fa(E0, fm(Li.rgb[0], g));
        E1 = fa(E1, fm(Li.rgb[1], g));
        E2 = fa(E2, fm(Li.rgb[2], g));
    }
    const float a0 = __ldg(S.albedo + 3 * (size_t)tri), a1 = __ldg(S.albedo + 3 * (size_t)tri + 1),
                a2 = __ldg(S.albedo + 3 * (size_t)tri + 2);
    float r0 = fm(fm(a0, kInvPi), E0), r1 = fm(fm(a1, kInvPi), E1), r2 = fm(fm(a2, kInvPi), E2);
    const float lo = fa(fa(fm(kLumR, r0), fm(kLumG, r1)), fm(kLumB, r2));
    if (bounce) {
        float3 Q = query_irr_at<kFmt, false>(V, irr, dep, o, t, d, n);
        r0 += a0 * Q.x;
        r1 += a1 * Q.y;
        r2 += a2 * Q.z;
    }
    rec[slot] = make_float4(r0, r1, r2, depth);
    if (lum) lum[slot] = lo;
}

}  // namespace

}  // namespace adgi
