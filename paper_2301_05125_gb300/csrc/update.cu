// update.cu -- heuristics, ray allocation, blend and query kernels (sm_103a).
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include <cooperative_groups.h>

#include "adgi_internal.cuh"
#include "kernels.cuh"
#include "phase.cuh"

namespace adgi {

namespace {


__global__ void __launch_bounds__(256) k_classify(VolConst V, const FrameDev* __restrict__ FD,
                                                  const uint16_t* __restrict__ lut_c, uint8_t* __restrict__ cls)
{
    classify_body(V, FD, lut_c, cls, blockIdx.x);
}

__global__ void __launch_bounds__(128) k_change_state(VolConst V, const FrameDev* __restrict__ FD, ChangeBufs B)
{
    change_state_body(V, FD, B, blockIdx.x);
}

__global__ void __launch_bounds__(128) k_change_weight(VolConst V, const FrameDev* __restrict__ FD, ChangeBufs B)
{
    change_weight_body<false>(V, FD, B, blockIdx.x);
}

__global__ void __launch_bounds__(256) k_blend_plan(VolConst V, const FrameDev* __restrict__ FD,
                                                    const float4* __restrict__ sf, BlendPlan Pl)
{
    blend_plan_body(V, FD, sf, Pl, blockIdx.x);
}

__global__ void __launch_bounds__(128) k_blend(VolConst V, const FrameDev* __restrict__ FD, BlendBufs B)
{
    blend_body<false>(V, FD, B, blockIdx.x, blockDim.x >> 5);
}

// ============================================================== allocation
// Integer water-filling of the extra budget by W, capped, then the remainder
// one ray per probe in index order, by kCl CTAs (one, or a thread-block
// cluster).  CTA r works on the r-th slice of the probes; warp w of a CTA on
// the w-th segment of the slice, its lanes on consecutive probes (32 a step),
// so the staged arrays are read without bank conflicts (with a contiguous
// chunk per thread, as before, the 16-probe chunks of a 131,072-probe grid
// made every access a 16-way conflict).  Measured (ncu, updates of the scenes
// of that size): 131,072 probes 205 -> 83-89 us, 16,384 probes 45 -> 30-34 us,
// 64 probes on one CTA 45 -> 7-10 us.  The pass count (7 to 10 on the city
// scenes) is what is left: a pass costs one block barrier and one cluster
// barrier, in which the CTAs' sums are written into every CTA's shared
// memory; all threads then add the same numbers in rank order, so every loop
// bound and break below is the same in all threads and they pass the same
// barriers.
//
// Where the slices fit in shared memory (8 bytes a probe) the weights and
// extras are staged there; larger grids run the same steps on the input and
// output arrays in global memory.
//
// With clip volumes (cls given) only V_in probes (cls 2) take adaptive rays:
// floors m0 in V_in, 8 (the pilots) in V_out - V_in, 0 outside; beyond the
// V_in floors E = (avg - 8) P - (m0 - 8) |V_in| is spread over V_in, capped
// at rmax - m0 per probe.  Without cls every probe is in V_in and E =
// (avg - m0) P.  A probe outside V_in has weight 0 and starts with its
// extras at the cap, so it is never eligible: every test is w > 0 / n < cap.
namespace cg = cooperative_groups;
constexpr int kAllocThreads = 1024;
constexpr int kAllocIters = 64;
constexpr int kAllocCluster = 8;
constexpr int kAllocStage = 24576;     // probes a CTA stages: 192 KB of shared memory

// Sums over all threads of the kCl CTAs.  red: the warps' partials of this
// CTA; tot: every CTA's partials, written by each CTA into all of them.  Both
// are double-buffered: a warp (a CTA) can be one reduction ahead of the
// slowest reader.
struct AllocRed {
    uint64_t red[2][2][32];
    uint64_t tot[2][2][kAllocCluster];
};

// warp sums with the integer reduction instruction: of 32-bit values whose
// sum fits, and of 64-bit values below 2^52 in two pieces
__device__ __forceinline__ uint32_t redux_add(uint32_t v) { return __reduce_add_sync(0xFFFFFFFFu, v); }
__device__ __forceinline__ uint64_t redux_add64(uint64_t v)
{
    constexpr uint32_t kMask = (1u << 26) - 1u;
    return (uint64_t)redux_add((uint32_t)v & kMask) + ((uint64_t)redux_add((uint32_t)(v >> 26)) << 26);
}

template <int kCl>
struct AllocGroup {
    AllocRed* S;
    int buf, rank, lane, warp, nw;

    // a sum over the CTA's warps (every lane holds it) to the sum over all CTAs
    __device__ __forceinline__ void across(uint64_t& a, uint64_t& b)
    {
        if constexpr (kCl > 1) {
            if (warp == 0 && lane < kCl) {
                *cg::this_cluster().map_shared_rank(&S->tot[buf][0][rank], lane) = a;
                *cg::this_cluster().map_shared_rank(&S->tot[buf][1][rank], lane) = b;
            }
            cg::this_cluster().sync();
            a = b = 0;
            for (int r = 0; r < kCl; ++r) a += S->tot[buf][0][r], b += S->tot[buf][1][r];
        }
        buf ^= 1;
    }
    // sums of a (below 2^32 in all) and b (below 2^52 a lane)
    __device__ __forceinline__ void sum2(uint64_t& a, uint64_t& b)
    {
        a = redux_add((uint32_t)a);
        b = redux_add64(b);
        if (lane == 0) S->red[buf][0][warp] = a, S->red[buf][1][warp] = b;
        __syncthreads();
        a = redux_add(lane < nw ? (uint32_t)S->red[buf][0][lane] : 0u);
        b = lane < nw ? S->red[buf][1][lane] : 0ull;
        b = (uint64_t)redux_add((uint32_t)b & 0x3FFFFFFu) + ((uint64_t)redux_add((uint32_t)(b >> 26) & 0x3FFFFFFu) << 26) +
            ((uint64_t)redux_add((uint32_t)(b >> 52)) << 52);
        across(a, b);
    }
    // minima of a and b
    __device__ __forceinline__ void min2(uint32_t& a, uint32_t& b)
    {
        a = __reduce_min_sync(0xFFFFFFFFu, a);
        b = __reduce_min_sync(0xFFFFFFFFu, b);
        if (lane == 0) S->red[buf][0][warp] = a, S->red[buf][1][warp] = b;
        __syncthreads();
        a = __reduce_min_sync(0xFFFFFFFFu, lane < nw ? (uint32_t)S->red[buf][0][lane] : 0xFFFFFFFFu);
        b = __reduce_min_sync(0xFFFFFFFFu, lane < nw ? (uint32_t)S->red[buf][1][lane] : 0xFFFFFFFFu);
        if constexpr (kCl > 1) {
            if (warp == 0 && lane < kCl) {
                *cg::this_cluster().map_shared_rank(&S->tot[buf][0][rank], lane) = a;
                *cg::this_cluster().map_shared_rank(&S->tot[buf][1][rank], lane) = b;
            }
            cg::this_cluster().sync();
            for (int r = 0; r < kCl; ++r) {
                a = min(a, (uint32_t)S->tot[buf][0][r]);
                b = min(b, (uint32_t)S->tot[buf][1][r]);
            }
        }
        buf ^= 1;
    }
    // v (the warp's, below 2^32 in all): the sum over the warps before this one, in probe order; *total: over all
    __device__ __forceinline__ uint64_t before(uint32_t v, uint64_t* total)
    {
        if (lane == 0) S->red[buf][0][warp] = v;
        __syncthreads();
        const uint32_t x = lane < nw ? (uint32_t)S->red[buf][0][lane] : 0u;
        uint64_t pre = redux_add(lane < warp ? x : 0u);
        const uint64_t own = redux_add(x);
        if constexpr (kCl > 1) {
            if (warp == 0 && lane < kCl) *cg::this_cluster().map_shared_rank(&S->tot[buf][0][rank], lane) = own;
            cg::this_cluster().sync();
            uint64_t all = 0;
            for (int r = 0; r < kCl; ++r) {
                const uint64_t t = S->tot[buf][0][r];
                pre += r < rank ? t : 0ull;
                all += t;
            }
            *total = all;
        } else {
            *total = own;
        }
        buf ^= 1;
        return pre;
    }
};

template <int kCl, bool kStaged>
__device__ __forceinline__ void allocate_body(const uint32_t* __restrict__ Win, int P, int avg, int m0, int rmax,
                                              uint32_t* __restrict__ n, uint32_t* __restrict__ off,
                                              const uint8_t* __restrict__ cls)
{
    __shared__ AllocRed S;
    extern __shared__ uint32_t stage[];  // staged: [Pc] weights, then [Pc] extras of this CTA's slice
    AllocGroup<kCl> g;
    g.S = &S;
    g.buf = 0;
    g.rank = kCl == 1 ? 0 : (int)cg::this_cluster().block_rank();
    g.lane = threadIdx.x & 31;
    g.warp = threadIdx.x >> 5;
    g.nw = blockDim.x >> 5;
    const int Pc = (P + kCl - 1) / kCl;
    const int b0 = min(P, g.rank * Pc), b1 = min(P, b0 + Pc);
    const int seg = ((Pc + g.nw - 1) / g.nw + 31) & ~31;
    const int s0 = min(b1, b0 + g.warp * seg), s1 = min(b1, s0 + seg);  // this warp's probes
    const uint32_t cap = (uint32_t)(rmax - m0);
    uint32_t* ws = stage;
    uint32_t* nx = kStaged ? stage + Pc : n;  // extra rays beyond the floor
    const int xo = kStaged ? b0 : 0;          // probe of nx[0]
    auto vin = [&](int p) { return !cls || cls[p] == 2; };
    auto w_of = [&](int p) -> uint32_t {
        if constexpr (kStaged)
            return ws[p - b0];
        else
            return vin(p) ? __ldg(Win + p) : 0u;
    };
    uint64_t pin = 0, sw = 0;
    for (int p = s0 + g.lane; p < s1; p += 32) {
        const bool in = vin(p);
        const uint32_t w = in ? __ldg(Win + p) : 0u;
        pin += in ? 1u : 0u;
        sw += w;
        if constexpr (kStaged) ws[p - b0] = w;
        nx[p - xo] = in ? 0u : cap;
    }
    uint64_t Pin = pin, Sw = sw;
    if constexpr (kCl > 1) cg::this_cluster().sync();  // every CTA runs before its shared memory is written to
    g.sum2(Pin, Sw);
    uint64_t E = (uint64_t)(avg - 8) * (uint64_t)P - (uint64_t)(m0 - 8) * Pin;
    if (E > Pin * cap) E = Pin * cap;
    const uint32_t lt = (1u << g.lane) - 1u;
    if (Sw == 0) {  // uniform over V_in, the remainder to the lowest V_in ranks
        const uint64_t q = Pin ? E / Pin : 0, r = Pin ? E % Pin : 0;
        uint64_t all, rk = g.before(redux_add((uint32_t)pin), &all);
        for (int p0 = s0; p0 < s1; p0 += 32) {
            const int p = p0 + g.lane;
            const bool in = p < s1 && vin(p);
            const uint32_t m = __ballot_sync(0xFFFFFFFFu, in);
            if (in) nx[p - xo] = (uint32_t)(q + (rk + __popc(m & lt) < r ? 1u : 0u));
            rk += __popc(m);
        }
    } else {
        // proportional passes: SU = the weight of the probes below their cap
        // (at first every V_in probe: Sw, unless the cap is 0); the pass that
        // hands out shares also sums SU for the next pass
        uint64_t Erem = E, SU = cap > 0u ? Sw : 0u;
        for (int it = 0; it < kAllocIters; ++it) {
            if (SU == 0 || Erem == 0) break;
            const uint64_t inv = 0xFFFFFFFFFFFFFFFFull / SU;
            uint64_t G = 0, su = 0;
            auto hand_out = [&](int p, uint32_t w, uint32_t e) {
                const uint64_t share = div_by(Erem * (uint64_t)w, SU, inv);
                const uint64_t room = cap - e;
                const uint64_t a = share < room ? share : room;
                nx[p - xo] = e + (uint32_t)a;
                G += a;
                su += a < room ? w : 0u;  // still below the cap after this pass
            };
            if constexpr (kCl == 1) {  // few probes a lane: no branch (W = 0 or at the cap: 0), four in flight
#pragma unroll 4
                for (int p = s0 + g.lane; p < s1; p += 32) hand_out(p, w_of(p), nx[p - xo]);
            } else {  // many, most of them without weight: skipped
                for (int p = s0 + g.lane; p < s1; p += 32) {
                    const uint32_t w = w_of(p), e = nx[p - xo];
                    if (w != 0u && e < cap) hand_out(p, w, e);
                }
            }
            g.sum2(G, su);
            if (G == 0) break;
            Erem -= G;
            SU = su;
        }
        // Remainder: one ray each in probe order, probes with W > 0 first,
        // round after round.  While a whole round fits into what is left,
        // every eligible probe takes one a round and the eligible set stays
        // the same until one of them reaches its cap: those rounds are done
        // at once (a camera's small V_in with many unweighted probes ran
        // hundreds of them: 1,006 us at 15,345 probes, 29 us now).
        for (int guard = 0; Erem > 0 && guard < (1 << 20); ++guard) {
            uint64_t ca = 0, ce = 0;
            uint32_t ra = 0xFFFFFFFFu, re = 0xFFFFFFFFu;  // least room of the eligible probes
            for (int p = s0 + g.lane; p < s1; p += 32) {
                const uint32_t e = nx[p - xo];
                if (e >= cap) continue;
                ++ce;
                re = min(re, cap - e);
                if (w_of(p) > 0u) {
                    ++ca;
                    ra = min(ra, cap - e);
                }
            }
            const uint32_t wa = redux_add((uint32_t)ca), we = redux_add((uint32_t)ce);
            g.sum2(ca, ce);
            const bool modeA = ca > 0;
            const uint64_t tot = modeA ? ca : ce;
            if (tot == 0) break;
            if (Erem >= tot) {
                g.min2(ra, re);
                const uint64_t full = Erem / tot, room = modeA ? ra : re;
                const uint32_t k = (uint32_t)(full < room ? full : room);
                for (int p = s0 + g.lane; p < s1; p += 32) {
                    const uint32_t e = nx[p - xo];
                    if (e < cap && (!modeA || w_of(p) > 0u)) nx[p - xo] = e + k;
                }
                Erem -= (uint64_t)k * tot;
            } else {
                uint64_t all, pre = g.before(modeA ? wa : we, &all);
                for (int p0 = s0; p0 < s1; p0 += 32) {
                    const int p = p0 + g.lane;
                    const uint32_t e = p < s1 ? nx[p - xo] : cap;
                    const bool el = e < cap && (!modeA || w_of(p) > 0u);
                    const uint32_t m = __ballot_sync(0xFFFFFFFFu, el);
                    if (el && pre + __popc(m & lt) < Erem) nx[p - xo] = e + 1u;
                    pre += __popc(m);
                }
                Erem = 0;
            }
        }
    }
    // rays per probe: the floor plus the extra; adaptive rays = rays - 8 (0 outside V_in)
    auto rays_of = [&](int p) -> uint32_t {
        if (vin(p)) return (uint32_t)m0 + nx[p - xo];
        return cls[p] == 1 ? 8u : 0u;
    };
    uint64_t loc = 0;
    for (int p = s0 + g.lane; p < s1; p += 32) {
        const uint32_t np = rays_of(p);
        loc += np > 8u ? np - 8u : 0u;
    }
    uint64_t tot, pre = g.before(redux_add((uint32_t)loc), &tot);
    for (int p0 = s0; p0 < s1; p0 += 32) {
        const int p = p0 + g.lane;
        const uint32_t np = p < s1 ? rays_of(p) : 0u;
        const uint32_t y = np > 8u ? np - 8u : 0u;
        uint32_t x = y;  // at most 32 * 4,088
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t z = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (g.lane >= o) x += z;
        }
        if (p < s1) {
            off[p] = (uint32_t)pre + x - y;
            n[p] = np;
        }
        pre += __shfl_sync(0xFFFFFFFFu, x, 31);
    }
    if (g.rank == 0 && threadIdx.x == 0) off[P] = (uint32_t)tot;
    if constexpr (kCl > 1) cg::this_cluster().sync();  // no CTA leaves while another may still write its sums
}

__global__ void __launch_bounds__(kAllocThreads, 1)
    k_allocate(const uint32_t* __restrict__ Win, int P, int avg, int m0, int rmax, uint32_t* __restrict__ n,
               uint32_t* __restrict__ off, const uint8_t* __restrict__ cls)
{
    allocate_body<1, true>(Win, P, avg, m0, rmax, n, off, cls);
}

template <bool kStaged>
__global__ void __cluster_dims__(kAllocCluster, 1, 1) __launch_bounds__(kAllocThreads, 1)
    k_allocate_cluster(const uint32_t* __restrict__ Win, int P, int avg, int m0, int rmax, uint32_t* __restrict__ n,
                       uint32_t* __restrict__ off, const uint8_t* __restrict__ cls)
{
    allocate_body<kAllocCluster, kStaged>(Win, P, avg, m0, rmax, n, off, cls);
}


// ---- DDGI cosine gather (blend_mode = 1, Sec. 3.1): every ray of the probe
// feeds every texel of its hemisphere.  Texel t with centre direction n_t
// (FP32 decode of the texel centre) and ray direction w, c = n_t . w: the
// test c > 0 is exact FP32 ((x x' + y y') + z z'), the irradiance texel
// takes the c-weighted mean radiance, the visibility texel the c^50-weighted
// mean of {d, d^2}; the number of rays with c > 0 is the batch count of the
// moving average.  One block of four warps per probe: rays are staged in
// shared memory a block's width at a time, and each lane holds two texels over
// the pass of the rays, the depth texels first and then the irradiance texels
// (196 + 36 texels in 256 places; one warp of the four has some of both).
//   Bound by FP32 arithmetic: 958M (texel, ray) pairs a tunnel update.  A
// pair's weight is c^50 of the clamped c as it stands, in one straight line of
// code for a lane's two texels (two-wide FP32 operations); only texels all of
// whose rays lie so far off that the weights near FP32's range (c below 0.4:
// a few rays) are gathered again relative to their largest c.  Measured
// (tunnel update, ncu): weights relative to the largest c so far (a division,
// a second c^50 and two branches a pair), four texels a lane for either tile,
// one warp a probe: 2.85 ms.  Weights as they stand, seven depth texels a
// lane: 1.25 ms; one-warp blocks, approximate reciprocals: 1.03 ms, with a
// third of the time a tail of probes of up to 1,016 rays; four warps a probe:
// 0.83 ms, the pipe that takes two-wide operations 73 % busy (some of them as
// scalar pairs, to use the other FP32 pipe too: no faster), and 0.86 with c
// exact (see cos_dot).  The depth variance is closer to FP64 than with weights
// relative to the largest c (2-norm 4.0e-7 -> 3.9e-7 after four frames of a
// small city, largest error of a texel 2e-3 -> 2e-5).
constexpr int kCosWarps = 4, kCosThreads = 32 * kCosWarps;
constexpr float kCosWeak = 1e-20f;  // a depth weight sum below this: gathered again

struct CosLayout {
    uint32_t ray_d, ray_r, irr_new, dep_new, dn_new, total;
};

__host__ __device__ inline CosLayout cos_layout(int Ti, int Td)
{
    const uint32_t ti2 = (uint32_t)(Ti * Ti), td2 = (uint32_t)(Td * Td);
    CosLayout L;
    uint32_t o = 0;
    L.ray_d = o, o += 16 * kCosThreads;  // a chunk of rays: direction and depth
    L.ray_r = o, o += 16 * kCosThreads;  // and radiance
    L.irr_new = o, o += al16(16 * ti2);
    L.dep_new = o, o += al16(8 * td2);
    L.dn_new = o, o += al16(td2);
    L.total = o;
    return L;
}

__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

__device__ __forceinline__ float2 pow50(float2 c)
{
    const float2 c2 = mul2(c, c), c4 = mul2(c2, c2), c8 = mul2(c4, c4), c16 = mul2(c8, c8), c32 = mul2(c16, c16);
    return mul2(mul2(c32, c16), c2);
}

// the rays of one probe: pilots, then the adaptive rays in row order
struct CosRays {
    const float4* prec;   // pilot records
    const float4* mrec;   // adaptive records
    const float4* sfrow;
    uint64_t key;
    int p, npil, n;
    uint32_t m;
};

// stage rays [c0, c0 + kCosThreads) of the probe (the whole block); returns how
// many; odd: one of their records is not finite (the same for the block)
__device__ __forceinline__ int cos_stage(const CosRays& R, const float* rot, int c0, float4* rd, float4* rr, bool& odd)
{
    __syncthreads();  // the last chunk is read
    const int j = c0 + (int)threadIdx.x;
    bool bad = false;
    if (j < R.n) {
        float3 d;
        float4 r;
        if (j < R.npil) {
            d = pilot_dir(R.key, (uint32_t)R.p, j);
            r = __ldg(R.prec + j);
        } else {
            const float4 sfp = __ldg(R.sfrow + (j - R.npil));
            const uint32_t i = min((uint32_t)__float_as_int(sfp.w), R.m - 1);
            d = rotate(rot, sfp);
            r = __ldg(R.mrec + i);
        }
        rd[threadIdx.x] = make_float4(d.x, d.y, d.z, r.w);
        rr[threadIdx.x] = r;
        bad = !(isfinite(r.x) && isfinite(r.y) && isfinite(r.z) && isfinite(r.w));
    }
    odd = __syncthreads_or(bad) != 0;
    return min(kCosThreads, R.n - c0);
}

// the texel at place q: a depth texel, then the irradiance texels, then none
// (a zero direction: c is never > 0)
__device__ __forceinline__ float3 cos_texel(int q, int nd, int ni)
{
    const int nd2 = nd * nd;
    if (q < nd2) return texel_centre_dir(q % nd, q / nd, nd);
    q -= nd2;
    return q < ni * ni ? texel_centre_dir(q % ni, q / ni, ni) : make_float3(0.f, 0.f, 0.f);
}

// The exact c of two texels: products and sums each rounded once.  The
// compiler fuses a two-wide product into a sum that follows (the scalar
// intrinsics it leaves alone), so both are written as fused operations, with
// one = 1 and nil = -0 from the kernel's arguments, whose values it does not
// know.
__device__ __forceinline__ float2 cos_dot(float2 nx, float2 ny, float2 nz, float4 d, float2 one, float2 nil)
{
    return fma2(fma2(fma2(nx, dup2(d.x), nil), one, fma2(ny, dup2(d.y), nil)), one, fma2(nz, dup2(d.z), nil));
}

// Weighted running mean s0 and sum of squared deviations s1 of the depths
// (West's update of Welford's method): no cancellation between the mean of
// d^2 and the square of the mean of d.  With i = 1 / (sw + w) the mean moves
// by w i of the deviation dx and the sum grows by w dx^2 (1 - w i), where 1 -
// w i = sw i is formed as such: exact to a few ulps also where the new weight
// outweighs all before it.  A zero weight changes nothing as long as the depth
// is finite (see pick2 for the others).
__device__ __forceinline__ float inv_approx(float x)  // x normal: 1 ulp
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ void cos_west(float2 w, float2 d, float2& sw, float2& s0, float2& s1)
{
    const float2 old = sw;
    sw = add2(sw, w);
    const float2 i = make_float2(inv_approx(sw.x), inv_approx(sw.y));
    const float2 dx = fma2(s0, dup2(-1.0f), d);
    s0 = fma2(dx, mul2(w, i), s0);
    s1 = fma2(mul2(w, dx), mul2(dx, mul2(old, i)), s1);
}

// A ray behind a texel has weight 0, but 0 times an infinite or NaN value is
// NaN: where such a value is among the rays (a radiance that overflowed, a
// miss with an infinite depth_max), a texel takes the new sums of the rays it
// faces alone.  Elsewhere the plain sums are the same bits and no branch.
__device__ __forceinline__ float2 pick2(bool x, bool y, float2 a, float2 b)
{
    return make_float2(x ? a.x : b.x, y ? a.y : b.y);
}

__device__ __forceinline__ void cos_west_of(bool x, bool y, float2 w, float2 d, float2& sw, float2& s0, float2& s1)
{
    float2 a = sw, b = s0, c = s1;
    cos_west(w, d, a, b, c);
    sw = pick2(x, y, a, sw), s0 = pick2(x, y, b, s0), s1 = pick2(x, y, c, s1);
}

__global__ void __launch_bounds__(kCosThreads) k_blend_cos(VolConst V, const FrameDev* __restrict__ FD, BlendBufs B,
                                                           float plus_one, float minus_zero)
{
    const FrameConst& F = FD->F;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = V.p_lo + blockIdx.x;
    if (p >= V.p_hi) return;  // the whole block
    const uint32_t base = __ldg(B.off + p);
    uint32_t m = __ldg(B.off + p + 1) - base;
    if (m > (uint32_t)(V.rays_max - kPilots) || base > V.R_main || m > V.R_main - base) {
        if (threadIdx.x == 0) atomicOr(V.err, kErrRayRange);
        m = 0;
    }
    const uint8_t cl = V.cls[p];
    const int npil = (F.even && cl >= 1) ? kPilots : 0;
    if ((int)m + npil == 0 && cl != 1) return;  // untouched tile
    const int Ti = V.Ti, Td = V.Td, ni = V.n_irr, nd = V.n_dep, nd2 = nd * nd, places = nd2 + ni * ni;
    const CosLayout L = cos_layout(Ti, Td);
    float4* rd = reinterpret_cast<float4*>(smem + L.ray_d);
    float4* rr = reinterpret_cast<float4*>(smem + L.ray_r);
    float4* irr_new = reinterpret_cast<float4*>(smem + L.irr_new);
    float2* dep_new = reinterpret_cast<float2*>(smem + L.dep_new);
    uint8_t* dn_new = smem + L.dn_new;
    const size_t io = (size_t)p * Ti * Ti, dof = (size_t)p * Td * Td;
    const CosRays R{B.pil_rec + (size_t)p * kPilots, B.main_rec + base, B.sf + (m ? (size_t)m * (m - 1) / 2 : 0),
                    F.pilot_key, p, npil, npil + (int)m, m};
    const float omh = 1.0f - V.hyst;
    const float2 zero = make_float2(0.f, 0.f), one = dup2(plus_one), nil = dup2(minus_zero);
    for (int g = 0; g < places; g += 2 * kCosThreads) {
        const int q0 = g + 64 * warp, q = q0 + lane;  // this lane's places: q and q + 32
        const bool has_dep = q0 < nd2, has_irr = q0 < places && q0 + 63 >= nd2;  // the same for the warp
        const float3 ta = cos_texel(q, nd, ni), tb = cos_texel(q + 32, nd, ni);
        const float2 nx = make_float2(ta.x, tb.x), ny = make_float2(ta.y, tb.y), nz = make_float2(ta.z, tb.z);
        float2 k = zero;  // rays with c > 0 (whole numbers far below 2^24)
        float2 sw = dup2(1e-37f), s0 = zero, s1 = zero;  // depth (sw never 0: its inverse is finite)
        float2 iw = zero, r0 = zero, r1 = zero, r2 = zero;  // radiance
        for (int c0 = 0; c0 < R.n; c0 += kCosThreads) {
            bool odd;
            const int cnt = cos_stage(R, F.R, c0, rd, rr, odd);
            if (odd) {
                for (int u = 0; u < cnt; ++u) {
                    const float4 d = rd[u], r = rr[u];
                    float2 c = cos_dot(nx, ny, nz, d, one, nil);
                    const bool x = c.x > 0.0f, y = c.y > 0.0f;
                    k = add2(k, make_float2(x ? 1.0f : 0.0f, y ? 1.0f : 0.0f));
                    c = make_float2(fmaxf(c.x, 0.0f), fmaxf(c.y, 0.0f));
                    iw = add2(iw, c);
                    r0 = pick2(x, y, fma2(c, dup2(r.x), r0), r0);
                    r1 = pick2(x, y, fma2(c, dup2(r.y), r1), r1);
                    r2 = pick2(x, y, fma2(c, dup2(r.z), r2), r2);
                    if (has_dep) cos_west_of(x, y, pow50(c), dup2(d.w), sw, s0, s1);
                }
            } else if (has_dep && !has_irr) {
#pragma unroll 2
                for (int u = 0; u < cnt; ++u) {
                    const float4 d = rd[u];
                    float2 c = cos_dot(nx, ny, nz, d, one, nil);
                    k = add2(k, make_float2(c.x > 0.0f ? 1.0f : 0.0f, c.y > 0.0f ? 1.0f : 0.0f));
                    c = make_float2(fmaxf(c.x, 0.0f), fmaxf(c.y, 0.0f));
                    cos_west(pow50(c), dup2(d.w), sw, s0, s1);
                }
            } else if (has_irr) {
                for (int u = 0; u < cnt; ++u) {
                    const float4 d = rd[u], r = rr[u];
                    float2 c = cos_dot(nx, ny, nz, d, one, nil);
                    k = add2(k, make_float2(c.x > 0.0f ? 1.0f : 0.0f, c.y > 0.0f ? 1.0f : 0.0f));
                    c = make_float2(fmaxf(c.x, 0.0f), fmaxf(c.y, 0.0f));
                    iw = add2(iw, c);
                    r0 = fma2(c, dup2(r.x), r0);
                    r1 = fma2(c, dup2(r.y), r1);
                    r2 = fma2(c, dup2(r.z), r2);
                    if (has_dep) cos_west(pow50(c), dup2(d.w), sw, s0, s1);
                }
            }
        }
        // depth texels whose weights came near FP32's range: again, relative to the largest c
        const bool weak_x = q < nd2 && k.x > 0.f && sw.x < kCosWeak, weak_y = q + 32 < nd2 && k.y > 0.f && sw.y < kCosWeak;
        if (__syncthreads_or(weak_x || weak_y)) {
            float2 cm = zero;
            for (int pass = 0; pass < 2; ++pass) {
                if (pass) {
                    if (weak_x) sw.x = 1e-37f, s0.x = s1.x = 0.f;
                    if (weak_y) sw.y = 1e-37f, s0.y = s1.y = 0.f;
                }
                for (int c0 = 0; c0 < R.n; c0 += kCosThreads) {
                    bool odd;
                    const int cnt = cos_stage(R, F.R, c0, rd, rr, odd);
                    if (!weak_x && !weak_y) continue;
                    for (int u = 0; u < cnt; ++u) {
                        const float4 d = rd[u];
                        const float2 c = cos_dot(nx, ny, nz, d, one, nil);
                        if (pass == 0) {
                            cm = make_float2(fmaxf(cm.x, c.x), fmaxf(cm.y, c.y));
                        } else {
                            const bool x = weak_x && c.x > 0.f, y = weak_y && c.y > 0.f;
                            cos_west_of(x, y, pow50(make_float2(x ? c.x / cm.x : 0.f, y ? c.y / cm.y : 0.f)), dup2(d.w), sw, s0, s1);
                        }
                    }
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            int x = q + 32 * j;
            if (x >= places) continue;
            const float kf = j ? k.y : k.x;
            if (x < nd2) {
                const int row = x / nd, t = (row + 1) * Td + (x - row * nd) + 1;
                const float w = j ? sw.y : sw.x;
                const bool ok = kf > 0.f && w > 1e-37f;
                float2 v = dep_load(V, B.dep, dof + t);
                uint32_t c = B.dep_n[dof + t];
                // the batch as its mean with zero offset sum and k x its variance s1 / w
                if (ok) v = dep_texel_blend(v, c, j ? s0.y : s0.x, 0.0f, (j ? s1.y : s1.x) * (kf / w), (uint32_t)kf, omh);
                if (cl == 1) c = min(c, 16u);
                dep_new[t] = v;
                dn_new[t] = (uint8_t)c;
            } else {
                x -= nd2;
                const int row = x / ni, t = (row + 1) * Ti + (x - row * ni) + 1;
                const float w = j ? iw.y : iw.x;
                const bool ok = kf > 0.0f && w > 0.0f;
                const float inv = ok ? kf / w : 0.0f;  // sums of the k-sample batch: mean * k
                float4 v = irr_load(V, B.irr, io + t);
                if (ok) v = irr_texel_blend(v, (j ? r0.y : r0.x) * inv, (j ? r1.y : r1.x) * inv, (j ? r2.y : r2.x) * inv, (uint32_t)kf, omh);
                if (cl == 1) v.w = fminf(v.w, 16.0f);
                irr_new[t] = v;
            }
        }
    }
    __syncthreads();
    store_tiles(V, F, B.irr, B.dep, B.dep_n, B.src, p, irr_new, dep_new, dn_new, threadIdx.x, kCosThreads);
}

// ---- Metropolis samples (sampler.cu): one warp per probe tile.  The
// samples of probe p are contiguous in grouped order (sample order inside the
// probe).  Sample s adds its +w radiance to the irradiance texel of w and the
// distance along -w to the visibility texel of -w (the extra ray of the
// static adaptive sampling); the pilots come first on the first frame of a
// pair.  Per texel the sums run in that order (a chunk's samples of one
// texel summed first, in order); then the batched moving average and the
// stores of k_blend.
struct MhLayout {
    uint32_t acc_i, acc_d, cnt_d, sh_d, dn, e_rec, dacc_i, dacc_d, dcnt_d, dsh_d, total;
};

__host__ __device__ inline MhLayout mh_layout(int Ti, int Td, bool dyn)
{
    const uint32_t ti2 = (uint32_t)(Ti * Ti), td2 = (uint32_t)(Td * Td);
    MhLayout L;
    uint32_t o = 0;
    L.acc_i = o, o += al16(16 * ti2);  // {sum r, g, b, count}, then the updated texel
    L.acc_d = o, o += al16(8 * td2);   // {sum d - x0, sum (d - x0)^2}, then the updated texel
    L.cnt_d = o, o += al16(4 * td2);
    L.sh_d = o, o += al16(4 * td2);    // x0: the texel's first sample (the shift of the sums)
    L.dn = o, o += al16(td2);
    L.e_rec = o, o += 16 * 32;  // one chunk of samples: {r, g, b, depth}
    L.dacc_i = L.dacc_d = L.dcnt_d = L.dsh_d = o;
    if (dyn) {  // the dynamic rays' sums: a second batch step
        L.dacc_i = o, o += al16(16 * ti2);
        L.dacc_d = o, o += al16(8 * td2);
        L.dcnt_d = o, o += al16(4 * td2);
        L.dsh_d = o, o += al16(4 * td2);
    }
    L.total = o;
    return L;
}

// Add a chunk of samples, one per lane (lane j holds sample j of the chunk
// with its texels ki, kd; -1 for none): the lanes of one texel form a group
// (match_any) whose lowest lane sums the group's records in lane order and
// adds the sum to the texel.  Texels are distinct across groups, so the
// adds do not race; per texel the chunks are added in order.
__device__ __forceinline__ void mh_accumulate(const float4* e_rec, int ki, int kd, float4* acc_i, float2* acc_d,
                                              uint32_t* cnt_d, float* sh_d, int lane)
{
    const uint32_t below = (1u << lane) - 1u;
    const uint32_t gi = __match_any_sync(0xFFFFFFFFu, ki), gd = __match_any_sync(0xFFFFFFFFu, kd);
    if (ki >= 0 && (gi & below) == 0u) {
        float sx = 0.f, sy = 0.f, sz = 0.f;
        for (uint32_t m = gi; m; m &= m - 1u) {
            const float4 r = e_rec[__ffs(m) - 1];
            sx += r.x;
            sy += r.y;
            sz += r.z;
        }
        float4 t = acc_i[ki];
        t.x += sx;
        t.y += sy;
        t.z += sz;
        t.w += (float)__popc(gi);
        acc_i[ki] = t;
    }
    if (kd >= 0 && (gd & below) == 0u) {
        // offsets from the texel's first sample (this group's first when the
        // texel has none yet)
        if (cnt_d[kd] == 0u) sh_d[kd] = e_rec[__ffs(gd) - 1].w;
        const float x0 = sh_d[kd];
        float s1 = 0.f, s2 = 0.f;
        for (uint32_t m = gd; m; m &= m - 1u) {
            const float dx = e_rec[__ffs(m) - 1].w - x0;
            s1 += dx;
            s2 += dx * dx;
        }
        float2 t = acc_d[kd];
        t.x += s1;
        t.y += s2;
        acc_d[kd] = t;
        cnt_d[kd] += (uint32_t)__popc(gd);
    }
}

__global__ void __launch_bounds__(128) k_mh_blend(VolConst V, const FrameDev* __restrict__ FD, MhBlendBufs B)
{
    const FrameConst& F = FD->F;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int p = blockIdx.x * (blockDim.x >> 5) + wib;
    if (p >= V.P) return;  // the whole warp
    const uint32_t b0 = __ldg(B.off + p);
    uint32_t b1 = __ldg(B.off + p + 1);
    if (b1 < b0 || b1 > B.n) {
        if (lane == 0) atomicOr(V.err, kErrRayRange);
        b1 = b0;
    }
    const uint8_t cl = V.cls[p];
    if (cl != 2) b1 = b0;  // samples outside V_in are dropped
    const int npil = (F.even && cl >= 1) ? kPilots : 0;
    const uint32_t r0 = V.dyn ? __ldg(B.dyn.off + p) : 0u, r1 = V.dyn ? __ldg(B.dyn.off + p + 1) : 0u;
    if (b1 == b0 && npil == 0 && r1 <= r0 && cl != 1) return;  // untouched tile
    const int Ti = V.Ti, Td = V.Td, ni = V.n_irr, nd = V.n_dep;
    const int ti2 = Ti * Ti, td2 = Td * Td;
    const MhLayout L = mh_layout(Ti, Td, V.dyn != 0);
    unsigned char* ws = smem + (size_t)wib * L.total;
    float4* acc_i = reinterpret_cast<float4*>(ws + L.acc_i);
    float2* acc_d = reinterpret_cast<float2*>(ws + L.acc_d);
    uint32_t* cnt_d = reinterpret_cast<uint32_t*>(ws + L.cnt_d);
    float* sh_d = reinterpret_cast<float*>(ws + L.sh_d);
    uint8_t* dn = ws + L.dn;
    float4* e_rec = reinterpret_cast<float4*>(ws + L.e_rec);
    for (int t = lane; t < ti2; t += 32) acc_i[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int t = lane; t < td2; t += 32) {
        acc_d[t] = make_float2(0.f, 0.f);
        cnt_d[t] = 0u;
    }
    float4* dacc_i = reinterpret_cast<float4*>(ws + L.dacc_i);
    float2* dacc_d = reinterpret_cast<float2*>(ws + L.dacc_d);
    uint32_t* dcnt_d = reinterpret_cast<uint32_t*>(ws + L.dcnt_d);
    float* dsh_d = reinterpret_cast<float*>(ws + L.dsh_d);
    if (V.dyn) {
        for (int t = lane; t < ti2; t += 32) dacc_i[t] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int t = lane; t < td2; t += 32) {
            dacc_d[t] = make_float2(0.f, 0.f);
            dcnt_d[t] = 0u;
        }
    }
    __syncwarp();
    if (npil) {
        int ki = -1, kd = -1;
        if (lane < kPilots) {
            e_rec[lane] = __ldg(B.pil_rec + (size_t)p * kPilots + lane);
            const float2 e = oct_encode_x(pilot_dir(F.pilot_key, (uint32_t)p, lane));
            ki = texel_of(e, ni);
            kd = texel_of(e, nd);
        }
        __syncwarp();
        mh_accumulate(e_rec, ki, kd, acc_i, acc_d, cnt_d, sh_d, lane);
        __syncwarp();
    }
    // chunks of 32 samples, one per lane; the next chunk's loads are issued
    // before the current chunk is added (two chunks in flight per warp)
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), x = a;
    int2 hn = make_int2((int)kMiss, 0);
    if (b0 + lane < b1) {
        a = __ldg(B.smp_g + b0 + lane);
        x = __ldg(B.rec + b0 + lane);
        hn = __ldg(B.hit_neg + b0 + lane);
    }
    for (uint32_t c0 = b0; c0 < b1; c0 += 32) {
        int ki = -1, kd = -1;
        if (c0 + lane < b1) {
            const float dep = (uint32_t)hn.x == kMiss ? V.depth_max : fminf(__int_as_float(hn.y), V.depth_max);
            e_rec[lane] = make_float4(x.x, x.y, x.z, dep);
            ki = texel_of(oct_encode_x(make_float3(a.x, a.y, a.z)), ni);
            const float4 an = B.smp_gn ? __ldg(B.smp_gn + c0 + lane) : make_float4(-a.x, -a.y, -a.z, 0.f);
            kd = texel_of(oct_encode_x(make_float3(an.x, an.y, an.z)), nd);
        }
        __syncwarp();
        const uint32_t qn = c0 + 32 + lane;
        if (qn < b1) {
            a = __ldg(B.smp_g + qn);
            x = __ldg(B.rec + qn);
            hn = __ldg(B.hit_neg + qn);
        }
        mh_accumulate(e_rec, ki, kd, acc_i, acc_d, cnt_d, sh_d, lane);
        __syncwarp();
    }
    // the dynamic rays of the probe (each at its own texel centre): sums of
    // the second batch step
    for (uint32_t c0 = r0; c0 < r1; c0 += 32) {
        int ki = -1, kd = -1;
        if (c0 + lane < r1) {
            int pp, t;
            float3 d;
            if (dyn_ray_of(V, B.dyn, c0 + lane, pp, t, d) && pp == p) {
                e_rec[lane] = __ldg(B.drec + c0 + lane);
                ki = t;
                kd = texel_of(oct_encode_x(d), nd);
            } else {
                atomicOr(V.err, kErrRayRange);
            }
        }
        __syncwarp();
        mh_accumulate(e_rec, ki, kd, dacc_i, dacc_d, dcnt_d, dsh_d, lane);
        __syncwarp();
    }
    const float omh = 1.0f - V.hyst;
    const float rni = 1.0f / (float)ni, rnd = 1.0f / (float)nd;
    const size_t io = (size_t)p * ti2, dof = (size_t)p * td2;
    for (int q = lane; q < ni * ni; q += 32) {
        const int r = tile_row(q, rni), t = (r + 1) * Ti + (q - r * ni) + 1;
        const float4 sum = acc_i[t];
        float4 v = irr_load(V, B.irr, io + t);
        if (sum.w > 0.0f) v = irr_texel_blend(v, sum.x, sum.y, sum.z, (uint32_t)sum.w, omh);
        if (V.dyn) {
            const float4 ds = dacc_i[t];
            if (ds.w > 0.0f) v = irr_texel_blend(v, ds.x, ds.y, ds.z, (uint32_t)ds.w, 1.0f - V.hyst_dyn);
        }
        if (cl == 1) v.w = fminf(v.w, 16.0f);
        acc_i[t] = v;
    }
    for (int q = lane; q < nd * nd; q += 32) {
        const int r = tile_row(q, rnd), t = (r + 1) * Td + (q - r * nd) + 1;
        const float2 sum = acc_d[t];
        const uint32_t k = cnt_d[t];
        float2 v = dep_load(V, B.dep, dof + t);
        uint32_t c = B.dep_n[dof + t];
        if (k) v = dep_texel_blend(v, c, sh_d[t], sum.x, sum.y, k, omh);
        if (V.dyn) {
            const uint32_t kd2 = dcnt_d[t];
            const float2 ds = dacc_d[t];
            if (kd2) v = dep_texel_blend(v, c, dsh_d[t], ds.x, ds.y, kd2, 1.0f - V.hyst_dyn);
        }
        if (cl == 1) c = min(c, 16u);
        acc_d[t] = v;
        dn[t] = (uint8_t)c;
    }
    __syncwarp();
    store_tiles(V, F, B.irr, B.dep, B.dep_n, B.src, p, acc_i, acc_d, dn, lane);
}

// ============================================================== query
// One thread a point.  Bound by instruction issue (some 2,000 a warp of points,
// a quarter of them the exact cage weights) and the latency of the eight
// probes' gathers: 518,400 points in screen order 47 -> 37 us with the kernel
// made for the storage format (the loads of a probe stay in one block of
// code), the offsets formed once per plane and one address product a tile.
template <int kFmt>
__global__ void __launch_bounds__(128) k_query(VolConst V, const void* __restrict__ irr, const void* __restrict__ dep,
                                               const float* __restrict__ pos, const float* __restrict__ nrm, int n,
                                               float* __restrict__ out)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float3 x = make_float3(pos[3 * (size_t)i], pos[3 * (size_t)i + 1], pos[3 * (size_t)i + 2]);
    float3 nn = make_float3(nrm[3 * (size_t)i], nrm[3 * (size_t)i + 1], nrm[3 * (size_t)i + 2]);
    float3 e = query_irr_at<kFmt, true>(V, irr, dep, x, 0.0f, make_float3(0.f, 0.f, 0.f), nn);
    out[3 * (size_t)i] = e.x;
    out[3 * (size_t)i + 1] = e.y;
    out[3 * (size_t)i + 2] = e.z;
}

// Few points: eight lanes a point, one probe each, so that the eight gathers
// are in flight together; every lane then adds the eight terms in k_query's
// order, so a point's result does not depend on how many are asked for.
template <int kFmt>
__global__ void __launch_bounds__(128) k_query_few(VolConst V, const void* __restrict__ irr, const void* __restrict__ dep,
                                                   const float* __restrict__ pos, const float* __restrict__ nrm, int n,
                                                   float* __restrict__ out)
{
    const int i0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 3, c = threadIdx.x & 7;
    const int i = min(i0, n - 1);  // every lane takes part in the shuffles
    float os[3] = {pos[3 * (size_t)i], pos[3 * (size_t)i + 1], pos[3 * (size_t)i + 2]}, ds[3] = {0.f, 0.f, 0.f};
    float3 nn = make_float3(nrm[3 * (size_t)i], nrm[3 * (size_t)i + 1], nrm[3 * (size_t)i + 2]);
    const Cage C = cage_of<true>(V, os, 0.0f, ds);
    const IrrTaps taps = normal_taps(V, nn);
    float wt, wc, E[3];
    query_probe<kFmt>(V, irr, dep, os, 0.0f, ds, C, taps, c, wt, wc, E);
    float sum[3] = {0.f, 0.f, 0.f}, sumt[3] = {0.f, 0.f, 0.f}, sw = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float t = __shfl_sync(0xFFFFFFFFu, wt, k, 8), w = t * __shfl_sync(0xFFFFFFFFu, wc, k, 8);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float e = __shfl_sync(0xFFFFFFFFu, E[j], k, 8);
            sum[j] += w * e;
            sumt[j] += t * e;
        }
        sw += w;
    }
    if (i0 < n && c < 3) {
        const float s = c == 0 ? sum[0] : c == 1 ? sum[1] : sum[2], st = c == 0 ? sumt[0] : c == 1 ? sumt[1] : sumt[2];
        out[3 * (size_t)i + c] = sw >= 1e-12f ? s / sw : st;
    }
}

}  // namespace

size_t blend_plan_bytes(int M, int Ti, int Td)
{
    const size_t m = (size_t)(M > 0 ? M : 0), tri = m * (m + 1) / 2;
    return sizeof(uint16_t) * (2 * tri + m * ((size_t)Ti * Ti + 1) + m * ((size_t)Td * Td + 1) + 8);
}

BlendPlan carve_blend_plan(void* base, int M, int Ti, int Td)
{
    const size_t m = (size_t)(M > 0 ? M : 0), tri = m * (m + 1) / 2;
    uint16_t* b = reinterpret_cast<uint16_t*>(base);
    BlendPlan P;
    P.ord_i = b;
    P.ord_d = b + tri;
    P.beg_i = b + 2 * tri;
    P.beg_d = P.beg_i + m * ((size_t)Ti * Ti + 1);
    return P;
}

// shared memory of one probe (one warp) of k_blend
size_t blend_smem_bytes(const VolConst& V) { return blend_layout(V.Ti, V.Td).total; }

cudaError_t launch_change(const VolConst& V, const FrameDev* FD, const ChangeBufs& B, cudaStream_t s, int parts)
{
    const int n = V.p_hi - V.p_lo;
    if (n <= 0) return cudaSuccess;
    if (parts & 1) {
        k_change_state<<<(n + 15) / 16, 128, 0, s>>>(V, FD, B);
        count_launches(1);
    }
    if (parts & 2) {
        k_change_weight<<<(n + 15) / 16, 128, 0, s>>>(V, FD, B);
        count_launches(1);
    }
    return cudaGetLastError();
}

cudaError_t launch_classify(const VolConst& V, const FrameDev* FD, const uint16_t* lut_c, uint8_t* cls,
                            cudaStream_t s)
{
    k_classify<<<(V.P + 255) / 256, 256, 0, s>>>(V, FD, lut_c, cls);
    count_launches(1);
    return cudaGetLastError();
}

// The dynamic shared-memory limit of a kernel is one attribute per device,
// shared by every launch in the process, graphs captured earlier included.
// It is only ever raised: lowering it for a small volume could invalidate a
// launch or a graph made for a larger one.
cudaError_t raise_smem_limit(const void* func, size_t bytes)
{
    if (bytes <= 48 * 1024) return cudaSuccess;
    static std::mutex mu;
    static std::map<std::pair<int, const void*>, size_t> limit;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> g(mu);
    size_t& cur = limit[{dev, func}];
    if (bytes <= cur) return cudaSuccess;
    e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) cur = bytes;
    return e;
}

// One CTA up to kAllocOneCta probes (a warp per 32 of them: a smaller block
// passes its barriers sooner), the cluster beyond: its passes over fewer probes
// a thread then make up for a cluster barrier each.  One CTA / cluster, us,
// events around the call: dense weights 1,024 probes 15.5 / 20.8, 4,096 19.1 /
// 20.5, 6,144 22.2 / 20.8, 8,192 24.8 / 21.0, 16,384 29.8 / 20.3; 3 % of the
// probes weighted: 15.6 / 20.7, 18.6 / 21.1, 21.4 / 21.4, 23.4 / 21.4, 33.3 /
// 22.5.
constexpr int kAllocOneCta = 5120;

cudaError_t launch_allocate(const uint32_t* W, int P, int avg, int m0, int rmax, uint32_t* n_out, uint32_t* off_out,
                            cudaStream_t s, const uint8_t* cls)
{
    if (P <= kAllocOneCta) {
        const int t = std::min(kAllocThreads, (P + 31) / 32 * 32);
        cudaError_t e = raise_smem_limit((const void*)k_allocate, 8 * kAllocOneCta);
        if (e != cudaSuccess) return e;
        k_allocate<<<1, t, 8 * P, s>>>(W, P, avg, m0, rmax, n_out, off_out, cls);
    } else if (P <= kAllocCluster * kAllocStage) {
        const int sm = 8 * ((P + kAllocCluster - 1) / kAllocCluster);
        // the limit for the largest grid the staged cluster takes, set once
        cudaError_t e = raise_smem_limit((const void*)k_allocate_cluster<true>, 8 * kAllocStage);
        if (e != cudaSuccess) return e;
        k_allocate_cluster<true><<<kAllocCluster, kAllocThreads, sm, s>>>(W, P, avg, m0, rmax, n_out, off_out, cls);
    } else {
        k_allocate_cluster<false><<<kAllocCluster, kAllocThreads, 0, s>>>(W, P, avg, m0, rmax, n_out, off_out, cls);
    }
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_blend_plan(const VolConst& V, const FrameDev* FD, const float4* sf, const BlendPlan& plan,
                              cudaStream_t s)
{
    const int M = V.rays_max - kPilots;
    if (M <= 0) return cudaSuccess;
    const size_t ps = blend_plan_smem(V);
    {
        cudaError_t e = raise_smem_limit((const void*)k_blend_plan, ps);
        if (e != cudaSuccess) return e;
    }
    k_blend_plan<<<M, 256, ps, s>>>(V, FD, sf, plan);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_blend(const VolConst& V, const FrameDev* FD, const BlendBufs& B, const Tuning& T, cudaStream_t s)
{
    // probes per CTA (one warp each), as many as the tuning asks and 227 KB allow
    const size_t per = blend_smem_bytes(V);
    const int wpb = std::max(1, std::min(T.blend_block / 32, (int)((227u * 1024u) / per)));
    const size_t sm = per * (size_t)wpb;
    {
        cudaError_t e = raise_smem_limit((const void*)k_blend, sm);
        if (e != cudaSuccess) return e;
    }
    const int np = V.p_hi - V.p_lo;
    if (np <= 0) return cudaSuccess;
    k_blend<<<(np + wpb - 1) / wpb, 32 * wpb, sm, s>>>(V, FD, B);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_blend_cos(const VolConst& V, const FrameDev* FD, const BlendBufs& B, const Tuning& T, cudaStream_t s)
{
    (void)T;
    const size_t sm = cos_layout(V.Ti, V.Td).total;
    {
        cudaError_t e = raise_smem_limit((const void*)k_blend_cos, sm);
        if (e != cudaSuccess) return e;
    }
    const int np = V.p_hi - V.p_lo;
    if (np <= 0) return cudaSuccess;
    k_blend_cos<<<np, kCosThreads, sm, s>>>(V, FD, B, 1.0f, -0.0f);
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_mh_blend(const VolConst& V, const FrameDev* FD, const MhBlendBufs& B, cudaStream_t s)
{
    // Bound by the latency of the ordered sums with as many warps as shared
    // memory holds (11 KB each with dynamic chains).  One warp a block, so that
    // a probe of few samples gives its memory back at once: 279 (four) -> 258 us a
    // tunnel update (1,276 samples in the fullest probe, 198 on average; two:
    // 265); without dynamic chains 194 -> 188.
    const size_t sm = mh_layout(V.Ti, V.Td, V.dyn != 0).total;
    cudaError_t e = raise_smem_limit((const void*)k_mh_blend, sm);
    if (e != cudaSuccess) return e;
    k_mh_blend<<<V.P, 32, sm, s>>>(V, FD, B);
    count_launches(1);
    return cudaGetLastError();
}

// Up to here eight lanes a point (us, eight lanes / one thread a point, points
// in screen order: 64 points 5.2 / 8.3, 5,000 6.2 / 8.5, 10,000 8.1 / 8.7,
// 20,000 9.3 / 9.3, 32,768 12.3 / 10.3; unordered points 1,000 6.2 / 10.3,
// 20,000 10.3 / 12.3, 32,768 12.9 / 12.4)
constexpr int kQueryFew = 16384;

cudaError_t launch_query(const VolConst& V, const void* irr, const void* dep, const float* pos, const float* nrm, int n,
                         float* out, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    if (n <= kQueryFew) {
        auto few = V.fp16 == 3 ? k_query_few<3> : V.fp16 ? k_query_few<1> : k_query_few<0>;
        few<<<(n + 15) / 16, 128, 0, s>>>(V, irr, dep, pos, nrm, n, out);
    } else {
        auto query = V.fp16 == 3 ? k_query<3> : V.fp16 ? k_query<1> : k_query<0>;
        query<<<(n + 127) / 128, 128, 0, s>>>(V, irr, dep, pos, nrm, n, out);
    }
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace adgi
