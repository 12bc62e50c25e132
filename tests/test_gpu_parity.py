"""GPU parity: the CUDA path (through the C ABI) against the CPU oracle.

Bit-exact: ray allocation, heuristics, pilot luminance, hit indices and t,
texel counts.  Tolerances (tests/_helpers.py): irradiance 1e-3 relative,
depth moments 1e-4 relative.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2301_05125_gb300 import scenegen as S

from _helpers import DEP_RTOL, IRR_RTOL, diag_path, gpu_volume, oracle_volume, rel_check

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def adgi():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_05125_gb300 import adgi as A
    from paper_2301_05125_gb300 import build

    build.build()
    A.load()
    return A


def _dump_rays(gv, ov, frame, what):
    def dump(rows):
        R = int(ov.off()[-1])
        np.savez(diag_path("fail_%s_f%d.npz" % (what.replace(" ", "_"), frame)), rows=rows[:64],
                 gpu_rec=gv.main_rec()[:R][rows[:64]], ora_rad=ov.main_rad()[rows[:64]],
                 ora_dep=ov.main_dep()[rows[:64]], tri=ov.main_tri()[rows[:64]], t=ov.main_t()[rows[:64]],
                 off=ov.off(), n=ov.n())
    return dump


def _compare_update(gv, ov, frame, check_atlas=True, what=""):
    tag = "%s frame %d" % (what, frame)
    gv.stats()  # raises if a device-side anomaly flag was set
    np.testing.assert_array_equal(gv.W(), ov.W(), err_msg=tag + " W")
    np.testing.assert_array_equal(gv.n(), ov.n(), err_msg=tag + " n")
    np.testing.assert_array_equal(gv.off(), ov.off(), err_msg=tag + " off")
    np.testing.assert_array_equal(gv.qv(), ov.qv(), err_msg=tag + " qv")
    np.testing.assert_array_equal(gv.qr(), ov.qr(), err_msg=tag + " qr")
    np.testing.assert_array_equal(gv.trv(), ov.trv(), err_msg=tag + " trv")
    np.testing.assert_array_equal(gv.trr(), ov.trr(), err_msg=tag + " trr")
    ph = gv.pilot_hit()
    from paper_2301_05125_gb300 import adgi as A

    np.testing.assert_array_equal(A.hit_tri(ph), ov.pilot_tri(), err_msg=tag + " pilot tri")
    hitm = ov.pilot_tri() >= 0
    np.testing.assert_array_equal(A.hit_t(ph)[hitm], ov.pilot_t()[hitm], err_msg=tag + " pilot t")
    np.testing.assert_array_equal(gv.pilot_lum(), ov.pilot_lum().astype(np.float32), err_msg=tag + " pilot lum")
    R = int(ov.off()[-1])
    mh = gv.main_hit()[:R]
    np.testing.assert_array_equal(A.hit_tri(mh), ov.main_tri(), err_msg=tag + " main tri")
    hm = ov.main_tri() >= 0
    np.testing.assert_array_equal(A.hit_t(mh)[hm], ov.main_t()[hm], err_msg=tag + " main t")
    rel_check(gv.main_rec()[:R, :3], ov.main_rad(), IRR_RTOL, tag + " main radiance",
              dump=_dump_rays(gv, ov, frame, what))
    rel_check(gv.main_rec()[:R, 3], ov.main_dep(), DEP_RTOL, tag + " main depth")
    if check_atlas:
        gi, oi = gv.irr(), ov.irr()
        np.testing.assert_array_equal(gi[..., 3].astype(np.int64), ov.irr_n().astype(np.int64),
                                      err_msg=tag + " irr counts")
        np.testing.assert_array_equal(gv.dep_n(), ov.dep_n(), err_msg=tag + " depth counts")
        e_i = rel_check(gi[..., :3], oi, IRR_RTOL, tag + " irradiance atlas")
        e_d = rel_check(gv.dep_moments(), ov.dep(), DEP_RTOL, tag + " depth atlas")
        return e_i, e_d
    return None


# ------------------------------------------------------------------ allocation
# 196608 is the largest grid of the 8-CTA cluster kernel, 196609 the smallest
# of the one-block kernel
@pytest.mark.parametrize("P", [1, 7, 64, 1000, 1025, 16384, 24576, 131072, 196608, 196609, 200000])
def test_allocation_bit_exact(adgi, P):
    rng = np.random.default_rng(P)
    cases = [
        (rng.integers(0, 1 << 24, P), 64, 8, 256),
        (rng.integers(0, 3, P), 64, 4, 512),
        (np.where(rng.random(P) < 0.01, rng.integers(1, 1 << 24, P), 0), 256, 8, 1024),
        (np.zeros(P, np.int64), 33, 8, 40),
        (np.full(P, 5), 9, 8, 9),
        (rng.integers(0, 2, P) * ((1 << 24) - 1), 100, 16, 101),
        (rng.integers(0, 1 << 32, P, dtype=np.uint64), 64, 8, 256),  # weights beyond what the heuristics make
    ]
    dev = torch.device("cuda")
    for W, avg, rmin, rmax in cases:
        W = W.astype(np.uint32)
        n_ref, off_ref = O.allocate(W, avg, rmin, rmax)
        Wd = torch.from_numpy(W.view(np.int32)).to(dev)
        nd = torch.empty(P, dtype=torch.int32, device=dev)
        od = torch.empty(P + 1, dtype=torch.int32, device=dev)
        adgi.adgi_allocate_rays(Wd, avg, rmin, rmax, nd, od, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(nd.cpu().numpy().view(np.uint32), n_ref)
        np.testing.assert_array_equal(od.cpu().numpy().view(np.uint32), off_ref)


# the edges of the one-CTA / cluster / global-memory rule, with weights that
# leave long remainders (few weighted probes at their cap, the rest one ray a
# round) and rounds that end when a probe reaches its cap
@pytest.mark.parametrize("P", [2, 31, 33, 1024, 8191, 8192, 8193, 196609])
def test_allocation_long_remainders(adgi, P):
    rng = np.random.default_rng(P + 5)
    dev = torch.device("cuda")
    few = np.where(rng.random(P) < 0.02, rng.integers(1, 9, P), 0)
    one = np.zeros(P, np.int64)
    one[P // 2] = 7
    for W, avg, rmin, rmax in [(few, 300, 8, 1024), (one, 97, 16, 200), (one, 200, 8, 200), (np.ones(P, np.int64), 33, 8, 34),
                               (rng.integers(0, 2, P), 63, 8, 64), (few, 8, 8, 64)]:
        W = W.astype(np.uint32)
        n_ref, off_ref = O.allocate(W, avg, rmin, rmax)
        Wd = torch.from_numpy(W.view(np.int32)).to(dev)
        nd = torch.empty(P, dtype=torch.int32, device=dev)
        od = torch.empty(P + 1, dtype=torch.int32, device=dev)
        adgi.adgi_allocate_rays(Wd, avg, rmin, rmax, nd, od, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(nd.cpu().numpy().view(np.uint32), n_ref)
        np.testing.assert_array_equal(od.cpu().numpy().view(np.uint32), off_ref)


@pytest.mark.parametrize("P", [5119, 5120, 5121])
def test_allocation_at_the_one_cta_edge(adgi, P):
    test_allocation_bit_exact(adgi, P)
    test_allocation_long_remainders(adgi, P)


def test_allocation_large_then_smaller_then_large(adgi):
    # the cluster kernel's shared memory grows with P (8 B a probe): a grid
    # above 49,152 probes, then a smaller one also above it, then the larger
    # again must all match the oracle (the kernel's shared-memory limit is
    # never lowered by the smaller grid)
    dev = torch.device("cuda")
    rng = np.random.default_rng(21)
    for P in (131072, 60000, 131072, 50000, 196608):
        W = rng.integers(0, 1 << 24, P).astype(np.uint32)
        n_ref, off_ref = O.allocate(W, 64, 8, 256)
        Wd = torch.from_numpy(W.view(np.int32)).to(dev)
        nd = torch.empty(P, dtype=torch.int32, device=dev)
        od = torch.empty(P + 1, dtype=torch.int32, device=dev)
        adgi.adgi_allocate_rays(Wd, 64, 8, 256, nd, od, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(nd.cpu().numpy().view(np.uint32), n_ref, err_msg="P=%d" % P)
        np.testing.assert_array_equal(od.cpu().numpy().view(np.uint32), off_ref, err_msg="P=%d" % P)


def test_graph_of_large_volume_replays_after_smaller_capture(adgi):
    # two volumes above 49,152 probes (cluster allocation with more than
    # 48 KB of shared memory): the larger one's captured update graph is
    # replayed after the smaller one was captured, and must still equal
    # plain updates of an identical volume
    w = S.box_room(1)
    big = dict(origin=(0.2, 0.2, 0.2), spacing=(7.6 / 63, 7.6 / 31, 7.6 / 63), dims=(64, 32, 64), rays_avg=9,
               rays_min=8, rays_max=24)
    small = dict(big, dims=(60, 25, 40), spacing=(7.6 / 59, 7.6 / 24, 7.6 / 39))
    g_big = gpu_volume(adgi, w, **big)
    p_big = gpu_volume(adgi, w, **big)
    g_small = gpu_volume(adgi, w, **small)
    wsum = 0
    for f in range(5):
        lights = w.lights_at(f)
        g_big.update_graph(f, w.seed, lights, w.sky)
        g_small.update_graph(f, w.seed, lights, w.sky)
        p_big.update(f, w.seed, lights, w.sky)
        torch.cuda.synchronize()
        g_big.stats()
        np.testing.assert_array_equal(g_big.W(), p_big.W(), err_msg="frame %d W" % f)
        np.testing.assert_array_equal(g_big.n(), p_big.n(), err_msg="frame %d n" % f)
        np.testing.assert_array_equal(g_big.main_hit(), p_big.main_hit(), err_msg="frame %d hits" % f)
        np.testing.assert_array_equal(g_big.irr(), p_big.irr(), err_msg="frame %d irradiance" % f)
        wsum += int(p_big.W().astype(np.int64).sum())
    assert wsum > 0  # some allocation was not uniform
    for v in (g_big, p_big, g_small):
        v.close()


def test_allocation_rejects_impossible_budget(adgi):
    dev = torch.device("cuda")
    W = torch.zeros(10, dtype=torch.int32, device=dev)
    n = torch.empty(10, dtype=torch.int32, device=dev)
    off = torch.empty(11, dtype=torch.int32, device=dev)
    with pytest.raises(adgi.AdgiError):
        adgi.adgi_allocate_rays(W, 300, 8, 256, n, off)


# ------------------------------------------------------------------ tracing
def _trace_case(adgi, w, O_, D, use_bvh):
    gv = gpu_volume(adgi, w)
    dev = torch.device("cuda")
    o = torch.from_numpy(O_).to(dev)
    d = torch.from_numpy(D).to(dev)
    n = O_.shape[0]
    t = torch.empty(n, dtype=torch.float32, device=dev)
    tri = torch.empty(n, dtype=torch.int32, device=dev)
    adgi.adgi_trace_closest(gv.h, o, d, 1e-4, float("inf"), t, tri)
    torch.cuda.synchronize()
    t_ref, tri_ref, det_ref = O.trace_closest(w.verts, w.idx, O_, D, 1e-4, np.inf, use_bvh=use_bvh)
    h = np.stack([tri.cpu().numpy(), t.cpu().numpy().view(np.int32)], 1)
    np.testing.assert_array_equal(adgi.hit_tri(h), tri_ref)
    np.testing.assert_array_equal(t.cpu().numpy(), t_ref)
    hit = tri_ref >= 0
    np.testing.assert_array_equal(adgi.hit_back(h)[hit], (det_ref < 0)[hit])
    gv.close()


def test_trace_room_bit_exact_vs_brute_force(adgi):
    rng = np.random.default_rng(11)
    w = S.box_room(1)
    n = 200000
    O_ = rng.uniform(0.1, 7.9, (n, 3)).astype(np.float32)
    D = rng.normal(size=(n, 3)).astype(np.float32)
    # rays aimed exactly at box edges and corners stress watertightness
    tgt = w.verts[rng.integers(0, len(w.verts), n // 4)]
    D[: n // 4] = (tgt - O_[: n // 4]).astype(np.float32)
    _trace_case(adgi, w, O_, D, use_bvh=False)


def test_trace_city_bit_exact_vs_oracle(adgi):
    rng = np.random.default_rng(12)
    w = S.small_city(3, n_boxes=2000)
    n = 100000
    O_ = rng.uniform(-40, 40, (n, 3)).astype(np.float32)
    O_[:, 1] = rng.uniform(0.5, 30, n)
    D = rng.normal(size=(n, 3)).astype(np.float32)
    _trace_case(adgi, w, O_, D, use_bvh=True)


def test_trace_axis_aligned_directions(adgi):
    # directions with exact zero components (axis-aligned rays, rays in a
    # coordinate plane, signed zeros): 1/0 in the box test must not reject boxes
    rng = np.random.default_rng(14)
    w = S.small_city(3, n_boxes=2000)
    n = 60000
    O_ = rng.uniform(-40, 40, (n, 3)).astype(np.float32)
    O_[:, 1] = rng.uniform(0.5, 30, n)
    D = rng.normal(size=(n, 3)).astype(np.float32)
    ax = rng.integers(0, 3, n)
    D[np.arange(n) % 3 == 0, :] = 0.0  # axis-aligned: keep one component
    keep = np.arange(n) % 3 == 0
    D[keep, ax[keep]] = np.where(rng.random(keep.sum()) < 0.5, -1.0, 1.0)
    one = np.arange(n) % 3 == 1  # one component zero (+0 or -0)
    D[one, ax[one]] = np.where(rng.random(one.sum()) < 0.5, 0.0, -0.0)
    _trace_case(adgi, w, O_, D, use_bvh=True)


def test_update_axis_aligned_sun(adgi):
    # a sun straight down: every shadow ray points straight up (two zero
    # direction components)
    w = S.small_city(4, n_boxes=800, dims=(9, 5, 7), rays_avg=40)
    sun = [(1, (0.0, -1.0, 0.0), (2.0, 2.0, 2.0))]
    gv = gpu_volume(adgi, w)
    ov = oracle_volume(O, w)
    for f in range(2):
        gv.update(f, w.seed, sun, w.sky)
        ov.update(f, w.seed, sun, w.sky)
        _compare_update(gv, ov, f, what="axis-aligned sun")
    gv.close()


def test_trace_degenerate_scenes(adgi):
    rng = np.random.default_rng(13)
    O_ = rng.uniform(-1, 1, (5000, 3)).astype(np.float32)
    D = rng.normal(size=(5000, 3)).astype(np.float32)
    one = S.Workload("one", 0, np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0]], np.float32),
                     np.array([[0, 1, 2]], np.int32), np.ones((1, 3), np.float32), S.box_room(1).volume, 1,
                     (0, 0, 0), lambda f: [])
    _trace_case(adgi, one, O_, D, use_bvh=False)
    # duplicated triangles: ties must resolve to the smaller index
    dup = S.Workload("dup", 0, one.verts, np.repeat(one.idx, 5, 0), np.ones((5, 3), np.float32),
                     S.box_room(1).volume, 1, (0, 0, 0), lambda f: [])
    _trace_case(adgi, dup, O_, D, use_bvh=False)


@pytest.mark.parametrize("n_quads", [1, 2, 3, 5, 400])
def test_trace_triangle_pairs(adgi, n_quads):
    # quads split along a shared edge, in every vertex order and orientation
    # of their two triangles, some degenerate, some with a duplicate; rays
    # through their corners, edges and diagonals; a moved triangle besides
    rng = np.random.default_rng(40 + n_quads)
    verts, idx = [], []
    for q in range(n_quads):
        c = rng.uniform(-4, 4, 3)
        a, b = rng.normal(size=3), rng.normal(size=3)
        if q % 7 == 3:
            b = 2.0 * a  # degenerate: a line
        k = len(verts)
        verts += [c, c + a, c + a + b, c + b]
        t1, t2 = [k, k + 1, k + 2], [k, k + 2, k + 3]
        if q % 5 == 4:
            t2.reverse()  # the shared edge in the same direction
        idx += [np.roll(t1, q % 3), np.roll(t2, (q // 3) % 3)]
        if q % 11 == 7:
            idx.append(np.roll(t2, 1))
    first = len(verts)
    verts += [(9.0, 9.0, 9.0), (9.5, 9.0, 9.0), (9.0, 9.5, 9.0)]
    idx.append([first, first + 1, first + 2])
    verts, idx = np.array(verts, np.float32), np.array(idx, np.int32)
    w = S.Workload("pairs", 0, verts, idx, np.ones((len(idx), 3), np.float32), S.box_room(1).volume, 1, (0, 0, 0),
                   lambda f: [])
    n = 40000
    o = rng.uniform(-6, 6, (n, 3)).astype(np.float32)
    d = rng.normal(size=(n, 3)).astype(np.float32)
    quad = 4 * rng.integers(0, n_quads, n)
    u = rng.random((n, 1)).astype(np.float32)
    on_diag = verts[quad] + u * (verts[quad + 2] - verts[quad])
    d[: n // 4] = (on_diag - o)[: n // 4]
    d[n // 4: n // 2] = (verts[quad + rng.integers(0, 4, n)] - o)[n // 4: n // 2]
    gv = gpu_volume(adgi, w)
    moved = verts[first:] + np.float32(0.25)
    gv.move_vertices(first, moved)
    now = verts.copy()
    now[first:] = moved
    dev = torch.device("cuda")
    t = torch.empty(n, dtype=torch.float32, device=dev)
    tri = torch.empty(n, dtype=torch.int32, device=dev)
    adgi.adgi_trace_closest(gv.h, torch.from_numpy(o).to(dev), torch.from_numpy(d).to(dev), 1e-4, float("inf"), t, tri)
    torch.cuda.synchronize()
    gv.stats()
    t_ref, tri_ref, det_ref = O.trace_closest(now, idx, o, d, 1e-4, np.inf, use_bvh=False)
    h = np.stack([tri.cpu().numpy(), t.cpu().numpy().view(np.int32)], 1)
    np.testing.assert_array_equal(adgi.hit_tri(h), tri_ref)
    np.testing.assert_array_equal(t.cpu().numpy(), t_ref)
    hit = tri_ref >= 0
    np.testing.assert_array_equal(adgi.hit_back(h)[hit], (det_ref < 0)[hit])
    gv.close()


@pytest.mark.parametrize("n_tris,moved", [(2, 0), (3, 0), (4, 1), (5, 0), (7, 2), (64, 0), (300, 30)])
def test_trace_rays_that_are_not_finite(adgi, n_tris, moved):
    # NaN and infinite components hit every box, the empty slots of the 4-wide
    # nodes too: no record outside the tree is read, and what is hit is what
    # the test of every triangle says (nothing, or the finite rays' hits)
    rng = np.random.default_rng(n_tris)
    verts = rng.normal(size=(3 * n_tris, 3)).astype(np.float32)
    idx = np.arange(3 * n_tris, dtype=np.int32).reshape(-1, 3)
    w = S.Workload("soup", 0, verts, idx, np.ones((n_tris, 3), np.float32), S.box_room(1).volume, 1, (0, 0, 0), lambda f: [])
    gv = gpu_volume(adgi, w)
    if moved:
        verts = verts.copy()
        verts[: 3 * moved] += np.float32(0.5)
        gv.move_vertices(0, verts[: 3 * moved])
    odd = np.array([0.0, -0.0, 1.0, -1.0, 1e-38, 1e30, -1e30, np.inf, -np.inf, np.nan], np.float32)
    n = 4096
    o, d = (rng.normal(size=(n, 3)).astype(np.float32) for _ in range(2))
    for a in (o, d):
        pick = rng.random((n, 3)) < rng.random((n, 1))
        a[pick] = odd[rng.integers(0, len(odd), int(pick.sum()))]
    o[:8], d[:8] = 0.0, [[x, y, z] for x in (np.inf, np.nan) for y in (np.inf, -np.inf) for z in (np.inf, np.nan)]
    dev = torch.device("cuda")
    t = torch.empty(n, dtype=torch.float32, device=dev)
    tri = torch.empty(n, dtype=torch.int32, device=dev)
    adgi.adgi_trace_closest(gv.h, torch.from_numpy(o).to(dev), torch.from_numpy(d).to(dev), 1e-4, float("inf"), t, tri)
    torch.cuda.synchronize()
    gv.stats()
    t_ref, tri_ref, _ = O.trace_closest(verts, idx, o, d, 1e-4, np.inf, use_bvh=False)
    real = np.isfinite(o).all(1) & np.isfinite(d).all(1)
    fin = real & (np.abs(o) < 1e6).all(1) & (np.abs(d) < 1e6).all(1) & (np.abs(d).max(1) > 1e-3)
    h = np.stack([tri.cpu().numpy(), t.cpu().numpy().view(np.int32)], 1)
    np.testing.assert_array_equal(adgi.hit_tri(h)[fin], tri_ref[fin])
    np.testing.assert_array_equal(t.cpu().numpy()[fin], t_ref[fin])
    assert (tri_ref[~real] == -1).all() and (tri.cpu().numpy()[~real] == -1).all()
    gv.close()


# ------------------------------------------------------------------ full update
def test_update_room_bit_exact_and_within_tolerance(adgi):
    w = S.box_room(1)
    gv = gpu_volume(adgi, w)
    ov = oracle_volume(O, w)
    for f in range(w.frames):
        gv.update(f, w.seed, w.lights_at(f), w.sky)
        ov.update(f, w.seed, w.lights_at(f), w.sky)
        _compare_update(gv, ov, f, what="room")
    rng = np.random.default_rng(3)
    pos = rng.uniform(0.5, 7.5, (4000, 3)).astype(np.float32)
    nrm = rng.normal(size=(4000, 3)).astype(np.float32)
    rel_check(gv.query(pos, nrm), ov.query(pos, nrm), IRR_RTOL, "room query")
    gv.close()


@pytest.mark.parametrize("kind,dims,avg", [("back", (4, 4, 4), 64), ("far", (4, 4, 4), 64), ("some", (3, 2, 5), 13)])
def test_update_few_front_hits(adgi, kind, dims, avg):
    # the finish step takes the front hits alone: none, hardly any, some; the
    # other rays' records come from the step before
    r = S.box_room(1)
    verts, idx = r.verts, r.idx
    if kind == "back":
        idx = np.ascontiguousarray(idx[:, ::-1])
    elif kind == "far":
        verts = verts + np.float32(40.0)
    else:
        idx = np.where((np.arange(len(idx)) % 3 == 0)[:, None], idx[:, ::-1], idx)
    w = S.Workload(r.name, r.seed, verts, np.ascontiguousarray(idx), r.albedo, dict(r.volume, dims=dims, rays_avg=avg),
                   r.frames, (0.2, 0.3, 0.4), r.lights_at)
    gv = gpu_volume(adgi, w)
    ov = oracle_volume(O, w)
    for f in range(2):
        gv.update(f, w.seed, w.lights_at(f), w.sky)
        ov.update(f, w.seed, w.lights_at(f), w.sky)
        _compare_update(gv, ov, f, what=kind)
    gv.close()


@pytest.mark.parametrize("n_lights", [0, 1, 4, 5, 64])
def test_update_light_counts(adgi, n_lights):
    # the shadow jobs are listed by light and warp within a block: no light, one
    # scan of 32 counts (4 lights of 8 warps), more than one, the most lights
    w = S.box_room(1)
    rng = np.random.default_rng(n_lights)
    lights = [(0, tuple(rng.uniform(1.0, 7.0, 3)), (9.0, 8.0, 7.0)) for _ in range(n_lights)]
    if n_lights > 1:
        lights[1] = (1, (-0.3, -1.0, -0.2), (0.4, 0.4, 0.3))
    gv = gpu_volume(adgi, w)
    ov = oracle_volume(O, w)
    for f in range(2):
        gv.update(f, w.seed, lights, w.sky)
        ov.update(f, w.seed, lights, w.sky)
        _compare_update(gv, ov, f, what="%d lights" % n_lights)
    gv.close()


@pytest.mark.parametrize("fp16", [0, 1, 3])
def test_query_few_and_many_points_agree(adgi, fp16):
    # eight lanes a point up to 16,384 points, one thread a point beyond: the
    # same bits for the same points, whatever the count
    w = S.small_city(4, n_boxes=500, dims=(6, 5, 7), rays_avg=40)
    gv = gpu_volume(adgi, w, atlas_fp16=fp16)
    for f in range(2):
        gv.update(f, w.seed, w.lights_at(f), w.sky)
    rng = np.random.default_rng(9)
    pos = rng.uniform(-45, 45, (16400, 3)).astype(np.float32)
    org, sp = np.array(w.volume["origin"]), np.array(w.volume["spacing"])
    pos[:2000] = org + sp * rng.integers(0, 5, (2000, 3))  # at probes and on probe planes
    pos[1000:2000, 0] += 0.25
    nrm = rng.normal(size=pos.shape).astype(np.float32)
    nrm[::97] = 0.0
    many = gv.query(pos, nrm)
    for n in (1, 3, 16, 17, 1000, 16383, 16384, 16385):
        np.testing.assert_array_equal(gv.query(pos[:n], nrm[:n]), many[:n], err_msg="%d points" % n)
    gv.close()


def test_update_small_city_ragged(adgi):
    # 9 x 5 x 7 probes (ragged against every block size), moving occluders
    w = S.small_city(4, n_boxes=800, dims=(9, 5, 7), rays_avg=40)
    gv = gpu_volume(adgi, w)
    ov = oracle_volume(O, w)
    for f in range(4):
        dv = w.dyn_at(f)
        gv.move_vertices(w.dyn_first, dv)
        ov.move_vertices(w.dyn_first, dv)
        gv.update(f, w.seed, w.lights_at(f), w.sky)
        ov.update(f, w.seed, w.lights_at(f), w.sky)
        _compare_update(gv, ov, f, what="small city")
    rng = np.random.default_rng(5)
    pos = rng.uniform(-40, 40, (4000, 3)).astype(np.float32)
    pos[:, 1] = rng.uniform(0, 40, 4000)
    nrm = rng.normal(size=(4000, 3)).astype(np.float32)
    rel_check(gv.query(pos, nrm), ov.query(pos, nrm), IRR_RTOL, "city query")
    gv.close()


@pytest.mark.parametrize("case", ["pilots_only", "uniform_forced", "empty_scene", "theta1_camera", "minimal_grid",
                                  "tiles_8_16", "tiles_5_9", "tiles_1_1"])
def test_update_edge_cases(adgi, case):
    w = S.box_room(2)
    over = {}
    cam = None
    if case == "pilots_only":
        over = dict(rays_avg=8, rays_min=8, rays_max=8)
    elif case == "uniform_forced":
        over = dict(rays_avg=32, rays_min=32, rays_max=32)
    elif case == "empty_scene":
        w = S.Workload("empty", 1, np.zeros((3, 3), np.float32), np.zeros((0, 3), np.int32),
                       np.zeros((0, 3), np.float32), w.volume, 3, (0.3, 0.5, 0.9), lambda f: [])
    elif case == "theta1_camera":
        over = dict(tr_theta=1)
        cam = ((2.0, 3.0, 2.5), 1.5)
    elif case == "minimal_grid":
        over = dict(dims=(2, 2, 2), spacing=(4.0, 4.0, 4.0), rays_avg=100, rays_max=300)
    elif case == "tiles_8_16":  # the 8 x 8 / 16 x 16 interiors of the DDGI paper
        over = dict(irr_interior=8, depth_interior=16)
    elif case == "tiles_5_9":  # odd tiles, and texel runs split across 32-sample passes
        over = dict(irr_interior=5, depth_interior=9, rays_avg=120, rays_max=300)
    elif case == "tiles_1_1":  # one texel per tile: every sample in one run, counts above 255
        over = dict(irr_interior=1, depth_interior=1, rays_avg=290, rays_min=290, rays_max=300)
    gv = gpu_volume(adgi, w, **over)
    ov = oracle_volume(O, w, **over)
    for f in range(4):
        gv.update(f, w.seed, w.lights_at(f), w.sky, camera=cam)
        ov.update(f, w.seed, w.lights_at(f), w.sky, camera=cam)
        _compare_update(gv, ov, f, what=case)
    gv.close()


def test_update_rejects_bad_calls(adgi):
    w = S.box_room(1)
    v = adgi.Volume(**w.volume)
    with pytest.raises(adgi.AdgiError) as e:
        v.update(0, 1, [])
    assert e.value.code == -4  # no scene
    v.set_scene(w.verts, w.idx, w.albedo)
    with pytest.raises(adgi.AdgiError):
        v.move_vertices(len(w.verts) - 1, np.zeros((2, 3), np.float32))
    bad = w.idx.copy()
    bad[0, 0] = len(w.verts)
    with pytest.raises(adgi.AdgiError):
        v.set_scene(w.verts, bad, w.albedo)
    v.close()


# ------------------------------------------------------------------ full size
def test_tunnel_city_full_size_two_frames(adgi):
    """The bench workload (16384 probes, 4.19M rays/update, ~200k triangles,
    moving occluders) on both sides for two frames: allocation, heuristics and
    every hit bit-exact; atlases within tolerance."""
    w = S.tunnel_city(1)
    gv = gpu_volume(adgi, w)
    ov = oracle_volume(O, w)
    for f in range(2):
        dv = w.dyn_at(f)
        gv.move_vertices(w.dyn_first, dv)
        ov.move_vertices(w.dyn_first, dv)
        gv.update(f, w.seed, w.lights_at(f), w.sky)
        ov.update(f, w.seed, w.lights_at(f), w.sky)
        _compare_update(gv, ov, f, what="tunnel")
    gv.close()


# ------------------------------------------------------------------ stand-alone BVH build
@pytest.mark.parametrize("scene", ["room", "city", "one", "two"])
def test_build_bvh_matches_volume_bvh(adgi, scene):
    if scene == "room":
        w = S.box_room(1)
    elif scene == "city":
        w = S.small_city(6, n_boxes=1500)
    else:
        nt = 1 if scene == "one" else 2
        v = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], np.float32)
        w = S.Workload(scene, 0, v, np.array([[0, 1, 2], [1, 2, 3]], np.int32)[:nt], np.ones((nt, 3), np.float32),
                       S.box_room(1).volume, 1, (0, 0, 0), lambda f: [])
    gv = gpu_volume(adgi, w)
    # moving every vertex (to where it is) makes every triangle part of the
    # moving set, whose BVH is the linear one adgi_build_bvh builds
    gv.move_vertices(0, w.verts)
    dev = torch.device("cuda")
    nt = w.n_tris
    V = torch.from_numpy(w.verts).to(dev)
    I = torch.from_numpy(w.idx).to(dev)
    nodes = torch.zeros(max(nt - 1, 1) * 16, dtype=torch.int32, device=dev)
    tris = torch.zeros(nt * 12, dtype=torch.float32, device=dev)
    adgi.adgi_build_bvh(V, I, adgi.scene_eps(w.verts), nodes, tris, torch.cuda.current_stream().cuda_stream)
    ref_nodes = gv.state("MOVING_BVH_NODES", np.int32)
    ref_tris = gv.state("MOVING_BVH_TRIS", np.int32)
    if nt > 1:
        np.testing.assert_array_equal(nodes.cpu().numpy(), ref_nodes)
    np.testing.assert_array_equal(tris.cpu().numpy().view(np.int32), ref_tris)
    # triangles in BVH order are a permutation of the input, tagged with their index
    t = tris.cpu().numpy().reshape(nt, 3, 4)
    orig = t[:, 0, 3].view(np.int32)
    assert sorted(orig.tolist()) == list(range(nt))
    np.testing.assert_array_equal(t[:, :, :3], w.verts[w.idx[orig]])
    gv.close()


def test_moving_bvh_after_static_part(adgi):
    """With static and moving triangles, the moving part is built after the
    static part's nodes and triangles and its references relocated; the
    state reader gives it back in the layout of a stand-alone build of the
    moving triangles (those touching a moved vertex, in index order)."""
    w = S.small_city(3, n_boxes=400, dims=(6, 4, 5), rays_avg=24)
    gv = gpu_volume(adgi, w)
    dv = w.dyn_at(1)
    gv.move_vertices(w.dyn_first, dv)
    gv.update(0, w.seed, w.lights_at(0), w.sky)
    verts = w.verts.copy()
    verts[w.dyn_first:w.dyn_first + len(dv)] = dv
    moved = np.zeros(len(verts), bool)
    moved[w.dyn_first:w.dyn_first + len(dv)] = True
    mov = np.flatnonzero(moved[w.idx].any(axis=1))
    assert 1 < len(mov) < w.n_tris  # both parts hold triangles
    dev = torch.device("cuda")
    nt = len(mov)
    nodes = torch.zeros((nt - 1) * 16, dtype=torch.int32, device=dev)
    tris = torch.zeros(nt * 12, dtype=torch.float32, device=dev)
    adgi.adgi_build_bvh(torch.from_numpy(verts).to(dev), torch.from_numpy(np.ascontiguousarray(w.idx[mov])).to(dev),
                        adgi.scene_eps(w.verts), nodes, tris, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(gv.state("MOVING_BVH_NODES", np.int32), nodes.cpu().numpy())
    got = gv.state("MOVING_BVH_TRIS", np.float32).reshape(nt, 3, 4)
    ref = tris.cpu().numpy().reshape(nt, 3, 4)
    np.testing.assert_array_equal(got[:, :, :3], ref[:, :, :3])
    # the volume tags each triangle with its scene index, the stand-alone build with its list position
    np.testing.assert_array_equal(got[:, 0, 3].view(np.int32), mov[ref[:, 0, 3].view(np.int32)])
    gv.close()


def _morton_keys(tv):
    """63-bit Morton codes of triangles (vertices tv[n, 3, 3]) in their
    centroid bounds, with the builder's FP32 steps"""
    f = np.float32
    c = ((tv[:, 0] + tv[:, 1]) + tv[:, 2]) * f(1.0 / 3.0)
    lo, hi = c.min(0), c.max(0)
    ext = np.maximum(hi - lo, f(1e-30))
    q = np.clip((c - lo) / ext * f(2097152.0), f(0), f(2097151.0)).astype(np.uint64)
    key = np.zeros(len(tv), np.uint64)
    for b in range(21):
        for k in range(3):
            key |= ((q[:, k] >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + 2 - k)
    return key


@pytest.mark.parametrize("nt", [5, 1500, 2048, 2049, 30000])
def test_build_order_is_stable_morton_order(adgi, nt):
    # below 2,049 triangles one block sorts (bitonic, by key then index),
    # above it the radix passes do: both must give the stable key order
    rng = np.random.default_rng(nt)
    verts = rng.uniform(-50, 50, (3 * nt, 3)).astype(np.float32)
    verts[: 3 * nt // 2] = np.round(verts[: 3 * nt // 2] / 8.0) * 8.0  # repeated centroids: equal keys
    idx = np.arange(3 * nt, dtype=np.int32).reshape(nt, 3)
    dev = torch.device("cuda")
    nodes = torch.zeros(max(nt - 1, 1) * 16, dtype=torch.int32, device=dev)
    tris = torch.zeros(nt * 12, dtype=torch.float32, device=dev)
    adgi.adgi_build_bvh(torch.from_numpy(verts).to(dev), torch.from_numpy(idx).to(dev), adgi.scene_eps(verts), nodes,
                        tris, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    t = tris.cpu().numpy().reshape(nt, 3, 4)
    orig = t[:, 0, 3].view(np.int32)
    assert sorted(orig.tolist()) == list(range(nt))
    key = _morton_keys(verts.reshape(nt, 3, 3))[orig]
    k0, k1 = key[:-1], key[1:]
    assert np.all((k0 < k1) | ((k0 == k1) & (orig[:-1] < orig[1:]))), "not the stable Morton order"
    assert (k0 == k1).any() or nt < 100  # the ties were exercised


def _morton_order(verts, idx):
    """stable order of the triangles by the 63-bit Morton code of their
    centroids, FP32 as the build takes it (sum / 3 - lo is one FMA there)"""
    f = np.float32
    t = verts[idx]
    total = (t[:, 0] + t[:, 1]) + t[:, 2]
    c = total * f(1.0 / 3.0)
    lo = c.min(0)
    ext = np.maximum(c.max(0) - lo, f(1e-30))
    off = (total.astype(np.float64) * np.float64(f(1.0 / 3.0)) - lo.astype(np.float64)).astype(f)
    q = np.clip(off / ext * f(2097152.0), f(0), f(2097151.0)).astype(np.uint64)
    key = np.zeros(len(idx), np.uint64)
    for b in range(21):
        for k in range(3):
            key |= ((q[:, k] >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + 2 - k)
    return np.argsort(key, kind="stable")


# the edges of the one-block build (2,048 triangles), of the sort's tiles (1,024
# keys, 2,048 beyond 524,288) and of its warps, with equal keys among them
@pytest.mark.parametrize("nt", [2, 3, 32, 33, 2047, 2048, 2049, 3072, 3073, 524288, 524289])
def test_build_bvh_sizes(adgi, nt):
    rng = np.random.default_rng(nt)
    verts = (rng.uniform(-5, 5, (nt, 1, 3)) + rng.normal(scale=0.3, size=(nt, 3, 3))).astype(np.float32)
    verts[nt // 3:nt // 3 + nt // 10] = verts[0]
    verts = verts.reshape(-1, 3)
    idx = np.arange(3 * nt, dtype=np.int32).reshape(-1, 3)
    dev = torch.device("cuda")
    nodes = torch.full((nt - 1, 16), -7, dtype=torch.int32, device=dev)
    tris = torch.full((nt, 12), -7.0, device=dev)
    eps = adgi.scene_eps(verts)
    adgi.adgi_build_bvh(torch.from_numpy(verts).to(dev), torch.from_numpy(idx).to(dev), eps, nodes, tris,
                        torch.cuda.current_stream().cuda_stream)
    order = tris[:, 3].cpu().numpy().view(np.int32)
    np.testing.assert_array_equal(order, _morton_order(verts, idx))
    n = nodes.cpu().numpy()
    ch, box = n[:, 12:14], n[:, :12].view(np.float32)
    leaves, inner = ~ch[ch < 0], ch[ch >= 0]
    np.testing.assert_array_equal(np.sort(leaves), np.arange(nt))
    np.testing.assert_array_equal(np.sort(inner), np.arange(1, nt - 1))
    # a child's box: the triangle's enlarged by eps, or the union of the node's two
    t = verts[idx[order]]
    for side in range(2):
        lo, hi, c = box[:, 6 * side:6 * side + 3], box[:, 6 * side + 3:6 * side + 6], ch[:, side]
        lf = c < 0
        e = np.maximum(np.float32(eps), np.float32(1e-5) * np.abs(t[~c[lf]]).max((1, 2)))[:, None]
        np.testing.assert_array_equal(lo[lf], t[~c[lf]].min(1) - e)
        np.testing.assert_array_equal(hi[lf], t[~c[lf]].max(1) + e)
        kid = box[c[~lf]]
        np.testing.assert_array_equal(lo[~lf], np.minimum(kid[:, 0:3], kid[:, 6:9]))
        np.testing.assert_array_equal(hi[~lf], np.maximum(kid[:, 3:6], kid[:, 9:12]))


def test_build_bvh_rejects_bad_index(adgi):
    dev = torch.device("cuda")
    w = S.box_room(1)
    idx = w.idx.copy()
    idx[5, 1] = len(w.verts) + 3
    nodes = torch.zeros((w.n_tris - 1) * 16, dtype=torch.int32, device=dev)
    tris = torch.zeros(w.n_tris * 12, dtype=torch.float32, device=dev)
    with pytest.raises(adgi.AdgiError) as e:
        adgi.adgi_build_bvh(torch.from_numpy(w.verts).to(dev), torch.from_numpy(idx).to(dev), 1e-4, nodes, tris)
    assert e.value.code == -1 and "index" in str(e.value)
