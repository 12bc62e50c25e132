"""One volume that takes several scenes: its arrays and build scratch are kept
at the largest size seen, and each scene has to come out as in a volume of its
own."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2301_05125_gb300 import scenegen as S

from _helpers import gpu_volume

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


def _soup(nt, seed):
    rng = np.random.default_rng(seed)
    size = 12.0 / nt ** (1 / 3)
    verts = rng.uniform(-6, 6, (nt, 1, 3)) + rng.normal(scale=size, size=(nt, 3, 3))
    return S.Workload("soup", 0, verts.reshape(-1, 3).astype(np.float32), np.arange(3 * nt, dtype=np.int32).reshape(-1, 3),
                      np.ones((nt, 3), np.float32), S.box_room(1).volume, 1, (0, 0, 0), lambda f: [])


def _trace(adgi, v, o, d):
    t, tri = torch.empty(len(o), device="cuda"), torch.empty(len(o), dtype=torch.int32, device="cuda")
    adgi.adgi_trace_closest(v.h, torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), 1e-4, float("inf"), t, tri)
    torch.cuda.synchronize()
    v.stats()  # raises on a device anomaly flag
    return t.cpu().numpy(), np.stack([tri.cpu().numpy(), t.cpu().numpy().view(np.int32)], 1)


def test_fewer_triangles_in_kept_scratch(adgi):
    # scratch for 600,000 triangles, then builds of fewer in it: the static part
    # (500,000 and 520,000 triangles left after a move, a smaller scene) and the
    # moving part (530,000, then 520,000)
    n = 4000
    rng = np.random.default_rng(3)
    o = rng.uniform(-7, 7, (n, 3)).astype(np.float32)
    d = rng.normal(size=(n, 3)).astype(np.float32)
    v = None
    for nt, moving in [(600_000, 100_000), (530_000, 10_000), (500_000, 0), (560_000, 530_000), (560_000, 520_000)]:
        w = _soup(nt, nt + moving)
        if v is None:
            v = gpu_volume(adgi, w)
        else:
            v.set_scene(w.verts, w.idx, w.albedo)
        now = w.verts.copy()
        if moving:
            now[: 3 * moving] += np.float32(0.125)
            v.move_vertices(0, now[: 3 * moving])
        t, h = _trace(adgi, v, o, d)
        t_ref, tri_ref, _ = O.trace_closest(now, w.idx, o, d, 1e-4, np.inf)
        np.testing.assert_array_equal(adgi.hit_tri(h), tri_ref, err_msg="%d, %d moving" % (nt, moving))
        np.testing.assert_array_equal(t, t_ref)
        assert (tri_ref >= 0).mean() > 0.5
    v.close()


@pytest.mark.parametrize("n", list(range(1, 12)))
def test_failed_scene_leaves_none(adgi, n):
    # a new scene that runs out of memory, at any of its allocations (seven
    # arrays, four of the static tree): the volume has no scene afterwards --
    # not the old one's captured graph or 4-wide tree over freed arrays -- and
    # takes the next one as if nothing had been
    small = S.small_city(4, n_boxes=100, dims=(5, 4, 5), rays_avg=24)
    big = _soup(9000, 2)
    stream = torch.cuda.Stream()  # (the default stream cannot be captured)
    v = gpu_volume(adgi, small, stream=stream.cuda_stream)
    B = adgi.Batch([v], stream.cuda_stream)
    fr = [adgi.make_frame(f, 3, small.lights_at(f), small.sky) for f in range(3)]
    adgi.adgi_update_graph(v.h, fr[0])
    B.update([fr[1]])
    rng = np.random.default_rng(n)
    o, d = (rng.normal(size=(2000, 3)).astype(np.float32) for _ in range(2))
    adgi.adgi_inject_alloc_failure(n)
    try:
        with pytest.raises(adgi.AdgiError) as e:
            v.set_scene(big.verts, big.idx, big.albedo)
        assert e.value.code == -2
    finally:
        adgi.adgi_inject_alloc_failure(0)
    for call in (lambda: adgi.adgi_update_graph(v.h, fr[2]), lambda: B.update([fr[2]]), lambda: adgi.adgi_update(v.h, fr[2]),
                 lambda: _trace(adgi, v, o, d), lambda: v.move_vertices(0, small.verts[:3]),
                 lambda: adgi.adgi_count_traversal(v.h, fr[2])):
        with pytest.raises(adgi.AdgiError) as e:
            call()
        assert e.value.code == -4  # no scene
    st = v.stats()
    assert st.n_tris == 0 and st.bvh_nodes == 0 and not v.state("BVH_NODES", np.uint8).any()
    for w in (small, big):
        v.set_scene(w.verts, w.idx, w.albedo)
        t, h = _trace(adgi, v, o, d)
        t_ref, tri_ref, _ = O.trace_closest(w.verts, w.idx, o, d, 1e-4, np.inf)
        np.testing.assert_array_equal(adgi.hit_tri(h), tri_ref)
        np.testing.assert_array_equal(t, t_ref)
        adgi.adgi_update_graph(v.h, fr[2])
    torch.cuda.synchronize()
    v.stats()
    B.close()
    v.close()


@pytest.mark.parametrize("n", [12, 13])
def test_scene_without_room_for_the_wide_tree(adgi, n):
    # the 4-wide tree (nodes, then leaf records) is an aid: a scene that fits
    # without it is taken, on the binary tree, and gets one at its next build
    small, w = S.small_city(4, n_boxes=100, dims=(5, 4, 5), rays_avg=24), _soup(9000, 2)
    v = gpu_volume(adgi, small)
    rng = np.random.default_rng(n)
    o, d = (rng.normal(size=(2000, 3)).astype(np.float32) for _ in range(2))
    whole = gpu_volume(adgi, small)
    whole.set_scene(w.verts, w.idx, w.albedo)
    adgi.adgi_inject_alloc_failure(n)
    try:
        v.set_scene(w.verts, w.idx, w.albedo)
    finally:
        adgi.adgi_inject_alloc_failure(0)
    assert v.stats().device_bytes < whole.stats().device_bytes  # the tree is missing
    whole.close()
    now = w.verts.copy()
    for moved in (0, 30):
        if moved:
            now[:moved] += np.float32(0.5)
            v.move_vertices(0, now[:moved])
        t, h = _trace(adgi, v, o, d)
        t_ref, tri_ref, _ = O.trace_closest(now, w.idx, o, d, 1e-4, np.inf)
        np.testing.assert_array_equal(adgi.hit_tri(h), tri_ref)
        np.testing.assert_array_equal(t, t_ref)
    v.close()


def test_wide_tree_pays_without_pairs(adgi):
    # triangles that share no edge have a leaf record each, half of it unused:
    # the 4-wide tree still is the faster one (the binary tree of the same
    # scene is what a volume without room for the 4-wide tree walks)
    small, w = S.small_city(4, n_boxes=100, dims=(5, 4, 5), rays_avg=24), _soup(50_000, 2)
    n = 1 << 20
    g = torch.Generator(device="cuda").manual_seed(1)
    o, d = torch.rand((n, 3), generator=g, device="cuda") * 12 - 6, torch.randn((n, 3), generator=g, device="cuda")
    t, tri = torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")
    ms, out = [], []
    for n_fail in (0, 12):
        v = gpu_volume(adgi, small)
        adgi.adgi_inject_alloc_failure(n_fail)
        try:
            v.set_scene(w.verts, w.idx, w.albedo)
        finally:
            adgi.adgi_inject_alloc_failure(0)
        runs = []
        for _ in range(13):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            adgi.adgi_trace_closest(v.h, o, d, 1e-4, float("inf"), t, tri)
            b.record()
            b.synchronize()
            runs.append(a.elapsed_time(b))
        ms.append(float(np.median(runs[3:])))
        out.append((t.clone(), tri.clone()))
        v.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert ms[0] < ms[1], ms


def test_equal_sort_keys_are_no_slower(adgi):
    # triangles around one point have one Morton code: the sort's counts of all
    # of them go to one digit, which must not queue them one by one
    nt = 200_000
    rng = np.random.default_rng(0)
    idx = torch.arange(3 * nt, dtype=torch.int32, device="cuda").reshape(-1, 3)
    nodes, tris = torch.empty((nt, 16), dtype=torch.int32, device="cuda"), torch.empty((nt, 12), device="cuda")
    ms = []
    for same in (0, 1):
        verts = rng.normal(size=(1 if same else nt, 3, 3)).astype(np.float32)
        verts = torch.from_numpy(np.broadcast_to(verts, (nt, 3, 3)).reshape(-1, 3).copy()).cuda()
        runs = []
        for _ in range(13):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            adgi.adgi_build_bvh(verts, idx, 1e-5, nodes, tris, torch.cuda.current_stream().cuda_stream)
            b.record()
            b.synchronize()
            runs.append(a.elapsed_time(b))
        ms.append(float(np.median(runs[3:])))
    np.testing.assert_array_equal(tris[:, 3].cpu().numpy().view(np.int32), np.arange(nt))  # stable
    assert ms[1] < 2.0 * ms[0], ms
