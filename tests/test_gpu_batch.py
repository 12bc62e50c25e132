"""Graph-captured, batched and autotuned updates give the results of the plain
update (same kernels; only the launch mechanism and block shapes differ).

Integer outputs (allocation, heuristics, hits, counts) must be identical;
float atlases may differ only by the order of shared-memory additions in the
blend (a few ulps), checked at 1e-5 relative.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2301_05125_gb300 import scenegen as S

from _helpers import gpu_volume, rel_check

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


def _same(a, b, tag):
    np.testing.assert_array_equal(a.W(), b.W(), err_msg=tag)
    np.testing.assert_array_equal(a.n(), b.n(), err_msg=tag)
    np.testing.assert_array_equal(a.trv(), b.trv(), err_msg=tag)
    np.testing.assert_array_equal(a.main_hit()[:, 0], b.main_hit()[:, 0], err_msg=tag)
    np.testing.assert_array_equal(a.pilot_hit(), b.pilot_hit(), err_msg=tag)
    np.testing.assert_array_equal(a.dep_n(), b.dep_n(), err_msg=tag)
    rel_check(a.irr(), b.irr(), 1e-5, tag + " irr")
    rel_check(a.dep_moments(), b.dep_moments(), 1e-5, tag + " dep")


def _step(v, w, f, mode):
    if w.dyn_at is not None and w.dyn_count:
        v.move_vertices(w.dyn_first, w.dyn_at(f))
    getattr(v, mode)(f, w.seed, w.lights_at(f), w.sky)


def test_graph_update_matches_plain(adgi):
    w = S.small_city(5, n_boxes=900, dims=(9, 5, 7), rays_avg=40)
    a, b = gpu_volume(adgi, w), gpu_volume(adgi, w)
    for f in range(6):
        _step(a, w, f, "update")
        _step(b, w, f, "update_graph")
        a.stats()
        b.stats()
        _same(a, b, "graph frame %d" % f)


def test_batch_matches_individual(adgi):
    ws = [S.box_room(1), S.small_city(5, n_boxes=900, dims=(9, 5, 7), rays_avg=40),
          S.small_city(6, n_boxes=500, dims=(6, 4, 5), rays_avg=24)]
    ref = [gpu_volume(adgi, w) for w in ws]
    bat = [gpu_volume(adgi, w, atlas_fp16=0) for w in ws]
    stream = torch.cuda.Stream()
    B = adgi.Batch(bat, stream.cuda_stream)
    for f in range(6):
        frames = []
        for v, w in zip(bat, ws):
            if w.dyn_at is not None and w.dyn_count:
                v.move_vertices(w.dyn_first, w.dyn_at(f))
            frames.append(adgi.make_frame(f, w.seed, w.lights_at(f), w.sky))
        B.update(frames)
        stream.synchronize()
        for v, w in zip(ref, ws):
            _step(v, w, f, "update")
        for i in range(len(ws)):
            bat[i].stats()
            _same(ref[i], bat[i], "batch vol %d frame %d" % (i, f))
    B.close()


def test_autotune_keeps_results(adgi):
    w = S.small_city(5, n_boxes=900, dims=(9, 5, 7), rays_avg=40)
    a, b = gpu_volume(adgi, w), gpu_volume(adgi, w)
    _step(a, w, 0, "update")
    _step(b, w, 0, "update")
    t = b.autotune(0, w.seed, w.lights_at(0), w.sky, reps=2)
    assert t.trace_block in (64, 128, 256) and t.blend_block in (32, 64, 128)
    assert t.ms_trace > 0 and t.ms_shade > 0 and t.ms_blend > 0
    _same(a, b, "after autotune")
    for f in range(1, 5):
        _step(a, w, f, "update")
        _step(b, w, f, "update")
        _same(a, b, "autotuned frame %d" % f)
    with pytest.raises(adgi.AdgiError):
        adgi.adgi_set_tuning(b.h, adgi.adgi_tuning(100, 128, 0, 128))


def test_graph_and_batch_follow_scene_changes(adgi):
    # the static / moving split and the scene's arrays change between replays
    # through other calls (a trace builds the split; a new scene of another
    # size): captured graphs must not be replayed on the old ones
    w, w2 = S.small_city(4, n_boxes=700, dims=(5, 4, 5), rays_avg=24), S.small_city(6, n_boxes=1500, dims=(5, 4, 5), rays_avg=24)
    stream = torch.cuda.Stream()
    plain, graph, bat = (gpu_volume(adgi, w, stream=stream.cuda_stream) for _ in range(3))
    B = adgi.Batch([bat], stream.cuda_stream)
    o = torch.zeros(64, 3, device="cuda") + 5.0
    d = torch.nn.functional.normalize(torch.randn(64, 3, device="cuda"), dim=1)
    t, tri = torch.empty(64, device="cuda"), torch.empty(64, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for f in range(7):
        if f == 2:  # occluders begin to move; a trace brings the split up to date first
            for v in (plain, graph, bat):
                v.move_vertices(w.dyn_first, w.dyn_at(f))
                adgi.adgi_trace_closest(v.h, o, d, 1e-4, 1e30, t, tri)
        if f == 4:  # another scene
            for v in (plain, graph, bat):
                v.set_scene(w2.verts, w2.idx, w2.albedo)
        lights = w.lights_at(f)
        plain.update(f, 3, lights, w.sky)
        graph.update_graph(f, 3, lights, w.sky)
        B.update([adgi.make_frame(f, 3, lights, w.sky)])
        torch.cuda.synchronize()
        for v in (graph, bat):
            np.testing.assert_array_equal(v.n(), plain.n(), err_msg="frame %d" % f)
            np.testing.assert_array_equal(v.pilot_hit(), plain.pilot_hit(), err_msg="frame %d" % f)
            np.testing.assert_array_equal(v.irr(), plain.irr(), err_msg="frame %d" % f)
            np.testing.assert_array_equal(v.dep(), plain.dep(), err_msg="frame %d" % f)
    B.close()
    for v in (plain, graph, bat):
        v.stats()
        v.close()


@pytest.mark.parametrize("nt", [2, 3, 31, 32, 33, 511, 513, 1025, 4100])
def test_static_build_sizes(adgi, nt):
    # the static build at the edges of its clustering (groups of 32, the
    # one-block tail, duplicates that tie everywhere) against brute force
    rng = np.random.default_rng(nt)
    n = 20000
    verts = rng.uniform(-4, 4, (nt, 1, 3)) + rng.normal(scale=0.4, size=(nt, 3, 3))
    verts[nt // 2:nt // 2 + nt // 8] = verts[0]  # duplicates
    verts = verts.reshape(-1, 3).astype(np.float32)
    idx = np.arange(3 * nt, dtype=np.int32).reshape(-1, 3)
    w = S.Workload("soup", 0, verts, idx, np.ones((nt, 3), np.float32), S.box_room(1).volume, 1, (0, 0, 0), lambda f: [])
    v = gpu_volume(adgi, w)
    o = rng.uniform(-6, 6, (n, 3)).astype(np.float32)
    d = rng.normal(size=(n, 3)).astype(np.float32)
    t, tri = torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")
    adgi.adgi_trace_closest(v.h, torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda(), 1e-4, float("inf"), t, tri)
    torch.cuda.synchronize()
    v.stats()
    t_ref, tri_ref, _ = O.trace_closest(verts, idx, o, d, 1e-4, np.inf, use_bvh=nt > 600)
    h = np.stack([tri.cpu().numpy(), t.cpu().numpy().view(np.int32)], 1)
    np.testing.assert_array_equal(adgi.hit_tri(h), tri_ref)
    np.testing.assert_array_equal(t.cpu().numpy(), t_ref)
    v.close()


@pytest.mark.parametrize("kind,nt", [("soup", 3), ("soup", 4), ("soup", 5), ("soup", 700), ("soup", 2049), ("soup", 2050),
                                     ("soup", 9001), ("same", 3000), ("line", 5000), ("quads", 10), ("quads", 6000), ("nested", 700),
                                     ("nested", 4500)])
def test_static_tree_sound(adgi, kind, nt):
    # the reinsertion rounds (one block up to 2,048 nodes besides pairs, many
    # beyond; ties, one point, one line): every triangle once, every box the
    # union of its children's, no way round in a circle, a bounded depth (a
    # nest of boxes, each around the one before, clusters into a chain)
    rng = np.random.default_rng(nt)
    if kind == "quads":
        c, a, b = (rng.normal(size=(nt // 2, 3)) for _ in range(3))
        verts = np.stack([8 * c, 8 * c + a, 8 * c + a + b, 8 * c + b], 1).reshape(-1, 3)
        q = 4 * np.arange(nt // 2)[:, None]
        idx = np.stack([q + [0, 1, 2], q + [0, 2, 3]], 1).reshape(-1, 3)
    elif kind == "nested":
        size = (1.0 + 20.0 / nt) ** np.arange(nt)
        verts = (rng.normal(size=(1, 3, 3)) * size[:, None, None]).reshape(-1, 3)
        idx = np.arange(3 * nt).reshape(-1, 3)
    else:
        c = rng.uniform(-9, 9, (nt, 1, 3)) * {"soup": 1.0, "same": 0.0, "line": np.array([1.0, 0.0, 0.0])}[kind]
        size = np.exp(rng.uniform(-4, 2, (nt, 1, 1))) if kind == "soup" else 0.3
        tri = rng.normal(size=(nt, 3, 3)) if kind != "same" else np.broadcast_to(rng.normal(size=(3, 3)), (nt, 3, 3))
        verts = (c + size * tri).reshape(-1, 3)
        idx = np.arange(3 * nt).reshape(-1, 3)
    verts, idx = verts.astype(np.float32), idx.astype(np.int32)
    w = S.Workload("soup", 0, verts, idx, np.ones((nt, 3), np.float32), S.box_room(1).volume, 1, (0, 0, 0), lambda f: [])
    v = gpu_volume(adgi, w)
    raw = v.state("BVH_NODES", np.float32).reshape(-1, 16)[:nt - 1]
    box = raw[:, :12].reshape(-1, 2, 6)
    ref = raw.view(np.int32)[:, 12:14]
    leaves = np.sort(~ref[ref < 0])
    np.testing.assert_array_equal(leaves, np.arange(nt))
    inner = np.sort(ref[ref >= 0])
    np.testing.assert_array_equal(inner, np.arange(1, nt - 1))
    level, seen, depth = np.array([0]), 0, 0
    while len(level):
        depth += 1
        seen += len(level)
        assert depth < 96
        kids = ref[level]
        m = kids >= 0
        sub = box[kids[m]]
        un = np.concatenate([sub[:, :, :3].min(1), sub[:, :, 3:].max(1)], 1)
        np.testing.assert_array_equal(box[level][m], un)
        level = kids[m]
    assert seen == nt - 1
    v.close()


@pytest.mark.parametrize("nt", [1152, 1153, 1154])
def test_static_tree_sound_at_the_one_block_edge(adgi, nt):
    # 1,152 internal nodes: the last tree that one block reinserts on its own
    test_static_tree_sound(adgi, "soup", nt)
    test_static_build_sizes(adgi, nt)
