"""GPU parity of the DDGI cosine-gather blend (blend_mode = 1) against the
oracle: allocation, hits and the per-texel ray counts (the rays with
n . w > 0, an exact FP32 test on both sides) bit-exact; irradiance within
1e-3 and depth moments within 1e-4 relative.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2301_05125_gb300 import scenegen as S

from _helpers import gpu_volume, oracle_volume, rel_check
from test_gpu_parity import _compare_update

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


@pytest.mark.parametrize("scene", ["room", "city"])
def test_cosine_gather_matches_oracle(adgi, scene):
    if scene == "room":
        w = S.box_room(1)
    else:
        w = S.small_city(4, n_boxes=800, dims=(9, 5, 7), rays_avg=40)
    gv, ov = gpu_volume(adgi, w, blend_mode=1), oracle_volume(O, w, blend_mode=1)
    for f in range(4):
        if w.dyn_at is not None and w.dyn_count:
            dv = w.dyn_at(f)
            gv.move_vertices(w.dyn_first, dv)
            ov.move_vertices(w.dyn_first, dv)
        gv.update(f, w.seed, w.lights_at(f), w.sky)
        ov.update(f, w.seed, w.lights_at(f), w.sky)
        _compare_update(gv, ov, f, what="cosine gather " + scene)
    gv.close()


# texel places at the edges of the gather's split (256 places a round, a
# warp's 64 all depth, all irradiance or both) and probes of few rays, whose
# far texels' weights come near FP32's range
@pytest.mark.parametrize("ni,nd,avg,lo,hi", [(6, 14, 9, 8, 10), (4, 6, 20, 8, 64), (8, 16, 70, 8, 400), (6, 8, 200, 8, 500)])
def test_cosine_gather_tiles_and_ray_counts(adgi, ni, nd, avg, lo, hi):
    w = S.small_city(4, n_boxes=500, dims=(5, 4, 6), rays_avg=avg)
    over = dict(blend_mode=1, irr_interior=ni, depth_interior=nd, rays_min=lo, rays_max=hi)
    gv, ov = gpu_volume(adgi, w, **over), oracle_volume(O, w, **over)
    for f in range(3):
        gv.update(f, w.seed, w.lights_at(f), w.sky)
        ov.update(f, w.seed, w.lights_at(f), w.sky)
        _compare_update(gv, ov, f, what="cosine gather %d %d" % (ni, nd))
    gv.close()


def test_cosine_gather_with_clip_volumes_and_fp16(adgi):
    w = S.small_city(5, n_boxes=600, dims=(6, 4, 5), rays_avg=24)
    from test_gpu_clip import view_proj

    gv = gpu_volume(adgi, w, blend_mode=1, atlas_fp16=1)
    ov = oracle_volume(O, w, blend_mode=1)
    for f in range(4):
        eye = (-30.0 + 5.0 * f, 12.0, -5.0)
        cam = (eye, 30.0, view_proj(eye, (0.0, 6.0, 0.0)))
        gv.update(f, w.seed, w.lights_at(f), w.sky, camera=cam)
        ov.update(f, w.seed, w.lights_at(f), w.sky, camera=cam)
        np.testing.assert_array_equal(gv.cls(), ov.cls())
        gi = gv.irr()
        np.testing.assert_array_equal(gi[..., 3].astype(np.int64), ov.irr_n().astype(np.int64))
        rel_check(gi[..., :3], ov.irr(), 6e-3, "fp16 cosine-gather irradiance")  # half storage (FP16 bounds)
    gv.close()


def test_cosine_gather_rejects_bad_modes(adgi):
    w = S.box_room(1)
    for over in (dict(blend_mode=2), dict(blend_mode=1, sampler=1), dict(blend_mode=1, atlas_fp16=3)):
        with pytest.raises(adgi.AdgiError):
            gpu_volume(adgi, w, **over)


@pytest.mark.parametrize("avg,hi", [(9, 10), (24, 64), (150, 400)])
@pytest.mark.parametrize("what", ["sky", "depth"])
def test_cosine_gather_infinite_values_stay_in_front(adgi, what, avg, hi):
    # rays that escape bring an infinite radiance (or an infinite depth): the
    # texels that face one are lost, the others are what they are without it
    w = S.small_city(4, n_boxes=500, dims=(5, 4, 6), rays_avg=avg)
    over = dict(blend_mode=1, rays_min=8, rays_max=hi)
    sky = w.sky
    if what == "sky":
        sky = (float("inf"), 0.25, float("inf"))
    else:
        over["depth_max"] = float("inf")
    gv, ov = gpu_volume(adgi, w, **over), oracle_volume(O, w, **over)
    gv.update(0, w.seed, w.lights_at(0), sky)
    ov.update(0, w.seed, w.lights_at(0), sky)
    gv.stats()
    np.testing.assert_array_equal(gv.n(), ov.n())
    gi, oi, gd, od = gv.irr()[..., :3], ov.irr(), gv.dep_moments(), ov.dep()
    ok = np.isfinite(oi)
    np.testing.assert_array_equal(np.isfinite(gi), ok)
    rel_check(gi[ok], oi[ok], 1e-3, "irradiance")
    ok = np.isfinite(od).all(-1)
    np.testing.assert_array_equal(np.isfinite(gd).all(-1), ok)
    rel_check(gd[ok], od[ok], 1e-4, "depth")
    lost = ~np.isfinite(oi if what == "sky" else od)
    assert lost.any() and not lost.all()
    gv.close()
