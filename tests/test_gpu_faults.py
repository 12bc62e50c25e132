"""Failure paths, with the failures made on the host.

A device allocation is made to fail the way cudaMalloc fails on a full
device (adgi_inject_alloc_failure: the call reports the error without
allocating), at the first, a middle and a late allocation of a volume.  The
call must return OOM, release everything it had allocated, and leave the
library able to build and update the next volume.  Nothing here faults,
traps or stalls a GPU.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

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


def test_allocation_failure_returns_oom_and_releases_memory(adgi):
    w = S.small_city(4, n_boxes=800, dims=(9, 5, 7), rays_avg=40)
    ref = gpu_volume(adgi, w)  # the same frames on an undisturbed volume
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    try:
        for n in (1, 9, 20):
            adgi.adgi_inject_alloc_failure(n)
            with pytest.raises(adgi.AdgiError) as e:
                adgi.Volume(**w.volume)
            assert e.value.code == -2, "allocation %d" % n
    finally:
        adgi.adgi_inject_alloc_failure(0)
    torch.cuda.synchronize()
    free1 = torch.cuda.mem_get_info()[0]
    assert free0 - free1 < (16 << 20), "device memory not released: %d bytes" % (free0 - free1)
    v = gpu_volume(adgi, w)
    for f in range(2):
        for x in (ref, v):
            if w.dyn_at is not None and w.dyn_count:
                x.move_vertices(w.dyn_first, w.dyn_at(f))
            x.update(f, w.seed, w.lights_at(f), w.sky)
    np.testing.assert_array_equal(v.n(), ref.n())
    np.testing.assert_array_equal(v.main_hit(), ref.main_hit())
    np.testing.assert_array_equal(v.irr(), ref.irr())
    v.close()
    ref.close()


def test_injection_rejects_negative_counts(adgi):
    with pytest.raises(adgi.AdgiError):
        adgi.adgi_inject_alloc_failure(-1)


_REFUSED = """
import sys
import numpy as np
import torch
from paper_2301_05125_gb300 import adgi

adgi.load()
rng = np.random.default_rng(1)
verts = torch.from_numpy(rng.normal(size=(300, 3)).astype(np.float32)).cuda()
idx = torch.arange(300, dtype=torch.int32, device="cuda").reshape(-1, 3)
nodes, tris = torch.zeros((99, 16), dtype=torch.int32, device="cuda"), torch.zeros((100, 12), device="cuda")
x, other = torch.zeros(10, device="cuda"), torch.cuda.Stream()
torch.cuda.synchronize()
code = 0
try:
    with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=torch.cuda.Stream()):
        x.add_(1)
        try:
            adgi.adgi_build_bvh(verts, idx, 1e-5, nodes, tris, other.cuda_stream)
        except adgi.AdgiError as e:
            code = e.code
        x.add_(1)
except RuntimeError:
    pass  # the refused call ended the capture
adgi.adgi_build_bvh(verts, idx, 1e-5, nodes, tris, other.cuda_stream)
torch.cuda.synchronize()
order = np.sort(tris[:, 3].cpu().numpy().view(np.int32))
print("code", code, "built", bool((order == np.arange(100)).all()))
"""


def test_build_refused_by_the_runtime_is_no_memory_shortage(adgi):
    # the stand-alone build asks for scratch while a stream is captured, which
    # CUDA refuses: a CUDA error, not OOM, and the next build works (in a
    # process of its own: a capture that fails leaves torch on its stream)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _REFUSED], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.stdout.split() == ["code", "-5", "built", "True"], r.stdout + r.stderr
