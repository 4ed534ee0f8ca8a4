"""Every potential loop, named by its tiles, cluster or launches, in the index-checking build and on
non-finite input, under the stopping rule and at a fixed count, over more than eight steps (so
that the eight-step graphs run too).  Checked build: no index out of range, fields bit for bit
those of the normal build (no tolerance).  Non-finite input: reported, one sub-iteration a
step, and a fresh simulation afterwards computes what it computed before."""
import hashlib
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2407_01654_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NONFINITE = 5

TILES, STREAM = dict(cluster_ctas=0), dict(kind=1, cluster_ctas=0)
# name: nx, ny, periodic in y, parameters, what loop_shape says
LOOPS = {
    "tiles": (70, 45, 1, dict(poisson_loop=2, tile_rows=16, precision=1), dict(TILES, kind=2, rows=16)),
    "two-step": (132, 100, 0, dict(poisson_loop=3, tile_rows=32), dict(TILES, kind=3, rows=32)),
    "three-step": (140, 106, 0, dict(poisson_loop=4, tile_rows=48), dict(TILES, kind=4, rows=48)),
    "one-cta": (21, 23, 0, dict(), dict(kind=2, cluster_ctas=1)),
    "cluster": (70, 45, 0, dict(precision=1), dict(kind=2, cluster_ctas=12, capacity=512)),
    "cluster-periodic": (128, 61, 1, dict(), dict(kind=2, cluster_ctas=16, capacity=512)),
    "cluster-addresses-formed": (160, 190, 0, dict(), dict(kind=2, capacity=1920)),
    "cluster-two-copies": (187, 194, 0, dict(), dict(kind=2, cluster_ctas=15, capacity=2432)),
    "own-two-step": (300, 300, 0, dict(), dict(TILES, kind=3, rows=40)),
    "stream": (70, 45, 0, dict(poisson_loop=1), dict(STREAM, launch_iters=1)),
    "stream-several": (641, 951, 0, dict(), dict(STREAM, launch_iters=5)),
    "stream-several-periodic": (1030, 590, 1, dict(), dict(STREAM, launch_iters=5)),
}
COUNTS = {"rule": dict(poisson_min_iter=2, poisson_max_iter=60), "fixed": dict(poisson_fixed_iter=7)}


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_01654_gb300 import build
    build.build()
    from paper_2407_01654_gb300 import ehd
    return ehd


def setup(name, count):
    nx, ny, periodic, over, _ = LOOPS[name]
    p = wl.make_params(nx=nx, ny=ny, walls_y=1 - periodic, eps_l=4.0, sigma_l=0.05, sigma_v=0.01,
                       neutralize_charge=periodic, varphi_top=0.0 if periodic else 0.3)
    p.update(over)
    p.update(COUNTS[count])
    rng = np.random.default_rng(nx + ny)
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    phi = wl.tanh_profile(0.3 * min(nx, ny) - np.hypot(x - nx / 2.1, y - ny / 2.3), 4.0)
    return p, [phi] + [a * rng.standard_normal((ny, nx)) for a in (1e-3, 1e-4, 1e-4)]


def run(ehd, name, count):
    p, f = setup(name, count)
    s = ehd.Sim(p)
    s.set_fields(*f)
    st = s.step(13)
    F = s.read_fields()
    out = dict(status=st["status"], iters=st["poisson_iters_total"], errors=s.index_errors(),
               fields={k: hashlib.sha256(np.ascontiguousarray(v)).hexdigest() for k, v in F.items()})
    s.close()
    return out


CHILD = r"""
import json, sys
sys.path.insert(0, {root!r}); sys.path.insert(0, {tests!r})
from paper_2407_01654_gb300 import build, ehd
ehd.LIB_PATH = build.build(checked=True)
import test_gpu_loop_coverage as t
print(json.dumps({{n + "/" + c: t.run(ehd, n, c) for n in t.LOOPS for c in t.COUNTS}}))
assert b"checked" in ehd.lib().ehd_version()
"""


@pytest.fixture(scope="module")
def checked():
    code = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=900,
                       cwd=ROOT)
    assert r.returncode == 0, r.stderr[-3000:]
    return json.loads(r.stdout.strip().splitlines()[-1])


@pytest.mark.parametrize("count", list(COUNTS))
@pytest.mark.parametrize("name", list(LOOPS))
def test_checked_indices(gpu, checked, name, count):
    got, want = checked[name + "/" + count], run(gpu, name, count)
    assert got["errors"] == 0 and want["errors"] == 0
    assert got == want


@pytest.mark.parametrize("count", list(COUNTS))
@pytest.mark.parametrize("name", list(LOOPS))
def test_non_finite_input(gpu, name, count):
    p, f = setup(name, count)
    before = run(gpu, name, count)
    ny, nx = f[0].shape
    bad = f[0].copy()
    bad[ny // 2, nx - 3] = np.nan
    s = gpu.Sim(p)
    got = s.loop_shape()
    shape = LOOPS[name][4]
    assert {k: got[k] for k in shape} == shape
    assert s.set_fields(bad, *f[1:]) == NONFINITE
    phi = s.read_fields(("phi",))["phi"]
    far = np.ones_like(phi, dtype=bool)
    far[ny // 2 - 2:ny // 2 + 3, np.arange(nx - 5, nx) % nx] = False
    assert np.isnan(phi[ny // 2, nx - 3]) and np.isfinite(phi[far]).all()
    st = s.step(11)
    assert st["status"] == NONFINITE and st["nonfinite"] == 1 and st["steps"] == 11
    assert st["poisson_iters_total"] == 11 and st["not_converged_steps"] == 11
    it, _, code = s.solve_potential()
    assert (it, code) == (1, NONFINITE)
    s.close()
    assert run(gpu, name, count) == before
