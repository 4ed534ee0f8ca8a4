"""Streaming with several sub-iterations per launch (lattices beyond the chip's storage) against
one slab of the slab decomposition, which streams one sub-iteration per launch: at a fixed
count the states are the same bit for bit (no tolerance); under the rule both stop alike, on the
last sub-iteration of a launch and inside one.  Sizes: ragged tiles in x and y, narrow and
flat lattices, y-periodic ones, both potential schemes."""
import numpy as np
import pytest

from paper_2407_01654_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(977, 811, 1, 0), (1024, 600, 0, 0), (8, 76000, 1, 0), (90001, 7, 0, 0), (641, 950, 1, 1)]


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_01654_gb300 import build
    build.build()
    from paper_2407_01654_gb300 import ehd
    return ehd


def setup(nx, ny, walls, scheme, **over):
    p = wl.make_params(nx=nx, ny=ny, walls_y=walls, eps_l=4.0, sigma_l=0.05, sigma_v=0.01,
                       varphi_top=0.3 if walls else 0.0, potential_scheme=scheme, chi=2.0)
    p.update(over)
    rng = np.random.default_rng(nx + ny)
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    phi = wl.tanh_profile(0.3 * min(nx, ny) - np.hypot(x - nx / 2.1, y - ny / 2.3), 4.0)
    return p, (phi,) + tuple(a * rng.standard_normal((ny, nx)) for a in (1e-3, 1e-4, 1e-4))


def both(gpu, p, f, steps):
    s, t = gpu.Sim(p), gpu.Slabs(p, 1)
    assert s.loop_kind() == 1
    s.set_fields(*f)
    t.set_fields(*f)
    a, b = s.step(steps), t.step(steps)
    out = s.read_fields(), t.read_fields(), a, b
    s.close()
    t.close()
    return out


@pytest.mark.parametrize("nx,ny,walls,scheme", SHAPES)
def test_fixed_count(gpu, nx, ny, walls, scheme):
    for k in (1, 4, 5, 7, 48):  # one launch, a full one, two unequal ones, a loop of launches
        p, f = setup(nx, ny, walls, scheme, poisson_fixed_iter=k)
        fa, fb, a, b = both(gpu, p, f, 1)
        assert a["poisson_iters_total"] == b["poisson_iters_total"] == k
        for name in fa:
            assert np.array_equal(fa[name], fb[name]), (name, k)


@pytest.mark.parametrize("nx,ny,walls,scheme", SHAPES[:3])
def test_rule(gpu, nx, ny, walls, scheme):
    ends = set()
    for tol in (1e-2, 1e-3, 5e-4, 3e-4, 2e-4):
        p, f = setup(nx, ny, walls, scheme, poisson_tol=tol)
        fa, fb, a, b = both(gpu, p, f, 2)
        assert a["poisson_iters_total"] == b["poisson_iters_total"]
        ends.add(a["poisson_iters_total"])
        for name in fa:
            assert np.array_equal(fa[name], fb[name]), (name, tol)
    assert len(ends) > 1
