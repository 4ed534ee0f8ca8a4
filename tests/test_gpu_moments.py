"""The moments pass of a node count that is no multiple of 4 (four nodes per thread, 1024 per CTA,
without the cross-CTA tail) against one that takes one node at a time with the tail (a batch
slot's; beyond the chip's storage one slab of the slab decomposition): at a fixed count the states
are the same bit for bit (no tolerance) for lattices below, at and beyond the edges of a CTA's
nodes, on the on-chip and on the streaming loop, in both storage precisions.  The sums it leaves
to the coupled pass are FP32 over at most 128 values and FP64 beyond: at most 128 roundings of
2^-24, 7.7e-6 of the sum of |phi|, from the FP64 sum of the field before the step."""
import numpy as np
import pytest

from paper_2407_01654_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [(nx, ny, h) for nx, ny in ((9, 7), (33, 31), (79, 13), (93, 11), (201, 101)) for h in (0, 1)]
CASES += [(977, 811, 0)]


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_01654_gb300 import build
    build.build()
    from paper_2407_01654_gb300 import ehd
    return ehd


@pytest.mark.parametrize("nx,ny,precision", CASES)
def test_odd_node_counts(gpu, nx, ny, precision):
    p = wl.make_params(nx=nx, ny=ny, walls_y=1, eps_l=4.0, sigma_l=0.05, sigma_v=0.01,
                       varphi_top=0.3, poisson_fixed_iter=3, precision=precision)
    rng = np.random.default_rng(nx + ny)
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    phi = wl.tanh_profile(0.3 * min(nx, ny) - np.hypot(x - nx / 2.1, y - ny / 2.3), 4.0)
    f = (phi,) + tuple(a * rng.standard_normal((ny, nx)) for a in (1e-3, 1e-4, 1e-4))
    s = gpu.Sim(p)
    s.set_fields(*f)
    s.step(2)
    before = s.read_fields()["phi"]
    st = s.step(1)
    fa = s.read_fields()
    s.close()
    if nx * ny > 600000:
        t = gpu.Slabs(p, 1)
        t.set_fields(*f)
        t.step(3)
        fb = t.read_fields()
    else:
        t = gpu.Batch(128 << 20, max_slots=1)
        slot = t.admit(p, dict(zip(("phi", "q", "ux", "uy"), f)), 0)
        t.run(3)
        fb = t.read_fields(slot)
    t.close()
    assert st["poisson_iters_total"] == 3
    for name in fb:
        assert np.array_equal(fa[name], fb[name]), name
    assert abs(st["sum_phi"] - before.sum()) <= 7.7e-6 * np.abs(before).sum()
