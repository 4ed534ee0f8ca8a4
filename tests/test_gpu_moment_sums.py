"""The sums of phi and q that a step reports, on node counts that are no multiple of 4: FP32 over 32
consecutive nodes (a fixed tree) and FP64 beyond.  The same is formed here from the fields before
the step, which the library reads with the moments pass's own arithmetic, so the two differ
only in the order of FP64 additions: at most N 2^-53 of the sum of the magnitudes."""
import numpy as np
import pytest

from paper_2407_01654_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_01654_gb300 import build
    build.build()
    from paper_2407_01654_gb300 import ehd
    return ehd


def by_warps(v):
    v = v.astype(np.float32).ravel()
    v = np.concatenate([v, np.zeros(-v.size % 32, np.float32)]).reshape(-1, 32)
    lane = np.arange(32)
    for o in (16, 8, 4, 2, 1):
        v = v + v[:, lane ^ o]
    return v[:, 0].astype(np.float64).sum()


@pytest.mark.parametrize("nx,ny", [(5, 3), (33, 31), (93, 11), (201, 101), (977, 811)])
def test_sums_are_formed_in_fp64_beyond_a_warp(gpu, nx, ny):
    p = wl.make_params(nx=nx, ny=ny, walls_y=1, eps_l=4.0, sigma_l=0.05, sigma_v=0.01,
                       varphi_top=0.3, poisson_fixed_iter=2)
    rng = np.random.default_rng(nx + ny)
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    phi = wl.tanh_profile(0.3 * min(nx, ny) - np.hypot(x - nx / 2.1, y - ny / 2.3), 4.0)
    s = gpu.Sim(p)
    s.set_fields(phi, *(a * rng.standard_normal((ny, nx)) for a in (1e-3, 1e-4, 1e-4)))
    s.step(2)
    before = s.read_fields(("phi", "q"))
    st = s.step(1)
    s.close()
    for name in ("phi", "q"):
        err = abs(st["sum_" + name] - by_warps(before[name]))
        assert err <= nx * ny * 2.0 ** -53 * np.abs(before[name]).sum(), name
