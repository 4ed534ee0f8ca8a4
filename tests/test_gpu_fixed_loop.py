"""The on-chip two-step loop's ending at a fixed count (no second sub-iteration of an odd count's
last cycle, no closing grid barrier; a single cycle writes back behind a barrier it arrived at
early): the same states as the streaming and the one-step loop bit for bit, for one cycle and
several, odd and even counts, every tile height, ragged tiles, both schemes.  The relative change
of the last sub-iteration is a quotient of FP32 sums (1e-5 of it, at most 160 roundings of 2^-24)
of a difference whose terms one loop may round once more than another (2^-24 of the potential, so
1.2e-7 for both).  The bounded wait reports an expired barrier for one cycle as for several."""
import numpy as np
import pytest

from paper_2407_01654_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(200, 100, 24, 1, 0), (133, 71, 32, 1, 1), (128, 80, 40, 0, 0), (196, 101, 48, 1, 0),
          (512, 1024, 56, 1, 0), (72, 68, 64, 0, 1)]


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
                       varphi_top=0.3 if walls else 0.0, potential_scheme=scheme, chi=2.0, **over)
    rng = np.random.default_rng(nx + ny)
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    phi = wl.tanh_profile(0.3 * min(nx, ny) - np.hypot(x - nx / 2.1, y - ny / 2.3), 4.0)
    return p, (phi,) + tuple(a * rng.standard_normal((ny, nx)) for a in (1e-3, 1e-4, 1e-4))


def run(gpu, p, f, loop, rows):
    s = gpu.Sim(dict(p, poisson_loop=loop, tile_rows=rows if loop > 1 else 0))
    assert s.loop_kind() == loop
    s.set_fields(*f)
    st = s.step(3)
    it, rel, code = s.solve_potential()
    out = s.read_fields()
    s.close()
    return out, st["poisson_iters_total"], it, rel, code


@pytest.mark.parametrize("k", (1, 2, 3, 4, 7))
@pytest.mark.parametrize("nx,ny,rows,walls,scheme", SHAPES)
def test_same_states_and_change(gpu, nx, ny, rows, walls, scheme, k):
    p, f = setup(nx, ny, walls, scheme, poisson_fixed_iter=k)
    two = run(gpu, p, f, 3, rows)
    stream, one = run(gpu, p, f, 1, 0), run(gpu, p, f, 2, rows)
    assert two[1:3] == stream[1:3] == one[1:3] == (3 * k, k) and two[4] == one[4] == 0
    assert abs(two[3] - one[3]) <= 1.2e-7 + 1e-5 * one[3]
    for name in two[0]:
        assert np.array_equal(two[0][name], stream[0][name]), name
        assert np.array_equal(two[0][name], one[0][name]), name


@pytest.mark.parametrize("k", (1, 2, 3))
def test_expired_barrier(gpu, k):
    p, f = setup(200, 100, 1, 0, poisson_fixed_iter=k, poisson_loop=3, tile_rows=24)
    s = gpu.Sim(p)
    s.set_fields(*f)
    s.diag_expire_barrier()
    with pytest.raises(gpu.EhdError) as err:
        s.step(1)
    assert err.value.code == 9  # EHD_ERR_TIMEOUT
    s.close()
