"""The one-cluster potential loop (the library's own choice on lattices that fit 16 SMs'
shared memory) at the edges of its shapes: one CTA and several, full and ragged last CTAs,
single rows and columns, every CTA capacity, both wall rules and both potential schemes.  At a
fixed count its state is the streaming loop's bit for bit (the arithmetic per node is the
same, so the tolerance is none); under the rule it stops where the tiled loop stops, also
where the tolerance lies between two neighbouring floats."""
import numpy as np
import pytest

from paper_2407_01654_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# nx, ny (CTAs, rows of each, capacity): one CTA, its largest and beyond; single rows and
# columns; every capacity, full and ragged; the largest that fits and one beyond
SHAPES = [(16, 32),    # 1, 32, 512
          (27, 19),    # 3, 7, 256
          (3, 7),      # 1, 7, 256
          (1, 600),    # 3, 200, 256
          (300, 9),    # 5, 2, 768
          (64, 64),    # 16, 4, 256
          (128, 128),  # 16, 8, 1024
          (200, 100),  # 15, 7, 1408
          (180, 149),  # 15, 10, 1920
          (187, 194),  # 15, 13, 2432
          (180, 256),  # 16, 16, 2880
          (181, 256)]  # beyond: the two-step tiled loop (a count of 1: the one-step loop)


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
                       width=4.0, varphi_top=0.3 if walls else 0.0, varphi_bottom=-0.1 if walls else 0.0,
                       neutralize_charge=0 if walls else 1, potential_scheme=scheme, chi=2.0)
    p.update(over)
    rng = np.random.default_rng(nx * 1009 + ny)
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    phi = wl.tanh_profile(0.3 * min(nx, ny) - np.hypot(x - nx / 2.1, y - ny / 2.3), 4.0)
    q, ux, uy = (a * rng.standard_normal((ny, nx)) for a in (1e-3, 1e-4, 1e-4))
    return p, (phi, q, ux, uy)


def own_rows(nx, ny, sms=152):
    """The height of the tiles that the library itself picks (about 2048 nodes each)."""
    ntx = -(-nx // 64)
    nty = max(1, min((nx * ny + 2047) // 2048, sms) // ntx)
    rows = -(-ny // nty)
    if rows > 64:
        rows = -(-ny // -(-ny // 64))
    return max(8, (rows + 7) // 8 * 8)


def states(gpu, p, f, steps):
    s = gpu.Sim(p)
    s.set_fields(*f)
    st = s.step(steps)
    out = s.read_fields(), st["poisson_iters_total"], s.loop_kind()
    s.close()
    return out


@pytest.mark.parametrize("nx,ny", SHAPES)
@pytest.mark.parametrize("walls,scheme", [(1, 0), (0, 0), (1, 1)])
def test_fixed_count_equals_streaming(gpu, nx, ny, walls, scheme):
    for k in (1, 2, 3, 8):  # every rotation of the copies
        p, f = setup(nx, ny, walls, scheme, poisson_fixed_iter=k)
        a, ia, kind = states(gpu, p, f, 2)
        b, ib, _ = states(gpu, dict(p, poisson_loop=1), f, 2)
        assert kind == (3 if nx == 181 and k > 1 else 2) and ia == ib == 2 * k
        for name in a:
            assert np.array_equal(a[name], b[name]), (name, k)


@pytest.mark.parametrize("nx,ny", SHAPES)
def test_rule_stops_where_the_tiled_loop_stops(gpu, nx, ny):
    p, f = setup(nx, ny, 1, 0, poisson_tol=1e-4)
    a, ia, _ = states(gpu, p, f, 3)
    b, ib, _ = states(gpu, dict(p, tile_rows=own_rows(nx, ny)), f, 3)
    assert ia == ib
    for name in a:
        assert np.array_equal(a[name], b[name]), name


@pytest.mark.parametrize("k", [40, 41])
@pytest.mark.parametrize("nx,ny,walls,scheme", [(4, 64, 1, 0), (64, 64, 0, 0), (64, 64, 1, 1),
                                                (200, 100, 1, 0), (180, 256, 1, 0),
                                                (60, 7, 1, 0), (64, 24, 1, 0), (100, 40, 0, 0),
                                                (128, 60, 1, 0)])
def test_rule_on_the_last_bit(gpu, nx, ny, walls, scheme, k):
    """The tolerance set to the tiled loop's own relative change after k sub-iterations, and to
    the next float above it: the first does not stop at k, the second does."""
    p, f = setup(nx, ny, walls, scheme, poisson_fixed_iter=k, tile_rows=own_rows(nx, ny))
    s = gpu.Sim(p)
    s.set_fields(*f)
    r = np.float32(s.step(1)["last_rel_change"])
    s.close()
    for tol, stops in ((float(r), False), (float(np.nextafter(r, np.float32(1))), True)):
        q = dict(p, poisson_fixed_iter=0, poisson_tol=tol, poisson_min_iter=k, poisson_max_iter=k + 1)
        # the same first solve (k sub-iterations), then one step under the rule
        got = []
        for rows in (p["tile_rows"], 0):
            s = gpu.Sim(dict(q, tile_rows=rows, poisson_max_iter=k))
            s.set_fields(*f)
            blob = s.save_state()
            s.close()
            s = gpu.Sim(dict(q, tile_rows=rows))
            s.load_state(blob)
            got.append(s.step(1)["poisson_iters_total"])
            s.close()
        assert got == [k if stops else k + 1] * 2, (tol, stops)
