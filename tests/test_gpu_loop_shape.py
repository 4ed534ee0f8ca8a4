"""Which potential loop a lattice gets, CTA for CTA: the shapes that the tests of the one-cluster
loop are written for, the lattices just beyond it, and the streaming loops on either side of
600 000 nodes."""
import numpy as np
import pytest

import test_gpu_cluster as cl
from paper_2407_01654_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# CTAs of the cluster, rows of each, node capacity, in the order of the
# shapes there (300 x 9 is one of nine single rows)
CLUSTERS = [(1, 32, 512), (3, 7, 256), (1, 7, 256), (3, 200, 256), (9, 1, 512), (16, 4, 256),
            (16, 8, 1024), (15, 7, 1408), (15, 10, 1920), (15, 13, 2432), (16, 16, 2880), None]


@pytest.fixture(scope="module")
def gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2407_01654_gb300 import build
    build.build()
    from paper_2407_01654_gb300 import ehd
    return ehd


def shape(gpu, nx, ny, **over):
    s = gpu.Sim(wl.make_params(nx=nx, ny=ny, **over))
    try:
        return s.loop_shape()
    finally:
        s.close()


@pytest.mark.parametrize("size,cluster", list(zip(cl.SHAPES, CLUSTERS)))
@pytest.mark.parametrize("scheme", [0, 1])
def test_small_lattices_run_on_one_cluster(gpu, size, cluster, scheme):
    for count in (0, 3):
        d = shape(gpu, *size, potential_scheme=scheme, chi=2.0, poisson_fixed_iter=count)
        # (under the rule the largest capacity is left to the two-step loop)
        if cluster is None or (cluster[2] == 2880 and count == 0):
            assert d["cluster_ctas"] == 0 and d["kind"] == 3
        else:
            assert (d["cluster_ctas"], d["rows"], d["capacity"]) == cluster and d["kind"] == 2
    # tiles where they are asked for
    d = shape(gpu, *size, potential_scheme=scheme, chi=2.0, poisson_loop=2, tile_rows=32)
    assert (d["cluster_ctas"], d["rows"], d["capacity"], d["launch_iters"]) == (0, 32, 0, 0)


@pytest.mark.parametrize("nx,ny", [(127, 90), (128, 96)])
def test_capacity_of_768_nodes(gpu, nx, ny):
    """The capacity that none of those shapes has, ragged and full: the same comparisons."""
    d = shape(gpu, nx, ny)
    assert (d["cluster_ctas"], d["rows"], d["capacity"]) == (15 if ny == 90 else 16, 6, 768)
    for walls, scheme in ((1, 0), (0, 0), (1, 1)):
        cl.test_fixed_count_equals_streaming(gpu, nx, ny, walls, scheme)
    cl.test_rule_stops_where_the_tiled_loop_stops(gpu, nx, ny)
    cl.test_rule_on_the_last_bit(gpu, nx, ny, 1, 0, 40)


@pytest.mark.parametrize("loop", [0, 2])
def test_largest_capacity_under_the_rule(gpu, loop):
    """2880 nodes a CTA with a last tile of one column, which the two-step loop does not take: the
    cluster, as when one sub-iteration per exchange is asked for; it stops where the tiles do."""
    for nx, ny, ctas, rows in ((193, 224, 16, 14), (200, 200, 16, 13)):
        d = shape(gpu, nx, ny, poisson_loop=loop)
        if nx == 193 or loop == 2:
            assert (d["cluster_ctas"], d["rows"], d["capacity"]) == (ctas, rows, 2880)
        else:
            assert d["kind"] == 3 and d["cluster_ctas"] == 0
    p, f = cl.setup(193, 224, 1, 0, poisson_tol=1e-4, poisson_loop=loop)
    a, ia, _ = cl.states(gpu, p, f, 3)
    b, ib, _ = cl.states(gpu, dict(p, poisson_loop=2, tile_rows=cl.own_rows(193, 224)), f, 3)
    assert ia == ib
    for name in a:
        assert np.array_equal(a[name], b[name]), name
    cl.test_rule_on_the_last_bit(gpu, 193, 224, 1, 0, 41)


def test_streaming_launches(gpu):
    assert shape(gpu, 64, 40, poisson_loop=1)["launch_iters"] == 1
    assert shape(gpu, 1000, 600, poisson_loop=1)["launch_iters"] == 1
    assert shape(gpu, 1000, 601)["launch_iters"] == 5
    assert shape(gpu, 1000, 601)["kind"] == 1
