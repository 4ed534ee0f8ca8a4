"""Launches of the streaming loop beyond the chip's storage under the stopping rule: a settled solve
of K sub-iterations makes ceil(K / 5) launches and repeats none, solves whose count changes from
step to step stop where one slab of the slab decomposition stops (one sub-iteration per launch;
states bit for bit, no tolerance), from the eight-step graphs, single ones and the host."""
import numpy as np
import pytest

from test_gpu_multi import setup

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


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 10, 11])
def test_settled_counts_need_no_repeat(gpu, k):
    p, f = setup(1000, 601, 1, 0, poisson_tol=1.0, poisson_min_iter=k)  # stops at k exactly
    s = gpu.Sim(p)
    s.set_fields(*f)
    for graphs in (True, False):
        s.use_graphs(graphs)
        s.step(2)
        st = s.step(12)
        assert st["poisson_iters_min"] == st["poisson_iters_max"] == k
        if graphs:  # the clearing of the statistics, moments and coupled pass, the loop
            assert st["kernel_launches"] == 1 + 12 * (2 + (k + 4) // 5)
    assert s.solve_potential()[0] == k
    s.close()


@pytest.mark.parametrize("nx,ny,walls,scheme", [(977, 811, 1, 0), (1024, 600, 0, 0), (641, 950, 1, 1)])
def test_changing_counts(gpu, nx, ny, walls, scheme):
    counts = set()
    for tol in (3e-3, 5e-4, 1e-4):
        p, f = setup(nx, ny, walls, scheme, poisson_tol=tol, ramp_steps=12,
                     varphi_bottom=-0.2 if walls else 0.0)
        s, h, t = gpu.Sim(p), gpu.Sim(p), gpu.Slabs(p, 1)
        h.use_graphs(False)
        for o in (s, h, t):
            o.set_fields(*f)
        for n in (1, 9, 3):
            got = [o.step(n) for o in (s, h, t)]
            assert len({g["poisson_iters_total"] for g in got}) == 1
            counts.add((got[0]["poisson_iters_min"], got[0]["poisson_iters_max"]))
        fields = [o.read_fields() for o in (s, h, t)]
        for o in (s, h, t):
            o.close()
        for name in fields[0]:
            assert np.array_equal(fields[0][name], fields[2][name]), (name, tol)
            assert np.array_equal(fields[1][name], fields[2][name]), (name, tol)
    assert any(a != b for a, b in counts)  # some call met several counts


def test_new_fields_forget_the_count(gpu):
    p, f = setup(1000, 601, 1, 0, poisson_tol=1e-4)
    ends = []
    for again in (False, True):
        s = gpu.Sim(p)
        s.set_fields(*f)
        if again:
            s.step(5)
            s.set_fields(*f)
        st = s.step(3)
        ends.append((st["poisson_iters_total"], st["kernel_launches"], s.read_fields()))
        s.close()
    assert ends[0][:2] == ends[1][:2]
    for name in ends[0][2]:
        assert np.array_equal(ends[0][2][name], ends[1][2][name]), name
