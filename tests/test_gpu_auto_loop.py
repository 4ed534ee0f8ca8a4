"""The library's own choice of loop under the stopping rule: on tall tiles steps whose solves settle
at one sub-iteration (on tiles of 56 rows also at three) move to the one-step loop, the others
keep the two-step loop; with the largest cluster, where the two-step loop does not fit, one and
two sub-iterations move; beyond the chip's storage one sub-iteration moves to launches of one.  New fields start with the other form again; the states are those of
one loop bit for bit (no tolerance).  The count is set by equal smallest and largest counts, which
the rule's kernels honour whatever the change of the potential."""
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


def setup(nx, ny, k, **over):
    p = wl.make_params(nx=nx, ny=ny, walls_y=1, eps_l=4.0, sigma_l=0.05, sigma_v=0.01, varphi_top=0.3,
                       poisson_tol=1e-12, poisson_min_iter=k, poisson_max_iter=k)
    p.update(over)
    y, x = np.meshgrid(np.arange(ny), np.arange(nx), indexing="ij")
    phi = wl.tanh_profile(0.3 * min(nx, ny) - np.hypot(x - nx / 2.1, y - ny / 2.3), 4.0)
    return p, (phi, 0 * phi, 0 * phi, 0 * phi)


# lattice, storage, count, the loop it settles on (2: one step, 3: two steps an exchange, 0: cluster)
CASES = [(200, 200, 0, 1, 2), (200, 200, 0, 2, 3), (193, 224, 0, 1, 2), (193, 224, 1, 2, 2),
         (193, 224, 0, 3, 0), (1000, 601, 0, 1, "single"), (1000, 601, 1, 2, "several"),
         (300, 300, 0, 1, 2), (300, 300, 1, 1, 2), (300, 300, 0, 2, 3), (300, 300, 0, 3, 3),
         (256, 256, 0, 1, 3), (512, 1024, 0, 1, 2), (512, 1024, 0, 3, 2), (512, 1024, 0, 5, 3)]


def loop_of(s):
    d = s.loop_shape()
    if d["kind"] == 1:
        return {1: "single", 5: "several"}[d["launch_iters"]]
    return 0 if d["cluster_ctas"] else d["kind"]


@pytest.mark.parametrize("nx,ny,precision,k,settled", CASES)
def test_settled_counts_choose_the_loop(gpu, nx, ny, precision, k, settled):
    p, f = setup(nx, ny, k, precision=precision)
    ends = []
    first = {193: 0, 1000: "several"}.get(nx, 3)
    one_loop = {193: dict(poisson_loop=2, tile_rows=32), 1000: dict(poisson_loop=1)}.get(
        nx, dict(poisson_loop=3))
    for over in (dict(), one_loop):
        s = gpu.Sim({**p, **over})
        if over.get("poisson_loop") == 1:
            s.use_graphs(False)  # steps from the host keep their launches of several
        s.set_fields(*f)
        stays = {1: first}.get(over.get("poisson_loop"), over.get("poisson_loop"))
        assert loop_of(s) == (stays or first)
        for n in (3, 60, 61, 700, 257):  # calls that end between two looks at the count, and odd ones
            st = s.step(n)
            assert st["poisson_iters_min"] == st["poisson_iters_max"] == k and st["steps"] == n
            if n < 64:  # neither a look's answer nor enough steps of one count
                assert loop_of(s) == (stays or first)
        assert loop_of(s) == (stays or settled)
        ends.append(s.read_fields())
        blob = s.save_state()
        if not over:
            for again in (lambda: s.set_fields(*f), lambda: s.load_state(blob)):
                again()
                assert loop_of(s) == first
                s.step(64)  # as many of one count as its statistics need to tell
                assert loop_of(s) == settled
        s.close()
    for name in ends[0]:
        assert np.array_equal(ends[0][name], ends[1][name]), name


def test_tallest_tiles_keep_the_one_step_loop(gpu):
    """64 rows: the one-step loop under the rule, the two-step loop at a fixed count."""
    p, f = setup(576, 1024, 2)
    for over, kind in ((dict(), 2), (dict(poisson_fixed_iter=2), 3)):
        s = gpu.Sim({**p, **over})
        s.set_fields(*f)
        s.step(600)
        s.step(300)
        assert s.loop_kind() == kind
        s.close()


def test_single_steps_and_profiling(gpu):
    """Steps one at a time follow the count too; steps under profiling run the chosen loop."""
    p, f = setup(300, 300, 1)
    s = gpu.Sim(p)
    s.set_fields(*f)
    for _ in range(600):
        s.step(1)
    assert s.loop_kind() == 2
    s.profile(True)
    s.step(4)
    assert s.profile_read()["potential"]["launches"] == 4
    s.profile(False)
    a = s.read_fields()
    s.close()
    s = gpu.Sim(dict(p, poisson_loop=3))
    s.set_fields(*f)
    s.step(604)
    b = s.read_fields()
    s.close()
    for name in a:
        assert np.array_equal(a[name], b[name]), name


def test_calls_without_statistics_follow_the_count(gpu):
    """Nothing is read back but the count; the answers of a long call arrive while it is queued or
    before the next one."""
    p, f = setup(300, 300, 1)
    s = gpu.Sim(p)
    s.set_fields(*f)
    for _ in range(4):
        s.step(200, stats=False)
        s.read_fields(("phi",))
    assert s.loop_kind() == 2
    st = s.read_stats()
    assert st["steps"] == 800 and st["poisson_iters_total"] == 800
    s.close()
