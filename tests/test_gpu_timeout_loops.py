"""Waits that run out, loop by loop: every on-chip loop has its own bounded wait and its own way
out, which differ between the stopping rule and a fixed count (tensor memory is held only under
the rule; the last barrier of a fixed count's single cycle is another than a full cycle's) and
between one and two spare copies of the one-cluster loop.  Each is named by its tiles or its
cluster, so that the library's choice cannot move the case elsewhere.  As in the other timeout
test a diagnostic makes the count unreachable for one solve, the waits run out after 2 s, the
call reports EHD_ERR_TIMEOUT and the context stays usable; the one-cluster loop, whose CTAs all
give up, leaves the state as it was."""
import time

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


# name: lattice side, parameters, the loop's shape (what loop_shape must say)
CASES = {
    "tiles-rule": (96, dict(poisson_loop=2, tile_rows=16), dict(kind=2, cluster_ctas=0, rows=16)),
    "tiles-fixed": (96, dict(poisson_loop=2, tile_rows=16, poisson_fixed_iter=5),
                    dict(kind=2, cluster_ctas=0, rows=16)),
    "two-step-rule": (96, dict(poisson_loop=3, tile_rows=32), dict(kind=3, rows=32)),
    "two-step-fixed-one-cycle": (96, dict(poisson_loop=3, tile_rows=32, poisson_fixed_iter=2),
                                 dict(kind=3, rows=32)),
    "two-step-fixed-odd": (96, dict(poisson_loop=3, tile_rows=32, poisson_fixed_iter=1),
                           dict(kind=3, rows=32)),
    "three-step-rule": (96, dict(poisson_loop=4, tile_rows=48), dict(kind=4, rows=48)),
    "cluster-rule": (96, dict(), dict(kind=2, cluster_ctas=16, capacity=768)),
    "cluster-fixed": (96, dict(poisson_fixed_iter=5), dict(kind=2, cluster_ctas=16, capacity=768)),
    "cluster-two-copies-rule": (187, dict(), dict(kind=2, cluster_ctas=16, capacity=2432)),
    "cluster-two-copies-fixed": (200, dict(poisson_fixed_iter=5),
                                 dict(kind=2, cluster_ctas=16, capacity=2880)),
    "one-cta": (16, dict(), dict(kind=2, cluster_ctas=1)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_expired_wait(gpu, name):
    n, over, shape = CASES[name]
    # at least three sub-iterations under the rule, so that every loop gets to wait
    p, f, _ = wl.droplet(N=n, r=0.15 * n, R=3.0, S=0.5, Ca=0.2, poisson_min_iter=3, **over)

    def run(steps):
        s = gpu.Sim(p)
        s.set_fields(f["phi"], f["q"], f["ux"], f["uy"])
        st = s.step(steps)
        out = s.read_fields()
        s.close()
        assert st["status"] == 0 and st["poisson_iters_min"] >= (over.get("poisson_fixed_iter") or 3)
        return out

    ref = run(6)
    s = gpu.Sim(p)
    got = s.loop_shape()
    assert {k: got[k] for k in shape} == shape
    s.set_fields(f["phi"], f["q"], f["ux"], f["uy"])
    s.step(2)
    before = s.read_fields(("varphi", "Ex", "Ey"))
    s.diag_expire_barrier()
    t0 = time.perf_counter()
    with pytest.raises(gpu.EhdError) as err:
        s.step(1)
    assert err.value.code == 9                            # EHD_ERR_TIMEOUT
    assert 1.5 < time.perf_counter() - t0 < 30.0          # the 2 s limit, not a hang
    if got["cluster_ctas"] > 1:
        after = s.read_fields(("varphi",))
        assert np.array_equal(after["varphi"], before["varphi"])
    s.close()
    again = run(6)
    for k in ref:
        assert np.array_equal(again[k], ref[k]), k
