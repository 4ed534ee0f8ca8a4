"""Device arrays that a caller hands to ehd_read_fields: which the output kernel writes itself, and
which go through checked copies.  The predicate is asked alone, with addresses that no kernel
then touches; a read into arrays that overlap is made and equals a read into arrays of its own."""
import ctypes

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


def direct(ehd, ptrs, nbytes):
    return ehd.lib().ehd_diag_direct_outputs((ctypes.c_void_p * len(ptrs))(*ptrs), len(ptrs), nbytes)


def test_only_whole_separate_arrays_are_written_by_the_kernel(gpu):
    import torch
    size = 64 << 20
    with torch.cuda.use_mem_pool(torch.cuda.MemPool()):  # an allocation of its own
        buf = torch.empty(size, dtype=torch.uint8, device="cuda")
    lo = buf.data_ptr()
    assert direct(gpu, [lo], size) == 1
    assert direct(gpu, [lo], size + 1) == 0                  # past the end
    assert direct(gpu, [lo + size - 4096], 4096) == 1        # up to the end
    assert direct(gpu, [lo + size - 4096], 4100) == 0        # past the end from inside
    assert direct(gpu, [lo + size - 4], 1 << 62) == 0        # no wrap in the arithmetic
    assert direct(gpu, [lo + 2], 4096) == 0                  # misaligned
    assert direct(gpu, [lo, lo + 4096], 4096) == 1           # side by side
    assert direct(gpu, [lo, lo + 4092], 4096) == 0           # overlapping
    assert direct(gpu, [lo + 4092, lo], 4096) == 0
    assert direct(gpu, [lo, lo], 4096) == 0                  # the same array twice
    host = torch.empty(4096, dtype=torch.uint8).pin_memory()
    assert direct(gpu, [host.data_ptr()], 4096) == 0
    plain = np.empty(4096, np.uint8)
    assert direct(gpu, [plain.ctypes.data], 4096) == 0
    assert direct(gpu, [lo], 0) == 1 and direct(gpu, [None], 4) == 0


def test_overlapping_outputs_keep_the_order_of_the_fields(gpu):
    import torch
    p, f, _ = wl.droplet(N=40, r=8.0, R=3.0, S=0.5, Ca=0.2, poisson_fixed_iter=2)
    s = gpu.Sim(p)
    s.set_fields(f["phi"], f["q"], f["ux"], f["uy"])
    s.step(3)
    own = s.read_fields(("phi", "varphi"), device=True)
    n = 40 * 40
    buf = torch.zeros(n + 40, dtype=torch.float32, device="cuda")
    out = {"phi": buf[:n].view(40, 40), "varphi": buf[40:].view(40, 40)}
    s.read_fields(("phi", "varphi"), device=True, out=out)
    s.close()
    assert torch.equal(buf[:40], own["phi"].reshape(-1)[:40])
    assert torch.equal(buf[40:], own["varphi"].reshape(-1))
