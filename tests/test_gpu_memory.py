"""Memory the library holds: F64 links without room for their second form, and
the pools' memory given back."""
import numpy as np
import pytest

from conftest import rel_l2
from gpu_helpers import dev, host
from paper_0710_2442_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def w():
    from paper_0710_2442_gb300 import build, wilson
    build.build()
    return wilson


def test_f64_handle_without_room_for_both_forms(w):
    """24^3 x 48 links take 382 MB in each form: with room for one and a half, the handle is
    made all the same and its hops run on the doubles.  Tolerance: two FP64 hops, as in the
    fixed-point tests."""
    import torch
    dims = (24, 24, 24, 48)
    L = w.lattice(dims)
    U = dev(inputs.gauge_field(dims, "weak", eps=0.3, seed=431))
    src = dev(inputs.gaussian_spinor(inputs.volume(dims) // 2, seed=432))
    a, b = w.Spinor(L, w.WILSON_ODD, w.WILSON_F64), w.Spinor(L, w.WILSON_EVEN, w.WILSON_F64)
    a.load(src)

    def hop():
        g = w.Gauge(U, L, w.WILSON_F64, 18)
        left = torch.cuda.mem_get_info()[0]
        w.wilson_dslash_h(b, g, a, 0.0, w.WILSON_OP_HOP)
        out = torch.empty_like(src)
        b.store(out)
        res = host(out)
        g.close()
        return res, left

    want, _ = hop()
    w.wilson_release_workspace()
    torch.cuda.empty_cache()
    links = 18 * 8 * 4 * inputs.volume(dims)
    free = torch.cuda.mem_get_info()[0]
    out = torch.empty_like(src)  # before the memory is taken, for the cache to hand out again
    del out
    fill = torch.empty(torch.cuda.mem_get_info()[0] - links * 3 // 2 - (64 << 20), dtype=torch.uint8, device="cuda")
    got, left = hop()
    assert left > links // 4, "the second form was made"
    del fill
    torch.cuda.empty_cache()
    assert torch.cuda.mem_get_info()[0] >= free - (128 << 20)
    assert rel_l2(got, want) <= 1e-14


def test_workspace_is_given_back(w):
    import torch
    dims = (16, 16, 16, 16)
    U = dev(inputs.gauge_field(dims, "weak", eps=0.3, seed=433))
    b = dev(inputs.gaussian_spinor(dims, seed=434))
    x = torch.zeros_like(b)
    L = w.lattice(dims)
    w.wilson_release_workspace()
    runs = []
    for _ in range(2):
        x.zero_()
        w.wilson_cg_solve(x, U, b, L, 0.13, w.solver_defaults(w.WILSON_F16))
        runs.append(host(x))
        torch.cuda.synchronize()
        kept = torch.cuda.mem_get_info()[0]
        w.wilson_release_workspace()
        assert torch.cuda.mem_get_info()[0] > kept  # a solve keeps its workspace, until it is asked for
    assert np.array_equal(runs[0], runs[1])
