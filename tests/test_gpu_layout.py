"""Import and export of several right-hand sides in one launch: bit for bit what
each right-hand side gives alone, and what the storage format makes of the values."""
import numpy as np
import pytest

from gpu_helpers import dev, host
from paper_0710_2442_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def w():
    from paper_0710_2442_gb300 import build, wilson
    build.build()
    return wilson


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 10, 4, 14), (14, 12, 6, 10)])
@pytest.mark.parametrize("prec", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("subset", [0, 1, 2])
def test_multi_rhs_round_trip(w, dims, prec, subset):
    import torch
    L = w.lattice(dims)
    n = inputs.volume(dims) // (1 if subset == 2 else 2)
    src = inputs.gaussian_spinor(n, seed=501, nrhs=3)
    a = w.Spinor(L, subset, w.PREC[prec], 3)
    a.load(dev(src))
    out = torch.full((3, n, 4, 3), float("nan"), dtype=torch.complex128, device="cuda")
    a.store(out)
    got = host(out)
    for k in range(3):
        b = w.Spinor(L, subset, w.PREC[prec])
        b.load(dev(src[k]))
        one = torch.full((n, 4, 3), float("nan"), dtype=torch.complex128, device="cuda")
        b.store(one)
        assert np.array_equal(got[k], host(one))
    if prec in ("f64", "f32"):
        assert np.array_equal(got, src if prec == "f64" else src.astype(np.complex64).astype(np.complex128))
    else:  # one rounding of a value below its site's largest component
        top = np.abs(src.view(np.float64)).reshape(3, n, -1).max(axis=2)[..., None, None]
        assert np.max(np.abs((got - src).view(np.float64).reshape(3, n, 4, 6)) / top) <= (2.0 ** -11 if prec == "f16" else 2.0 ** -8)


def test_default_stream_is_torchs_current_one(w):
    import torch
    side = torch.cuda.Stream()
    assert w._stream(None) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(side):
        assert w._stream(None) == side.cuda_stream == w._stream(side)
    assert w._stream(None) == torch.cuda.current_stream().cuda_stream
