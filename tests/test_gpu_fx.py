"""The F64 hops in block fixed point (dslash_fx.cuh) at the edges of their tiles
and of the rule that chooses between the two kernels, against the FP64 oracle;
and fields and links out of the fixed-point ranges against the FP64 stencil.

Tolerance: a term is exact to 2^-56 of its half spinor's scale and the sum of eight hops of
at most 12 scales is rounded to FP64 once, so a component is off by at most
8 * 12 * 2^-56 scales + 2^-53 of itself: 1.4e-15 scales, with a scale of at most
about 8 rms of the output.  1e-14 relative L2 holds all of it, oracle rounding included.
"""
import numpy as np
import pytest

from conftest import assert_parity
from gpu_helpers import handle_hop
from paper_0710_2442_gb300 import inputs

pytestmark = pytest.mark.gpu

PHASES = (np.exp(0.4j), 1.0, np.exp(-2.2j), -1.0)
TOL = 1e-14

# half volumes 16 (less than a tile), 1680 (a ragged tile), 13440 (a half field below the
# rule's 20000 sites, a full field above), 20480 (above), 20748 (above, ragged)
DIMS = [(2, 2, 4, 2), (6, 10, 4, 14), (12, 14, 16, 10), (16, 16, 16, 10), (14, 14, 12, 18)]


@pytest.fixture(scope="module")
def w():
    from paper_0710_2442_gb300 import build, wilson
    build.build()
    return wilson


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("recon,op", [(18, "hop"), (12, "hop"), (18, "schur_dag"), (18, "m")])
def test_fixed_point_hops(w, oracle_mod, dims, recon, op):
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=401)
    if op == "m":
        src = inputs.gaussian_spinor(dims, seed=402)
        got = handle_hop(w, U, src, dims, PHASES, w.WILSON_F64, recon, w.WILSON_FULL, w.WILSON_FULL, w.WILSON_OP_M, 0.135)
        want = oracle_mod.wilson_m(U, src, dims, 0.135, PHASES)
    elif op == "hop":
        src = inputs.gaussian_spinor(inputs.volume(dims) // 2, seed=403)
        got = handle_hop(w, U, src, dims, PHASES, w.WILSON_F64, recon, 1, 0, w.WILSON_OP_HOP)
        want = oracle_mod.dslash_eo(U, src, dims, 0, PHASES)
    else:
        src = inputs.gaussian_spinor(inputs.volume(dims) // 2, seed=404)
        got = handle_hop(w, U, src, dims, PHASES, w.WILSON_F64, recon, 1, 1, w.WILSON_OP_SCHUR_DAG, 0.135)
        want = oracle_mod.schur(U, src, dims, 0.135, 1, True, PHASES)
    assert_parity(got, want, TOL)


def test_fixed_point_multi_rhs(w, oracle_mod):
    dims = (8, 10, 8, 22)  # 3 x 7040 sites: above the rule's line together
    U = inputs.gauge_field(dims, "random", seed=405)
    src = inputs.gaussian_spinor(inputs.volume(dims) // 2, seed=406, nrhs=3)
    got = handle_hop(w, U, src, dims, PHASES, w.WILSON_F64, 18, 0, 0, w.WILSON_OP_SCHUR, 0.13, nrhs=3)
    for k in range(3):
        assert_parity(got[k], oracle_mod.schur(U, src[k], dims, 0.13, 0, False, PHASES), TOL)


@pytest.mark.parametrize("dims", [(4, 4, 4, 6), (12, 14, 16, 16)])
@pytest.mark.parametrize("case", ["nan", "inf", "large links", "small links", "one link", "denormal", "huge", "zero", "point"])
def test_out_of_range(w, monkeypatch, dims, case):
    """What does not fit runs on the FP64 stencil site by site: the same NaN, Inf
    and zero patterns as with that stencil throughout, and the same values."""
    U = inputs.gauge_field(dims, "random", seed=407)
    src = inputs.gaussian_spinor(inputs.volume(dims) // 2, seed=408)
    if case in ("nan", "inf"):
        src[17, 2, 1] = np.nan if case == "nan" else np.inf
    elif case == "large links":
        U = U * 7.5
    elif case == "small links":
        U = U * 1e-9
    elif case == "one link":
        U[101, 2] *= 3.0
    elif case in ("denormal", "huge"):
        src = src * (1e-312 if case == "denormal" else 1e200)
    elif case in ("zero", "point"):
        src = src * 0
        if case == "point":
            src[3, 1, 2] = -1.0
    args = (w, U, src, dims, PHASES, w.WILSON_F64, 18, 0, 0, w.WILSON_OP_SCHUR, 0.13)
    with np.errstate(all="ignore"):
        got = handle_hop(*args)
        monkeypatch.setenv("WILSON_HOP_VARIANT", "0")
        want = handle_hop(*args)
        for part in ("real", "imag"):
            a, b = getattr(got, part), getattr(want, part)
            assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(a[~np.isfinite(b)], b[~np.isfinite(b)], equal_nan=True)
            f = np.isfinite(b)
            if case == "zero":
                assert np.all(a == 0)
            else:
                assert np.max(np.abs(a[f] - b[f])) <= TOL * np.max(np.abs(b[f]))


@pytest.mark.parametrize("dims", [(4, 4, 4, 6), (14, 14, 12, 18)])
def test_output_over_an_input(w, dims):
    """An output that overlaps the links or part of the input is what it is in
    memory of its own (the kernels read their inputs while they write)."""
    import torch
    L = w.lattice(dims, PHASES)
    V = inputs.volume(dims)
    U = torch.from_numpy(inputs.gauge_field(dims, "random", seed=409)).cuda()
    src = torch.from_numpy(inputs.gaussian_spinor(V // 2, seed=410)).cuda()
    want = torch.empty_like(src)
    for op in (w.WILSON_OP_HOP, w.WILSON_OP_SCHUR):
        w.wilson_dslash_eo(want, U, src, L, 0, 0.13, op)
        links = U.clone()
        out = links.reshape(-1)[: src.numel()].view_as(src)
        w.wilson_dslash_eo(out, links, src, L, 0, 0.13, op)
        assert torch.equal(out, want)
        both = torch.cat([src.reshape(-1), torch.zeros(1200, dtype=src.dtype, device="cuda")])
        out = both[1200:].view_as(src)
        w.wilson_dslash_eo(out, U, both[: src.numel()].view_as(src), L, 0, 0.13, op)
        assert torch.equal(out, want)


@pytest.mark.parametrize("scale", [1.0, 2.0**-400, 2.0**450])
def test_conversions_agree(w, scale):
    """The split kernel rounds its sums to FP64 with FP64 additions at up to one tile per SM
    (53 tiles, one right-hand side) and with integers beyond (three): the same bits."""
    dims = (6, 10, 4, 14)
    U = inputs.gauge_field(dims, "random", seed=409)
    src = inputs.gaussian_spinor(inputs.volume(dims) // 2, seed=410) * scale
    src[::3] = 0.0  # exact zeros and sums of few terms, of either sign
    src[1::3] = np.where(np.abs(src[1::3].real) > scale, src[1::3], -scale * 2.0**-30)
    args = (dims, PHASES, w.WILSON_F64, 18, 1, 0, w.WILSON_OP_HOP)
    three = handle_hop(w, U, np.stack([src, -src, src]), *args, nrhs=3)
    for k, sign in enumerate((1.0, -1.0, 1.0)):
        assert np.array_equal(three[k], handle_hop(w, U, sign * src, *args))


@pytest.mark.parametrize("dims", [(4, 2, 4, 6), (12, 14, 16, 16)])
@pytest.mark.parametrize("case", ["mean link", "all entries", "third row"])
def test_links_at_the_edge_of_the_range(w, monkeypatch, dims, case):
    """Entries up to 1.25 stay in fixed point: SU(3) over a mean link of 0.8, and links whose every entry is as large
    as it may be, with a field that adds all products up; 12-real links whose third row leaves the range do not.
    Against the FP64 stencil, whose own error is at most 16 roundings of a sum of moduli."""
    V = inputs.volume(dims)
    U = inputs.gauge_field(dims, "random", seed=411)
    src = inputs.gaussian_spinor(V // 2, seed=412)
    recon = 18
    if case == "mean link":
        U = U / 0.8
    elif case == "all entries":
        U = np.full_like(U, 1.25 - 1.25j)
        src = np.full_like(src, 1.0 + 1.0j)
    else:
        recon = 12
        U[..., 0, :] = 0.95 + 0.95j
        U[..., 1, :] = (0.95 - 0.95j) * np.array([1.0, -1.0, 1.0])
    args = (w, U, src, dims, PHASES, w.WILSON_F64, recon, 1, 0, w.WILSON_OP_HOP)
    got = handle_hop(*args)
    monkeypatch.setenv("WILSON_HOP_VARIANT", "0")
    assert_parity(got, handle_hop(*args), TOL)
