"""GPU CG solves against the FP64 oracle.

The binding check is each GPU solution's true residual |b - M x| / |b|
recomputed by the oracle's FP64 Wilson matrix (<= 1e-10, the solve target,
with 10% slack for the different summation order), plus agreement with the
oracle's own solution within cond(M) * 1e-10.
"""
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


def solve(w, U, b, dims, kappa, inner, reliable=1, recon=None, maxiter=100000, tol=1e-10, phases=None, check=True):
    phases = inputs.DEFAULT_PHASES if phases is None else phases
    L = w.lattice(dims, phases)
    p = w.solver_defaults(inner)
    p.reliable = reliable
    p.tol = tol
    p.maxiter = maxiter
    if recon is not None:
        p.recon = recon
    x = dev(np.zeros_like(b))
    st = w.wilson_cg_solve(x, dev(U), dev(b), L, kappa, p, check=check)
    return host(x), st


def true_resid(oracle_mod, U, x, b, dims, kappa, phases=None):
    r = b - oracle_mod.wilson_m(U, x, dims, kappa, phases)
    return np.linalg.norm(r) / np.linalg.norm(b)


@pytest.mark.parametrize("inner", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("reliable", [1, 0])
def test_solve_matches_oracle(w, oracle_mod, inner, reliable):
    dims = (4, 4, 4, 8)
    kappa = 0.1350
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=201)
    b = inputs.gaussian_spinor(dims, seed=202)
    x, st = solve(w, U, b, dims, kappa, w.PREC[inner], reliable)
    assert st["rc"] == 0 and st["true_rel_resid"] <= 1e-10
    assert true_resid(oracle_mod, U, x, b, dims, kappa) <= 1.1e-10
    xo, info = oracle_mod.cg_solve(U, b, dims, kappa, tol=1e-12)
    assert info["converged"]
    # cond(M) of this 4^3 x 8 weak field is below 100: solutions agree to ~1e-8
    assert rel_l2(x, xo) <= 1e-7


def test_solve_complex_phases_random_field(w, oracle_mod):
    dims = (4, 2, 4, 6)
    kappa = 0.124
    phases = (np.exp(0.7j), 1.0, np.exp(-1.9j), -1.0)
    U = inputs.gauge_field(dims, "random", seed=203)
    b = inputs.gaussian_spinor(dims, seed=204)
    for inner in ("f64", "f32", "f16"):
        x, st = solve(w, U, b, dims, kappa, w.PREC[inner], recon=18 if inner == "f64" else 12, phases=phases)
        assert true_resid(oracle_mod, U, x, b, dims, kappa, phases) <= 1.1e-10


def test_solve_ragged_lattice(w, oracle_mod):
    dims = (6, 4, 6, 10)  # Vh = 720: several blocks and a ragged tail
    kappa = 0.13
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=205)
    b = inputs.gaussian_spinor(dims, seed=206)
    x, st = solve(w, U, b, dims, kappa, w.WILSON_F16)
    assert true_resid(oracle_mod, U, x, b, dims, kappa) <= 1.1e-10


def test_maxiter_reports_noconv(w):
    dims = (4, 4, 4, 8)
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=207)
    b = inputs.gaussian_spinor(dims, seed=208)
    x, st = solve(w, U, b, dims, 0.135, w.WILSON_F32, maxiter=5, check=False)
    assert st["rc"] == w.WILSON_ERR_NOCONV
    assert st["inner_iters"] <= 5 + 16


def test_nan_source_reports_numeric(w):
    dims = (4, 4, 4, 4)
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=209)
    b = inputs.gaussian_spinor(dims, seed=210)
    b[5, 1, 2] = np.nan
    x, st = solve(w, U, b, dims, 0.13, w.WILSON_F32, check=False)
    assert st["rc"] == w.WILSON_ERR_NUMERIC


def test_zero_source(w):
    dims = (4, 4, 4, 4)
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=211)
    b = np.zeros((inputs.volume(dims), 4, 3), dtype=np.complex128)
    x, st = solve(w, U, b, dims, 0.13, w.WILSON_F16)
    assert st["rc"] == 0 and np.all(x == 0)


@pytest.mark.parametrize("inner", ["f64", "f16", "f32"])
def test_multi_rhs_solve(w, oracle_mod, inner):
    """12 right-hand sides (point sources and Gaussian noise) sharing one gauge
    field, solved together; each reaches the target against the oracle's M."""
    dims = (4, 4, 4, 8)
    kappa = 0.1350
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=212)
    V = inputs.volume(dims)
    b = np.concatenate([inputs.point_sources(dims, site=5)[:8],
                        inputs.gaussian_spinor(dims, seed=213, nrhs=4)], axis=0)
    L = w.lattice(dims)
    x = dev(np.zeros_like(b))
    rc, st = w.wilson_cg_solve_multi(x, dev(U), dev(b), 12, L, kappa, w.solver_defaults(w.PREC[inner]))
    xs = host(x)
    assert rc == 0
    for k in range(12):
        assert st[k]["true_rel_resid"] <= 1e-10
        assert true_resid(oracle_mod, U, xs[k], b[k], dims, kappa) <= 1.1e-10
    # the lockstep solve gives the single-rhs solution
    x1, _ = solve(w, U, b[9], dims, kappa, w.PREC[inner])
    assert rel_l2(xs[9], x1) <= 1e-8


def test_multi_rhs_with_zero_and_easy_rhs(w, oracle_mod):
    """Right-hand sides that finish at different times (a zero source finishes
    at once) are skipped while the others continue."""
    dims = (4, 4, 4, 4)
    kappa = 0.13
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=214)
    b = inputs.gaussian_spinor(dims, seed=215, nrhs=3)
    b[1] = 0
    L = w.lattice(dims)
    x = dev(np.zeros_like(b))
    rc, st = w.wilson_cg_solve_multi(x, dev(U), dev(b), 3, L, kappa, w.solver_defaults(w.WILSON_F16))
    xs = host(x)
    assert rc == 0 and np.all(xs[1] == 0)
    for k in (0, 2):
        assert true_resid(oracle_mod, U, xs[k], b[k], dims, kappa) <= 1.1e-10


def multi(w, U, b, dims, kappa, inner, block, phases=None, check=True):
    L = w.lattice(dims, inputs.DEFAULT_PHASES if phases is None else phases)
    p = w.solver_defaults(inner)
    p.block_cg = block
    x = dev(np.zeros_like(b))
    rc, st = w.wilson_cg_solve_multi(x, dev(U), dev(b), b.shape[0], L, kappa, p, check=check)
    return rc, host(x), st


@pytest.mark.parametrize("inner", ["f64", "f32", "f16", "bf16"])
def test_block_cg_solve(w, oracle_mod, inner):
    """Block CG over 12 right-hand sides (8 point sources and 4 Gaussian
    sources): every column reaches the target against the oracle's M, and
    the solutions agree with the independent CGs' solutions."""
    dims, kappa = (4, 4, 4, 8), 0.1350
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=230)
    b = np.concatenate([inputs.point_sources(dims, site=7)[:8],
                        inputs.gaussian_spinor(dims, seed=231, nrhs=4)], axis=0)
    rc, xb, st = multi(w, U, b, dims, kappa, w.PREC[inner], 1)
    assert rc == 0
    for k in range(12):
        assert st[k]["status"] == 0 and st[k]["true_rel_resid"] <= 1e-10
        assert true_resid(oracle_mod, U, xb[k], b[k], dims, kappa) <= 1.1e-10
    rc, xi, _ = multi(w, U, b, dims, kappa, w.PREC[inner], 0)
    for k in range(12):
        assert rel_l2(xb[k], xi[k]) <= 1e-8


def test_block_cg_shares_the_krylov_space(w, oracle_mod):
    """In FP64 the block method needs fewer iterations than the slowest of
    the independent CGs (each iteration widens the search space by all 12
    columns' directions)."""
    dims, kappa = (4, 4, 4, 8), 0.1355
    U = inputs.gauge_field(dims, "weak", eps=0.35, seed=232)
    b = inputs.gaussian_spinor(dims, seed=233, nrhs=12)
    _, xb, sb = multi(w, U, b, dims, kappa, w.WILSON_F64, 1)
    _, xi, si = multi(w, U, b, dims, kappa, w.WILSON_F64, 0)
    blk = max(s["inner_iters"] for s in sb)
    ind = max(s["inner_iters"] for s in si)
    assert blk < 0.8 * ind, (blk, ind)
    for k in range(12):
        assert true_resid(oracle_mod, U, xb[k], b[k], dims, kappa) <= 1.1e-10


def test_block_cg_degenerate_columns(w, oracle_mod):
    """A zero source (finished before the block starts), a source that
    repeats another one and one that is a multiple of a third: the block
    loses rank, falls back to independent CGs, and every column still
    reaches the target."""
    dims, kappa = (4, 4, 4, 4), 0.13
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=234)
    b = inputs.gaussian_spinor(dims, seed=235, nrhs=6)
    b[1] = 0
    b[3] = b[2]
    b[5] = (0.5 - 2j) * b[4]
    rc, x, st = multi(w, U, b, dims, kappa, w.WILSON_F16, 1)
    assert rc == 0 and np.all(x[1] == 0)
    for k in (0, 2, 3, 4, 5):
        assert true_resid(oracle_mod, U, x[k], b[k], dims, kappa) <= 1.1e-10


def test_block_cg_nan_source_is_per_column(w, oracle_mod):
    """A NaN in one source is caught by the FP64 residual before the block
    starts; that column reports WILSON_ERR_NUMERIC and the others converge."""
    dims, kappa = (4, 4, 4, 4), 0.13
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=236)
    b = inputs.gaussian_spinor(dims, seed=237, nrhs=4)
    b[2, 5, 1, 1] = np.nan
    rc, x, st = multi(w, U, b, dims, kappa, w.WILSON_F16, 1, check=False)
    assert rc == w.WILSON_ERR_NUMERIC and st[2]["status"] == w.WILSON_ERR_NUMERIC
    for k in (0, 1, 3):
        assert st[k]["status"] == 0
        assert true_resid(oracle_mod, U, x[k], b[k], dims, kappa) <= 1.1e-10


@pytest.mark.parametrize("inner", ["f64", "f16"])
def test_kappa_zero_is_identity(w, inner):
    """kappa = 0 makes M the identity: the solve returns x = b."""
    dims = (4, 4, 4, 6)
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=240)
    b = inputs.gaussian_spinor(dims, seed=241)
    x, st = solve(w, U, b, dims, 0.0, w.PREC[inner])
    assert st["rc"] == 0 and st["true_rel_resid"] <= 1e-10
    assert rel_l2(x, b) <= 1e-10


@pytest.mark.parametrize("inner", ["f16", "bf16", "f32"])
def test_fp32_outer_residuals(w, oracle_mod, inner):
    """The early corrections of an F16/BF16 solve compute their residual with
    FP32 fields and links (expected residual above 1e-4 |bhat|); an F32 solve
    (inner reduction 1e-4) has none.  Every solve still reaches the 1e-10
    true residual by the oracle's FP64 M, also in the lockstep multi-RHS
    form.  A target at or above 1e-7 uses only FP64 residuals."""
    dims = (8, 6, 4, 10)
    kappa = 0.1350
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=161)
    b = inputs.gaussian_spinor(dims, seed=162)
    x, st = solve(w, U, b, dims, kappa, w.PREC[inner])
    assert st["rc"] == 0
    if inner == "f32":
        assert st["outer_f32"] == 0
    else:
        assert st["outer_f32"] >= 1
        assert st["outer_f32"] < st["outer_iters"]  # the last corrections are FP64
    assert true_resid(oracle_mod, U, x, b, dims, kappa) <= 1.1e-10
    x, st = solve(w, U, b, dims, kappa, w.PREC[inner], tol=1e-6)
    assert st["rc"] == 0 and st["outer_f32"] == 0
    assert true_resid(oracle_mod, U, x, b, dims, kappa) <= 1.1e-6
    bs = inputs.gaussian_spinor(dims, seed=163, nrhs=3)
    bs[1] *= 1e-4  # a right-hand side of another scale: its own |bhat| sets its threshold
    xs = dev(np.zeros_like(bs))
    rc, sts = w.wilson_cg_solve_multi(xs, dev(U), dev(bs), 3, w.lattice(dims), kappa, w.solver_defaults(w.PREC[inner]))
    assert rc == 0 and (sts[0]["outer_f32"] >= 1) == (inner != "f32")
    xh = host(xs)
    for k in range(3):
        assert true_resid(oracle_mod, U, xh[k], bs[k], dims, kappa) <= 1.1e-10


@pytest.mark.parametrize("inner", ["f16", "f32"])
def test_lockstep_solve_repeats_itself(w, inner):
    """Kernels of a 12-right-hand-side iteration run in several waves (12 x 144 blocks of 256
    threads), with blocks of a right-hand side starting while its first block
    records that it has finished: every run takes the same iterations and gives the same bits.
    The sources span scales and shapes, so that they finish at different times."""
    dims, kappa = (24, 16, 12, 16), 0.13
    U = dev(inputs.gauge_field(dims, "weak", eps=0.3, seed=250))
    b = inputs.gaussian_spinor(dims, seed=251, nrhs=12)
    b[3] = 0
    b[5:9] = inputs.point_sources(dims, site=9)[:4]
    db = dev(b)
    runs = []
    for _ in range(4):
        x = dev(np.zeros_like(b))
        rc, st = w.wilson_cg_solve_multi(x, U, db, 12, w.lattice(dims), kappa, w.solver_defaults(w.PREC[inner]))
        assert rc == 0
        runs.append((host(x), [s["inner_iters"] for s in st], st[0]["outer_iters"]))
    for x, it, outer in runs[1:]:
        assert it == runs[0][1] and outer == runs[0][2]
        assert np.array_equal(x, runs[0][0])


def test_block_cg_beside_a_busy_default_stream(w):
    """A solve's set-up is ordered on its own stream alone: work queued on the legacy default
    stream, which the solve does not wait for, changes nothing."""
    import torch
    dims, kappa = (4, 4, 4, 8), 0.1350
    U = dev(inputs.gauge_field(dims, "weak", eps=0.3, seed=252))
    b = dev(inputs.gaussian_spinor(dims, seed=253, nrhs=4))
    L = w.lattice(dims)
    p = w.solver_defaults(w.WILSON_F32)
    p.block_cg = 1
    side = torch.cuda.Stream()
    load = torch.ones(2048, 2048, device="cuda")
    runs = []
    for busy in (False, True, True):
        x = torch.zeros_like(b)
        torch.cuda.synchronize()
        if busy:
            for _ in range(200):
                load @ load
        rc, st = w.wilson_cg_solve_multi(x, U, b, 4, L, kappa, p, stream=side)
        assert rc == 0
        runs.append((host(x), [s["inner_iters"] for s in st]))
    for x, it in runs[1:]:
        assert it == runs[0][1] and np.array_equal(x, runs[0][0])
