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

from conftest import assert_parity, parity_merge, parity_split
from gpu_helpers import dev, empty_like_dev, handle_hop, host
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
@pytest.mark.parametrize("case", ["mean link", "all entries", "third row", "third row of 4"])
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
    elif case == "third row of 4":  # its limb is 2^31
        recon = 12
        U[..., 0, :] = 1.0 + 1.0j
        U[..., 1, :] = [1.0 - 1.0j, -1.0 + 1.0j, 1.0 - 1.0j]
    else:
        recon = 12
        U[..., 0, :] = 0.95 + 0.95j
        U[..., 1, :] = (0.95 - 0.95j) * np.array([1.0, -1.0, 1.0])
    args = (w, U, src, dims, PHASES, w.WILSON_F64, recon, 1, 0, w.WILSON_OP_HOP)
    got = handle_hop(*args)
    monkeypatch.setenv("WILSON_HOP_VARIANT", "0")
    assert_parity(got, handle_hop(*args), TOL)


def hop_moduli(U, a, dims):
    """Each component's sum of the moduli of its terms: a = (|re|, |im|) of a full field [V, 4, 3],
    as [2, V, 4, 3]; boundary phases +-1.  Partner spins: 3 - s in x and y, s ^ 2 in z and t, with a factor i in x and z."""
    L = tuple(reversed(dims))
    u = np.stack([np.abs(U.real), np.abs(U.imag)]).reshape(2, *L, 4, 3, 3)
    a = a.reshape(2, *L, 4, 3)
    s = np.zeros_like(a)
    for mu in range(4):
        axis = 3 - mu  # of the lattice: t, z, y, x
        h = a + (a[:, ..., [3, 2, 1, 0], :] if mu < 2 else a[:, ..., [2, 3, 0, 1], :])[::-1 if mu in (0, 2) else 1]
        f = np.roll(h, -1, axis=axis + 1)
        m = u[..., mu, :, :]
        for re, im, links in ((f[0], f[1], m), (h[0], h[1], np.swapaxes(m, -1, -2))):
            x = np.stack([np.einsum("...ik,...sk->...si", links[0], re) + np.einsum("...ik,...sk->...si", links[1], im),
                          np.einsum("...ik,...sk->...si", links[0], im) + np.einsum("...ik,...sk->...si", links[1], re)])
            s += x if links is m else np.roll(x, 1, axis=axis + 1)
    return s.reshape(2, -1, 4, 3)


def graded_field(kind, V, seed):
    rng = np.random.default_rng(seed)
    psi = inputs.gaussian_spinor(V, seed=seed)
    if kind == "colour":
        return psi * np.array([1.0, 1e-4, 1e-8])
    if kind == "spin":
        return psi * np.array([1e-10, 1.0, 1e-2, 1e-6])[:, None]
    if kind == "imaginary":
        return psi.real + 1e-9j * psi.imag
    if kind == "component":
        return psi.real * 2.0 ** -rng.integers(0, 40, psi.shape) + 1j * psi.imag * 2.0 ** -rng.integers(0, 40, psi.shape)
    if kind == "one spin":
        psi[:, [0, 1, 3]] = 0
        return psi
    if kind == "site":
        return psi * 2.0 ** -rng.integers(0, 40, V)[:, None, None]
    return psi


def links_of(kind, dims):
    if kind == "abelian":
        U = inputs.gauge_field(dims, "unit")
        a = np.random.default_rng(421).standard_normal(U.shape[:-1])
        a[..., 2] = -a[..., 0] - a[..., 1]
        return U * np.exp(1j * a)[..., None]
    if kind == "slice of zeros":
        U = inputs.gauge_field(dims, "random", seed=422).reshape(-1, 4, 3, 3)
        U[: V3(dims), 3] = 0
        return U
    return inputs.gauge_field(dims, "weak", eps=1e-6, seed=423) if kind == "near unit" else inputs.gauge_field(dims, kind, seed=424)


def V3(dims):
    return dims[0] * dims[1] * dims[2]


@pytest.mark.parametrize("dims", [(4, 4, 4, 6), (14, 14, 12, 18)])
@pytest.mark.parametrize("links", ["unit", "abelian", "near unit", "random", "slice of zeros"])
@pytest.mark.parametrize("field", ["gaussian", "colour", "spin", "imaginary", "component", "one spin", "site"])
def test_component_accuracy(w, oracle_mod, dims, links, field):
    """Every component as accurate as FP64 arithmetic leaves it, whatever the others of its site are: a component of the
    hop is 13 roundings (1 projection, 6 products, 7 sums) of a sum of terms, so two FP64 evaluations
    differ by at most 28 units 2^-53 of its terms' moduli; M adds 2 more; a Schur operator applies it twice.  Stateless and on
    handles; one lattice on each of the two kernels."""
    V, kappa = inputs.volume(dims), 0.13
    U = links_of(links, dims)
    psi = graded_field(field, V, 425)
    mod = np.stack([np.abs(psi.real), np.abs(psi.imag)])
    s1 = hop_moduli(U, mod, dims)
    unit = 2.0 ** -53
    L = w.lattice(dims)

    def check(got, want, bound, what):
        err = np.stack([np.abs((got - want).real), np.abs((got - want).imag)])
        assert np.all(err <= bound), (what, float(np.max(err / np.maximum(bound, 1e-300))))

    out = empty_like_dev(psi)
    w.wilson_dslash(out, dev(U), dev(psi), L, kappa, w.WILSON_OP_M)
    want = oracle_mod.wilson_m(U, psi, dims, kappa)
    check(host(out), want, 32 * unit * (kappa * s1 + mod), "m")
    got = handle_hop(w, U, psi, dims, inputs.DEFAULT_PHASES, w.WILSON_F64, 18, w.WILSON_FULL, w.WILSON_FULL, w.WILSON_OP_M, kappa)
    check(got, want, 32 * unit * (kappa * s1 + mod), "m on handles")

    even, odd = parity_split(psi, dims)
    s2 = hop_moduli(U, hop_moduli(U, np.stack([np.abs(parity_merge(even, 0 * odd, dims).real),
                                               np.abs(parity_merge(even, 0 * odd, dims).imag)]), dims), dims)
    bound = np.stack([parity_split(s2[z], dims)[0] for z in (0, 1)]) * kappa ** 2 * 64 * unit
    bound += 4 * unit * np.stack([np.abs(even.real), np.abs(even.imag)])
    want = oracle_mod.schur(U, even, dims, kappa, 0)
    out = empty_like_dev(even)
    w.wilson_dslash_eo(out, dev(U), dev(even), L, 0, kappa, w.WILSON_OP_SCHUR)
    check(host(out), want, bound, "schur")
    got = handle_hop(w, U, even, dims, inputs.DEFAULT_PHASES, w.WILSON_F64, 18, 0, 0, w.WILSON_OP_SCHUR, kappa)
    check(got, want, bound, "schur on handles")


def test_captured_handle_operators(w, oracle_mod):
    """Under stream capture an F64 operator takes no workspace (a captured call allocates
    nothing), so that its hops of a large lattice run on the other kernel: the same operator."""
    import torch
    dims = (14, 14, 12, 18)
    L = w.lattice(dims, PHASES)
    U = inputs.gauge_field(dims, "random", seed=435)
    src = inputs.gaussian_spinor(inputs.volume(dims) // 2, seed=436)
    g = w.Gauge(U, L, w.WILSON_F64, 18)
    a, b, c = (w.Spinor(L, w.WILSON_EVEN, w.WILSON_F64) for _ in range(3))
    d = w.Spinor(L, w.WILSON_ODD, w.WILSON_F64)
    a.load(dev(src))
    w.wilson_dslash_h(b, g, a, 0.13, w.WILSON_OP_SCHUR)  # the handle's intermediate field
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        w.wilson_dslash_h(c, g, a, 0.13, w.WILSON_OP_SCHUR)
        w.wilson_dslash_h(d, g, a, 0.0, w.WILSON_OP_HOP)
    got = []
    for _ in range(2):
        graph.replay()
        got.append([np.empty_like(src), np.empty_like(src)])
        for f, x in zip((c, d), got[-1]):
            out = empty_like_dev(src)
            f.store(out)
            x[:] = host(out)
    for x, y in zip(*got):
        assert np.array_equal(x, y)
    assert_parity(got[0][0], oracle_mod.schur(U, src, dims, 0.13, 0, False, PHASES), TOL)
    assert_parity(got[0][1], oracle_mod.dslash_eo(U, src, dims, 1, PHASES), TOL)


@pytest.mark.parametrize("dims", [(4, 4, 4, 6), (14, 14, 12, 18)])
@pytest.mark.parametrize("part", [40, 20, 6, 1])
def test_links_out_of_range_in_part(w, oracle_mod, dims, part):
    """Every part-th link twice as large: a few are done over site by site, from a twelfth of them on
    the handle runs on the FP64 stencil."""
    U = inputs.gauge_field(dims, "random", seed=437)
    U.reshape(-1, 3, 3)[::part] *= 2.0
    src = inputs.gaussian_spinor(inputs.volume(dims) // 2, seed=438)
    got = handle_hop(w, U, src, dims, PHASES, w.WILSON_F64, 18, 0, 0, w.WILSON_OP_SCHUR, 0.13)
    assert_parity(got, oracle_mod.schur(U, src, dims, 0.13, 0, False, PHASES), TOL)


@pytest.mark.parametrize("inner", ["f64", "f32"])
def test_solve_with_links_out_of_range(w, oracle_mod, inner):
    """Links twice as large and half of kappa are the same matrix."""
    dims, kappa = (4, 4, 4, 8), 0.0675
    U = 2.0 * inputs.gauge_field(dims, "weak", eps=0.3, seed=439)
    b = inputs.gaussian_spinor(dims, seed=440)
    p = w.solver_defaults(w.PREC[inner])
    p.recon = 18
    x = dev(np.zeros_like(b))
    st = w.wilson_cg_solve(x, dev(U), dev(b), w.lattice(dims), kappa, p)
    assert st["rc"] == 0
    r = b - oracle_mod.wilson_m(U, host(x), dims, kappa)
    assert np.linalg.norm(r) <= 1.1e-10 * np.linalg.norm(b)


def test_reducing_hop_does_sites_over(w, oracle_mod):
    """FP64 CG on 80000 sites a parity, three turns of each block of the reducing hop, with a link in 500 out of
    range: the sites that are done over are in its sums (a wrong |Mhat p|^2 ends in
    another iteration count or none: the count is that of the FP64 stencil, within one)."""
    dims, kappa = (20, 20, 20, 20), 0.11
    U = inputs.gauge_field(dims, "weak", eps=0.3, seed=441)
    U.reshape(-1, 3, 3)[::500] *= 2.0
    b = inputs.gaussian_spinor(dims, seed=442)
    p = w.solver_defaults(w.WILSON_F64)
    p.recon = 18
    x = dev(np.zeros_like(b))
    st = w.wilson_cg_solve(x, dev(U), dev(b), w.lattice(dims), kappa, p)
    assert st["rc"] == 0
    r = b - oracle_mod.wilson_m(U, host(x), dims, kappa)
    assert np.linalg.norm(r) <= 1.1e-10 * np.linalg.norm(b)
    stencil = 2.0 * U  # all of them out of range: the FP64 stencil, the same matrix with half of kappa
    y = dev(np.zeros_like(b))
    ref = w.wilson_cg_solve(y, dev(stencil), dev(b), w.lattice(dims), kappa / 2, p)
    assert ref["rc"] == 0 and abs(ref["inner_iters"] - st["inner_iters"]) <= 1
