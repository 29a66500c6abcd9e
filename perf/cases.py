"""Workloads of the Wilson operator library, as its users run them: one pass of
each goes through the public binding (paper_0710_2442_gb300.wilson) from the
fields a program holds to the result it goes on with.

Kinds of case:
  stateless  wilson_dslash / wilson_dslash_eo / wilson_dslash_eo_noalloc on
             canonical complex128 device fields: the simplest calls, made where
             an operator is applied once or twice to a field (a residual, a
             measurement, a force term with new links each time).
  handle     prepared links; a source is imported, the operator is applied
             ``apps`` times and the result exported: what an eigensolver, a
             polynomial filter or a smearing does.  The result goes on in the
             precision it was computed in (complex64 for F32 storage, 16-bit
             reals for F16 and BF16).
  solve      wilson_cg_solve(_multi), mixed precision, to a residual of 1e-12.
  batch      wilson_batch_solve of lattices of several sizes.

All inputs are seeded and made on the GPU: links exp(i eps H) projected to
SU(3) (eps = 0: Gaussian rows orthonormalised, a disordered field), Gaussian
sources, antiperiodic t; ``twist`` adds a boundary phase exp(i twist) in x.
"""
import math

import torch

from paper_0710_2442_gb300 import wilson as w

OPS = {"hop": w.WILSON_OP_HOP, "m": w.WILSON_OP_M, "schur": w.WILSON_OP_SCHUR, "schur_dag": w.WILSON_OP_SCHUR_DAG}
LINK_BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
SITE_BYTES = {"f64": 192, "f32": 96, "f16": 52, "bf16": 52}  # stored spinor, with the scale of the 16-bit formats


def listed():
    return [
        # a single small call, where launches and latency count (unit tests, small physics lattices)
        dict(name="eo_hop_f64_8x8x8x8", kind="stateless", entry="eo", op="hop", x=8, y=8, z=8, t=8, eps=0.0, twist=0.0),
        # the same for hosts that own the device memory, with a twisted boundary
        dict(name="noalloc_schur_f64_12x12x12x12", kind="stateless", entry="noalloc", op="schur_dag",
             x=12, y=12, z=12, t=12, eps=0.3, twist=0.4),
        # an ordinary residual: M on a full field
        dict(name="full_m_f64_16x16x16x32", kind="stateless", entry="full", op="m", x=16, y=16, z=16, t=32, eps=0.3, twist=0.0),
        # the largest stateless call
        dict(name="eo_schur_f64_32x32x32x64", kind="stateless", entry="eo", op="schur", x=32, y=32, z=32, t=64, eps=0.3,
             twist=0.0),
        # double-precision operator on prepared fields (an eigensolver's step)
        dict(name="handle_f64_schur_24x24x24x48", kind="handle", prec="f64", recon=18, op="schur", apps=2, nrhs=1,
             x=24, y=24, z=24, t=48, eps=0.3, twist=0.0),
        # single precision on the largest lattice
        dict(name="handle_f32_hop_32x32x32x64", kind="handle", prec="f32", recon=12, op="hop", apps=8, nrhs=1,
             x=32, y=32, z=32, t=64, eps=0.3, twist=0.0),
        # a small lattice with extents that divide nothing evenly, full links
        dict(name="handle_f32_m_10x14x6x18", kind="handle", prec="f32", recon=18, op="m", apps=4, nrhs=1,
             x=10, y=14, z=6, t=18, eps=0.0, twist=0.0),
        # the inner operator of the mixed-precision solvers on its own
        dict(name="handle_f16_schur_24x24x24x48", kind="handle", prec="f16", recon=12, op="schur", apps=4, nrhs=1,
             x=24, y=24, z=24, t=48, eps=0.3, twist=0.0),
        # twelve right-hand sides (spin x colour of a propagator) on one set of links
        dict(name="handle_f32_hop_12rhs_24x24x24x48", kind="handle", prec="f32", recon=12, op="hop", apps=4, nrhs=12,
             x=24, y=24, z=24, t=48, eps=0.3, twist=0.0),
        dict(name="handle_bf16_schur_12rhs_16x16x16x32", kind="handle", prec="bf16", recon=12, op="schur_dag", apps=4, nrhs=12,
             x=16, y=16, z=16, t=32, eps=0.3, twist=0.0),
        # a whole solve of an ordinary lattice
        dict(name="cg_f16_16x16x16x32", kind="solve", prec="f16", nrhs=1, kappa=0.135, x=16, y=16, z=16, t=32, eps=0.3, twist=0.0),
        # many lattices at once, small ones on chip, larger ones on their own loops
        dict(name="batch_f16_8_12_16", kind="batch", prec="f16", sizes="8x8x8x8*8,12x12x12x12*4,16x16x16x32*2", eps=0.3, kappa=0.13),
    ]


def _extents(rng, lo, hi):
    """Even extents >= 4 with a volume spread over the logarithm of [lo, hi]."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        d = [max(4, 2 * round(v ** 0.25 * math.exp(rng.uniform(-0.35, 0.35)) / 2)) for _ in range(3)]
        t = max(4, 2 * round(v / (d[0] * d[1] * d[2]) / 2))
        if t <= 128 and lo * 0.8 <= d[0] * d[1] * d[2] * t <= hi:
            return dict(x=d[0], y=d[1], z=d[2], t=t)


def draw(rng):
    big = 32 * 32 * 32 * 64
    kind = rng.choice(["stateless", "stateless", "handle", "handle", "handle", "multi", "solve", "batch"])
    eps = rng.choice([0.0, 0.2, 0.3, 0.4])
    twist = rng.choice([0.0, 0.0, round(rng.uniform(0.1, 3.0), 3)])
    if kind == "stateless":
        entry = rng.choice(["eo", "full", "noalloc"])
        op = rng.choice(["hop", "m"]) if entry == "full" else rng.choice(["hop", "schur", "schur_dag"])
        top = 2 * 18000 if entry == "noalloc" else big
        return dict(kind="stateless", entry=entry, op=op, eps=eps, twist=twist, **_extents(rng, 256, top))
    if kind in ("handle", "multi"):
        prec = rng.choice(["f32", "f16", "bf16"] if kind == "multi" else ["f64", "f32", "f16", "bf16"])
        op = rng.choice(["hop", "m", "schur", "schur_dag"])
        nrhs = rng.choice([2, 3, 4, 6, 8, 12]) if kind == "multi" else 1
        apps = rng.choice([1, 2]) if prec == "f64" else 2 * rng.choice([1, 2])
        recon = 12 if kind == "multi" else rng.choice([12, 18])
        return dict(kind="handle", prec=prec, recon=recon, op=op, apps=2 if op == "hop" else apps, nrhs=nrhs, eps=eps, twist=twist,
                    **_extents(rng, 256, big / nrhs))
    prec = rng.choice(["f16", "f32", "bf16"])
    kappa = round(rng.uniform(0.12, 0.13), 4)
    eps = rng.choice([0.2, 0.3, 0.4])
    if kind == "solve":
        return dict(kind="solve", prec=prec, nrhs=rng.choice([1, 1, 4, 12]), kappa=kappa, eps=eps, twist=twist,
                    **_extents(rng, 256, 8 ** 4 * 16))
    few = [_extents(rng, 256, 8 ** 4 * 8) for _ in range(rng.randint(2, 3))]
    return dict(kind="batch", prec=prec, kappa=kappa, eps=eps,
                sizes=",".join("%dx%dx%dx%d*%d" % (*d.values(), rng.randint(1, 4)) for d in few))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, k):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 64 + k)


def _gaussian(shape, gen):
    return torch.randn(*shape, 2, dtype=torch.float64, device="cuda", generator=gen).view(torch.complex128).squeeze(-1)


def _mul3(a, b):
    return sum(a[..., :, k, None] * b[..., None, k, :] for k in range(3))


def _links(V, eps, gen):
    """complex128 [V, 4, 3, 3] in SU(3)."""
    m = _gaussian((V * 4, 3, 3), gen)
    if eps > 0:
        # i eps H, H = (m + m^dag) / (2 sqrt 2) without its trace: components as of sum_a h_a lambda_a / 2
        h = (m + m.mH) * (eps / (2 * math.sqrt(2.0)))
        h -= torch.diag_embed((h.diagonal(dim1=-2, dim2=-1).sum(-1, keepdim=True) / 3).expand(-1, 3))
        h = 1j * h
        one = torch.eye(3, dtype=torch.complex128, device="cuda")
        m = one + h / 12
        for k in range(11, 0, -1):
            m = one + _mul3(h, m) / k
        del h
    r0, r1 = m[:, 0], m[:, 1]
    r0 = r0 / torch.linalg.vector_norm(r0, dim=1, keepdim=True)
    for _ in range(2):
        r1 = r1 - (r0.conj() * r1).sum(1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
    return torch.stack([r0, r1, torch.linalg.cross(r0, r1, dim=1).conj()], dim=1).reshape(V, 4, 3, 3)


def _dims(case):
    return tuple(case[k] for k in "xyzt")


def _phases(case):
    th = case.get("twist", 0.0)
    return (complex(math.cos(th), math.sin(th)) if th else 1.0, 1.0, 1.0, -1.0)


def _subset(case):
    """Sites of the input field: a full field for M (and the full hop), else one parity."""
    if case["kind"] in ("solve", "batch") or case["op"] == "m" or case.get("entry") == "full":
        return "full"
    return "half"


def _fields(case, seed):
    """(links, source) of one lattice, canonical complex128."""
    V = math.prod(_dims(case))
    n = V if _subset(case) == "full" else V // 2
    nrhs = case.get("nrhs", 1)
    shape = (n, 4, 3) if nrhs == 1 else (nrhs, n, 4, 3)
    return _links(V, case["eps"], _gen(seed, 0)), _gaussian(shape, _gen(seed, 1))


def _batch_cases(case):
    got = []
    for part in case["sizes"].split(","):
        size, count = part.split("*")
        x, y, z, t = (int(v) for v in size.split("x"))
        for _ in range(int(count)):
            k = len(got)
            # neighbouring kappas and roughnesses, as of an ensemble scan
            got.append(dict(kind="solve", x=x, y=y, z=z, t=t, eps=case["eps"] * (1 + 0.02 * (k % 5)),
                            kappa=case["kappa"] - 0.0005 * (k % 7), twist=0.0))
    return got


def _params(case):
    """The defaults of the inner precision with a residual of 1e-12: a propagator that enters a
    difference or a force has to be solved further than the default 1e-10."""
    p = w.solver_defaults(w.PREC[case["prec"]])
    p.tol = 1e-12
    return p


def prepare(case, seed):
    if case["kind"] == "batch":
        probs = []
        for k, c in enumerate(_batch_cases(case)):
            U, b = _fields(c, seed * 97 + k)
            probs.append(dict(L=w.lattice(_dims(c), _phases(c)), kappa=c["kappa"], gauge=U, b=b, x=torch.zeros_like(b)))
        return dict(case=case, probs=probs, params=_params(case))
    U, src = _fields(case, seed)
    L = w.lattice(_dims(case), _phases(case))
    s = dict(case=case, L=L, src=src, out=torch.zeros_like(src))
    if case["kind"] == "handle":
        prec = w.PREC[case["prec"]]
        s["gauge"] = w.Gauge(U, L, prec, case["recon"])
        full = _subset(case) == "full"
        to_other = case["op"] == "hop"  # the hop maps odd to even and back
        s["a"] = w.Spinor(L, w.WILSON_FULL if full else w.WILSON_EVEN, prec, case["nrhs"])
        s["b"] = w.Spinor(L, w.WILSON_FULL if full else w.WILSON_ODD if to_other else w.WILSON_EVEN, prec, case["nrhs"])
        return s
    s["U"] = U
    if case["kind"] == "solve":
        s["params"] = _params(case)
    return s


KAPPA = 0.13  # of the operator cases


def run(s):
    c = s["case"]
    if c["kind"] == "stateless":
        op = OPS[c["op"]]
        if c["entry"] == "full":
            w.wilson_dslash(s["out"], s["U"], s["src"], s["L"], KAPPA, op)
        elif c["entry"] == "eo":
            w.wilson_dslash_eo(s["out"], s["U"], s["src"], s["L"], 0, KAPPA, op)
        else:
            w.wilson_dslash_eo_noalloc(s["out"], s["U"], s["src"], s["L"], 0, KAPPA, op)
        return s["out"]
    if c["kind"] == "handle":
        a, b = s["a"], s["b"]
        a.load(s["src"])
        for _ in range(c["apps"]):
            w.wilson_dslash_h(b, s["gauge"], a, KAPPA, OPS[c["op"]])
            a, b = b, a
        a.store(s["out"])
        if c["prec"] == "f64":
            return s["out"]
        if c["prec"] == "f32":
            return s["out"].to(torch.complex64)
        return torch.view_as_real(s["out"]).to(torch.float16 if c["prec"] == "f16" else torch.bfloat16)
    if c["kind"] == "solve":
        if c["nrhs"] == 1:
            w.wilson_cg_solve(s["out"], s["U"], s["src"], s["L"], c["kappa"], s["params"])
        else:
            w.wilson_cg_solve_multi(s["out"], s["U"], s["src"], c["nrhs"], s["L"], c["kappa"], s["params"])
        return s["out"]
    w.wilson_batch_solve(s["probs"], s["params"])
    return [p["x"] for p in s["probs"]]


# ---------------------------------------------------------------------------
# work: every application is a call that reads its links and fields and
# writes its result; 1320 flops per hopping term and output site
# ---------------------------------------------------------------------------
def work(case):
    if case["kind"] == "batch":
        parts = [work(dict(c, nrhs=1)) for c in _batch_cases(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    V = math.prod(_dims(case))
    if case["kind"] == "solve":
        # fields in and out once; about 100 iterations of four half-lattice hops
        return {"bytes": V * (576 + 2 * 192 * case["nrhs"]), "flops": 100 * 4 * 1320 * (V // 2) * case["nrhs"]}
    n = V if _subset(case) == "full" else V // 2
    hops = 2 if case["op"].startswith("schur") else 1
    if case["kind"] == "stateless":
        return {"bytes": V * 576 + 2 * 192 * n, "flops": 1320 * hops * n}
    one = V * 4 * case["recon"] * LINK_BYTES[case["prec"]] + 2 * SITE_BYTES[case["prec"]] * n * case["nrhs"]
    back = 192 + 192 * LINK_BYTES[case["prec"]] // 8  # export, and the result in its own precision
    return {"bytes": case["apps"] * one + (192 + (back if case["prec"] != "f64" else 192)) * n * case["nrhs"],
            "flops": case["apps"] * 1320 * hops * n * case["nrhs"]}


# ---------------------------------------------------------------------------
# the same in 64 bits, from the operator's definition
#   D psi(x) = sum_mu (1 - g_mu) U_mu(x) psi(x+mu) + (1 + g_mu) U_mu(x-mu)^dag psi(x-mu)
# with the DeGrand-Rossi matrices: (g_mu psi)_s = GAMMA[mu][s][1] psi_{GAMMA[mu][s][0]}
# ---------------------------------------------------------------------------
GAMMA = (((3, 1j), (2, 1j), (1, -1j), (0, -1j)), ((3, -1), (2, 1), (1, 1), (0, -1)),
         ((2, 1j), (3, -1j), (0, -1j), (1, 1j)), ((2, 1), (3, 1), (0, 1), (1, 1)))


def _gamma(mu, psi):
    return torch.stack([c * psi[..., s, :] for s, c in GAMMA[mu]], dim=-2)


def _g5(psi):
    return torch.cat([psi[..., :2, :], -psi[..., 2:, :]], dim=-2)


def _shift(f, mu, step, phase):
    """f at x + step*mu on [t, z, y, x, ...] with the boundary phase where it wraps."""
    dim = 3 - mu
    g = torch.roll(f, -step, dims=dim)
    if phase != 1:
        edge = g.narrow(dim, g.shape[dim] - 1 if step > 0 else 0, 1)
        edge *= phase if step > 0 else complex(phase).conjugate()
    return g


def _colour(u, psi, adj):
    """u psi (or u^dag psi) on the colours of every spin."""
    return sum((u[..., k, :].conj() if adj else u[..., :, k])[..., None, :] * psi[..., :, k, None] for k in range(3))


def _hop(U, psi, dims, phases):
    shape = tuple(reversed(dims))
    p = psi.reshape(*shape, 4, 3)
    u = U.reshape(*shape, 4, 3, 3)
    out = torch.zeros_like(p)
    for mu in range(4):
        f = _colour(u[..., mu, :, :], _shift(p, mu, 1, phases[mu]), False)
        out += f - _gamma(mu, f)
        f = _shift(_colour(u[..., mu, :, :], p, True), mu, -1, phases[mu])
        out += f + _gamma(mu, f)
    return out.reshape(psi.shape)


def _parity(dims):
    ax = [torch.arange(d, device="cuda") for d in reversed(dims)]
    t, z, y, x = torch.meshgrid(*ax, indexing="ij")
    return ((x + y + z + t) & 1).reshape(-1)


def _half_hop(U, half, p, dims, phases, par):
    """D_{p,1-p}: from parity 1 - p to parity p."""
    full = torch.zeros((par.numel(), 4, 3), dtype=torch.complex128, device="cuda")
    full[par == 1 - p] = half
    return _hop(U, full, dims, phases)[par == p]


def _exact_op(case, U, psi, parity, par):
    """(result, its parity) of one application on one field (parity None: a full field)."""
    dims, ph, op = _dims(case), _phases(case), case["op"]
    if op == "m":
        return psi - KAPPA * _hop(U, psi, dims, ph), parity
    if op == "hop":
        if parity is None:
            return _hop(U, psi, dims, ph), None
        return _half_hop(U, psi, 1 - parity, dims, ph, par), 1 - parity
    v = _g5(psi) if op == "schur_dag" else psi
    v = v - KAPPA ** 2 * _half_hop(U, _half_hop(U, v, 1 - parity, dims, ph, par), parity, dims, ph, par)
    return (_g5(v) if op == "schur_dag" else v), parity


def _exact_solve(case, U, b):
    """M x = b by conjugate gradients on the normal equations, to about 1e-14."""
    dims, ph, k = _dims(case), _phases(case), case["kappa"]
    mul = lambda v: v - k * _hop(U, v, dims, ph)  # noqa: E731
    adj = lambda v: _g5(mul(_g5(v)))  # noqa: E731
    x = torch.zeros_like(b)
    for _ in range(3):  # the residual is taken anew twice
        s = b - mul(x)
        r = adj(s)
        p, gam = r, torch.linalg.vector_norm(r).item() ** 2
        stop = max(1e-14 * torch.linalg.vector_norm(b).item(), 1e-8 * torch.linalg.vector_norm(s).item())
        for _ in range(2000):
            if torch.linalg.vector_norm(s).item() <= stop or gam == 0.0:
                break
            q = mul(p)
            a = gam / torch.linalg.vector_norm(q).item() ** 2
            x, s = x + a * p, s - a * q
            r = adj(s)
            new = torch.linalg.vector_norm(r).item() ** 2
            p, gam = r + (new / gam) * p, new
    return x


def exact(case, seed):
    if case["kind"] == "batch":
        cases = _batch_cases(case)
        if sum(math.prod(_dims(c)) + 20000 for c in cases) > 800_000:
            return None
        return [_exact_solve(c, *_fields(c, seed * 97 + k)) for k, c in enumerate(cases)]
    U, src = _fields(case, seed)
    nrhs = case.get("nrhs", 1)
    if case["kind"] == "solve":
        if math.prod(_dims(case)) * nrhs > 300_000 or nrhs > 4:
            return None
        got = [_exact_solve(case, U, b) for b in (src if nrhs > 1 else [src])]
        return torch.stack(got) if nrhs > 1 else got[0]
    par = _parity(_dims(case))
    got = []
    for psi in src if nrhs > 1 else [src]:
        # the stateless calls return the even half; handles start from an even field
        parity = None if _subset(case) == "full" else 1 if case["kind"] == "stateless" and case["op"] == "hop" else 0
        for _ in range(case.get("apps", 1)):
            psi, parity = _exact_op(case, U, psi, parity, par)
        got.append(psi)
    v = torch.stack(got) if nrhs > 1 else got[0]
    return torch.view_as_real(v) if case.get("prec") in ("f16", "bf16") else v
