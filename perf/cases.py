"""Performance cases of the clover-Wilson library: what its users have it do, over the sizes they use.

A case names one call sequence through the torch-facing API (``CloverWilson`` and
``CloverPseudofermionAction``), a lattice X x Y x Z x T, a precision and a number of right-hand sides:

* ``apply``  -- one operator (hopping term, Mhat, Mhat^dag Mhat, clover, inverse clover) on fields of
  the canonical layout, as a measurement or an outer solver written by the user calls it;
* ``solve``  -- Mhat^dag Mhat x = b to a true relative residual of 1e-8: plain FP64, or FP32 / FP16
  iterations with FP64 reliable updates;
* ``ingest`` -- a new gauge configuration: links packed, clover term built and inverted, its
  log-determinant, and the first operator application on it;
* ``force``  -- the molecular-dynamics force of known solutions, with the clover determinant term;
* ``action`` -- the differentiable pseudofermion action, forward and backward through torch.autograd;
* ``rstep``  -- one R-algorithm step on links and momenta, and the plaquette of the new links.

The inputs follow the repository's synthetic recipe (links exp(i eps H) near unity, projected to SU(3);
complex Gaussian sources; kappa 0.12, c_sw 1), drawn here on the GPU.  ``exact`` restates every
operator in plain torch, complex128 on the full lattice, and takes its gradients from torch.autograd.
"""

import math

import torch

from paper_0910_0262_gb300 import qcd
from paper_0910_0262_gb300.qcd import CloverPseudofermionAction, CloverWilson

KAPPA, CSW, T_BC = 0.12, 1.0, -1.0
TOL = 1e-8         # true relative residual of the solves
BETA, DTAU = 5.6, 0.02

OPS = {"dslash_eo": qcd.QCD_OP_DSLASH_EO, "dslash_oe": qcd.QCD_OP_DSLASH_OE, "mhat": qcd.QCD_OP_MHAT,
       "mdagm": qcd.QCD_OP_MDAGM, "clover": qcd.QCD_OP_CLOVER, "clover_inv": qcd.QCD_OP_CLOVER_INV}


def _case(kind, dims, name=None, **kw):
    c = {} if name is None else {"name": name}
    c.update(kind=kind, X=dims[0], Y=dims[1], Z=dims[2], T=dims[3], **kw)
    return c


def listed():
    return [
        # the smallest call: one operator on a test lattice, where launches and latency count
        _case("apply", (4, 4, 4, 8), "apply_mhat_fp64_4x4x4x8", op="mhat", dagger=False, prec=64, nrhs=1, recon12=False),
        # an outer solver's operator on an ordinary lattice, FP32 storage, reconstructed links
        _case("apply", (16, 16, 16, 16), "apply_mdagm_fp32_16x16x16x16", op="mdagm", dagger=False, prec=32, nrhs=1,
              recon12=True),
        # the daggered operator in FP64 on a ragged lattice, an odd number of fields
        _case("apply", (22, 18, 14, 26), "apply_mhatdag_fp64_22x18x14x26_rhs3", op="mhat", dagger=True, prec=64, nrhs=3,
              recon12=False),
        # the largest call: a batch of fields on a production lattice in FP16 storage
        _case("apply", (32, 32, 32, 64), "apply_mdagm_fp16_32x32x32x64_rhs8", op="mdagm", dagger=False, prec=16, nrhs=8,
              recon12=True),
        # the solve of a molecular-dynamics step on the smallest workload lattice
        _case("solve", (8, 8, 16, 16), "solve_fp32_8x8x16x16", prec=32, nrhs=1, recon12=True),
        # the same on the ordinary workload lattice
        _case("solve", (16, 16, 16, 16), "solve_fp32_16x16x16x16", prec=32, nrhs=1, recon12=True),
        # plain FP64 conjugate gradients (a reference or ill-conditioned solve), ragged lattice
        _case("solve", (10, 12, 14, 18), "solve_fp64_10x12x14x18_rhs2", prec=64, nrhs=2, recon12=False),
        # a propagator: a batch of sources on a large lattice, FP16 inner iterations
        _case("solve", (24, 24, 24, 48), "solve_fp16_24x24x24x48_rhs8", prec=16, nrhs=8, recon12=True),
        # a new configuration of a stream of configurations
        _case("ingest", (24, 24, 24, 32), "ingest_24x24x24x32", recon12=True),
        # the force evaluation of a molecular-dynamics integrator that has its solutions
        _case("force", (16, 16, 16, 16), "force_det_16x16x16x16", nrhs=1, det=True),
        # a training step through the differentiable action: forward, and gradients of links and field
        _case("action", (12, 12, 12, 20), "action_fwd_bwd_12x12x12x20", prec=32, nrhs=1),
        # one step of the R-algorithm trajectory
        _case("rstep", (16, 16, 16, 16), "rstep_16x16x16x16", prec=32, nrhs=1),
    ]


def _dims(rng, vmax):
    """Even extents, the volume spread over its logarithm between 512 and vmax."""
    v = math.exp(rng.uniform(math.log(512.0), math.log(vmax)))
    side = v ** 0.25
    d = [max(4, min(48, 2 * round(0.5 * side * math.exp(rng.uniform(-0.35, 0.35))))) for _ in range(4)]
    d[3] = max(4, min(64, 2 * round(0.5 * v / (d[0] * d[1] * d[2]))))
    while d[0] * d[1] * d[2] * d[3] > vmax:
        k = max(range(4), key=lambda j: d[j])
        d[k] -= 2
    return tuple(d)


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "solve", "solve", "solve", "ingest", "force", "action", "rstep"])
    prec = rng.choice([64, 32, 16])
    nrhs = rng.choice([1, 1, 1, 2, 3, 4, 5, 8])
    recon12 = rng.random() < 0.6
    if kind == "apply":
        op = rng.choice(["mhat", "mdagm", "mhat", "mdagm", "dslash_eo", "dslash_oe", "clover", "clover_inv"])
        dims = _dims(rng, 2.0e6 / (2 if nrhs > 2 else 1))
        return _case(kind, dims, op=op, dagger=rng.random() < 0.4, prec=prec, nrhs=nrhs, recon12=recon12)
    if kind == "solve":
        dims = _dims(rng, (4.0e5 if prec == 64 else 1.6e6) / nrhs)
        return _case(kind, dims, prec=prec, nrhs=nrhs, recon12=recon12)
    if kind == "ingest":
        return _case(kind, _dims(rng, 6.0e5), recon12=recon12)
    if kind == "force":
        return _case(kind, _dims(rng, 3.0e5), nrhs=min(nrhs, 4), det=rng.random() < 0.5)
    if kind == "action":
        return _case(kind, _dims(rng, 1.6e5), prec=rng.choice([64, 32]), nrhs=min(nrhs, 2))
    return _case("rstep", _dims(rng, 1.6e5), prec=32, nrhs=min(nrhs, 2))


# ------------------------------------------------------------------------------------------ inputs ----
def _shape(case):
    return case["T"], case["Z"], case["Y"], case["X"]


def _volume(case):
    return case["X"] * case["Y"] * case["Z"] * case["T"]


def _hermitian(gen, n):
    """sum_a h_a lambda_a / 2 for h_a ~ N(0, 1): n traceless Hermitian 3x3 matrices."""
    h = 0.5 * torch.randn(8, n, generator=gen, device="cuda", dtype=torch.float64)
    d8 = h[7] / math.sqrt(3.0)
    z = torch.zeros_like(d8)
    c = torch.complex
    m = [c(h[2] + d8, z), c(h[0], -h[1]), c(h[3], -h[4]),
         c(h[0], h[1]), c(d8 - h[2], z), c(h[5], -h[6]),
         c(h[3], h[4]), c(h[5], h[6]), c(-2 * d8, z)]
    return torch.stack(m, -1).reshape(n, 3, 3)


def _project(u):
    """SU(3): rows 0, 1 orthonormalised, row 2 = conj(row 0 x row 1)."""
    r0 = u[..., 0, :]
    r0 = r0 / r0.abs().square().sum(-1, keepdim=True).sqrt()
    r1 = u[..., 1, :]
    r1 = r1 - (r0.conj() * r1).sum(-1, keepdim=True) * r0
    r1 = r1 / r1.abs().square().sum(-1, keepdim=True).sqrt()
    r2 = torch.linalg.cross(r0, r1, dim=-1).conj()
    return torch.stack([r0, r1, r2], -2)


def _links(case, gen):
    """Links exp(i eps H), by their series to fifth order and projected to SU(3)."""
    n = _volume(case) * 4
    eps = 0.2 if _volume(case) <= 70000 else 0.15
    out = torch.empty(n, 3, 3, dtype=torch.complex128, device="cuda")
    step = 1 << 21
    for k in range(0, n, step):
        m = min(step, n - k)
        a = 1j * eps * _hermitian(gen, m)
        u = torch.eye(3, dtype=a.dtype, device=a.device).expand_as(a)
        for j in range(5, 0, -1):
            u = torch.eye(3, dtype=a.dtype, device=a.device) + (a @ u) / j
        out[k:k + m] = _project(u)
    return out.reshape(_shape(case) + (4, 3, 3))


def _fields(case, gen, n):
    vh = _volume(case) // 2
    return torch.view_as_complex(torch.randn(n, vh, 4, 3, 2, generator=gen, device="cuda", dtype=torch.float64))


def _inputs(case, seed):
    """(links, fields): the numbers of a case, the same for prepare and exact."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    U = _links(case, gen)
    v = {"links": U}
    if case["kind"] in ("ingest", "apply", "solve", "force", "action", "rstep"):
        v["field"] = _fields(case, gen, case.get("nrhs", 1))
    if case["kind"] == "rstep":
        h = _hermitian(gen, _volume(case) * 4)
        v["momenta"] = (1j * h).reshape(U.shape)
    return v


def prepare(case, seed):
    v = _inputs(case, seed)
    op = CloverWilson((case["X"], case["Y"], case["Z"], case["T"]), T_BC)
    s = {"case": case, "op": op, **v}
    kind = case["kind"]
    if kind in ("apply", "solve", "force", "rstep"):
        # the configuration a program has loaded before these calls
        op.load_gauge(v["links"], recon12=case.get("recon12", True))
        op.clover_build(KAPPA, CSW)
    if kind not in ("ingest", "rstep", "action"):
        del s["links"]
    return s


def run(state):
    case, op = state["case"], state["op"]
    kind = case["kind"]
    if kind == "apply":
        return op.dslash(state["field"], OPS[case["op"]], dagger=case["dagger"], precision=case["prec"])
    if kind == "solve":
        x, _, _ = op.cg_solve(state["field"], tol=TOL, inner_prec=case["prec"])
        return x
    if kind == "ingest":
        op.load_gauge(state["links"], recon12=case["recon12"])
        op.clover_build(KAPPA, CSW)
        even, odd = op.clover_logdet()
        return {"mhat": op.dslash(state["field"], OPS["mhat"]), "logdet": [even, odd]}
    if kind == "force":
        F, _ = op.fermion_force(state["field"], input_is_solution=True, clover_det=case["det"])
        return F
    if kind == "action":
        U = state["links"].detach().requires_grad_(True)
        phi = state["field"].detach().requires_grad_(True)
        S = CloverPseudofermionAction.apply(U, phi, op, KAPPA, CSW, {"tol": TOL, "inner_prec": case["prec"]})
        gU, gphi = torch.autograd.grad(S, (U, phi))
        return {"S": S.detach(), "gU": gU, "gphi": gphi}
    U, P = state["links"].clone(), state["momenta"].clone()
    op.r_step(U, P, state["field"], DTAU, BETA, clover_det=True, tol=TOL, inner_prec=case["prec"])
    return {"U": U, "P": P, "plaquette": op.plaquette()}


# -------------------------------------------------------------------------------------------- work ----
def _hop_flops(vh, nrhs):
    return vh * nrhs * (1320.0 + 504.0)


def work(case):
    """Bytes and flops a pass cannot do without: inputs and outputs once (canonical complex128 fields), the
    links and clover blocks of the precision once; the conventional flops of the operators.  A solve is
    counted with 60 iterations, what these inputs take to 1e-8."""
    V = _volume(case)
    vh = V / 2.0
    nrhs = case.get("nrhs", 1)
    field = vh * 12 * 16.0 * nrhs
    links64, clover64 = V * 4 * 144.0, V * 72 * 8.0
    kind = case["kind"]
    if kind == "apply":
        b = case["prec"] / 8.0
        links = V * 4 * (12 if case["recon12"] and case["prec"] < 64 else 18) * b
        clover = V * 72 * b / 2  # one parity's blocks
        op = case["op"]
        if op in ("clover", "clover_inv"):
            return {"bytes": 2 * field + clover, "flops": vh * nrhs * 504.0}
        if op.startswith("dslash"):
            return {"bytes": 2 * field + links, "flops": vh * nrhs * 1320.0}
        hops = 2 if op == "mhat" else 4
        return {"bytes": 2 * field + links + 2 * clover, "flops": hops * _hop_flops(vh, nrhs)}
    if kind == "solve":
        return {"bytes": 2 * field + links64 + clover64, "flops": 60 * 4 * _hop_flops(vh, nrhs)}
    if kind == "ingest":
        # links in three precisions; A and its inverse on both parities in three precisions
        return {"bytes": links64 + V * 4 * 12 * 6.0 + links64 + 2 * V * 72 * 14.0 + 2 * field,
                "flops": V * (6 * 10 * 198.0 + 2000.0) + 2 * _hop_flops(vh, 1)}
    force = V * (6 * 20 * 198.0 + 4 * nrhs * 744.0 + 4 * 274.0) + 3 * _hop_flops(vh, nrhs)
    if kind == "force":
        return {"bytes": field + 2 * links64 + clover64, "flops": force}
    build = V * (6 * 10 * 198.0 + 2000.0)
    solve = 60 * 4 * _hop_flops(vh, nrhs)
    if kind == "action":
        return {"bytes": 2 * field + 2 * links64, "flops": solve + force + 2 * build}
    return {"bytes": field + 4 * links64, "flops": solve + force + 2 * build + V * 4 * (13 + 20) * 198.0}


# --------------------------------------------------------------------------------------- tolerance ----
def tolerance(case):
    """About four times the differences seen against ``exact``: FP64 operators 2e-16 (their sums in another
    order 5e-16), FP32 1.4e-7, FP16 storage 5.2e-4; forces 5e-16.  The solves stop at a relative residual of
    1e-8, so two correct ones differ by that times the operator's conditioning: solutions 8e-8, the
    gradients of the action 1.8e-7, the momenta of a step 1.6e-9."""
    kind = case["kind"]
    if kind == "apply":
        rel = {64: 2e-15, 32: 6e-7, 16: 2e-3}[case["prec"]]
    elif kind in ("ingest", "force"):
        rel = 2e-15
    else:
        rel = {"solve": 3.2e-7, "action": 7.2e-7, "rstep": 6.4e-9}[kind]
    return {"rel": rel, "max": 40 * rel}


# ------------------------------------------------------------------- plain torch, complex128, exact ----
# (g_mu psi)_s = COEF[mu][s] psi_{PERM[mu][s]} in the DeGrand-Rossi basis
_I = 1j
_PERM = [[3, 2, 1, 0], [3, 2, 1, 0], [2, 3, 0, 1], [2, 3, 0, 1]]
_COEF = [[_I, _I, -_I, -_I], [-1, 1, 1, -1], [_I, -_I, -_I, _I], [1, 1, 1, 1]]
_PLANES = [(m, n) for m in range(4) for n in range(m + 1, 4)]


def _gamma(mu):
    g = torch.zeros(4, 4, dtype=torch.complex128, device="cuda")
    for s in range(4):
        g[s, _PERM[mu][s]] = _COEF[mu][s]
    return g


def _dag(m):
    return m.transpose(-1, -2).conj()


def _at(f, mu, n):
    """f(x + n mu) of a site field [T, Z, Y, X, ...]."""
    return torch.roll(f, -n, 3 - mu)


def _leaves(U, mu, nu):
    m, n = U[..., mu, :, :], U[..., nu, :, :]
    n_xm, m_xn = _at(n, mu, 1), _at(m, nu, 1)                # U_nu(x+mu), U_mu(x+nu)
    m_bm, n_bm = _at(m, mu, -1), _at(n, mu, -1)              # at x-mu
    m_bn, n_bn = _at(m, nu, -1), _at(n, nu, -1)              # at x-nu
    q = m @ n_xm @ _dag(m_xn) @ _dag(n)
    q = q + n @ _dag(_at(m_xn, mu, -1)) @ _dag(n_bm) @ m_bm
    q = q + _dag(m_bm) @ _dag(_at(n_bm, nu, -1)) @ _at(m_bm, nu, -1) @ n_bn
    return q + _dag(n_bn) @ m_bn @ _at(n_xm, nu, -1) @ _dag(m)


def _clover(U):
    """The clover term's two chiral 6x6 blocks [T, Z, Y, X, 2, 6, 6]."""
    lat = U.shape[:4]
    one = torch.eye(3, dtype=U.dtype, device=U.device)
    blocks = [torch.eye(6, dtype=U.dtype, device=U.device).expand(lat + (6, 6)) for _ in range(2)]
    for mu, nu in _PLANES:
        Q = _leaves(U, mu, nu)
        F = (Q - _dag(Q)) / 8j
        F = F - F.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None] * one / 3
        gm, gn = _gamma(mu), _gamma(nu)
        sig = 0.5j * (gm @ gn - gn @ gm)
        for b in range(2):
            s = sig[2 * b:2 * b + 2, 2 * b:2 * b + 2]
            k = s[:, None, :, None] * F[..., None, :, None, :]
            blocks[b] = blocks[b] - KAPPA * CSW * k.reshape(lat + (6, 6))
    return torch.stack(blocks, -3)


def _site(A, psi):
    """A psi for the two chiral blocks; psi [T, Z, Y, X, spin, colour, n]."""
    v = psi.reshape(psi.shape[:4] + (2, 6, psi.shape[-1]))
    return (A @ v).reshape(psi.shape)


def _hop(U, psi):
    """D psi on the full lattice; psi [T, Z, Y, X, spin, colour, n]."""
    out = torch.zeros_like(psi)
    n = psi.shape[-1]
    for mu in range(4):
        u = U[..., mu, :, :]
        if mu == 3:
            u = torch.cat([u[:-1], T_BC * u[-1:]], 0)
        coef = torch.tensor(_COEF[mu], dtype=psi.dtype, device=psi.device)[:, None, None]
        for sgn, link, nb in ((-1, u, _at(psi, mu, 1)), (1, _dag(_at(u, mu, -1)), _at(psi, mu, -1))):
            h = (nb + sgn * coef * nb[..., _PERM[mu], :, :])
            h = h.transpose(-3, -2).reshape(h.shape[:4] + (3, 4 * n))
            h = (link @ h).reshape(psi.shape[:4] + (3, 4, n)).transpose(-3, -2)
            out = out + h
    return out


def _parity(case):
    t, z, y, x = torch.meshgrid(*(torch.arange(k, device="cuda") for k in _shape(case)), indexing="ij")
    return (x + y + z + t) % 2


class _Schur:
    """Mhat on full-lattice fields that are zero on the other parity."""

    def __init__(self, case, U):
        self.U = U
        self.A = _clover(U)
        self.inv = torch.linalg.inv(self.A)
        p = _parity(case)
        self.even = (p == 0).to(U.dtype)[..., None, None, None]
        self.odd = 1 - self.even
        self.index = [(p == k).reshape(-1).nonzero()[:, 0] for k in range(2)]
        self.shape = _shape(case)

    def full(self, f, parity):
        """[n, V/2, 4, 3] on one parity -> [T, Z, Y, X, 4, 3, n], zero elsewhere."""
        n = f.shape[0]
        out = torch.zeros(self.even.numel(), 4, 3, n, dtype=f.dtype, device=f.device)
        out[self.index[parity]] = f.permute(1, 2, 3, 0)
        return out.reshape(self.shape + (4, 3, n))

    def half(self, f, parity):
        n = f.shape[-1]
        return f.reshape(-1, 4, 3, n)[self.index[parity]].permute(3, 0, 1, 2).contiguous()

    def g5(self, f):
        return torch.cat([f[..., :2, :, :], -f[..., 2:, :, :]], -3)

    def mhat(self, x, dagger=False):
        if dagger:
            return self.g5(self.mhat(self.g5(x)))
        t = _site(self.inv, self.odd * _hop(self.U, x))
        return _site(self.A, x) - KAPPA ** 2 * self.even * _hop(self.U, t)

    def mdagm(self, x):
        return self.mhat(self.mhat(x), True)

    def solve(self, b, tol):
        """Conjugate gradients per right-hand side (the last axis) to |r| <= tol |b|."""
        def dot(u, v):
            return (u.conj() * v).real.sum(dim=tuple(range(u.ndim - 1)))
        x, r, p = torch.zeros_like(b), b.clone(), b.clone()
        rr = dot(r, r)
        stop = tol ** 2 * rr
        for k in range(1000):
            if k % 8 == 0 and bool((rr <= stop).all()):
                break
            ap = self.mdagm(p)
            a = rr / dot(p, ap)
            x = x + a * p
            r = r - a * ap
            new = dot(r, r)
            p = r + (new / rr) * p
            rr = new
        return x


def _gradients(case, U, x, det):
    """The Wirtinger gradient of the pseudofermion action at the solutions x (full lattice), with
    det of S_det = -2 sum_{x odd} log det A: dS = -2 Re <Mhat x, (dMhat) x>."""
    U = U.detach().requires_grad_(True)
    S = _Schur(case, U)
    L = 0.0
    if x is not None:
        y = S.mhat(x)
        L = L - 2 * (y.detach().conj() * y).real.sum()
    if det:
        ld = torch.linalg.slogdet(S.A)[1].sum(-1)
        L = L - 2 * (ld * S.odd[..., 0, 0, 0].real).sum()
    return torch.autograd.grad(L, U)[0]


def _ta(m):
    a = (m - _dag(m)) / 2
    tr = a.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None]
    return a - tr * torch.eye(3, dtype=m.dtype, device=m.device) / 3


def _plaquette_sum(U):
    s = 0.0
    for mu, nu in _PLANES:
        m, n = U[..., mu, :, :], U[..., nu, :, :]
        p = m @ _at(n, mu, 1) @ _dag(_at(m, nu, 1)) @ _dag(n)
        s = s + p.diagonal(dim1=-2, dim2=-1).sum().real / 3
    return s


def _move(U, P, eps):
    return _project(torch.linalg.matrix_exp(eps * P) @ U)


def exact(case, seed):
    kind = case["kind"]
    n = case.get("nrhs", 1)
    V = _volume(case)
    # conjugate gradients in plain torch take too long on the largest batches
    if (kind == "solve" and V * n > 1_500_000) or (kind in ("rstep", "action", "force") and V > 200_000):
        return None
    v = _inputs(case, seed)
    U, f = v["links"], v["field"]
    if kind == "apply":
        return _exact_apply(case, U, f)
    if kind == "solve":
        S = _Schur(case, U)
        return S.half(S.solve(S.full(f, 0), 1e-13), 0)
    if kind == "ingest":
        S = _Schur(case, U)
        ld = torch.linalg.slogdet(S.A)[1].sum(-1)
        odd = S.odd[..., 0, 0, 0].real
        return {"mhat": S.half(S.mhat(S.full(f, 0)), 0),
                "logdet": [float((ld * (1 - odd)).sum()), float((ld * odd).sum())]}
    if kind == "force":
        S = _Schur(case, U)
        G = _gradients(case, U, S.full(f, 0), case["det"])
        return -0.5 * _ta(U @ _dag(G))
    if kind == "action":
        S = _Schur(case, U)
        phi = S.full(f, 0)
        x = S.solve(phi, 1e-13)
        return {"S": (phi.conj() * x).real.sum(), "gU": _gradients(case, U, x, False), "gphi": 2 * S.half(x, 0)}
    P = v["momenta"]
    U = _move(U, P, 0.5 * DTAU)
    S = _Schur(case, U)
    x = S.solve(S.mhat(S.full(f, 0), True), 1e-13)
    G = _gradients(case, U, x, True)
    W = U.detach().requires_grad_(True)
    G = G + torch.autograd.grad(-BETA * _plaquette_sum(W), W)[0]
    P = P - DTAU * (-0.5 * _ta(U @ _dag(G)))
    U = _move(U, P, 0.5 * DTAU)
    return {"U": U, "P": P, "plaquette": float(_plaquette_sum(U) / (6 * V))}


def _exact_apply(case, U, f):
    S = _Schur(case, U)
    outs = []
    for k in range(0, f.shape[0], 2):  # two fields at a time
        g = f[k:k + 2]
        op, dag = case["op"], case["dagger"]
        if op in ("mhat", "mdagm"):
            x = S.full(g, 0)
            outs.append(S.half(S.mdagm(x) if op == "mdagm" else S.mhat(x, dag), 0))
        elif op == "clover":
            outs.append(S.half(_site(S.A, S.full(g, 0)), 0))
        elif op == "clover_inv":
            outs.append(S.half(_site(S.inv, S.full(g, 1)), 1))
        else:
            to = 0 if op == "dslash_eo" else 1
            x = S.full(g, 1 - to)
            outs.append(S.half(S.g5(_hop(U, S.g5(x))) if dag else _hop(U, x), to))
    return torch.cat(outs)
