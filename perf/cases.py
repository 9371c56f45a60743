"""The calls that stand for what this library is used for, with their inputs, their
results in 64 bits and the memory traffic and arithmetic they cannot do without.

Lattices and parameters are those of the configurations that the tests and bench.py run
(8^4, 24^3x48 with 1 and 12 right-hand sides and ten shifts, 32^3x64 with C* boundaries,
16^4 for the learned preconditioner, two-flavour C* systems with BF16 inner solves), the
mid-size ones with smaller extents where the exact result would take long.  Extents are
given in the order (x0, x1, x2, x3) of the physical lattice; with cstar > 0 the simulated
lattice is twice as long in x1.
"""
import math

import numpy as np
import torch

from paper_1908_11673_gb300 import qxd

C64, C128 = torch.complex64, torch.complex128

# link, phase and site-diagonal bytes per site as the library's FP32 and FP64 operators need
# them at least: two rows of SU(3) and a U(1) phase, or a full 3x3 matrix, in four directions;
# two Hermitian 6x6 blocks
LINKS = {qxd.FP32: 4 * 56, qxd.FP64: 4 * 144}
DIAG = {qxd.FP32: 288, qxd.FP64: 576}
SPINOR = {qxd.FP32: 96, qxd.FP64: 192}
FLOPS_D = 2112  # per site and application of D or Dhat (hop, U(1) phases, two 6x6 products)

# the ten shifts of the printed degree-10 approximation's range
SHIFTS = np.geomspace(1.2e-3, 8.4, 10)


def _case(name, op, L, cstar=0, **more):
    c = {"name": name, "op": op, "L0": L[0], "L1": L[1], "L2": L[2], "L3": L[3], "cstar": cstar}
    c.update(more)
    return c


def listed():
    up = {"qhat": 4, "kappa": 0.137312, "u1csw": 1.0}
    down = {"qhat": -2, "kappa": 0.136377, "u1csw": 1.0}
    return [
        # one operator application on the smallest lattice in use: launches and host time count
        _case("dhat_fp32_8x8x8x8", "dhat", (8, 8, 8, 8), prec=qxd.FP32, dagger=False, nrhs=1, **down),
        # Dhat^+ in the FP32 that inner solves and external Krylov loops use, ordinary size
        _case("dhat_dag_fp32_48x24x24x24", "dhat", (48, 24, 24, 24), prec=qxd.FP32, dagger=True, nrhs=1, **down),
        # the same on the large C* lattice (64 x 64 x 32 x 32 simulated)
        _case("dhat_fp32_64x32x32x32_c3", "dhat", (64, 32, 32, 32), 3, prec=qxd.FP32, dagger=False, nrhs=1, **up),
        # twelve spin-colour sources of a propagator at once
        _case("dw_fp32_12rhs_48x24x24x24", "dw", (48, 24, 24, 24), prec=qxd.FP32, nrhs=12, **down),
        # the full operator in FP64: residual checks of a user's own solver
        _case("dw_fp64_48x24x24x24", "dw", (48, 24, 24, 24), prec=qxd.FP64, nrhs=1, **down),
        # a new gauge configuration: links, site-diagonal terms, first application
        _case("configuration_32x16x16x16", "configuration", (32, 16, 16, 16), 1, **up),
        # mixed-precision solve to 1e-10, the library's headline
        _case("solve_fgcr_64x32x32x32_c3", "solve", (64, 32, 32, 32), 3, nrhs=1, inner=qxd.FP32, nkv=8, precond="none",
              sigma=0.3, tol=1e-10, **up),
        # four sources in lockstep with bfloat16 storage in the inner solves
        _case("solve_bf16_4rhs_32x16x16x16_c3", "solve", (32, 16, 16, 16), 3, nrhs=4, inner=qxd.BF16, nkv=8,
              precond="none", sigma=0.3, tol=1e-11, u1_steps=5, qhat=4, kappa=0.137312, u1csw=1.90952),
        # light quark on a rough field: deflation and SAP in flexible GCR
        _case("solve_dfl_32x16x16x16", "solve", (32, 16, 16, 16), nrhs=1, inner=qxd.FP32, nkv=16, precond="dfl",
              sigma=0.6, tol=1e-11, qhat=-2, kappa=0.130, u1csw=1.0),
        # the Schwarz preconditioner alone with the paper's 5 cycles of 5 steps
        _case("sap_apply_48x24x24x24", "sap", (48, 24, 24, 24), ncy=5, nmr=5, **down),
        # the shifted systems of the rational approximation (RHMC, reweighting)
        _case("multishift_32x16x16x16", "multishift", (32, 16, 16, 16), nshift=10, **down),
        # one training batch of the learned preconditioner: loss and gradient, 4 layers of 8 channels
        _case("train_16x16x16x16", "train", (16, 16, 16, 16), nlayers=4, nch=8, npairs=10, kind=qxd.LOSS_RESIDUAL, **down),
    ]


def _extents(rng, step, lo, hi):
    """Four extents (multiples of step) whose product is spread over the logarithm of lo..hi."""
    while True:
        side = math.exp(rng.uniform(math.log(lo), math.log(hi)) / 4)
        L = [max(step if step > 4 else 4, step * round(side * 2 ** rng.uniform(-0.6, 0.6) / step)) for _ in range(4)]
        if lo <= math.prod(L) <= hi:
            return tuple(L)


def draw(rng):
    op = rng.choice(["dhat", "dhat", "dhat", "dw", "dw", "dw", "configuration", "solve", "solve", "sap", "sap", "multishift",
                     "train"])
    cstar = rng.randint(0, 3)
    quark = rng.choice([{"qhat": 4, "kappa": 0.137312, "u1csw": 1.0}, {"qhat": -2, "kappa": 0.136377, "u1csw": 1.0}])
    half = 2 if cstar else 1  # the simulated lattice is twice the physical one
    if op == "dhat":
        return _case(None, op, _extents(rng, 2, 8 ** 4, 2 ** 20), cstar, prec=rng.choice([qxd.FP32, qxd.FP32, qxd.FP64]),
                     dagger=rng.random() < 0.5, nrhs=rng.choice([1, 1, 1, 2, 3, 4]), **quark)
    if op == "dw":
        return _case(None, op, _extents(rng, 2, 8 ** 4, 2 ** 19), cstar, prec=rng.choice([qxd.FP32, qxd.FP32, qxd.FP64]),
                     nrhs=rng.choice([1, 1, 2, 3, 4, 6, 12]), **quark)
    if op == "configuration":
        return _case(None, op, _extents(rng, 2, 8 ** 4, 2 ** 18), cstar, **quark)
    if op == "solve":
        inner = rng.choice([qxd.FP32, qxd.BF16])
        precond = rng.choice(["none", "sap", "dfl"]) if inner == qxd.FP32 else "none"
        L = _extents(rng, 8 if precond != "none" else 2, 8 ** 4, 2 ** 17 // half)
        if precond == "dfl":
            return _case(None, op, L, cstar, nrhs=1, inner=inner, nkv=16, precond=precond, sigma=0.6, tol=1e-11, qhat=-2,
                         kappa=0.130, u1csw=1.0)
        return _case(None, op, L, cstar, nrhs=rng.choice([1, 2, 4]) if precond == "none" else 1, inner=inner,
                     nkv=rng.choice([8, 12, 16]), precond=precond, sigma=0.6, tol=1e-11, qhat=quark["qhat"], kappa=0.126,
                     u1csw=1.0)
    if op == "sap":
        return _case(None, op, _extents(rng, 8, 8 ** 4, 2 ** 19), cstar, ncy=rng.randint(2, 5), nmr=rng.randint(3, 5), **quark)
    if op == "multishift":
        return _case(None, op, _extents(rng, 2, 8 ** 4, 2 ** 17 // half), cstar, nshift=rng.randint(4, 10), **quark)
    return _case(None, op, _extents(rng, 2, 8 ** 4, 2 ** 16 // half), cstar, nlayers=rng.randint(2, 4),
                 nch=rng.choice([4, 6, 8]), npairs=rng.randint(2, 8), kind=rng.choice([qxd.LOSS_ERROR, qxd.LOSS_RESIDUAL]),
                 **quark)


# ---- inputs ---------------------------------------------------------------------------
def _geometry(case):
    L = tuple(case["L%d" % i] for i in range(4))
    N = (L[0], 2 * L[1], L[2], L[3]) if case["cstar"] else L
    return L, N


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _unitary(U):
    """SU(3) from complex 3x3 matrices near it: Gram-Schmidt on two rows, third row their conjugate cross product."""
    a, b = U[..., 0, :], U[..., 1, :]
    a = a / a.abs().square().sum(-1, keepdim=True).sqrt()
    b = b - (a.conj() * b).sum(-1, keepdim=True) * a
    b = b / b.abs().square().sum(-1, keepdim=True).sqrt()
    return torch.stack((a, b, torch.linalg.cross(a, b, dim=-1).conj()), -2)


def _mm(a, b):
    """Products of small matrices (faster than a batched library product for 3x3)."""
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _gauge_field(L, gen, sigma, u1_steps=0, steps=5, alpha=0.6):
    """Links (complex128 [V][4][3][3]) and photon angles ([V][4]) as the path meets them: noise of width
    sigma, smeared `steps` times with all six staples (APE weights, projected to SU(3)); Gaussian angles of width 0.2, u1_steps abelian stout steps (0.1)."""
    dev = gen.device
    h = sigma * torch.randn(*L, 4, 3, 3, 2, generator=gen, device=dev)
    h = torch.view_as_complex(h)
    h = (h + h.mH) / math.sqrt(2)
    one = torch.eye(3, dtype=C64, device=dev)
    U = _unitary(one + 1j * h - 0.5 * _mm(h, h))
    for _ in range(steps):
        new = torch.empty_like(U)
        for mu in range(4):
            a = U[..., mu, :, :]
            s = (1 - alpha) * a
            for nu in range(4):
                if nu != mu:
                    b = U[..., nu, :, :]
                    b_mu = torch.roll(b, -1, mu)
                    up = _mm(_mm(b, torch.roll(a, -1, nu)), b_mu.mH)
                    s = s + alpha / 6 * (up + torch.roll(_mm(_mm(b.mH, a), b_mu), 1, nu))
            new[..., mu, :, :] = _unitary(s)
        U = new
    U = _unitary(U.to(C128)).reshape(-1, 4, 3, 3).contiguous()
    A = 0.2 * torch.randn(*L, 4, generator=gen, device=dev, dtype=torch.float64)
    for _ in range(u1_steps):
        new = A.clone()
        for mu in range(4):
            a = A[..., mu]
            for nu in range(4):
                if nu != mu:
                    b = A[..., nu]
                    b_mu = torch.roll(b, -1, mu)
                    new[..., mu] += 0.1 * torch.sin(b + torch.roll(a, -1, nu) - b_mu - a)
                    new[..., mu] += 0.1 * torch.sin(torch.roll(b_mu + a - b, 1, nu) - a)
        A = new
    return U, A.reshape(-1, 4).contiguous()


def _noise(gen, dtype, *shape):
    real = torch.float64 if dtype == C128 else torch.float32
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device=gen.device, dtype=real))


def _theta(case):
    return (math.pi, 0.0, 0.0, 0.0)


def _inputs(case, seed):
    """Everything random of a case: gauge field and the fields that go in."""
    gen = torch.Generator(device=_device()).manual_seed(int(seed))
    L, N = _geometry(case)
    V = math.prod(N)
    sigma = case.get("sigma", 0.3)
    U, A = _gauge_field(L, gen, sigma, case.get("u1_steps", 0))
    s = {"U": U, "A": A}
    op = case["op"]
    if op == "dhat":
        s["x"] = _noise(gen, C128 if case["prec"] == qxd.FP64 else C64, case["nrhs"], V // 2, 4, 3)
    elif op == "dw":
        s["x"] = _noise(gen, C128 if case["prec"] == qxd.FP64 else C64, case["nrhs"], V, 4, 3)
    elif op == "configuration":
        s["x"] = _noise(gen, C128, V, 4, 3)
    elif op == "solve":
        s["x"] = _noise(gen, C128, case["nrhs"], V, 4, 3)
        if case["precond"] == "dfl":
            s["seeds"] = _noise(gen, C64, 12, V, 4, 3)
    elif op == "sap":
        s["x"] = _noise(gen, C64, V, 4, 3)
    elif op == "multishift":
        s["x"] = _noise(gen, C128, V // 2, 4, 3)
    else:
        s["r"] = _noise(gen, C64, case["npairs"], V // 2, 4, 3)
        s["e"] = _noise(gen, C64, case["npairs"], V // 2, 4, 3)
        # weights as in the course of a training: the start 2 kappa on the first channels plus noise
        parts = []
        for cin, cout in _layers(case):
            w = 0.02 * _noise(gen, C64, cout, cin, 9, 4, 4)
            for c in range(min(cin, cout)):
                w[c, c, 0] += (2 * case["kappa"]) ** (1 / case["nlayers"]) * torch.eye(4, dtype=C64, device=w.device)
            parts.append(w.reshape(-1))
        s["W"] = torch.cat(parts)
    return s


def _layers(case):
    n, c = case["nlayers"], case["nch"]
    return [(1 if l == 0 else c, 1 if l == n - 1 else c) for l in range(n)]


def prepare(case, seed):
    s = _inputs(case, seed)
    L, N = _geometry(case)
    ctx = qxd.Context(L, case["cstar"], _theta(case))
    s["ctx"], s["case"] = ctx, case
    op = case["op"]
    if op != "configuration":
        ctx.set_links(s["U"], s["A"])
        ctx.set_clover(0, case["qhat"], case["kappa"], 1.90952, case["u1csw"])
    if op == "sap":
        ctx.set_sap(case["ncy"], case["nmr"])
    if op == "solve" and case["precond"] != "none":
        ctx.set_sap(3, 4)
        if case["precond"] == "dfl":
            ctx.dfl_setup(0, s.pop("seeds"), 12, 2)
    if op == "multishift":
        s["out"] = torch.empty((case["nshift"],) + tuple(s["x"].shape), dtype=C128, device=s["x"].device)
    elif op == "train":
        s["out"] = torch.empty_like(s["W"])
    else:
        s["out"] = torch.empty_like(s["x"])
    return s


_PRECOND = {"none": qxd.PRECOND_NONE, "sap": qxd.PRECOND_SAP, "dfl": qxd.PRECOND_DFL}


def run(s):
    ctx, case, op = s["ctx"], s["case"], s["case"]["op"]
    if op == "dhat":
        ctx.apply_Dhat_eo(0, case["prec"], s["x"], s["out"], dagger=case["dagger"], nrhs=case["nrhs"])
    elif op == "dw":
        ctx.apply_Dw(0, case["prec"], s["x"], s["out"], nrhs=case["nrhs"])
    elif op == "configuration":
        ctx.set_links(s["U"], s["A"])
        ctx.set_clover(0, case["qhat"], case["kappa"], 1.90952, case["u1csw"])
        ctx.apply_Dw(0, qxd.FP64, s["x"], s["out"])
    elif op == "solve":
        ctx.solve(0, s["x"], s["out"], kind=qxd.FGCR, tol=case["tol"], nkv=case["nkv"], inner=case["inner"],
                  precond=_PRECOND[case["precond"]], nrhs=case["nrhs"])
    elif op == "sap":
        ctx.sap_apply(0, s["x"], s["out"])
    elif op == "multishift":
        ctx.solve_multishift(0, SHIFTS[: case["nshift"]], s["x"], s["out"], tol=1e-11, inner=qxd.FP32)
    else:
        loss = ctx.ptc_loss_grad(0, s["W"], case["nlayers"], case["nch"], s["r"], s["e"], case["npairs"], s["out"],
                                 kind=case["kind"])
        return {"loss": loss, "grad": s["out"]}
    return s["out"]


def work(case):
    """Traffic with every array read or written once per operator application, and flops."""
    V = math.prod(_geometry(case)[1])
    op = case["op"]
    if op in ("dhat", "dw"):
        p, n = case["prec"], case["nrhs"]
        sites = V // 2 if op == "dhat" else V  # sites of the fields that go in and come out
        return {"bytes": V * (LINKS[p] + DIAG[p]) + sites * 2 * SPINOR[p] * n, "flops": V * FLOPS_D * n}
    if op == "configuration":
        # links and angles in; the terms and their inverses out in both precisions, links in both; 24 clover leaves of
        # which each plaquette's four share half their 3x3 products, two 6x6 inverses, one application
        phys = V // 2 if case["cstar"] else V
        return {"bytes": phys * (576 + 32) + V * (576 + 192 + 32 + 2 * (576 + 288) + 576 + 2 * 192),
                "flops": V * (6 * 8 * 198 + 2 * 1728 + FLOPS_D)}
    fp32_dhat = V * (LINKS[qxd.FP32] + DIAG[qxd.FP32]) + V * SPINOR[qxd.FP32]
    if op == "solve":
        # the iterations that GCR of this restart length takes at the listed sizes, each one operator application
        # and one new direction kept; the preconditioners' own work once per iteration
        its = {"none": 50, "sap": 15, "dfl": 12}[case["precond"]] * case["nrhs"]
        f = 1 if case["precond"] == "none" else 20
        return {"bytes": its * f * fp32_dhat, "flops": its * f * V * FLOPS_D}
    if op == "sap":
        # per half sweep: links, terms, source and solution of the colour once; the block hops and products of the steps
        return {"bytes": case["ncy"] * V * (LINKS[qxd.FP32] + DIAG[qxd.FP32] + 144 + 3 * SPINOR[qxd.FP32]),
                "flops": case["ncy"] * V * FLOPS_D * (case["nmr"] + 2)}
    if op == "multishift":
        its = 300
        return {"bytes": its * (2 * fp32_dhat + V // 2 * SPINOR[qxd.FP32] * 2 * case["nshift"]), "flops": its * 2 * V * FLOPS_D}
    mix = sum(cin * cout for cin, cout in _layers(case)) * 9 * 16 * 3 * 8
    field = sum(cin + cout for cin, cout in _layers(case)) * SPINOR[qxd.FP32] + case["nlayers"] * LINKS[qxd.FP32]
    return {"bytes": 3 * case["npairs"] * V * field, "flops": 3 * case["npairs"] * V * mix}


# ---- the same in 64 bits, in plain torch -----------------------------------------------
# gamma_mu = [[0, B], [B^+, 0]]; B has one entry in each row: its column and its value
_GAMMA = [((0, 1), (-1, -1)), ((1, 0), (-1j, -1j)), ((1, 0), (-1, 1)), ((0, 1), (-1j, 1j))]


class _Operator:
    """D = 1/(2 kappa) + SW term + hopping term on the simulated lattice, complex128.  Fields are kept by
    parity: a half field lists the sites of one parity in lexicographic order, [V/2, 4, 3]."""

    def __init__(self, case, U, A):
        L, N = _geometry(case)
        self.N, self.cstar, self.L1 = N, case["cstar"], L[1]
        dev = U.device
        U, A = U.reshape(*L, 4, 3, 3), A.reshape(*L, 4)
        if self.cstar:
            U, A = torch.cat((U, U.conj()), 1), torch.cat((A, -A), 1)
        self.V = math.prod(N)
        site = torch.arange(self.V, device=dev).reshape(N)
        self.fwd = [self._shift(site, mu, 1).reshape(-1) for mu in range(4)]
        self.bwd = [self._shift(site, mu, -1).reshape(-1) for mu in range(4)]
        x = torch.stack(torch.meshgrid(*[torch.arange(n, device=dev) for n in N], indexing="ij"), -1).reshape(-1, 4)
        self.x = x
        self.sites = [(x.sum(1) % 2 == p).nonzero()[:, 0] for p in range(2)]
        U, A = U.reshape(-1, 4, 3, 3), A.reshape(-1, 4)
        ang = case["qhat"] * A
        th = _theta(case)
        for mu in range(4):
            if not (self.cstar and 1 <= mu <= self.cstar):
                ang[:, mu] = ang[:, mu] + th[mu] * (x[:, mu] == N[mu] - 1).double()
        link = U * torch.polar(torch.ones_like(ang), ang)[..., None, None]
        # hop d = mu from x + mu, 4 + mu from x - mu: sites and colour matrices, on the whole lattice and by parity
        self.from_ = self.fwd + self.bwd
        self.colour = [link[:, mu].contiguous() for mu in range(4)]
        self.colour += [link[self.bwd[mu], mu].mH.contiguous() for mu in range(4)]
        self.half = [[(f[s] // 2, m[s]) for f, m in zip(self.from_, self.colour)] for s in self.sites]
        self.g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device=dev)[:, None]
        diag = self._diagonal(case, U, A)
        self.diag = [diag[s] for s in self.sites]  # [V/2, chirality, 6, 6]
        self.inv = [torch.linalg.inv(d) for d in self.diag]

    def _shift(self, f, mu, sign):
        """f(x + sign mu): crossing a C* direction 2 or 3 moves x1 by half its extent."""
        g = torch.roll(f, -sign, mu)
        if mu >= 2 and mu <= self.cstar:
            at = [slice(None)] * 4
            at[mu] = self.N[mu] - 1 if sign > 0 else 0
            g = g.clone()
            g[tuple(at)] = torch.roll(g[tuple(at)], self.L1, 1)
        return g

    def _diagonal(self, case, U, A):
        """1/(2 kappa) + sum_{mu < nu} (i/2) sigma_{mu nu} G_{mu nu}, block diagonal in the chirality."""
        V, f, b, dev = self.V, self.fwd, self.bwd, U.device
        gamma = torch.zeros(4, 4, 4, dtype=C128)
        for mu, (col, val) in enumerate(_GAMMA):
            for r in range(2):
                gamma[mu, r, 2 + col[r]] = val[r]
                gamma[mu, 2 + col[r], r] = complex(val[r]).conjugate()
        M = torch.zeros(V, 2, 2, 3, 2, 3, dtype=C128, device=dev)
        for mu in range(4):
            for nu in range(mu + 1, 4):
                lo, ln, both = b[mu], b[nu], b[nu][b[mu]]
                Q = _mm(_mm(U[:, mu], U[f[mu], nu]), _mm(U[:, nu], U[f[nu], mu]).mH) + self._leaves(U, mu, nu, lo, ln, both)
                p = torch.sin(A[:, mu] + A[f[mu], nu] - A[f[nu], mu] - A[:, nu])
                p = p + p[lo] + p[ln] + p[both]
                G = 1.90952 * (Q - Q.mH) / 8 + (0.25j * case["u1csw"] * case["qhat"]) * p[:, None, None] * torch.eye(
                    3, dtype=C128, device=dev)
                s = 0.5j * (gamma[mu] @ gamma[nu] - gamma[nu] @ gamma[mu])
                s = torch.stack((s[:2, :2], s[2:, 2:])).to(dev)
                M += 0.5j * s[None, :, :, None, :, None] * G[:, None, None, :, None, :]
        return M.reshape(V, 2, 6, 6) + torch.eye(6, dtype=C128, device=dev) / (2 * case["kappa"])

    def _leaves(self, U, mu, nu, lo, ln, both):
        """The clover leaves at x whose plaquettes have their lower corners at x - mu, x - mu - nu and x - nu."""
        f = self.fwd
        Um, Un = U[:, mu], U[:, nu]
        Q = _mm(_mm(Un, Um[f[nu][lo]].mH), _mm(Un[lo].mH, Um[lo]))
        Q = Q + _mm(_mm(Um[lo].mH, Un[both].mH), _mm(Um[both], Un[ln]))
        return Q + _mm(_mm(Un[ln].mH, Um[ln]), _mm(Un[f[mu][ln]], Um.mH))

    def transport(self, d, f):
        """T_d of a field [V, channels, 4, 3]: 0 the field, 1 + mu from x + mu, 5 + mu from x - mu."""
        if d == 0:
            return f
        g = f[self.from_[d - 1]]
        return (g.reshape(self.V, -1, 3) @ self.colour[d - 1].mT).reshape(g.shape)

    def hop(self, f, p, keep=None):
        """Hopping term at the sites of parity p from the half field f; keep: masks of the hops of that parity."""
        out = torch.zeros_like(f)
        for d, (idx, M) in enumerate(self.half[p]):
            col, val = _GAMMA[d % 4]
            sign = -1 if d < 4 else 1  # 1 - gamma forwards, 1 + gamma backwards
            b = torch.tensor(val, dtype=C128, device=f.device)[:, None] * sign
            g = f[idx]
            h = g[:, :2] + b * g[:, [2 + col[0], 2 + col[1]]]
            h = (M[:, None] * h[:, :, None, :]).sum(-1)
            if keep is not None:
                h = h * keep[p][d][:, None, None]
            out[:, :2] -= 0.5 * h
            out[:, 2:] -= 0.5 * (b.conj() * h)[:, [col[0], col[1]]]
        return out

    def mul(self, M, f):
        return (M @ f.reshape(-1, 2, 6, 1)).reshape(f.shape)

    def split(self, f):
        return f[self.sites[0]], f[self.sites[1]]

    def join(self, e, o):
        f = torch.empty((self.V,) + e.shape[1:], dtype=e.dtype, device=e.device)
        f[self.sites[0]], f[self.sites[1]] = e, o
        return f

    def D(self, e, o):
        return self.mul(self.diag[0], e) + self.hop(o, 0), self.mul(self.diag[1], o) + self.hop(e, 1)

    def dhat(self, e, dagger=False):
        e = self.g5 * e if dagger else e
        out = self.mul(self.diag[0], e) - self.hop(self.mul(self.inv[1], self.hop(e, 1)), 0)
        return self.g5 * out if dagger else out

    def normal(self, e):
        return self.dhat(self.dhat(e), True)

    def solve(self, eta):
        """D^-1 eta by CG on the normal equations of Dhat, to rounding."""
        e, o = self.split(eta)
        b = e - self.hop(self.mul(self.inv[1], o), 0)
        x = self.cg(self.dhat(b, True), 1e-9)
        x = x + self.cg(self.dhat(b - self.dhat(x), True), 1e-6)
        return self.join(x, self.mul(self.inv[1], o - self.hop(x, 1)))

    def cg(self, b, tol):
        return self.cg_shifted(b, [0.0], tol)[0]

    def cg_shifted(self, b, shifts, tol=1e-14):
        """(normal + s)^-1 b for ascending shifts s: one Krylov space, the recursion of the shifted residuals."""
        n = len(shifts)
        d = [float(s - shifts[0]) for s in shifts]
        X, P = [torch.zeros_like(b) for _ in d], [b.clone() for _ in d]
        z, zo = [1.0] * n, [1.0] * n
        r, p = b.clone(), b.clone()
        rr = start = float(r.abs().square().sum())
        a_old, beta = 1.0, 0.0
        for _ in range(20000):
            w = self.normal(p) + float(shifts[0]) * p
            a = rr / float((p.conj() * w).sum().real)
            r = r - a * w
            new = float(r.abs().square().sum())
            b_new = new / rr
            for j in range(n):
                if j and abs(z[j]) ** 2 * rr < 1e-30 * start:
                    continue
                zn = z[j] * zo[j] * a_old / (a * beta * (zo[j] - z[j]) + zo[j] * a_old * (1 + d[j] * a))
                X[j] += (a * zn / z[j]) * P[j]
                P[j] = zn * r + (b_new * (zn / z[j]) ** 2) * P[j]
                zo[j], z[j] = z[j], zn
            rr, a_old, beta = new, a, b_new
            p = r + beta * p
            if new <= tol * tol * start:
                break
        return torch.stack(X)

    def sap(self, eta, ncy, nmr):
        nb = [n // 4 for n in self.N]
        bc = self.x // 4
        block = ((bc[:, 0] * nb[1] + bc[:, 1]) * nb[2] + bc[:, 2]) * nb[3] + bc[:, 3]
        inside = [(block[f] == block).double() for f in self.from_]
        keep = [[m[s] for m in inside] for s in self.sites]
        colour = [(bc.sum(1) % 2)[s] for s in self.sites]
        even = block[self.sites[0]]

        def total(v):
            return torch.zeros(math.prod(nb), dtype=v.dtype, device=v.device).index_add_(0, even, v)[even]

        eta = self.split(eta)
        psi, rho = [torch.zeros_like(f) for f in eta], eta
        for k in range(2 * ncy):
            ev, od = [(c == k % 2).double()[:, None, None] for c in colour]
            r = ev * (rho[0] - self.hop(od * self.mul(self.inv[1], rho[1]), 0, keep))
            y = torch.zeros_like(r)
            for _ in range(nmr):
                p = self.mul(self.diag[0], r) - self.hop(self.mul(self.inv[1], self.hop(r, 1, keep)), 0, keep)
                pp = total(p.abs().square().sum((1, 2)))
                pr = total((p.conj() * r).sum((1, 2)))
                a = torch.where(pp > 0, pr / torch.where(pp > 0, pp, torch.ones_like(pp)), torch.zeros_like(pr))
                y, r = y + a[:, None, None] * r, r - a[:, None, None] * p
            psi = [psi[0] + y, psi[1] + od * self.mul(self.inv[1], rho[1] - self.hop(y, 1, keep))]
            rho = [n - f for n, f in zip(eta, self.D(*psi))]
        return self.join(*psi)


def _exact_train(o, case, s):
    Ws, at = [], 0
    for cin, cout in _layers(case):
        n = cout * cin * 144
        Ws.append(s["W"][at:at + n].to(C128).reshape(cout, cin, 9, 4, 4).clone().requires_grad_(True))
        at += n
    loss = 0.0
    for r, e in zip(s["r"].to(C128), s["e"].to(C128)):
        a = o.join(r, torch.zeros_like(r))[:, None]  # [V, channel, spin, colour]
        for W in Ws:
            cout, cin = W.shape[:2]
            T = torch.stack([o.transport(d, a) for d in range(9)], 1)  # [V, 9, cin, 4, 3]
            w = W.permute(0, 3, 2, 1, 4).reshape(cout * 4, 9 * cin * 4)
            a = torch.matmul(w, T.reshape(o.V, 9 * cin * 4, 3)).reshape(o.V, cout, 4, 3)
        out = a[o.sites[0], 0]
        if case["kind"] == qxd.LOSS_ERROR:
            one = (out - e).abs().square().sum() / e.abs().square().sum()
        else:
            one = (r - o.dhat(out)).abs().square().sum() / r.abs().square().sum()
        one.backward()
        loss += float(one.detach())
    # torch's gradient of a real loss is dL/dRe + i dL/dIm = 2 dL/dW^*
    return {"loss": loss, "grad": torch.cat([0.5 * W.grad.reshape(-1) for W in Ws])}


def exact(case, seed):
    op = case["op"]
    V = math.prod(_geometry(case)[1])
    if V > 2 ** 20 or op in ("solve", "multishift") and V * case.get("nrhs", 1) > 2 ** 20:
        return None
    s = _inputs(case, seed)
    s.pop("seeds", None)
    o = _Operator(case, s["U"], s["A"])
    if op == "dhat":
        return torch.stack([o.dhat(x.to(C128), case["dagger"]) for x in s["x"]])
    if op == "dw":
        return torch.stack([o.join(*o.D(*o.split(x.to(C128)))) for x in s["x"]])
    if op == "configuration":
        return o.join(*o.D(*o.split(s["x"])))
    if op == "solve":
        return torch.stack([o.solve(x) for x in s["x"]])
    if op == "sap":
        return o.sap(s["x"].to(C128), case["ncy"], case["nmr"])
    if op == "multishift":
        return o.cg_shifted(s["x"], SHIFTS[: case["nshift"]])
    return _exact_train(o, case, s)
