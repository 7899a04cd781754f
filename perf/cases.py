"""Performance cases: the calls a user of this framework makes, over the sizes it is used at.

Workloads are the ones of the repository's configurations, studies and tests: Hubbard rings and
lattices at half filling, and linear STO-3G hydrogen chains in Loewdin orbitals (spacing 1.8 bohr)
with 20 to 160 atoms, 256 to 32,768 walkers, thresholds 1e-6 (benchmark) and 1e-4 (studies), in the
mixed and the FP64 form, with and without the 5-site correlator product.

A case is {"op", "system", "W", "eps", "form", "cps", "sweeps"}:
  eloc     Engine.local_energy: the screened local energy and residence time of every walker
  sweep    one sampling sweep, Engine.local_energy + Engine.ctmc_step, with the periodic recompute
           of the tables (Engine.refresh) every 64 moves
  refresh  Engine.refresh: every table recomputed for the current parameters
  grad     vmc_accumulate_gradient into zeroed sums (the energy-gradient pieces of one sweep)
  logpsi   LogPsi forward and backward (ln|psi| of every walker, its vector-Jacobian product)
  batch    Batch.local_energy + Batch.ctmc_step over seven systems of uneven size, `sweeps` times,
           then the recompute of every system's tables
  iter     one iteration of optimize.optimize: `sweeps` x (local energy, gradient sums, move), then
           energy gradient, AMSGrad and the recompute of the tables
"""
import math

import numpy as np
import torch

from paper_1807_10633_gb300 import optimize as O
from paper_1807_10633_gb300 import systems as S
from paper_1807_10633_gb300 import vmc

DEV = "cuda"
RECOMPUTE = 64                     # moves between recomputes of the walker tables
UNEVEN = "hubbard4x4 hubbard6x6 hubbard8x8 hubbard10x10 H40 H60 H100"


def _case(name, op, system, W, form, eps=1e-6, cps=False, sweeps=0):
    return dict(name=name, op=op, system=system, W=W, form=form, eps=eps, cps=cps, sweeps=sweeps)


def listed():
    return [
        # the 10-site ring of the plain method: the smallest call, one sampling sweep at eps = 0
        _case("sweep_ring10_w256_fp64", "sweep", "hubbard10", 256, "fp64", eps=0.0),
        # the optimisation command line's defaults: H20, 4096 walkers, 16 sweeps per iteration
        _case("iter_H20_w4096_mixed", "iter", "H20", 4096, "mixed", sweeps=16),
        # an odd chain with an odd number of walkers (31 alpha + 30 beta electrons, unaligned rows)
        _case("eloc_H61_w5003_mixed", "eloc", "H61", 5003, "mixed"),
        # the benchmark's local energy, in both precision forms
        _case("eloc_H160_w32768_mixed", "eloc", "H160", 32768, "mixed"),
        _case("eloc_H160_w32768_fp64", "eloc", "H160", 32768, "fp64"),
        # the wavefunction of the paper's chains: 5-site correlators on every site
        _case("eloc_cps_H160_w8192_mixed", "eloc", "H160", 8192, "mixed", cps=True),
        # the recompute after every parameter update, at the benchmark's size and at an odd one
        _case("refresh_H160_w32768_mixed", "refresh", "H160", 32768, "mixed"),
        _case("refresh_H61_w5003_fp64", "refresh", "H61", 5003, "fp64"),
        # the backward direction of one sweep: the H80 configuration's walkers in FP64
        _case("grad_H80_w16384_fp64", "grad", "H80", 16384, "fp64"),
        # ln|psi| as a differentiable function: forward and backward
        _case("logpsi_H40_w4096_fp64", "logpsi", "H40", 4096, "fp64"),
        # lattices and chains of uneven size in one persistent launch
        _case("batch_uneven_w2048_mixed", "batch", UNEVEN, 2048, "mixed", sweeps=4),
        # the benchmark's whole step: 8 sweeps, gradient, AMSGrad, recompute
        _case("iter_H160_w32768_mixed", "iter", "H160", 32768, "mixed", sweeps=8),
    ]


def draw(rng):
    op = rng.choice(["eloc", "eloc", "sweep", "refresh", "grad", "logpsi", "iter"])
    form = rng.choice(["mixed", "mixed", "fp64"])
    n = int(round(math.exp(rng.uniform(math.log(14), math.log(128)))))
    # walkers: 64 up to the memory and work of the largest listed case
    top = 32768 if op in ("eloc", "refresh", "grad") else 8192
    if op == "logpsi":
        form, top = "fp64", 4096
    W = int(round(math.exp(rng.uniform(math.log(64), math.log(top)))))
    cps = op in ("eloc", "sweep") and rng.random() < 0.25
    if cps:
        W = max(1, W // 4)
    system = "H%d" % n
    if rng.random() < 0.15:
        system = rng.choice(["hubbard10", "hubbard4x4", "hubbard6x6", "hubbard8x8", "hubbard14"])
    eps = rng.choice([1e-6, 1e-6, 1e-4])
    return dict(op=op, system=system, W=W, form=form, eps=eps, cps=cps, sweeps=rng.choice([2, 4, 8]) if op == "iter" else 0)


# ------------------------------------------------------------------------------------ inputs
_systems = {}


def _f0(x):
    """Boys function F0."""
    y = torch.clamp(x, min=1e-8)
    return torch.where(x < 1e-8, 1.0 - x / 3.0, 0.5 * torch.sqrt(math.pi / y) * torch.erf(torch.sqrt(y)))


def _chain(n, spacing=1.8):
    """Linear H_n, STO-3G 1s functions, closed-form s-Gaussian integrals in Loewdin orbitals, the
    two-electron integrals in the 8-fold packed form."""
    ex = torch.tensor(S.STO3G_H_EXP, dtype=torch.float64)
    d = torch.tensor(S.STO3G_H_COEF, dtype=torch.float64) * (2.0 * ex / math.pi) ** 0.75
    a, b = ex[:, None], ex[None, :]
    p = (a + b).reshape(-1)                                   # [9] primitive pairs
    dd = (d[:, None] * d[None, :]).reshape(-1)
    mu = (a * b / (a + b)).reshape(-1)
    frac = (b / (a + b)).expand(3, 3).reshape(-1)
    sites = torch.arange(n, dtype=torch.float64)
    r = spacing * (sites[None, :] - sites[:, None])[..., None]    # B - A
    K = dd * torch.exp(-mu * r * r)
    ov = (math.pi / p) ** 1.5
    Sm = (K * ov).sum(-1)
    T = (K * mu * (3.0 - 2.0 * mu * r * r) * ov).sum(-1)
    P = spacing * sites[:, None, None] + frac * r                 # [n, n, 9]
    V = torch.zeros(n, n, dtype=torch.float64)
    for c in range(n):
        V -= (K * 2.0 * math.pi / p * _f0(p * (P - spacing * c) ** 2)).sum(-1)
    # (mu nu|la si) depends on the two pair lengths and the offset alone: a small table, gathered
    D = min(n - 1, 24)
    Kl, sh = K[0, :D + 1], spacing * torch.arange(D + 1, dtype=torch.float64)[:, None] * frac
    off = spacing * torch.arange(-(n - 1), n, dtype=torch.float64)
    g = lambda t, *shape: t.reshape(*shape).to(DEV)  # noqa: E731
    pa, qa = g(p, 1, 1, 1, 9, 1), g(p, 1, 1, 1, 1, 9)
    tab = torch.empty(D + 1, D + 1, 2 * n - 1, dtype=torch.float64, device=DEV)
    for x in range(D + 1):
        x2 = (g(sh[x], 1, 1, 1, 9, 1) - g(off, 1, 1, -1, 1, 1) - g(sh, 1, D + 1, 1, 1, 9)) ** 2
        v = 2.0 * math.pi ** 2.5 / (pa * qa * torch.sqrt(pa + qa)) * _f0(pa * qa / (pa + qa) * x2)
        tab[x] = (v * g(Kl[x], 1, 1, 1, 9, 1) * g(Kl, 1, D + 1, 1, 1, 9)).sum((-1, -2))[0]
    i = torch.arange(n, device=DEV)
    lo, ln = torch.minimum(i[:, None], i[None, :]), (i[:, None] - i[None, :]).abs()
    keep = (ln <= D).reshape(-1)
    lo, ln = lo.reshape(-1), torch.clamp(ln, max=D).reshape(-1)
    E = torch.empty(n * n, n * n, dtype=torch.float64, device=DEV)
    for k in range(0, n * n, 2048):
        s = slice(k, k + 2048)
        E[s] = tab[ln[s, None], ln[None, :], lo[None, :] - lo[s, None] + (n - 1)] * (keep[s, None] & keep[None, :])
    w, U = torch.linalg.eigh(Sm)
    X = (U * w ** -0.5) @ U.T
    h1 = X.T @ (T + V) @ X
    Xg = X.to(DEV)
    E = E.view(n, n, n * n)
    E = torch.matmul(Xg.T, torch.matmul(Xg.T, E.reshape(n, -1)).view(n, n, n * n))
    E = torch.matmul(Xg.T, torch.matmul(E.view(n * n, n, n), Xg)).view(n * n, n * n)
    pq = torch.tril_indices(n, n, device=DEV)
    pq = pq[0] * n + pq[1]
    E = E[pq][:, pq]
    t = torch.tril_indices(pq.numel(), pq.numel(), device=DEV)
    packed = E[t[0], t[1]].cpu().numpy()
    del E, t
    torch.cuda.empty_cache()
    core = sum((n - k) / (spacing * k) for k in range(1, n))
    return S.System("H%d" % n, n, (n + 1) // 2, n // 2, (0.5 * (h1 + h1.T)).numpy(), packed, core,
                    dict(spacing=spacing, basis="sto-3g", orbitals="lowdin"))


def _system(name):
    if name not in _systems:
        if len(_systems) > 8:
            _systems.clear()
        _systems[name] = _chain(int(name[1:])) if name[0] == "H" else S.named_system(name)
    return _systems[name]


def _rows(C, W, gen):
    """W draws of n rows of C (M x n) with probability proportional to det(C[rows])^2 (sequential
    sampling of the projection determinantal point process), sorted: the typical starting
    determinants the framework's own init_occupations gives, drawn on the GPU."""
    n = C.shape[1]
    Q = torch.as_tensor(np.linalg.qr(C)[0], device=DEV)
    left = (Q * Q).sum(1).expand(W, -1).clone()
    basis = torch.zeros(W, n, n, dtype=torch.float64, device=DEV)
    rows = torch.empty(W, n, dtype=torch.int64, device=DEV)
    at = torch.arange(W, device=DEV)
    for k in range(n):
        c = torch.cumsum(left.clamp(min=0.0), 1)
        u = torch.rand(W, 1, dtype=torch.float64, device=DEV, generator=gen) * c[:, -1:]
        i = (c <= u).sum(1).clamp(max=C.shape[0] - 1)
        rows[:, k] = i
        v = Q[i].clone()
        for _ in range(2 if k else 0):
            v -= torch.bmm(torch.bmm(v[:, None], basis[:, :k].transpose(1, 2)), basis[:, :k])[:, 0]
        v /= torch.linalg.norm(v, dim=1, keepdim=True)
        basis[:, k] = v
        left -= (v @ Q.T) ** 2
        left[at, i] = 0.0
    return rows.sort(1).values


def _parts(case, seed, name, shift=0):
    """Hamiltonian, seeded parameters, seeded starting determinants and correlators of one system."""
    sy = _system(name)
    prm = S.make_params(sy, seed=seed + shift)
    gen = torch.Generator(device=DEV).manual_seed(1000003 * (seed + shift) + 17)
    occ = torch.cat([_rows(C, case["W"], gen) for C in (prm.C_alpha, prm.C_beta)], 1)
    cps = S.make_cps(sy, seed=seed + shift) if case["cps"] else None
    return sy, prm, occ.cpu().numpy().astype(np.uint16), cps, gen


def _weights(case, gen):
    """Residence times and energies as a sweep leaves them: positive with a long tail, and spread by
    a few per cent around the mean."""
    W = case["W"]
    t = 0.02 * torch.empty(W, dtype=torch.float64, device=DEV).exponential_(1.0, generator=gen)
    e = -20.0 + torch.randn(W, dtype=torch.float64, device=DEV, generator=gen)
    return t, e


def _engine(case, seed, name, shift=0):
    sy, prm, occ, cps, gen = _parts(case, seed, name, shift)
    eng = vmc.Engine(sy, prm, occ, eps=case["eps"], precision=vmc.VMC_MIXED if case["form"] == "mixed" else vmc.VMC_FP64,
                     cps=cps)
    return eng, gen


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        engs = [_engine(case, seed, name, 7919 * k)[0] for k, name in enumerate(case["system"].split())]
        bat = vmc.Batch(engs)
        bat.autotune()                      # as the benchmark does before it samples
        return dict(op=op, bat=bat, engs=engs, seed=seed, sweeps=case["sweeps"])
    eng, gen = _engine(case, seed, case["system"])
    st = dict(op=op, eng=eng, seed=seed, k=0)
    if op in ("eloc", "iter") and not case["cps"]:
        vmc.Batch([eng]).autotune()         # as the optimisation command line does
    if op == "grad":
        st["t"], st["e"] = _weights(case, gen)
        st["sums"] = torch.zeros(2 * eng.n_params + 2, dtype=torch.float64, device=DEV)
    if op == "logpsi":
        st["w"] = _weights(case, gen)[0]
        st["leaves"] = [x.detach().clone().requires_grad_(True) for x in (eng.J, eng.Ca, eng.Cb)]
    if op == "iter":
        st["opt"], st["sweeps"] = O.OptState.fresh(eng), case["sweeps"]
    return st


# ------------------------------------------------------------------------------------- the calls
def _tables(eng):
    w = eng.walkers
    return dict(G=w.G, AinvT=w.AinvT, S=w.S, F=w.F)


def run(st):
    op = st["op"]
    if op == "batch":
        out = {}
        for k in range(st["sweeps"]):
            st["bat"].local_energy()
            st["bat"].ctmc_step(st["seed"] + k)
        for k, e in enumerate(st["engs"]):
            e.refresh()
            out[str(k)] = dict(e_loc=e.e_loc, t_res=e.t_res, moves=e.moves, occ=e.walkers.occ_bits, G=e.walkers.G)
        return out
    eng = st["eng"]
    if op == "eloc":
        e, t = eng.local_energy()
        return dict(e_loc=e, t_res=t)
    if op == "sweep":
        e, t = eng.local_energy()
        moves = eng.ctmc_step(st["seed"])
        st["k"] += 1
        if st["k"] % RECOMPUTE == 0:
            eng.refresh()
        w = eng.walkers
        return dict(e_loc=e, t_res=t, moves=moves, occ=w.occ_bits, e_diag=w.e_diag, **_tables(eng))
    if op == "refresh":
        eng.refresh()
        return _tables(eng)
    if op == "grad":
        n, red = eng.n_params, st["sums"].zero_()
        vmc.vmc_accumulate_gradient(eng.ctx, eng.walkers.struct(), st["t"], st["e"], eng.split(red[:n]),
                                    eng.split(red[n:2 * n]), red[2 * n:])
        return dict(AO=red[:n], AEO=red[n:2 * n], sums=red[2 * n:])
    if op == "logpsi":
        out = vmc.LogPsi.apply(*st["leaves"], eng)
        g = torch.autograd.grad(out, st["leaves"], st["w"])
        return dict(log_psi=out.detach(), dJ=g[0], dCa=g[1], dCb=g[2])
    it = O.optimize(eng, 1, st["sweeps"], seed=st["seed"], alpha1=0.001, state=st["opt"])[0]
    return dict(energy=it.energy, t_sum=it.t_sum, grad_norm=it.grad_norm, p=eng.p, m=st["opt"].m, v=st["opt"].v,
                occ=eng.walkers.occ_bits, moves=eng.moves, e_diag=eng.walkers.e_diag)


# ------------------------------------------------------------------------------------- the work
def _one(case, name):
    """Bytes and operations of every step for one system: tables, lists and sums, once each."""
    W, M = case["W"], _size(name)
    n = (M + 1) // 2 if name[0] == "H" else M // 2
    nb = M // 2
    r = 4 if case["form"] == "mixed" else 8
    lists = name[0] == "H"
    loose = 0.35 if case["eps"] > 1e-5 else 1.0
    singles = (22.0 if lists else 4.0) * M * loose
    entries = (1000.0 if lists else 0.0) * M * loose            # stored doubles
    moves = ((95.0 if lists else 1.0) * M) * loose              # free single and double moves
    tabs = W * r * ((M - n) * n + (M - nb) * nb)
    inv = W * r * (n * n + nb * nb)
    small = W * (r * 2 * M + 4 * M + 16)
    fock = W * r * 2 * singles
    par = 8.0 * (4 * M * M + M * (n + nb))
    cube = W * (float(n) ** 3 + float(nb) ** 3)
    eloc = (tabs + small + W * r * singles / 4 + 4 * r * entries, W * moves * (60.0 if case["cps"] else 8.0))
    move = (2 * (tabs + inv + fock + small), 2.0 * (tabs + inv) / r * 2)
    grad = (inv + W * M + 2 * par, 2.0 * 2 * (W * (n + nb) ** 2 / 2 + inv / r))
    back = (inv + tabs + small + (fock if r == 4 else 0) + par, 2.0 * 2 * cube)
    logp = (W * (n + nb) * 2.0 + par, 2.0 / 3.0 * cube)
    return dict(eloc=eloc, move=move, grad=grad, back=back, logp=logp, par=(4 * par, 8 * par / 8))


def _size(name):
    if name[0] == "H":
        return int(name[1:])
    return math.prod(int(x) for x in name[len("hubbard"):].split("x"))


def work(case):
    op, k = case["op"], max(1, case["sweeps"])
    steps = dict(eloc={"eloc": 1}, sweep={"eloc": 1, "move": 1, "back": 1.0 / RECOMPUTE}, refresh={"back": 1},
                 grad={"grad": 1}, logpsi={"logp": 1, "grad": 0.5}, batch={"eloc": k, "move": k, "back": 1},
                 iter={"eloc": k, "move": k, "grad": k, "back": 1, "par": 1})[op]
    by = fl = 0.0
    for name in case["system"].split():
        one = _one(case, name)
        by += sum(v * one[s][0] for s, v in steps.items())
        fl += sum(v * one[s][1] for s, v in steps.items())
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------------------- 64-bit results
def _dense(sy):
    """(pq|rs) as a dense tensor on the GPU."""
    M = sy.M
    if sy.eri.size == M ** 4:
        return torch.as_tensor(sy.eri, device=DEV).view(M, M, M, M)
    i = torch.arange(M, device=DEV)
    hi, lo = torch.maximum(i[:, None], i[None, :]), torch.minimum(i[:, None], i[None, :])
    pair = (hi * (hi + 1) // 2 + lo).reshape(-1)
    v = torch.as_tensor(sy.eri, device=DEV)
    E = torch.empty(M * M, M * M, dtype=torch.float64, device=DEV)
    for k in range(0, M * M, 4096):
        A = torch.maximum(pair[k:k + 4096, None], pair[None, :])
        B = torch.minimum(pair[k:k + 4096, None], pair[None, :])
        E[k:k + 4096] = v[A * (A + 1) // 2 + B]
    return E.view(M, M, M, M)


class _Exact:
    """The walkers' tables and sums in 64 bits, with plain torch operations."""

    def __init__(self, case, seed):
        self.sy, prm, occ, self.cps, self.gen = _parts(case, seed, case["system"])
        self.case, self.M, self.n = case, self.sy.M, (self.sy.n_alpha, self.sy.n_beta)
        J = torch.as_tensor(prm.J, device=DEV)
        self.J = torch.triu(J) + torch.triu(J, 1).T
        self.C = [torch.as_tensor(c, device=DEV) for c in (prm.C_alpha, prm.C_beta)]
        o = torch.as_tensor(occ.astype(np.int64), device=DEV)
        self.occ = [o[:, :self.n[0]], o[:, self.n[0]:]]
        self.N = torch.zeros(case["W"], 2 * self.M, dtype=torch.float64, device=DEV)
        for s in (0, 1):
            self.N.scatter_(1, self.occ[s] + s * self.M, 1.0)

    def inverse(self, s, w):
        return torch.linalg.inv(self.C[s][self.occ[s][w]])          # rows x, columns c

    def sums(self, w=slice(None)):
        N = self.N[w]
        return N @ self.J - N * torch.diagonal(self.J)

    def chunks(self, k):
        return [slice(a, min(a + k, self.case["W"])) for a in range(0, self.case["W"], k)]

    def virt(self, s):
        n = self.N[:, s * self.M:(s + 1) * self.M]
        return torch.argsort(n, dim=1, stable=True)[:, :self.M - self.n[s]]

    def tables(self):
        G, A = [], []
        for w in self.chunks(4096):
            g, a = [], []
            for s in (0, 1):
                inv = self.inverse(s, w)
                a.append(inv.transpose(1, 2).reshape(inv.shape[0], -1))
                g.append(torch.bmm(self.C[s][self.virt(s)[w]], inv).reshape(inv.shape[0], -1))
            G.append(torch.cat(g, 1))
            A.append(torch.cat(a, 1))
        return torch.cat(G).reshape(-1), torch.cat(A).reshape(-1)

    def gradient(self, weights):
        """For each weight: sum_w c_w d ln psi / d (J, C_alpha, C_beta)."""
        dC = [[torch.zeros_like(c) for c in self.C] for _ in weights]
        for w in self.chunks(4096):
            for s in (0, 1):
                a = self.inverse(s, w).transpose(1, 2)                # [walker, column, x]
                for k, c in enumerate(weights):
                    v = (c[w, None, None] * a).reshape(-1, self.n[s])
                    dC[k][s].index_add_(0, self.occ[s][w].reshape(-1), v)
        return [(torch.triu(self.N.T @ (c[:, None] * self.N)), *dC[k]) for k, c in enumerate(weights)]

    def log_psi(self):
        out = 0.5 * ((self.N @ self.J) * self.N).sum(1) + 0.5 * self.N @ torch.diagonal(self.J)
        for s in (0, 1):
            for w in self.chunks(4096):
                out[w] += torch.linalg.slogdet(self.C[s][self.occ[s][w]])[1]
        return out

    def energy(self):
        """Screened local energy and residence time: every single and double whose bound or
        magnitude exceeds eps, from the integrals."""
        M, eps, E = self.M, self.case["eps"], _dense(self.sy)
        h = torch.as_tensor(self.sy.h1, device=DEV)
        i = torch.arange(M, device=DEV)
        co = E[:, :, i, i]                                            # (ai|kk)
        ex = E.permute(0, 3, 1, 2)[:, :, i, i]                        # (ak|ki)
        Tjk, d = co - ex, torch.diagonal(self.J)
        bound = h.abs() + Tjk.abs().sum(2) + co.abs().sum(2)
        bound[i, i] = 0.0
        a1, i1 = torch.nonzero(bound > eps, as_tuple=True)
        opp, same = [], []
        for p in range(M):                                            # (ap|bq)
            A = E[:, p]                                               # [a, b, q]
            ok = A.abs() > eps
            ok[p] = False
            ok[:, i, i] = False
            a, b, q = torch.nonzero(ok, as_tuple=True)
            opp.append(torch.stack([a, torch.full_like(a, p), b, q]))
            X = A - A.permute(1, 0, 2)                                # (ap|bq) - (aq|bp)
            X = torch.where((i[:, None, None] < i[None, :, None]) & (i[None, None, :] > p), X, 0.0)
            X[p] = 0.0
            X[:, p] = 0.0
            X[:, i, i] = 0.0
            X[i, :, i] = 0.0
            a, b, q = torch.nonzero(X.abs() > eps, as_tuple=True)
            same.append(torch.stack([a, torch.full_like(a, p), b, q]))
        opp, same = torch.cat(opp, 1), torch.cat(same, 1)

        def factor(A, I, B, Q):                                       # Jastrow part that no sum holds
            J = self.J
            return torch.exp(-J[A, I] - J[A, Q] - J[B, I] - J[B, Q] + J[A, B] + J[I, Q] + d[A] + d[B] - d[I] - d[Q])

        a, p, b, q = opp
        v2, w2 = E[a, p, b, q], factor(a, p, b + M, q + M)
        f2 = (a * M + p, b * M + q)
        a, p, b, q = same
        v1 = E[a, p, b, q] - E[a, q, b, p]
        w1 = [factor(a + s * M, p + s * M, b + s * M, q + s * M) for s in (0, 1)]
        f1 = (a * M + p, b * M + q, a * M + q, b * M + p)
        w0 = [torch.exp(-self.J[a1 + s * M, i1 + s * M] + d[a1 + s * M] - d[i1 + s * M]) for s in (0, 1)]
        f0 = a1 * M + i1
        tj, tjk = co[a1, i1], Tjk[a1, i1]                             # [single, k]
        dg_j, dg_k = E[i, i][:, i, i], E.permute(0, 3, 1, 2)[i, i][:, i, i]
        hd = torch.diagonal(h)
        e_out, t_out = [], []
        for w in self.chunks(max(16, min(2048, 30_000_000 // max(1, opp.shape[1] + same.shape[1])))):
            N = self.N[w]
            Na, Nb = N[:, :M], N[:, M:]
            k = N.shape[0]
            expS = torch.exp(self.sums(w))
            R = []
            for s in (0, 1):                                          # G[a, i] exp(S_a - S_i), 0 unless a empty, i filled
                x = torch.bmm(self.C[s].expand(k, -1, -1), self.inverse(s, w))
                n, es = N[:, s * M:(s + 1) * M], expS[:, s * M:(s + 1) * M]
                full = torch.zeros(k, M, M, dtype=torch.float64, device=DEV)
                full.scatter_(2, self.occ[s][w][:, None, :].expand(-1, M, -1), x)
                R.append((full * ((1 - n) * es)[:, :, None] / es[:, None, :]).view(k, -1))
            e = self.sy.e_core + (Na + Nb) @ hd + ((Na + Nb) @ dg_j * (Na + Nb)).sum(1) / 2
            e -= ((Na @ dg_k * Na).sum(1) + (Nb @ dg_k * Nb).sum(1)) / 2
            rate = torch.zeros_like(e)
            for s, (n, o) in enumerate(((Na, Nb), (Nb, Na))):
                r = R[s][:, f0] * w0[s]
                F = h[a1, i1] + n @ tjk.T + o @ tj.T
                e += (r * F).sum(1)
                rate += r.abs().sum(1)
                r = (R[s][:, f1[0]] * R[s][:, f1[1]] - R[s][:, f1[2]] * R[s][:, f1[3]]) * w1[s]
                e += r @ v1
                rate += r.abs().sum(1)
            r = R[0][:, f2[0]] * R[1][:, f2[1]] * w2
            e_out.append(e + r @ v2)
            t_out.append(1.0 / (rate + r.abs().sum(1)))
        return torch.cat(e_out), torch.cat(t_out)


def exact(case, seed):
    op = case["op"]
    if op in ("batch", "iter") or case["cps"]:
        return None
    x = _Exact(case, seed)
    if op == "eloc":
        e, t = x.energy()
        return dict(e_loc=e, t_res=t)
    if op == "sweep":                        # what follows the chosen move has no value of its own
        e, t = x.energy()
        return dict(e_loc=e, t_res=t, moves=None, occ=None, e_diag=None, G=None, AinvT=None, S=None, F=None)
    if op == "refresh":
        G, A = x.tables()
        return dict(G=G, AinvT=A, S=x.sums().reshape(-1), F=None)
    if op == "grad":
        t, e = _weights(case, x.gen)
        (g0, g1), sums = x.gradient([t, t * e]), torch.stack([t.sum(), (t * e).sum()])
        return dict(AO=torch.cat([y.reshape(-1) for y in g0]), AEO=torch.cat([y.reshape(-1) for y in g1]), sums=sums)
    w = _weights(case, x.gen)[0]
    g = x.gradient([w])[0]
    return dict(log_psi=x.log_psi(), dJ=g[0], dCa=g[1], dCb=g[2])
