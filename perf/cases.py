"""Performance cases of the MLCC3 triples library: the calls a response calculation makes.

A case is one pass through a public entry point (`paper_2202_08612_gb300.binding`,
`.autograd`, `.cnto`) on one system of N_O / N_V occupied / virtual, n_o / n_v active orbitals and
N_J Cholesky vectors, in one of the two precisions:

  ground      one ground-state iteration: the integral build for new amplitudes, then Omega
  davidson    one iteration of an eigenvalue solver: rho = A R and sigma = A^T L of `vec` vectors
  adjoint     rho through the torch.autograd Function and its backward pass
  densities   the transition densities of `vec` states (with D^{0-0}) and their oscillator strengths
  sweep       rho of `vec` vectors of several uneven systems in one captured CUDA graph
  cnto        the CNTO matrices M and N of one state in full doubles storage
  gemm        C = A B^T to FP64 accuracy on the tensor cores (`slices` digits)

Inputs follow the repository's synthetic recipe (`synth.py`: uniform orbital energies, Gaussian
Cholesky vectors, MP2-like doubles scaled to a molecule's norm, singles-dominated trial vectors),
drawn on the GPU.
"""
import math

import numpy as np
import torch

from paper_2202_08612_gb300 import autograd, binding, cnto

F64 = torch.float64

# Leading operation counts of the quantities in units of N_V n_v^3 n_o^3 (the paper's Sec. 3).
UNITS_OMEGA, UNITS_RHO, UNITS_SIGMA, UNITS_LEFT, UNITS_RIGHT = 4, 8, 8, 10, 16

# The uneven systems of the sweep, (n_o, n_v, N_V) with N_O = n_o + 8: the first ones of the
# benchmark's six.
SWEEP = [(8, 40, 120), (11, 60, 216), (14, 80, 312)]


def _system(op, prec, NO, NV, no, nv, NJ, vec=1, core=False):
    return {"op": op, "precision": prec, "NO": NO, "NV": NV, "no": no, "nv": nv, "NJ": NJ, "vec": vec,
            "core": core}


def listed():
    def named(name, case):
        return dict(case, name=name)
    return [
        # the smallest system of the tests: a call is launches and host work
        named("davidson_fp64_tiny", _system("davidson", "fp64", 6, 24, 4, 8, 72)),
        # the differentiable transformation of the FP64 path at the size it is quoted on
        named("adjoint_fp64", _system("adjoint", "fp64", 20, 200, 12, 60, 600)),
        # FP64 densities of a small molecule, no extent a multiple of a tile
        named("densities_fp64_ragged", _system("densities", "fp64", 13, 101, 7, 37, 303)),
        # a ground-state iteration: new t1 and t2, so new integrals each time
        named("ground_split", _system("ground", "split", 20, 200, 12, 60, 600)),
        # an iteration of the eigenvalue solver with two trial vectors at the benchmark's small size
        named("davidson_split", _system("davidson", "split", 20, 200, 12, 60, 600, vec=2)),
        # densities and f of one state, ragged extents
        named("densities_split_ragged", _system("densities", "split", 19, 187, 11, 57, 561)),
        # the middle-sized molecule of the configurations, its triples blocks in chunks
        named("davidson_split_large", _system("davidson", "split", 40, 500, 20, 120, 1500)),
        # two states at the virtual extent of the largest molecule (150), few occupied orbitals
        named("densities_split_wide", _system("densities", "split", 28, 260, 6, 150, 780, vec=2)),
        # a core-excited state: the skip rule leaves the batches that hold the core orbital
        named("davidson_split_core", _system("davidson", "split", 24, 240, 10, 80, 720, core=True)),
        # trial vectors of several systems in one graph
        named("sweep_split", {"op": "sweep", "precision": "split", "systems": 3, "vec": 4}),
        # the choice of the active space, once per calculation, at the size of a small molecule
        named("cnto", {"op": "cnto", "precision": "fp64", "NO": 39, "NV": 263}),
        # the FP64-accurate tensor-core product at the benchmark's size
        named("gemm_fp64emu", {"op": "gemm", "precision": "fp64", "M": 4096, "N": 4096, "K": 4096, "slices": 5}),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    while True:
        op = rng.choice(["ground", "davidson", "davidson", "adjoint", "densities", "densities", "sweep", "cnto",
                         "gemm"])
        if op == "sweep":
            case = {"op": op, "precision": rng.choice(["fp64", "split"]), "systems": rng.randint(1, 3),
                    "vec": rng.randint(1, 6)}
            if work(case)["flops"] <= (8e11 if case["precision"] == "fp64" else 6e13):
                return case
            continue
        if op == "cnto":
            return {"op": op, "precision": "fp64", "NO": _log(rng, 6, 48), "NV": _log(rng, 24, 263)}
        if op == "gemm":
            return {"op": op, "precision": "fp64", "M": _log(rng, 60, 4096), "N": _log(rng, 60, 4096),
                    "K": _log(rng, 60, 4096), "slices": rng.randint(3, 6)}
        prec = rng.choice(["fp64", "split"])
        no = _log(rng, 3, 20)
        NO = no + _log(rng, 2, 22)
        nv = _log(rng, 8, 150)
        NV = nv + _log(rng, 8, 380)
        case = _system(op, prec, NO, NV, no, nv, 3 * NV, vec=rng.randint(1, 3) if op in ("davidson", "densities") else 1,
                       core=op == "davidson" and rng.random() < 0.25)
        flops = work(case)["flops"]
        if 5e6 <= flops <= (8e11 if prec == "fp64" else 6e13):
            return case


def _dims(case):
    return case["NO"], case["NV"], case["no"], case["nv"], case["NJ"]


def work(case):
    op = case["op"]
    if op == "cnto":
        NO, NV = case["NO"], case["NV"]
        # two symmetric Gram matrices: the upper triangle's multiply-adds of each
        n = float((NO * NV) ** 2)
        return {"bytes": 8.0 * n, "flops": n * (NO + 1) + n * (NV + 1)}
    if op == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 8.0 * (M * K + N * K + M * N), "flops": 2.0 * M * N * K}
    if op == "sweep":
        b = f = 0.0
        for no, nv, NV in SWEEP[:case["systems"]]:
            w = work(_system("rho", case["precision"], no + 8, NV, no, nv, 3 * NV, vec=case["vec"]))
            b, f = b + w["bytes"], f + w["flops"]
        return {"bytes": b, "flops": f}
    NO, NV, no, nv, NJ = _dims(case)
    vec = case["vec"]
    blk, nmo = float(no * nv * NO * NV), NO + NV
    vector = NO * NV + blk
    held = NJ * nmo * nmo + blk  # Cholesky vectors and amplitudes
    if op == "ground":
        units, words = UNITS_OMEGA, held + blk + vector
    elif op == "rho":
        units, words = UNITS_RHO * vec, held + 2 * vec * vector
    elif op in ("davidson", "adjoint"):
        units, words = (UNITS_RHO + UNITS_SIGMA) * vec, held + 4 * vec * vector
    else:
        units, words = UNITS_LEFT + (UNITS_LEFT + UNITS_RIGHT) * vec, held + blk + (1 + 2 * vec) * vector + 3 * vec * nmo * nmo
    triples = float(no ** 3)
    if case["core"]:  # the ordered triples that hold the core orbital
        triples -= float((no - 1) ** 3)
    return {"bytes": 8.0 * words, "flops": units * NV * float(nv) ** 3 * triples}


# ---- inputs ----------------------------------------------------------------------------------
def _uniform(gen, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, dtype=F64, device=gen.device, generator=gen)


def _normal(gen, *shape):
    return torch.randn(*shape, dtype=F64, device=gen.device, generator=gen)


def _weights(no, nv, NO, NV, dev):
    """1/2 on the doubles that the active-pair block stores twice, else 1."""
    w = torch.ones(no, nv, NO, NV, dtype=F64, device=dev)
    w[:, :, :no, :nv] = 0.5
    i, a = torch.arange(no, device=dev)[:, None], torch.arange(nv, device=dev)[None, :]
    w[i, a, i, a] = 1.0
    return w


def _symmetrize(x, no, nv):
    aa = x[:, :, :no, :nv].clone()
    x[:, :, :no, :nv] = 0.5 * (aa + aa.permute(2, 3, 0, 1))
    return x


def _make_system(case, gen):
    """Orbital energies, Cholesky vectors, amplitudes, and R, L, multipliers, dipole integrals."""
    NO, NV, no, nv, NJ = _dims(case)
    nmo, dev = NO + NV, gen.device
    eps = torch.cat([_uniform(gen, -1.5, -0.3, NO), _uniform(gen, 0.1, 3.0, NV)])
    if case["core"]:
        eps[0] = -10.0
    chol = _normal(gen, NJ, nmo, nmo).mul_(0.05).triu_()
    chol += chol.triu(1).transpose(1, 2)
    t1 = 0.01 * _normal(gen, NV, NO)
    vo = chol[:, NO:, :NO]
    act = vo[:, :nv, :no]
    den = (eps[:no, None, None, None] + eps[None, None, :NO, None] - eps[None, NO:NO + nv, None, None]
           - eps[None, None, None, NO:])
    t2c = torch.einsum("Jai,JDL->iaLD", act, vo) / den
    t2x = torch.einsum("JaL,JDi->iaLD", vo[:, :nv], vo[:, :, :no]) / den
    scale = min(1.0, 0.3 / float(t2c.norm()))  # a closed-shell molecule's doubles norm
    chol *= math.sqrt(scale)
    sys = {"eps": eps, "chol": chol, "t1": t1, "t2c": (t2c * scale).contiguous(), "t2x": (t2x * scale).contiguous()}

    w = _weights(no, nv, NO, NV, dev)
    core = torch.zeros(NO, dtype=torch.bool, device=dev)
    core[0] = case["core"]

    def project(x1, x2):
        if not case["core"]:
            return x1, x2
        keep = core[:no, None, None, None] | core[None, None, :, None]
        return x1 * core, x2 * keep

    R1, R2, L1, L2 = [], [], [], []
    for _ in range(case["vec"]):
        x1, x2 = project(_normal(gen, NV, NO), _symmetrize(_normal(gen, no, nv, NO, NV), no, nv))
        x1 = x1 * math.sqrt(0.95 / float((x1 * x1).sum()))
        x2 = x2 * math.sqrt(0.05 / float((w * x2 * x2).sum()))
        y1 = x1 + 0.3 / math.sqrt(x1.numel()) * _normal(gen, NV, NO)
        y2 = x2 + 0.3 / math.sqrt(x2.numel()) * _symmetrize(_normal(gen, no, nv, NO, NV), no, nv)
        y1, y2 = project(y1, y2)
        s = float((y1 * x1).sum() + (w * y2 * x2).sum())
        R1.append(x1), R2.append(x2), L1.append(y1 / s), L2.append(y2 / s)
    omega = [10.2] * case["vec"] if case["core"] else _uniform(gen, 0.3, 0.6, case["vec"]).tolist()
    mu = 0.1 * _normal(gen, 3, nmo, nmo)
    sys.update(R1=torch.stack(R1), R2=torch.stack(R2), L1=torch.stack(L1), L2=torch.stack(L2), omega=omega,
               lam1=0.01 * _normal(gen, NV, NO), lam2=sys["t2c"].clone(), mu=0.5 * (mu + mu.transpose(1, 2)).contiguous(),
               core=core)
    return sys


def _generator(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(1_000_003 * int(seed) + 17)


def _context(case):
    NO, NV, no, nv, NJ = _dims(case)
    mask = None
    if case["core"]:
        mask = np.zeros(NO, dtype=np.uint8)
        mask[0] = 1
    ctx = binding.Context(NO, NV, no, nv, NJ, core_mask=mask,
                          precision=binding.MLCC3_FP64 if case["precision"] == "fp64" else binding.MLCC3_SPLIT_BF16X3)
    # several contexts share the card: a bound on the blocks each holds instead of half of what is free
    ctx.set_param("chunk_blocks", max(1, int(4e10 / (156 * nv ** 3))))
    return ctx


def _build(ctx, s):
    ctx.build_integrals(s["chol"], s["t1"], s["eps"], s["t2c"], s["t2x"])


def _reference_densities(s, NO):
    """Leading-order CCSD-level densities that f needs beside the triples parts."""
    nmo, n = s["eps"].numel(), len(s["omega"])
    D00 = torch.zeros(nmo, nmo, dtype=F64, device=s["eps"].device)
    D00.diagonal()[:NO] = 2.0
    Dm0, D0m = (torch.zeros(n, nmo, nmo, dtype=F64, device=D00.device) for _ in range(2))
    Dm0[:, :NO, NO:] = s["L1"].transpose(1, 2)
    D0m[:, NO:, :NO] = s["R1"]
    return D00, Dm0, D0m


def prepare(case, seed):
    gen, op = _generator(seed), case["op"]
    if op == "cnto":
        NO, NV = case["NO"], case["NV"]
        R1, R2 = _normal(gen, NV, NO), _normal(gen, NV * NO, NV * NO)
        R2 += R2.t().clone()
        R1 *= math.sqrt(0.95) / R1.norm()
        R2 *= math.sqrt(0.05) / R2.norm()
        return {"case": case, "R1": R1, "R2": R2.view(NV, NO, NV, NO)}
    if op == "gemm":
        M, N, K = case["M"], case["N"], case["K"]
        return {"case": case, "A": _normal(gen, M, K), "B": _normal(gen, N, K),
                "C": torch.empty(M, N, dtype=F64, device="cuda")}
    if op == "sweep":
        systems = []
        for no, nv, NV in SWEEP[:case["systems"]]:
            one = _system("rho", case["precision"], no + 8, NV, no, nv, 3 * NV, vec=case["vec"])
            s = _make_system(one, gen)
            s["ctx"] = _context(one)
            _build(s["ctx"], s)
            for name in ("R1", "R2"):
                s["rho" + name[1]] = torch.empty_like(s[name])
            systems.append(s)
        # without the tuner, whose choices (and with them the order of sums) follow its own timings
        sweep = binding.Sweep([s["ctx"] for s in systems], tune=False)
        for q, s in enumerate(systems):
            sweep.set_system(q, s["R1"], s["R2"], s["rho1"], s["rho2"])
        return {"case": case, "sweep": sweep, "systems": systems, "omega": [w for s in systems for w in s["omega"]]}
    s = _make_system(case, gen)
    s.update(case=case, ctx=_context(case))
    NO = case["NO"]
    if op == "ground":
        s.update(o1=torch.empty_like(s["t1"]), o2=torch.empty_like(s["t2c"]))
        return s
    _build(s["ctx"], s)
    if op == "davidson":
        s.update({name: torch.empty_like(s[like]) for name, like in
                  (("rho1", "R1"), ("rho2", "R2"), ("sigma1", "L1"), ("sigma2", "L2"))})
    elif op == "adjoint":
        s.update(x1=s["R1"][0].clone().requires_grad_(), x2=s["R2"][0].clone().requires_grad_())
    else:
        s["D00_in"], s["Dm0_in"], s["D0m_in"] = _reference_densities(s, NO)
        s.update(D00=torch.empty_like(s["D00_in"]), Dm0=torch.empty_like(s["Dm0_in"]), D0m=torch.empty_like(s["D0m_in"]))
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "cnto":
        return cnto.cnto_matrices(s["R1"], s["R2"])
    if op == "gemm":
        binding.fp64emu_gemm(s["A"], s["B"], s["C"], slices=case["slices"])
        return s["C"]
    if op == "sweep":
        s["sweep"].run(s["omega"])
        return [(y["rho1"], y["rho2"]) for y in s["systems"]]
    ctx = s["ctx"]
    if op == "ground":
        _build(ctx, s)
        ctx.triples_omega(s["o1"], s["o2"])
        return s["o1"], s["o2"]
    if op == "davidson":
        ctx.jacobian_right(s["omega"], s["R1"], s["R2"], s["rho1"], s["rho2"])
        ctx.jacobian_left(s["omega"], s["L1"], s["L2"], s["sigma1"], s["sigma2"])
        return s["rho1"], s["rho2"], s["sigma1"], s["sigma2"]
    if op == "adjoint":
        rho1, rho2 = autograd.jacobian_right(ctx, s["omega"][0], s["x1"], s["x2"])
        g1, g2 = torch.autograd.grad((rho1, rho2), (s["x1"], s["x2"]), (s["L1"][0], s["L2"][0]))
        return rho1.detach(), rho2.detach(), g1, g2
    ctx.transition_densities(s["omega"], s["lam1"], s["lam2"], s["R1"], s["R2"], s["L1"], s["L2"], s["D00_in"],
                             s["D00"], s["Dm0"], s["D0m"])
    right, left = s["D0m"] + s["D0m_in"], s["Dm0"] + s["Dm0_in"]
    f = [ctx.oscillator_strength(w, right[q], left[q], s["mu"]) for q, w in enumerate(s["omega"])]
    return s["D00"], s["Dm0"], s["D0m"], f


# ---- the same quantities from the equations, every sum over all ordered triples, in 64 bits -----
_PAIRS = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))
_ein = torch.einsum


class _Exact:
    """Triples quantities with triples tensors [i][j][k][a][b][c] and doubles X[A][I][B][J]."""

    def __init__(self, case, s):
        self.NO, self.NV, self.no, self.nv, _ = _dims(case)
        NO, NV, no, nv = self.NO, self.NV, self.no, self.nv
        self.s, self.dev = s, s["eps"].device
        self.blocked = s["core"][:no] if case["core"] else None
        t = torch.zeros(NO + NV, NO + NV, dtype=F64, device=self.dev)
        t[NO:, :NO] = s["t1"]
        one = torch.eye(NO + NV, dtype=F64, device=self.dev)
        self.mut = (one - t) @ s["mu"] @ (one + t)
        Lt = ((one - t) @ s["chol"]) @ (one + t)
        self.Loo, self.Lov, self.Lvo, self.Lvv = Lt[:, :NO, :NO], Lt[:, :NO, NO:], Lt[:, NO:, :NO], Lt[:, NO:, NO:]
        self.t2 = self.full(s["t2c"])
        self.tA, self.tB = self.views(self.t2)
        self.vVvo = _ein("JbD,Jck->bDck", self.Lvv[:, :nv], self.Lvo[:, :nv, :no])
        self.Oovo = _ein("JLj,Jck->Ljck", self.Loo[:, :, :no], self.Lvo[:, :nv, :no])
        self.Vvov = _ein("JDb,Jkc->Dbkc", self.Lvv[:, :, :nv], self.Lov[:, :no, :nv])
        self.oOov = _ein("JjL,Jkc->jLkc", self.Loo[:, :no], self.Lov[:, :no, :nv])
        self.ovov = _ein("Jjb,Jkc->jbkc", self.Lov[:, :no, :nv], self.Lov[:, :no, :nv])
        self.F = self.fock(s["t1"])
        eo, ev = s["eps"][:no], s["eps"][NO:NO + nv]
        self.eps3 = ((ev[:, None, None] + ev[None, :, None] + ev[None, None, :])[None, None, None]
                     - (eo[:, None, None] + eo[None, :, None] + eo[None, None, :])[:, :, :, None, None, None])
        self.tau = self.solve(self.w_term(self.tA, self.tB, self.vVvo, self.Oovo), 0.0)

    def full(self, blk):
        X = torch.zeros(self.NV, self.NO, self.NV, self.NO, dtype=F64, device=self.dev)
        b = blk.permute(1, 0, 3, 2)
        X[:self.nv, :self.no] = b
        X[:, :, :self.nv, :self.no] = b.permute(2, 3, 0, 1)
        return X

    def block(self, X):
        return X[:self.nv, :self.no].permute(1, 0, 3, 2).contiguous()

    def views(self, X):
        nv, no = self.nv, self.no
        return X[:nv, :no, :, :no].permute(1, 3, 0, 2), X[:nv, :no, :nv].permute(1, 0, 2, 3)

    def diagonal(self, X, factor):
        X = X.clone()
        a, i = torch.arange(self.NV, device=self.dev)[:, None], torch.arange(self.NO, device=self.dev)[None, :]
        X[a, i, a, i] *= factor
        return X

    @staticmethod
    def covariant(X):
        return (2.0 * X + X.permute(2, 1, 0, 3)) / 3.0

    def fock(self, x):
        no, nv = self.no, self.nv
        Lov = self.Lov
        y = 2.0 * _ein("Jkc,J->kc", Lov[:, :no, :nv], _ein("JLD,DL->J", Lov, x))
        return y - _ein("JkL,JLc->kc", _ein("JkD,DL->JkL", Lov[:, :no], x), Lov[:, :, :nv])

    @staticmethod
    def w_term(XA, XB, vVvo, Oovo):
        W = _ein("ijaD,bDck->ijkabc", XA, vVvo)
        W -= _ein("iabL,Ljck->ijkabc", XB, Oovo)
        return W

    def solve(self, W, omega, masked=False):
        X = torch.zeros(W.shape, dtype=F64, device=self.dev)
        for p in _PAIRS:  # the six permutations of the pairs (i,a), (j,b), (k,c)
            X += W.permute(*p, *(3 + q for q in p))
        X /= omega - self.eps3
        return self.mask(X) if masked else X

    def mask(self, X):
        if self.blocked is None:
            return X
        c = self.blocked
        return X * (c[:, None, None] | c[None, :, None] | c[None, None, :])[:, :, :, None, None, None]

    @staticmethod
    def contra(X):
        p = X.permute
        return (4.0 * X - 2.0 * p(0, 1, 2, 4, 3, 5) - 2.0 * p(0, 1, 2, 5, 4, 3) - 2.0 * p(0, 1, 2, 3, 5, 4)
                + p(0, 1, 2, 4, 5, 3) + p(0, 1, 2, 5, 3, 4))

    def back(self, Xt, F, oOov, Vvov):
        NO, NV, no, nv = self.NO, self.NV, self.no, self.nv
        Z = torch.zeros(NV, NO, NV, NO, dtype=F64, device=self.dev)
        Z[:nv, :no, :nv, :no] += 0.5 * _ein("ijkabc,kc->aibj", Xt, F)
        Z[:nv, :no, :nv] -= _ein("ijkabc,jLkc->aibL", Xt, oOov)
        Z[:nv, :no, :, :no] += _ein("ijkabc,Dbkc->aiDj", Xt, Vvov)
        return Z

    def singles(self, Xt):
        s1 = torch.zeros(self.NV, self.NO, dtype=F64, device=self.dev)
        s1[:self.nv, :self.no] = 0.5 * _ein("ijkabc,jbkc->ai", Xt, self.ovov)
        return s1

    def finish(self, Z):
        return self.block(self.covariant(self.diagonal(Z + Z.permute(2, 3, 0, 1), 0.5)))

    def omega(self):
        tt = self.contra(self.tau)
        return self.singles(tt), self.finish(self.back(tt, self.F, self.oOov, self.Vvov))

    def right(self, omega, R1, R2):
        no, nv = self.no, self.nv
        RA, RB = self.views(self.diagonal(self.full(R2), 2.0))
        R1o, R1v = R1[:, :no], R1[:nv]
        bD = -_ein("bM,JMD->JbD", R1v, self.Lov)
        ck = _ein("JcE,Ek->Jck", self.Lvv[:, :nv], R1o) - _ein("cM,JMk->Jck", R1v, self.Loo[:, :, :no])
        Lj = _ein("JLE,Ej->JLj", self.Lov, R1o)
        Uv = _ein("JbD,Jck->bDck", bD, self.Lvo[:, :nv, :no]) + _ein("JbD,Jck->bDck", self.Lvv[:, :nv], ck)
        Uo = _ein("JLj,Jck->Ljck", Lj, self.Lvo[:, :nv, :no]) + _ein("JLj,Jck->Ljck", self.Loo[:, :, :no], ck)
        W = self.w_term(RA, RB, self.vVvo, self.Oovo)
        W += self.w_term(self.tA, self.tB, Uv, Uo)
        return self.solve(W, omega, True), RA, RB

    def rho(self, omega, R1, R2):
        no, nv = self.no, self.nv
        Rt = self.contra(self.right(omega, R1, R2)[0])
        tt = self.contra(self.mask(self.tau))
        Z = self.back(Rt, self.F, self.oOov, self.Vvov)
        jL = _ein("JjD,DL->JjL", self.Lov[:, :no], R1)
        bD = -_ein("JLb,DL->JbD", self.Lov[:, :, :nv], R1)
        Lkc = self.Lov[:, :no, :nv]
        Z += self.back(tt, self.fock(R1), _ein("JjL,Jkc->jLkc", jL, Lkc), _ein("JbD,Jkc->Dbkc", bD, Lkc))
        return self.singles(Rt), self.finish(Z)

    def left(self, omega, L1, L2, masked=True):
        no, nv = self.no, self.nv
        Lc = self.covariant(self.full(L2))
        Q = 0.5 * _ein("ai,jbkc->ijkabc", L1[:nv, :no], self.ovov)
        Q += 0.5 * _ein("aibj,kc->ijkabc", Lc[:nv, :no, :nv, :no], self.F)
        Q -= _ein("aibL,jLkc->ijkabc", Lc[:nv, :no, :nv], self.oOov)
        Q += _ein("aiDj,Dbkc->ijkabc", Lc[:nv, :no, :, :no], self.Vvov)
        return self.solve(Q, omega, masked), Lc

    def sigma(self, omega, L1, L2):
        NO, NV, no, nv = self.NO, self.NV, self.no, self.nv
        Lt, Lc = self.left(omega, L1, L2)
        Lt = self.contra(Lt)
        S = torch.zeros(NV, NO, NV, NO, dtype=F64, device=self.dev)
        S[:nv, :no, :, :no] += _ein("ijkabc,bDck->aiDj", Lt, self.vVvo)
        S[:nv, :no, :nv] -= _ein("ijkabc,Ljck->aibL", Lt, self.Oovo)
        Y1 = _ein("ijkabc,ijaD->bDck", Lt, self.tA)
        Y2 = _ein("ijkabc,iabL->Ljck", Lt, self.tB)
        tt = self.contra(self.mask(self.tau))
        # everything that meets a four-index integral goes through its Cholesky factors
        Loo, Lov, Lvo, Lvv = self.Loo, self.Lov, self.Lvo, self.Lvv
        W = _ein("bDck,JbD->Jck", Y1, Lvv[:, :nv]) - _ein("Ljck,JLj->Jck", Y2, Loo[:, :, :no])
        bD = _ein("bDck,Jck->JbD", Y1, Lvo[:, :nv, :no])
        Lj = _ein("Ljck,Jck->JLj", Y2, Lvo[:, :nv, :no])
        s1 = torch.zeros(NV, NO, dtype=F64, device=self.dev)
        s1[:, :no] += _ein("Jck,JcE->Ek", W, Lvv[:, :nv]) - _ein("JLj,JLE->Ej", Lj, Lov)
        s1[:nv] -= _ein("Jck,JMk->cM", W, Loo[:, :, :no]) + _ein("JbD,JMD->bM", bD, Lov)
        Lkc = Lov[:, :no, :nv]
        Y3 = 0.5 * _ein("aibj,ijkabc->kc", Lc[:nv, :no, :nv, :no], tt)
        s1 += 2.0 * _ein("J,JLD->DL", _ein("kc,Jkc->J", Y3, Lkc), Lov)
        s1 -= _ein("JkL,JkD->DL", _ein("kc,JLc->JkL", Y3, Lov[:, :, :nv]), Lov[:, :no])
        P1 = _ein("aibL,ijkabc->jkcL", Lc[:nv, :no, :nv], tt)
        s1 -= _ein("JjL,JjD->DL", _ein("jkcL,Jkc->JjL", P1, Lkc), Lov[:, :no])
        P2 = _ein("aiDj,ijkabc->bDkc", Lc[:nv, :no, :, :no], tt)
        s1 -= _ein("JbD,JLb->DL", _ein("bDkc,Jkc->JbD", P2, Lkc), Lov[:, :, :nv])
        return s1, self.block(S + S.permute(2, 3, 0, 1))

    def density_left(self, Lt, L2):
        NO, no, nv = self.NO, self.no, self.nv
        D = torch.zeros(NO + self.NV, NO + self.NV, dtype=F64, device=self.dev)
        Lc = self.covariant(self.full(L2))
        D[:no, :no] -= 0.5 * _ein("ijlabc,ijkabc->kl", Lt, self.tau)
        D[:no, NO:NO + nv] += 0.5 * _ein("aibj,ijlabd->ld", Lc[:nv, :no, :nv, :no], self.contra(self.tau))
        D[:NO, NO:] -= _ein("jkbL,jkbD->LD", _ein("ijkabc,iacL->jkbL", Lt, self.tB), self.tA)
        D[NO:NO + nv, NO:NO + nv] += 0.5 * _ein("ijkabc,ijkabd->cd", Lt, self.tau)
        return D

    def densities(self, n):
        NO, no, nv, s = self.NO, self.no, self.nv, self.s
        R1, R2, w = s["R1"][n], s["R2"][n], s["omega"][n]
        lt = self.contra(self.left(0.0, s["lam1"], s["lam2"], False)[0])
        D00 = self.density_left(lt, s["lam2"])
        Dm0 = self.density_left(self.contra(self.left(w, s["L1"][n], s["L2"][n])[0]), s["L2"][n])
        R3, RA, RB = self.right(w, R1, R2)
        tau, tA, tB = self.tau, self.tA, self.tB
        D = torch.zeros_like(D00)
        U = _ein("ijkabc,ai->jkbc", lt, R1[:nv, :no])
        D[:NO, :no] -= _ein("jlbc,jbcK->Kl", U, tB)
        D[:no, :no] -= 0.5 * _ein("ijlabc,ijkabc->kl", lt, R3)
        D[:no, NO:NO + nv] += _ein("jkbc,jklbcd->ld", U, tau) - _ein("jkbc,jlkbcd->ld", U, tau)
        lc = self.covariant(self.full(s["lam2"]))
        D[:no, NO:NO + nv] += 0.5 * _ein("aibj,ijlabd->ld", lc[:nv, :no, :nv, :no], self.contra(R3))
        W3 = 0.5 * _ein("ijkabc,ijab->kc", lt, RA[:, :, :, :nv])
        D[:NO, NO:] += _ein("kc,kcLD->LD", W3, 2.0 * s["t2c"] - s["t2x"])
        D[:NO, NO:] -= _ein("jkbL,jkbD->LD", _ein("ijkabc,iacL->jkbL", lt, RB), tA)
        D[:NO, NO:] -= _ein("ikaL,ikaD->LD", _ein("ijkabc,jbcL->ikaL", lt, tB), RA)
        D[:no, NO:] -= 0.5 * _ein("kl,Dk->lD", _ein("ijkabc,ijlabc->kl", lt, tau), R1[:, :no])
        D[:NO, NO:NO + nv] -= 0.5 * _ein("cd,cL->Ld", _ein("ijkabc,ijkabd->cd", lt, tau), R1[:nv])
        D[NO:NO + nv, :no] += W3.t()
        D[NO:NO + nv, NO:] += _ein("jkbc,jkbD->cD", U, tA)
        D[NO:NO + nv, NO:NO + nv] += 0.5 * _ein("ijkabc,ijkabd->cd", lt, R3)
        lr3 = (lt * R3).sum() / 6.0
        D.diagonal()[:NO] += 2.0 * lr3
        D00_in = _reference_densities(s, NO)[0]
        wt = _weights(no, nv, NO, self.NV, self.dev)
        sd = (s["lam1"] * R1).sum() + (wt * s["lam2"] * R2).sum()
        return D00, Dm0, D - lr3 * (D00_in + D00) - sd * D00


def _pairs(outs):
    return tuple(torch.stack(x) for x in zip(*outs))


def exact(case, seed, device="cuda"):
    op = case["op"]
    if op == "cnto":
        s = prepare(case, seed)
        R1, R2 = s["R1"], s["R2"]
        NV, NO = R1.shape
        d = _ein("aiai->ai", R2)
        M = R1.t() @ R1 + 0.5 * (_ein("aibk,ajbk->ij", R2, R2) + torch.diag((d * d).sum(0)))
        return M, R1 @ R1.t() + 0.5 * (_ein("aicj,bicj->ab", R2, R2) + torch.diag((d * d).sum(1)))
    if op == "gemm":
        s = prepare(case, seed)
        return s["A"] @ s["B"].t()
    gen = _generator(seed, device)
    if op == "sweep":
        out = []
        for no, nv, NV in SWEEP[:case["systems"]]:
            one = _system("rho", case["precision"], no + 8, NV, no, nv, 3 * NV, vec=case["vec"])
            s = _make_system(one, gen)
            x = _Exact(one, s)
            out.append(_pairs(x.rho(s["omega"][q], s["R1"][q], s["R2"][q]) for q in range(case["vec"])))
        return out
    # 64-bit sums over all ordered triples: about 1 TFLOP/s, and tensors of n_o^3 n_v^3 values
    if work(dict(case, core=False))["flops"] > 8e12 or (case["no"] * case["nv"]) ** 3 > 2e9:
        return None
    s = _make_system(case, gen)
    x = _Exact(case, s)
    vectors = range(case["vec"])
    if op == "ground":
        return x.omega()
    if op == "davidson":
        return (_pairs(x.rho(s["omega"][q], s["R1"][q], s["R2"][q]) for q in vectors)
                + _pairs(x.sigma(s["omega"][q], s["L1"][q], s["L2"][q]) for q in vectors))
    if op == "adjoint":
        w = _weights(x.no, x.nv, x.NO, x.NV, x.dev)
        g1, g2 = x.sigma(s["omega"][0], s["L1"][0], _symmetrize(s["L2"][0].clone(), x.no, x.nv) / w)
        return *x.rho(s["omega"][0], s["R1"][0], s["R2"][0]), g1, w * g2
    D = [x.densities(q) for q in vectors]
    _, Dm0_in, D0m_in = _reference_densities(s, x.NO)
    f = []
    for q in vectors:
        T0m, Tm0 = (_ein("pq,xpq->x", d, x.mut) for d in (D[q][2] + D0m_in[q], D[q][1] + Dm0_in[q]))
        f.append(2.0 / 3.0 * s["omega"][q] * float(T0m @ Tm0))
    return D[0][0], torch.stack([d[1] for d in D]), torch.stack([d[2] for d in D]), f
