"""What a user of the library has it do, as measurable cases.

A case is one call (or one captured MD step) through the Python binding of the
C ABI, at the sizes of the repository's own workloads and at odd ones between
them.  `listed()` names twelve, `draw()` gives more of the same kinds.

Kinds of case:
  step        an MD step captured as a CUDA graph (StepGraph.launch)
  predict     energies, local energies, forces and virials of new structures
  energies    energies alone of new structures (screening, Monte Carlo)
  energy_grad the differentiable energy and its backward pass
  knm         the energy and force rows of K_NM of a training batch
  solve       the regularised least-squares solve of a fit
  descriptor  descriptors of candidate cells (sparse-point selection)

The results of the reduced-precision forms (bf16x3, bf16x6, fp32) are kept in
FP32: the library's buffers are FP64, but the arithmetic behind them is FP32
outside the sums per configuration, and a program that chose these forms has
no use for more.  The plain FP64 path and the solve keep FP64.

Structures are near-crystalline diamond supercells and random packings (here
jittered lattices, which are quick to make) at the densities of the workloads.
Sparse points are descriptors of other such cells, computed here in FP64 by
plain torch, so that they depend on the seed alone; `exact()` uses the same
plain torch for the whole method.
"""
import math

import numpy as np
import torch

from paper_2310_03921_gb300 import gap

F64 = torch.float64
SI = 5.431  # diamond lattice parameter, Angstrom

# Descriptor and model settings by name: (n_max, l_max, cutoff, sigma, species,
# mixed channels, zeta).  The shapes are those of the five workloads and of the
# silicon model of the paper's Sec. 4.1.
SOAPS = {
    "n6l4": (6, 4, 5.0, 0.5, 1, 0, 4),
    "n6l6": (6, 6, 5.0, 0.5, 1, 0, 4),
    "n8l6": (8, 6, 5.0, 0.5, 1, 0, 4),
    "n8l8": (8, 8, 5.0, 0.5, 1, 0, 4),
    "n8l6k4": (8, 6, 5.0, 0.5, 4, 4, 4),
    "n10l8": (10, 8, 4.5, 0.5, 1, 0, 4),
}


def listed():
    return [
        # The smallest MD step: 64 atoms, launches and latency only.
        dict(name="step_64", kind="step", soap="n6l4", structure="diamond", cells=1, reps=2, vacancies=0, M=100,
             precision="bf16x3", virial=False, two_body=False),
        # The plain FP64 path on the same cell: reference energies, finite differences.
        dict(name="predict_64_fp64", kind="predict", soap="n6l4", structure="diamond", cells=1, reps=2, vacancies=0,
             M=100, precision="fp64", virial=True, two_body=False),
        # One new structure (a vacancy cell of 215 atoms) under the fitted silicon model, as in active learning.
        dict(name="predict_215", kind="predict", soap="n8l6", structure="diamond", cells=1, reps=3, vacancies=1,
             M=2000, precision="bf16x3", virial=True, two_body=False),
        # Differentiable energy of a 1000-atom cell with the paper's silicon descriptor.
        dict(name="energy_grad_1000", kind="energy_grad", soap="n6l6", structure="diamond", cells=1, reps=5,
             vacancies=0, M=1500, precision="bf16x3", virial=True, two_body=False),
        # MD of 32768 atoms, energies, forces and virial.
        dict(name="step_32768", kind="step", soap="n8l8", structure="diamond", cells=1, reps=16, vacancies=0, M=4000,
             precision="bf16x3", virial=True, two_body=False),
        # 512 four-species boxes of 8 to 256 atoms in one call, four GPs.
        dict(name="predict_512_alloys", kind="predict", soap="n8l6k4", structure="boxes", cells=512, atoms_lo=8,
             atoms_hi=256, M=3000, precision="bf16x3", virial=True, two_body=False),
        # MD of a 110592-atom network with the two-body term.
        dict(name="step_110592", kind="step", soap="n10l8", structure="network", cells=1, side=48, M=9000,
             precision="bf16x3", virial=True, two_body=True),
        # K_NM of the 200-cell silicon fit (cells of 64 to 216 atoms).
        dict(name="knm_200_cells", kind="knm", soap="n8l6", structure="strained", cells=200, M=2000,
             precision="bf16x3"),
        # K_NM rows of a few four-species boxes (descriptors of 1008 entries, four GPs).
        dict(name="knm_24_alloys", kind="knm", soap="n8l6k4", structure="boxes", cells=24, atoms_lo=8, atoms_hi=64,
             M=500, precision="bf16x3"),
        # The least-squares solve of the 200-cell fit: 24992 atoms, 75176 rows.
        dict(name="solve_75176x2000", kind="solve", configs=200, atoms=24992, D=252, M=2000, zeta=4),
        # A first fit on few cells.
        dict(name="solve_2648x300", kind="solve", configs=8, atoms=880, D=252, M=300, zeta=4),
        # Candidate pool of the sparse-point selection: 12 cells of 216 atoms in FP64.
        dict(name="descriptor_2592_fp64", kind="descriptor", soap="n8l6", structure="diamond", cells=12, reps=3,
             vacancies=0, precision="fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "predict", "energies", "energy_grad", "knm", "solve", "descriptor"])
    if kind == "solve":
        atoms = _log_int(rng, 400, 24000)
        return dict(kind="solve", configs=max(1, atoms // rng.randint(60, 220)), atoms=atoms,
                    D=rng.choice([105, 252, 324]), M=_log_int(rng, 60, 1900), zeta=rng.choice([2, 4]))
    if kind == "knm":
        if rng.random() < 0.3:
            return dict(kind="knm", soap="n8l6k4", structure="boxes", cells=rng.randint(2, 24), atoms_lo=8,
                        atoms_hi=rng.randint(16, 64), M=_log_int(rng, 40, 500), precision="bf16x3")
        return dict(kind="knm", soap=rng.choice(["n6l4", "n6l6", "n8l6"]), structure="strained",
                    cells=_log_int(rng, 1, 150), M=_log_int(rng, 50, 2000), precision="bf16x3")
    if kind == "descriptor":
        return dict(kind="descriptor", soap=rng.choice(["n6l4", "n6l6", "n8l6", "n8l8"]), structure="diamond",
                    cells=rng.randint(1, 12), reps=rng.randint(1, 4), vacancies=rng.randint(0, 2),
                    precision=rng.choice(["fp64", "bf16x3"]))
    case = dict(kind=kind, precision="bf16x3", virial=rng.random() < 0.7, two_body=False)
    form = rng.random()
    if form < 0.55:
        case.update(soap=rng.choice(["n6l4", "n6l6", "n8l6", "n8l8"]), structure="diamond", cells=rng.randint(1, 3),
                    reps=rng.randint(1, 14), vacancies=rng.randint(0, 3), M=_log_int(rng, 50, 4000))
        if case["reps"] <= 3 and kind != "step":
            case["precision"] = rng.choice(["bf16x3", "fp32", "fp64", "bf16x6"])
    elif form < 0.8 and kind in ("predict", "energies"):
        case.update(soap="n8l6k4", structure="boxes", cells=_log_int(rng, 1, 300), atoms_lo=8,
                    atoms_hi=rng.randint(24, 256), M=_log_int(rng, 50, 2000))
    else:
        case.update(soap="n10l8", structure="network", cells=1, side=rng.randint(6, 36), M=_log_int(rng, 100, 6000),
                    two_body=True)
    return case


# ------------------------------------------------------------- structures
def _diamond(reps):
    base = torch.tensor([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0],
                         [.25, .25, .25], [.25, .75, .75], [.75, .25, .75], [.75, .75, .25]], dtype=F64)
    n = torch.tensor(reps, dtype=F64)
    grid = torch.cartesian_prod(*[torch.arange(r, dtype=F64) for r in reps]).reshape(-1, 1, 3)
    return ((grid + base[None]) / n).reshape(-1, 3), torch.diag(n * SI)


def _structures(case, seed, pool=0):
    """(positions [N][3], species [N], cells [C][3][3], offsets [C+1]) on the host.  With pool > 0: at least that many
    atoms of every species in cells like the case's own, none of them the case's."""
    g = torch.Generator().manual_seed(1000003 * (seed + 1) + (17 if pool else 0))
    sizes = torch.Generator().manual_seed(9)  # a batch's cell sizes are the case's, not the seed's
    species = SOAPS[case["soap"]][4]
    kind = case["structure"]
    out, have, c = [], 0, 0
    while (have < pool) if pool else (c < case["cells"]):
        if kind in ("diamond", "strained"):
            if kind == "strained":
                reps = [int(v) for v in torch.randint(2, 4, (3,), generator=sizes)] if not pool else [3, 3, 3]
                sigma = 0.05 + 0.15 * float(torch.rand((), generator=g))
                e = (torch.rand(6, generator=g, dtype=F64) * 2 - 1) * 0.03
                eps = torch.stack([e[0], e[3], e[4], e[3], e[1], e[5], e[4], e[5], e[2]]).reshape(3, 3)
            else:
                reps, sigma, eps = [3 if pool else case["reps"]] * 3, 0.1, torch.zeros(3, 3, dtype=F64)
            frac, cell = _diamond(reps)
            cell = cell @ (torch.eye(3, dtype=F64) + eps)
            pos = frac @ cell + sigma * torch.randn(frac.shape[0], 3, generator=g, dtype=F64)
            if kind == "diamond" and case["vacancies"] and not pool:
                pos = pos[torch.randperm(pos.shape[0], generator=g)[case["vacancies"]:].sort().values]
        else:
            # jittered simple cubic lattice: 0.05 atoms / A^3 no closer than
            # ~1.8 A (boxes of four species), 0.1 / A^3 and ~1.4 A (network)
            if kind == "network":
                side = 13 if pool else case["side"]
                n, density, d_min = side ** 3, 0.1, 1.4
            else:
                n = 216 if pool else int(torch.randint(case["atoms_lo"], case["atoms_hi"] + 1, (), generator=sizes))
                side, density, d_min = math.ceil(n ** (1 / 3) - 1e-9), 0.05, 1.8
            L = (n / density) ** (1 / 3)
            sites = torch.cartesian_prod(*[torch.arange(side, dtype=F64)] * 3).reshape(-1, 3)
            sites = sites[torch.randperm(side ** 3, generator=g)[:n].sort().values]
            room = max(0.0, L / side - d_min) / 2
            pos = sites * (L / side) + (torch.rand(n, 3, generator=g, dtype=F64) * 2 - 1) * max(room, 0.1)
            cell = torch.eye(3, dtype=F64) * L
        z = torch.randint(0, species, (pos.shape[0],), generator=g, dtype=torch.int32)
        out.append((pos, z, cell))
        have += min(int((z == s).sum()) for s in range(species))
        c += 1
    counts = torch.tensor([0] + [p.shape[0] for p, _, _ in out])
    return (torch.cat([p for p, _, _ in out]), torch.cat([z for _, z, _ in out]),
            torch.stack([b for _, _, b in out]), counts.cumsum(0).to(torch.int32))


def _mix(case):
    species, K = SOAPS[case["soap"]][4:6]
    if not K:
        return None
    return torch.randn(K, species, generator=torch.Generator().manual_seed(4), dtype=F64)


def _model_arrays(case, seed, device):
    """Sparse points [M][D] and coefficients [M] of every GP, and the two-body sparse distances and coefficients."""
    species = SOAPS[case["soap"]][4]
    pos, z, cell, off = _structures(case, seed, pool=case["M"])
    pool = _Soap(case, device).descriptors(pos, z, cell, off)
    g = torch.Generator().manual_seed(7 * seed + 3)
    X, a = [], []
    for s in range(species):
        rows = torch.nonzero(z == s)[:, 0]
        pick = rows[torch.randperm(rows.numel(), generator=g)[:case["M"]]]
        X.append(pool[pick.to(pool.device)])
        a.append(0.1 * torch.randn(case["M"], generator=g, dtype=F64))
    tb = None
    if case.get("two_body"):
        rc = SOAPS[case["soap"]][2]
        tb = (1.4 + (rc - 1.4) * (torch.arange(50, dtype=F64) + 0.5) / 50, 0.1 * torch.randn(50, generator=g, dtype=F64))
    return X, a, tb


class _TwoBody:
    def __init__(self, rc, x, alpha):
        self.rc, self.d, self.theta, self.delta, self.x, self.alpha = rc, 1.0, 1.0, 10.0, x.numpy(), alpha.numpy()


def _gap_soap(case):
    n, l, rc, sigma, species, K, _ = SOAPS[case["soap"]]
    w = _mix(case)
    return gap.Soap(n, l, rc, sigma, n_species=species, mix_K=K, mix_w=None if w is None else w.numpy())


# -------------------------------------------------------- prepare and run
def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    state = {"case": case}
    if case["kind"] == "solve":
        K, y, sigma, X = _solve_inputs(case, seed, dev)
        state.update(K=K, y=y, sigma=sigma)
        # a solve needs the sparse points (K_MM) only: any descriptor of their size will do
        state["soap"] = gap.Soap(*{105: (6, 4), 252: (8, 6), 324: (8, 8)}[case["D"]], 5.0, 0.5)
        state["model"] = gap.Model(state["soap"], [X.cpu().numpy()], [np.zeros(case["M"])], 1.0, case["zeta"])
        return state
    pos, z, cell, off = _structures(case, seed)
    state.update(pos=pos.to(dev), species=z.to(dev), cell=cell.numpy(), off=off.numpy(),
                 pbc=np.ones((cell.shape[0], 3), np.int32), soap=_gap_soap(case))
    if case["kind"] == "descriptor":
        return state
    X, a, tb = _model_arrays(case, seed, dev)
    rc = SOAPS[case["soap"]][2]
    state["model"] = gap.Model(state["soap"], [x.cpu().numpy() for x in X], [v.numpy() for v in a], 1.0,
                               SOAPS[case["soap"]][6], two_body=None if tb is None else _TwoBody(rc, *tb))
    if case["kind"] == "step":
        state["batch"] = _batch(state)
        state["graph"] = gap.StepGraph(state["model"], state["batch"], case["precision"], pair_capacity=1.2,
                                       virial=case["virial"])
    return state


def _batch(s):
    return gap.Batch(s["pos"], s["species"], s["cell"], s["pbc"], s["off"])


def _kept(x, precision):
    return x if precision == "fp64" or x is None else x.float()


def run(state):
    case = state["case"]
    kind, prec = case["kind"], case.get("precision")
    if kind == "solve":
        return {"alpha": state["model"].solve(state["K"], state["y"], state["sigma"], jitter=1e-8)}
    if kind == "step":
        state["graph"].launch()
        return {k: _kept(v, prec) for k, v in state["graph"].outputs.items() if v is not None}
    if kind == "descriptor":
        return {"p": _kept(state["soap"].descriptor(_batch(state), prec), prec)}
    if kind == "knm":
        return {"knm": _kept(state["model"].assemble_knm(_batch(state), prec), prec)}
    if kind == "energy_grad":
        pos = state["pos"].detach().requires_grad_(True)
        E, V = gap.energy(state["model"], pos, state["species"], state["cell"], state["pbc"], state["off"], prec)
        grad, = torch.autograd.grad(E.sum(), pos)
        return {"energy": _kept(E.detach(), prec), "grad": _kept(grad, prec), "virial": _kept(V, prec)}
    full = kind == "predict"
    out = state["model"].predict(_batch(state), prec, local=True, forces=full, virial=full and case["virial"])
    return {k: _kept(v, prec) for k, v in out.items() if v is not None}


def _sizes(case):
    """(atoms, configurations) of a case, random counts by their mean."""
    s = case["structure"]
    if s == "diamond":
        n = 8 * case["reps"] ** 3 - case["vacancies"]
    elif s == "strained":
        n = 125
    elif s == "network":
        n = case["side"] ** 3
    else:
        n = (case["atoms_lo"] + case["atoms_hi"]) / 2
    return n * case["cells"], case["cells"]


def work(case):
    if case["kind"] == "solve":
        rows, M = case["configs"] + 3 * case["atoms"], case["M"]
        # the symmetric Gram matrix, one factorisation, and the sparse points' Gram matrix
        return {"bytes": 8 * (rows * M + 2 * rows + M * case["D"] + M),
                "flops": rows * M * M + M ** 3 / 3 + M * M * case["D"]}
    n, l, rc, _, species, K, _ = SOAPS[case["soap"]]
    lm, blocks = (l + 1) ** 2, K or 1
    nc = n if K else n * species
    npair = blocks * nc * (nc + 1) // 2
    D, chans = npair * (l + 1), n * (K or species)
    N, C = _sizes(case)
    density = {"diamond": 8 / SI ** 3, "strained": 8 / SI ** 3, "network": 0.1, "boxes": 0.05}[case["structure"]]
    pairs = N * density * 4 / 3 * math.pi * rc ** 3
    item = 8 if case["precision"] == "fp64" else 4
    flops = 2 * pairs * chans * lm + 2 * N * npair * lm
    read = 28 * N
    if case["kind"] == "descriptor":
        return {"bytes": read + item * N * D, "flops": flops}
    M = case["M"]
    read += item * M * D * species
    if case["kind"] == "knm":
        rows = C + 3 * N
        return {"bytes": read + item * rows * M * species, "flops": flops + 2 * 3 * (N + pairs) * D * M + 2 * N * D * M}
    if case["kind"] == "energies":
        return {"bytes": read + item * (N + C), "flops": flops + 2 * N * D * M}
    wrote = item * (4 * N + C * (10 if case["virial"] else 1))
    return {"bytes": read + wrote, "flops": flops + 4 * N * D * M + 2 * N * npair * lm + 4 * pairs * n * lm}


# ----------------------------------------------- the solve's inputs and value
def _solve_inputs(case, seed, dev):
    """K_NM [C + 3N][M], targets, regularisation per row and sparse points: rows of the kernel and of its derivative
    along random Jacobian rows, at unit descriptors spread about a common mean."""
    g = torch.Generator(dev).manual_seed(seed + 11)
    D, M, C, N, z = case["D"], case["M"], case["configs"], case["atoms"], case["zeta"]
    rn = lambda *s: torch.randn(*s, generator=g, device=dev, dtype=F64)  # noqa: E731
    mean = rn(D)
    mean /= mean.norm()

    def unit(k):
        x = mean + rn(k, D) / math.sqrt(D)
        return x / x.norm(dim=1, keepdim=True)

    X = unit(M)
    q = unit(N) @ X.T
    rows = C + 3 * N
    K = torch.empty(rows, M, dtype=F64, device=dev)
    first = [(c * N) // C for c in range(C + 1)]
    k = q ** z
    W = z * q ** (z - 1)
    for c in range(C):
        a, b = first[c], first[c + 1]
        K[c + 3 * a] = k[a:b].sum(0)
        J = rn(3 * (b - a), D) * (0.5 / math.sqrt(D))
        K[c + 1 + 3 * a:c + 1 + 3 * b] = -W[a:b].repeat_interleave(3, 0) * (J @ X.T)
    sigma = torch.full((rows,), 0.1, dtype=F64, device=dev)
    for c in range(C):
        sigma[c + 3 * first[c]] = 0.01 * math.sqrt(first[c + 1] - first[c])
    y = K @ (0.1 * rn(M)) + sigma * rn(rows)
    return K, y, sigma, X


def _solve_exact(case, seed, dev):
    K, y, sigma, X = _solve_inputs(case, seed, dev)
    M = case["M"]
    kmm = (X @ X.T) ** case["zeta"] + 1e-8 * torch.eye(M, dtype=F64, device=dev)
    A = torch.cat([K / sigma[:, None], torch.linalg.cholesky(kmm).T])
    b = torch.cat([y / sigma, torch.zeros(M, dtype=F64, device=dev)])
    del K
    Q, R = torch.linalg.qr(A)
    return {"alpha": torch.linalg.solve_triangular(R, (Q.T @ b)[:, None], upper=True)[:, 0]}


# -------------------------------------------------- the method in plain torch
class _Soap:
    """SOAP descriptors, the sparse GP and its derivatives in FP64 (Eqs. 1-3, 10-13, 18-25)."""

    def __init__(self, case, device):
        self.n, self.l, self.rc, self.sigma, self.species, self.K, self.zeta = SOAPS[case["soap"]]
        self.dev = device
        w = _mix(case)
        self.w = (torch.eye(self.species, dtype=F64) if w is None else w).to(device)  # [groups][species]
        s, ws = np.polynomial.legendre.leggauss(128)
        self.s = torch.tensor((s + 1) * self.rc / 2, device=device)
        ws = torch.tensor(ws * self.rc / 2, device=device)
        self.gw = self._radial(self.s) * (4 * math.pi * ws * self.s ** 2)  # [n][nodes]
        self.R0 = self._integrals(torch.full((1,), 1e-9, dtype=F64, device=device))[0][0, :, 0]

    def _radial(self, r):
        """Orthonormal g_n of (rc - r)^(k+2), k = 1..n: u^3 P_k^(2,6)(2u - 1) with u = 1 - r / rc."""
        def poly(r):
            u = 1 - r / self.rc
            x, a, b = 2 * u - 1, 2, 6
            p = [torch.ones_like(x), (a + 1) + (a + b + 2) * (x - 1) / 2]
            for k in range(2, self.n):
                c = 2 * k + a + b
                p.append(((c - 1) * (c * (c - 2) * x + a * a - b * b) * p[-1]
                          - 2 * (k + a - 1) * (k + b - 1) * c * p[-2]) / (2 * k * (k + a + b) * (c - 2)))
            return torch.stack(p[:self.n]) * u ** 3
        s, ws = np.polynomial.legendre.leggauss(64)
        s, ws = torch.tensor((s + 1) * self.rc / 2, device=r.device), torch.tensor(ws * self.rc / 2, device=r.device)
        norm = (poly(s) ** 2 * (ws * s ** 2)).sum(1).sqrt()
        return poly(r) / norm[:, None]

    def _integrals(self, r):
        """I_nl(r) and dI_nl/dr, [P][n][l+1], by quadrature over s."""
        out, dout = [], []
        for rr in r.split(1 << 17):
            x = rr[:, None] * self.s / self.sigma ** 2
            top = self.l + 90
            ratio, keep = torch.zeros_like(x), {}
            for l in range(top, 0, -1):  # i_l / i_(l-1)
                ratio = x / ((2 * l + 1) + x * ratio)
                if l <= self.l + 1:
                    keep[l] = ratio
            e = torch.exp(-(self.s - rr[:, None]) ** 2 / (2 * self.sigma ** 2))
            i = [-torch.expm1(-2 * x) / (2 * x) * e]
            for l in range(1, self.l + 2):
                i.append(i[-1] * keep[l])
            I, dI = [], []
            for l in range(self.l + 1):
                d = (i[l + 1] + (l / x) * i[l]) * (self.s / self.sigma ** 2) - (rr[:, None] / self.sigma ** 2) * i[l]
                I.append(i[l] @ self.gw.T)
                dI.append(d @ self.gw.T)
            out.append(torch.stack(I, 2))
            dout.append(torch.stack(dI, 2))
        return torch.cat(out), torch.cat(dout)

    def _cut(self, r, d=1.0):
        t = math.pi * ((r - self.rc + d) / d).clamp(min=0)
        return 0.5 * (torch.cos(t) + 1), -0.5 * math.pi / d * torch.sin(t)

    def _ylm(self, x, y, z):
        """Real spherical harmonics of unit vectors, a list of [..., 2l+1] by l."""
        C, S = [torch.ones_like(x)], [torch.zeros_like(x)]
        for m in range(1, self.l + 1):
            C.append(x * C[-1] - y * S[-1])
            S.append(x * S[m - 1] + y * C[m - 1])
        Q = {}  # d^m P_l / dz^m
        out = []
        for l in range(self.l + 1):
            row = [None] * (2 * l + 1)
            for m in range(l, -1, -1):
                if m == l:
                    Q[l, m] = torch.full_like(x, float(math.prod(range(1, 2 * l, 2))))
                elif m == l - 1:
                    Q[l, m] = (2 * l - 1) * z * Q[l - 1, m]
                else:
                    Q[l, m] = ((2 * l - 1) * z * Q[l - 1, m] - (l + m - 1) * Q[l - 2, m]) / (l - m)
                k = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m))
                if m == 0:
                    row[l] = k * Q[l, 0]
                else:
                    row[l + m] = math.sqrt(2) * k * Q[l, m] * C[m]
                    row[l - m] = math.sqrt(2) * k * Q[l, m] * S[m]
            out.append(torch.stack(row, -1))
        return out

    def neighbours(self, pos, cells, off):
        """(i, j, r_ij) of all pairs within the cutoff, images included, ordered by i."""
        I, J, V = [], [], []
        off = off.tolist()
        pos, cells = pos.to(self.dev), cells.to(self.dev)
        for c in range(len(off) - 1):
            cell, x = cells[c], pos[off[c]:off[c + 1]]
            inv = torch.linalg.inv(cell)
            reach = (self.rc * inv.norm(dim=0) + 0.5).floor().int().tolist()
            frac = x @ inv
            shifts = torch.cartesian_prod(*[torch.arange(-k, k + 1, dtype=F64) for k in reach]).to(self.dev).reshape(-1, 3)
            step = max(1, (1 << 25) // (x.shape[0] * shifts.shape[0]))
            for a in range(0, x.shape[0], step):
                d = frac[None] - frac[a:a + step, None]
                d = (d - d.round())[:, :, None] + shifts
                v = d @ cell
                r2 = (v * v).sum(-1)
                own = torch.arange(d.shape[0], device=self.dev)
                i, j, t = torch.nonzero((r2 < self.rc ** 2) & (r2 > 1e-12), as_tuple=True)
                I.append(own[i] + a + off[c])
                J.append(j + off[c])
                V.append(v[i, j, t])
        return torch.cat(I), torch.cat(J), torch.cat(V)

    def chunks(self, pos, z, cells, off, size):
        """Per run of atoms: (first, last, mask [A][J], j, displacement, their r, unit vector, R, dR/dr, Y by l, group
        weights [A][J][G], coefficients by l [A][G][n][2l+1])."""
        i, j, v = self.neighbours(pos, cells, off)
        z = z.to(self.dev).long()
        N = z.numel()
        count = torch.bincount(i, minlength=N)
        start = count.cumsum(0) - count
        for a in range(0, N, size):
            b = min(N, a + size)
            width = max(1, int(count[a:b].max()))
            p = torch.arange(width, device=self.dev)
            mask = p < count[a:b, None]
            at = torch.where(mask, start[a:b, None] + p, 0)
            if i.numel():
                jj, vv = j[at], torch.where(mask[..., None], v[at], torch.tensor([1.0, 0.0, 0.0], dtype=F64, device=self.dev))
            else:
                jj = torch.zeros_like(at)
                vv = torch.ones(*at.shape, 3, dtype=F64, device=self.dev)
            r = vv.norm(dim=-1)
            u = vv / r[..., None]
            I, dI = self._integrals(r.reshape(-1))
            f, df = self._cut(r)
            f, df = (f * mask)[..., None, None], (df * mask)[..., None, None]
            I, dI = I.reshape(*r.shape, self.n, -1), dI.reshape(*r.shape, self.n, -1)
            R, dR = f * I, df * I + f * dI
            Y = self._ylm(u[..., 0], u[..., 1], u[..., 2])
            w = self.w.T[z[jj]]
            coef = []
            for l in range(self.l + 1):
                wR = w[..., :, None] * R[..., None, :, l]
                c = wR.flatten(2).transpose(1, 2) @ Y[l]
                c = c.reshape(b - a, w.shape[-1], self.n, 2 * l + 1)
                if l == 0:
                    c = c + (self.w.T[z[a:b]][:, :, None] * self.R0 / math.sqrt(4 * math.pi))[..., None]
                coef.append(c)
            yield a, b, mask, jj, vv, r, u, R, dR, Y, w, coef

    def _pairs(self, left, right):
        """sum_m left_a right_b for a <= b, sqrt 2 off the diagonal: [..., groups][pairs] of [..., G][n][m] pairs."""
        if not self.K:
            left, right = left.flatten(-3, -2)[..., None, :, :], right.flatten(-3, -2)[..., None, :, :]
        p = left @ right.transpose(-1, -2)
        k = p.shape[-1]
        a, b = torch.triu_indices(k, k, device=p.device)
        return p, a, b, torch.where(a == b, 1, 2).to(F64).sqrt()

    def spectrum(self, coef):
        out = []
        for c in coef:
            p, a, b, s = self._pairs(c, c)
            out.append(p[..., a, b] * s)
        return torch.stack(out, -1).flatten(1)

    def descriptors(self, pos, z, cells, off):
        out = []
        for ch in self.chunks(pos, z, cells, off, 2048):
            p = self.spectrum(ch[-1])
            out.append(p / p.norm(dim=1, keepdim=True))
        return torch.cat(out)

    def _dylm(self, u, r):
        """d Y / d r_ij by l, [..., 3][2l+1]."""
        out = [[] for _ in range(self.l + 1)]
        for x in range(3):
            t = -u * u[..., x:x + 1]
            t[..., x] += 1
            t = t / r[..., None]
            _, d = torch.func.jvp(lambda *q: tuple(self._ylm(*q)), tuple(u[..., k] for k in range(3)),
                                  tuple(t[..., k].contiguous() for k in range(3)))
            for l in range(self.l + 1):
                out[l].append(d[l])
        return [torch.stack(o, -2) for o in out]

    def predict(self, pos, z, cells, off, X, alpha, tb, grad):
        N, C = z.numel(), len(off) - 1
        eps = torch.zeros(N, dtype=F64, device=self.dev)
        F = torch.zeros(N, 3, dtype=F64, device=self.dev)
        W = torch.zeros(N, 3, 3, dtype=F64, device=self.dev)
        zd = z.to(self.dev).long()
        for a, b, mask, jj, vv, r, u, R, dR, Y, w, coef in self.chunks(pos, z, cells, off, 1024):
            if grad:
                coef = [c.detach().requires_grad_(True) for c in coef]
            p = self.spectrum(coef)
            ph = p / p.norm(dim=1, keepdim=True)
            e = torch.zeros(b - a, dtype=F64, device=self.dev)
            for s in range(self.species):
                at = torch.nonzero(zd[a:b] == s)[:, 0]
                if at.numel():
                    e = e.index_add(0, at, ((ph[at] @ X[s].T) ** self.zeta) @ alpha[s])
            eps[a:b] = e.detach()
            dv = torch.zeros_like(vv)
            if grad:
                G = torch.autograd.grad(e.sum(), coef)
                dY = self._dylm(u, r)
                for l in range(self.l + 1):
                    gz = (w @ G[l].flatten(2)).reshape(*r.shape, self.n, 2 * l + 1)
                    sR = (gz * dR[..., l, None]).sum(-2)
                    sY = (gz * R[..., l, None]).sum(-2)
                    dv += (sR * Y[l]).sum(-1, keepdim=True) * u + (dY[l] * sY[..., None, :]).sum(-1)
            if tb is not None:
                f, df = self._cut(r)
                x, al = tb
                k = torch.exp(-(r[..., None] - x) ** 2 / 2)  # theta = 1, delta = 10
                e2, d2 = (k @ al) * 100, (k * (r[..., None] - x)) @ al * -100
                eps[a:b] += 0.5 * (f * e2 * mask).sum(1)
                dv += (0.5 * (df * e2 + f * d2) * mask)[..., None] * u
            if grad:
                dv = dv * mask[..., None]
                F[a:b] += dv.sum(1)
                F.index_add_(0, jj[mask], -dv[mask])
                W[a:b] -= (dv[..., :, None] * vv[..., None, :]).sum(1)
        cfg = torch.repeat_interleave(torch.arange(C, device=self.dev), (off[1:] - off[:-1]).to(self.dev).long())
        E = torch.zeros(C, dtype=F64, device=self.dev).index_add_(0, cfg, eps)
        V = torch.zeros(C, 3, 3, dtype=F64, device=self.dev).index_add_(0, cfg, W)
        return E, eps, F, V

    def knm(self, pos, z, cells, off, X):
        N, C, M = z.numel(), len(off) - 1, X[0].shape[0]
        K = torch.zeros(C + 3 * N, M * self.species, dtype=F64, device=self.dev)
        zd = z.to(self.dev).long()
        cfg = torch.repeat_interleave(torch.arange(C), (off[1:] - off[:-1]).long()).to(self.dev)
        row = cfg + 1 + 3 * torch.arange(N, device=self.dev)  # first force row of an atom
        first = (torch.arange(C) + 3 * off[:-1].long()).to(self.dev)
        D = X[0].shape[1]
        for a, b, mask, jj, vv, r, u, R, dR, Y, w, coef in self.chunks(pos, z, cells, off, max(16, 256 * 252 // D)):
            p = self.spectrum(coef)
            nrm = p.norm(dim=1, keepdim=True)
            ph = p / nrm
            dY = self._dylm(u, r)
            J = []
            for l in range(self.l + 1):
                # d c [A][J][3][G][n][m] of this l
                dc = (dR[..., None, :, l, None] * u[..., None, None] * Y[l][..., None, None, :]
                      + R[..., None, :, l, None] * dY[l][..., None, :])
                dc = w[:, :, None, :, None, None] * dc[:, :, :, None]
                q, ia, ib, s = self._pairs(dc, coef[l][:, None, None])
                J.append((q[..., ia, ib] + q[..., ib, ia]) * s)
            J = torch.stack(J, -1).flatten(3)  # d p / d r_ij [A][J][3][D]
            J = (J - (J * ph[:, None, None]).sum(-1, keepdim=True) * ph[:, None, None]) / nrm[:, None, None]
            for s in range(self.species):
                at = torch.nonzero(zd[a:b] == s)[:, 0]
                if not at.numel():
                    continue
                q = ph[at] @ X[s].T
                cols = slice(s * M, (s + 1) * M)
                K[:, cols].index_add_(0, first[cfg[a + at]], q ** self.zeta)
                T = (J[at] @ X[s].T) * (self.zeta * q ** (self.zeta - 1))[:, None, None]  # [A][J][3][M]
                own, ok = row[a + at], mask[at]
                for x in range(3):
                    K[:, cols].index_add_(0, own + x, T[:, :, x].sum(1))
                    K[:, cols].index_add_(0, (row[jj[at]] + x)[ok], -T[:, :, x][ok])
        return K


def exact(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device()) if torch.cuda.is_available() else torch.device("cpu")
    if case["kind"] == "solve":
        return _solve_exact(case, seed, dev)
    pos, z, cell, off = _structures(case, seed)
    soap = _Soap(case, dev)
    if case["kind"] == "descriptor":
        return {"p": soap.descriptors(pos, z, cell, off)}
    X, a, tb = _model_arrays(case, seed, dev)
    if case["kind"] == "knm":
        return {"knm": soap.knm(pos, z, cell, off, X)}
    a = [v.to(dev) for v in a]
    tb = None if tb is None else tuple(v.to(dev) for v in tb)
    E, eps, F, V = soap.predict(pos, z, cell, off, X, a, tb, case["kind"] != "energies")
    if case["kind"] == "energy_grad":
        return {"energy": E, "grad": -F, "virial": V}
    out = {"energy": E}
    if case["kind"] != "step":
        out["local_e"] = eps
    if case["kind"] != "energies":
        out["forces"] = F
        if case["virial"]:
            out["virial"] = V
    return out
