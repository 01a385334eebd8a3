"""Performance cases of the framework: the calls that a program makes through the Python API
(``paper_2411_19030_gb300``), over the sizes, precisions and options that are in use.

A case is a dict of plain values; ``prepare`` makes what a program holds before the call (the
operator handle, the buffers, a design and the coarse states of the previous design iteration),
``run`` makes the call, ``exact`` restates it in plain FP64 torch (block-tridiagonal direct solves).

Kinds
-----
sequential  assemble the design, step the state and the adjoint through all Nt steps
            (``sequential_pass``): the first iteration of a design loop.
oneshot     assemble the design and run one one-shot Parareal pass (``oneshot_pass``) from the
            coarse states of a design 1% away: every later iteration of a design loop.  With
            ``design`` set, the density filter and projection before it and their chain rule
            after it too (``DesignMap``), as the loop does.
gradient    ``ParaTopoFn``: objective and backward through torch autograd.
batch       several designs of uneven size in one captured graph (``Batch``).
sens        the sensitivity reduction over stored state and adjoint histories.

All solves run at rtol 1e-12: the class default is 1e-13, which the FP64 coarse-step CG with an
FP32 preconditioner does not reach on every problem; at 1e-12 the results are reproducible to
about 1e-11, so outputs of two versions of the code can be compared.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2411_19030_gb300 import Operator, PassBuffers, SolveConfig, oneshot_pass, parareal_pass, sequential_pass
from paper_2411_19030_gb300.autograd import ParaTopoFn
from paper_2411_19030_gb300.batch import Batch
from paper_2411_19030_gb300.design import DesignMap

RTOL = 1e-12
# The two material sets: conductivity-only SIMP with unit capacity, and Table 1 of the paper.
MATERIALS = {
    "simp_k": dict(k0=1.0, kmin=1e-3, pk=3.0, c0=1.0, cmin=1.0, pc=1.0),
    "table1": dict(k0=3.0, kmin=0.03, pk=3.0, c0=1.0, cmin=0.5, pc=2.0),
}
# Side, steps and slices of the first designs of the 48-design batching workload.
BATCH_SIDES = (64, 96, 128, 192, 256)
BATCH_TIMES = ((512, 16), (1024, 32), (2048, 64))


def _case(name, kind, nx, ny, Nt, Ntau, precision="fp64", p=8.0, material="simp_k", sink="left", load="constant",
          objective="power_mean", lo=0.2, hi=0.8, design=False, warm="sequential", count=1, t_end=1.0):
    return dict(name=name, kind=kind, nx=nx, ny=ny, Nt=Nt, Ntau=Ntau, precision=precision, p=p, material=material,
                sink=sink, load=load, objective=objective, lo=lo, hi=hi, design=design, warm=warm, count=count, t_end=t_end)


def listed():
    return [
        # the plain method on the smallest grid in use: launches and latency are all of it
        _case("seq_32_fp64", "sequential", 32, 32, 100, 1, lo=0.4, hi=0.6, t_end=0.1),
        # a small design iteration
        _case("oneshot_64_mixed", "oneshot", 64, 64, 512, 16, "fp32_refine"),
        # the paper's test problem: its materials, sink, load and exponent
        _case("oneshot_100_paper", "oneshot", 100, 100, 480, 16, "fp32_refine", p=20.0, material="table1",
              sink="bottom", load="paper", lo=0.05, hi=0.95),
        # odd sides, no 2h level, every solve in FP64, the modified objective
        _case("oneshot_97x61_fp64", "oneshot", 97, 61, 240, 8, material="table1", load="paper", objective="modified"),
        # the headline design iteration, with the filter and projection around it
        _case("oneshot_128_mixed", "oneshot", 128, 128, 1024, 32, "fp32_refine", design=True),
        # the same pass with every solve in FP64
        _case("oneshot_128_fp64", "oneshot", 128, 128, 1024, 32),
        # a rectangle that is a multiple of nothing in the launch geometry
        _case("oneshot_200x150_mixed", "oneshot", 200, 150, 768, 24, "fp32_refine"),
        # the high-contrast 256 x 256 design of the differentiation workload
        _case("oneshot_256_mixed", "oneshot", 256, 256, 2048, 64, "fp32_refine", lo=0.0, hi=1.0),
        # the largest: an iteration of the full design loop
        _case("loop_512_mixed", "oneshot", 512, 512, 4096, 128, "fp32_refine", design=True, warm="parareal"),
        # differentiation through autograd: checkpointed forward, slice by slice backward
        _case("gradient_96_fp64", "gradient", 96, 96, 256, 8, lo=0.0, hi=1.0),
        # designs of uneven size advanced together
        _case("batch_10_mixed", "batch", 256, 256, 2048, 64, "fp32_refine", count=10),
        # the sensitivity sums alone, over histories that a program stored
        _case("sens_256", "sens", 256, 256, 512, 16, material="table1"),
    ]


def draw(rng):
    """One more case of the same kinds: sides 24 to 288, odd ones and rectangles among them."""
    kind = rng.choice(("sequential", "oneshot", "oneshot", "oneshot", "oneshot", "gradient", "batch", "sens"))
    precision = "fp64" if kind == "gradient" else rng.choice(("fp64", "fp32_refine", "fp32_refine"))
    most = {"sequential": 128, "gradient": 112, "batch": 128, "sens": 320}.get(kind, 160 if precision == "fp64" else 288)
    nx = int(round(math.exp(rng.uniform(math.log(24), math.log(most)))))
    ny = max(24, min(most, int(round(nx * rng.uniform(0.7, 1.4)))))
    if rng.random() < 0.6:                       # most programs take even sides
        nx, ny = nx + nx % 2, ny + ny % 2
    if kind == "batch":
        Ntau, M, count = 16, 32, rng.randint(2, 8)
    else:
        Ntau, M, count = rng.choice((6, 8, 12, 16, 24, 32, 48)), rng.choice((8, 12, 16, 20, 32)), 1
        if kind in ("sequential", "gradient"):
            Ntau = rng.choice((4, 8, 12, 16))
    material = rng.choice(("simp_k", "simp_k", "table1"))
    lo, hi = rng.choice(((0.2, 0.8), (0.05, 0.95), (0.4, 0.6)))
    c = _case("", kind, nx, ny, Ntau * M, Ntau, precision, p=rng.choice((2.0, 8.0, 8.0, 20.0)), material=material,
              sink=rng.choice(("left", "bottom")), load=rng.choice(("constant", "paper")),
              objective=rng.choice(("power_mean", "power_mean", "modified")), lo=lo, hi=hi,
              design=kind == "oneshot" and rng.random() < 0.3, count=count)
    del c["name"]
    return c


# ------------------------------------------------------------------------------- inputs

def _designs_of(case):
    """(nx, ny, Nt, Ntau) of every design of a case."""
    if case["kind"] != "batch":
        return [(case["nx"], case["ny"], case["Nt"], case["Ntau"])]
    if case["nx"] == 256:                        # the first designs of the 48-design workload
        return [(BATCH_SIDES[i % 5], BATCH_SIDES[i % 5], *BATCH_TIMES[i % 3]) for i in range(case["count"])]
    out = []
    for i in range(case["count"]):               # sides shrinking from the drawn one
        f = 1.0 - 0.5 * i / case["count"]
        out.append((max(12, int(case["nx"] * f)), max(12, int(case["ny"] * f)), case["Nt"], case["Ntau"]))
    return out


def _sink(case, nx, ny):
    """The centred tenth of the left or of the bottom edge, as a node mask."""
    h = 1.0 / nx
    y, x = np.meshgrid(np.arange(ny + 1) * h, np.arange(nx + 1) * h, indexing="ij")
    s, L, edge = (y, ny * h, x) if case["sink"] == "left" else (x, nx * h, y)
    m = (edge < 1e-12) & (np.abs(s - 0.5 * L) <= max(0.05 * L + 1e-12, 0.51 * h))
    return m.reshape(-1).astype(np.uint8)


def _load(case, Nt):
    """The time factor of the source: one, or (1 - t)(1 + cos 50 t)/2."""
    if case["load"] == "constant":
        return None
    t = case["t_end"] * np.arange(Nt + 1) / Nt
    return 0.5 * (1.0 - t) * (1.0 + np.cos(50.0 * t))


def _rho(case, nx, ny, seed):
    """The previous design and the one at hand, 1% away, per element."""
    rng = np.random.default_rng([seed, nx, ny])
    old = rng.uniform(case["lo"], case["hi"], nx * ny)
    return old, np.clip(old + rng.uniform(-0.01, 0.01, nx * ny), 0.0, 1.0)


def _dev(a):
    return torch.tensor(a, dtype=torch.float64, device="cuda")


def _operator(case, size, precision):
    nx, ny, Nt, Ntau = size
    return Operator(nx, ny, 1.0 / nx, MATERIALS[case["material"]], Nt, Ntau, case["t_end"] / Nt, case["p"], _sink(case, nx, ny),
                    q_time=_load(case, Nt), solve=SolveConfig(precision, rtol=RTOL, cg_iters_max=8000),
                    objective=case["objective"])


def _histories(case, seed):
    """A state and an adjoint history [Nt + 1][Nn] and [Nt][Nn]: smooth fields that grow and decay
    in time, with the roughness of a per-element design."""
    nx, ny, Nt = case["nx"], case["ny"], case["Nt"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.linspace(0, 1, nx + 1, dtype=torch.float64, device="cuda")
    y = torch.linspace(0, 1, ny + 1, dtype=torch.float64, device="cuda")[:, None]
    shape = ((1 + torch.sin(1.5 * x)) * (1 + torch.cos(2.0 * y)) / 4).reshape(-1)
    t = torch.arange(Nt + 1, dtype=torch.float64, device="cuda")[:, None] / Nt

    def rough(rows):
        return 0.01 * torch.rand(rows, shape.numel(), dtype=torch.float64, device="cuda", generator=g)

    T = (1 - torch.exp(-3 * t)) * (shape + rough(Nt + 1))
    lam = torch.exp(-2 * t[1:]) * (shape + rough(Nt))
    return T, lam


# The filter radius, projection and chi range of the design loop.
FILTER = dict(r_fil=0.03, beta=32.0)


def _chi(case, seed):
    """The design variables of the previous iteration and of this one."""
    rng = np.random.default_rng([seed, 7])
    n = case["nx"] * case["ny"]
    old = rng.uniform(0.3, 0.7, n)
    return old, np.clip(old + rng.uniform(-0.01, 0.01, n), 0.0, 1.0)


def prepare(case, seed):
    kind = case["kind"]
    sizes = _designs_of(case)
    if kind == "batch":
        ops = [_operator(case, s, case["precision"]) for s in sizes]
        batch = Batch(ops)
        rhos = [_rho(case, s[0], s[1], seed + 100 * i) for i, s in enumerate(sizes)]
        for d, (old, _) in enumerate(rhos):
            batch.buffers(d)["rho"].copy_(_dev(old))
        batch.assemble()
        batch.sequential_pass()
        for d, (_, new) in enumerate(rhos):
            batch.buffers(d)["rho"].copy_(_dev(new))
        batch.capture()
        return dict(case=case, batch=batch, ops=ops)
    op = _operator(case, sizes[0], case["precision"])
    nx, ny = case["nx"], case["ny"]
    old, new = _rho(case, nx, ny, seed)
    s = dict(case=case, op=op, rho=_dev(new))
    if kind == "gradient":
        s["rho"].requires_grad_(True)
    elif kind == "sens":
        op.assemble(s["rho"])
        s["T"], s["lam"] = _histories(case, seed)
        s["grad"] = op.zeros(op.Ne)
    elif kind == "sequential":
        s["buf"] = PassBuffers(op)
    else:
        s["buf"] = buf = PassBuffers(op)
        old = _dev(old)
        if case["design"]:
            s["map"] = DesignMap(nx, ny, 1.0 / nx, **FILTER)
            chi_old, chi = _chi(case, seed)
            s["chi"] = _dev(chi)
            s["dproj"], s["g_chi"], s["v_chi"], s["vol"] = op.zeros(op.Ne), op.zeros(op.Ne), op.zeros(op.Ne), op.zeros(1)
            s["map"].forward(_dev(chi_old), old, s["dproj"])
        if case["warm"] == "parareal":           # a loop whose first iteration was one Parareal iteration
            op.assemble(old)
            parareal_pass(op, buf, 1)
        else:                                    # a loop whose first iteration was sequential
            first = _operator(case, sizes[0], "fp64")
            first.assemble(old)
            sequential_pass(first, buf)
            torch.cuda.synchronize()
            first.close()
    return s


# ------------------------------------------------------------------------------- the calls

def _held(view, owner):
    """A view of memory that the batch owns, which keeps the batch: the memory goes with it."""
    view = view.view(view.shape)
    view.owner = owner
    return view


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        batch = state["batch"]
        batch.replay()
        return [{k: _held(batch.buffers(d)[k], state) for k in ("T_hist", "U_T_new", "U_theta_new", "V_lam_new", "V_g_new")}
                for d in range(len(state["ops"]))]
    op, rho = state["op"], state["rho"]
    if kind == "gradient":
        rho.grad = None
        Theta = ParaTopoFn.apply(rho, op)
        Theta.backward()
        return dict(Theta=Theta.detach(), grad=rho.grad)
    if kind == "sens":
        state["grad"].zero_()
        op.sensitivities(state["lam"], 1, op.Nt, state["T"], state["grad"])
        return dict(grad=state["grad"])
    buf = state["buf"]
    if kind == "sequential":
        op.assemble(rho)
        Theta, grad = sequential_pass(op, buf)
        return dict(Theta=Theta, grad=grad, T_hist=buf.T_hist, U_theta=buf.U_th, V_lam=buf.V_l, V_g=buf.V_g)
    if case["design"]:
        state["map"].forward(state["chi"], rho, state["dproj"])
    op.assemble(rho)
    Theta, grad = oneshot_pass(op, buf)
    out = dict(Theta=Theta, grad=grad, T_hist=buf.T_hist, U_T=buf.U_T_new, U_theta=buf.U_th_new, V_lam=buf.V_l_new,
               V_g=buf.V_g_new)
    if case["design"]:
        m = state["map"]
        m.backward(state["dproj"], grad, state["g_chi"])
        m.volume(rho, state["vol"])
        m.backward(state["dproj"], None, state["v_chi"])
        out.update(g_chi=state["g_chi"], v_chi=state["v_chi"], volume=state["vol"])
    return out


def work(case):
    """Bytes: the design, the start states and (sens) the histories read once, the results written
    once.  Operations: per fine solve and node the right-hand side, one residual and one
    application of the operator (two operations for each of 9 couplings each)."""
    nbytes = flops = 0
    for nx, ny, Nt, Ntau in _designs_of(case):
        Nn, Ne = (nx + 1) * (ny + 1), nx * ny
        if case["kind"] == "sens":
            nbytes += 8 * (2 * Nt * Nn + 2 * Ne)
            flops += 2 * 20 * Nt * Ne
            continue
        states = (Ntau + 1) * (2 * Nn + Ne)
        if case["kind"] == "gradient":
            nbytes += 8 * (2 * Ne + 2 * (Ntau + 1) * Nn)
            solves = 3 * Nt
        elif case["kind"] == "sequential":
            nbytes += 8 * (Ne + 2 * Nt * Nn + states)
            solves = 2 * Nt
        else:
            nbytes += 8 * (Ne + 2 * Nt * Nn + 2 * states)
            solves = 2 * (Nt + 2 * Ntau)
        flops += 54 * Nn * solves
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------- 64-bit values

_AT = ((0, 0), (0, 1), (1, 1), (1, 0))           # row and column of the element corners SW, SE, NE, NW
_KE = torch.tensor([[4., -1, -2, -1], [-1, 4, -1, -2], [-2, -1, 4, -1], [-1, -2, -1, 4]], dtype=torch.float64) / 6
_ME = torch.tensor([[4., 2, 1, 2], [2, 4, 2, 1], [1, 2, 4, 2], [2, 1, 2, 4]], dtype=torch.float64) / 36


class _Heat:
    """Backward-Euler steps of the heat equation on bilinear squares for one design, with a direct
    block-tridiagonal factorisation per step size; fields are [R][ny + 1][nx + 1]."""

    def __init__(self, case, size, rho):
        self.nx, self.ny, self.Nt, self.Ntau = nx, ny, Nt, Ntau = size
        m, self.p, self.modified = MATERIALS[case["material"]], case["p"], case["objective"] == "modified"
        self.h, self.dt, self.M = 1.0 / nx, case["t_end"] / Nt, Nt // Ntau
        self.Ne = nx * ny
        r = rho.reshape(ny, nx)
        self.k = m["kmin"] + (m["k0"] - m["kmin"]) * r ** m["pk"]
        self.c = m["cmin"] + (m["c0"] - m["cmin"]) * r ** m["pc"]
        self.dk = m["pk"] * (m["k0"] - m["kmin"]) * r ** (m["pk"] - 1)
        self.dc = m["pc"] * (m["c0"] - m["cmin"]) * r ** (m["pc"] - 1)
        self.free = _dev(1.0 - _sink(case, nx, ny)).reshape(ny + 1, nx + 1)
        q = _load(case, Nt)
        self.q = [1.0] * (Nt + 1) if q is None else q.tolist()
        f = torch.zeros_like(self.free)
        for i, j in _AT:
            f[i:i + ny, j:j + nx] += self.h ** 2 / 4
        self.f = f * self.free
        self.factors = {}

    def _factor(self, step):
        if step not in self.factors:
            nx, ny, nn = self.nx, self.ny, self.nx + 1
            D = torch.zeros(ny + 1, nn, nn, dtype=torch.float64, device="cuda")
            U = torch.zeros_like(D)              # coupling of row i to row i + 1
            e = torch.arange(nx, device="cuda")
            for a, (ia, ja) in enumerate(_AT):
                for b, (ib, jb) in enumerate(_AT):
                    v = self.k * float(_KE[a, b]) + self.c * float(_ME[a, b] * self.h ** 2 / step)
                    if ia == ib:
                        D[ia:ia + ny, e + ja, e + jb] += v
                    elif ia < ib:
                        U[:ny, e + ja, e + jb] += v
            free = self.free
            D = D * free[:, :, None] * free[:, None, :] + torch.diag_embed(1 - free)
            U[:ny] *= free[:-1, :, None] * free[1:, None, :]
            S = torch.empty_like(D)              # inverses of the Schur complements
            for i in range(ny + 1):
                S[i] = torch.linalg.inv(D[i] if i == 0 else D[i] - U[i - 1].T @ (S[i - 1] @ U[i - 1]))
            # y_i = b_i - y_{i-1} G_i, z = y S, x_i = z_i - x_{i+1} H_i on row vectors
            G = torch.bmm(S[:-1], U[:-1])
            H = torch.bmm(U[:-1].transpose(1, 2), S[:-1].transpose(1, 2))
            self.factors[step] = (S.transpose(1, 2).contiguous(), G.contiguous(), H.contiguous())
        return self.factors[step]

    def _solve(self, step, b):
        S, G, H = self._factor(step)
        y = (b * self.free).transpose(0, 1).contiguous()
        for i in range(1, self.ny + 1):
            torch.addmm(y[i], y[i - 1], G[i - 1], alpha=-1, out=y[i])
        x = torch.bmm(y, S)
        for i in range(self.ny - 1, -1, -1):
            torch.addmm(x[i], x[i + 1], H[i], alpha=-1, out=x[i])
        return x.transpose(0, 1).contiguous()

    def _mass(self, x):
        ny, nx = self.ny, self.nx
        y = torch.zeros_like(x)
        c = self.c * self.h ** 2
        v = [x[:, i:i + ny, j:j + nx] * c for i, j in _AT]
        for a, (ia, ja) in enumerate(_AT):
            y[:, ia:ia + ny, ja:ja + nx] += sum(v[b] * float(_ME[a, b]) for b in range(4))
        return y

    def _corners(self, x):
        return torch.stack([x[:, i:i + self.ny, j:j + self.nx] for i, j in _AT], 1)

    def term(self, lam, T, Tp, step):
        """lambda_e^T (dk Ke T_e + dc Me (T - T_prev)_e / step) per element"""
        l, t, d = self._corners(lam), self._corners(T), self._corners(T - Tp)
        kt = torch.einsum("raij,ab,rbij->rij", l, _KE.cuda(), t)
        ct = torch.einsum("raij,ab,rbij->rij", l, (_ME * self.h ** 2).cuda(), d)
        return self.dk * kt + self.dc * ct / step

    def primal(self, T, theta, j, step, N):
        q = _dev([self.q[i] for i in j])[:, None, None]
        T = self._solve(step, self._mass(T) / step + q * self.f)
        inc = (T ** self.p).sum((1, 2)) / (N * self.Ne)
        return T, theta + inc if self.modified else (theta ** self.p + inc) ** (1 / self.p)

    def adjoint(self, lam, g, T, Tp, Theta, step, N):
        scale = (self.p if self.modified else Theta ** (1 - self.p)) / self.Ne
        lam = self._solve(step, self._mass(lam) / step + scale * T ** (self.p - 1))
        return lam, g - self.term(lam, T, Tp, step) / N

    def sequential(self):
        """(T history, theta at the slice ends, (lambda, g) at the first step of every slice)"""
        M, Nt, Ntau = self.M, self.Nt, self.Ntau
        T = torch.zeros(1, self.ny + 1, self.nx + 1, dtype=torch.float64, device="cuda")
        theta = torch.zeros(1, dtype=torch.float64, device="cuda")
        hist, th = [T], [theta]
        for j in range(1, Nt + 1):
            T, theta = self.primal(T, theta, [j], self.dt, Nt)
            hist.append(T)
            if j % M == 0:
                th.append(theta)
        lam, g = torch.zeros_like(T), torch.zeros(1, self.ny, self.nx, dtype=torch.float64, device="cuda")
        V = [(lam, g)]
        for j in range(Nt, 0, -1):
            lam, g = self.adjoint(lam, g, hist[j], hist[j - 1], theta, self.dt, Nt)
            if (j - 1) % M == 0:
                V.append((lam, g))
        V.reverse()
        return torch.cat(hist), torch.cat(th), torch.cat([v[0] for v in V]), torch.cat([v[1] for v in V])

    def oneshot(self, U_T, U_th, V_l, V_g):
        """One modified forward and one reverse Parareal iteration from the given coarse states."""
        M, Nt, Ntau, dtau = self.M, self.Nt, self.Ntau, self.M * self.dt
        hist = torch.empty(Nt + 1, self.ny + 1, self.nx + 1, dtype=torch.float64, device="cuda")
        s = torch.arange(Ntau, device="cuda")
        T, th = U_T[:-1], U_th[:-1]
        for i in range(1, M + 1):
            T, th = self.primal(T, th, [M * n + i for n in range(Ntau)], self.dt, Nt)
            hist[M * s + i] = T
        G, Gth = self.primal(U_T[:-1], U_th[:-1], [M * (n + 1) for n in range(Ntau)], dtau, Ntau)
        X, Xth = [U_T[:1]], [U_th[:1]]
        for n in range(Ntau):
            a, b = self.primal(X[-1], Xth[-1], [M * (n + 1)], dtau, Ntau)
            X.append(a + T[n] - G[n])
            Xth.append(b + th[n] - Gth[n])
        X, Xth = torch.cat(X), torch.cat(Xth)
        hist[0] = X[0]
        hist[M * (s + 1)] = X[1:]
        Theta = Xth[-1:]
        lam, g = V_l[1:], V_g[1:]
        for i in range(M, 0, -1):
            lam, g = self.adjoint(lam, g, hist[M * s + i], hist[M * s + i - 1], Theta, self.dt, Nt)
        k = M * s + 1
        kp = (k - M).clamp(min=0)
        Gl, Gg = self.adjoint(V_l[1:], V_g[1:], hist[k], hist[kp], Theta, dtau, Ntau)
        Y = [(torch.zeros_like(V_l[:1]), torch.zeros_like(V_g[:1]))]
        for n in range(Ntau - 1, -1, -1):
            a, b = self.adjoint(*Y[-1], hist[k[n:n + 1]], hist[kp[n:n + 1]], Theta, dtau, Ntau)
            Y.append((a + lam[n] - Gl[n], b + g[n] - Gg[n]))
        Y.reverse()
        return hist, X, Xth, torch.cat([v[0] for v in Y]), torch.cat([v[1] for v in Y])


def _seconds(case):
    """About what the direct solves of ``exact`` take: one call per node row each way."""
    t = 0.0
    for nx, ny, Nt, Ntau in _designs_of(case):
        solves = 2 * (Nt + Ntau + Nt // Ntau) if case["kind"] in ("oneshot", "batch") else 2 * Nt
        t += solves * (2 * (ny + 1) * 8e-6 + 1e-3)
    return t


def _filtered(nx, ny, chi):
    """The filtered and projected design, its derivative, and the filter's rows as a function"""
    h, beta, eta = 1.0 / nx, FILTER["beta"], 0.5
    R = math.ceil(FILTER["r_fil"] / h)
    d = torch.arange(-R, R + 1, dtype=torch.float64, device="cuda") * h
    w = (FILTER["r_fil"] - torch.sqrt(d[:, None] ** 2 + d ** 2)).clamp(min=0)

    def cone(a):
        pad = torch.nn.functional.pad(a.reshape(ny, nx), (R, R, R, R))
        return sum(w[i, j] * pad[i:i + ny, j:j + nx] for i in range(2 * R + 1) for j in range(2 * R + 1))

    S = cone(torch.ones(ny * nx, dtype=torch.float64, device="cuda"))
    t = torch.tanh(beta * (cone(chi) / S - eta))
    den = math.tanh(beta * (1 - eta)) + math.tanh(beta * eta)
    rho, dproj = (t + math.tanh(beta * eta)) / den, beta * (1 - t * t) / den
    return rho.reshape(-1), lambda y: cone(dproj.reshape(-1) * y / S.reshape(-1)).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "sens":
        T, lam = _histories(case, seed)
        nx, ny, Nt = case["nx"], case["ny"], case["Nt"]
        heat = _Heat(case, _designs_of(case)[0], _dev(_rho(case, nx, ny, seed)[1]))
        T, lam = T.reshape(-1, ny + 1, nx + 1), lam.reshape(-1, ny + 1, nx + 1)
        g = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
        for a in range(0, Nt, 64):
            b = min(Nt, a + 64)
            g -= heat.term(lam[a:b], T[a + 1:b + 1], T[a:b], heat.dt).sum(0) / Nt
        return dict(grad=g.reshape(-1))
    if _seconds(case) > 11 or case["warm"] == "parareal":
        return None
    out = []
    for i, size in enumerate(_designs_of(case)):
        nx, ny = size[0], size[1]
        old, new = (_dev(a) for a in _rho(case, nx, ny, seed + 100 * i))
        back = None
        if case["design"]:
            chi_old, chi = _chi(case, seed)
            old = _filtered(nx, ny, _dev(chi_old))[0]
            new, back = _filtered(nx, ny, _dev(chi))
        flat = lambda x: x.reshape(x.shape[0], -1)  # noqa: E731
        if kind in ("sequential", "gradient"):
            hist, th, lam, g = _Heat(case, size, new).sequential()
            if kind == "gradient":
                return dict(Theta=th[-1], grad=g[0].reshape(-1))
            return dict(Theta=th[-1:], grad=g[0].reshape(-1), T_hist=flat(hist), U_theta=th, V_lam=flat(lam), V_g=flat(g))
        hist, th, lam, g = _Heat(case, size, old).sequential()
        T, X, Xth, Y, Yg = _Heat(case, size, new).oneshot(hist[::size[2] // size[3]], th, lam, g)
        if kind == "batch":
            out.append(dict(T_hist=flat(T), U_T_new=flat(X), U_theta_new=Xth, V_lam_new=flat(Y), V_g_new=flat(Yg)))
            continue
        res = dict(Theta=Xth[-1:], grad=Yg[0].reshape(-1), T_hist=flat(T), U_T=flat(X), U_theta=Xth, V_lam=flat(Y),
                   V_g=flat(Yg))
        if back is not None:
            ones = torch.full((nx * ny,), 1.0 / (nx * ny), dtype=torch.float64, device="cuda")
            res.update(g_chi=back(Yg[0].reshape(-1)), v_chi=back(ones), volume=new.mean().reshape(1))
        return res
    return out
