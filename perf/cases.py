"""What this library is measured on: passes through its public entry points
(``paper_2004_05566_gb300.hifcn``) as a user's program makes them.

A user factors an operator once (``hif_setup``), keeps the handle and the state
vectors on the GPU, and then

* steps it in time: ``cn_step`` for a step at a time, ``cn_steps`` for a queue of
  steps, ``cn_step_batched`` for many operators, ``cn_step_multi`` for many states;
* solves with it (``pcg_solve``) or applies the approximate inverse (``hif_apply``)
  inside a solver of their own;
* refactors it when the coefficient has moved (``hif_refactor``).

Sizes are those of the repository's workloads, tests and benchmark (63^2 to 2047^2,
3D up to 63^3, leaves 8 to 16, sides n = leaf 2^L) and sizes between them.  The
fields follow the same recipes: lognormal coefficients of a filtered Gaussian random
field with a given contrast, and smooth or noisy states.
"""

from __future__ import annotations

import math

import torch

import paper_2004_05566_gb300.hifcn as H

PRECISION = {"fp64": H.HIF_FP64, "fp32": H.HIF_FP32, "bf16top": H.HIF_FP32_BF16TOP}

DEFAULTS = {"dim": 2, "leaf": 16, "eps": 1e-6, "precision": "fp32", "tol": 1e-10, "dt": 1.0,
            "contrast": 1e3, "logistic": True, "theta": 0.5, "warm": False, "steps": 1,
            "states": 1, "count": 1, "side_to": 0}


def _case(**kw) -> dict:
    return {**DEFAULTS, **kw}


def listed() -> list[dict]:
    return [
        # the smallest call: one step of the 2D heat equation at 63^2 with the library's
        # default options (FP64 factor), a step at a time as an interactive loop takes it
        _case(name="step2d_63_fp64", kind="step", n=64, leaf=8, precision="fp64", dt=1e-2,
              contrast=1.0, logistic=False),
        # a small reaction-diffusion run at a side that is no power of two, steps queued
        _case(name="steps2d_351_fp32", kind="steps", n=352, leaf=11, dt=0.1, steps=10),
        # the benchmark's operator: Fisher-KPP at 1023^2, mixed precision
        _case(name="steps2d_1023_fp32", kind="steps", n=1024, contrast=1e4, steps=10),
        # the same operator with the default (FP64) factor, to the paper's tolerance
        _case(name="steps2d_1023_fp64", kind="steps", n=1024, contrast=1e4, precision="fp64",
              tol=1e-12, steps=4),
        # the largest 2D operator of the serving mix
        _case(name="steps2d_2047_fp32", kind="steps", n=2048, dt=0.3, steps=4),
        # a solve to the paper's tolerance with the paper's looser factor, several iterations
        _case(name="solve2d_703_fp32", kind="solve", n=704, leaf=11, eps=1e-3, tol=1e-12, dt=0.1),
        # the approximate inverse as an operator in a user's own Krylov loop
        _case(name="apply2d_511_fp64", kind="apply", n=512, precision="fp64", dt=0.1),
        # many small operators of uneven size stepped together (one tick of the step server)
        _case(name="batched2d_24_fp32", kind="batched", n=64, side_to=512, leaf=0, count=24, dt=0.1),
        # 3D heat equation, single trajectory
        _case(name="steps3d_63_fp32", kind="steps", dim=3, n=64, leaf=8, eps=1e-4, dt=0.1,
              logistic=False, steps=4),
        # an ensemble of 16 states of one 3D operator, BF16 top levels
        _case(name="multi3d_63_bf16top", kind="multi", dim=3, n=64, leaf=8, eps=1e-4, dt=0.1,
              logistic=False, precision="bf16top", states=16),
        # coefficients that move in time: factor again, then a few steps
        _case(name="refactor2d_511_fp32", kind="refactor", n=512, dt=0.1, steps=4),
        _case(name="refactor3d_47_fp32", kind="refactor", dim=3, n=48, leaf=6, eps=1e-4, dt=0.1,
              steps=2),
    ]


def _log_uniform(rng, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _snap(side: float, leafs) -> tuple[int, int]:
    """The admissible (n, leaf) with n = leaf 2^L, L >= 1, whose n is nearest to side."""
    return min(((m << L, m) for m in leafs for L in range(1, 12)),
               key=lambda nm: (abs(nm[0] - side), nm[0], nm[1]))


def draw(rng) -> dict:
    """A case of the same ranges: entry point, size, leaf, precision and options drawn."""
    kind = rng.choice(["step", "steps", "steps", "solve", "apply", "batched", "steps", "multi",
                       "refactor"])
    dim = 3 if kind in ("steps", "multi", "refactor", "solve") and rng.random() < 0.35 else 2
    if kind == "apply":
        precision = "fp64"
    elif kind == "multi":
        precision = "bf16top"
    elif kind == "batched":
        precision = "fp32"
    else:
        precision = rng.choice(["fp32", "fp32", "fp64"])
    if dim == 3:
        n, leaf = _snap(_log_uniform(rng, 16, 60 if kind != "refactor" else 44),
                        [rng.choice([4, 5, 6, 7, 8])])
        eps = rng.choice([1e-3, 1e-4])
    else:
        n, leaf = _snap(_log_uniform(rng, 64, 1280 if kind not in ("refactor", "multi") else 700),
                        [rng.choice([8, 9, 10, 11, 12, 13, 14, 15, 16])])
        eps = rng.choice([1e-6, 1e-6, 1e-3])
    c = _case(kind=kind, dim=dim, n=n, leaf=leaf, eps=eps, precision=precision,
              tol=rng.choice([1e-10, 1e-12]), dt=round(_log_uniform(rng, 1e-2, 1.0), 4),
              contrast=rng.choice([1e2, 1e3]), logistic=rng.random() < 0.6,
              theta=1.0 if rng.random() < 0.2 else 0.5, warm=kind == "solve" and rng.random() < 0.3,
              steps=rng.randint(1, 6) if kind in ("steps", "refactor") else 1)
    if kind == "multi":
        c["states"] = rng.choice([3, 8, 16, 24])
    if kind == "batched":
        c.update(n=64, side_to=rng.choice([256, 384, 512]), leaf=0, count=rng.randint(5, 24))
    return c


# ------------------------------------------------------------------------- inputs


def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _field(n: int, dim: int, corr_len: float, gen) -> torch.Tensor:
    """Zero-mean Gaussian random field on the (n+1)^dim nodes, filtered to corr_len."""
    shape = (n + 1,) * dim
    spec = torch.fft.fftn(torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64))
    k = 2.0 * math.pi * torch.fft.fftfreq(n + 1, d=1.0 / n, device="cuda", dtype=torch.float64)
    for ax in range(dim):
        s = [1] * dim
        s[ax] = n + 1
        spec = spec * torch.exp(-0.5 * (k * corr_len) ** 2).reshape(s)
    g = torch.fft.ifftn(spec).real
    return g - g.mean()


def _coefficient(n: int, dim: int, contrast: float, gen) -> torch.Tensor:
    """Nodal a(x) > 0 with max a / min a = contrast (1: a = 1, the heat equation)."""
    g = _field(n, dim, 0.05, gen)
    return torch.exp(g * (math.log(contrast) / (g.max() - g.min()))).contiguous()


def _state(n: int, dim: int, gen, logistic: bool) -> torch.Tensor:
    """A state u on the interior nodes: the bump of the logistic examples with a smooth
    perturbation, or for the heat equation a smooth field of both signs with 1% noise."""
    g = _field(n, dim, 0.1, gen)[(slice(1, n),) * dim]
    g = g / g.abs().max()
    if logistic:
        t = torch.arange(1, n, device="cuda", dtype=torch.float64) / n - 0.5
        r2 = sum((t ** 2).reshape([-1 if d == ax else 1 for d in range(dim)]) for ax in range(dim))
        amp = 2.0 / (3.0 * math.sqrt(2.0 * math.pi * 0.05))
        u = amp * torch.exp(-r2 / 0.05) * (1.0 + 0.2 * g)
    else:
        u = g + 0.01 * torch.randn(g.shape, generator=gen, device="cuda", dtype=torch.float64)
    return u.reshape(-1).contiguous()


def _problems(case: dict) -> list[tuple[int, int]]:
    """(n, leaf) of each operator: one, or the uneven sides of a batch."""
    if case["kind"] != "batched":
        return [(case["n"], case["leaf"])]
    lo, hi, m = math.log(case["n"]), math.log(case["side_to"]), case["count"]
    # sides spread evenly over their logarithm
    return [_snap(math.exp(lo + (hi - lo) * i / max(1, m - 1)), range(8, 17)) for i in range(m)]


def _inputs(case: dict, seed: int) -> list[dict]:
    """The device inputs of each operator: coefficient(s) and state(s)."""
    out = []
    for i, (n, leaf) in enumerate(_problems(case)):
        gen = _gen(1000003 * int(seed) + 7919 * i + 11)
        p = {"n": n, "leaf": leaf, "a": _coefficient(n, case["dim"], case["contrast"], gen)}
        u = _state(n, case["dim"], gen, case["logistic"])
        if case["kind"] == "multi":
            k = case["states"]
            scale = 1.0 + 0.05 * torch.arange(k, device="cuda", dtype=torch.float64)
            u = u[None, :] * scale[:, None]
            u = (u + 0.01 * torch.randn(u.shape, generator=gen, device="cuda", dtype=torch.float64)).contiguous()
        if case["kind"] == "refactor":  # the coefficient one interval later
            p["a0"] = p["a"]
            p["a"] = (p["a"] * torch.exp(0.3 * torch.sin(
                3.0 * torch.arange(p["a"].numel(), device="cuda", dtype=torch.float64)
                / p["a"].numel())).reshape(p["a"].shape)).contiguous()
        p["u"] = u
        out.append(p)
    return out


def prepare(case: dict, seed: int) -> dict:
    opt = H.default_options(eps=case["eps"], precision=PRECISION[case["precision"]],
                            cg_tol=case["tol"], theta=case["theta"], x0_mode=1 if case["warm"] else 0)
    s = {"case": case, "problems": _inputs(case, seed), "handles": []}
    for p in s["problems"]:
        h = H.hif_setup(case["dim"], p["n"], p["leaf"], p.get("a0", p["a"]), case["dt"], opt)
        if case["logistic"]:
            H.hif_set_reaction(h, 1, 1.0, 1.0)
        s["handles"].append(h)
        p["out"] = torch.empty_like(p["u"])
    return s


def run(s: dict):
    """One pass.  The library also tells the number of CG iterations; it is a diagnostic, and
    the outputs are the new states."""
    case, p, h = s["case"], s["problems"][0], s["handles"][0]
    kind = case["kind"]
    if kind == "step":
        return H.cn_step(h, p["u"], out=p["out"])[0]
    if kind == "steps":
        p["out"].copy_(p["u"])
        H.cn_steps(h, p["out"], case["steps"])
        return p["out"]
    if kind == "solve":
        if case["warm"]:
            p["out"].copy_(p["u"])
        return H.pcg_solve(h, p["u"], x=p["out"])[0]
    if kind == "apply":
        return H.hif_apply(h, p["u"], y=p["out"])
    if kind == "multi":
        return H.cn_step_multi(h, p["u"], out=p["out"])[0]
    if kind == "batched":
        return H.cn_step_batched(s["handles"], [q["u"] for q in s["problems"]],
                                 outs=[q["out"] for q in s["problems"]])[0]
    if kind == "refactor":
        H.hif_refactor(h, p["a"])
        p["out"].copy_(p["u"])
        H.cn_steps(h, p["out"], case["steps"])
        return p["out"]
    raise ValueError(kind)


# --------------------------------------------------------------------------- work


def _factor_model(dim: int, n: int, leaf: int, eps: float) -> tuple[float, float]:
    """(stored factor values, flops of forming them), estimated from the geometry: cell and
    separator sizes per level, separators above the leaf level holding the ranks that the
    interpolative decompositions keep (measured on the 2D and 3D recipes)."""
    values = flops = 0.0
    side, nc, level = leaf, n // leaf, 0
    edge, face, inner = leaf - 1, (leaf - 1) ** 2, (leaf - 1) ** dim
    while nc >= 1:
        cells = nc ** dim
        if nc == 1:  # the root
            values += inner * inner / 2
            flops += inner ** 3 * 2 / 3
            break
        share = (nc - 1) / nc  # of the sides that are no boundary of the domain
        if dim == 2:
            nB = 4 * share * (edge + 1)
            groups, gsize = 2 * nc * (nc - 1), edge
        else:
            nB = 6 * share * face + 12 * share * share * edge
            groups, gsize = 3 * nc * nc * (nc - 1), face
        values += cells * (inner * inner / 2 + inner * nB) + groups * gsize * gsize
        flops += cells * (inner ** 3 * 2 / 3 + 2 * inner * inner * nB + inner * nB * nB)
        flops += groups * 2 * gsize * gsize * nB
        # the next level's cells hold the sides between their 2^dim children
        if dim == 2:
            keep = min(edge, 8 + 2.5 * level if eps > 1e-5 else 13 + 4 * level)
            inner, edge = 4 * keep + 1, 2 * keep + 1
        else:
            keep = min(face, (5.5 if eps > 5e-4 else 7.5) * side)
            inner, face, edge = 12 * keep + 6 * edge + 1, 4 * keep + 4 * edge, 2 * edge + 1
        side, nc, level = 2 * side, nc // 2, level + 1
    return values, flops


def work(case: dict) -> dict:
    """Every preconditioner application of a pass reads each factor value once, and every CG
    iteration reads and writes its vectors once; a factorization writes each value once."""
    size = {"fp64": 8, "fp32": 4, "bf16top": 4}[case["precision"]]
    bytes_, flops = 0.0, 0.0
    for n, leaf in _problems(case):
        N = (n - 1) ** case["dim"]
        values, setup_flops = _factor_model(case["dim"], n, leaf, case["eps"])
        if case["kind"] == "apply":
            applies = 1
        else:  # a CG iteration gains a little less than |log10 eps| digits
            applies = case["steps"] * round(-math.log10(case["tol"]) / (-math.log10(case["eps"]) - 0.7))
        k = case["states"]
        bytes_ += applies * (values * size + (2 if case["kind"] == "apply" else 12) * 8 * N * k)
        flops += applies * k * (4 * values + 26 * N)
        if case["kind"] == "refactor":
            bytes_ += 8 * values
            flops += setup_flops
    return {"bytes": bytes_, "flops": flops}


# -------------------------------------------------------------------------- exact


class _Direct:
    """A = I - theta dt M by block tridiagonal elimination in 64 bits: the unknowns of a grid
    line (2D) or plane (3D) are a block, the coupling of neighbouring blocks is diagonal."""

    def __init__(self, a: torch.Tensor, n: int, dim: int, dt: float, theta: float):
        c = theta * dt * n * n
        self.dim, self.n, S = dim, n, n - 1
        inner = (slice(1, n),) * dim
        self.w = []  # coupling to the next node along array axis d, zero at the boundary
        diag = torch.ones((S,) * dim, device=a.device, dtype=a.dtype)
        for d in range(dim):
            f = 0.5 * c * (a.narrow(d, 0, n) + a.narrow(d, 1, n))  # face (j, j+1)
            sel = [slice(1, n)] * dim
            sel[d] = slice(0, n)
            f = f[tuple(sel)]
            diag += f.narrow(d, 0, S) + f.narrow(d, 1, S)
            w = f.narrow(d, 1, S).clone()
            w.narrow(d, S - 1, 1).zero_()
            self.w.append(w)
        self.diag = diag
        B = S ** (dim - 1)
        i = torch.arange(B, device=a.device)
        self.inv = []
        for b in range(S):
            D = torch.zeros((B, B), device=a.device, dtype=a.dtype)
            D[i, i] = diag[b].reshape(-1)
            for d in range(1, dim):
                step = S ** (dim - 1 - d)
                wd = self.w[d][b].reshape(-1)[: B - step]
                D[i[: B - step], i[step:]] -= wd
                D[i[step:], i[: B - step]] -= wd
            if b > 0:
                e = self.w[0][b - 1].reshape(-1)
                D -= e[:, None] * self.inv[-1] * e[None, :]
            self.inv.append(torch.cholesky_inverse(torch.linalg.cholesky(D)))

    def matvec(self, u):
        v = u.reshape((self.n - 1,) * self.dim)
        out = self.diag * v
        for d, w in enumerate(self.w):
            m = w.narrow(d, 0, self.n - 2)
            out.narrow(d, 0, self.n - 2).sub_(m * v.narrow(d, 1, self.n - 2))
            out.narrow(d, 1, self.n - 2).sub_(m * v.narrow(d, 0, self.n - 2))
        return out.reshape(-1)

    def _eliminate(self, g):
        S = self.n - 1
        g = g.reshape(S, -1)
        y = [g[0]]
        for b in range(1, S):
            y.append(g[b] + self.w[0][b - 1].reshape(-1) * (self.inv[b - 1] @ y[-1]))
        x = [None] * S
        x[S - 1] = self.inv[S - 1] @ y[S - 1]
        for b in range(S - 2, -1, -1):
            x[b] = self.inv[b] @ (y[b] + self.w[0][b].reshape(-1) * x[b + 1])
        return torch.stack(x).reshape(-1)

    def solve(self, g):
        x = self._eliminate(g)
        return x + self._eliminate(g - self.matvec(x))  # one refinement


def exact(case: dict, seed: int):
    out = []
    for p in _inputs(case, seed):
        if (p["n"] - 1) ** (3 * case["dim"] - 2) > 5e12:  # work of the elimination: over 20 s
            return None
        A = _Direct(p["a"], p["n"], case["dim"], case["dt"], case["theta"])

        def step(u):
            kappa = (1.0 - case["theta"]) / case["theta"]
            g = u + kappa * (u - A.matvec(u))
            if case["logistic"]:
                g = g + case["dt"] * (u * (1.0 - u))
            return A.solve(g)

        u = p["u"]
        if case["kind"] in ("solve", "apply"):  # the apply is the inverse up to eps
            out.append(A.solve(u))
        elif case["kind"] == "multi":
            out.append(torch.stack([step(u[c]) for c in range(u.shape[0])]))
        else:
            for _ in range(case["steps"]):
                u = step(u)
            out.append(u)
    return out if case["kind"] == "batched" else out[0]
