"""What a user of this library has it do, as cases that can be timed.

The library solves 2D Helmholtz problems -Lap u - k^2 u = g with the Wave-ADR
cycle (arXiv 2404.02493).  Its users
  - apply the cycle as the preconditioner of an iteration of their own
    (`mg_cycle`, from a zero iterate, on a residual),
  - let the library iterate (`mg_solve_begin / steps / end`, flexible GMRES
    around complex-FP32 cycles with an FP64 residual), one medium or many
    media of uneven sizes at once,
  - train the phase and the smoother weights through the cycles
    (`autograd.cycles`, FP64),
  - compute the travel-time phase of a medium (`mg_eikonal`),
  - check a field with the FP64 residual (`mg_residual_norm_noalloc`),
  - go from a new medium to a field (`mg_setup`, iterations, `mg_destroy`).

Media are seeded Gaussian random fields (log-normal or layered speeds with a
max/min ratio of 3), phases are travel times: the eikonal equation solved on a
coarse grid and interpolated in the factored form tau = |x - x0| tau_1 of the
paper's Section 3.2.1.  The recipes and sizes are those of the repository's
tests and benchmark.  `exact` restates the method in complex128 with plain
torch operations.
"""
import math
import random  # noqa: F401  (draw takes a random.Random)

import numpy as np
import torch
import torch.nn.functional as F

from paper_2404_02493_gb300 import autograd as AG
from paper_2404_02493_gb300 import binding as B

DEV = "cuda"
RESTART = 20


def listed():
    return [
        # the smallest call: one preconditioner application on a coarse model
        # (the oracle-sized problem, the benchmark's M = 2 and absorbing ADR
        # closure); launches and latency decide
        dict(name="cycle_127", op="cycle", prec="mixed", n=127, ny=0, count=1, medium="lognormal", kh=0.31, M=2,
             bc="abc1", adr_bc="abc"),
        # the paper's N = 1024: an even grid
        dict(name="cycle_1024", op="cycle", prec="mixed", n=1024, ny=0, count=1, medium="layered", kh=0.49, M=2,
             bc="abc1", adr_bc="abc"),
        # a non-square section with a sponge layer: ragged, even sides, the
        # level-1 passes at streaming size
        dict(name="cycle_2300x1000_sponge", op="cycle", prec="mixed", n=2300, ny=1000, count=1, medium="layered",
             kh=0.25, M=2, bc="sponge", adr_bc="zero"),
        # the same cycle wholly in FP64 (what training runs forward)
        dict(name="cycle_fp64_511", op="cycle", prec="fp64", n=511, ny=0, count=1, medium="lognormal", kh=0.39, M=8,
             bc="abc1", adr_bc="zero"),
        # the headline workload: FGMRES steps on the n = 4095, omega = 2000
        # layered medium with M = 2 and the absorbing ADR closure
        dict(name="solve_4095", op="solve", prec="mixed", n=4095, ny=0, count=1, medium="layered", kh=0.49, M=2,
             bc="abc1", adr_bc="abc", steps=10),
        # one restart on a medium-sized log-normal medium (n = 511, omega = 200)
        # with the paper's M = 8 corrections
        dict(name="solve_511", op="solve", prec="mixed", n=511, ny=0, count=1, medium="lognormal", kh=0.39, M=8,
             bc="abc1", adr_bc="zero", steps=20),
        # the batched workload: 64 media of 255, 511 and 1023 in turn
        dict(name="solve_batch64", op="solve", prec="mixed", n=1023, ny=0, count=64, medium="lognormal", kh=0.25, M=2,
             bc="abc1", adr_bc="abc", steps=3),
        # a training step: two FP64 cycles forward and their adjoint
        dict(name="train_255", op="train", n=255, ny=0, medium="lognormal", kh=0.39, M=8, bc="abc1", K=2),
        # the travel time of a layered medium, source at no node
        dict(name="eikonal_2047", op="eikonal", n=2047, ny=0, medium="layered"),
        # the FP64 residual and its norm of a field, nothing allocated
        dict(name="residual_1023", op="residual", n=1023, ny=0, medium="layered", kh=0.49, bc="abc1"),
        # a new medium: setup, one FGMRES restart, the handle freed
        dict(name="medium_511", op="medium", prec="mixed", n=511, ny=0, count=1, medium="lognormal", kh=0.39, M=2,
             bc="abc1", adr_bc="abc", steps=20),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def side(n):
        return 0 if rng.random() < 0.5 else max(40, int(n * rng.uniform(0.4, 1.0)))

    op = rng.choice(["cycle", "cycle", "cycle64", "solve", "solve", "batch", "train", "eikonal", "residual", "medium"])
    medium = rng.choice(["lognormal", "layered"])
    kh = round(rng.uniform(0.2, 0.49), 3)
    bc = rng.choice(["abc1", "abc1", "sponge", "dirichlet"])
    # the absorbing ADR closure belongs to the absorbing boundary
    adr_bc = "abc" if bc == "abc1" else "zero"
    if op == "cycle":
        n = logint(100, 2300)
        return dict(op="cycle", prec="mixed", n=n, ny=side(n), count=1, medium=medium, kh=kh,
                    M=2 if adr_bc == "abc" or n > 1100 else 1, bc=bc, adr_bc=adr_bc)
    if op == "cycle64":
        n = logint(100, 511)
        return dict(op="cycle", prec="fp64", n=n, ny=side(n), count=1, medium=medium, kh=kh, M=rng.choice([2, 4, 8]),
                    bc=bc, adr_bc=adr_bc)
    if op == "solve":
        n = logint(127, 3000)
        paper = 250 < n < 600 and rng.random() < 0.5        # the paper's M = 8 on a whole restart
        return dict(op="solve", prec="mixed", n=n, ny=side(n), count=1, medium=medium, kh=0.39 if paper else kh,
                    M=8 if paper else 2, bc="abc1", adr_bc="zero" if paper else "abc",
                    steps=20 if paper else rng.randint(3, 10))
    if op == "batch":
        return dict(op="solve", prec="mixed", n=logint(400, 1023), ny=0, count=rng.randint(2, 24), medium="lognormal",
                    kh=kh, M=2, bc="abc1", adr_bc="abc", steps=3)
    if op == "train":
        return dict(op="train", n=logint(95, 255), ny=0, medium=medium, kh=kh, M=rng.choice([2, 8]), bc="abc1",
                    K=rng.randint(1, 2))
    if op == "eikonal":
        n = logint(127, 2047)
        return dict(op="eikonal", n=n, ny=side(n), medium=medium)
    if op == "residual":
        n = logint(100, 4095)
        return dict(op="residual", n=n, ny=side(n), medium=medium, kh=kh, bc=rng.choice(["abc1", "sponge"]))
    return dict(op="medium", prec="mixed", n=logint(127, 600), ny=0, count=1, medium=medium, kh=kh, M=2, bc="abc1",
                adr_bc="abc", steps=rng.randint(10, 20))


# ------------------------------------------------------------------ inputs
def _shape(case):
    n = case["n"]
    return n, case["ny"] or n


def _sizes(case):
    """(n, ny) of every instance of a case (a batch: a quarter, a half and
    the whole of n in turn, as 255, 511 and 1023)."""
    n, ny = _shape(case)
    if case.get("count", 1) == 1:
        return [(n, ny)]
    turn = [n // 4, n // 2, n]
    return [(turn[i % 3], turn[i % 3]) for i in range(case["count"])]


def _grid(n, ny):
    h = 1.0 / (max(n, ny) + 1)
    x = (torch.arange(n, device=DEV, dtype=torch.float64) + 1) * h
    y = (torch.arange(ny, device=DEV, dtype=torch.float64) + 1) * h
    return x[None, :], y[:, None], h


def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, device=DEV, dtype=torch.float64)


def _filter(w, corr, h):
    """Periodic Gaussian filter of standard deviation `corr`, then mean 0 and
    standard deviation 1 (per part of a complex field)."""
    ny, n = w.shape[-2:]
    fx = torch.fft.fftfreq(n, d=h, device=DEV, dtype=torch.float64)[None, :]
    fy = torch.fft.fftfreq(ny, d=h, device=DEV, dtype=torch.float64)[:, None]
    z = torch.fft.ifft2(torch.fft.fft2(w) * torch.exp(-2.0 * math.pi ** 2 * corr ** 2 * (fx ** 2 + fy ** 2)))
    return z if w.is_complex() else z.real


def _slowness(kind, n, ny, gen):
    """s = min c / c of a log-normal medium c = 3^z, or of six smoothed
    horizontal layers with c from 1.5 to 4.5 times (1 + 0.1 z)."""
    x, y, h = _grid(n, ny)
    z = _filter(_randn(gen, ny, n), 0.1, h)
    z = (z - z.mean()) / z.std()
    if kind == "lognormal":
        z = (z - z.min()) / (z.max() - z.min())
        c = 3.0 ** z
        return c.min() / c
    layer = torch.clamp(torch.floor(6 * y[:, 0] / ((ny + 1) * h)), 0, 5)
    prof = 1.5 + 3.0 * layer / 5
    rad = 16
    t = torch.arange(-rad, rad + 1, device=DEV, dtype=torch.float64)
    ker = torch.exp(-0.5 * (t / 4.0) ** 2)
    prof = F.conv1d(F.pad(prof[None, None], (rad, rad), mode="replicate"), (ker / ker.sum())[None, None])[0, 0]
    c = torch.clamp(prof[:, None] * (1 + 0.1 * z), 1.5, 4.5)
    return 1.5 / c


def _godunov(tau, f):
    """One update of every node from its neighbours (tau = inf outside)."""
    p = F.pad(tau, (1, 1, 1, 1), value=1e300)
    a = torch.minimum(p[..., 1:-1, :-2], p[..., 1:-1, 2:])
    b = torch.minimum(p[..., :-2, 1:-1], p[..., 2:, 1:-1])
    d = a - b
    two = d.abs() < f
    root = torch.sqrt(torch.where(two, 2 * f * f - d * d, torch.zeros_like(d)))
    return torch.where(two, 0.5 * (a + b + root), torch.minimum(a, b) + f)


def _travel_time(s, x0, y0, tol):
    """Fixed point of the first-order Godunov scheme, nodes within 3h of the
    source at s(x0) |x - x0| (fields of shape (..., ny, n))."""
    ny, n = s.shape[-2:]
    x, y, h = _grid(n, ny)
    r = torch.sqrt((x - x0) ** 2 + (y - y0) ** 2)
    i0 = min(max(int(math.floor(x0 / h - 0.5)), 0), n - 1)
    j0 = min(max(int(math.floor(y0 / h - 0.5)), 0), ny - 1)
    fixed = r <= 3 * h
    start = torch.where(fixed, s[..., j0, i0, None, None] * r, torch.full_like(s, 1e300))
    f, tau = s * h, start
    for it in range(20 * (n + ny)):
        new = torch.where(fixed, start, torch.minimum(tau, _godunov(tau, f)))
        if it % 64 == 63 and bool((tau - new).max() <= tol):
            return new
        tau = new
    return tau


def _at(field, n, ny, x, y, mode):
    """The grid field (ny rows of n) at the coordinates x (row), y (column)."""
    h = 1.0 / (max(n, ny) + 1)
    gx = (2 * (x / h - 1) + 1) / n - 1
    gy = (2 * (y / h - 1) + 1) / ny - 1
    g = torch.stack([gx.expand(y.shape[0], x.shape[1]), gy.expand(y.shape[0], x.shape[1])], -1)
    return F.grid_sample(field[None, None], g[None], mode=mode, padding_mode="border", align_corners=False)[0, 0]


def _phase(s, x0, y0):
    """Travel-time phase |x - x0| tau_1, tau_1 from a coarse eikonal solve."""
    ny, n = s.shape
    x, y, h = _grid(n, ny)
    m = max(n, ny)
    mc = min(m, 95)
    cx, cy = max(8, round(n * mc / m)), max(8, round(ny * mc / m))
    xc, yc, hc = _grid(cx, cy)
    tc = _travel_time(_at(s, n, ny, xc, yc, "bilinear"), x0, y0, 1e-9)
    rc = torch.sqrt((xc - x0) ** 2 + (yc - y0) ** 2)
    tau1 = tc / rc.clamp_min(1e-9)
    return torch.sqrt((x - x0) ** 2 + (y - y0) ** 2) * _at(tau1, cx, cy, x, y, "bicubic")


def _medium(case, n, ny, gen, seed):
    """k, phi, omega and the source position of one instance."""
    pick = np.random.default_rng([seed, n, ny])
    h = 1.0 / (max(n, ny) + 1)
    fx, fy = pick.uniform(0.3, 0.7, 2)
    # the centre of a grid cell: at no node
    x0 = (math.floor(fx * (n + 1)) + 0.5) * h
    y0 = (math.floor(fy * (ny + 1)) + 0.5) * h
    s = _slowness(case["medium"], n, ny, gen)
    omega = case.get("kh", 0.4) / h
    return s, omega, x0, y0


def _instances(case, seed):
    out = []
    for b, (n, ny) in enumerate(_sizes(case)):
        gen = torch.Generator(DEV).manual_seed(1000003 * seed + b)
        s, omega, x0, y0 = _medium(case, n, ny, gen, seed + 7919 * b)
        x, y, h = _grid(n, ny)
        if case["op"] in ("cycle", "train"):
            # a residual of an outer iteration: waves of the medium's length
            g = _filter(torch.complex(_randn(gen, ny, n), _randn(gen, ny, n)), 0.5 / omega, h)
            g = g / torch.linalg.vector_norm(g)
        else:
            # a Gaussian source two spacings wide
            sg = 2 * h
            g = torch.exp(-((x - x0) ** 2 + (y - y0) ** 2) / (2 * sg * sg)) / (2 * math.pi * sg * sg)
            g = g.to(torch.complex128)
        out.append(dict(n=n, ny=ny, omega=omega, k=omega * s, phi=_phase(s, x0, y0), g=g))
    return out


def _params(case):
    return dict(precision=case["prec"], M=case["M"], adr_bc=case["adr_bc"], outer="fgmres", restart=RESTART, tol=0.0,
                maxit=1 << 30)


def _spec(insts, bc):
    return [(I["n"], I["omega"], I["k"], I["phi"], bc, I["ny"]) for I in insts]


class _Handle:
    def __init__(self, insts, bc, params):
        self.h = B.mg_setup(_spec(insts, bc), B.default_params(**params))

    def __del__(self):
        B.mg_destroy(self.h)


def prepare(case, seed):
    op = case["op"]
    if op == "eikonal":
        n, ny = _shape(case)
        gen = torch.Generator(DEV).manual_seed(seed)
        s, _, x0, y0 = _medium(case, n, ny, gen, seed)
        return dict(op=op, n=n, ny=ny, s=s.contiguous(), x0=x0, y0=y0)
    if op == "residual":
        n, ny = _shape(case)
        gen = torch.Generator(DEV).manual_seed(seed)
        s, omega, _, _ = _medium(case, n, ny, gen, seed)
        h = 1.0 / (max(n, ny) + 1)
        u = _filter(torch.complex(_randn(gen, ny, n), _randn(gen, ny, n)), 0.5 / omega, h).contiguous()
        g = torch.complex(_randn(gen, ny, n), _randn(gen, ny, n))
        return dict(op=op, n=n, ny=ny, omega=omega, k=(omega * s).contiguous(), bc=case["bc"], u=u, g=g)
    insts = _instances(case, seed)
    for I in insts:
        I["k"], I["phi"], I["g"] = (I[f].contiguous() for f in ("k", "phi", "g"))
    if op == "train":
        I = insts[0]
        gen = torch.Generator(DEV).manual_seed(seed + 1)
        want = torch.complex(_randn(gen, I["ny"], I["n"]), _randn(gen, I["ny"], I["n"]))
        lv = _levels(I, case["bc"], "zero")
        w = torch.tensor([_jacobi_weight(lv[0])] + [_alpha(lv[q]) for q in _cheb_levels(lv)], dtype=torch.float64,
                         device=DEV)
        return dict(op=op, I=I, M=case["M"], bc=case["bc"], K=case["K"], w=w, want=want * 1e-4, u0=torch.zeros_like(I["g"]))
    st = dict(op=op, insts=insts, bc=case["bc"], params=_params(case), steps=case.get("steps", 0),
              shapes=[(I["ny"], I["n"]) for I in insts])
    dt = torch.complex128 if case["prec"] == "fp64" or op != "cycle" else torch.complex64
    st["g"] = torch.cat([I["g"].reshape(-1) for I in insts]).to(dt)
    if op != "medium":
        st["handle"] = _Handle(insts, case["bc"], st["params"])
        for I in insts:
            I.clear()
    return st


# ------------------------------------------------------------------ runs
def _iterate(h, g, steps):
    """FGMRES steps from zero; the field is kept in single precision, as the
    complex-FP32 cycles that built it, with the FP64 relative residual."""
    u = torch.zeros_like(g)
    B.mg_solve_begin(h, u, g)
    B.mg_solve_steps(h, steps)
    rel = B.mg_solve_end(h, u)
    return {"u": u.to(torch.complex64), "residual": rel}


def run(state):
    op = state["op"]
    if op == "cycle":
        u = torch.zeros_like(state["g"])
        B.mg_cycle(state["handle"].h, u, state["g"], 1)
        return u
    if op == "solve":
        return _iterate(state["handle"].h, state["g"], state["steps"])
    if op == "medium":
        h = B.mg_setup(_spec(state["insts"], state["bc"]), B.default_params(**state["params"]))
        out = _iterate(h, state["g"], state["steps"])
        B.mg_destroy(h)
        return out
    if op == "train":
        I = state["I"]
        phi, w = I["phi"].detach().requires_grad_(), state["w"].detach().requires_grad_()
        u = AG.cycles(phi, w, state["u0"], I["g"], n=I["n"], omega=I["omega"], k=I["k"], bc=state["bc"], K=state["K"],
                      M=state["M"])
        loss = (u - state["want"]).abs().square().sum()
        gphi, gw = torch.autograd.grad(loss, (phi, w))
        return {"u": u.detach(), "phi": gphi, "weights": gw}
    if op == "eikonal":
        tau = torch.empty_like(state["s"])
        B.mg_eikonal_rect(state["n"], state["ny"], state["s"], state["x0"], state["y0"], tau)
        return tau
    r = torch.empty_like(state["u"])
    norm2 = torch.empty(1, dtype=torch.float64, device=DEV)
    B.mg_residual_norm_noalloc_rect(state["n"], state["ny"], state["omega"], state["k"], state["bc"], state["u"],
                                    state["g"], r, norm2)
    return {"r": r, "norm2": norm2}


# ------------------------------------------------------------------ work
def _cycle_work(n, ny, M, C, R):
    """Bytes and operations of one cycle: every pass that a global sum or the
    recursion forces reads its operands once and writes its results once
    (C, R: bytes of a complex and a real value; the ADR coefficients are two
    reals and a complex)."""
    by = fl = 0.0
    level = 1
    while max(n, ny) > 15:
        p = n * ny
        if level == 1:
            by += p * ((2 * C + R + C / 4) + (3 * C + R + C / 4))
            fl += p * 120
        elif level == 3:
            by += p * (C + C / 4 + C / 4 + C)
            fl += p * 30
        else:
            by += p * ((2 * C + R) + (2 * C + R + C / 4) + (3 * C + R + C / 4))
            fl += p * (10 * 56 + 60)
        if level >= 2:
            Q = 2 * R + C
            pre = (C + Q) + (2 * C + Q + C / 4)            # Gram sums; x, restricted residual
            post = (2 * C + Q + C / 4) + (3 * C + Q + C / 4)   # Gram sums of b - L x'; x
            by += M * p * (pre + post + ((4 * C + R) if level == 2 else 0))
            fl += M * p * (2 * (3 * 46 + 80) + 150)
        n, ny, level = n // 2, ny // 2, level + 1
    N = n * ny
    by += (M + 1) * N * N * C
    fl += (M + 1) * 8 * N * N
    return by, fl


def work(case):
    op = case["op"]
    n, ny = _shape(case)
    p = n * ny
    if op == "eikonal":
        return {"bytes": 16.0 * p, "flops": 12.0 * p}
    if op == "residual":
        return {"bytes": 56.0 * p, "flops": 30.0 * p}
    if op == "train":
        by, fl = _cycle_work(n, ny, case["M"], 16, 8)
        # a forward cycle, the same again for the tape, twice that in reverse
        return {"bytes": 4 * case["K"] * by, "flops": 4 * case["K"] * fl}
    by = fl = 0.0
    C, R = (16, 8) if case["prec"] == "fp64" else (8, 4)
    for m, my in _sizes(case):
        b, f = _cycle_work(m, my, case["M"], C, R)
        if op == "cycle":
            by, fl = by + b, fl + f
            continue
        q, S = m * my, case["steps"]
        # step j: z and A z written, two passes over the j + 2 Krylov vectors; at the end u and r
        by += S * b + q * sum(2 * (j + 2) * C + 3 * C for j in range(S)) + q * (S * C + 6 * 16)
        fl += S * f + q * sum(32 * (j + 1) + 30 for j in range(S))
        if op == "medium":
            by += 4.0 / 3 * q * 100
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ exact values
# The method in complex128, written from the paper with plain torch operations.
def _inject(a):
    ny, n = a.shape
    return a[1: 2 * (ny // 2): 2, 1: 2 * (n // 2): 2]


def _edges(ny, n):
    m = torch.zeros(ny, n, dtype=torch.float64, device=DEV)
    m[:, 0] += 1
    m[:, -1] += 1
    m[0] += 1
    m[-1] += 1
    return m


def _diag(k, sig, h, bc):
    """h^2 times the diagonal of the 5-point operator with its boundary."""
    d = (4.0 - (k * h) ** 2).to(torch.complex128)
    if bc == "abc1":
        d = d - _edges(*k.shape) * (1 + 1j * k * h)
    elif bc == "sponge":
        d = d - 1j * h * h * sig
    return d


def _nb(u):
    p = F.pad(torch.view_as_real(u), (0, 0, 1, 1, 1, 1))
    p = torch.view_as_complex(p)
    return p[1:-1, :-2], p[1:-1, 2:], p[:-2, 1:-1], p[2:, 1:-1]


def _A(lv, u, conj=False):
    w, e, s, t = _nb(u)
    d = lv["d"].conj() if conj else lv["d"]
    return (d * u - (w + e + s + t)) / lv["h"] ** 2


def _sponge(n, ny, omega, k):
    x, y, h = _grid(n, ny)
    lx, ly = (n + 1) * h, (ny + 1) * h
    dist = torch.minimum(torch.minimum(x, lx - x), torch.minimum(y, ly - y))
    W = 2 * math.pi / omega
    gam = torch.where(dist < W, omega * ((W - dist) / W) ** 2, torch.zeros_like(dist))
    return omega * gam * (k / omega) ** 2


def _extend(p):
    p = torch.cat([2 * p[:, :1] - p[:, 1:2], p, 2 * p[:, -1:] - p[:, -2:-1]], 1)
    return torch.cat([2 * p[:1] - p[1:2], p, 2 * p[-1:] - p[-2:-1]], 0)


def _adr(k, sig, phi, h, omega, bc, closure):
    """Upwind stencil (centre, W, E, S, N) of the ADR operator."""
    q = _extend(phi)
    W, E, S, N = q[1:-1, :-2], q[1:-1, 2:], q[:-2, 1:-1], q[2:, 1:-1]
    px, py = (E - W) / (2 * h), (N - S) / (2 * h)
    lap = (E + W + N + S - 4 * phi) / (h * h)
    ax, ay = px.abs(), py.abs()
    d = torch.complex(4 / (h * h) + omega ** 2 * (px ** 2 + py ** 2) - k ** 2, -2 * omega * (ax + ay) / h - omega * lap)
    if bc == "sponge":
        d = d - 1j * sig
    one = torch.full_like(px, -1 / (h * h))
    c = [torch.complex(one, omega * (px + ax) / h), torch.complex(one, omega * (ax - px) / h),
         torch.complex(one, omega * (py + ay) / h), torch.complex(one, omega * (ay - py) / h)]
    if closure == "abc" and bc == "abc1":
        add = torch.zeros_like(d)
        for cf, at, inner in ((c[0], np.s_[:, :1], np.s_[:, 1:2]), (c[1], np.s_[:, -1:], np.s_[:, -2:-1]),
                              (c[2], np.s_[:1], np.s_[1:2]), (c[3], np.s_[-1:], np.s_[-2:-1])):
            g = torch.zeros_like(d)
            g[at] = cf[at] * (1 + 1j * k[at] * h) * torch.exp(-1j * omega * (phi[at] - phi[inner]))
            add = add + g
        d = d + add
    return d, c


def _L(lv, a):
    w, e, s, t = _nb(a)
    c = lv["c"]
    return lv["c0"] * a + c[0] * w + c[1] * e + c[2] * s + c[3] * t


def _levels(I, bc, closure, phi=None):
    n, ny, omega = I["n"], I["ny"], I["omega"]
    k, phi = I["k"], I["phi"] if phi is None else phi
    sig = _sponge(n, ny, omega, k) if bc == "sponge" else None
    out = []
    while True:
        h = 1.0 / (max(n, ny) + 1)
        lv = dict(n=n, ny=ny, h=h, k=k, d=_diag(k, sig, h, bc), bc=bc)
        if out:
            lv["c0"], lv["c"] = _adr(k, sig, phi, h, omega, bc, closure)
        if len(out) == 1:
            lv["mod"] = torch.exp(1j * omega * phi)
        out.append(lv)
        if max(n, ny) <= 15:
            break
        n, ny, k, phi = n // 2, ny // 2, _inject(k), _inject(phi)
        sig = None if sig is None else _inject(sig)
    eye = torch.eye(n * ny, dtype=torch.complex128, device=DEV).reshape(-1, ny, n)
    lv = out[-1]
    lv["A"] = torch.stack([_A(lv, e).reshape(-1) for e in eye], 1)
    lv["LA"] = torch.stack([_L(lv, e).reshape(-1) for e in eye], 1)
    return out


def _cheb_levels(lv):
    return [q for q in range(1, len(lv) - 1) if q != 2]


def _jacobi_weight(lv):
    kap = (lv["h"] * float(lv["k"].max())) ** 2
    return (4 - kap) / (5 - kap)


def _alpha(lv):
    """Largest over median squared eigenvalue of the constant-k operator."""
    n, ny, h, k = lv["n"], lv["ny"], lv["h"], float(lv["k"].max())

    def sines(m):
        return 4 * torch.sin(torch.arange(1, m + 1, device=DEV, dtype=torch.float64) * math.pi / (2 * (m + 1))) ** 2 / h ** 2

    ev = (sines(ny)[:, None] + sines(n)[None, :] - k * k).square().reshape(-1).sort()[0]
    N = ev.numel()
    med = ev[N // 2] if N % 2 else 0.5 * (ev[N // 2 - 1] + ev[N // 2])
    return float(ev[-1] / med)


def _restrict(r):
    ny, n = r.shape
    p = torch.view_as_complex(F.pad(torch.view_as_real(r), (0, 0, 1, 1, 1, 1)))
    cy, cx = ny // 2, n // 2
    out = 0
    for b, wb in enumerate((1, 2, 1)):
        for a, wa in enumerate((1, 2, 1)):
            out = out + wa * wb / 16 * p[b + 1: b + 1 + 2 * cy: 2, a + 1: a + 1 + 2 * cx: 2]
    return out


def _prolong(e, n, ny):
    # along each direction: the coarse value at odd nodes, the mean of the two neighbours at even ones
    def lines(a, m):
        z = torch.zeros_like(a[:1])
        q = torch.cat([z, a, z], 0)
        mid = 0.5 * (q[:-1] + q[1:])
        o = torch.stack([mid[:-1], a], 1).reshape(-1, a.shape[1])
        return torch.cat([o, mid[-1:]], 0)[:m] if m % 2 else o
    return lines(lines(e, ny).T, n).T


def _cheb(lv, x, g, lam, alpha, q=5):
    a = lam / alpha
    theta, delta = 0.5 * (a + lam), 0.5 * (lam - a)
    sigma = theta / delta
    rho = 1 / sigma
    d = 0
    for m in range(q):
        s = _A(lv, g - _A(lv, x), conj=True)
        if m == 0:
            d = s / theta
        else:
            new = 1 / (2 * sigma - rho)
            d = new * rho * d + (2 * new / delta) * s
            rho = new
        x = x + d
    return x


def _gmres3(lv, b, x):
    """One GMRES(3) sweep from x (None: zero)."""
    r = b if x is None else b - _L(lv, x)
    beta = torch.sqrt((r.conj() * r).real.sum())
    V = [r / beta]
    H = []
    for j in range(3):
        w = _L(lv, V[j])
        col = []
        for v in V:
            hij = (v.conj() * w).sum()
            w = w - hij * v
            col.append(hij)
        nw = torch.sqrt((w.conj() * w).real.sum())
        H.append(torch.stack(col + [nw.to(torch.complex128)] + [torch.zeros_like(hij)] * (2 - j)))
        V.append(w / nw)
    H = torch.stack(H, 1)
    Q, R = torch.linalg.qr(H)
    y = torch.linalg.solve(R, Q[0].conj() * beta)
    z = y[0] * V[0] + y[1] * V[1] + y[2] * V[2]
    return z if x is None else x + z


def _adr_cycle(lvs, l, b):
    lv = lvs[l]
    if l == len(lvs) - 1:
        return torch.linalg.solve(lv["LA"], b.reshape(-1)).reshape(b.shape)
    x = _gmres3(lv, b, None)
    e = _adr_cycle(lvs, l + 1, _restrict(b - _L(lv, x)))
    return _gmres3(lv, b, x + _prolong(e, lv["n"], lv["ny"]))


def _cycle(lvs, l, u, g, M, wj, alphas):
    lv = lvs[l]
    if l == len(lvs) - 1:
        return torch.linalg.solve(lv["A"], g.reshape(-1)).reshape(g.shape)
    n, ny, h2 = lv["n"], lv["ny"], lv["h"] ** 2
    smooth = l in alphas
    if l == 0:
        u = u + wj * h2 * (g - _A(lv, u)) / lv["d"]
    elif smooth:
        nbr = 4 - _edges(ny, n)
        lam = ((lv["d"].abs() + nbr) / h2).max() ** 2
        u = _cheb(lv, u, g, lam, alphas[l])
    e = _cycle(lvs, l + 1, torch.zeros(ny // 2, n // 2, dtype=torch.complex128, device=DEV), _restrict(g - _A(lv, u)),
               M, wj, alphas)
    u = u + _prolong(e, n, ny)
    if l == 0:
        return u + wj * h2 * (g - _A(lv, u)) / lv["d"]
    if smooth:
        u = _cheb(lv, u, g, lam, alphas[l])
    if l == 1:
        for _ in range(M):
            b = lv["mod"].conj() * (g - _A(lv, u))
            u = u + lv["mod"] * _adr_cycle(lvs, 1, b)
    return u


def _exact_cycle(lvs, M):
    alphas = {q: _alpha(lvs[q]) for q in _cheb_levels(lvs)}
    wj = _jacobi_weight(lvs[0])
    return lambda g: _cycle(lvs, 0, torch.zeros_like(g), g, M, wj, alphas)


def _exact_fgmres(lvs, M, g, steps):
    """`steps` <= RESTART flexible GMRES iterations from zero."""
    pre = _exact_cycle(lvs, M)
    beta = torch.linalg.vector_norm(g)
    V, Z, H = [g / beta], [], torch.zeros(steps + 1, steps, dtype=torch.complex128, device=DEV)
    for j in range(steps):
        z = pre(V[j])
        w = _A(lvs[0], z)
        for _ in range(2):
            for i, v in enumerate(V):
                c = (v.conj() * w).sum()
                H[i, j] += c
                w = w - c * v
        nw = torch.linalg.vector_norm(w)
        H[j + 1, j] = nw
        V.append(w / nw)
        Z.append(z)
    Q, R = torch.linalg.qr(H)
    y = torch.linalg.solve(R, Q[0].conj() * beta)
    u = sum(y[j] * Z[j] for j in range(steps))
    return u, float(torch.linalg.vector_norm(g - _A(lvs[0], u)) / beta)


def exact(case, seed):
    op = case["op"]
    if op == "eikonal":
        st = prepare(case, seed)
        return _travel_time(st["s"], st["x0"], st["y0"], 1e-14)
    if op == "residual":
        n, ny = _shape(case)
        st = prepare(case, seed)
        sig = _sponge(n, ny, st["omega"], st["k"]) if st["bc"] == "sponge" else None
        h = 1.0 / (max(n, ny) + 1)
        lv = dict(h=h, d=_diag(st["k"], sig, h, st["bc"]))
        r = st["g"] - _A(lv, st["u"])
        return {"r": r, "norm2": r.abs().square().sum().reshape(1)}
    insts = _instances(case, seed)
    if op == "train":
        I = insts[0]
        st = prepare(case, seed)
        phi = I["phi"].clone().requires_grad_()
        w = st["w"].clone().requires_grad_()
        lvs = _levels(I, case["bc"], "zero", phi)
        alphas = {q: w[1 + i] for i, q in enumerate(_cheb_levels(lvs))}
        u = torch.zeros_like(I["g"])
        for _ in range(case["K"]):
            u = _cycle(lvs, 0, u, I["g"], case["M"], w[0], alphas)
        loss = (u - st["want"]).abs().square().sum()
        gphi, gw = torch.autograd.grad(loss, (phi, w))
        return {"u": u.detach(), "phi": gphi, "weights": gw}
    parts, rel = [], 0.0
    for I in insts:
        lvs = _levels(I, case["bc"], case["adr_bc"])
        if op == "cycle":
            g = I["g"] if case["prec"] == "fp64" else I["g"].to(torch.complex64).to(torch.complex128)
            u = _exact_cycle(lvs, case["M"])(g)
        else:
            u, r = _exact_fgmres(lvs, case["M"], I["g"], case["steps"])
            rel = max(rel, r)
        parts.append(u.reshape(-1))
    u = torch.cat(parts)
    return u if op == "cycle" else {"u": u, "residual": rel}
