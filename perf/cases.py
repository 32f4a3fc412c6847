"""What a user of this framework has it do, as cases that can be timed and compared.

A case is a dict of plain values.  `listed()` gives the fixed ones, `draw(rng)`
more of the same ranges, `prepare(case, seed)` what a program holds before the
call (an `AllAtOnce` solver and its inputs), `run(state)` one pass through the
public entry points, `work(case)` the bytes and operations no implementation
can do without, and `exact(case, seed)` the same outputs in 64-bit torch.

kind        entry point
----------  -----------------------------------------------------------------
apply       AllAtOnce.precond_apply: y = P^{-1} x or P^{-T} x
neumann     AllAtOnce.neumann_apply: y = Q_i^{-1} x on a perturbed time grid
matvec_f32  AllAtOnce.matvec_f32: A x - v of an FP32 basis vector
dots        AllAtOnce.matvec_dots: w = A x - v with v0.w, v.w, w.w
residual    AllAtOnce.residual: r = A x - b and its squared norm
solve       AllAtOnce.build_rhs + solve: flexible GMRES from initial data
gradient    AAOSolve forward and backward: d loss / d u0, d loss / d kappa

The plain FP32 preconditioner's results are FP32 numbers widened to FP64; a
mixed-precision program keeps them as FP32, so those passes end in that cast.
"""
import math

import numpy as np
import torch

from paper_1810_00615_gb300 import AAOSolve, AllAtOnce

F64 = torch.float64


def _case(name, kind, n, ell, **kw):
    c = {"name": name, "kind": kind, "n": n, "ell": ell, "equation": "heat", "precision": "fp32_refined",
         "transpose": False, "terms": 1, "delta": 0.0, "restart": 30, "rtol": 1e-10}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest solve: a coarse heat problem inside someone's outer loop,
        # all FP64; launches and host round trips are what it costs
        _case("solve_n63_l64", "solve", 63, 64, precision="fp64"),
        # the headline: heat, 16.8 million unknowns, refined FP32 circulant
        _case("solve_n4095_l4096", "solve", 4095, 4096),
        # an inverse problem's step: forward solve, adjoint solve, both gradients
        _case("gradient_n16383_l1024", "gradient", 16383, 1024, rtol=5e-9),
        # the preconditioner alone, as an outer Krylov method of the user's own
        # calls it: smallest transform that is split into four steps
        _case("apply32_n255_l256", "apply", 255, 256, precision="fp32"),
        # ... the benchmark size
        _case("apply32_n4095_l4096", "apply", 4095, 4096, precision="fp32"),
        # ... refined, for the paper's largest Table 1 problem: ell not a power of two, a row
        # length that does not divide into whole chunks, transposed (adjoint)
        _case("apply_t_n1568_l1440", "apply", 1568, 1440, transpose=True),
        # ... the paper's Table 2 (f) problem with the FP64 preconditioner
        _case("apply64_n1024_l1024", "apply", 1024, 1024, precision="fp64"),
        # ... the finest grid: frequency rows longer than one CTA can hold
        _case("apply32_n65535_l512", "apply", 65535, 512, precision="fp32"),
        # the Neumann-series preconditioner with two extra terms on a perturbed
        # time grid, plain FP32
        _case("neumann32_n4095_l4096", "neumann", 4095, 4096, precision="fp32", terms=3, delta=0.5),
        # the Arnoldi product of the FP64 and refined solves
        _case("dots_n4095_l4096", "dots", 4095, 4096),
        # the Arnoldi product of the plain FP32 solve's adjoint, ragged sizes
        _case("matvec32_t_n1000_l900", "matvec_f32", 1000, 900, transpose=True),
        # the true residual of the wave system (BD2: three block bands)
        _case("residual_bd2_n8191_l2048", "residual", 8191, 2048, equation="wave_bd2"),
    ]


#: Lengths 2^a 3^b 5^c that the time transforms take.
_LENGTHS = sorted({2 ** a * 3 ** b * 5 ** c for a in range(13) for b in range(6) for c in range(5)
                   if 16 <= 2 ** a * 3 ** b * 5 ** c <= 4096})


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["solve", "gradient", "apply", "apply", "apply", "neumann", "dots", "matvec_f32", "residual"])
    # half the lengths are powers of two, as in most uses
    ell = 2 ** rng.randint(4, 12) if rng.random() < 0.5 else min(_LENGTHS, key=lambda v, t=_log_int(rng, 16, 4096): abs(v - t))
    precision = rng.choice(["fp32", "fp32_refined", "fp32_refined", "fp64"])
    if kind == "apply" and rng.random() < 0.15:
        n = rng.choice([32767, 49151, 65535])
    elif rng.random() < 0.5:
        n = 2 ** rng.randint(5, 13) - 1
    else:
        n = _log_int(rng, 31, 16383)
    most = 2 ** 21 if precision == "fp64" else 2 ** 24
    while n * ell > most and ell > 16:
        ell = max(v for v in _LENGTHS if v < ell)
    if n * ell > most:
        n = 2047
    # a refined result is short of FP64 by about n^2 2^-48 (the pair arithmetic
    # of its residual); finer grids get their accuracy from the solver around it
    if precision == "fp32_refined" and (kind == "apply" and n > 2047 or kind == "neumann" and n > 1023):
        precision = "fp32"
    c = _case("", kind, n, ell, precision=precision, transpose=rng.random() < 0.4)
    del c["name"]
    if kind == "neumann":
        c.update(terms=rng.choice([2, 3]), delta=rng.choice([0.1, 0.5, 0.9]))
    elif kind in ("dots", "matvec_f32", "residual"):
        c.update(precision="fp32_refined", equation=rng.choice(["heat", "heat", "wave_bd2", "wave_bd4"]))
    elif kind == "solve":
        # finer grids at larger steps put the tolerance below what FP64 can
        # attain (eps |A| |U| / |b|, which grows like n^2 / ell)
        c.update(n=min(n, int(4096 * math.sqrt(ell / 512))), transpose=False)
        if rng.random() < 0.4:
            c.update(delta=0.5, terms=rng.choice([1, 2]))
    elif kind == "gradient":
        c.update(transpose=False, rtol=5e-9, n=min(n, int(16384 * math.sqrt(ell / 2048))))
    return c


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=F64)


def _steps(case, seed):
    """The perturbed time grid t_j = (j + delta (R_j - 1/2)) / ell, as steps."""
    ell = case["ell"]
    t = np.arange(ell + 1, dtype=np.float64)
    t[1:ell] += case["delta"] * (np.random.default_rng(seed).random(ell - 1) - 0.5)
    return np.diff(t / ell)


def _initial(n, seed):
    """Eight sine modes with coefficients N(0, 1) / j^2 at the interior nodes."""
    c = np.random.default_rng(seed).standard_normal(8) / np.arange(1, 9) ** 2
    x = torch.arange(1, n + 1, device="cuda", dtype=F64) / (n + 1)
    return sum(float(cj) * torch.sin(j * math.pi * x) for j, cj in enumerate(c, start=1))


def _field(case, g):
    """A block vector like a solution: smooth in space and time, with noise."""
    n, ell = case["n"], case["ell"]
    x = torch.arange(1, n + 1, device="cuda", dtype=F64) / (n + 1)
    t = torch.arange(1, ell + 1, device="cuda", dtype=F64) / ell
    j = torch.arange(1, 9, device="cuda", dtype=F64)
    a = _randn(g, 8) / j ** 2
    return (a * torch.exp(-j * t[:, None])) @ torch.sin(math.pi * j[:, None] * x) + 1e-3 * _randn(g, ell, n)


def _inputs(case, seed):
    """The inputs alone, the same for `prepare` and `exact`."""
    n, ell, kind, g = case["n"], case["ell"], case["kind"], _gen(seed)
    if kind in ("apply", "neumann"):
        return {"x": _randn(g, ell, n)}
    if kind == "matvec_f32":
        return {"x": _field(case, g).to(torch.float32), "v": _randn(g, ell, n)}
    if kind == "dots":
        return {"x": _field(case, g), "v": _randn(g, ell, n), "v0": _randn(g, ell, n)}
    if kind == "residual":
        return {"x": _field(case, g), "b": _randn(g, ell, n)}
    if kind == "solve":
        return {"u0": _initial(n, seed)}
    # observations: the solution of other initial data would do as well; a
    # decaying field with measurement noise has the same loss gradient scale
    return {"u0": _initial(n, seed), "obs": _field(case, g)}


def prepare(case, seed):
    kind = case["kind"]
    solver = AllAtOnce(case["n"], case["ell"], 1.0 / case["ell"], equation=case["equation"],
                       precision=case["precision"],
                       restart=case["restart"] if kind in ("solve", "gradient") else 1)
    if case["delta"]:
        solver.set_steps(_steps(case, seed))
    s = dict(_inputs(case, seed), case=case, solver=solver)
    if kind == "gradient":
        s["u0"].requires_grad_(True)
        s["kappa"] = torch.tensor(1.0, dtype=F64, requires_grad=True)
    return s


def _kept(case, y):
    return y.to(torch.float32) if case["precision"] == "fp32" else y


def run(s):
    c, a = s["case"], s["solver"]
    kind, tr = c["kind"], c["transpose"]
    if kind == "apply":
        return _kept(c, a.precond_apply(s["x"], transpose=tr))
    if kind == "neumann":
        return _kept(c, a.neumann_apply(s["x"], c["terms"], transpose=tr))
    if kind == "matvec_f32":
        return a.matvec_f32(s["x"], transpose=tr, sub=s["v"])
    if kind == "dots":
        w, d = a.matvec_dots(s["x"], s["v"], v0=s["v0"], transpose=tr)
        return [w, d]
    if kind == "residual":
        r, norm2 = a.residual(s["x"], s["b"], transpose=tr)
        return [r, norm2]
    if kind == "solve":
        U, _ = a.solve(a.build_rhs(s["u0"]), restart=c["restart"], rtol=c["rtol"], precond=c["terms"])
        return U
    u0, kappa = s["u0"], s["kappa"]
    u0.grad = kappa.grad = None
    U = AAOSolve.apply(u0, kappa, a, c["rtol"], c["restart"])
    loss = 0.5 * (U - s["obs"]).square().sum()
    loss.backward()
    return [U.detach(), loss.detach(), u0.grad, kappa.grad]


# -------------------------------------------------------------------- work

def work(case):
    n, ell, kind = case["n"], case["ell"], case["kind"]
    N = n * ell
    # one application of P^{-1}: two real FFTs along time (2.5 log2 ell per
    # point each) and a complex tridiagonal solve per stored frequency (about
    # 30 operations per unknown with the factors at hand: 15 per real point)
    apply = N * (5.0 * math.log2(ell) + 15.0)
    mv = N * {"heat": 9.0, "wave_bd2": 11.0, "wave_bd4": 13.0}[case["equation"]]
    if kind == "apply":
        return {"bytes": (12.0 if case["precision"] == "fp32" else 16.0) * N, "flops": apply}
    if kind == "neumann":
        return {"bytes": (12.0 if case["precision"] == "fp32" else 16.0) * N,
                "flops": case["terms"] * apply + (case["terms"] - 1) * 6.0 * N}
    if kind == "matvec_f32":
        return {"bytes": 20.0 * N, "flops": mv}
    if kind == "dots":
        return {"bytes": 32.0 * N, "flops": mv + 6.0 * N}
    if kind == "residual":
        return {"bytes": 24.0 * N, "flops": mv + 2.0 * N}
    if kind == "solve":
        # the initial data in, the solution out; exact time stepping (a
        # tridiagonal solve per step) is the least arithmetic known
        return {"bytes": 8.0 * (n + N), "flops": 13.0 * N}
    # observations in, U and the gradients out; a forward and a backward sweep
    return {"bytes": 16.0 * N + 16.0 * n, "flops": 32.0 * N}


# ------------------------------------------------------------------- exact

def _sine_symbols(n):
    """Eigenvalues of M and K (uniform P1 elements) on the sine modes 1..n."""
    h = 1.0 / (n + 1)
    s2 = torch.sin(torch.arange(1, n + 1, device="cuda", dtype=F64) * (math.pi / (2 * (n + 1)))) ** 2
    return h * (1.0 - (2.0 / 3.0) * s2), (4.0 / h) * s2


def _dst(x):
    """sum_i x_i sin(pi i j / (n+1)) along the last axis (its own inverse times 2/(n+1))."""
    n = x.shape[-1]
    z = x.new_zeros(*x.shape[:-1], 2 * (n + 1))
    z[..., 1:n + 1] = x
    z[..., n + 2:] = -x.flip(-1)
    f = torch.fft.fft(z) if x.is_complex() else torch.fft.rfft(z)
    y = f[..., 1:n + 1]
    return 0.5j * y if x.is_complex() else -0.5 * y.imag


def _circulant_inverse(case, x):
    """P^{-1} x (P^{-T} x): Fourier modes in time, sine modes in space."""
    n, ell = case["n"], case["ell"]
    tau = 1.0 / ell
    m, k = _sine_symbols(n)
    f = torch.fft.rfft(x, dim=0)
    out = torch.empty_like(f)
    th = torch.arange(f.shape[0], device="cuda", dtype=F64) * (2 * math.pi / ell)
    om = torch.complex(2 * torch.sin(th / 2) ** 2, torch.sin(th))      # 1 - w_k
    if case["transpose"]:
        om = om.conj()
    rows = max(1, (1 << 25) // (n + 1))
    for a in range(0, f.shape[0], rows):
        lam = om[a:a + rows, None] * m + tau * k
        out[a:a + rows] = _dst(_dst(f[a:a + rows].contiguous()) / lam) * (2.0 / (n + 1))
    return torch.fft.irfft(out, n=ell, dim=0)


def _stiff(x):
    """2 x_i - x_{i-1} - x_{i+1} along the last axis."""
    s = 2.0 * x
    s[..., 1:] -= x[..., :-1]
    s[..., :-1] -= x[..., 1:]
    return s


def _lag(q, j, transpose):
    """q_{t-j} (q_{t+j} for the transpose), zero outside."""
    out = torch.zeros_like(q)
    if j < q.shape[0]:
        if transpose:
            out[:q.shape[0] - j] = q[j:]
        else:
            out[j:] = q[:q.shape[0] - j]
    return out


def _product(case, x):
    """A x (A^T x) of the all-at-once system with uniform steps."""
    n, ell, tr = case["n"], case["ell"], case["transpose"]
    h, tau = 1.0 / (n + 1), 1.0 / ell
    s = _stiff(x)
    q = 6.0 * x - s
    if case["equation"] == "heat":
        return (h / 6.0) * (q - _lag(q, 1, tr)) + (tau / h) * s
    b = tau * tau / h
    w = [1.0, -2.0, 1.0] if case["equation"] == "wave_bd2" else [2.0, -5.0, 4.0, -1.0]
    S = sum(wj * _lag(q, j, tr) for j, wj in enumerate(w))
    if case["equation"] == "wave_bd4":
        # the two start-up block rows are the BD2 ones: M x_1 and M (x_2 - 2 x_1)
        if not tr:
            S[0] = q[0]
            if ell > 1:
                S[1] = q[1] - 2.0 * q[0]
        else:
            S[0] = q[0] - (2.0 * q[1] if ell > 1 else 0) + (4.0 * q[2] if ell > 2 else 0) - (q[3] if ell > 3 else 0)
            if ell > 1:
                S[1] = q[1] - (5.0 * q[2] if ell > 2 else 0) + (4.0 * q[3] if ell > 3 else 0) - (q[4] if ell > 4 else 0)
    return (h / 6.0) * S + b * s


def _heat_solution(case, u0, taus):
    """Implicit Euler from u0, mode by mode: factors m / (m + tau_t k)."""
    n = case["n"]
    m, k = _sine_symbols(n)
    r = m / (m + torch.as_tensor(taus, device="cuda", dtype=F64)[:, None] * k)
    return _dst(torch.cumprod(r, dim=0) * _dst(u0)) * (2.0 / (n + 1))


def exact(case, seed):
    n, ell, kind = case["n"], case["ell"], case["kind"]
    inp = _inputs(case, seed)
    if kind == "apply":
        return _circulant_inverse(case, inp["x"])
    if kind == "neumann":
        x = inp["x"]
        sig = torch.as_tensor(_steps(case, seed) - 1.0 / ell, device="cuda", dtype=F64)[:, None] * (n + 1)
        y = _circulant_inverse(case, x)
        for _ in range(1, case["terms"]):
            y = _circulant_inverse(case, x - sig * _stiff(y))
        return y
    if kind == "matvec_f32":
        return _product(case, inp["x"].to(F64)) - inp["v"]
    if kind == "dots":
        w = _product(case, inp["x"]) - inp["v"]
        return [w, [float((inp["v0"] * w).sum()), float((inp["v"] * w).sum()), float((w * w).sum())]]
    if kind == "residual":
        r = _product(case, inp["x"]) - inp["b"]
        return [r, float((r * r).sum())]
    if kind == "solve":
        return _heat_solution(case, inp["u0"], _steps(case, seed))
    # gradient: the adjoint recursion (m + tau k) l_t - m l_{t+1} = g_t per mode
    tau = 1.0 / ell
    m, k = _sine_symbols(n)
    U = _heat_solution(case, inp["u0"], np.full(ell, tau))
    g = U - inp["obs"]
    loss = 0.5 * g.square().sum()
    gh, uh = _dst(g), _dst(U)
    lam, gk = torch.zeros(n, device="cuda", dtype=F64), torch.zeros((), device="cuda", dtype=F64)
    for t in range(ell - 1, -1, -1):
        lam = (gh[t] + m * lam) / (m + tau * k)
        gk -= tau * (lam * k * uh[t]).sum()
    c = 2.0 / (n + 1)
    return [U, loss, _dst(m * lam) * c, gk * c]
