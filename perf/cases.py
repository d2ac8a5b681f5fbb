"""What a user of this library has it do, as cases that can be timed and compared.

Each case is a dict of plain values with a "kind"; prepare() makes the device inputs and the
context a program would hold before the call, run() makes one pass through the public binding,
exact() gives the same outputs in 64 bits with plain torch (no code of this package).

Kinds:
  update     one iteration of a caller's own loop: fot_u_update, then fot_v_update, from an
             iterate the caller holds
  solve      Algorithm 1 from the standard start: fot_solve, then fot_potentials
  batch      independent problems of their own sizes: fot_batch_solve, then every problem's
             potentials
  phase      the phase step from a converged iterate: fot_moments (Dx, Dy and the phase)
  backward   a training step: fot_phase_fn and the gradients of a loss of the phase and the
             target potential with respect to both amplitudes
  intensity  the far field and the L1 intensity loss of a phase: fot_intensity_loss
  cfot       the FFT-convolution form at large eps: fot_cfot_solve, then fot_potentials
  rect       input and output grids of different sizes: fot_solve_rect
"""
import math
import random

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2512_19072_gb300 import binding as B

PRECISION = {"fp32": B.FOT_FP32, "mixed": B.FOT_MIXED, "bf16": B.FOT_BF16, "dense": B.FOT_FP32_DENSE}
BATCH_SIZES = (128, 192, 256, 384, 512)


def listed():
    return [
        # A caller's own loop on a small ragged grid: a handful of launches per call, rows that
        # are not 16-byte aligned.
        dict(name="update_257x201_fp32", kind="update", rows=257, cols=201, precision="fp32", eps=20.0),
        # The smallest solve of the configurations: 64^2, a fixed eps of one square pixel, 200
        # iterations; latency of the launches.
        dict(name="solve_64_fp32", kind="solve", rows=64, cols=64, precision="fp32", eps0=1.0, eps1=1.0, iters=200),
        # The annealed 256^2 solve, eps 64 to 1 over 300 iterations: wide kernels first, narrow
        # ones at the end.
        dict(name="solve_256_anneal_mixed", kind="solve", rows=256, cols=256, precision="mixed", eps0=64.0, eps1=1.0,
             iters=300),
        # The working size: 1024^2 at the paper's eps (2e-4 n^2), 200 iterations, in both forms.
        dict(name="solve_1024_fp32", kind="solve", rows=1024, cols=1024, precision="fp32", eps0=209.7152,
             eps1=209.7152, iters=200),
        dict(name="solve_1024_mixed", kind="solve", rows=1024, cols=1024, precision="mixed", eps0=209.7152,
             eps1=209.7152, iters=200),
        # The largest size of the configurations.
        dict(name="solve_2048_mixed", kind="solve", rows=2048, cols=2048, precision="mixed", eps0=838.8608,
             eps1=838.8608, iters=100),
        # Many independent problems of uneven size, annealed 32 to 1.
        dict(name="batch_20_fp32", kind="batch", count=20, precision="fp32", eps0=32.0, eps1=1.0, iters=40),
        # The phase that ends every solve at the working size.
        dict(name="phase_1024", kind="phase", rows=1024, cols=1024, eps=209.7152),
        # A training step through 30 unrolled iterations.
        dict(name="backward_256_fp32", kind="backward", rows=256, cols=256, precision="fp32", eps=130.0, iters=30,
             every=10),
        # The loss a user looks at after each solve of an eps sweep.
        dict(name="intensity_1024", kind="intensity", rows=1024, cols=1024),
        # The FFT form, where eps is large enough for it.
        dict(name="cfot_512", kind="cfot", rows=512, cols=512, eps=20000.0, iters=50),
        # Different grids on the two planes, none of the four sizes aligned with another.
        dict(name="rect_300x257_to_385x212", kind="rect", rows=300, cols=257, rows_out=385, cols_out=212, eps=60.0,
             iters=30),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, lo, hi):
    """Two sides within a factor of two of each other; odd and unaligned ones as often as not."""
    a = _log_int(rng, lo, hi)
    b = min(hi, max(lo, int(round(a * math.exp(rng.uniform(-0.7, 0.7))))))
    if rng.random() < 0.5:
        a, b = max(lo, a // 16 * 16), max(lo, b // 16 * 16)
    return a, b


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "update", "update", "batch", "phase", "backward",
                       "intensity", "cfot", "rect"])
    if kind == "update":
        r, c = _sides(rng, 48, 2048)
        n = max(r, c)
        eps = math.exp(rng.uniform(math.log(max(1.0, 5e-5 * n * n)), math.log(2e-3 * n * n + 1.0)))
        prec = rng.choice(["fp32", "mixed", "mixed", "bf16"] + (["dense"] if n <= 512 else []))
        return dict(kind=kind, rows=r, cols=c, precision=prec, eps=round(eps, 4))
    if kind == "solve":
        r, c = _sides(rng, 48, 1536)
        n = max(r, c)
        prec = rng.choice(["fp32", "mixed", "mixed"])
        if n <= 320 and rng.random() < 0.6:                 # annealed to small eps
            eps1 = math.exp(rng.uniform(0.0, math.log(4.0)))
            eps0 = eps1 * math.exp(rng.uniform(math.log(4.0), math.log(64.0)))
        else:
            eps0 = eps1 = math.exp(rng.uniform(math.log(max(1.0, 1e-4 * n * n)), math.log(1e-3 * n * n + 1.0)))
        cost = 2.0 * r * c * (r + c)                        # terms of one dense iteration
        iters = int(max(16, min(rng.randint(40, 200), 60e10 / cost)))
        return dict(kind=kind, rows=r, cols=c, precision=prec, eps0=round(eps0, 4), eps1=round(eps1, 4), iters=iters)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 20), precision=rng.choice(["fp32", "mixed"]),
                    eps0=round(rng.uniform(20.0, 64.0), 3), eps1=round(rng.uniform(1.0, 8.0), 3),
                    iters=rng.randint(20, 40))
    if kind == "phase":
        r, c = _sides(rng, 64, 1536)
        n = max(r, c)
        return dict(kind=kind, rows=r, cols=c, eps=round(n * n * math.exp(rng.uniform(math.log(1.5e-4), math.log(2e-3))), 4))
    if kind == "backward":
        r, c = _sides(rng, 64, 320)
        n = max(r, c)
        return dict(kind=kind, rows=r, cols=c, precision="fp32", eps=round(n * n * rng.uniform(1.5e-3, 4e-3), 4),
                    iters=rng.randint(15, 30), every=rng.randint(4, 10))
    if kind == "intensity":
        return dict(kind=kind, rows=2 ** rng.randint(6, 11), cols=2 ** rng.randint(6, 11))
    if kind == "cfot":
        r, c = _sides(rng, 64, 1024)
        n = max(r, c)
        return dict(kind=kind, rows=r, cols=c, eps=round(n * n * rng.uniform(0.06, 0.15), 2), iters=rng.randint(10, 50))
    r, c = _sides(rng, 48, 512)
    ro, co = _sides(rng, 48, 512)
    n = max(r, c, ro, co)
    return dict(kind="rect", rows=r, cols=c, rows_out=ro, cols_out=co,
                eps=round(n * n * math.exp(rng.uniform(math.log(2e-4), math.log(2e-3))), 4), iters=rng.randint(10, 30))


# ---- inputs --------------------------------------------------------------------------------

def _axes(rows, cols):
    j = torch.arange(rows, dtype=torch.float64, device="cuda")[:, None] - rows // 2
    k = torch.arange(cols, dtype=torch.float64, device="cuda")[None, :] - cols // 2
    return j, k


def _beam(rng, rows, cols):
    """The input amplitude: two overlapping Gaussians, seeded a few pixels off (amplitude float32)."""
    j, k = _axes(rows, cols)
    s = min(rows, cols) / 256.0
    d = [rng.uniform(-4.0, 4.0) * s for _ in range(4)]
    sa, sb = 40.0 * s, 25.0 * s
    g = (0.6 * torch.exp(-((j - 20.0 * s - d[0]) ** 2 + (k - d[1]) ** 2) / (2 * sa * sa))
         + 0.4 * torch.exp(-((j + 20.0 * s - d[2]) ** 2 + (k - d[3]) ** 2) / (2 * sb * sb)))
    return (g / torch.sqrt((g * g).sum())).float()


def _target(rng, rows, cols, shapes, pedestal):
    """The target amplitude: flat rectangles, disks and rings with a two-pixel cosine edge on a
    dark background (or on a faint pedestal inside a dark frame)."""
    j, k = _axes(rows, cols)
    s = min(rows, cols) / 256.0
    G = torch.zeros(rows, cols, dtype=torch.float64, device="cuda")
    for i in range(shapes):
        cj, ck = rng.uniform(-80.0, 80.0) * s, rng.uniform(-80.0, 80.0) * s
        if i % 3 == 0:
            hj, hk = rng.uniform(8.0, 30.0) * s, rng.uniform(8.0, 30.0) * s
            d = torch.maximum((j - cj).abs() - hj, (k - ck).abs() - hk)
        else:
            r = torch.sqrt((j - cj) ** 2 + (k - ck) ** 2)
            if i % 3 == 1:
                d = r - rng.uniform(15.0, 30.0) * s
            else:
                R, w = rng.uniform(20.0, 60.0) * s, max(1.0, rng.uniform(4.0, 8.0) * s)
                d = (r - R).abs() - w / 2
        edge = torch.where(d <= 0, 1.0, torch.where(d < 2, 0.5 * (1 + torch.cos(math.pi * d / 2)), 0.0))
        G = torch.maximum(G, edge)
    if pedestal:
        frame = max(1, int(round(7 * s)))
        inside = torch.zeros_like(G)
        inside[frame:-frame, frame:-frame] = 1.0
        G = torch.maximum(G, torch.full_like(G, 0.02)) * inside
    return (G / torch.sqrt((G * G).sum())).float()


def _pair(case, seed, shapes=9, pedestal=False):
    rng = random.Random("%s/%s" % (case["kind"], seed))
    rows, cols = case["rows"], case["cols"]
    return (_beam(rng, rows, cols),
            _target(rng, case.get("rows_out", rows), case.get("cols_out", cols), shapes, pedestal))


def _noise(seed, *shape):
    """Uniform in [0, 1), the same on every machine."""
    return torch.from_numpy(np.random.default_rng(seed).random(shape)).cuda()


def _schedule(case):
    e0, e1, T = case["eps0"], case["eps1"], case["iters"]
    if e0 == e1:
        return [e0]
    return [e0 * (e1 / e0) ** (t / (T - 1)) for t in range(T)]


def _batch_problems(case, seed):
    # sizes are the case's own (a program's problem set); contents come from the seed
    sizes = [BATCH_SIZES[(7 * i + 3 * case["count"]) % 5] for i in range(case["count"])]
    out = []
    for i, n in enumerate(sizes):
        rng = random.Random("batch/%s/%d" % (seed, i))
        out.append((_beam(rng, n, n), _target(rng, n, n, rng.randint(2, 6), False)))
    return sizes, out


def _warm_iterate(g, G, eps, rounds):
    """A partly converged iterate in 64 bits: what a caller holds in the middle of a run."""
    la, lb = _log_marginal(g), _log_marginal(G)
    psi = torch.full_like(lb, eps * math.log(1.0 / lb.numel()))
    S = f = None
    for t in range(rounds):
        e = eps * 8.0 ** (1.0 - t / (rounds - 1.0))         # annealed: few rounds suffice
        S = _log_apply(psi, e)
        f = e * (la - S)
        psi = e * (lb - _log_apply(f, e))
    return f, psi, S


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        g, G = _pair(case, seed)
        ctx = B.fot_create(case["rows"], case["cols"], PRECISION[case["precision"]])
        return dict(case=case, ctx=ctx, g=g, G=G, eps=np.array(_schedule(case)))
    if kind == "update":
        g, G = _pair(case, seed)
        ctx = B.fot_create(case["rows"], case["cols"], PRECISION[case["precision"]])
        B.fot_set_problem(ctx, g, G)
        _, psi, _ = _warm_iterate(g, G, case["eps"], 6)
        return dict(case=case, ctx=ctx, g=g, G=G, psi=psi.float().contiguous())
    if kind == "batch":
        sizes, probs = _batch_problems(case, seed)
        batch = B.fot_batch_create([(n, n) for n in sizes], PRECISION[case["precision"]])
        return dict(case=case, batch=batch, gs=[p[0] for p in probs], Gs=[p[1] for p in probs],
                    eps=np.tile(np.array(_schedule(case)), (len(sizes), 1)))
    if kind == "phase":
        psi, S = _phase_inputs(case, seed)
        return dict(case=case, ctx=B.fot_create(case["rows"], case["cols"]), psi=psi, S=S)
    if kind == "backward":
        g, G, wphi, wpsi = _backward_inputs(case, seed)
        return dict(case=case, g=g.requires_grad_(), G=G.requires_grad_(), wphi=wphi, wpsi=wpsi)
    if kind == "intensity":
        g, G, phi = _intensity_inputs(case, seed)
        ctx = B.fot_create(case["rows"], case["cols"])
        B.fot_set_problem(ctx, g, G)
        return dict(case=case, ctx=ctx, g=g, G=G, phi=phi)
    if kind == "cfot":
        g, G = _cfot_inputs(case, seed)
        return dict(case=case, ctx=B.fot_create(case["rows"], case["cols"]), g=g, G=G)
    g, G = _pair(case, seed, pedestal=True)
    return dict(case=case, g=g, G=G)


def _phase_inputs(case, seed):
    g, G = _pair(case, seed, pedestal=True)
    f, psi, S = _warm_iterate(g, G, case["eps"], 8)
    return psi.float().contiguous(), S.float().contiguous()


def _backward_inputs(case, seed):
    g, G = _pair(case, seed, pedestal=True)
    g = (g + 0.02 * g.max()).contiguous()                   # a beam on a faint floor
    w = _noise(seed, 2, case["rows"], case["cols"])
    return g, G, w[0].float().contiguous(), (w[1] * (G > 0)).float().contiguous()


def _intensity_inputs(case, seed):
    g, G = _pair(case, seed)
    j, k = _axes(case["rows"], case["cols"])
    rng = random.Random("phi/%s" % seed)
    # a quadratic phase that spreads the beam over about a third of the far field, a smooth
    # ripple and a little roughness, in cycles
    a, b = rng.uniform(0.1, 0.2) / case["rows"], rng.uniform(0.1, 0.2) / case["cols"]
    phi = (a * j * j + b * k * k + 0.3 * torch.cos(2 * math.pi * (2 * j / case["rows"] + 3 * k / case["cols"]))
           + 0.05 * _noise(seed, case["rows"], case["cols"]))
    return g, G, phi.float().contiguous()


def _cfot_inputs(case, seed):
    """Two beams over a flat floor on both planes: the regime the exponential domain holds in."""
    rows, cols = case["rows"], case["cols"]
    rng = random.Random("cfot/%s" % seed)
    g, G = _beam(rng, rows, cols), _beam(rng, rows, cols)
    return (g + 0.3 * g.max()).contiguous(), (G.flip(0, 1) + 0.3 * G.max()).contiguous()


# ---- one pass --------------------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        B.fot_solve(state["ctx"], state["g"], state["G"], state["eps"], case["iters"])
        return B.fot_potentials(state["ctx"])
    if kind == "update":
        f = B.fot_u_update(state["ctx"], state["psi"], case["eps"])
        return f, B.fot_v_update(state["ctx"], f, case["eps"])
    if kind == "batch":
        B.fot_batch_solve(state["batch"], state["gs"], state["Gs"], state["eps"], case["iters"])
        return [B.fot_potentials(B.fot_batch_context(state["batch"], q)) for q in range(case["count"])]
    if kind == "phase":
        return B.fot_moments(state["ctx"], state["psi"], state["S"], case["eps"])
    if kind == "backward":
        phi, f, psi = B.fot_phase_fn(state["g"], state["G"], [case["eps"]], case["iters"],
                                     precision=PRECISION[case["precision"]], checkpoint_every=case["every"])
        return torch.autograd.grad([phi, psi], [state["g"], state["G"]], [state["wphi"], state["wpsi"]])
    if kind == "intensity":
        loss, inten = B.fot_intensity_loss(state["ctx"], state["phi"], with_intensity=True)
        return loss, inten
    if kind == "cfot":
        B.fot_cfot_solve(state["ctx"], state["g"], state["G"], [case["eps"]], case["iters"])
        return B.fot_potentials(state["ctx"])
    return B.fot_solve_rect(state["g"], state["G"], [case["eps"]], case["iters"])


def work(case):
    """Bytes: each input image read once, each output image written once.  Flops: the separable
    contraction itself, one multiply-add per (row, output, input) term of every axis pass; for
    the FFT forms, 5 N log2 N per transform."""
    kind = case["kind"]

    def half(r, c):                                         # one half-step: a pass along each axis
        return 2.0 * r * c * (r + c)

    if kind == "batch":
        sizes = [BATCH_SIZES[(7 * i + 3 * case["count"]) % 5] for i in range(case["count"])]
        return {"bytes": sum(16.0 * n * n for n in sizes), "flops": sum(2 * case["iters"] * half(n, n) for n in sizes)}
    r, c = case["rows"], case["cols"]
    if kind == "rect":
        ro, co = case["rows_out"], case["cols_out"]
        it = 2.0 * (ro * co * c + c * ro * r) + 2.0 * (r * c * co + co * r * ro)
        return {"bytes": 8.0 * (r * c + ro * co), "flops": case["iters"] * it}
    if kind == "solve":
        return {"bytes": 16.0 * r * c, "flops": 2 * case["iters"] * half(r, c)}
    if kind == "update":
        return {"bytes": 20.0 * r * c, "flops": 2 * half(r, c)}
    if kind == "phase":
        return {"bytes": 20.0 * r * c, "flops": 2 * half(r, c)}      # two weighted sums per term
    if kind == "backward":
        # forward, its recomputation, and two kernel applications per half-step's adjoint
        return {"bytes": 24.0 * r * c, "flops": 8 * case["iters"] * half(r, c)}
    fft = 5.0 * r * c * math.log2(r * c)
    if kind == "intensity":
        return {"bytes": 16.0 * r * c, "flops": fft}
    # cfot: a convolution per half-step, each a forward and an inverse transform of the padded lines
    return {"bytes": 16.0 * r * c, "flops": case["iters"] * 2 * 2 * 5.0 * 2 * r * c * math.log2(4.0 * r * c)}


# ---- the same in 64 bits ------------------------------------------------------------------

FLOOR = -1e30                                               # stands for log 0


def _log_marginal(amp):
    a = amp.double()
    p = a * a / (a * a).sum()
    return torch.where(p > 0, torch.log(torch.where(p > 0, p, 1.0)), -math.inf)


def _axis_lse(x, n_out, shift, eps, weights=()):
    """x [rows][len] natural logs -> (log sum_m exp(x - (o - m + shift)^2 / (2 eps)) as
    [n_out][rows], and the mean of each weight [rows][len] under those terms)."""
    rows, n_in = x.shape
    m = torch.arange(n_in, dtype=torch.float64, device=x.device)
    x = torch.where(torch.isinf(x), FLOOR, x)
    out = torch.empty(n_out, rows, dtype=torch.float64, device=x.device)
    means = [torch.empty_like(out) for _ in weights]
    # a tile of outputs o = kc + t shares the offset of its centre; the rest of the kernel,
    # exp((t (m - shift - kc) - t^2 / 2) / eps), is a matrix that no row changes, while its
    # exponents stay far inside the range of 64 bits
    half = int(200.0 * eps / (n_in + n_out))
    if half >= 4:
        half = min(half, 32)
        for k0 in range(0, n_out, 2 * half):
            o = torch.arange(k0, min(n_out, k0 + 2 * half), dtype=torch.float64, device=x.device)
            kc = k0 + half
            E = x - (kc + shift - m) ** 2 / (2 * eps)
            top = E.max(dim=1, keepdim=True).values
            A = torch.exp(E - top)
            t = (o - kc)[None, :]
            mat = torch.exp((t * (m[:, None] - shift - kc) - t * t / 2) / eps)
            s = A @ mat
            out[k0:k0 + o.numel()] = (torch.log(s) + top).T
            for w, q in zip(weights, means):
                q[k0:k0 + o.numel()] = ((A * w) @ mat / s).T
    else:
        o = torch.arange(n_out, dtype=torch.float64, device=x.device)
        K = (o[:, None] + shift - m[None, :]) ** 2 / (2 * eps)
        step = max(1, int(3e7) // (n_out * n_in))
        for r0 in range(0, rows, step):
            E = x[r0:r0 + step, None, :] - K[None]
            top = E.max(dim=2, keepdim=True).values
            E = torch.exp(E - top)
            s = E.sum(dim=2)
            out[:, r0:r0 + step] = (torch.log(s) + top[..., 0]).T
            for w, q in zip(weights, means):
                q[:, r0:r0 + step] = ((E * w[r0:r0 + step, None, :]).sum(dim=2) / s).T
    return out, means


def _log_apply(pot, eps, rows_out=None, cols_out=None):
    """log of the separable Gaussian kernel applied to exp(pot / eps)."""
    r, c = pot.shape
    ro, co = rows_out or r, cols_out or c
    R, _ = _axis_lse(pot / eps, co, (c - co) / 2, eps)
    return _axis_lse(R, ro, (r - ro) / 2, eps)[0]


def _infinite(x):
    """Zero mass as the library writes it."""
    return torch.where(x < FLOOR / 1e6, -math.inf, x)


def _exact_solve(g, G, eps, iters):
    la, lb = _log_marginal(g), _log_marginal(G)
    psi = torch.full_like(lb, eps[0] * math.log(1.0 / lb.numel()))
    f = None
    for t in range(iters):
        e = eps[0] if len(eps) == 1 else eps[t]
        f = e * (la - _log_apply(psi, e, *la.shape))
        psi = e * (lb - _log_apply(f, e, *lb.shape))
    return f, psi


def _trapezoid(Dx, Dy, h):
    rows, cols = Dx.shape
    col = torch.cat([torch.zeros_like(Dx[:1, 0]), torch.cumsum(0.5 * h * (Dx[1:, cols // 2] + Dx[:-1, cols // 2]), 0)])
    col = col - col[rows // 2]
    row = torch.cat([torch.zeros_like(Dy[:, :1]), torch.cumsum(0.5 * h * (Dy[:, 1:] + Dy[:, :-1]), 1)], 1)
    return col[:, None] + row - row[:, cols // 2:cols // 2 + 1]


def _coordinates(rows, cols, h, device):
    X = (torch.arange(rows, dtype=torch.float64, device=device) - rows // 2) / (rows * h)
    Y = (torch.arange(cols, dtype=torch.float64, device=device) - cols // 2) / (cols * h)
    return X, Y


def _exact_phase(psi, S, eps):
    rows, cols = psi.shape
    h = 1.0 / math.sqrt(max(rows, cols))
    X, Y = _coordinates(rows, cols, h, psi.device)
    R, (my,) = _axis_lse(psi / eps, cols, 0.0, eps, [Y[None, :].expand(rows, cols)])
    T, (mx, mm) = _axis_lse(R, rows, 0.0, eps, [X[None, :].expand(cols, rows), my])
    w = torch.exp(T - S)
    Dx, Dy = mx * w, mm * w
    return _trapezoid(Dx, Dy, h), Dx, Dy


def _exact_backward(g, G, wphi, wpsi, eps, iters):
    rows, cols = g.shape
    h = 1.0 / math.sqrt(max(rows, cols))
    g, G = g.detach().double().requires_grad_(), G.detach().double().requires_grad_()

    def log_marginal(a):
        safe = torch.where(a > 0, a, 1.0)
        return torch.where(a > 0, 2 * torch.log(safe) - torch.log((a * a).sum()), FLOOR)

    def kernel(n):
        i = torch.arange(n, dtype=torch.float64, device=g.device)
        return (i[:, None] - i[None, :]) ** 2 / (2 * eps)

    Kr, Kc = kernel(rows), kernel(cols)

    def apply(pot):                                         # both passes, direct
        R = torch.logsumexp(pot[:, None, :] / eps - Kc[None], dim=2)            # [L][k]
        return torch.logsumexp(R.T[:, None, :] - Kr[None], dim=2).T              # [j][k]

    la, lb = log_marginal(g), log_marginal(G)
    psi = torch.full_like(g, eps * math.log(1.0 / g.numel()))
    S = f = None
    for _ in range(iters):
        S = checkpoint(apply, psi, use_reentrant=False)
        f = eps * (la - S)
        psi = eps * (lb - checkpoint(apply, f, use_reentrant=False))
    X, Y = _coordinates(rows, cols, h, g.device)

    def moments(psi, S):
        E = psi[:, None, :] / eps - Kc[None]
        R = torch.logsumexp(E, dim=2)
        my = (torch.softmax(E, dim=2) * Y).sum(dim=2)
        E = R.T[:, None, :] - Kr[None]
        T = torch.logsumexp(E, dim=2)
        P = torch.softmax(E, dim=2)
        mx, mm = (P * X).sum(dim=2), (P * my.T[:, None, :]).sum(dim=2)
        w = torch.exp(T.T - S)
        return mx.T * w, mm.T * w

    Dx, Dy = checkpoint(moments, psi, S, use_reentrant=False)
    phi = _trapezoid(Dx, Dy, h)
    psi = torch.where(G > 0, psi, 0.0)
    loss = (phi * wphi.double()).sum() + (psi * wpsi.double()).sum()
    return torch.autograd.grad(loss, [g, G])


def _exact_intensity(g, G, phi):
    field = torch.polar(g.double(), 2 * math.pi * phi.double())
    far = torch.fft.fft2(field).abs() ** 2
    far = far.roll((g.shape[0] // 2, g.shape[1] // 2), (0, 1))
    far = far / far.sum()
    b = G.double() ** 2
    return float((far - b / b.sum()).abs().sum()), far


def _exact_cfot(g, G, eps, iters):
    rows, cols = g.shape

    def kernel(n):
        i = torch.arange(n, dtype=torch.float64, device=g.device)
        return torch.exp(-(i[:, None] - i[None, :]) ** 2 / (2 * eps))

    Kr, Kc = kernel(rows), kernel(cols)
    a, b = (torch.exp(_log_marginal(x)) for x in (g, G))
    v = torch.full_like(a, 1.0 / a.numel())
    u = None
    for _ in range(iters):
        u = a / (Kr @ v @ Kc)
        v = b / (Kr @ u @ Kc)
    return eps * torch.log(u), eps * torch.log(v)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        g, G = _pair(case, seed)
        return tuple(_infinite(x) for x in _exact_solve(g, G, _schedule(case), case["iters"]))
    if kind == "update":
        g, G = _pair(case, seed)
        e = case["eps"]
        psi = _warm_iterate(g, G, e, 6)[1].float().double()
        f = e * (_log_marginal(g) - _log_apply(psi, e))
        return _infinite(f), _infinite(e * (_log_marginal(G) - _log_apply(f, e)))
    if kind == "batch":
        return [tuple(_infinite(x) for x in _exact_solve(g, G, _schedule(case), case["iters"]))
                for g, G in _batch_problems(case, seed)[1]]
    if kind == "phase":
        psi, S = _phase_inputs(case, seed)
        return _exact_phase(psi.double(), S.double(), case["eps"])
    if kind == "backward":
        return _exact_backward(*_backward_inputs(case, seed), case["eps"], case["iters"])
    if kind == "intensity":
        return _exact_intensity(*_intensity_inputs(case, seed))
    if kind == "cfot":
        return _exact_cfot(*_cfot_inputs(case, seed), case["eps"], case["iters"])
    g, G = _pair(case, seed, pedestal=True)
    return tuple(_infinite(x) for x in _exact_solve(g, G, [case["eps"]], case["iters"]))
