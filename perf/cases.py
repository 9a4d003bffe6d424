"""Performance cases of the library: the calls that a training program makes, over the sizes it makes them at.

``listed()`` are the cases that are timed, ``draw(rng)`` gives more of the same ranges, ``prepare(case, seed)``
makes what a program has in hand before the call, ``run(state)`` is one pass through the public entry points,
``work(case)`` what that pass cannot do without, ``tolerance(case)`` how far another correct implementation
may be off, and ``exact(case, seed)`` the same results in 64 bits, in plain torch.

The calls ("call" of a case):

  step        one ``RIKFAD.step`` over a parameter list (R-iKFAD, full-friction iKFAD, or iKFAD with shadow
              factors), optionally with the read-back of the friction denominators that a training loop logs
  optim       one ``RIKFADOptimizer.step`` (the torch.optim front end) with a learning-rate schedule
  checkpoint  ``RIKFAD.canonical_momentum`` and ``RIKFAD.export_state``: what is written to a checkpoint
  diagnose    ``RIKFAD.friction_diagnostics`` of every matrix of a list (shadow handle)
  noalloc     one ``step_matrix_noalloc``
  quadratic   one ``quadratic_run``: batched BACD integration of small dense quadratics

Parameter lists: "matrix" is one rows x cols matrix and a vector of ``cols`` elements (a layer and its bias),
"gpt2" the GPT-2-shaped list of the package's workloads (layers, width, vocab, ctx), "block" the six matrices of
one of its transformer blocks.  A list's tensors are views into one flat buffer each for parameters, gradients
and momenta, so a pass returns whole buffers.  Every optimiser has taken one step before the timed pass (factors
and a pending half-damp are in place, as in the middle of training).
"""
import math

import torch

from paper_2609_30342_gb300 import rikfad, workloads
from paper_2609_30342_gb300.optim import RIKFADOptimizer

# The paper's GPT2-S hyperparameters (R-iKFAD0).
H, ALPHA, MU, EPS = 0.0918, 0.0579, 1.3637e-6, 1e-16
X_STD, G_STD = 0.02, 1e-3
# The batched quadratics' (numerical set-up of the rate validation).
QH, QALPHA, QMU = 0.02, 1.0, 1.0

DEVICE = "cuda"
ALIGN = 64          # elements: every tensor of a flat buffer starts on 256 bytes (128 for bf16)


# ------------------------------------------------------------------ cases

def _step(name, **kw):
    case = dict(name=name, call="step", method="rikfad", grad="bf16", gamma=0.0, vary_h=False, denominators=False)
    case.update(kw)
    return case


def listed():
    return [
        # The smallest step: one layer of a small model, fp32 gradients; latency and launches.
        _step("step-256x512-f32", params="matrix", rows=256, cols=512, grad="f32"),
        # A small model's whole parameter list in mixed precision (100 tensors, 30M parameters).
        _step("step-nano", params="gpt2", layers=6, width=384, vocab=50304, ctx=256),
        # The benchmark's list (196 tensors, 124M parameters), in a training loop that logs 1^T R of every matrix.
        _step("step-gpt2s", params="gpt2", layers=12, width=768, vocab=50257, ctx=1024, denominators=True),
        # The largest: 1557.6M parameters, 15.6 GB touched per step, rows of 1600.
        _step("step-gpt2xl", params="gpt2", layers=48, width=1600, vocab=50257, ctx=1024),
        # A ragged matrix: rows start at any 4-byte address (a layer whose width is not a multiple of 8).
        _step("step-ragged-f32", params="matrix", rows=10007, cols=3001, grad="f32"),
        # Full-friction iKFAD, the method that R-iKFAD is compared with, on the benchmark's list.
        _step("step-ikfad-gpt2s", params="gpt2", layers=12, width=768, vocab=50257, ctx=1024, method="ikfad"),
        # The torch.optim front end with autograd's fp32 gradients, linear damping and a changing learning rate.
        dict(name="optim-nano", call="optim", params="gpt2", layers=6, width=384, vocab=50304, ctx=256, grad="f32",
             gamma=0.1, vary_h=True),
        # A checkpoint of the benchmark's list: the paper's momentum out of place, and the state image.
        dict(name="checkpoint-gpt2s", call="checkpoint", params="gpt2", layers=12, width=768, vocab=50257, ctx=1024,
             grad="bf16", gamma=0.0, vary_h=False),
        # The rank-1 friction's distance from the best one, for the layers of one transformer block (six calls).
        dict(name="diagnose-block", call="diagnose", params="block", width=768, grad="bf16", gamma=0.0, vary_h=False),
        # The allocation-free step of one matrix, called between a service's other work.
        dict(name="noalloc-16384x768", call="noalloc", rows=16384, cols=768, grad="bf16", gamma=0.0, vary_h=False),
        # Many small quadratics at once: throughput.
        dict(name="quadratic-65536x6x5", call="quadratic", batch=65536, m=6, n=5, steps=1000, eps=0.1, gamma=0.0),
        # One row of the decay-slope table (16 instances): latency of the sequential steps, with energies recorded.
        dict(name="quadratic-16x4x3", call="quadratic", batch=16, m=4, n=3, steps=8192, eps=0.0, gamma=0.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi):
    """A column count: half of them multiples of 64, the others any number."""
    n = _log_int(rng, lo, hi)
    return max(64, n // 64 * 64) if rng.random() < 0.5 else n


def _draw_params(rng, most):
    """One matrix with its bias, or a GPT-2-shaped list, of at most ``most`` elements."""
    if rng.random() < 0.6:
        cols = _width(rng, 24, 16384)
        rows = _log_int(rng, 16, max(17, min(65536, most // cols)))
        return dict(params="matrix", rows=rows, cols=cols)
    while True:
        p = dict(params="gpt2", layers=rng.randint(1, 24), width=32 * rng.randint(2, 48),
                 vocab=_log_int(rng, 500, 51000), ctx=rng.choice((128, 256, 512, 1024)))
        if sum(workloads.numel(s) for s in _shapes(p)) <= most:
            return p


def draw(rng):
    call = rng.choice(("step", "step", "step", "step", "optim", "checkpoint", "diagnose", "noalloc", "quadratic",
                       "quadratic"))
    common = dict(grad=rng.choice(("bf16", "f32")), gamma=rng.choice((0.0, 0.0, 0.1)), vary_h=rng.random() < 0.3)
    if call == "step":
        return dict(call=call, **_draw_params(rng, 400_000_000), method=rng.choice(("rikfad",) * 4 + ("ikfad", "ikfad_shadow")),
                    denominators=rng.random() < 0.3, **common)
    if call == "optim":
        common["grad"] = "f32"
        return dict(call=call, **_draw_params(rng, 100_000_000), **common)
    if call == "checkpoint":
        return dict(call=call, **_draw_params(rng, 400_000_000), **common)
    if call == "diagnose":
        cols = _width(rng, 64, 4096)
        return dict(call=call, params="matrix", rows=_log_int(rng, 64, 16384), cols=cols, **common)
    if call == "noalloc":
        return dict(call=call, rows=_log_int(rng, 8, 65536), cols=min(1024, _width(rng, 8, 1024)), **common)
    while True:
        m, n = rng.randint(1, 8), rng.randint(1, 8)
        if m * n <= 32:
            break
    batch = _log_int(rng, 1, 65536)
    steps = _log_int(rng, 64, min(8192, max(65, (1 << 25) // batch)))
    return dict(call=call, batch=batch, m=m, n=n, steps=steps, eps=rng.choice((0.0, 0.1)),
                gamma=rng.choice((0.0, 0.0, 0.05)))


# ----------------------------------------------------------------- inputs

def _shapes(case):
    if case["params"] == "matrix":
        return [(case["rows"], case["cols"]), (case["cols"], 0)]
    if case["params"] == "block":
        d = case["width"]
        return [(d, d)] * 4 + [(4 * d, d), (d, 4 * d)]
    return [s for _, s in workloads.gpt2_shapes(case["layers"], case["width"], case["vocab"], case["ctx"])]


def _offsets(shapes):
    offs, at = [], 0
    for s in shapes:
        offs.append(at)
        at += -(-workloads.numel(s) // ALIGN) * ALIGN
    return offs, at


def _views(flat, shapes):
    offs, _ = _offsets(shapes)
    return [flat[o:o + workloads.numel(s)].view(workloads.array_shape(s)) for o, s in zip(offs, shapes)]


def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


class _Inputs:
    """The seeded parameters (N(0, 0.02^2)) and gradients (N(0, 1e-3^2), one draw per step) of a list; the gaps
    between its tensors are zero."""

    def __init__(self, shapes, grad, seed):
        self.shapes, self.gen = shapes, _generator(seed)
        self.dtype = torch.bfloat16 if grad == "bf16" else torch.float32
        self.size = _offsets(shapes)[1]

    def _normal(self, std):
        flat = torch.randn(self.size, generator=self.gen, device=DEVICE).mul_(std)
        for (o, s), nxt in zip(zip(_offsets(self.shapes)[0], self.shapes), _offsets(self.shapes)[0][1:] + [self.size]):
            end = o + workloads.numel(s)
            if end < nxt:
                flat[end:nxt] = 0
        return flat

    def x(self):
        return self._normal(X_STD)

    def grad(self):
        return self._normal(G_STD).to(self.dtype)


def _h(case, k):
    """The step size of step k: constant, or alternating (a schedule that changes it at every step)."""
    return H * 0.9 if case["vary_h"] and k % 2 else H


def _warm_steps(case):
    return 3 if case["call"] == "diagnose" else 1


def _quadratic_inputs(case, seed):
    """The paper's instances: A = B B^T / d + 0.8 I, X ~ N(0, 0.4^2), P ~ N(0, 0.3^2) (float64), and the steps whose
    energies are recorded: the first and last, and a few per decade between them."""
    gen = _generator(seed)
    b, m, n = case["batch"], case["m"], case["n"]
    d = m * n
    B = torch.randn(b, d, d, generator=gen, device=DEVICE, dtype=torch.float64)
    A = torch.bmm(B, B.transpose(1, 2)) / d + 0.8 * torch.eye(d, device=DEVICE, dtype=torch.float64)
    A = 0.5 * (A + A.transpose(1, 2))
    X = 0.4 * torch.randn(b, m, n, generator=gen, device=DEVICE, dtype=torch.float64)
    P = 0.3 * torch.randn(b, m, n, generator=gen, device=DEVICE, dtype=torch.float64)
    rec = {0, case["steps"]}
    t = 1.0
    while t < case["steps"]:
        rec.add(int(t))
        t *= 1.8
    return A.float(), X.float(), P.float(), sorted(rec)


# ------------------------------------------------------------ prepare, run

class _Case:
    """What a program keeps between passes."""


def prepare(case, seed):
    s = _Case()
    s.case, s.call = case, case["call"]
    if s.call == "quadratic":
        s.A, s.X, s.P, rec = _quadratic_inputs(case, seed)
        b, m, n = s.X.shape
        s.R, s.C = torch.zeros(b, m, device=DEVICE), torch.zeros(b, n, device=DEVICE)
        s.rec = torch.tensor(rec, dtype=torch.int64, device=DEVICE)
        s.E = torch.zeros(len(rec), b, device=DEVICE)
        return s
    shapes = [(case["rows"], case["cols"])] if s.call == "noalloc" else _shapes(case)
    inp = _Inputs(shapes, case["grad"], seed)
    s.x, s.p = inp.x(), torch.zeros(inp.size, device=DEVICE)
    s.g = torch.zeros(inp.size, dtype=inp.dtype, device=DEVICE)
    s.xs, s.ps, s.gs = _views(s.x, shapes), _views(s.p, shapes), _views(s.g, shapes)
    s.k = 0
    if s.call == "noalloc":
        s.R, s.C = torch.zeros(case["rows"], device=DEVICE), torch.zeros(case["cols"], device=DEVICE)
        s.pending = 0.0
        step = _noalloc_step
    elif s.call == "optim":
        params = [torch.nn.Parameter(v) for v in s.xs]
        s.opt = RIKFADOptimizer(params, lr=H, alpha=ALPHA, mu=MU, gamma=case["gamma"], eps_stab=EPS)
        for v, g, p in zip(params, s.gs, s.ps):
            v.grad = g
            s.opt.state[v]["momentum"] = p
        step = _optim_step
    else:
        method = "ikfad_shadow" if s.call == "diagnose" else case.get("method", "rikfad")
        s.opt = rikfad.RIKFAD(shapes, ALPHA, MU, case["gamma"], EPS, case["grad"], method=method)
        s.ptrs = s.opt.pack(s.xs, s.gs, s.ps)
        if case.get("denominators"):
            s.den = torch.zeros(len(shapes), pin_memory=True)
        step = _list_step
    for _ in range(_warm_steps(case)):
        s.g.copy_(inp.grad())
        step(s)
    s.g.copy_(inp.grad())
    if s.call == "checkpoint":
        s.out = torch.zeros_like(s.p)
        s.outs = _views(s.out, shapes)
        s.image = torch.zeros(s.opt.state_image_bytes(), dtype=torch.uint8, device=DEVICE)
    elif s.call == "diagnose":
        s.matrices = [t for t, (_, n) in enumerate(shapes) if n]
    return s


def _list_step(s):
    s.opt.step(_h(s.case, s.k), ptrs=s.ptrs)
    s.k += 1


def _optim_step(s):
    s.opt.param_groups[0]["lr"] = _h(s.case, s.k)
    s.opt.step()
    s.k += 1


def _noalloc_step(s):
    h = _h(s.case, s.k)
    rikfad.step_matrix_noalloc(s.case["rows"], s.case["cols"], h, s.pending, ALPHA, MU, s.case["gamma"], EPS,
                               s.case["grad"], s.xs[0], s.gs[0], s.ps[0], s.R, s.C)
    s.pending = h
    s.k += 1


def run(s):
    if s.call == "step":
        _list_step(s)
        if s.case["denominators"]:
            s.opt.enqueue_denominators(s.den)
            return {"x": s.x, "p": s.p, "den": s.den}
        return {"x": s.x, "p": s.p}
    if s.call == "optim":
        _optim_step(s)
        return {"x": s.x, "p": s.p}
    if s.call == "noalloc":
        _noalloc_step(s)
        return {"x": s.x, "p": s.p, "R": s.R, "C": s.C}
    if s.call == "checkpoint":
        s.opt.canonical_momentum(s.ps, s.outs)
        s.opt.export_state(s.image)
        return {"momentum": s.out, "factors": s.image[64:].view(torch.float32)}     # after the image's header
    if s.call == "diagnose":
        # rel_err, Eckart-Young floor, stable rank, sigma_1, ||xi||; the iteration count is not a result
        return [list(s.opt.friction_diagnostics(t)[:5]) for t in s.matrices]
    rikfad.quadratic_run(s.A, s.X, s.P, s.R, s.C, QH, QALPHA, QMU, s.case["gamma"], s.case["eps"], s.case["steps"],
                         s.rec, s.E)
    return {"X": s.X, "P": s.P, "R": s.R, "C": s.C, "E": s.E}


# ------------------------------------------------------- work and tolerance

def work(case):
    """Bytes: every input read once, every output written once (parameters, gradients, momenta, factors or
    frictions).  Operations: the method's, an exponential counted as one."""
    if case["call"] == "quadratic":
        b, m, n, steps = case["batch"], case["m"], case["n"], case["steps"]
        d = m * n
        return {"bytes": 4 * b * (d * d + 2 * (2 * d + m + n)), "flops": b * steps * (2 * d * d + 13 * d + 5 * m + 3 * n)}
    gb = 2 if case["grad"] == "bf16" else 4
    shapes = [(case["rows"], case["cols"])] if case["call"] == "noalloc" else _shapes(case)
    nbytes = flops = 0
    for m, n in shapes:
        e = workloads.numel((m, n))
        if case["call"] == "checkpoint":
            nbytes += 8 * e + (8 * (m + n) if n else 8 * m)
            flops += 3 * e if n else 0
        elif case["call"] == "diagnose":
            if n:           # the friction read once; the norms and one power iteration
                nbytes += 4 * (e + m + n)
                flops += 9 * e
        elif n == 0 or case.get("method") in ("ikfad", "ikfad_shadow"):
            nbytes += (24 + gb) * e + (8 * (m + n) if n and case["method"] == "ikfad_shadow" else 0)
            flops += 14 * e
        else:
            nbytes += (16 + gb) * e + 8 * (m + n)
            flops += 12 * e
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the measured distance of a pass from exact().  One step's parameters, momenta, factors and
    denominators are 3.6e-8 to 9.8e-8 off (2-norm), the diagnostic's five numbers about 1e-7 to 2e-7 (float32 sums over
    a row or a matrix), checkpoints 6.3e-8.  The quadratics' rounding adds up over the steps: 1e-6 after 1000 of
    them, 5.7e-6 after 8192."""
    if case["call"] == "quadratic":
        return {"rel": 4e-6 + 2.5e-9 * case["steps"]}
    return {"rel": 1e-6 if case["call"] == "diagnose" else 5e-7}


# ------------------------------------------------------------------ exact

def _exact_tensor(x, grads, hs, gamma, matrix, shadow):
    """BACD steps of one tensor in float64 from P = 0 and zero factors (R, C of a rank-1 friction; with
    ``matrix`` false an element-wise friction, with ``shadow`` R, C beside it).  Returns x, the half-damped P^(1)
    and P_{n+1} of the last step, the friction, R, C."""
    x = x.double()
    p = torch.zeros_like(x)
    xi = torch.zeros_like(x)
    R = x.new_zeros(x.shape[0]) if x.dim() == 2 else None
    C = x.new_zeros(x.shape[1]) if x.dim() == 2 else None

    def friction():
        if not matrix:
            return xi
        den = R.sum() + EPS
        return torch.outer(R / den if den else R, C)

    p1 = p
    for g, h in zip(grads, hs):
        decay, gain = math.exp(-ALPHA * h), -math.expm1(-ALPHA * h) / (MU * ALPHA)
        p = p - h * g.double()
        x = x + h * p
        p1 = p * torch.exp(-0.5 * h * friction())
        q = p1 * p1
        if matrix or shadow:
            R = decay * R + gain * q.sum(1)
            C = decay * C + gain * q.sum(0)
        if not matrix:
            xi = decay * xi + gain * q
        p = p1 * torch.exp(-0.5 * h * friction()) * math.exp(-gamma * h)
    return x, p1, p, xi, R, C


def _exact_list(case, seed):
    call = case["call"]
    shapes = [(case["rows"], case["cols"])] if call == "noalloc" else _shapes(case)
    inp = _Inputs(shapes, case["grad"], seed)
    x0 = inp.x()
    steps = _warm_steps(case) + (0 if call in ("checkpoint", "diagnose") else 1)
    gs = [inp.grad() for _ in range(steps)]
    hs = [_h(case, k) for k in range(steps)]
    full = call == "diagnose" or case.get("method") in ("ikfad", "ikfad_shadow")
    shadow = call == "diagnose" or case.get("method") == "ikfad_shadow"
    if call == "diagnose":
        out = []
        for v, *g in zip(*(_views(t, shapes) for t in [x0] + gs)):
            if v.dim() == 2:
                _, _, _, xi, R, C = _exact_tensor(v, g, hs, case["gamma"], False, True)
                f2 = (xi * xi).sum()
                e2 = ((xi - torch.outer(R / (R.sum() + EPS), C)) ** 2).sum()
                gram = xi.t() @ xi if xi.shape[0] >= xi.shape[1] else xi @ xi.t()
                s2 = torch.linalg.eigvalsh(gram)[-1]
                out.append([float(v) for v in ((e2 / f2).sqrt(), (1 - s2 / f2).clamp(min=0).sqrt(), f2 / s2, s2.sqrt(),
                                               f2.sqrt())])
        return [[torch.tensor(v, dtype=torch.float64) for v in row] for row in out]
    x, p = (torch.zeros(inp.size, dtype=torch.float64, device=DEVICE) for _ in range(2))
    den = []
    for v, xv, pv, *g in zip(*(_views(t, shapes) for t in [x0, x, p] + gs)):
        matrix = v.dim() == 2 and not full
        xe, p1, pe, _, R, C = _exact_tensor(v, g, hs, case["gamma"], matrix, shadow and v.dim() == 2)
        xv.copy_(xe)
        # between steps a rank-1 matrix's momentum buffer holds the half-damped P^(1)
        pv.copy_(p1 if matrix and call != "checkpoint" else pe)
        den.append(float(R.sum()) if v.dim() == 2 and (matrix or shadow) else 0.0)
    if call == "checkpoint":
        return {"momentum": p, "factors": None}         # the image's layout is the library's own
    if call == "noalloc":
        return {"x": x, "p": p, "R": R, "C": C}
    if case.get("denominators"):
        return {"x": x, "p": p, "den": torch.tensor(den, dtype=torch.float64)}
    return {"x": x, "p": p}


def _exact_quadratic(case, seed):
    A, X, P, rec = _quadratic_inputs(case, seed)
    b, m, n = X.shape
    A, x, p = A.double(), X.double().reshape(b, m * n, 1), P.double().reshape(b, m * n, 1)
    R, C = x.new_zeros(b, m), x.new_zeros(b, n)
    gamma, eps, h = case["gamma"], case["eps"], QH
    decay, gain, damp = math.exp(-QALPHA * h), -math.expm1(-QALPHA * h) / (QMU * QALPHA), math.exp(-gamma * h)

    def half():
        den = R.sum(1) + eps
        inv = torch.where(den == 0, torch.zeros_like(den), 1 / den)
        return torch.exp((R * inv[:, None])[:, :, None] * C[:, None, :] * (-0.5 * h)).reshape(b, m * n, 1)

    E, at, want = [], 0, set(rec)
    for k in range(case["steps"] + 1):
        g = torch.bmm(A, x)
        if k in want:
            E.append((0.5 * (x * g).sum(1) + 0.5 * (p * p).sum(1))[:, 0])
        if k == case["steps"]:
            break
        e = half() if k == 0 else e
        p = p - h * g
        x = x + h * p
        p = p * e
        q = (p * p).reshape(b, m, n)
        R, C = decay * R + gain * q.sum(2), decay * C + gain * q.sum(1)
        e = half()
        p = p * e * damp
    return {"X": x.reshape(b, m, n), "P": p.reshape(b, m, n), "R": R, "C": C, "E": torch.stack(E)}


def exact(case, seed):
    with torch.no_grad():
        return _exact_quadratic(case, seed) if case["call"] == "quadratic" else _exact_list(case, seed)
