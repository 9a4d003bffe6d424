"""Matrices whose rows are not 8-aligned (cols % 8 != 0), on the GPU against
the oracle: widths at the edges of the kernels' tiles (32-element load
instructions, 8 per lane; 4, 2 and 1 rows per warp up to 64, 128 and more
columns; panels of 1024), odd row counts, and buffers that start at any
element address."""
import numpy as np
import pytest
import torch

from oracle import HParams
from paper_2609_30342_gb300 import build as pkg_build
from paper_2609_30342_gb300 import workloads

from gpu_helpers import DeviceRun, Tracked
from test_gpu_diagnostics import HP as SHADOW_HP, ShadowRef, _compare, _gpu_state

pytestmark = pytest.mark.gpu

WIDTHS = [1, 31, 33, 63, 65, 127, 129, 255, 257, 511, 1023, 1025, 2051]
SHAPES = [(r, w) for w, r in zip(WIDTHS, [70, 9, 33, 31, 1, 17, 66, 8, 23, 5, 16, 3, 2])] + [(40, 64), (13, 0)]


@pytest.fixture(scope="module", autouse=True)
def built():
    pkg_build.build()
    yield


def _off_by_one(run):
    """Move the ragged matrices' buffers one element on: 4-byte (fp32) and
    2-byte (bf16) aligned bases."""
    for lst in (run.x, run.p, run.g, run.out):
        for t, (m, n) in enumerate(run.shapes):
            if n % 8:
                flat = torch.empty(m * n + 1, dtype=lst[t].dtype, device="cuda")
                v = flat[1:].view(m, n)
                v.copy_(lst[t])
                lst[t] = v
    run.ptrs = run.opt.pack(run.x, run.g, run.p)


@pytest.mark.parametrize("shift", [False, True])
@pytest.mark.parametrize("grad_bf16", [True, False])
def test_ragged_steps_match_oracle(grad_bf16, shift):
    """Constant and changing step sizes (one and two exponentials per element),
    from the GPU's own state at every step: 1e-5, per-element rounding bound
    beyond it.  Summation depths: a lane's <= 8 columns a pass, 5 butterfly
    levels and 3 panels; a warp's rows, 8 warps x 4 groups and the slots; 64 covers
    both."""
    hp = HParams(alpha=0.3, mu=1e-3, gamma=0.05, eps_stab=1e-8)
    inp = workloads.ModelInputs(SHAPES, seed=61, g_std=1e-2, grad_bf16=grad_bf16)
    run = DeviceRun(SHAPES, hp, grad_bf16, inp.X, inp.P)
    if shift:
        _off_by_one(run)
    for k, h in enumerate((0.1, 0.1, 0.05)):
        seeded = Tracked.from_gpu(run)
        g = inp.grads(k)
        run.set_grads(g)
        run.step(h)
        seeded.step(g, h, hp, run.factors())
        seeded.check(run, 1e-5, "step%d" % (k + 1))
    # in place: the same bits as out of place
    want = run.canonical_P()
    run.opt.materialize(run.p)
    torch.cuda.synchronize()
    for p, w in zip(run.p, want):
        assert np.array_equal(p.double().cpu().numpy(), w)
    run.close()


@pytest.mark.parametrize("grad_bf16", [True, False])
def test_ragged_shadow_steps_match_oracle(grad_bf16):
    inp = workloads.ModelInputs(SHAPES, seed=62, g_std=1e-2, grad_bf16=grad_bf16)
    run = DeviceRun(SHAPES, SHADOW_HP, grad_bf16, inp.X, inp.P, method="ikfad_shadow")
    for k, h in enumerate((0.1, 0.05)):
        seeded = ShadowRef(SHAPES, *_gpu_state(run))
        g = inp.grads(k)
        run.set_grads(g)
        run.step(h)
        seeded.step(g, h)
        _compare(run, seeded, 1e-5, "reseeded step%d " % (k + 1))
    run.close()


@pytest.mark.parametrize("method", ["rikfad", "ikfad_shadow"])
@pytest.mark.parametrize("grad_bf16", [True, False])
def test_narrow_panels_match_oracle(method, grad_bf16):
    """8-wide panels of every number of rows per warp (8, 4, 2, 1 up to 32, 64,
    512 and more columns), with row counts that leave lane groups idle, and
    matrices whose last panel is narrow: from the GPU's own state at 1e-5."""
    widths = [8, 16, 24, 32, 40, 64, 72, 128, 200, 256, 384, 512, 520, 1096, 1376, 1600]
    shapes = [(r, w) for w, r in zip(widths, [129, 65, 63, 9, 33, 31, 17, 15, 7, 9, 13, 3, 5, 9, 7, 18])]
    inp = workloads.ModelInputs(shapes, seed=63, g_std=1e-2, grad_bf16=grad_bf16)
    run = DeviceRun(shapes, SHADOW_HP, grad_bf16, inp.X, inp.P, method=method)
    for k, h in enumerate((0.1, 0.1, 0.05)):
        g = inp.grads(k)
        if method == "rikfad":
            seeded = Tracked.from_gpu(run)
        else:
            seeded = ShadowRef(shapes, *_gpu_state(run))
        run.set_grads(g)
        run.step(h)
        if method == "rikfad":
            seeded.step(g, h, SHADOW_HP, run.factors())
            seeded.check(run, 1e-5, "step%d" % (k + 1))
        else:
            seeded.step(g, h)
            _compare(run, seeded, 1e-5, "step%d " % (k + 1))
    run.close()


@pytest.mark.parametrize("grad_bf16", [True, False])
def test_bands_match_oracle(grad_bf16):
    """Matrices whose last panels are walked together: partial chunks of 8, 24,
    40 and 136 columns, a band that is the whole row and one that is its end,
    beside panels of whole chunks; constant and changing step sizes, from the
    GPU's own state at every step (1e-5, per-element bound beyond)."""
    shapes = [(5000, 1800), (2500, 1048), (2000, 1928), (1500, 2600), (300, 768), (77, 40), (1000, 0)]
    from paper_2609_30342_gb300 import rikfad
    blocks = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    plan = rikfad.plan_query(shapes, "bf16" if grad_bf16 else "f32", blocks)
    same = (plan[1:, [0, 1, 5, 6]] == plan[:-1, [0, 1, 5, 6]]).all(axis=1) & (plan[1:, 2] == 0)
    assert set(plan[1:][same][:, 1]) == {0, 1, 2, 3}       # these matrices have bands
    hp = HParams(alpha=0.3, mu=1e-3, gamma=0.05, eps_stab=1e-8)
    inp = workloads.ModelInputs(shapes, seed=64, g_std=1e-2, grad_bf16=grad_bf16)
    run = DeviceRun(shapes, hp, grad_bf16, inp.X, inp.P)
    depths = {t: (64.0, 128.0) for t in range(len(shapes))}     # 30 rows a warp, 8 warps, up to 50 slots
    for k, h in enumerate((0.1, 0.1, 0.05)):
        seeded = Tracked.from_gpu(run, depths)
        g = inp.grads(k)
        run.set_grads(g)
        run.step(h)
        seeded.step(g, h, hp, run.factors())
        seeded.check(run, 1e-5, "step%d" % (k + 1))
    run.close()


FEW = [(5, 7), (1, 1), (9, 33), (3, 1025), (70, 1), (17, 129), (2, 2051)]


@pytest.mark.parametrize("method,base", [("rikfad", [(4000, 768), (33, 40), (1000, 0)]),
                                         ("rikfad", [(5000, 1800), (300, 768), (1000, 0)]),
                                         ("ikfad_shadow", [(4000, 768), (33, 40), (1000, 0)])])
@pytest.mark.parametrize("grad_bf16", [True, False])
def test_few_ragged_rows_match_oracle(method, base, grad_bf16):
    """Lists that are 8-wide but for one element in 256 at most, without and with
    bands: their ragged matrices (one panel and several, odd rows, buffers one
    element on) and the others, from the GPU's own state at every step."""
    shapes = base[:1] + FEW + base[1:]
    ragged = sum(m * n for m, n in FEW)
    assert ragged * 256 <= sum(workloads.numel(s) for s in shapes)
    hp = SHADOW_HP if method == "ikfad_shadow" else HParams(alpha=0.3, mu=1e-3, gamma=0.05, eps_stab=1e-8)
    inp = workloads.ModelInputs(shapes, seed=65, g_std=1e-2, grad_bf16=grad_bf16)
    run = DeviceRun(shapes, hp, grad_bf16, inp.X, inp.P, method=method)
    _off_by_one(run)
    depths = {t: (64.0, 128.0) for t in range(len(shapes))}
    for k, h in enumerate((0.1, 0.1, 0.05)):
        g = inp.grads(k)
        seeded = Tracked.from_gpu(run, depths) if method == "rikfad" else ShadowRef(shapes, *_gpu_state(run))
        run.set_grads(g)
        run.step(h)
        if method == "rikfad":
            seeded.step(g, h, hp, run.factors())
            seeded.check(run, 1e-5, "step%d" % (k + 1))
        else:
            seeded.step(g, h)
            _compare(run, seeded, 1e-5, "step%d " % (k + 1))
    run.close()
