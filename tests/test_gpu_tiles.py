"""The passes over tiles (canonical momentum; the step of lists without
matrices), on the GPU against the oracle, at the edges of their tiles."""
import numpy as np
import pytest
import torch

from oracle import HParams
from paper_2609_30342_gb300 import build as pkg_build
from paper_2609_30342_gb300 import workloads

from gpu_helpers import DeviceRun, Tracked

pytestmark = pytest.mark.gpu

HP = HParams(alpha=0.3, mu=1e-3, gamma=0.05, eps_stab=1e-8)


@pytest.fixture(scope="module", autouse=True)
def built():
    pkg_build.build()
    yield


def test_canonical_momentum_at_tile_edges():
    """8-wide widths on both sides of the flat path (128 columns), of the tile
    heights (512) and of a panel (1024), with row counts around a tile: the
    canonical momentum after two steps against the oracle from the GPU's state
    before the last (1e-5, per-element bound beyond), and in place bit for bit
    as out of place."""
    shapes = [(1, 8), (1023, 8), (1025, 8), (129, 64), (127, 64), (31, 120), (65, 128), (64, 136), (33, 384),
              (15, 512), (32, 520), (17, 768), (1, 1024), (16, 1032), (33, 1600), (7, 3072), (0, 16), (5, 0)]
    inp = workloads.ModelInputs(shapes, seed=71, g_std=1e-2)
    run = DeviceRun(shapes, HP, True, inp.X, inp.P)
    for k, h in enumerate((0.1, 0.05)):
        seeded = Tracked.from_gpu(run)
        g = inp.grads(k)
        run.set_grads(g)
        run.step(h)
        seeded.step(g, h, HP, run.factors())
        seeded.check(run, 1e-5, "step%d" % (k + 1))
    want = run.canonical_P()
    run.opt.materialize(run.p)
    torch.cuda.synchronize()
    for p, w in zip(run.p, want):
        assert np.array_equal(p.double().cpu().numpy(), w)
    run.close()


@pytest.mark.parametrize("grad_bf16", [True, False])
def test_element_lists_at_tile_edges(grad_bf16):
    """Lists of vectors alone, with sizes around a tile of 2048 elements and
    its 8-element loads, and an empty matrix whose C only decays."""
    shapes = [(n, 0) for n in (1, 7, 8, 9, 2047, 2048, 2049, 4095, 4097, 6144, 0, 10000)] + [(0, 24)]
    inp = workloads.ModelInputs(shapes, seed=72, g_std=1e-2, grad_bf16=grad_bf16)
    run = DeviceRun(shapes, HP, grad_bf16, inp.X, inp.P)
    C0 = np.linspace(0.1, 1.0, 24).astype(np.float32)
    run.opt.set_factors(len(shapes) - 1, np.zeros(0, np.float32), C0)
    for k, h in enumerate((0.1, 0.1, 0.05)):
        seeded = Tracked.from_gpu(run)
        g = inp.grads(k)
        run.set_grads(g)
        run.step(h)
        seeded.step(g, h, HP, run.factors())
        seeded.check(run, 1e-5, "step%d" % (k + 1))
    run.close()


RAGGED_SHAPES = [(8193, 1), (8192, 1), (3, 1), (1639, 5), (1638, 5), (64, 129), (63, 129), (32, 255), (33, 257),
                 (16, 513), (15, 1001), (16, 1025), (7, 2047), (40, 3001), (1, 1027), (4096, 1), (4097, 1), (819, 5), (820, 5), (10007, 1003)]


@pytest.mark.parametrize("method", ["rikfad", "ikfad_shadow"])
def test_ragged_canonical_momentum_at_tile_edges(method):
    """Ragged widths on both sides of a block's 256 threads and of a panel, with
    row counts around a tile of 4096 elements (8192 for the
    last, of 10 M).  Rank-1 friction: against the
    oracle, and in place bit for bit as out of place; element-wise friction (with
    8-wide matrices beside): a copy of the stored momentum, bit for bit."""
    shapes = RAGGED_SHAPES + ([(1023, 8), (65, 1032)] if method == "ikfad_shadow" else [])
    inp = workloads.ModelInputs(shapes, seed=73, g_std=1e-2)
    run = DeviceRun(shapes, HP, True, inp.X, inp.P, method=method)
    for k, h in enumerate((0.1, 0.05)):
        seeded = Tracked.from_gpu(run) if method == "rikfad" else None
        g = inp.grads(k)
        run.set_grads(g)
        run.step(h)
        if seeded:
            seeded.step(g, h, HP, run.factors())
            seeded.check(run, 1e-5, "step%d" % (k + 1))
    out = [torch.full_like(p, float("nan")) for p in run.p]
    run.opt.canonical_momentum(run.p, out)
    if method == "rikfad":
        run.opt.materialize(run.p)
    torch.cuda.synchronize()
    for p, o in zip(run.p, out):
        assert torch.equal(p, o)
    run.close()
