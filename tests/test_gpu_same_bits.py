"""The result of a solve, bit for bit, whichever kernels take it: every tile shape, and (FP32) the tile
kernels of a solve alone against the marching kernels of a large batch, for the precision forms, schemes
and tableaux that select different instantiations."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2512_19847_gb300 import api, tableaux  # noqa: E402

pytestmark = pytest.mark.gpu
TABS = {"gsa2": tableaux.gsa2, "euler": tableaux.euler, "type_a3": tableaux.type_a3, "ars4": tableaux.ars4}


def _params(nx, ny, scheme, tab, prec, eps):
    return api.default_params(nx, ny, eps=eps, dt=0.1 * 2 * math.pi / max(nx, ny), tau=0.05, mach=1e-2, space_scheme=scheme,
                              tableau=TABS[tab](), precision=prec)


def _state(nx, ny, seed=2):
    """Smooth on one half, noise on the other."""
    rng = np.random.default_rng(seed)
    x, y = 2 * math.pi * np.arange(nx)[None, :] / nx, 2 * math.pi * np.arange(ny)[:, None] / ny
    f = np.stack([np.sin(x + k) * np.cos(2 * y + 0.3 * k) for k in range(6)])
    return torch.from_numpy(f + np.where(x > math.pi, 0.2, 0.0) * rng.standard_normal(f.shape)).cuda()


def _alone(nx, ny, p, steps, tile=-1):
    s = api.Solver(p)
    s.set_tile(tile)
    s.set_state(_state(nx, ny))
    s.step(steps)
    s.sync_status()
    return s.get_state()


@pytest.mark.parametrize("prec", [api.FP64, api.FP32_DEV, api.FP32_DEV_TH])
@pytest.mark.parametrize("scheme", ["LF1_C2", "WENO3_C4", "WENO5_C4"])
@pytest.mark.parametrize("tab", ["gsa2", "type_a3"])
def test_every_tile(tab, scheme, prec):
    nx, ny = 75, 66
    p = _params(nx, ny, scheme, tab, prec, 1e-2)
    want = _alone(nx, ny, p, 3, tile=0)
    for tile in range(1, 6):
        assert torch.equal(_alone(nx, ny, p, 3, tile=tile), want), tile


@pytest.mark.parametrize("prec", [api.FP32_DEV, api.FP32_DEV_TH])
@pytest.mark.parametrize("scheme", ["LF1_C2", "WENO3_C4", "WENO5_C4"])
@pytest.mark.parametrize("tab,eps", [("gsa2", 1e-2), ("gsa2", 1e-5), ("euler", 1e-2), ("type_a3", 1e-2), ("ars4", 1e-5)])
def test_marching_in_a_batch_equals_tiles_alone(tab, eps, scheme, prec):
    sizes = [(256, 256), (128, 128), (100, 200), (300, 300), (360, 350)]   # none large enough to march alone, all together are
    b = api.Batch(_params(1024, 1024, scheme, tab, prec, eps), len(sizes))
    want = []
    for k, (nx, ny) in enumerate(sizes):
        p = _params(nx, ny, scheme, tab, prec, eps)
        b.attach(k, p)
        b.set_state(_state(nx, ny), slot=k)
        want.append(_alone(nx, ny, p, 2))
    b.step(2)
    b.sync_status()
    for k in range(len(sizes)):
        assert torch.equal(b.get_state(k), want[k]), sizes[k]
