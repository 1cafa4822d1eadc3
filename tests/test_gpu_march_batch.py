"""FP32 batches that hold solves of the tile kernels beside solves of the marching kernels, and whose set of
solves crosses, between graph launches, the number of cells from which all of them march: the launches
of a step follow the set, and every solve gets the bits it gets alone."""
import math

import pytest

torch = pytest.importorskip("torch")

from paper_2512_19847_gb300 import api, tableaux, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _params(nx, ny, prec):
    return api.default_params(nx, ny, eps=1e-3, dt=0.1 * 2 * math.pi / max(nx, ny), tau=0.05, mach=1e-2,
                              tableau=tableaux.gsa2(), precision=prec)


def _state(nx, ny, seed):
    return torch.from_numpy(W.random_moment_state(nx, ny, seed)).cuda()


@pytest.mark.parametrize("graph", [0, 2])
@pytest.mark.parametrize("prec", [api.FP32_DEV, api.FP32_DEV_TH])
def test_kinds_change_between_steps(prec, graph):
    # 400^2 marches by itself, 32x300 is too narrow ever to; the others march with it once the
    # second 400^2 brings the batch past 2 x 384^2 cells
    sizes = {0: (400, 400), 1: (64, 64), 2: (100, 96), 3: (32, 300), 4: (400, 400)}
    b = api.Batch(_params(1024, 1024, prec), 5)
    b.set_graph_steps(graph)
    done = {}

    def attach(k):
        b.attach(k, _params(*sizes[k], prec))
        b.set_state(_state(*sizes[k], k), slot=k)
        done[k] = 0

    def detach(k):
        b.detach(k)
        del done[k]

    def step(n, only=None):
        if only is None:
            b.step(n)
        else:
            b.step_slots(n, {k: only.get(k, n) for k in done})
        b.sync_status()
        for k in done:
            done[k] += n if only is None else only.get(k, n)
            s = api.Solver(_params(*sizes[k], prec))
            s.set_state(_state(*sizes[k], k))
            s.step(done[k])
            assert torch.equal(b.get_state(k), s.get_state()), (k, done)

    for k in (0, 1, 2):
        attach(k)
    mixed = b.launches_per_step   # one kind of stencil kernel less is 4 launches less: explicit and update of two stages
    step(3)
    attach(4)                     # all march
    assert b.launches_per_step == mixed - 4
    step(3)
    step(4, {1: 1, 4: 2})         # paused solves still count
    assert b.launches_per_step == mixed - 4
    attach(3)                     # too narrow: tiles again
    assert b.launches_per_step == mixed
    step(2)
    detach(4)                     # tiles for the small ones
    step(3)
    detach(0)                     # no marching solve left
    assert b.launches_per_step == mixed - 4
    step(2)
    attach(4)
    assert b.launches_per_step == mixed
    step(3)
