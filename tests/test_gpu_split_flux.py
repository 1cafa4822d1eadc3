"""FP64 WENO solves of at least 256 cells a side take the split fluxes (FP32 pairs for the
nonlinear part): parity with the oracle on both sides of that line, on every tile
shape, over the range of the WENO epsilon and of the fields' scale, and in a batch
that holds both kinds."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ap_dvm_oracle as O  # noqa: E402
from paper_2512_19847_gb300 import api, tableaux, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
TABS = {"gsa2": tableaux.gsa2, "euler": tableaux.euler, "type_a3": tableaux.type_a3, "ars4": tableaux.ars4}


def _setup(nx, ny, scheme, tab="gsa2", eps=1e-2, weno_eps=1e-6, amp=1.0, seed=3):
    A_ex, A_im = TABS[tab]()
    X0 = W.random_moment_state(nx, ny, seed, amp=amp)
    dt = 0.2 * (2 * math.pi / max(nx, ny)) / amp
    p = api.default_params(nx, ny, eps=eps, dt=dt, tau=0.05, space_scheme=scheme, tableau=(A_ex, A_im), weno_eps=weno_eps)
    o = O.Params(nx, ny, eps, 0.05, dt, np.array(A_ex), np.array(A_im), scheme=scheme, weno_eps=weno_eps)
    return X0, p, o


def _check(X0, p, o, tile=-1, steps=1):
    s = api.Solver(p)
    s.set_tile(tile)
    s.set_state(torch.from_numpy(X0).cuda())
    s.step(steps)
    s.sync_status()
    got, ref = s.get_state().cpu().numpy(), O.run(X0, o, steps)
    err = np.max(np.abs(got - ref), axis=(1, 2)) / np.maximum(np.max(np.abs(ref), axis=(1, 2)), 1e-300)
    assert np.all(err <= 1e-12), err   # the parity bound of every FP64 test


@pytest.mark.parametrize("scheme", ["WENO3_C4", "WENO5_C4"])
@pytest.mark.parametrize("nx,ny", [(256, 256), (255, 256), (256, 255), (257, 259), (300, 256), (258, 512)])
def test_sizes_about_the_line(nx, ny, scheme):
    _check(*_setup(nx, ny, scheme))


@pytest.mark.parametrize("scheme", ["WENO3_C4", "WENO5_C4"])
@pytest.mark.parametrize("tile", [0, 1, 2, 3, 4, 5])
def test_every_tile(tile, scheme):
    _check(*_setup(260, 262, scheme, tab="ars4"), tile=tile)


@pytest.mark.parametrize("tab", ["euler", "type_a3"])
def test_tableaux(tab):
    _check(*_setup(256, 256, "WENO5_C4", tab=tab, eps=1e-4))


@pytest.mark.parametrize("scheme", ["WENO3_C4", "WENO5_C4"])
@pytest.mark.parametrize("weno_eps,amp", [(1e-30, 1.0), (1e-12, 1e-6), (1e-6, 1e6), (1.0, 1e-3)])
def test_range_of_scales(weno_eps, amp, scheme):
    _check(*_setup(256, 256, scheme, weno_eps=weno_eps, amp=amp))


def test_zero_and_constant_planes():
    """q = 0, tau = 0 and constant velocities: increments and nonlinear terms that are exactly zero."""
    n = 256
    X0 = np.zeros((6, n, n))
    X0[0], X0[2], X0[3] = 1.0, 0.5, -0.5
    A_ex, A_im = tableaux.gsa2()
    p = api.default_params(n, n, eps=1e-3, dt=1e-3, tau=0.0, tableau=(A_ex, A_im))
    s = api.Solver(p)
    s.set_state(torch.from_numpy(X0).cuda())
    s.step(2)
    s.sync_status()
    got = s.get_state().cpu().numpy()
    assert np.max(np.abs(got - X0)) <= 1e-12


def test_non_finite_values_reach_the_status():
    X0, p, _ = _setup(256, 256, "WENO5_C4")
    X0[3, 7, 9] = np.nan
    s = api.Solver(p)
    s.set_state(torch.from_numpy(X0).cuda())
    s.step(1)
    with pytest.raises(api.ApDvmError) as e:
        s.sync_status()
    assert e.value.status == 5


@pytest.mark.parametrize("graph", [0, 2])
def test_batch_of_both_kinds_equals_alone(graph):
    sizes = [(64, 64), (256, 256), (96, 300), (300, 257)]
    A_ex, A_im = tableaux.gsa2()
    tmpl = api.default_params(300, 512, eps=1e-2, dt=1e-3, tau=0.05, tableau=(A_ex, A_im))
    b = api.Batch(tmpl, len(sizes))
    want = []
    for k, (nx, ny) in enumerate(sizes):
        X0, p, _ = _setup(nx, ny, "WENO5_C4", seed=k)
        b.attach(k, p)
        b.set_state(torch.from_numpy(X0).cuda(), slot=k)
        s = api.Solver(p)
        s.set_state(torch.from_numpy(X0).cuda())
        s.step(3)
        want.append(s.get_state())
    b.set_graph_steps(graph)
    assert b.launches_per_step > api.Solver(_setup(64, 64, "WENO5_C4")[1]).launches_per_step
    b.step(3)
    b.sync_status()
    for k in range(len(sizes)):
        assert torch.equal(b.get_state(k), want[k])
    b.step_slots(2, {0: 2, 1: 0, 2: 1, 3: 2})
    b.detach(1)
    b.detach(3)          # only one kind left
    b.step(1)
    b.sync_status()
