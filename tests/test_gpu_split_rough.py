"""FP64 WENO solves with split fluxes on data that is rough at the mesh scale, or of a size beyond what
pairs of floats hold: there the whole FP64 form must come out, cell by cell.

A state that repeats itself, on a grid of 256 x 256 (split), is compared with one period of it on a
grid of 128 x 128 (below the line, whole), at eps = 1 and tau = 50, where v and q keep their values over a step and the
pressure follows them loosely.  The two solves differ in the transforms' lengths only: rounding of at most 2 log2(256^2)
2^-53 = 4e-15 of the pressure, which enters the velocity times (4/3) dt/h = 0.27, so 1e-15, and the roundings
of the sums it joins, at most 16 of 2^-53: 3e-15 together, of each plane's largest value.  Pairs of floats
are off by 1e-14 and more of it on white noise.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2512_19847_gb300 import api, tableaux  # noqa: E402

pytestmark = pytest.mark.gpu
N = 128


def _state(kind, amp=(1.0, 1.0), seed=5):
    rng = np.random.default_rng(seed)
    t = 2 * math.pi * np.arange(N) / N
    x, y = t[None, :], t[:, None]
    f = np.stack([np.sin(x + k) * np.cos(2 * y + 0.3 * k) + 0.3 * np.cos(3 * y + k + 0 * x) for k in range(6)])
    if kind == "noise":
        f = rng.standard_normal((6, N, N))
    elif kind == "small_noise":
        f = f + 0.03 * rng.standard_normal((6, N, N))
    elif kind == "jumps":
        f = np.sign(f) + 0.25 * (x > 2)
    elif kind == "half":
        f = f + np.where(x > math.pi, 0.5, 0.0) * rng.standard_normal((6, N, N))
    scale = np.array([amp[0], amp[0], amp[0], amp[1], amp[1], amp[1]])   # of u and theta, of v and q
    return f * scale[:, None, None]


def _solve(X0, nx, ny, scheme, dt, tile=-1, steps=1, weno_eps=1e-6, tab=tableaux.gsa2, graph=0, eps=1.0, tau=50.0):
    L = 2 * math.pi
    p = api.default_params(nx, ny, eps=eps, dt=dt, tau=tau, space_scheme=scheme, tableau=tab(), weno_eps=weno_eps,
                           Lx=L * nx / N, Ly=L * ny / N)
    s = api.Solver(p)
    s.set_tile(tile)
    s.set_graph_steps(graph)
    s.set_state(torch.from_numpy(X0).cuda())
    s.step(steps)
    return s


def _periods(kind, scheme, amp=(1.0, 1.0), weno_eps=1e-6, tab=tableaux.gsa2):
    X0 = _state(kind, amp)
    dt = 0.2 * (2 * math.pi / N) * amp[0] / amp[1]
    small = _solve(X0, N, N, scheme, dt, weno_eps=weno_eps, tab=tab).get_state().cpu().numpy()
    big = _solve(np.tile(X0, (1, 2, 2)), 2 * N, 2 * N, scheme, dt, weno_eps=weno_eps, tab=tab).get_state().cpu().numpy()
    assert np.all(np.isfinite(small))
    err = [np.max(np.abs(big[m] - np.tile(small[m], (2, 2)))) / np.max(np.abs(small[m])) for m in (0, 1, 3, 4, 5)]
    assert max(err) <= 3e-15, err


@pytest.mark.parametrize("scheme", ["WENO3_C4", "WENO5_C4"])
@pytest.mark.parametrize("kind", ["noise", "small_noise", "jumps", "half"])
def test_rough_data(kind, scheme):
    _periods(kind, scheme)


@pytest.mark.parametrize("tab", [tableaux.euler, tableaux.ars4, tableaux.type_a3])
def test_rough_data_of_other_tableaux(tab):
    _periods("noise", "WENO5_C4", tab=tab)


# Values whose squares leave the float range (the whole WENO5 form has no more range than the pairs), values
# below the pairs' low parts, indicators that differ by more than the float range
@pytest.mark.parametrize("scheme,kind,amp,weno_eps", [("WENO3_C4", "smooth", (1e6, 1e24), 1e-6), ("WENO3_C4", "jumps", (1e6, 1e24), 1e-6),
                                                      ("WENO3_C4", "noise", (1e-35, 1e-35), 1e-6),
                                                      ("WENO5_C4", "smooth", (1e-38, 1e-38), 1e-6),
                                                      ("WENO5_C4", "jumps", (1.0, 1e9), 1e-30), ("WENO5_C4", "smooth", (1.0, 1.0), 1e-30),
                                                      ("WENO3_C4", "jumps", (1.0, 1.0), 1e38), ("WENO5_C4", "noise", (1.0, 1.0), 1e33)])
def test_range_of_values(scheme, kind, amp, weno_eps):
    _periods(kind, scheme, amp=amp, weno_eps=weno_eps)


@pytest.mark.parametrize("scheme", ["WENO3_C4", "WENO5_C4"])
def test_same_bits_on_every_tile_and_in_a_batch(scheme):
    """Which interfaces are rough depends on the field, not on the tile: rough and smooth parts, 5 steps."""
    X0 = np.tile(_state("half"), (1, 3, 3))[:, :262, :300].copy()
    dt = 0.1 * 2 * math.pi / N
    want = _solve(X0, 300, 262, scheme, dt, steps=5, graph=2)
    want.sync_status()
    want = want.get_state()
    for tile in range(6):
        assert torch.equal(_solve(X0, 300, 262, scheme, dt, tile=tile, steps=5).get_state(), want), tile
    L = 2 * math.pi
    p = api.default_params(300, 262, eps=1.0, dt=dt, tau=50.0, space_scheme=scheme, Lx=L * 300 / N, Ly=L * 262 / N,
                           tableau=tableaux.gsa2())
    b = api.Batch(api.default_params(300, 512, eps=1.0, dt=dt, tau=50.0, space_scheme=scheme, tableau=tableaux.gsa2()), 3)
    for k in range(3):   # the first is ahead by two steps, the second holds smaller values
        b.attach(k, p)
        b.set_state(torch.from_numpy(X0 * (1e-3 if k == 1 else 1.0)).cuda(), slot=k)
    b.step_slots(2, {0: 2, 1: 1, 2: 0})
    b.step_slots(5, {0: 3, 1: 4, 2: 5})
    b.sync_status()
    for k in (0, 2):
        assert torch.equal(b.get_state(k), want), k


def test_state_from_a_restart_gives_the_same_bits():
    X0 = np.tile(_state("half"), (1, 2, 2))
    dt = 0.1 * 2 * math.pi / N
    one = _solve(X0, 256, 256, "WENO5_C4", dt, steps=4).get_state()
    half = _solve(X0, 256, 256, "WENO5_C4", dt, steps=2).get_state()
    assert torch.equal(_solve(half.cpu().numpy(), 256, 256, "WENO5_C4", dt, steps=2).get_state(), one)
