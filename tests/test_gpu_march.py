"""FP32 solves of at least 384 x 384 cells are taken by the marching kernels: against the
oracle at column counts about multiples of a warp's 26, ragged row segments, every tableau
form (stored terms: the second-order tableau's and the general ones), every scheme, with and without the
relaxation in pairs, and in a batch beside solves of the tile kernels."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ap_dvm_oracle as O  # noqa: E402
from paper_2512_19847_gb300 import api, tableaux, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu
TABS = {"gsa2": tableaux.gsa2, "euler": tableaux.euler, "type_a3": tableaux.type_a3, "ars4": tableaux.ars4}


def _setup(nx, ny, tab, eps, prec=api.FP32_DEV, scheme="WENO5_C4"):
    A_ex, A_im = TABS[tab]()
    X, Y = W.cell_centres(nx, ny)
    u1 = np.sin(X + 0.3) * np.cos(2 * Y) + 0.3 * np.cos(3 * Y + 0.1)
    u2 = -0.5 * np.cos(X + 0.3) * np.sin(2 * Y) + 0.2 * np.sin(2 * X)
    X0 = O.equilibrium_state(u1, u2, 0.25 * np.cos(X + Y))
    dt = W.stable_dt(u1, u2, 2 * math.pi / max(nx, ny), 0.05)
    p = api.default_params(nx, ny, eps=eps, dt=dt, tau=0.05, mach=1e-2, tableau=(A_ex, A_im), precision=prec,
                           space_scheme=scheme)
    return X0, p, O.Params(nx, ny, eps, 0.05, dt, np.array(A_ex), np.array(A_im), scheme=scheme)


def _run(X0, p, steps, graph=0):
    s = api.Solver(p)
    s.set_graph_steps(graph)
    s.set_state(torch.from_numpy(X0).cuda())
    s.step(steps)
    s.sync_status()
    return s


# The FP32 form's bound of the other tests, 1e-5 of the plane's maximum; at eps = 0.5 for u, theta and v
# (theta and v ride at eps in the populations), at 1e-5 for u.  q rides at eps^2: q = (d2 - d1 - d3) /
# (4 eps^2) from six populations of |f| <= 0.6 rounded to 2^-25, 1.1e-7 at eps = 0.5, and as much from
# D_0 . v of the rounded v: 1e-6, four to five times their sum.
def _check(X0, p, o, eps, steps=2, graph=0):
    got = _run(X0, p, steps, graph).get_state().cpu().numpy()
    ref = O.run(X0, o, steps)
    for m in range(5) if eps > 0.1 else (0, 1):
        err = np.max(np.abs(got[m] - ref[m])) / np.max(np.abs(ref[m]))
        assert err <= 1e-5, (m, err)
    if eps > 0.1:
        assert np.max(np.abs(got[5] - ref[5])) <= 1e-6


@pytest.mark.parametrize("nx,ny", [(384, 384), (390, 384), (391, 400), (416, 355), (509, 291), (1000, 150), (156, 1001), (2048, 73)])
def test_sizes(nx, ny):
    X0, p, o = _setup(nx, ny, "gsa2", 0.5)
    _check(X0, p, o, 0.5)


@pytest.mark.parametrize("scheme", ["LF1_C2", "WENO3_C4"])
@pytest.mark.parametrize("nx,ny,tab", [(390, 384, "gsa2"), (509, 291, "gsa2"), (391, 400, "ars4")])
def test_schemes(nx, ny, tab, scheme):
    X0, p, o = _setup(nx, ny, tab, 0.5, scheme=scheme)
    _check(X0, p, o, 0.5)


@pytest.mark.parametrize("tab", ["euler", "ars4", "type_a3"])
@pytest.mark.parametrize("eps", [0.5, 1e-5])
def test_tableaux(tab, eps):
    X0, p, o = _setup(400, 390, tab, eps)
    _check(X0, p, o, eps, graph=2)


@pytest.mark.parametrize("prec", [api.FP32_DEV, api.FP32_DEV_TH])
def test_batch_beside_tiles_equals_alone(prec):
    sizes = [(64, 64), (400, 400), (384, 32), (512, 300)]
    tmpl = _setup(1024, 1024, "gsa2", 1e-4, prec)[1]   # transforms as long as any of them needs
    b = api.Batch(tmpl, len(sizes))
    want = []
    for k, (nx, ny) in enumerate(sizes):
        X0, p, _ = _setup(nx, ny, "gsa2", 1e-4, prec)
        b.attach(k, p)
        b.set_state(torch.from_numpy(X0).cuda(), slot=k)
        want.append([_run(X0, p, n).get_state() for n in (3, 2, 1, 3)[k:k + 1]][0])
    b.step_slots(3, {0: 3, 1: 2, 2: 1, 3: 3})
    b.sync_status()
    for k in range(len(sizes)):
        assert torch.equal(b.get_state(k), want[k])
    b.detach(0)
    b.detach(2)          # the tile kernels' solves are gone
    b.step(2)
    b.sync_status()


@pytest.mark.parametrize("scheme", ["LF1_C2", "WENO3_C4", "WENO5_C4"])
@pytest.mark.parametrize("eps,tab", [(1e-2, "gsa2"), (1e-5, "gsa2"), (1e-2, "ars4")])
def test_small_solves_of_a_large_batch_equal_alone(scheme, eps, tab):
    """Enough cells together, so that every solve of the batch is taken by the marching kernels (but the
    one too narrow for them): bit for bit what the tile kernels give each alone."""
    sizes = [(256, 256), (128, 128), (64, 64), (100, 200), (127, 255), (300, 300), (40, 400), (210, 300)]
    tmpl = _setup(1024, 1024, tab, eps, scheme=scheme)[1]
    b = api.Batch(tmpl, len(sizes))
    want = []
    for k, (nx, ny) in enumerate(sizes):
        X0, p, _ = _setup(nx, ny, tab, eps, scheme=scheme)
        b.attach(k, p)
        b.set_state(torch.from_numpy(X0).cuda(), slot=k)
        want.append(_run(X0, p, 2).get_populations(dtype=torch.float32))
    b.step(2)
    b.sync_status()
    for k in range(len(sizes)):
        assert torch.equal(b.get_populations(k, dtype=torch.float32), want[k]), sizes[k]


def test_non_finite_values_reach_the_status():
    X0, p, _ = _setup(400, 400, "gsa2", 1e-2)
    X0[0, 11, 399] = np.inf
    s = api.Solver(p)
    s.set_state(torch.from_numpy(X0).cuda())
    s.step(2)
    with pytest.raises(api.ApDvmError) as e:
        s.sync_status()
    assert e.value.status == 5
