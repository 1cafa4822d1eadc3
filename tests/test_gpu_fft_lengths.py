"""Power-of-two transforms of every length, along rows and along columns: the steps that are left
over when log2 n is no multiple of three, the length that needs one step, odd numbers of rows
(one row without a partner) and column groups that the spectrum does not fill.

FP64 against the oracle to 1e-12 (relative max-norm per moment plane, the bound of the size
tests); FP32 velocity on a resolved flow to 1e-5 (the bound of the mixed-radix FP32 test).
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ap_dvm_oracle as O  # noqa: E402
from paper_2512_19847_gb300 import api, tableaux, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _run(nx, ny, X0, steps, precision, **kw):
    A_ex, A_im = tableaux.gsa2()
    p = api.default_params(nx, ny, tau=0.05, tableau=(A_ex, A_im), **kw)
    p.precision = precision
    s = api.Solver(p)
    s.set_state(torch.from_numpy(X0).cuda())
    s.step(steps)
    s.sync_status()
    o = O.Params(nx, ny, kw["eps"], 0.05, kw["dt"], np.array(A_ex), np.array(A_im), scheme=kw["space_scheme"])
    return s.get_state().cpu().numpy(), O.run(X0, o, steps)


@pytest.mark.parametrize("other", [8, 9])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("k", range(3, 13))
def test_every_length_fp64(k, axis, other):
    nx, ny = (2 ** k, other) if axis == 0 else (other, 2 ** k)
    X0 = W.random_moment_state(nx, ny, seed=10 * k + axis, amp=0.4)
    got, ref = _run(nx, ny, X0, 2, api.FP64, eps=1e-2, dt=1e-3, space_scheme="LF1_C2")
    scale = np.max(np.abs(ref), axis=(1, 2), keepdims=True)
    assert np.max(np.abs(got - ref) / scale) <= 1e-12


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("k", range(4, 13))
def test_every_length_fp32(k, axis):
    nx, ny = (2 ** k, 16) if axis == 0 else (16, 2 ** k)
    u1, u2, pr = W.taylor_green(nx, ny)
    X0 = O.equilibrium_state(u1, u2, pr)
    dt = W.stable_dt(u1, u2, 2 * math.pi / max(nx, ny), 0.05)
    got, ref = _run(nx, ny, X0, 3, api.FP32_DEV, eps=1e-4, dt=dt, mach=1e-3, space_scheme="WENO5_C4")
    err = np.max(np.hypot(got[0] - ref[0], got[1] - ref[1])) / np.max(np.hypot(ref[0], ref[1]))
    assert err <= 1e-5, err
