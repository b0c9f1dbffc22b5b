"""Rows far from the interface on the compensated FP32 state, whose psi rate
takes constants for phi and the coupling term.

NaN and infinities there reach the same cells as in the oracle, which evaluates
every term (exact: sets of cells).  A coupling term that is large enough to
matter is not left out: with uniform psi of +-25 to +-32 (no gradients, so the rate
is sqrt2 (phi - lambda (1 - phi^2) U) / a_s^2, a_s = 1), psi' with U minus psi' with
U = 0 is -dt sqrt2 lambda (1 - phi^2) U, 1 - phi^2 = 4 e / (1 + e)^2 with e =
e^{-sqrt2 |psi|} (the oracle's phi, an FP64 tanh, does not hold it), within 1e-13 +
1e-8 of itself: half a unit in the last place of two lo halves (5.7e-14), what the
kernel leaves out below its bound (2.1e-14), and the FP32 part of a_s^2 (4e-9)."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from tests.helpers import oracle_params, small_workload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_12448_gb300 import native as N
    N.lib()
    return N


def both(N, w, psi, U):
    s = N.Sim(N.make_params(2, w.nx, w.ny, 1, w.h, w.dt, w.k, w.eps4, w.lam, w.D, w.U0, w.scheme, "f32c"))
    s.set_fields(psi, U)
    s.step(1)
    got = s.get_fields()
    s.close()
    return got, O.step(oracle_params(w), np.eye(3).reshape(1, 9), np.zeros(psi.shape, np.int16), psi, U, 1)


@pytest.mark.parametrize("scheme", ["SBAR21", "S10", "S21"])
@pytest.mark.parametrize("psi0", [-40.0, 28.0])
@pytest.mark.parametrize("field,value", [("psi", np.nan), ("U", np.nan), ("U", np.inf)])
def test_not_finite(native, field, value, psi0, scheme):
    w = small_workload(2, 124, 40, scheme=scheme)
    for at in ((20, 61), (0, 0), (33, 123)):
        f = {"psi": np.full((w.ny, w.nx), psi0), "U": np.full((w.ny, w.nx), -0.3)}
        f[field][at] = value
        (gp, gu), (op, ou) = both(native, w, f["psi"], f["U"])
        assert np.array_equal(np.isfinite(gp), np.isfinite(op))
        assert np.array_equal(np.isfinite(gu), np.isfinite(ou))


@pytest.mark.parametrize("U0", [-0.55, 3.0, 1e4, 1e9])
@pytest.mark.parametrize("psi0", [-25.0, 26.0, -32.0])
def test_coupling(native, psi0, U0):
    w = small_workload(2, 124, 24)
    (gp, _), _ = both(native, w, np.full((w.ny, w.nx), psi0), np.full((w.ny, w.nx), U0))
    (gz, _), _ = both(native, w, np.full((w.ny, w.nx), psi0), np.zeros((w.ny, w.nx)))
    e = math.exp(-math.sqrt(2.0) * abs(psi0))
    want = -w.dt * math.sqrt(2.0) * w.lam * 4.0 * e / (1.0 + e) ** 2 * U0
    assert np.abs((gp - gz) - want).max() <= 1e-13 + 1e-8 * abs(want)
