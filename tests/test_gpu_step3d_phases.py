"""Planes of one phase in the 3D U pass, whose weights are constants and whose
anti-trapping term is left out.  A NaN or an infinity in or beside such planes
reaches the same cells of psi' and U' as in the oracle, which evaluates every
term (exact: sets of cells).  And the constants give the bits of the full
evaluation: the same state at different sweep lengths and at the library's own,
whose first planes are always evaluated in full, has the same bits in FP32 and
FP64, T1 and T0."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2110_12448_gb300 import synth
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


def step(N, w, prec, psi, U, steps=1, sweep=None, time_level=0):
    p = N.make_params(3, w.nx, w.ny, w.nz, w.h, w.dt, w.k, w.eps4, w.lam, w.D, w.U0, w.scheme, prec,
                      time_level=time_level)
    s = N.Sim(p)
    if sweep:
        s.set_tile(34, 10, sweep)
    dt = np.float32 if prec == "f32" else np.float64
    s.set_fields(psi.astype(dt), U.astype(dt))
    s.step(steps)
    out = s.get_fields()
    s.close()
    return out


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("time_level", [0, 1])
@pytest.mark.parametrize("scheme", ["SBAR120", "S100"])
@pytest.mark.parametrize("phase", [-1.0, 1.0])
@pytest.mark.parametrize("field,value", [("psi", np.nan), ("U", np.nan), ("U", np.inf)])
def test_not_finite(native, field, value, phase, scheme, time_level, prec):
    w = small_workload(3, 62, 25, 22, scheme=scheme)
    for at in ((10, 12, 31), (9, 5, 29), (0, 24, 61)):
        f = {"psi": np.full((w.nz, w.ny, w.nx), 40.0 * phase), "U": np.full((w.nz, w.ny, w.nx), -0.3)}
        f[field][at] = value
        op, ou = O.step(oracle_params(w, time_level=time_level), np.eye(3).reshape(1, 9), np.zeros(f["U"].shape, np.int16),
                        f["psi"], f["U"], 1)
        gp, gu = step(native, w, prec, f["psi"], f["U"], time_level=time_level)
        assert np.array_equal(np.isfinite(gp), np.isfinite(op))
        assert np.array_equal(np.isfinite(gu), np.isfinite(ou))


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("time_level", [0, 1])
@pytest.mark.parametrize("scheme", ["SBAR120", "S100"])
def test_sweeps_have_the_same_bits(native, scheme, time_level, prec):
    w = small_workload(3, 61, 23, 50, scheme=scheme)
    z, y, x = np.meshgrid(*[np.arange(n) * w.h for n in (w.nz, w.ny, w.nx)], indexing="ij")
    # solid, liquid and solid again along z, steep enough that phi = +-1 a few planes from the interfaces
    psi = 5.0 * (np.abs(z - 0.5 * w.nz * w.h) - 0.22 * w.nz * w.h + 0.5 * np.cos(x / 5.0))
    U = w.U0 + 0.1 * np.sin(x / 4.0 + z / 3.0) * np.cos(y / 5.0)
    out = [step(native, w, prec, psi, U, 4, sweep, time_level) for sweep in (None, 8, 11, 50)]
    assert np.isfinite(out[0][1]).all()
    for a in out[1:]:
        assert np.array_equal(a[0], out[0][0]) and np.array_equal(a[1], out[0][1])
