"""The observe's sums over fields whose U is finite but large, as a run that
diverges leaves them: all of it, or cells of it among ordinary ones, near the
interface and in both bulks.

Reference: numpy in extended precision.  Tolerance 1e-13 of the sum of the
terms' magnitudes, as for ordinary fields: the sums are FP64."""
import numpy as np
import pytest

from paper_2110_12448_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_12448_gb300 import native as N
    N.lib()
    return N


@pytest.mark.parametrize("prec,large", [("f32", 3e38), ("f32", 1e19), ("f64", 1e300), ("f64", 1e39), ("f32c", 1e30)])
@pytest.mark.parametrize("share", [1.0, 0.02])
@pytest.mark.parametrize("nx", [64, 61])
def test_sums(native, nx, share, prec, large):
    rng = np.random.default_rng(nx)
    ny = 70
    w = synth.free_dendrite_2d(nx, ny=ny)
    dt = np.float32 if prec == "f32" else np.float64
    psi = rng.uniform(-45.0, 45.0, (ny, nx)).astype(dt)
    psi[:20] = rng.uniform(-900.0, 900.0, (20, nx)).astype(dt)
    U = np.where(rng.random((ny, nx)) < share, large, rng.uniform(-0.7, 0.1, (ny, nx))).astype(dt)
    s = native.Sim(native.make_params(2, nx, ny, 1, w.h, w.dt, w.k, w.eps4, w.lam, w.D, w.U0, "SBAR21", prec))
    s.set_fields(psi, U)
    psi, U = s.get_fields()  # F32C: as its pairs hold them
    o = s.observe()
    s.close()
    assert o["nonfinite"] == 0
    ph = np.tanh(psi.astype(np.longdouble) / np.sqrt(np.longdouble(2)))
    k = np.longdouble(w.k)
    t = (1 + k - (1 - k) * ph) * (1 + (1 - k) * U.astype(np.longdouble)) / 2
    assert abs(o["solute"] - float(t.sum()) * w.h**2) <= 1e-13 * float(np.abs(t).sum()) * w.h**2
    assert abs(o["solid_fraction"] - float(((1 + ph) / 2).mean())) <= 1e-13
