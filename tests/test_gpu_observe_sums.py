"""The observe's sums over fields whose |psi| spans every way a cell is summed
(near the interface, the bulk with its exponential tail, the bulk where phi is
+-1), on row lengths read four cells at a time and one by one, with queues that
fill, spill over and stay short.

Reference: numpy in extended precision.  Tolerance 1e-13 of the sum of the
terms' magnitudes: a cell's phi is within 4e-16, and a thread adds at most a few
hundred FP64 terms (rounding below 1e-16 of the running sum each)."""
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


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("reach", [3.0, 17.9, 45.0])
@pytest.mark.parametrize("nx,ny", [(4, 5), (61, 40), (64, 33), (130, 700), (1024, 610)])
def test_sums(native, nx, ny, reach, prec):
    rng = np.random.default_rng(nx + ny)
    w = synth.free_dendrite_2d(nx, ny=ny)
    dt = np.float32 if prec == "f32" else np.float64
    psi = rng.uniform(-reach, reach, (ny, nx)).astype(dt)
    psi[:, : nx // 4] = dt(40.0)
    psi[: ny // 5] = dt(-50.0)
    U = rng.uniform(-0.7, 0.1, (ny, nx)).astype(dt)
    s = native.Sim(native.make_params(2, nx, ny, 1, w.h, w.dt, w.k, w.eps4, w.lam, w.D, w.U0, "SBAR21", prec))
    s.set_fields(psi, U)
    o = s.observe()
    s.close()
    ph = np.tanh(psi.astype(np.longdouble) / np.sqrt(np.longdouble(2)))
    k = np.longdouble(w.k)
    t = (1 + k - (1 - k) * ph) * (1 + (1 - k) * U.astype(np.longdouble)) / 2
    assert abs(o["solute"] - float(t.sum()) * w.h**2) <= 1e-13 * float(np.abs(t).sum()) * w.h**2
    assert abs(o["solid_fraction"] - float(((1 + ph) / 2).mean())) <= 1e-13
