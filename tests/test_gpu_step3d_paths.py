"""The 3D step's two passes against the FP64 oracle where the U pass changes
between its ways: planes of one phase (liquid, solid) before, at and after
planes with the interface, sweeps that begin and end in each of them, both
orders of the phases along z, and strips and row pairs at the edges of the
grid.  psi is five times a signed distance, so that phi is exactly +-1 a few
cells from the interface.  FP64, one and three steps: 1e-12 relative per step,
as in the other parity tests of this kernel.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2110_12448_gb300 import synth
from tests.helpers import oracle_params, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_12448_gb300 import native as N
    N.lib()
    return N


def state(nx, ny, nz, scheme, shape, n_grains):
    rng = np.random.default_rng(nx * ny + nz)
    w = synth.free_dendrite_3d(nx, scheme=scheme)
    w.ny, w.nz = ny, nz
    z, y, x = np.meshgrid(*[np.arange(n) * w.h for n in (nz, ny, nx)], indexing="ij")
    if shape == "slab":  # solid below, liquid above
        d = 0.45 * nz * w.h - z + 0.6 * np.sin(x / 3.0) * np.cos(y / 4.0)
    elif shape == "hole":  # liquid between solids
        d = np.abs(z - 0.5 * nz * w.h) - 0.22 * nz * w.h + 0.5 * np.cos(x / 5.0)
    else:
        d = 0.3 * min(nx, ny, nz) * w.h - np.sqrt((x - 0.5 * nx * w.h) ** 2 + (y - 0.4 * ny * w.h) ** 2 + (z - 0.5 * nz * w.h) ** 2)
    U = w.U0 + 0.1 * np.sin(x / 4.0 + z / 3.0) * np.cos(y / 5.0)
    g, rots = synth.random_grains(rng, w, max(1, n_grains))
    return w, 5.0 * d, U, (g if n_grains > 1 else np.zeros_like(g)), rots


def check(N, w, psi, U, g, rots, sweep, steps, time_level=0):
    p = N.make_params(3, w.nx, w.ny, w.nz, w.h, w.dt, w.k, w.eps4, w.lam, w.D, w.U0, w.scheme, "f64",
                      max_grains=rots.shape[0], time_level=time_level)
    s = N.Sim(p)
    s.set_tile(34, 10, sweep)
    s.set_grains(rots)
    s.set_grain_index(g)
    s.set_fields(psi, U)
    s.step(steps)
    gp, gu = s.get_fields()
    s.close()
    op, ou = O.step(oracle_params(w, time_level=time_level), rots, g, psi, U, steps)
    assert rel_err(gp, op) < steps * 1e-12 and rel_err(gu, ou) < steps * 1e-12


@pytest.mark.parametrize("sweep", [8, 11, 64])
@pytest.mark.parametrize("shape", ["slab", "hole", "ball"])
@pytest.mark.parametrize("scheme", ["SBAR120", "S100"])
def test_phases_along_the_sweep(native, scheme, shape, sweep):
    w, psi, U, g, rots = state(34, 19, 50, scheme, shape, 1)
    check(native, w, psi, U, g, rots, sweep, 3)


@pytest.mark.parametrize("time_level,n_grains", [(0, 1), (0, 3), (1, 1)])
@pytest.mark.parametrize("nx,ny", [(4, 13), (29, 6), (30, 7), (31, 12), (60, 5), (62, 14), (92, 9)])
def test_strip_and_row_edges(native, nx, ny, time_level, n_grains):
    w, psi, U, g, rots = state(nx, ny, 21, "SBAR120", "slab", n_grains)
    check(native, w, psi, U, g, rots, 8, 1, time_level)
