"""The 2D step's paths: strips wholly inside the grid with rows of even and of
odd length, strips that touch a wall, one crystal frame for all cells and
per-cell frames, orthonormal frames (J - g from the reflection about the crystal
axes) and matrices that are not (J - g by rotation into the frame and back).

FP64 against the oracle over one step: 1e-12 relative.  FP32 across the ways a
strip reaches its rows: every cell gets the same operations on the same values,
so cells further from the walls than the stencil reaches have the same bits.
FP32 with matrices that are not orthonormal against the oracle: 2e-6 on phi and
5e-6 on U, the figures of the one-step parity tests of this scheme.  A frame
1e-7 off orthonormal changes J - g by less than 1e-7 of the gradient, below
FP32's own rounding of it, and takes the reflection in FP32 but not in FP64.
"""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2110_12448_gb300 import synth
from tests.helpers import max_abs, oracle_params, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_12448_gb300 import native as N
    N.lib()
    return N


def check(N, w, scheme, prec, g, rots, psi, U, time_level=0):
    if prec == "f32":
        psi, U = psi.astype(np.float32), U.astype(np.float32)
    p = N.make_params(2, w.nx, w.ny, 1, w.h, w.dt, w.k, w.eps4, w.lam, w.D, w.U0, scheme, prec,
                      max_grains=rots.shape[0], time_level=time_level)
    s = N.Sim(p)
    s.set_tile(64, 1, 16)
    s.set_grains(rots)
    s.set_grain_index(g)
    s.set_fields(psi, U)
    s.step(1)
    gp, gu = s.get_fields()
    s.close()
    psi, U = psi.astype(np.float64), U.astype(np.float64)
    op, ou = O.step(oracle_params(w, scheme, time_level=time_level), rots, g, psi, U, 1)
    if prec == "f64":
        assert rel_err(gp, op) < 1e-12 and rel_err(gu, ou) < 1e-12
    else:
        assert max_abs(np.tanh(gp.astype(np.float64) / math.sqrt(2)), np.tanh(op / math.sqrt(2))) < 2e-6
        assert max_abs(gu, ou) < 5e-6


def state(seed, nx, ny, scheme, n_grains):
    rng = np.random.default_rng(seed)
    w = synth.free_dendrite_2d(nx, ny=ny, scheme=scheme, eps4=0.05)
    psi, U = synth.random_state(rng, w)
    g, rots = synth.random_grains(rng, w, max(1, n_grains))
    return w, psi, U, (g if n_grains > 1 else np.zeros_like(g)), rots


@pytest.mark.parametrize("n_grains", [1, 4])
@pytest.mark.parametrize("nx,ny", [(61, 17), (122, 33), (123, 16), (124, 15), (182, 40), (243, 9)])
@pytest.mark.parametrize("scheme", ["SBAR21", "S21", "S10"])
def test_strips_and_frames_against_the_oracle(native, scheme, nx, ny, n_grains):
    w, psi, U, g, rots = state(nx + ny, nx, ny, scheme, n_grains)
    check(native, w, scheme, "f64", g, rots, psi, U)


@pytest.mark.parametrize("prec", ["f32", "f32c"])
@pytest.mark.parametrize("n_grains", [1, 4])
@pytest.mark.parametrize("cut", [1, 2, 5])
@pytest.mark.parametrize("scheme", ["SBAR21", "S21", "S10"])
def test_fp32_does_not_depend_on_the_strips(native, scheme, cut, n_grains, prec):
    w, psi, U, g, rots = state(7, 252, 37, scheme, n_grains)
    out = []
    for lo in (0, cut):  # the same cells in a grid without its first `cut` columns
        p = native.make_params(2, w.nx - lo, w.ny, 1, w.h, w.dt, w.k, w.eps4, w.lam, w.D, w.U0, scheme, prec,
                               max_grains=rots.shape[0])
        s = native.Sim(p)
        s.set_tile(64, 1, 16 if lo == 0 else 9)
        s.set_grains(rots)
        s.set_grain_index(np.ascontiguousarray(g[:, lo:]))
        s.set_fields(np.ascontiguousarray(psi[:, lo:]), np.ascontiguousarray(U[:, lo:]))
        s.step(1)
        out.append([f[:, cut - lo + 6:] for f in s.get_fields()])
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("time_level", [0, 1])
@pytest.mark.parametrize("shear", [0.2, 1e-7])
@pytest.mark.parametrize("n_grains", [1, 3])
def test_matrices_that_are_not_orthonormal(native, n_grains, shear, time_level, prec):
    w, psi, U, g, rots = state(5, 129, 41, "SBAR21", n_grains)
    rots = rots.reshape(-1, 3, 3).copy()
    rots[-1, 0, 1] += shear
    check(native, w, "SBAR21", prec, g, rots.reshape(-1, 9), psi, U, time_level)


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_reflected_frame(native, prec):
    w, psi, U, g, rots = state(6, 130, 37, "SBAR21", 1)
    rots = rots.reshape(-1, 3, 3).copy()
    rots[0, :, 1] *= -1.0  # orthonormal, determinant -1
    check(native, w, "SBAR21", prec, g, rots.reshape(-1, 9), psi, U)
