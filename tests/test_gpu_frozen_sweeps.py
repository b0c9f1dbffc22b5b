"""Frozen-temperature runs do not depend on how the grid is cut into sweeps: the
same bits at every sweep length, alone at the library's own choice and in a
group, whose members share another."""
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


def make(N, w, psi, U, prec, scheme, st, **kw):
    p = N.make_params(2, w.nx, w.ny, 1, w.h, w.dt, w.k, w.eps4, w.lam, w.D, w.U0, scheme, prec,
                      thermal=1, Vp=0.1, lT=1000.0, yT=20.0, **kw)
    s = N.Sim(p, stream=st)
    s.set_grains(synth.rot2d(20.0).reshape(1, 9))
    dt = np.float32 if prec == "f32" else np.float64
    s.set_fields(psi.astype(dt), U.astype(dt))
    return s


def state(seed, nx, ny):
    """A front with fingers, its solute profile and a little noise."""
    w = synth.free_dendrite_2d(nx, ny=ny)
    rng = np.random.default_rng(seed)
    y, x = np.meshgrid(np.arange(ny) * w.h, np.arange(nx) * w.h, indexing="ij")
    psi = 30.0 + 4.0 * np.sin(x / 7.0) + 3.0 * np.cos(x / 4.0) - y
    U = -0.5 * (1.0 - np.exp(np.minimum(psi, 0.0) / 10.0)) + 0.01 * rng.standard_normal(psi.shape)
    return w, psi, U


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("scheme,kw", [("SBAR21", {}), ("S10", {"bc_x": 1}), ("S21", {"time_level": 1}),
                                       ("SBAR21", {"time_level": 1, "kernels": 1})])
def test_sweeps(native, scheme, kw, prec):
    w, psi, U = state(1, 130, 200)
    out = []
    for sweep in (None, 8, 10, 31, 32, 38, 200):
        s = make(native, w, psi, U, prec, scheme, None, **kw)
        if sweep:
            s.set_tile(64, 1, sweep)
        s.step(5)
        out.append(s.get_fields())
        s.close()
    assert np.isfinite(out[0][0]).all() and np.isfinite(out[0][1]).all()
    for a in out[1:]:
        assert np.array_equal(a[0], out[0][0]) and np.array_equal(a[1], out[0][1])


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_alone_and_in_a_group(native, prec):
    import torch
    st = torch.cuda.Stream()
    states = [state(i, nx, ny) for i, (nx, ny) in enumerate([(130, 200), (301, 640), (1024, 777)])]
    alone, sweeps = [], set()
    for w, psi, U in states:
        s = make(native, w, psi, U, prec, "SBAR21", st, bc_x=1)
        sweeps.add(s.get_tile()[2])
        s.step(20)
        alone.append(s.get_fields())
        s.close()
    assert len(sweeps) > 1  # the choices differ, so a shared one differs from some member's own
    ss = [make(native, w, psi, U, prec, "SBAR21", st, bc_x=1) for w, psi, U in states]
    g = native.Group(len(ss), sum(native.Group.work_items(s) for s in ss), stream=st)
    for s in ss:
        g.add(s)
    g.step(20)
    st.synchronize()
    for s, a in zip(ss, alone):
        g.remove(s)
        b = s.get_fields()
        s.close()
        assert np.isfinite(b[0]).all() and np.isfinite(b[1]).all()
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    g.close()
