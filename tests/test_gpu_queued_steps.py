"""Queued steps, whose launches begin before the one ahead has ended, against
the same steps with a synchronisation after each: bit for bit, at the library's
own sweeps, in the two-kernel form, with a frozen temperature (whose step clock a
kernel advances between the steps), in groups of several classes as direct
launches and as a graph, and as depth-2 wavefronts."""
import numpy as np
import pytest

from paper_2110_12448_gb300 import synth

pytestmark = pytest.mark.gpu

T0, TWO, FROZEN = {"time_level": 1}, {"time_level": 1, "kernels": 1}, {"thermal": 1, "Vp": 0.1, "lT": 1000.0, "yT": 20.0}
ALONE = [("f32", (128, 128), "SBAR21", {}), ("f64", (200, 190), "SBAR21", {}), ("f32c", (127, 130), "S10", {}),
         ("f32", (301, 200), "S21", {}), ("f32", (130, 120), "SBAR21", TWO), ("f64", (90, 120), "S10", TWO),
         ("f32", (130, 200), "SBAR21", {**FROZEN, "bc_x": 1}), ("f32", (48, 40, 44), "SBAR120", {}),
         ("f64", (31, 33, 40), "S100", T0)]
MIXED = [ALONE[0], ALONE[5], ALONE[6], ALONE[7], ("f32", (70, 90), "SBAR21", FROZEN), ("f32c", (64, 70), "SBAR21", {})]
PLAIN = [ALONE[0], ALONE[3], ALONE[7], ("f64", (100, 90), "SBAR21", {}), ("f32", (62, 33, 70), "S100", {})]


@pytest.fixture(scope="module")
def native():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2110_12448_gb300 import native as N
    N.lib()
    return N


def make(N, prec, shape, scheme, kw, st):
    dim = len(shape)
    h = 0.8
    p = N.make_params(dim, *shape, h=h, scheme=scheme, precision=prec, **({"dt": 0.01} if dim == 3 else {}), **kw)
    s = N.Sim(p, stream=st)
    s.set_grains(synth.rot2d(20.0).reshape(1, 9))
    x = np.meshgrid(*[np.arange(n) * h for n in reversed(shape)], indexing="ij")
    psi = 0.3 * min(shape) * h - np.sqrt(sum((c - 0.45 * n * h) ** 2 for c, n in zip(x, reversed(shape)))) + np.sin(x[-1] / 3.0)
    U = -0.5 * (1.0 - np.exp(np.minimum(psi, 0.0) / 10.0))
    dt = np.float32 if prec == "f32" else np.float64
    s.set_fields(psi.astype(dt), U.astype(dt))
    return s


def same(a, b):
    for x, y in zip(a, b):
        assert np.isfinite(x[0]).all() and np.isfinite(x[1]).all()
        assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])


@pytest.mark.parametrize("case", ALONE)
def test_alone(native, case):
    import torch
    st, out = torch.cuda.Stream(), []
    for queued in (False, True):
        s = make(native, *case, st)
        for _ in range(1 if queued else 24):
            s.step(24 if queued else 1)
            st.synchronize()
        out.append([s.get_fields()])
        s.close()
    same(*out)


@pytest.mark.parametrize("members,depth", [(MIXED, 1), (PLAIN, 1), (PLAIN, 2)])
@pytest.mark.parametrize("graph", [False, True])
def test_group(native, graph, members, depth):
    import torch
    st, out = torch.cuda.Stream(), []
    for queued in (False, True):
        sims = [make(native, *m, st) for m in members]
        g = native.Group(len(sims), sum(native.Group.work_items(s) for s in sims), stream=st)
        for s in sims:
            g.add(s)
        g.set_depth(depth, 1)
        for _ in range(1 if queued else 40 // depth):
            g.step(40 if queued else depth, use_graph=graph and queued)
            st.synchronize()
        assert g.depth()[2] == depth
        for s in sims:
            g.remove(s)
        out.append([s.get_fields() for s in sims])
        g.close()
        for s in sims:
            s.close()
    same(*out)
