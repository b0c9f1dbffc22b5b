"""Steps whose launches begin before the step ahead of them has ended: a queue
of steps gives the bits of the same steps with a synchronisation after each,
with as many blocks as the GPU has SMs, one row of blocks fewer and more, and
on full grids; launched directly and as a group's graph; 2D in each precision
and 3D, whose passes follow one another in the same way."""
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


# 8 strips (2D: 60 columns, 8 rows) or 4 x 2 columns (3D: 30 x 6, 8 planes) times
# 18, 19 = 152 / 8 and 20 sweeps; one block; many more blocks than the GPU holds
@pytest.mark.parametrize("dim,prec,sweeps", [(2, "f32", 1), (2, "f32", 18), (2, "f32", 19), (2, "f32", 20), (2, "f32", 160),
                                             (2, "f64", 19), (2, "f64", 20), (2, "f32c", 19), (2, "f32c", 20),
                                             (3, "f32", 1), (3, "f32", 19), (3, "f32", 20), (3, "f64", 19)])
def test_queued_steps_equal_single_ones(native, dim, prec, sweeps):
    import torch
    if dim == 2:
        w = synth.free_dendrite_2d(480 if sweeps > 1 else 60, ny=8 * sweeps)
    else:
        w = synth.free_dendrite_3d(118 if sweeps > 1 else 28)
        w.ny, w.nz = 12 if sweeps > 1 else 6, 8 * sweeps
    rng = np.random.default_rng(dim + sweeps)
    psi, U = synth.random_state(rng, w)
    dt = np.float32 if prec == "f32" else np.float64
    out = []
    for how in ("single", "queued", "graph"):
        st = torch.cuda.Stream()
        p = native.make_params(dim, w.nx, w.ny, w.nz, w.h, w.dt, w.k, w.eps4, w.lam, w.D, w.U0, w.scheme, prec)
        s = native.Sim(p, stream=st)
        s.set_grains(w.rots)
        s.set_tile(*((64, 1, 8) if dim == 2 else (34, 10, 8)))
        s.set_fields(psi.astype(dt), U.astype(dt))
        if how == "graph":
            g = native.Group(1, native.Group.work_items(s), stream=st)
            g.add(s)
            g.step(12, use_graph=True)
            st.synchronize()
            g.remove(s)
            g.close()
        else:
            for _ in range(12 if how == "single" else 1):
                s.step(1 if how == "single" else 12)
                st.synchronize()
        out.append(s.get_fields())
        s.close()
    for a in out[1:]:
        assert np.array_equal(a[0], out[0][0]) and np.array_equal(a[1], out[0][1])
