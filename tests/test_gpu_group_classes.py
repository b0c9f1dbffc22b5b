"""A group member whose matrices are not orthonormal takes other arithmetic than
its orthonormal classmates; their fields are those they get alone."""
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


def make(N, prec, shape, scheme, st=None, **kw):
    dim = len(shape)
    if dim == 3:
        kw = {"dt": 0.01, **kw}
    s = N.Sim(N.make_params(dim, *shape, scheme=scheme, precision=prec, **kw), stream=st)
    r0 = 0.3 * min(shape) * 0.8
    s.init_seeds([[0.4 * shape[0], 0.4 * shape[1], 0.4 * shape[-1] if dim == 3 else 0.0, r0]], [0])
    return s


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_members_with_any_matrices_leave_the_others_alone(native, prec):
    import torch
    st = torch.cuda.Stream()
    rot = synth.rot2d(20.0).reshape(3, 3).copy()
    bent = rot.copy()
    bent[0, 1] += 0.1
    kws = [dict(bc_x=1), dict(bc_x=1), {}, dict(thermal=1, Vp=0.1, lT=900.0, yT=30.0)]

    def sims():
        out = []
        for i, kw in enumerate(kws):
            s = make(native, prec, (150 + 20 * i, 130), "SBAR21", st, **kw)
            s.set_grains((bent if i in (1, 2) else rot).reshape(1, 9))
            out.append(s)
        return out

    alone = []
    for s in sims():
        s.step(6)
        alone.append(s.get_fields())
        s.close()
    ss = sims()
    g = native.Group(len(ss), sum(native.Group.work_items(s) for s in ss), stream=st)
    for s in ss:
        g.add(s)
    g.step(6)
    st.synchronize()
    for s, a in zip(ss, alone):
        g.remove(s)
        for x, y in zip(s.get_fields(), a):
            assert np.array_equal(x, y)
        s.close()
    g.close()
