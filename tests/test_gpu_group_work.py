"""A group whose work list is sized as the header says (the sum of its members'
pf_group_work_items), or for sweeps of 32 rows, steps: with several classes, of
very different members, at depth 2, where its own choice for one class or depth
is longer or shorter than its members'; each member's fields are those it gets
alone."""
import numpy as np
import pytest

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


F32C_2048 = [("f32c", (2048, 2048), "SBAR21")]
F64_1536 = [("f64", (1536, 1536), "SBAR21")]
CLASSES_C = [("f32c", (300, 661), "SBAR21"), ("f32c", (300, 538), "S10"), ("f32c", (120, 103), "S10")]
CLASSES_F = [("f32", (2040, 1784), "SBAR21"), ("f32", (300, 133), "S10"), ("f32", (1200, 542), "S10")]
SMALL = [("f32", (300, 300), "SBAR21"), ("f32", (400, 400), "S10"), ("f32", (200, 900), "S21")]
CUBES = [("f32", (62, 45, 40), "SBAR120"), ("f32", (33, 64, 48), "S100"), ("f32", (250, 250), "SBAR21")]


@pytest.mark.parametrize("depth,bands", [(1, 1), (2, 1), (2, 3)])
@pytest.mark.parametrize("members", [F32C_2048, F64_1536, CLASSES_C, CLASSES_F, SMALL, CUBES])
@pytest.mark.parametrize("sized", ["recipe", "rows of 32", "generous"])
def test_groups_step(native, sized, members, depth, bands):
    import torch
    st = torch.cuda.Stream()
    sims = [make(native, *m, st=st) for m in members]
    work = sum(native.Group.work_items(s) for s in sims)
    if sized == "rows of 32":
        cut = lambda n, k: -(-n // k)
        work = sum(cut(m[1][0], 60) * cut(m[1][1], 32) if len(m[1]) == 2 else
                   cut(m[1][0] + 1, 30) * cut(m[1][1], 6) * cut(m[1][2], 32) for m in members)
    elif sized == "generous":
        work *= 20
    g = native.Group(len(sims), work, stream=st)
    for s in sims:
        g.add(s)
    g.set_depth(depth, bands)
    g.step(4)
    assert g.depth()[2] == depth
    st.synchronize()
    for s, m in zip(sims, members):
        g.remove(s)
        ref = make(native, *m, st=st)
        ref.step(4)
        for x, y in zip(s.get_fields(), ref.get_fields()):
            assert np.array_equal(x, y)
        s.close()
        ref.close()
    g.close()
