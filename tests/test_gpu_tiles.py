"""Tiles at the library's own choice: pf_set_tile takes what pf_get_tile reports,
on the same handle and on handles of other sizes, with the same fields; block
shapes that are not compiled and sweeps below the shortest choice are refused."""
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


@pytest.mark.parametrize("prec", ["f32", "f64", "f32c"])
@pytest.mark.parametrize("scheme,small,large", [("SBAR21", (128, 128), (700, 650)), ("SBAR21", (4, 4), (61, 2000)),
                                                ("S10", (512, 512), (200, 200)), ("SBAR120", (64, 64, 64), (40, 37, 90)),
                                                ("S100", (4, 4, 4), (61, 13, 33))])
def test_reported_tiles_are_taken(native, scheme, small, large, prec):
    if prec == "f32c" and len(small) == 3:
        pytest.skip("2D only")
    for a in (small, large):
        own = make(native, prec, a, scheme)
        t = own.get_tile()
        own.step(3)
        for b in (small, large):
            s, ref = make(native, prec, b, scheme), make(native, prec, b, scheme)
            s.set_tile(*t)
            assert s.get_tile() == t
            s.step(3)
            ref.step(3)
            for x, y in zip(s.get_fields(), ref.get_fields()):
                assert np.array_equal(x, y)
            s.close()
            ref.close()
        own.close()


def test_refused_tiles(native):
    s = make(native, "f32", (128, 128), "SBAR21")
    t = s.get_tile()
    for bad in ((4, 1, 0), (100, 1, 0), (64, 1, 1), (64, 1, -8), (64, 1, (1 << 20) + 1)):
        with pytest.raises(native.PfError):
            s.set_tile(*bad)
        assert s.get_tile() == t
    s = make(native, "f32", (64, 64, 64), "SBAR120")
    for bad in ((4, 10, 0), (34, 4, 0), (34, 10, 3)):
        with pytest.raises(native.PfError):
            s.set_tile(*bad)


def test_another_block_shape_gets_its_own_choice(native):
    a, b = (make(native, "f32", (160, 150, 140), "SBAR120") for _ in range(2))
    a.set_tile(34, 18, 0)
    assert a.get_tile()[:2] == (34, 18)
    a.set_tile(34, 10, 0)
    assert a.get_tile() == b.get_tile()  # still the library's choice
    a.set_tile(0, 0, 16)
    a.set_tile(34, 18, 0)
    assert a.get_tile() == (34, 18, 16)
