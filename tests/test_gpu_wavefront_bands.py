"""The bands of depth-2 wavefronts: over members whose tile nobody has set they
are as high as sweeps of 32 rows or planes make them, and over the shortest
sweeps that can be set the fields are those of depth 1, bit for bit."""
import ctypes as C

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


def launches(stream, call):
    """Kernel nodes of a capture of `call` on the stream."""
    cu, st = C.CDLL("libcuda.so.1"), C.c_void_p(stream.cuda_stream)
    graph, n = C.c_void_p(), C.c_size_t()
    assert cu.cuStreamBeginCapture_v2(st, 2) == 0
    call()
    assert cu.cuStreamEndCapture(st, C.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    assert cu.cuGraphDestroy(graph) == 0
    return n.value


@pytest.mark.parametrize("prec,shape,scheme,rows", [("f32", (64, 64, 64), "SBAR120", (34, 10, 32)), ("f64", (48, 40, 96), "S100", (34, 10, 32)),
                                                    ("f32", (256, 256), "SBAR21", (64, 1, 32))])
def test_wavefront_bands_of_default_tiles(native, prec, shape, scheme, rows):
    """Every band is a launch: a wavefront over members whose tile nobody has set
    takes as many as over sweeps of 32 rows or planes."""
    import torch
    st = torch.cuda.Stream()
    out = []
    for tile in (None, rows):
        s = make(native, prec, shape, scheme, st)
        if tile:
            s.set_tile(*tile)
        g = native.Group(1, 4096, stream=st)
        g.add(s)
        g.set_depth(2, 1)
        g.step(2, use_graph=False)
        st.synchronize()
        out.append(launches(st, lambda: g.step(2, use_graph=False)))
        g.remove(s)
        s.close()
        g.close()
    assert out[0] == out[1] > 0


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("shape,scheme,tile", [((70, 41), "SBAR21", (64, 1, 2)), ((130, 30), "S21", (64, 1, 3)),
                                               ((33, 14, 21), "SBAR120", (34, 10, 4)), ((62, 13, 18), "S100", (34, 10, 5))])
def test_lowest_bands(native, shape, scheme, tile, prec):
    import torch
    st, out = torch.cuda.Stream(), []
    for depth in (1, 2):
        s = make(native, prec, shape, scheme, st)
        s.set_tile(*tile)
        g = native.Group(1, native.Group.work_items(s), stream=st)
        g.add(s)
        g.set_depth(depth, 1)
        g.step(6)
        assert g.depth()[2] == depth
        st.synchronize()
        g.remove(s)
        out.append(s.get_fields())
        s.close()
        g.close()
    for x, y in zip(*out):
        assert np.isfinite(x).all() and np.array_equal(x, y)
