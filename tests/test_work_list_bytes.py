"""pf_required_bytes leaves room for the work list of the shortest sweep that the
library chooses or pf_set_tile takes (host only): the fields, the grain map, the
304 observe partials of 72 bytes and a 32-byte item per strip and sweep."""
import pytest

from paper_2110_12448_gb300 import native as N


def cut(n, k):
    return -(-n // k)


@pytest.mark.parametrize("prec,cell", [("f32", 18), ("f64", 34), ("f32c", 34)])
@pytest.mark.parametrize("nx,ny", [(4, 4), (61, 4000), (60, 4001), (1024, 1024), (781, 781), (4, 65536), (4096, 63)])
def test_2d(nx, ny, prec, cell):
    lists = 32 * cut(nx, 60) * cut(ny, 2)
    assert N.required_bytes(N.make_params(2, nx, ny, precision=prec)) >= cell * nx * ny + 304 * 72 + lists


@pytest.mark.parametrize("prec,cell", [("f32", 18), ("f64", 34)])
@pytest.mark.parametrize("nx,ny,nz", [(4, 4, 4), (12, 4, 4000), (60, 61, 999), (30, 300, 65), (157, 121, 189)])
def test_3d(nx, ny, nz, prec, cell):
    p = N.make_params(3, nx, ny, nz, scheme="SBAR120", dt=0.01, precision=prec)
    lists = 32 * cut(nx + 1, 30) * cut(ny, 6) * cut(nz, 4)  # 30 x 6 columns, outputs from one column before a strip
    assert N.required_bytes(p) >= cell * nx * ny * nz + 304 * 72 + lists
