"""The default tile of an instance (host only): its work list fits the buffer
that pf_required_bytes asks for, so that pf_create succeeds on a device for
every size; checked through the byte counts of grids from the smallest to large
ones, which grow with the cells and never shrink below their fields."""
import pytest

from paper_2110_12448_gb300 import native as N


@pytest.mark.parametrize("prec,cell", [("f32", 18), ("f64", 34), ("f32c", 34)])
@pytest.mark.parametrize("nx,ny", [(4, 4), (61, 5), (128, 128), (200, 200), (1024, 1024), (4096, 64), (64, 4096)])
def test_required_bytes_2d(nx, ny, prec, cell):
    n = N.required_bytes(N.make_params(2, nx, ny, precision=prec))
    lists = 32 * (-(-nx // 60)) * (-(-ny // 2))  # sweeps of two rows, the shortest default
    assert cell * nx * ny <= n <= cell * nx * ny + lists + 40_000


@pytest.mark.parametrize("time_level,cell", [(0, 18), (1, 22)])
@pytest.mark.parametrize("n", [4, 31, 64, 157])
def test_required_bytes_3d(n, time_level, cell):
    b = N.required_bytes(N.make_params(3, n, n, n, scheme="SBAR120", dt=0.01, time_level=time_level))
    assert cell * n**3 <= b <= cell * n**3 + 32 * (n // 12 + 1) * (n // 4 + 1) ** 2 + 40_000
