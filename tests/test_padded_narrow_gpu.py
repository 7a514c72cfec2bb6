"""The narrowest grids whose rows are padded (a quarter more at most: 7, 13 to
15, 20 to 23, 26 to 28 voxels): one x-tile, rows far shorter than the copied
boxes.  Bit for bit the direct kernels' results, without CPML, with one cell
of it and with as much as fits."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("pml", ["none", "thin", "thick"])
@pytest.mark.parametrize("nx,n_sls", [(7, 2), (13, 2), (15, 1), (20, 2), (23, 0), (26, 2)])
def test_gpu_narrow_padded_rows_match_direct_kernels_bitwise(nx, n_sls, pml, storage, monkeypatch):
    from tests import test_padded_rows_gpu as padded
    from paper_2301_12727_gb300 import bvf
    n_pml = {"none": 0, "thin": 1, "thick": (nx - 2) // 2}[pml]
    ny, nz = max(19, 2 * n_pml + 2), max(14, 2 * n_pml + 3)
    s = bvf.Solver(nx, ny, nz, 0.5e-3, 4e-8, 5e5, n_sls=n_sls, n_pml=n_pml, storage=storage)
    for kernel in (1, 2):
        bvf.bvf_test_withhold_tma(s.ctx, kernel, 3, 64)      # refused on the direct kernels
    s.close()
    padded.test_padded_rows_match_direct_kernels_bitwise(nx, ny, nz, n_pml, n_sls, storage, monkeypatch)
