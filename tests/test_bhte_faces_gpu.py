"""The TMA-fed BHTE step takes a voxel's lower z-face from the plane before
where its chunk has one.  Grids whose chunks hold several planes, materials
that change along z every one to five planes (uniform planes, uniform columns
and neither, border rows and planes): the direct kernel's results bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,n_mat", [(128, 120, 90, 250), (200, 150, 61, 7), (136, 200, 128, 64)])
def test_gpu_layers_match_direct_kernel_bitwise(nx, ny, nz, n_mat, monkeypatch):
    torch = pytest.importorskip("torch")
    from paper_2301_12727_gb300 import bvf
    rng = np.random.default_rng(n_mat)
    mat = np.stack([rng.uniform(900, 1900, n_mat), rng.uniform(1450, 2900, n_mat), np.zeros(n_mat),
                    rng.uniform(1, 80, n_mat), np.zeros(n_mat), rng.uniform(0.2, 0.7, n_mat),
                    rng.uniform(1300, 4200, n_mat), rng.uniform(0, 0.01, n_mat),
                    rng.uniform(0, 1, n_mat)], axis=1)
    index = rng.integers(0, n_mat, (nz, ny, nx)).astype(np.uint8)
    z = 0
    while z < nz:                           # uniform layers between mixed ones
        n = int(rng.integers(1, 6))
        if rng.random() < 0.5:
            index[z:z + n] = rng.integers(0, n_mat)
        z += n
    index[:, 20:40, 30:60] = index[0, 20, 30]            # a uniform column
    index[:, 60:80, 64:100] = rng.integers(0, n_mat, (nz, 1, 1))   # changes along z only
    amp = torch.from_numpy(rng.uniform(0.0, 4e6, (nz, ny, nx))).cuda()
    T0 = torch.from_numpy(rng.uniform(36.0, 46.0, (nz, ny, nx)).astype(np.float32)).cuda()
    out = []
    for direct in (False, True):
        if direct:
            monkeypatch.setenv("BVF_NO_TMA", "1")
        s = bvf.Solver(nx, ny, nz, 0.5e-3, 5e-8, 5e5, n_sls=2, n_pml=0)
        s.set_materials(torch.from_numpy(index).cuda(), mat)
        r = s.thermal(amp, 0.02, 6, 4, 0.3, T=T0.clone())
        torch.cuda.synchronize()
        monkeypatch.delenv("BVF_NO_TMA", raising=False)
        out.append([t.cpu().numpy() for t in r])
        s.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
    assert np.isfinite(out[0][0]).all()
