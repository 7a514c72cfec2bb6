"""The pairwise, class-coded BHTE step equals the direct kernel (BVF_NO_TMA) bit
for bit: materials that share a conductivity and materials that all differ (up
to 200 of them), grids with ragged y tiles, a single tile and thin z, step counts
on both sides of the 32-step flush of the dose partial, a source that is never
on, and an infinite source entry (kept in the sum also while the source is
off)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,n_mat,shared,n_on,n_off,bad", [
    (8, 3, 3, 2, False, 5, 4, False), (32, 16, 5, 4, True, 31, 1, False),
    (40, 17, 9, 5, False, 0, 33, False), (64, 33, 31, 200, False, 20, 13, False),
    (72, 19, 21, 200, True, 33, 32, False), (96, 41, 12, 3, True, 3, 62, True)])
def test_matches_direct_kernel_bitwise(nx, ny, nz, n_mat, shared, n_on, n_off, bad, monkeypatch):
    torch = pytest.importorskip("torch")
    from paper_2301_12727_gb300 import bvf
    rng = np.random.default_rng(nx + n_mat)
    # rho, cL, cS, alphaL, alphaS, k, c_th, perf, heat_frac
    mat = np.stack([rng.uniform(900, 1900, n_mat), rng.uniform(1450, 2900, n_mat), np.zeros(n_mat),
                    rng.uniform(1, 80, n_mat), np.zeros(n_mat),
                    rng.choice([0.3, 0.5], n_mat) if shared else rng.uniform(0.2, 0.7, n_mat),
                    rng.uniform(1300, 4200, n_mat), rng.uniform(0, 0.01, n_mat),
                    rng.uniform(0, 1, n_mat)], axis=1)
    index = rng.integers(0, n_mat, (nz, ny, nx)).astype(np.uint8)
    index[:, :, nx // 2:] = n_mat - 1                  # a homogeneous half
    amp = rng.uniform(0.0, 4e6, (nz, ny, nx))
    if bad:
        amp[nz // 2, ny // 2, 5] = np.inf
    T0 = torch.from_numpy(rng.uniform(36.0, 46.0, (nz, ny, nx)).astype(np.float32)).cuda()
    out = []
    for direct in (False, True):
        if direct:
            monkeypatch.setenv("BVF_NO_TMA", "1")
        s = bvf.Solver(nx, ny, nz, 0.5e-3, 5e-8, 5e5, n_sls=2, n_pml=0)
        s.set_materials(torch.from_numpy(index).cuda(), mat)
        r = s.thermal(torch.from_numpy(amp).cuda(), 0.02, n_on, n_off, 0.3, T=T0.clone())
        torch.cuda.synchronize()
        monkeypatch.delenv("BVF_NO_TMA", raising=False)
        out.append([t.cpu().numpy() for t in r])
        s.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
    if not bad:
        assert np.isfinite(out[0][0]).all() and (out[0][0] != T0.cpu().numpy()).any()
