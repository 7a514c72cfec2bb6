"""Grids whose rows are no multiple of 8 voxels run the TMA-fed kernels on
padded rows; their results equal the direct kernels' (BVF_NO_TMA) bit for bit:
every state array, the peak map, amplitude and phase, for odd and even nx, no
or thin CPML slabs, 0 to 2 SLS mechanisms, both storages.  Snapshots keep
dense rows, so one made with padded rows continues in a context without them
and the other way round; what needs nx % 8 == 0 stays refused."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _make(bvf, synth, torch, nx, ny, nz, n_pml, n_sls, storage):
    f0, dx = 5e5, 0.5e-3
    rng = np.random.default_rng(nx * ny + nz)
    table = np.array([synth.water_row(f0), synth.bone_row_from_hu(900.0, f0),
                      synth.bone_row_from_hu(1900.0, f0)])
    if n_sls == 0:
        table[:, 3:5] = 0.0
    dt, _ = synth.choose_dt(dx, table[:, 1].max(), f0)
    s = bvf.Solver(nx, ny, nz, dx, dt, f0, n_sls=n_sls, n_pml=n_pml, storage=storage)
    s.set_materials(torch.from_numpy(rng.integers(0, 3, (nz, ny, nx)).astype(np.uint8)).cuda(), table)
    s.set_source(torch.from_numpy(rng.standard_normal((ny, nx, 2)).astype(np.float32) * 1e4).cuda(),
                 nz // 2, 1500.0, bvf.BVF_ENV_RAMP_CW)
    v = rng.standard_normal((nz, ny, nx)).astype(np.float32)
    s.set_field("sxx", v * 1e3)
    s.set_field("vy", v * 1e-3)
    if n_sls:
        s.set_field(s.memory_id(n_sls - 1, 3), v * 1e9)
    return s


def _outputs(s):
    out = [s.field(f).cpu().numpy() for f in range(9 + 6 * s.n_sls)]
    return out + [s.peak().cpu().numpy(), s.pressure().cpu().numpy()] + \
        [t.cpu().numpy() for t in s.amp_phase()]


@pytest.mark.parametrize("nx,ny,nz,n_pml,n_sls", [
    (29, 13, 11, 0, 2), (33, 18, 17, 3, 2), (37, 24, 20, 4, 1), (63, 33, 19, 4, 0),
    (65, 40, 37, 6, 2), (98, 21, 18, 4, 2), (100, 17, 30, 4, 2), (197, 41, 26, 8, 2)])
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_padded_rows_match_direct_kernels_bitwise(nx, ny, nz, n_pml, n_sls, storage, monkeypatch):
    torch = pytest.importorskip("torch")
    from paper_2301_12727_gb300 import bvf, synth
    got, snaps = [], []
    for direct in (False, True):
        if direct:
            monkeypatch.setenv("BVF_NO_TMA", "1")
        s = _make(bvf, synth, torch, nx, ny, nz, n_pml, n_sls, storage)
        monkeypatch.delenv("BVF_NO_TMA", raising=False)
        s.run(12, peak_from=2, dft_start=6, dft_steps=20)
        s.synchronize()
        snaps.append(s.save_state())
        s.run(9, peak_from=2, dft_start=6, dft_steps=20)
        s.synchronize()
        got.append((s, _outputs(s)))
    for a, b in zip(got[0][1], got[1][1]):
        assert np.array_equal(a, b)
    # each context continues from the other's snapshot
    for (s, ref), snap in zip(got, reversed(snaps)):
        s.load_state(snap)
        s.run(9, peak_from=2, dft_start=6, dft_steps=20)
        s.synchronize()
        for a, b in zip(_outputs(s), ref):
            assert np.array_equal(a, b)
        s.close()


def test_what_needs_whole_rows_stays_refused():
    torch = pytest.importorskip("torch")
    from paper_2301_12727_gb300 import bvf, synth
    s = _make(bvf, synth, torch, 98, 21, 18, 4, 2, "f32")
    with pytest.raises(bvf.BvfError):
        bvf.Batch([s])
    for kernel in (1, 2, 3):
        with pytest.raises(bvf.BvfError):
            bvf.bvf_test_withhold_copy(s.ctx, kernel, 3, 64)
    s.close()
