"""The z-chunks the TMA-fed kernels choose by grid size change no bit: at the
edges of the rules (one plane a block, two, the caps of 5 and 6, a last chunk
of one plane) every output equals that of a single chunk over all planes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,n_pml", [(16, 16, 13, 0), (64, 64, 65, 4), (96, 90, 95, 4),
                                            (256, 160, 37, 4)])
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_default_chunks_agree_with_one_chunk_bitwise(nx, ny, nz, n_pml, storage):
    torch = pytest.importorskip("torch")
    from paper_2301_12727_gb300 import bvf, synth
    f0, dx = 5e5, 0.5e-3
    rng = np.random.default_rng(nx + nz)
    table = np.array([synth.water_row(f0), synth.bone_row_from_hu(900.0, f0),
                      synth.bone_row_from_hu(1900.0, f0)])
    dt, M = synth.choose_dt(dx, table[:, 1].max(), f0)
    index = torch.from_numpy(rng.integers(0, 3, (nz, ny, nx)).astype(np.uint8)).cuda()
    plane = torch.from_numpy(rng.standard_normal((ny, nx, 2)).astype(np.float32) * 1e4).cuda()
    got = []
    for kchunk in (0, nz):
        s = bvf.Solver(nx, ny, nz, dx, dt, f0, n_pml=n_pml, storage=storage)
        s.set_materials(index, table)
        s.set_source(plane, nz // 2, 1500.0, bvf.BVF_ENV_RAMP_CW)
        s.set_tile(kchunk=kchunk)
        s.run(23, peak_from=2, dft_start=10, dft_steps=12)
        s.synchronize()
        out = [s.field(f).cpu().numpy() for f in range(9 + 6 * 2)]
        out += [s.peak().cpu().numpy()] + [t.cpu().numpy() for t in s.amp_phase()]
        got.append(out)
        s.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    assert np.abs(got[0][3]).max() > 0.0
