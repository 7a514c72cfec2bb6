"""Copies between a context's padded rows and dense arrays: snapshots, fields,
the peak map, the source plane and the padded index, at row lengths around the
128 elements a warp takes at a time, and with snapshot buffers that start on
any byte."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,n_sls,storage", [
    (7, 5, 4, 2, "f32"), (29, 9, 7, 1, "f16"), (98, 12, 9, 2, "f16"), (127, 6, 5, 0, "f32"),
    (129, 7, 6, 1, "f32"), (257, 6, 5, 2, "f16")])
def test_gpu_snapshots_and_fields_of_padded_rows(nx, ny, nz, n_sls, storage):
    torch = pytest.importorskip("torch")
    from paper_2301_12727_gb300 import bvf, synth
    f0, dx = 5e5, 0.5e-3
    rng = np.random.default_rng(nx)
    table = np.array([synth.water_row(f0), synth.bone_row_from_hu(1200.0, f0)])
    if n_sls == 0:
        table[:, 3:5] = 0.0
    dt, _ = synth.choose_dt(dx, table[:, 1].max(), f0)
    s, t = (bvf.Solver(nx, ny, nz, dx, dt, f0, n_sls=n_sls, n_pml=1, storage=storage) for _ in range(2))
    bvf.bvf_test_withhold_tma(s.ctx, 1, 0, 64)               # padded rows: the TMA-fed kernels
    bvf.bvf_test_withhold_tma(s.ctx, 0, 0, 0)
    index = torch.from_numpy(rng.integers(0, 2, (nz, ny, nx)).astype(np.uint8)).cuda()
    plane = torch.from_numpy(rng.standard_normal(ny * nx * 2 + 1).astype(np.float32) * 1e4).cuda()
    for c in (s, t):
        c.set_materials(index, table)
    # a source plane that starts on 4 bytes, not 8
    src = ctypes.c_void_p(plane.data_ptr() + 4)
    bvf._check(bvf.lib().bvf_set_source(s.ctx, nz // 2, src, 1500.0, bvf.BVF_ENV_RAMP_CW, 0, None), s.ctx)
    for f in range(9 + 6 * n_sls):
        v = torch.from_numpy(rng.standard_normal((nz, ny, nx)).astype(np.float32)).cuda()
        s.set_field(f, v)
        if storage == "f32":
            assert torch.equal(s.field(f), v)
    s.run(3, peak_from=0, dft_start=1, dft_steps=3)
    s.synchronize()
    want = [s.field(f) for f in range(9 + 6 * n_sls)] + [s.peak(), *s.amp_phase()]
    n = bvf.bvf_state_bytes(s.ctx)
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    big = torch.empty(n + 16, dtype=torch.uint8, device="cuda")
    for off in (0, 1, 2, 4, 8):
        big.fill_(0xA5)
        p = ctypes.c_void_p(big.data_ptr() + off)
        bvf._check(bvf.lib().bvf_state_save(s.ctx, p, n, stream), s.ctx)
        torch.cuda.synchronize()
        assert (big[:off] == 0xA5).all() and (big[off + n:] == 0xA5).all()
        t.reset()
        bvf._check(bvf.lib().bvf_state_load(t.ctx, p, n, stream), t.ctx)
        got = [t.field(f) for f in range(9 + 6 * n_sls)] + [t.peak(), *t.amp_phase()]
        for a, b in zip(got, want):
            assert torch.equal(a, b), off
    s.close()
    t.close()
