"""Time-outs of the TMA-fed acoustic kernels at the chunk lengths they run at
and on padded rows: a copy that is withheld (nothing in flight) ends in an
error that bvf_synchronize reports, and the context runs on after a reset."""
import numpy as np
import pytest

from tests import host_cuda

HOST = r"""
# the hook takes a context where its kernel is the TMA-fed one, and the armed
# step is launched as any other
for nx, tma in ((48, True), (45, True), (50, True), (41, True), (9, False), (12, False)):
    for storage in (0, 1):
        c = context(nx, 40, 33, [WATER, BONE], storage=storage)
        launches()
        assert L.bvf_run_acoustic(c, 1, None, None) == OK
        want = launches()
        assert any("_tma" in n for n, _, _ in want) == tma
        for kernel in (1, 2):
            assert L.bvf_test_withhold_tma(c, kernel, 3, 64) == (OK if tma else ARG), nx
            assert L.bvf_run_acoustic(c, 1, None, None) == OK
            assert launches() == want, (nx, kernel)
            assert L.bvf_test_withhold_copy(c, kernel, 3, 64) == (OK if nx % 8 == 0 else ARG)
            assert L.bvf_test_withhold_tma(c, 0, 0, 0) == OK
            for bad in ((4, 3), (kernel, -1), (kernel, 33)):
                assert L.bvf_test_withhold_tma(c, *bad, 64) == ARG
        assert L.bvf_test_withhold_tma(c, 3, 3, 64) == (OK if nx % 8 == 0 else ARG)
        L.bvf_test_withhold_tma(c, 0, 0, 0)
"""


def test_the_hook_follows_the_kernels(tmp_path):
    host_cuda.run(HOST, tmp_path)


@pytest.mark.gpu
@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("nx", [45, 50, 48])
def test_gpu_withheld_copies_time_out_and_the_context_recovers(nx, storage):
    """The plane whose copies are withheld (plane + 1 for the velocity, + 2 for
    the stress kernel) begins a z-chunk, lies inside one or ends it, for chunks
    of 1, 2 and 6 planes and the default ones."""
    torch = pytest.importorskip("torch")
    from paper_2301_12727_gb300 import bvf, synth
    c = synth.skull_case(nx, 40, 33, dx=0.5e-3, n_steps=30, aperture=16e-3, roc=15e-3, n_pml=4)

    def solver():
        s = bvf.Solver(c.nx, c.ny, c.nz, c.dx, c.dt, c.f0, n_sls=2, n_pml=c.n_pml, storage=storage)
        s.set_materials(c.index, c.materials)
        s.set_source(bvf.rs_plane(c.bowl, c.nx, c.ny, c.dx, c.k_src * c.dx, c.f0), c.k_src, c.c0,
                     c.envelope)
        return s

    def outputs(s):
        s.run(8, peak_from=0)
        s.synchronize()
        return [s.field(f).cpu().numpy() for f in range(21)] + [s.peak().cpu().numpy()]

    s, ref = solver(), solver()
    want = outputs(ref)
    assert want[-1].max() > 0
    for kernel, ahead in ((1, 1), (2, 2)):
        for kchunk, planes in ((1, (12, 32)), (2, (12, 13)), (6, (12, 14, 17)), (0, (12, 13))):
            s.set_tile(0, 0, kchunk)
            for plane in planes:
                bvf.bvf_test_withhold_tma(s.ctx, kernel, plane - ahead, 4096)
                s.run(2, peak_from=0)
                with pytest.raises(bvf.BvfError) as ei:
                    s.synchronize()
                assert ei.value.code == bvf.BVF_E_CUDA and "wait limit" in str(ei.value)
                s.reset()
                for a, b in zip(outputs(s), want):
                    assert np.array_equal(a, b), (kernel, kchunk, plane)
                s.reset()
    s.close()
    ref.close()
    torch.cuda.synchronize()
