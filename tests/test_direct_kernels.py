"""The direct acoustic kernels (csrc/bvf_acoustic.cu) run where rows stay
dense and are no multiple of 8 elements, where BVF_NO_TMA asks for them, and
for more than two SLS mechanisms.  Which contexts those are is asserted here,
and the oracle and chunk comparisons of test_parity_gpu.py run on them."""
import pytest

from tests import host_cuda

FAMILIES = r"""
def family(nx, **kw):
    c = context(nx, 12, 12, [WATER], **kw)
    launched()
    assert L.bvf_run_acoustic(c, 1, None, None) == OK
    names = {n for n, _ in launched()}
    L.bvf_destroy(c)
    direct = names == {"k_velocity", "k_stress"}
    assert direct or all("_tma" in n for n in names), names
    return "direct" if direct else "tma"

# rows padded where that adds at most a quarter: 4 ceil8(nx) <= 5 nx
for nx in range(6, 70):
    padded = (nx + 7) // 8 * 8
    want = "tma" if 4 * padded <= 5 * nx else "direct"
    for storage in (0, 1):
        assert family(nx, storage=storage) == want, nx
    for n_sls in (0, 1):
        assert family(nx, n_sls=n_sls) == want, nx
    assert family(nx, n_sls=3) == "direct"
assert [nx for nx in range(6, 40) if family(nx) == "direct"] == [6, 9, 10, 11, 12, 17, 18, 19, 25]
os.environ["BVF_NO_TMA"] = "1"
for nx in (42, 45, 48, 50):
    assert family(nx) == "direct"
"""


def test_which_contexts_run_the_direct_kernels(tmp_path):
    host_cuda.run(FAMILIES, tmp_path)


@pytest.fixture(scope="module")
def bvf():
    import torch
    assert torch.cuda.is_available()
    from paper_2301_12727_gb300 import build
    build.build()
    from paper_2301_12727_gb300 import bvf as m
    return m


def _is_direct(bvf, nx, ny, nz, n_pml):
    s = bvf.Solver(nx, ny, nz, 0.5e-3, 4e-8, 5e5, n_sls=2, n_pml=n_pml)
    for kernel in (1, 2):
        with pytest.raises(bvf.BvfError):
            bvf.bvf_test_withhold_tma(s.ctx, kernel, 3, 64)
    s.close()


@pytest.mark.gpu
@pytest.mark.parametrize("nx,no_tma", [(45, True), (48, True), (12, False), (25, False)])
def test_gpu_random_state_on_the_direct_kernels(bvf, orc, monkeypatch, nx, no_tma):
    """Random state in a heterogeneous medium against the oracle, every array:
    forced at a padded and an aligned width, and at widths that stay dense."""
    from tests import test_parity_gpu as parity
    if no_tma:
        monkeypatch.setenv("BVF_NO_TMA", "1")
    _is_direct(bvf, nx, 38, 29, 5)
    parity.test_gpu_random_state_all_fields(bvf, orc, nx, 38, 29)


@pytest.mark.gpu
@pytest.mark.parametrize("nx,no_tma", [(50, True), (25, False)])
def test_gpu_chunks_on_the_direct_kernels(bvf, monkeypatch, nx, no_tma):
    from tests import test_parity_gpu as parity
    if no_tma:
        monkeypatch.setenv("BVF_NO_TMA", "1")
    _is_direct(bvf, nx, 41, 37, 5)
    parity.test_gpu_zchunk_invariance(bvf, monkeypatch, nx)
