"""The Rayleigh-Sommerfeld sums over elements: the kernel with one thread per
point where few elements (or a large plane) would leave most of eight idle, the
one with eight threads elsewhere, and the same bits from both."""
import numpy as np
import pytest

from tests import host_cuda

HOST = r"""
def kernel(n, ne):
    el = (ctypes.c_double * (6 * ne))(*([0.0, 0.0, -1.0, 1e-6, 1.0, 0.0] * ne))
    launched()
    assert L.bvf_rs_elements(el, ne, 1e5, 1500.0, n, n, 5e-4, 0.0, 5e5, buf(8 * n * n), None) == OK
    (name, _), = launched()
    return name

L.bvf_rs_elements.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_int,
                              ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_double,
                              ctypes.c_void_p, ctypes.c_void_p]
# (points per side, elements, eight threads a point measured faster by)
for n, ne, split in ((8, 1, False), (64, 256, False), (64, 512, True), (64, 6150, True),
                     (160, 256, False), (190, 600, False), (190, 1024, True), (240, 300, False),
                     (240, 1024, True), (240, 6150, True), (512, 256, False), (512, 768, False),
                     (512, 1500, True), (700, 900, False), (1024, 256, False), (1024, 1024, False)):
    assert kernel(n, ne) == ("k_rs" if split else "k_rs_point"), (n, ne)
"""


def test_which_kernel_sums(tmp_path):
    host_cuda.run(HOST, tmp_path)


@pytest.mark.gpu
@pytest.mark.parametrize("ne", [1, 31, 255, 256, 257, 511, 700, 2047, 2049, 2300])
def test_gpu_both_kernels_sum_the_same_bits(ne):
    """The points of a small plane, summed with eight threads each from about
    400 elements on, are the first rows of a plane so large that one thread
    sums each; unweighted sums are weighted ones with weight 1."""
    pytest.importorskip("torch")
    from paper_2301_12727_gb300 import bvf
    rng = np.random.default_rng(ne)
    f0, c0, dx, nx = 5e5, 1500.0, 5e-4, 61
    el = np.zeros((ne, 6))
    el[:, :2] = rng.random((ne, 2)) * nx * dx
    el[:, 2] = -0.01 - 0.02 * rng.random(ne)
    el[:, 3] = 1e-6 * (1 + rng.random(ne))
    el[:, 4:] = rng.standard_normal((ne, 2))
    small = bvf.bvf_rs_elements(el, 1e5, c0, nx, 7, dx, 0.0, f0).cpu().numpy()
    large = bvf.bvf_rs_elements(el, 1e5, c0, nx, 20011, dx, 0.0, f0)[:7].cpu().numpy()
    assert np.array_equal(small, large)
    # the sum itself, in FP64
    x, y = np.meshgrid(np.arange(nx) * dx, np.arange(7) * dx)
    r = np.sqrt((x[..., None] - el[:, 0]) ** 2 + (y[..., None] - el[:, 1]) ** 2 + el[:, 2] ** 2)
    k = 2 * np.pi * f0 / c0
    ref = (1j * k * 1e5 / (2 * np.pi) *
           (el[:, 3] * (el[:, 4] + 1j * el[:, 5]) * np.exp(-1j * k * r) / r).sum(-1))
    got = small[..., 0] + 1j * small[..., 1]
    # of the sum of the terms' magnitudes: k r / pi of up to 30 rounds three
    # times (1.7e-5 rad), the coordinates once (2^-24 of 0.04 m, 5e-6 rad), and
    # a tile's 256 additions err by 256 * 2^-24 = 1.5e-5 at most
    terms = el[:, 3] * np.hypot(el[:, 4], el[:, 5]) / r
    assert (np.abs(got - ref) <= 4e-5 * terms.sum(-1) * k * 1e5 / (2 * np.pi)).all()
