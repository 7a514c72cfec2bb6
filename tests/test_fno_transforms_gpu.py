"""The folded y and z transforms and the projection's output counts against
the FP64 oracle: the smallest grids of a mode count (2m samples, the halves
meet in the middle), odd and even lengths, the mode counts at the edges of
the kernels' class bounds (8, 9, 12, 13, 16), 1 to 8 outputs.  Within 2e-5 of
the largest |ref|, the FP32 bound of test_fno_gpu.py."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,nx,ny,nz,width,c_out", [
    (1, 3, 2, 2, 16, 1), (1, 2, 3, 5, 16, 2), (4, 9, 8, 9, 32, 3), (8, 17, 17, 16, 16, 4),
    (9, 20, 18, 19, 16, 5), (12, 24, 25, 24, 32, 6), (13, 27, 26, 27, 16, 7),
    (16, 33, 33, 32, 16, 8), (5, 12, 41, 64, 48, 2)])
def test_inference_matches_oracle(m, nx, ny, nz, width, c_out):
    torch = pytest.importorskip("torch")
    from oracle import fno as ofno
    from paper_2301_12727_gb300 import fno, synth
    dims = dict(c_in=3, width=width, modes=m, n_layers=2, hidden=40, c_out=c_out)
    w = synth.fno_weights(dims, 10 * m + c_out)
    a = synth.fno_inputs(3, nx, ny, nz, m)
    net = fno.Surrogate(dims, w)
    got = net(torch.from_numpy(a).cuda()).cpu().numpy()
    net.synchronize()
    net.close()
    ref = ofno.forward(a.astype(np.float64), w.astype(np.float64), **dims)
    assert np.abs(got - ref).max() <= 2e-5 * np.abs(ref).max()
