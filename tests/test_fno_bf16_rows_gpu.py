"""The fused row passes of the BF16 path against the FP64 oracle at the edges
of their tiles: several rows a tile (nx <= 64, a last group with fewer rows),
one tile and a remainder (65, 128, 129, 301), rows too long for the fused
kernel (6600), every width, padded hidden layers, 1 to 16 input and 1 to 8
output channels, two samples.  Relative L2 below 3e-2: the chain of products
with BF16 operands (relative 2^-9 each), as in test_fno_bf16_gpu.py."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,width,m,c_in,hidden,c_out", [
    (17, 11, 13, 16, 4, 1, 20, 1), (32, 9, 9, 32, 4, 9, 128, 2), (40, 11, 9, 32, 3, 8, 64, 8),
    (65, 10, 9, 48, 4, 16, 48, 3), (128, 8, 9, 64, 4, 8, 256, 2), (129, 9, 8, 32, 4, 2, 17, 1),
    (301, 9, 10, 16, 4, 8, 16, 2), (6600, 8, 8, 16, 4, 8, 32, 2)])
def test_forward_matches_oracle_at_tile_edges(nx, ny, nz, width, m, c_in, hidden, c_out):
    torch = pytest.importorskip("torch")
    from oracle import fno as ofno
    from paper_2301_12727_gb300 import fno, synth
    dims = dict(c_in=c_in, width=width, modes=m, n_layers=2, hidden=hidden, c_out=c_out)
    w = synth.fno_weights(dims, nx + width)
    a = np.stack([synth.fno_inputs(c_in, nx, ny, nz, s) for s in (1, 2)])
    net = fno.Bf16Net(dims, w, (nx, ny, nz), max_batch=2)
    got = net.forward(torch.from_numpy(a).cuda()).cpu().numpy()
    net.synchronize()
    net.close()
    for b in range(2):
        ref = ofno.forward(a[b].astype(np.float64), w.astype(np.float64), **dims)
        assert np.linalg.norm(got[b] - ref) <= 3e-2 * np.linalg.norm(ref)
