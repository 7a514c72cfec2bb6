"""The forward x transform fed by TMA against the FP64 oracle at its edges:
the shortest rows it takes (32: a chunk of padding), rows with a partial last
chunk (36, 100, 132, 700), rows that are no whole 16-byte pieces and take the
other kernel (33, 66), both operand widths (2m <= 16, 2m <= 32), row counts
that are no multiple of 128, and long rows with one block per SM or too long
for the resident operand (700, m = 9).  FP32 within 2e-5 of the largest |ref|
(the bound of test_fno_gpu.py), BF16 within 3e-2 in relative L2 (that of
test_fno_bf16_gpu.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,m", [
    (32, 9, 8, 4), (33, 9, 8, 4), (36, 9, 11, 4), (64, 18, 19, 9), (66, 18, 18, 9), (100, 16, 17, 8),
    (132, 8, 9, 4), (700, 9, 8, 4), (700, 18, 18, 9)])
@pytest.mark.parametrize("bf16", [False, True])
def test_matches_oracle(nx, ny, nz, m, bf16):
    torch = pytest.importorskip("torch")
    from oracle import fno as ofno
    from paper_2301_12727_gb300 import fno, synth
    dims = dict(c_in=3, width=16, modes=m, n_layers=2, hidden=24, c_out=2)
    w = synth.fno_weights(dims, nx + m)
    a = synth.fno_inputs(3, nx, ny, nz, m)
    x = torch.from_numpy(a).cuda()
    ref = ofno.forward(a.astype(np.float64), w.astype(np.float64), **dims)
    if bf16:
        net = fno.Bf16Net(dims, w, (nx, ny, nz))
        got = net.forward(x[None]).cpu().numpy()[0]
    else:
        net = fno.Surrogate(dims, w)
        got = net(x).cpu().numpy()
    net.synchronize()
    net.close()
    if bf16:
        assert np.linalg.norm(got - ref) <= 3e-2 * np.linalg.norm(ref)
    else:
        assert np.abs(got - ref).max() <= 2e-5 * np.abs(ref).max()


def test_long_rows_of_a_wide_layer():
    """Width 64, 16 modes, rows of 300: the layer output holds one x tile's
    table and so takes rows that a table for the whole row did not fit."""
    torch = pytest.importorskip("torch")
    from oracle import fno as ofno
    from paper_2301_12727_gb300 import fno, synth
    dims = dict(c_in=3, width=64, modes=16, n_layers=2, hidden=24, c_out=1)
    w = synth.fno_weights(dims, 5)
    a = synth.fno_inputs(3, 300, 32, 33, 6)
    net = fno.Surrogate(dims, w)
    got = net(torch.from_numpy(a).cuda()).cpu().numpy()
    net.synchronize()
    net.close()
    ref = ofno.forward(a.astype(np.float64), w.astype(np.float64), **dims)
    assert np.abs(got - ref).max() <= 2e-5 * np.abs(ref).max()
