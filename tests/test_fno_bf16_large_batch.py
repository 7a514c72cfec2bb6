"""Training batches beyond the tiled mode mix (a block's spectra of all samples
and channels no longer fit its shared memory): the mix and its adjoints then
run one thread per output.  A batch's outputs are its samples', and its
gradient the mean of its parts', up to the scaling of the loss's gradient by 1
/ batch ahead of its BF16 rounding (2^-9 relative, at most 5e-3 through four
rounded products) and the order of float sums."""
import numpy as np
import pytest

from tests import host_cuda

HOST = r"""
F = fno.lib()
dims = fno.FnoDims(3, 64, 2, 2, 16, 1)
n_w = F.bvf_fno_weight_count(ctypes.byref(dims))
N, B = 8 * 6 * 6, 80
t = ctypes.c_void_p()
assert F.bvf_fno_bf16_create(ctypes.byref(t), ctypes.byref(dims), (ctypes.c_float * n_w)(), n_w,
                             8, 6, 6, B) == OK
a, y, g = buf(12 * N * B), buf(4 * N * B), buf(4 * n_w)
loss = ctypes.c_double()
for batch, forward, backward in ((19, "tile", "tile"), (20, "tile", "plain"), (73, "tile", "plain"),
                                 (74, "plain", "plain")):
    launched()
    assert F.bvf_fno_bf16_gradient(t, batch, a, y, None, 0.0, g, ctypes.byref(loss), None) == OK
    names = {n for n, _ in launched()}
    assert ("k_mix_fwd_tile" in names, "k_mix_fwd" in names) == (forward == "tile", forward == "plain")
    assert ("k_mix_bwd_tile" in names, "k_mix_adj" in names) == (backward == "tile", backward == "plain")
"""


def test_batches_that_leave_the_tiles(tmp_path):
    host_cuda.run(HOST, tmp_path)


@pytest.mark.gpu
@pytest.mark.parametrize("batch", [24, 80])
def test_gpu_large_batch_is_the_mean_of_its_parts(batch):
    torch = pytest.importorskip("torch")
    from paper_2301_12727_gb300 import fno, synth
    nx, ny, nz, part = 8, 6, 6, 8
    dims = dict(c_in=3, width=64, modes=2, n_layers=2, hidden=16, c_out=2)
    w = synth.fno_weights(dims, 9)
    a = np.stack([synth.fno_inputs(3, nx, ny, nz, s) for s in range(batch)])
    y = np.random.default_rng(3).standard_normal((batch, nz, ny, nx)).astype(np.float32)
    el = np.linspace(0.1, 0.5, batch).astype(np.float32)
    A, Y, E = (torch.from_numpy(v.astype(np.float32)).cuda() for v in (a, y, el))
    net = fno.Bf16Net(dims, w, (nx, ny, nz), max_batch=batch)
    out = net.forward(A).cpu().numpy().astype(np.float64)
    loss, g = net.gradient(A, Y, el=E, el_weight=0.3)
    g = g.cpu().numpy().astype(np.float64)
    cut = [slice(b, b + part) for b in range(0, batch, part)]
    outs = np.concatenate([net.forward(A[c]).cpu().numpy() for c in cut]).astype(np.float64)
    parts = [net.gradient(A[c].contiguous(), Y[c].contiguous(), el=E[c].contiguous(), el_weight=0.3)
             for c in cut]
    mean = np.mean([p[1].cpu().numpy().astype(np.float64) for p in parts], axis=0)
    net.synchronize()
    net.close()
    assert np.linalg.norm(out - outs) <= 5e-3 * np.linalg.norm(outs)
    assert abs(loss - np.mean([p[0] for p in parts])) <= 1e-5 * abs(loss)
    assert np.linalg.norm(g - mean) <= 5e-3 * np.linalg.norm(mean)
