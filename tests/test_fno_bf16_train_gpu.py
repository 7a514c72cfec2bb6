"""The training pass of the BF16 path at the edges of its tiles: voxel counts
that are no multiple of 128, every width, hidden layers that need padding, 1 to
8 outputs, batches of 1, 3 and 5.  The gradient of a batch is the mean of its
samples' gradients: both run the same products on the same roundings, up to
the scaling of the loss's gradient by 1 / batch ahead of its BF16 rounding
(2^-9 relative, at most 5e-3 through four rounded products) and the order of
float sums."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,width,m,c_in,hidden,c_out,batch", [
    (17, 11, 13, 16, 4, 1, 20, 1, 3), (32, 12, 9, 32, 4, 9, 128, 2, 5),
    (65, 10, 9, 48, 4, 8, 17, 8, 3), (40, 9, 11, 64, 3, 4, 256, 2, 5), (24, 9, 8, 16, 3, 8, 16, 3, 1)])
def test_batch_gradient_is_the_mean(nx, ny, nz, width, m, c_in, hidden, c_out, batch):
    torch = pytest.importorskip("torch")
    from paper_2301_12727_gb300 import fno, synth
    dims = dict(c_in=c_in, width=width, modes=m, n_layers=2, hidden=hidden, c_out=c_out)
    w = synth.fno_weights(dims, nx + width)
    a = np.stack([synth.fno_inputs(c_in, nx, ny, nz, s) for s in range(batch)])
    y = np.random.default_rng(3).standard_normal((batch, nz, ny, nx)).astype(np.float32)
    el = np.linspace(0.1, 0.5, batch).astype(np.float32)
    A, Y, E = (torch.from_numpy(v).cuda() for v in (a, y, el))
    net = fno.Bf16Net(dims, w, (nx, ny, nz), max_batch=batch)
    loss, g = net.gradient(A, Y, el=E, el_weight=0.3)
    g = g.cpu().numpy().astype(np.float64)
    one = [net.gradient(A[b:b + 1], Y[b:b + 1], el=E[b:b + 1], el_weight=0.3) for b in range(batch)]
    net.close()
    mean = np.mean([o[1].cpu().numpy().astype(np.float64) for o in one], axis=0)
    assert abs(loss - np.mean([o[0] for o in one])) <= 1e-5 * abs(loss)
    assert np.linalg.norm(g - mean) <= 5e-3 * np.linalg.norm(mean)


@pytest.mark.parametrize("grid,width,hidden,c_in,c_out,batch", [
    ((8, 7, 5), 16, 20, 3, 1, 2), ((9, 7, 5), 32, 16, 3, 2, 2), ((12, 11, 9), 64, 64, 16, 2, 1),
    ((8, 6, 6), 32, 128, 4, 8, 3), ((10, 10, 8), 64, 256, 4, 2, 2)])
def test_gradient_matches_oracle_along_itself(grid, width, hidden, c_in, c_out, batch):
    """Every parameter group's gradient g: the FP64 oracle's derivative along
    g / |g| is |g| (within 5e-2, the bound of test_fno_bf16_gpu.py), for all
    row counts of the weight gradients (up to 64, 128, 192 and 384 rows), two
    row tiles, and volumes that are no whole 16-byte pieces."""
    torch = pytest.importorskip("torch")
    from oracle import fno as ofno
    from paper_2301_12727_gb300 import fno, synth
    from tests.test_fno_bf16_gpu import groups, oracle_loss
    nx, ny, nz = grid
    dims = dict(c_in=c_in, width=width, modes=2, n_layers=2, hidden=hidden, c_out=c_out)
    w = synth.fno_weights(dims, nx + hidden)
    a = np.stack([synth.fno_inputs(c_in, nx, ny, nz, s) for s in range(batch)])
    y = np.random.default_rng(7).standard_normal((batch, nz, ny, nx))
    el = np.linspace(0.2, 0.6, batch)
    A, Y, E = (torch.from_numpy(v.astype(np.float32)).cuda() for v in (a, y, el))
    net = fno.Bf16Net(dims, w, grid, max_batch=batch)
    loss, g = net.gradient(A, Y, el=E, el_weight=2.0)
    g = g.cpu().numpy().astype(np.float64)
    net.close()
    w64 = w.astype(np.float64)
    eps = 1e-3
    for name, start, n in groups(dims):
        norm = np.linalg.norm(g[start:start + n])
        assert norm > 0.0, name
        step = np.zeros_like(w64)
        step[start:start + n] = eps * g[start:start + n] / norm
        fd = (oracle_loss(ofno, a, w64 + step, dims, y, el, 2.0) -
              oracle_loss(ofno, a, w64 - step, dims, y, el, 2.0)) / (2 * eps)
        assert abs(fd - norm) <= 5e-2 * norm, (name, fd, norm)
