"""The persistent sweep (bvf_batch_run) takes its contexts' material tables as
they are at the run, not as they were when the batch was made."""
import numpy as np
import pytest

from tests import host_cuda

HOST = r"""
NX, NY, NZ = 32, 16, 16
N = NX * NY * NZ
for storage in (0, 1):
    ctxs = [context(NX, NY, NZ, [WATER, BONE], storage=storage) for _ in range(2)]
    steps = (ctypes.c_int * 2)(2, 3)

    def batch():
        b = ctypes.c_void_p()
        assert L.bvf_batch_create((ctypes.c_void_p * 2)(*ctxs), 2, ctypes.byref(b)) == OK
        return b

    def shared_memory(b, graph_steps):
        launched()
        assert L.bvf_batch_run(b, steps, None, 0, graph_steps, None) == OK
        return {s for n, s in launched() if n == "k_stress_batch"}

    old = batch()
    short = shared_memory(old, 0)
    materials(ctxs[1], N, [WATER, BONE] * 20)
    # a batch made now asks for 38 rows of 32 bytes more; so does the old one
    want = shared_memory(batch(), 0)
    assert want == {max(short) + 38 * 32}
    assert shared_memory(old, 0) == want and shared_memory(old, 2) == want
    materials(ctxs[1], N, [WATER])
    assert shared_memory(old, 0) == short
    # an index beyond the table leaves nothing to run
    fake.fake_read_u32(7)
    assert L.bvf_set_materials(ctxs[0], buf(N), bvf.material_array([WATER]), 1) != OK
    fake.fake_read_u32(-1)
    launched()
    assert L.bvf_batch_run(old, steps, None, 0, 0, None) == ARG
    assert not launched()
"""


def test_shared_memory_follows_the_tables(tmp_path):
    host_cuda.run(HOST, tmp_path)


LIMITS = r"""
# 240 rows need more than the 48 KB every kernel may use: a batch of short
# tables made afterwards leaves the long one's launches as they were
NX, NY, NZ = 32, 16, 16
steps = (ctypes.c_int * 1)(2)

def batch(rows):
    c = context(NX, NY, NZ, [WATER] * rows)
    b = ctypes.c_void_p()
    assert L.bvf_batch_create((ctypes.c_void_p * 1)(c), 1, ctypes.byref(b)) == OK
    return b

long = batch(240)
assert L.bvf_batch_run(long, steps, None, 0, 0, None) == OK
assert max(s for n, s in launched()) > 48 * 1024
short = batch(2)
for b in (short, long, short):
    assert L.bvf_batch_run(b, steps, None, 0, 0, None) == OK, L.bvf_last_error(None)
"""


def test_a_batch_of_short_tables_leaves_the_limit_of_a_long_one(tmp_path):
    host_cuda.run(LIMITS, tmp_path)


@pytest.mark.gpu
def test_gpu_longer_table_after_the_batch_was_made():
    """96 rows set after the batch was made from 2: the sweep equals
    bvf_run_acoustic bit for bit."""
    torch = pytest.importorskip("torch")
    from paper_2301_12727_gb300 import bvf, synth
    f0, dx, n = 5e5, 0.5e-3, 32
    rng = np.random.default_rng(4)
    rows = [synth.water_row(f0)] + [synth.bone_row_from_hu(h, f0) for h in np.linspace(500, 1900, 95)]
    dt, _ = synth.choose_dt(dx, max(r[1] for r in rows), f0)
    plane = torch.from_numpy(rng.standard_normal((n, n, 2)).astype(np.float32) * 1e4).cuda()
    s = [bvf.Solver(n, n, n, dx, dt, f0, n_sls=2, n_pml=4) for _ in range(2)]
    for t in s:
        t.set_materials(torch.zeros((n, n, n), dtype=torch.uint8, device="cuda"), rows[:2])
        t.set_source(plane, 12, 1500.0, bvf.BVF_ENV_RAMP_CW)
    batch = bvf.Batch(s[:1])
    index = torch.from_numpy(rng.integers(0, 96, (n, n, n)).astype(np.uint8)).cuda()
    for t in s:
        t.set_materials(index, rows)
    batch.run(25, caps=[(0, 0, 0)], graph_steps=5)
    s[1].run(25, peak_from=0)
    out = []
    for t in s:
        t.synchronize()
        out.append([t.field(f).cpu().numpy() for f in range(21)] + [t.peak().cpu().numpy()])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    batch.close()
    for t in s:
        t.close()
