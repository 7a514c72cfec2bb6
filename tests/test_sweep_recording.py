"""bvf_batch_run_graph replays its recording only for what it was recorded
for: the recorded launches hold the sources' plane, speed, envelope and cycle
count and the length of the material tables by value."""
import numpy as np
import pytest

from tests import host_cuda

HOST = r"""
TABLE = [WATER, BONE]
NX, NY, NZ = 32, 16, 16
N = NX * NY * NZ
ctxs = [context(NX, NY, NZ, TABLE) for _ in range(2)]
plane = buf(8 * NX * NY)

def source(c, k=3, c0=1500.0, env=bvf.BVF_ENV_RAMP_CW, cycles=0):
    assert L.bvf_set_source(c, k, plane, c0, env, cycles, None) == OK

for c in ctxs:
    source(c)
b = ctypes.c_void_p()
assert L.bvf_batch_create((ctypes.c_void_p * 2)(*ctxs), 2, ctypes.byref(b)) == OK
steps = (ctypes.c_int * 2)(4, 5)

def sweep():
    # recordings made by one sweep from the start
    for c in ctxs:
        assert L.bvf_reset(c, None) == OK
    before = fake.fake_instantiated()
    rc = L.bvf_batch_run_graph(b, steps, None, 2, None)
    return rc, fake.fake_instantiated() - before

assert sweep() == (OK, 1)
assert sweep() == (OK, 0)
c = ctxs[1]
for change in (dict(k=5), dict(c0=1490.0), dict(env=bvf.BVF_ENV_BURST, cycles=3),
               dict(env=bvf.BVF_ENV_BURST, cycles=4), dict(env=bvf.BVF_ENV_NONE), dict()):
    source(c, **change)
    assert sweep() == (OK, 1), change
    source(c, **change)
    assert sweep() == (OK, 0), change
# a longer table: shared memory and table strides of the launches change
materials(c, N, TABLE + [BONE])
assert sweep() == (OK, 1)
materials(c, N, TABLE + [WATER])
assert sweep() == (OK, 0)
# an index beyond the table: refused, and so is a replay
fake.fake_read_u32(7)
assert L.bvf_set_materials(c, buf(N), bvf.material_array(TABLE + [WATER]), 3) != OK
fake.fake_read_u32(-1)
assert sweep() == (ARG, 0)
materials(c, N, TABLE + [WATER])
assert sweep()[0] == OK
"""


def test_what_the_launches_hold_is_recorded_anew(tmp_path):
    host_cuda.run(HOST, tmp_path)


@pytest.mark.gpu
def test_gpu_replay_after_a_new_source_matches_single_runs_bitwise():
    """A sweep is recorded, then one context's source changes plane, speed and
    envelope, then its materials grow by a row: after each change the sweep
    equals bvf_run_acoustic on that context bit for bit, and differs from the
    sweep before."""
    torch = pytest.importorskip("torch")
    from paper_2301_12727_gb300 import bvf, synth
    f0, dx, n, steps = 5e5, 0.5e-3, 32, 40
    rng = np.random.default_rng(3)
    rows = [synth.water_row(f0), synth.bone_row_from_hu(900.0, f0), synth.bone_row_from_hu(1900.0, f0)]
    dt, _ = synth.choose_dt(dx, max(r[1] for r in rows), f0)
    index = torch.from_numpy(rng.integers(0, 2, (n, n, n)).astype(np.uint8)).cuda()
    longer = index + (torch.arange(n, device="cuda") > 20).to(torch.uint8)[:, None, None]
    plane = torch.from_numpy(rng.standard_normal((n, n, 2)).astype(np.float32) * 1e4).cuda()

    def solver():
        return bvf.Solver(n, n, n, dx, dt, f0, n_sls=2, n_pml=4)

    def outputs(s):
        return [s.field(f).cpu().numpy() for f in range(9)] + [s.peak().cpu().numpy()]

    changes = [(index, rows[:2], 10, 1500.0, bvf.BVF_ENV_RAMP_CW, 0),
               (index, rows[:2], 17, 1480.0, bvf.BVF_ENV_BURST, 2),
               (longer, rows, 17, 1480.0, bvf.BVF_ENV_BURST, 2),
               (longer, rows, 17, 1480.0, bvf.BVF_ENV_NONE, 0)]
    s = [solver() for _ in range(2)]
    s[0].set_materials(index, rows[:2])
    s[0].set_source(plane, 12, 1500.0, bvf.BVF_ENV_RAMP_CW)
    s[1].set_materials(index, rows[:2])
    batch, last = bvf.Batch(s), None
    for idx, table, k, c0, env, cycles in changes:
        ref = solver()
        for t in (s[1], ref):
            t.set_materials(idx, table)
            t.set_source(plane, k, c0, env, cycles)
            t.reset()
        s[0].reset()
        batch.run_graph(steps, caps=[(0, 0, 0)] * 2, n_branches=2)
        ref.run(steps, peak_from=0)
        for t in s + [ref]:
            t.synchronize()
        got = outputs(s[1])
        for a, b in zip(got, outputs(ref)):
            assert np.array_equal(a, b)
        assert last is None or not np.array_equal(got[-1], last)
        last = got[-1]
        ref.close()
    batch.close()
    for t in s:
        t.close()
