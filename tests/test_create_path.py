"""What bvf_create decides on the host: the layout of a context's rows, the
kernels that run on it, and what it leaves behind."""
from tests import host_cuda

PENDING = r"""
# an error that is pending when a context is made is the caller's
for nx in (48, 41, 45, 9):
    fake.fake_set_pending(1)
    rc, c = create(nx)
    assert rc == OK and fake.fake_pending() == 1, nx
    L.bvf_destroy(c)
    fake.fake_set_pending(0)
"""


def test_a_pending_error_of_the_caller_stays(tmp_path):
    host_cuda.run(PENDING, tmp_path)


FALLBACK = r"""
# padded rows that cannot be had (any allocation of them fails): dense ones, on
# the direct kernels, with no error left behind
before = fake.fake_mallocs()
rc, c = create(45)
n = fake.fake_mallocs() - before
for k in range(1, n + 1):
    fake.fake_fail_malloc(k)
    c = context(45, table=[WATER, BONE])
    assert fake.fake_pending() == 0, k
    launched()
    assert L.bvf_run_acoustic(c, 1, None, None) == OK
    assert [name for name, _ in launched()] == ["k_velocity", "k_stress"], k
    L.bvf_destroy(c)
"""


def test_dense_rows_where_padded_ones_cannot_be_had(tmp_path):
    host_cuda.run(FALLBACK, tmp_path)


INDEX_RANGE = r"""
# the memories of an axis (six slabs of 2 n_pml + 1 layers) are indexed with 32
# bits: 6 * 39 * 48 * 200000 elements of padded rows are too many where the
# 6 * 39 * 41 * 200000 of dense rows are not
def made(*shape, **kw):
    before = fake.fake_malloc_bytes()
    rc, c = create(*shape, **kw)
    if rc == OK:
        L.bvf_destroy(c)
    return rc, fake.fake_malloc_bytes() - before

def state_bytes(pitch, ny, nz, W):      # fields and CPML memories, FP32, no SLS
    return 4 * (9 * pitch * ny * nz + 6 * W * (nz * ny + nz * pitch + ny * pitch))

for ny, pitch in ((190000, 48), (200000, 41)):
    rc, n = made(41, ny, 40, n_sls=0, n_pml=19)
    low = state_bytes(pitch, ny, 40, 39)
    # the peak map, the index and its padded copy, tables, the CPML profile
    assert rc == OK and low < n < low + (4 * pitch + 41 + 48) * ny * 40 + (2 << 20) + (8 * pitch + 48) * ny, ny
# dense rows beyond the range are refused
assert made(41, 230000, 40, n_sls=0, n_pml=19)[0] == ARG
assert made(800, 800, 800, n_sls=0, n_pml=340)[0] == ARG
assert made(700, 700, 700, n_sls=0, n_pml=300)[0] == OK
"""


def test_cpml_memories_stay_within_32_bits(tmp_path):
    host_cuda.run(INDEX_RANGE, tmp_path)


ROOM = r"""
# A context of dense rows, with its DFT sums, thermal buffers and the staging of
# bvf_plan_host, against the memory there is.  Where padded rows would take a
# quarter more than dense ones (nx = 13), a program whose two contexts just fit
# with dense rows finds room for both, in the order create, create, use, use.
nx, ny, nz = 13, 64, 60
N = nx * ny * nz
cap, th = bvf.Capture(0, 1, 4), bvf.Thermal(1e-3, 2, 1, 0.3, 37.0, 2.2e6, 1.0)

def use(c):
    materials(c, N, [WATER])
    assert L.bvf_run_acoustic(c, 1, ctypes.byref(cap), None) == OK
    assert L.bvf_run_thermal(c, ctypes.byref(th), buf(8 * N), buf(4 * N), buf(4 * N), buf(8 * N), None) == OK

def two_contexts(free):
    start, cs = fake.fake_malloc_bytes(), []
    for _ in range(2):
        fake.fake_free_mem(max(0, int(free - (fake.fake_malloc_bytes() - start))))
        rc, c = create(nx, ny, nz)
        assert rc == OK
        cs.append(c)
    launched()
    for c in cs:
        use(c)
    taken = fake.fake_malloc_bytes() - start
    padded = [n for n, _ in launched()].count("k_velocity_tma")
    return taken, padded

staging = 29 * N
dense, none = two_contexts(1)
assert none == 0
exact = dense + 2 * staging                 # what two dense contexts come to hold
for free in (exact, 1.02 * exact, 1.1 * exact, 1.2 * exact, 1.3 * exact, 2 * exact):
    taken, padded = two_contexts(free)
    assert taken + 2 * staging <= free, (free / exact, padded)
assert padded == 2                          # room enough: both padded
"""


def test_padded_rows_leave_room_for_what_dense_rows_held(tmp_path):
    host_cuda.run(ROOM, tmp_path)
