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
