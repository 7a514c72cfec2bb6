"""A device allocation, stream or event that cannot be made leaves a context
that can go on: the call that needed it returns an error, and the same call
made again makes what is missing and does all of its work, for every one of
those that a call makes on first use."""
from tests import host_cuda

COMMON = r"""
NX, NY, NZ = 32, 16, 16
N = NX * NY * NZ
cap = bvf.Capture(0, 1, 4)
th = bvf.Thermal(1e-3, 3, 2, 0.3, 37.0, 2.2e6, 1.0)

def plan_host(c):
    water = context(NX, NY, NZ, [WATER])
    bowl = bvf.Bowl(8e-3, 9e-3, (ctypes.c_double * 3)(8e-3, 4e-3, -2e-2),
                    (ctypes.c_double * 3)(0, 0, 1), 1e5, 1500.0, 0.25)
    pp = bvf.PlanParams(4, 1, 3, 0.0, th, 0)
    out = bvf.PlanOut()
    h = [buf(N), buf(4 * N), buf(4 * N), buf(4 * N), buf(8 * N)]
    mat = bvf.material_array([WATER])
    # without kernels the water field is zero, which the plan refuses at its
    # end: the work up to there is what counts
    def call():
        rc = L.bvf_plan_host(c, water, h[0], mat, 1, mat, ctypes.byref(bowl), 2, ctypes.byref(pp),
                             h[1], h[2], h[3], h[4], ctypes.byref(out), None)
        return OK if rc == ARG and b"zero water intensity" in L.bvf_last_error(None) else rc
    return call
"""

ACOUSTIC = COMMON + r"""

def dft(c):
    return lambda: L.bvf_run_acoustic(c, 2, ctypes.byref(cap), None)

def thermal(c):
    d = [buf(4 * N), buf(4 * N), buf(8 * N)]
    return lambda: L.bvf_run_thermal(c, ctypes.byref(th), buf(8 * N), *d, None)

def load(c):
    # a snapshot with DFT sums, loaded into a context that has none yet
    n = ctypes.c_size_t()
    assert L.bvf_state_bytes(c, ctypes.byref(n)) == OK
    full = context(NX, NY, NZ, [WATER])
    assert dft(full)() == OK
    snap = buf(n.value)
    assert L.bvf_state_save(full, snap, n, None) == OK
    return lambda: L.bvf_state_load(c, snap, n, None)

for make in (dft, thermal, load, plan_host):
    # what the call launches and allocates with nothing failing
    c = context(NX, NY, NZ, [WATER])
    call = make(c)
    launched()
    before = fake.fake_mallocs()
    assert call() == OK, (make.__name__, L.bvf_last_error(None))
    want, n = launched(), fake.fake_mallocs() - before
    assert n > 1
    L.bvf_destroy(c)
    for k in range(1, n + 1):
        c = context(NX, NY, NZ, [WATER])
        call = make(c)
        fake.fake_fail_malloc(k)
        assert call() == NOMEM, (make.__name__, k)
        launched()
        before = fake.fake_mallocs()
        assert call() == OK, (make.__name__, k, L.bvf_last_error(None))
        assert launched() == want, (make.__name__, k)
        assert fake.fake_mallocs() > before, (make.__name__, k)
        # reset walks over the lazily made buffers
        assert L.bvf_reset(c, None) == OK
        L.bvf_destroy(c)
"""


def test_calls_after_a_failed_allocation(tmp_path):
    host_cuda.run(ACOUSTIC, tmp_path)


SURROGATE = r"""
F = fno.lib()
dims = fno.FnoDims(3, 16, 4, 2, 16, 1)
n_w = F.bvf_fno_weight_count(ctypes.byref(dims))
w = (ctypes.c_float * n_w)()

def net():
    f = ctypes.c_void_p()
    assert F.bvf_fno_create(ctypes.byref(f), ctypes.byref(dims), w, n_w) == OK
    return f

def forward(f, nx, ny, nz):
    n = 4 * nx * ny * nz
    return F.bvf_fno_forward(f, nx, ny, nz, buf(3 * n), buf(n), None)

small, large = (16, 12, 10), (32, 24, 20)
f = net()
launched()
assert forward(f, *small) == OK
want, before = launched(), fake.fake_mallocs()
assert forward(f, *large) == OK
n = fake.fake_mallocs() - before
assert n > 4
for k in range(1, n + 1):
    f = net()
    assert forward(f, *small) == OK
    fake.fake_fail_malloc(k)
    assert forward(f, *large) == NOMEM, k
    # back on the grid it had: whatever the failed call gave up is made again
    launched()
    before = fake.fake_mallocs()
    assert forward(f, *small) == OK, (k, L.bvf_last_error(None))
    assert launched() == want and fake.fake_mallocs() > before, k
    assert forward(f, *large) == OK
    F.bvf_fno_destroy(f)

# the BF16 network: a failed creation leaves no error behind for the next one
for k in (1, 5, 20):
    t = ctypes.c_void_p()
    fake.fake_fail_malloc(k)
    assert F.bvf_fno_bf16_create(ctypes.byref(t), ctypes.byref(dims), w, n_w, 16, 12, 10, 1) == NOMEM
    assert not t.value
    assert F.bvf_fno_bf16_create(ctypes.byref(t), ctypes.byref(dims), w, n_w, 16, 12, 10, 1) == OK
    assert F.bvf_fno_bf16_forward(t, 1, buf(12 * 1920), buf(4 * 1920), None) == OK, L.bvf_last_error(None)
    F.bvf_fno_bf16_destroy(t)
"""


def test_surrogate_after_a_failed_grid_change(tmp_path):
    host_cuda.run(SURROGATE, tmp_path)


STREAMS = COMMON + r"""
def batch(run):
    def make(c):
        b = ctypes.c_void_p()
        ctxs = (ctypes.c_void_p * 2)(c, context(NX, NY, NZ, [WATER]))
        steps = (ctypes.c_int * 2)(2, 2)
        assert L.bvf_batch_create(ctxs, 2, ctypes.byref(b)) == OK
        return lambda: run(b, steps, None, 3, None)
    return make

for make, objects in ((plan_host, 3), (batch(L.bvf_batch_run_streams), 7), (batch(L.bvf_batch_run_graph), 7)):
    c = context(NX, NY, NZ, [WATER])
    call = make(c)
    launched()
    assert call() == OK
    want = launched()
    for k in range(1, objects + 1):
        c = context(NX, NY, NZ, [WATER])
        call = make(c)
        fake.fake_fail_object(k)
        assert call() == bvf.BVF_E_CUDA, (objects, k)
        launched()
        assert call() == OK, (objects, k, L.bvf_last_error(None))
        assert launched() == want, (objects, k)
        fake.fake_fail_object(1)
        assert call() == OK          # nothing left to make
        fake.fake_fail_object(0)
"""


def test_calls_after_a_stream_or_event_that_could_not_be_made(tmp_path):
    host_cuda.run(STREAMS, tmp_path)
