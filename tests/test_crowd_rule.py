"""Domains side by side take the long z-chunks of the batch rule only where
together they fill the GPU; few or small ones are launched as a domain alone."""
from tests import host_cuda

HOST = r"""
def grids(c):
    launches()
    assert L.bvf_run_acoustic(c, 1, None, None) == OK
    return [(n, g) for n, g, _ in launches()]

def sweep(ctxs, run, lanes):
    b = ctypes.c_void_p()
    n = len(ctxs)
    assert L.bvf_batch_create((ctypes.c_void_p * n)(*ctxs), n, ctypes.byref(b)) == OK
    launches()
    assert run(b, (ctypes.c_int * n)(*[1] * n), None, lanes, None) == OK
    out = [(k, g) for k, g, _ in launches()]
    L.bvf_batch_destroy(b)
    return out

# (cells per side, domains, streams, long chunks measured the faster in a graph, on streams)
for n, domains, lanes, storage, graph, streams in (
        (32, 8, 8, 0, False, False), (48, 8, 8, 0, False, False), (64, 1, 4, 0, False, False),
        (64, 2, 2, 0, False, False), (64, 8, 4, 0, False, False), (72, 6, 4, 0, False, False),
        (64, 7, 7, 0, True, False), (64, 8, 8, 0, True, True), (96, 8, 4, 0, True, True),
        (128, 2, 2, 0, True, True), (64, 7, 7, 1, False, False), (64, 8, 8, 1, True, False),
        (128, 2, 2, 1, True, True)):
    ctxs = [context(n, n, n, [WATER, BONE], storage=storage) for _ in range(domains)]
    alone = grids(ctxs[0])
    for run, long in ((L.bvf_batch_run_graph, graph), (L.bvf_batch_run_streams, streams)):
        got = sweep(ctxs, run, lanes)
        assert len(got) == 2 * domains
        assert (got[:2] != alone) == long, (n, domains, lanes, storage, long)
        if long:                        # the batch rule: 8 planes a block on these grids
            assert [g[2] for _, g in got[:2]] == [-(-n // 8)] * 2
        L.bvf_reset(ctxs[0], None)
    for c in ctxs:
        L.bvf_destroy(c)
"""


def test_long_chunks_only_where_domains_fill_the_gpu(tmp_path):
    host_cuda.run(HOST, tmp_path)
