"""The default candidates of the tile tuners hold what a context runs without
tuning, so tuning does not have to make it slower."""
from tests import host_cuda


def test_every_pair_of_heights_has_the_rules_own_chunk():
    from paper_2301_12727_gb300 import bvf
    rows = {(s, v) for s, v, _ in bvf.TILE_CANDIDATES}
    assert {(s, v) for s, v, k in bvf.TILE_CANDIDATES if k == 0} == rows
    assert len(set(bvf.TILE_CANDIDATES)) == len(bvf.TILE_CANDIDATES)


HOST = r"""
# every trial takes the same time here: both tuners keep the untuned tile
ctxs = [context(nx, 24, 20, [WATER, BONE]) for nx in (32, 48)]
b = ctypes.c_void_p()
assert L.bvf_batch_create((ctypes.c_void_p * 2)(*ctxs), 2, ctypes.byref(b)) == OK

def launched_now():
    out = []
    for c in ctxs:
        launches()
        assert L.bvf_run_acoustic(c, 1, None, None) == OK
        out.append(launches())
    return out

untuned = launched_now()
cand = (bvf.Tile * len(bvf.TILE_CANDIDATES))(*[bvf.Tile(*t) for t in bvf.TILE_CANDIDATES])
best, ms = (bvf.Tile * 2)(), ctypes.c_double()
assert L.bvf_batch_tune_domains(b, 3, cand, len(cand), best, None) == OK
assert launched_now() == untuned
assert L.bvf_batch_tune_graph(b, 3, cand, len(cand), 2, best, ctypes.byref(ms), None) == OK
assert launched_now() == untuned
"""


def test_tuning_that_finds_nothing_faster_keeps_the_default(tmp_path):
    host_cuda.run(HOST, tmp_path)
