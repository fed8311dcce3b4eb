"""Chained passes queued back to back, bit-exact against the oracle, many times
over: a longer pass of another lattice on the stream holds the queue up while one
short sweep a call is issued, so that the passes then follow one another at the
GPU's pace and each is placed on the SMs before the one ahead of it has ended.
The lattices are small enough for several passes to fit the GPU together; a pass
that read the other colour before it was complete, or from a copy of it that an
SM had kept, would change spins."""
import functools

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

INT8, BITPACK = 0, 1
METROPOLIS, HEATBATH, MULTIHIT = 0, 1, 3
SWEEPS, EVERY, HITS, REPEATS = 30, 2, 3, 200


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_cs_0312006_gb300 import _build, engine
    _build.build()
    engine.load_library()
    return engine


@pytest.fixture(scope="module")
def ahead(eng):
    lat = eng.Lattice(2, 16384, 0.4, 1, layout=BITPACK)  # ~0.1 ms a pass
    yield lat
    lat.close()


@functools.lru_cache(maxsize=None)
def wanted(dims, L, rule):
    beta = 0.43 if dims == 2 else 0.22
    if rule == MULTIHIT:
        return oracle.run_multihit(dims, L, beta, 3 * L, SWEEPS, HITS, measure_every=EVERY)
    return oracle.run(dims, L, beta, 3 * L, SWEEPS, EVERY, heatbath=rule == HEATBATH)


def check(eng, ahead, dims, L, layout, rule, **kw):
    import torch
    s_o, E_o, M_o = wanted(dims, L, rule)
    want = torch.from_numpy(s_o).cuda()
    got = torch.empty_like(want)
    lat = eng.Lattice(dims, L, 0.43 if dims == 2 else 0.22, 3 * L, layout=layout, rule=rule, **kw)
    lat.set_hits(HITS)
    for k in range(REPEATS):
        lat.init()
        ahead.sweep(2, 2)
        for _ in range(SWEEPS):
            lat.sweep(1, EVERY)
        lat.get_spins_async(got.data_ptr())
        E, M = lat.observables()
        ahead.observables()
        assert np.array_equal(E, E_o) and np.array_equal(M, M_o), (dims, L, layout, rule, k)
        assert torch.equal(got, want), (dims, L, layout, rule, k)
    lat.close()


# rows of one full word and of many, rows that start on a draw group and inside one
@pytest.mark.parametrize("dims,L", [(3, 64), (2, 512), (2, 1024), (2, 600), (3, 98)])
@pytest.mark.parametrize("rule", [METROPOLIS, HEATBATH, MULTIHIT])
def test_packed(eng, ahead, dims, L, rule):
    check(eng, ahead, dims, L, BITPACK, rule)
