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


# strips, strips in 3D, rows that end inside a vector, the staged kernel
@pytest.mark.parametrize("dims,L,staged", [(2, 512, False), (3, 64, False), (2, 600, False),
                                           (3, 98, False), (2, 512, True), (3, 64, True)])
@pytest.mark.parametrize("rule", [METROPOLIS, HEATBATH, MULTIHIT])
def test_int8(eng, ahead, dims, L, staged, rule):
    check(eng, ahead, dims, L, INT8, rule,
          kernel=eng.KERNEL_TMA if staged else eng.KERNEL_STRIP)


@pytest.mark.parametrize("L,layout", [(512, INT8), (600, INT8), (512, BITPACK), (600, BITPACK)])
def test_demon(eng, ahead, L, layout):
    import torch
    q = np.random.default_rng(L).integers(0, 4, L * L, dtype=np.uint8)
    s = oracle.init(2, L, 7)
    s_o, q_o, E_o, M_o = oracle.run_demon(2, L, s, q, 3, SWEEPS, EVERY)
    want, start = torch.from_numpy(s_o).cuda(), torch.from_numpy(s).cuda()
    got = torch.empty_like(want)
    lat = eng.Lattice(2, L, 0.43, 7, layout=layout)
    for k in range(REPEATS // 2):
        lat.set_demons(q, qmax=3)
        lat.set_rule(2)
        lat.set_spins_async(start.data_ptr())
        ahead.sweep(2, 2)
        for _ in range(SWEEPS):
            lat.sweep(1, EVERY)
        lat.get_spins_async(got.data_ptr())
        E, M = lat.observables()
        ahead.observables()
        assert np.array_equal(E, E_o) and np.array_equal(M, M_o), (L, layout, k)
        assert torch.equal(got, want) and np.array_equal(lat.get_demons(), q_o), (L, layout, k)
    lat.close()


def test_joint(eng, ahead):
    """A batch's joint passes, launch after launch (each reads the job table that
    the end of the launch before it has moved on)."""
    import torch
    shapes = [(3, 64, BITPACK), (2, 512, INT8), (2, 600, BITPACK), (3, 98, INT8)]
    lats = [eng.Lattice(d, L, 0.43 if d == 2 else 0.22, 3 * L, layout=y) for d, L, y in shapes]
    want = [wanted(d, L, METROPOLIS) for d, L, _ in shapes]
    got = [torch.empty(L ** d, dtype=torch.int8, device="cuda") for d, L, _ in shapes]
    batch = eng.Batch(lats, [EVERY] * len(lats), [EVERY] * len(lats), big_sites=1)
    for k in range(REPEATS):
        for lat in lats:
            lat.init()
        ahead.sweep(2, 2)
        for _ in range(SWEEPS // EVERY):
            batch.launch()
        batch.sync()
        ahead.observables()
        for lat, g, (s_o, E_o, M_o) in zip(lats, got, want):
            lat.get_spins_async(g.data_ptr())
            E, M = lat.observables()
            assert np.array_equal(E, E_o) and np.array_equal(M, M_o), k
            assert np.array_equal(g.cpu().numpy(), s_o), k
    batch.close()
    for lat in lats:
        lat.close()
