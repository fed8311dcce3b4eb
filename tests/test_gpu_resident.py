"""Runs of sweeps in one launch (the cluster-resident kernel) against the oracle,
bit-exact, at the sizes where its slabs and rows change: one CTA, two to sixteen,
slabs of unequal heights, rows that end inside a word and start inside a Philox
group, rows shorter than a word, both layouts and rules, records at intervals
that do not divide the first sweep's number, and the sizes on both sides of the
line to the pass kernels; and the pass kernels' int8 vectors where rows end
inside them, at the lattice's edges and at its ragged end."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

INT8, BITPACK = 0, 1


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_cs_0312006_gb300 import _build, engine
    _build.build()
    engine.load_library()
    return engine


SHAPES = [(2, L) for L in (2, 4, 6, 8, 10, 22, 30, 32, 34, 62, 66, 90, 92, 126, 128, 130, 258, 328,
                           340, 418, 420, 430, 470)]
SHAPES += [(3, L) for L in (2, 4, 6, 8, 10, 14, 18, 24, 34, 38, 46, 64)]


@pytest.mark.parametrize("dims,L", SHAPES)
@pytest.mark.parametrize("layout", [INT8, BITPACK])
def test_runs(eng, dims, L, layout):
    beta, seed = (0.43 if dims == 2 else 0.22), 11 + L
    for heatbath in (False, True):
        lat = eng.Lattice(dims, L, beta, seed, layout=layout, rule=int(heatbath))
        lat.sweep(5, 3)   # records after sweeps 2, 5, 8, ...
        lat.sweep(1, 3)
        lat.sweep(6, 3)
        E, M = lat.observables()
        s = lat.get_spins()
        lat.close()
        s_o, E_o, M_o = oracle.run(dims, L, beta, seed, 12, 3, heatbath=heatbath)
        assert np.array_equal(s, s_o), (dims, L, layout, heatbath)
        assert np.array_equal(E, E_o) and np.array_equal(M, M_o), (dims, L, layout, heatbath)


@pytest.mark.parametrize("dims,L", [(2, L) for L in (32, 34, 36, 38, 46, 50, 62, 78, 94, 130, 258)]
                         + [(3, L) for L in (32, 34, 36, 38, 46)])
@pytest.mark.parametrize("rule", [0, 1, 3])
def test_int8_vectors(eng, dims, L, rule):
    """One sweep a call: the pass kernels (rows of at least a vector)."""
    beta, seed, n = (0.43 if dims == 2 else 0.22), 5 + L, 3
    lat = eng.Lattice(dims, L, beta, seed, layout=INT8, kernel=eng.KERNEL_STRIP, rule=rule)
    lat.set_hits(2)
    for _ in range(n):
        lat.sweep(1, 1)
    E, M = lat.observables()
    s = lat.get_spins()
    lat.close()
    want = (oracle.run_multihit(dims, L, beta, seed, n, 2) if rule == 3
            else oracle.run(dims, L, beta, seed, n, heatbath=rule == 1))
    assert np.array_equal(s, want[0])
    assert np.array_equal(E, want[1]) and np.array_equal(M, want[2])


def test_last_sweeps(eng):
    """A run up to sweep 2^32 - 1, records at an interval that reaches it."""
    t0 = 2 ** 32 - 6
    got = []
    for whole in (True, False):
        lat = eng.Lattice(2, 66, 0.4, 3, layout=BITPACK)
        lat.set_spins(oracle.init(2, 66, 3), t=t0)
        for n in ([6] if whole else [1] * 6):
            lat.sweep(n, 2)
        E, M = lat.observables()
        got.append((lat.get_spins().tobytes(), E.tolist(), M.tolist()))
        lat.close()
    assert got[0] == got[1]
