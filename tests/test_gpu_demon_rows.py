"""The bit-packed demon pass by the shapes its rows are taken in, bit-exact: one
row and two rows an item on both sides of the line between them (the demons'
storage row wraps inside a pair of rows once their offset is odd), and lattices
out of L2 with and without E and M, whose grids differ."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

BITPACK, RULE_DEMON, QMAX = 1, 2, 3


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_cs_0312006_gb300 import _build, engine
    _build.build()
    engine.load_library()
    return engine


def state(L, dims=2):
    rng = np.random.default_rng(L)
    n = L ** dims
    s = np.resize(rng.choice(np.array([-1, 1], dtype=np.int8), size=1000003), n)
    q = np.resize(rng.integers(0, QMAX + 1, size=1000033).astype(np.uint8), n)
    return s, q


def run(eng, dims, L, s, q, n, every):
    lat = eng.Lattice(dims, L, 0.4, 1, layout=BITPACK)
    lat.set_spins(s, 0)
    lat.set_demons(q, qmax=QMAX)
    lat.set_rule(RULE_DEMON)
    lat.sweep(n, every)
    E, M = lat.observables()
    out = lat.get_spins(), lat.get_demons(), E, M
    lat.close()
    return out


@pytest.mark.parametrize("L", [5888, 6400, 8192])
def test_rows(eng, L):
    s, q = state(L)
    want = oracle.run_demon(2, L, s, q, QMAX, 3)
    got = run(eng, 2, L, s, q, 3, 1)
    for g, w in zip(got, want):
        assert np.array_equal(g, w), L


def test_out_of_l2(eng):
    L = 19200
    s, q = state(L)
    plain = run(eng, 2, L, s, q, 3, 3)     # two sweeps without a record, one with
    measured = run(eng, 2, L, s, q, 3, 1)
    assert np.array_equal(plain[0], measured[0]) and np.array_equal(plain[1], measured[1])
    assert plain[2][-1] == measured[2][-1] and plain[3][-1] == measured[3][-1]
