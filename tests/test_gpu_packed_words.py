"""Packed words at the sizes where their walk changes, against the oracle
(bit-exact): half rows just below, at and above a word and two words; rows of
at most 13 sites, whose words skip their second half's draws; rows that start
inside a Philox group (a warp takes 31 words, the last lane lending its draws)
with word counts around a warp's step; full words.  And the joint passes of a
batch: the same for lattices of every kind together, sweep counts and intervals
that differ, a continued launch, and sweep indices up to the last."""
import numpy as np
import pytest

import oracle

INT8, BITPACK = 0, 1
METROPOLIS, HEATBATH, MULTIHIT = 0, 1, 3


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_cs_0312006_gb300 import _build, engine
    _build.build()
    engine.load_library()
    return engine


SHAPES = [(2, L) for L in (4, 24, 26, 28, 30, 60, 62, 64, 66, 68, 72, 122, 124, 126, 128, 130, 200,
                           254, 320)]
SHAPES += [(3, L) for L in (4, 10, 26, 30, 34, 36)]


@pytest.mark.gpu
@pytest.mark.parametrize("dims,L", SHAPES)
@pytest.mark.parametrize("rule", [METROPOLIS, HEATBATH, MULTIHIT])
def test_words(eng, dims, L, rule):
    beta, seed, n = (0.42 if dims == 2 else 0.21), 70 + L, 4
    lat = eng.Lattice(dims, L, beta, seed, layout=BITPACK, rule=rule)
    lat.set_hits(3)
    for _ in range(n):  # one sweep a call: the pass kernels, whatever the size
        lat.sweep(1, 1)
    E, M = lat.observables()
    s = lat.get_spins()
    lat.close()
    if rule == MULTIHIT:
        want = oracle.run_multihit(dims, L, beta, seed, n, 3)
    else:
        want = oracle.run(dims, L, beta, seed, n, heatbath=rule == HEATBATH)
    assert np.array_equal(s, want[0])
    assert np.array_equal(E, want[1]) and np.array_equal(M, want[2])


@pytest.mark.gpu
@pytest.mark.parametrize("big_sites", [0, 1])
def test_joint_passes(eng, big_sites):
    """Every lattice of a batch with the cluster size left open, two launches."""
    specs = [(dims, L, layout, rule, 1 + (3 * k) % 7, 1 + k % 3)
             for k, (dims, L, layout, rule) in enumerate(
                 (d, L, y, r) for d, L in ((2, 2), (2, 26), (2, 62), (2, 66), (2, 126), (2, 256),
                                           (3, 6), (3, 16), (3, 22), (3, 36))
                 for y in (INT8, BITPACK) for r in (METROPOLIS, HEATBATH))]
    beta = {2: 0.43, 3: 0.22}
    lats = [eng.Lattice(d, L, beta[d], 900 + k, layout=y, rule=r)
            for k, (d, L, y, r, _, _) in enumerate(specs)]
    batch = eng.Batch(lats, [sp[4] for sp in specs], [sp[5] for sp in specs], big_sites=big_sites)
    batch.launch()
    batch.launch()
    batch.sync()
    for k, (lat, (d, L, y, r, n, every)) in enumerate(zip(lats, specs)):
        E, M = lat.observables()
        s_o, E_o, M_o = oracle.run(d, L, beta[d], 900 + k, 2 * n, every, heatbath=r == HEATBATH)
        assert np.array_equal(lat.get_spins(), s_o), specs[k]
        assert np.array_equal(E, E_o) and np.array_equal(M, M_o), specs[k]
        lat.close()
    batch.close()


@pytest.mark.gpu
def test_joint_passes_to_the_last_sweep(eng):
    """The record after sweep 2^32 - 1 (its number plus one needs 64 bits)."""
    t0, n = 2 ** 32 - 3, 3
    for every in (1, 2, 4):
        got = []
        for joint in (False, True):
            lat = eng.Lattice(2, 96, 0.4, 5, layout=BITPACK)
            lat.set_spins(oracle.init(2, 96, 5), t=t0)
            if joint:
                b = eng.Batch([lat], [n], [every], big_sites=1)
                b.launch()
                b.sync()
                b.close()
            else:
                for _ in range(n):
                    lat.sweep(1, every)
            E, M = lat.observables()
            got.append((lat.get_spins().tobytes(), E.tolist(), M.tolist()))
            lat.close()
        assert got[0] == got[1], every


def test_quotients():
    """FastDiv's quotients, restated: floor(n / d) for n < 2^31."""
    rng = np.random.default_rng(1)
    ds = list(range(1, 3000)) + [int(x) for x in rng.integers(3000, 2 ** 31, 3000)]
    for d in ds:
        s, one = d.bit_length() - 1, 0
        if d == 1:
            m, one = 0, 0xFFFFFFFF
        elif d & (d - 1) == 0:
            m, s = 1 << 31, s - 1
        else:
            m = ((1 << (32 + s)) + d - 1) // d
        assert m < 1 << 32
        for q in [0, 1, 2, (2 ** 31 - 1) // d] + [int(x) for x in rng.integers(0, 2 ** 31, 8) // d]:
            for n in (q * d - 1, q * d, q * d + 1, 2 ** 31 - 1):
                if 0 <= n < 2 ** 31:
                    assert (((n * m) >> 32) >> s) + (n & one) == n // d, (n, d)
