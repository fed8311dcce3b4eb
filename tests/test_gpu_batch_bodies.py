"""The persistent batch launch and the bit-packed pass by the ways they walk a
lattice's rows, bit-exact against the oracle: packed words of rows that need four,
five or eight calls, starting on a draw group or inside one; int8 rows of 16-site
vectors (whole and ragged, and too few of them for the CTAs), of whole words, and
words of any rows; one CTA and clusters."""
import functools

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

INT8, BITPACK = 0, 1
SHAPES = [(2, L) for L in (6, 24, 26, 28, 30, 32, 34, 36, 38, 40, 42, 44, 64, 90, 100, 126, 128, 130)]
SHAPES += [(3, L) for L in (8, 26, 30, 32, 34, 36, 38, 40, 128)]
SWEEPS, EVERY = 4, 2


@pytest.fixture(scope="module")
def eng():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_cs_0312006_gb300 import _build, engine
    _build.build()
    engine.load_library()
    return engine


def beta(dims):
    return 0.43 if dims == 2 else 0.22


@functools.lru_cache(maxsize=None)
def wanted(dims, L, heatbath):
    return oracle.run(dims, L, beta(dims), 60 + L, SWEEPS, EVERY, heatbath=heatbath)


def same(lat, dims, L, heatbath, what):
    s, E, M = wanted(dims, L, heatbath)
    E_g, M_g = lat.observables()
    assert np.array_equal(lat.get_spins(), s), what
    assert np.array_equal(E_g, E) and np.array_equal(M_g, M), what


@pytest.mark.parametrize("opts", [dict(cluster_size=1), dict(cluster_size=1, block_threads=128),
                                  dict(cluster_size=2, big_sites=1),
                                  dict(cluster_size=8, big_sites=1)])
@pytest.mark.parametrize("heatbath", [False, True])
def test_batch(eng, opts, heatbath):
    specs = [(d, L, y) for d, L in SHAPES for y in (INT8, BITPACK)]
    lats = [eng.Lattice(d, L, beta(d), 60 + L, layout=y, rule=int(heatbath)) for d, L, y in specs]
    batch = eng.Batch(lats, SWEEPS // 2, EVERY, **opts)
    batch.launch()
    batch.launch()
    batch.sync()
    for lat, (d, L, y) in zip(lats, specs):
        same(lat, d, L, heatbath, (d, L, y, opts))
        lat.close()
    batch.close()


@pytest.mark.parametrize("heatbath", [False, True])
@pytest.mark.parametrize("dims,L", [(d, L) for d, L in SHAPES if L < 64])
def test_packed_pass(eng, dims, L, heatbath):
    lat = eng.Lattice(dims, L, beta(dims), 60 + L, layout=BITPACK, rule=int(heatbath))
    for _ in range(SWEEPS):  # one sweep a call: the pass kernel
        lat.sweep(1, EVERY)
    same(lat, dims, L, heatbath, (dims, L))
    lat.close()
