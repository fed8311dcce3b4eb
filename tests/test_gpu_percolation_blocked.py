"""Blocked growth of 2D media against the oracle (bit-exact) at the sizes where
its geometry changes: one CTA for a whole medium up to L = 256, tiles with a
halo beyond (64 rows inside a tile, one tile across up to 16 words, then
several), rows that are no whole block, and in the batch every lane count and
media whose clusters leave as bytes or as 16-byte stores.  Clusters, sizes,
spanning and the number of passes must equal the oracle's; a corner source
makes growth enter tiles from their corners."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

POINT, FACE = 0, 1


@pytest.fixture(scope="module")
def perc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_cs_0312006_gb300 import _build, percolation
    _build.build()
    return percolation


@pytest.mark.parametrize("L", [4, 65, 255, 256, 257, 320, 512, 513, 769, 1300])
@pytest.mark.parametrize("P", [0.61, 0.75])
def test_medium(perc, L, P):
    m = perc.Medium(2, L, 40 + L)
    m.generate(P)
    pore = oracle.perc_pores(2, L, 40 + L, P)
    for source, site in ((FACE, 0), (POINT, 0), (POINT, L * L - 1), (POINT, L // 2 * (L + 1))):
        r = m.invade(source, site)
        c_o, size, spans, steps = oracle.perc_invade(2, L, pore, source, site)
        assert np.array_equal(m.cluster(), c_o), (L, P, source, site)
        assert (r.size, bool(r.spans), r.steps) == (size, spans, steps), (L, P, source, site)
    m.close()


def test_modes_agree(perc):
    """The graph's band passes and the blocked growth give the same answers."""
    m = perc.Medium(2, 700, 9)
    m.generate(0.6)
    got = []
    for mode in (perc.PASSES_AUTO, perc.PASSES_GRAPH, perc.PASSES_AUTO):
        m.set_passes(mode)
        r = m.invade(FACE)
        got.append((r.size, r.spans, r.steps, m.cluster().tobytes()))
    m.close()
    assert got[0] == got[1] == got[2]


@pytest.mark.parametrize("L", [1, 4, 5, 63, 64, 65, 100, 129, 255, 257, 511])
@pytest.mark.parametrize("offset", [0, 1])
def test_batch(perc, L, offset):
    import torch
    n, P = 5, 0.62
    seeds = [300 + 7 * k for k in range(n)]
    buf = torch.full((n * L * L + 16,), 9, dtype=torch.uint8, device="cuda")
    for source, site in ((FACE, 0), (POINT, L // 2 * (L + 1))):
        res = perc.batch(2, L, P, seeds, source, site, buf.data_ptr() + offset)
        got = buf.cpu().numpy()
        assert (got[:offset] == 9).all() and (got[offset + n * L * L:] == 9).all()
        got = got[offset:offset + n * L * L].reshape(n, -1)
        for k, seed in enumerate(seeds):
            c_o, size, spans, steps = oracle.perc_invade(
                2, L, oracle.perc_pores(2, L, seed, P), source, site)
            assert np.array_equal(got[k], c_o), (L, source, k)
            assert (res[k].size, bool(res[k].spans), res[k].steps) == (size, spans, steps)
