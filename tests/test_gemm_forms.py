"""Which form the Newton-Schulz GEMM launches of a set take (dpo_muon_test_tiles),
for a GPU that holds 76 CTA pairs or 152 single CTAs, without one: the sets of the
GPU tests of each form take it, so a change of the rule that empties one shows
here first."""
from __future__ import annotations

import pytest

from paper_2606_30634_gb300 import dpo, muon
from test_muon_worklist import EDGE_TILES, FORMS, HALVES, LONG_K

PAIRS, CTAS = 76, 152


def tiles(shapes, product, pairs=PAIRS, ctas=CTAS):
    return muon.gemm_tiles(shapes, product, pairs, ctas)


@pytest.mark.parametrize("product", [0, 1, 2])
def test_sets_of_the_gpu_tests_take_their_forms(product):
    single, pair, _, _ = tiles(EDGE_TILES, product)
    assert single > 0 and pair == 0
    single, pair, half, four = tiles(HALVES, product)
    assert single == 0 and 0 < half < pair and four == 0
    for shape, copies, forms in FORMS:
        got = tiles([shape] * copies, product)
        assert got[forms[product] - 1] > 0 and got[2 - forms[product]] == 0, shape
    single, pair, half, four = tiles(LONG_K, product)
    assert single == 0 and four == pair and half > 0


@pytest.mark.parametrize("shapes,product,want", [
    ([], 0, (0, 0, 0, 0)), ([(0, 5), (5, 0)], 2, (0, 0, 0, 0)),
    ([(1, 1)], 0, (1, 0, 0, 0)),
    # 3 x 6 tiles of 128 x 128; the triangle of 3 x 3
    ([(384, 700)], 2, (18, 0, 0, 0)), ([(700, 384)], 0, (6, 0, 0, 0)),
    # 18 x 19 pair tiles; the last row and column hold 1 row and 92 columns
    ([(4353, 4700)], 2, (0, 342, 36, 342)), ([(4353, 4700)], 1, (0, 171, 18, 0))])
def test_tile_counts(shapes, product, want):
    assert tiles(shapes, product) == want


@pytest.mark.parametrize("kw", [dict(product=3), dict(product=-1), dict(pairs=0), dict(ctas=0),
                                dict(pairs=-1), dict(shapes=[(-1, 4)]),
                                dict(shapes=[(1 << 26, 1 << 26)])])
def test_bad_arguments(kw):
    with pytest.raises(dpo.DpoError):
        tiles(**dict(dict(shapes=[(4, 4)], product=0), **kw))


@pytest.mark.parametrize("pairs", [1 << 28, (1 << 29) - 1, 1 << 29, 1 << 30])
def test_rounds_of_a_failed_residency_query(pairs):
    """Fewer than one round of tiles, however many pairs: not the four warps of long
    launches. (A residency query that fails leaves 2^30.)"""
    for product in range(3):
        assert tiles(LONG_K, product, pairs)[3] == 0
