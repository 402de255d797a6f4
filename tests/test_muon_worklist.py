"""The flat work lists of delayed Muon's element-wise passes against the
oracle (Alg. 2), at the sizes where the split can go wrong: matrices one
element short of, at and past one round of a CTA (2048), widths that are no
whole packets (a packet of the update then spans two or more rows), a last
partial packet, empty matrices at either end, and more matrices than one warp
searches at a time (32); and of the GEMMs' tiles, by every form a launch takes.
Which form a set takes is asked of the library (muon.gemm_tiles), so that a
change of the rule cannot leave a test without its subject."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from paper_2606_30634_gb300 import muon
from parity_util import TOL_ONE_STEP, TOL_RUN, rel_err
from test_muon_parity import F, NS_BARS, Pair, _flat, close_with_flips

pytestmark = pytest.mark.gpu

EDGES = [(0, 4), (1, 2047), (1, 2048), (1, 2049), (2049, 1), (683, 3), (7, 293), (64, 33), (5, 0)]
MANY = [(1 + i % 5, (3 * i) % 23) for i in range(70)] + [(9, 515), (0, 0)]


@pytest.mark.parametrize("shapes", [EDGES, MANY], ids=["edges", "many"])
@pytest.mark.parametrize("correction", [0, 2])
def test_flat_chunks_match_the_oracle(cuda_device, shapes, correction):
    """Three calls, no Newton-Schulz steps, so O is M / ||M||_F in bf16 and
    the weights, momentum and history are held element by element; an O that
    rounds the other way (an inverse norm one ulp off) moves U by at most
    lr r 2^-8."""
    p = Pair(shapes, cuda_device, ns_steps=0, ef=True, sdt=F, correction=correction)
    du = p.lr * 0.2 * np.sqrt(max(max(s) for s in shapes)) * 2.0 ** -8
    try:
        for k in range(3):
            p.step()
            assert rel_err(p.cat(p.gpu.mom), _flat(p.ref.mom)) <= (TOL_ONE_STEP if k == 0
                                                                   else TOL_RUN)
            close_with_flips(p.cat(p.gpu.master), _flat(p.ref.x), TOL_RUN, (k + 1) * du, 1e-3)
            close_with_flips(p.cat(p.gpu.ef), _flat(p.ref.u_prev), 1e-5, du, 2e-3)
            close_with_flips(p.cat(p.gpu.stash), _flat(p.ref.stash), TOL_RUN, (k + 1) * du, 1e-3)
    finally:
        p.close()


def test_more_shape_groups_than_one_launch_takes(cuda_device):
    """Ten matrix shapes: one GEMM launch takes up to eight, so each product
    of a Newton-Schulz step is two launches; one step at its normwise and
    differing-elements bars, and each matrix's output on its own."""
    p = Pair([(64 + i, 96 + 3 * i) for i in range(10)], cuda_device, ns_steps=1)
    try:
        p.step()
        for g, r in zip(*p.o_pairs()):
            assert np.linalg.norm(g - r) <= NS_BARS[1][0] * np.linalg.norm(r)
            assert np.mean(g != r) <= NS_BARS[1][1]
    finally:
        p.close()


# sizes on either side of a single CTA's tile (128) and of a pair's (256), in
# both dimensions; few enough tiles that single CTAs take them
EDGE_TILES = [(127, 129), (128, 128), (129, 384), (256, 385), (257, 640), (384, 257),
              (385, 513), (512, 641), (640, 640)]
# wide, tall and square matrices whose sizes, rounded up to 128, are odd
# multiples of it in one dimension, the other or both, and enough of them that
# CTA pairs take all three products
HALVES = [(640, 640), (600, 1100), (1100, 600), (897, 1152), (1152, 897)] * 6


def near_oracle(p, steps, calls=1):
    """Each matrix's Newton-Schulz output, call by call, at the normwise and
    differing-elements bars of its steps."""
    for _ in range(calls):
        p.step()
        for i, (g, r) in enumerate(zip(*p.o_pairs())):
            assert np.linalg.norm(g - r) <= NS_BARS[steps][0] * np.linalg.norm(r), (i, p.shapes[i])
            assert np.mean(g != r) <= NS_BARS[steps][1], (i, p.shapes[i])


@pytest.mark.parametrize("steps", [1, 2])
def test_tiles_of_single_ctas_at_their_edges(cuda_device, steps):
    for product in range(3):
        single, pair, _, _ = muon.gemm_tiles(EDGE_TILES, product)
        assert single > 0 and pair == 0
    p = Pair(EDGE_TILES, cuda_device, ns_steps=steps)
    try:
        near_oracle(p, steps, calls=2)
    finally:
        p.close()


@pytest.mark.parametrize("steps", [1, 2])
def test_tiles_half_in_the_padding(cuda_device, steps):
    """CTA pairs skip the padded half of a tile in all three products, wide and
    tall (which store X^T alone), over two calls (the second reads scratch that
    the first left)."""
    for product in range(3):
        single, pair, half, four = muon.gemm_tiles(HALVES, product)
        assert single == 0 and 0 < half < pair and four == 0
    p = Pair(HALVES, cuda_device, ns_steps=steps)
    try:
        near_oracle(p, steps, calls=2)
    finally:
        p.close()


# with the form of each product: by single CTAs (1) or by pairs (2)
FORMS = [((128, 128), 1, (1, 1, 1)), ((129, 257), 1, (1, 1, 1)), ((256, 768), 2, (1, 1, 1)),
         ((640, 300), 3, (1, 1, 1)), ((512, 2048), 40, (1, 1, 2)), ((768, 768), 60, (2, 2, 2))]


@pytest.mark.parametrize("shape,copies,forms", FORMS)
def test_tiles_by_single_ctas_and_by_pairs(cuda_device, shape, copies, forms):
    """One shape from one tile to several rounds of them: the small sets' GEMMs
    go to single CTAs (128 x 128 tiles), the large sets' to CTA pairs. Two
    Newton-Schulz steps, so each product reads what the other forms wrote."""
    for product, form in enumerate(forms):
        tiles = muon.gemm_tiles([shape] * copies, product)
        assert tiles[form - 1] > 0 and tiles[2 - form] == 0, (product, tiles)
    p = Pair([shape] * copies, cuda_device, ns_steps=2)
    try:
        near_oracle(p, 2)
    finally:
        p.close()


LONG_K = [(4098, 4100), (4100, 4098)]


def test_four_epilogue_warps_match_eight(cuda_device):
    """K of 4098 and 4100 (33 blocks, the last nearly empty): a wide and a tall
    matrix together are 578 pair tiles in B X + a X, which four epilogue warps
    drain; each alone is 289, which eight do. The same tiles either way, so the
    same bits. The symmetric products of one alone go to single CTAs, which
    compute the same elements from the same K blocks."""
    shapes = LONG_K
    for product in range(3):
        _, pair, half, four = muon.gemm_tiles(shapes, product)
        assert four == pair > 0 and half > 0
        for shape in shapes:
            assert muon.gemm_tiles([shape], product)[3] == 0
    assert muon.gemm_tiles(shapes[:1], 2)[:3] == (0, 289, 33)
    gen = torch.Generator().manual_seed(7)
    grads = [torch.randn(s, generator=gen) for s in shapes]

    def outputs(which):
        m = muon.DelayedMuon([shapes[i] for i in which], ns_steps=2, lr=0.02, momentum=0.95,
                             device=cuda_device, x0=[torch.zeros(shapes[i]) for i in which])
        try:
            for q, i in enumerate(which):
                m.grads(q).copy_(grads[i])
            m.step()
            torch.cuda.synchronize()
            return [m.last_update(q).clone() for q in range(len(which))]
        finally:
            m.close()

    for i, got in enumerate(outputs([0, 1])):
        assert torch.equal(got, outputs([i])[0]), shapes[i]
        assert got.float().abs().sum() > 0
