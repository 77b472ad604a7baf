"""Fits over bf16 weights with so many blocks that their addresses are put in order tile by tile (2^19 and more in a launch of 64
tensors), against the oracle: tensors that end inside tiles and inside groups of eight blocks, more than one launch, magnitudes that
fill more slots than a tile has threads, one magnitude alone."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

I = 32
BLOCKS = 1 << 19


@pytest.fixture(scope="module")
def bof4():
    import __graft_entry__ as entry
    entry.build()
    import paper_2505_06653_b200 as m
    return m


def _sizes(kind):
    if kind == "one":
        return [BLOCKS * I]
    if kind == "fewer":                  # one block below the line: written directly
        return [(BLOCKS - 1) * I]
    # 70 tensors: odd block counts, some without a whole block, ragged ends; 64 of them in the first launch
    sizes = [(4001 + 137 * k) * I + (k % 3) * 11 for k in range(69)]
    sizes[5], sizes[6] = 31, 7
    return sizes + [max(0, BLOCKS * I * 2 - sum(sizes))]


def _weights(n, seed, scales):
    w = workloads.gaussian(n, 0.02, seed, torch.float32)
    g = torch.Generator().manual_seed(seed + 1)
    blocks = (n + I - 1) // I
    if scales == "many":                 # 30 binades of block constants: thousands of magnitudes in a tile
        w *= torch.exp2(30 * torch.rand(blocks, generator=g) - 15).repeat_interleave(I)[:n]
    elif scales == "single":             # every block has the same constant
        w = w.clamp(-0.06, 0.06)
        w[::I] = 0.0625
    return w.to(torch.bfloat16)


@pytest.mark.parametrize("sizes", ["one", "fewer", "list"])
@pytest.mark.parametrize("scales", ["plain", "many", "single"])
@pytest.mark.parametrize("metric", [0, 1])
def test_blocks_in_order(bof4, sizes, scales, metric):
    ws = [_weights(n, 300 + k, scales) for k, n in enumerate(_sizes(sizes))]
    lv, mask = bof4.bof4_default_init(bof4.NORM_SIGNED)
    cb, log = bof4.bof4_fit_codebook([w.cuda() for w in ws], I, bof4.NORM_SIGNED, metric, lv, mask, 4)
    ref, ref_log = oracle.fit(ws, I, bof4.NORM_SIGNED, metric, lv, mask, 4)
    if metric == bof4.METRIC_MAE:
        assert np.array_equal(cb.cpu().numpy(), ref)
    else:
        np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=1e-5, atol=1e-7)
    np.testing.assert_allclose(log.cpu().numpy(), ref_log, rtol=1e-5, atol=1e-12)


CTAS, TILE, LAUNCH = 148, 8192, 64   # CTAs of the ordering, blocks of a tile, tensors of a launch


def _launches(sizes):
    """(first block, blocks) of every launch: tensors without a whole block are in none."""
    blocks = [n // I for n in sizes if n >= I]
    first, out = 0, []
    for k in range(0, len(blocks), LAUNCH):
        out.append((first, sum(blocks[k:k + LAUNCH])))
        first += out[-1][1]
    return out


def _ragged(kind):
    if kind == "launches":               # the second launch begins inside a group of eight blocks
        sizes = [(9001 + 138 * k) * I + (k % 3) * 11 for k in range(71)]
        sizes[5], sizes[6] = 31, 7
        sizes.append((BLOCKS + 4099) * I + 5)
        (_, n0), (first, n1) = _launches(sizes)
        assert n0 >= BLOCKS and n1 >= BLOCKS and first % 8
    else:                                # every CTA takes three tiles; tensors end inside them
        sizes = [(70001 + 137 * k) * I + (k % 3) * 11 for k in range(36)]
        (_, n0), = _launches(sizes)
        assert n0 > 2 * CTAS * TILE and n0 < 3 * CTAS * TILE
    return sizes


@pytest.mark.parametrize("kind,scales", [("launches", "plain"), ("launches", "many"), ("launches", "single"), ("tiles", "plain"), ("tiles", "many")])
def test_tiles_and_launches(bof4, kind, scales):
    """Launches that share a group of blocks, and CTAs of several tiles: against the oracle, and bit for bit against the same blocks in
    tensors so small that every launch writes its addresses directly (sums of integers: no order of blocks changes a bit)."""
    ws = [_weights(n, 900 + k, scales) for k, n in enumerate(_ragged(kind))]
    lv, mask = bof4.bof4_default_init(bof4.NORM_SIGNED)
    cuda = [w.cuda() for w in ws]
    cb, log = bof4.bof4_fit_codebook(cuda, I, bof4.NORM_SIGNED, bof4.METRIC_MSE, lv, mask, 4)
    piece = 8000 * I
    split = [p for w in cuda for p in w.split(piece)]
    assert all(n < BLOCKS for _, n in _launches([p.numel() for p in split]))
    cb2, log2 = bof4.bof4_fit_codebook(split, I, bof4.NORM_SIGNED, bof4.METRIC_MSE, lv, mask, 4)
    assert torch.equal(cb, cb2) and torch.equal(log, log2)
    ref, ref_log = oracle.fit(ws, I, bof4.NORM_SIGNED, bof4.METRIC_MSE, lv, mask, 4)
    np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=1e-5, atol=1e-7)
    np.testing.assert_allclose(log.cpu().numpy(), ref_log, rtol=1e-5, atol=1e-12)
