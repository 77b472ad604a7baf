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
