"""Batches whose tensors begin and end about the rows of a CTA: the first row of the next tensor is requested with the last
one of the tensor before, and a codebook's tables serve all of them.  Codes and constants are those of the calls on one tensor
(which the other tests hold against the oracle), bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu

ROW = {torch.bfloat16: 512 * 32, torch.float32: 512 * 16}   # weights of a CTA's row
CTAS = 2 * 148


@pytest.fixture(scope="module")
def bof4():
    import paper_2505_06653_b200 as m
    return m


@pytest.mark.parametrize("block", [32, 64, 2048])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("levels", ["printed", "rational", "crowded"])
def test_rows_across_tensors(bof4, block, dtype, levels):
    row = ROW[dtype]
    lv = {"printed": [-0.8568463921546936, -0.6692874431610107, -0.5235266089439392, -0.4004882574081421, -0.2910638153553009,
                      -0.1900092959403992, -0.0938529595732689, 0.0, 0.0887671709060669, 0.1794802695512772, 0.2743096053600311,
                      0.3760197460651398, 0.4886530041694641, 0.6188603639602661, 0.7791395783424377, 1.0],
          "rational": [k / 8 for k in range(-7, 9)],
          # several thresholds in one bin of the table: no table serves it
          "crowded": [-1.0, -0.5, -0.25] + [0.001 * k for k in range(-4, 6)] + [0.25, 0.5, 1.0]}[levels]
    lv = torch.tensor(lv, device="cuda")
    sizes = [row, block, row - block, row + block, 1, row * CTAS, 33, 2 * row + 5, row * CTAS + row // 2, row * 3 - 1, block + 1]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(block)
    w = [(torch.randn(n, generator=gen, device="cuda") * 0.02).to(dtype) for n in sizes]
    code = bof4.BF16 if dtype == torch.bfloat16 else bof4.F32
    codes, consts = bof4.bof4_quantize_batch(w, block, bof4.NORM_SIGNED, lv, code)
    for t, c, s in zip(w, codes, consts):
        c1, s1 = bof4.bof4_quantize(t, block, bof4.NORM_SIGNED, lv, code)
        assert torch.equal(c, c1) and torch.equal(s, s1)
    out = bof4.bof4_dequantize_batch(codes, consts, sizes, block, lv, code)
    for n, c, s, o in zip(sizes, codes, consts, out):
        assert torch.equal(o, bof4.bof4_dequantize(c, s, block, lv, code, n=n))
