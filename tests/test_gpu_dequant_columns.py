"""Decoding on both sides of the size from which the table of level pairs has 32 columns, not 16: the same, bit for bit, as the tensor
decoded in pieces of 2^24 weights (which the other tests hold against the oracle)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

LINE = 1 << 27   # weights
PIECE = 1 << 24


@pytest.mark.parametrize("n", [LINE - 64, LINE, LINE + 37])
@pytest.mark.parametrize("block,dtype", [(64, torch.bfloat16), (1024, torch.float32)])
def test_both_column_counts(n, block, dtype):
    import paper_2505_06653_b200 as bof4
    code = bof4.BF16 if dtype == torch.bfloat16 else bof4.F32
    gen = torch.Generator(device="cuda")
    gen.manual_seed(n & 0xffff)
    codes = torch.randint(0, 256, ((n + 1) // 2,), dtype=torch.uint8, device="cuda", generator=gen)
    scales = (torch.rand((n + block - 1) // block, device="cuda", generator=gen) + 0.5).to(dtype)
    levels = torch.linspace(-0.9, 1.0, 16, device="cuda")
    out = bof4.bof4_dequantize(codes, scales, block, levels, code, n=n)
    for a in range(0, n, PIECE):
        m = min(PIECE, n - a)
        piece = bof4.bof4_dequantize(codes[a // 2:(a + m + 1) // 2], scales[a // block:(a + m + block - 1) // block], block, levels, code, n=m)
        assert torch.equal(out[a:a + m], piece)
