"""The streaming squared-error pass on weights of any magnitude: m^2 is kept in units that follow the data."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

LV = np.array(workloads.BOF4S_MSE_I64, np.float32)


@pytest.fixture(scope="module")
def bof4():
    import __graft_entry__ as entry
    entry.build()
    import paper_2505_06653_b200 as m
    assert torch.cuda.is_available()
    return m


def _weights(kind, n, dtype):
    w = workloads.gaussian(n, 1.0, 17, torch.float32)
    blocks = (n + 63) // 64
    if kind == "mixed":          # constants over forty binades, block by block
        w *= torch.exp2(torch.randint(-20, 20, (blocks,), generator=torch.Generator().manual_seed(1)).float()).repeat_interleave(64)[:n]
    elif kind == "growing":      # a thread meets ever larger ones: its unit has to change
        w *= torch.exp2(torch.linspace(-120, 120, blocks)).repeat_interleave(64)[:n]
    elif kind == "shrinking":
        w *= torch.exp2(torch.linspace(120, -120, blocks)).repeat_interleave(64)[:n]
    elif kind == "zeros first":
        w[: n // 2] = 0.0
        w *= 1e-21
    else:
        w *= float(kind)
    return w.to(dtype)


@pytest.mark.parametrize("kind", ["1e-43", "1e-38", "1e-25", "1e-19", "0.02", "1e19", "1e30", "3e37", "mixed", "growing", "shrinking",
                                  "zeros first"])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("metric", [0, 2])
def test_squares_neither_underflow_nor_overflow(bof4, kind, dtype, metric):
    w = _weights(kind, (1 << 19) + 40, dtype)
    dev = [w.cuda()]
    if metric == 0:
        st, got = oracle.em_accumulate_mse(w, 64, 1, LV), bof4.bof4_em_step(dev, 64, 1, metric, LV)
        assert np.array_equal(got["count"], st["count"])
        np.testing.assert_allclose(got["s0"], st["s0"], rtol=1e-5)
        np.testing.assert_allclose(got["s1"], st["s1"], rtol=1e-5, atol=1e-6 * np.abs(st["s1"]).max())
        np.testing.assert_allclose(got["err_sum"], st["err_sum"], rtol=1e-5)
    for iters in (1, 3):
        ref, ref_log = oracle.fit([w], 64, 1, metric, LV, 0x8080, iters)
        ws = torch.empty(bof4.bof4_workspace_bytes(bof4.OP_EM, 0, 64, metric), dtype=torch.uint8, device="cuda")
        cb, log = bof4.bof4_fit_codebook(dev, 64, 1, metric, LV, 0x8080, iters, workspace=ws)
        np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=1e-5, atol=1e-7)
        np.testing.assert_allclose(log.cpu().numpy(), ref_log, rtol=1e-5)


def test_a_larger_workspace_makes_no_median_slower(bof4):
    """2^24 weights of sixteen levels: candidate lists as long as a workspace of 16 bytes per weight would hold are never filled."""
    g = torch.Generator().manual_seed(3)
    n = 1 << 24
    q = torch.randint(-7, 9, (n // 64, 64), generator=g).float()
    q[:, 0] = 8
    w = (q * torch.rand(n // 64, 1, generator=g) * 0.01).reshape(-1).cuda()
    lv, mask = bof4.bof4_default_init(0)
    ms = []
    for nbytes in (bof4.bof4_workspace_bytes(bof4.OP_EM, n, 64, 1), 16 * n):
        ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        best = 1e9
        for _ in range(3):
            s, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            s.record()
            bof4.bof4_fit_codebook(w, 64, 0, 1, lv, mask, 2, workspace=ws, sync=False)
            e.record()
            torch.cuda.synchronize()
            best = min(best, s.elapsed_time(e))
        ms.append(best)
    assert ms[1] < 2 * ms[0], ms
