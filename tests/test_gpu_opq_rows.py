"""The outlier pass where its row-wise decisions could go wrong: weights at and around the threshold, blocks that the
threshold's interval cannot bound, rows in which every lane holds a candidate, the length at which the list's
positions are found another way, and the count's way back to the host."""
import threading

import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

LV = np.array(workloads.init_levels_7_0_8(), np.float32)


@pytest.fixture(scope="module")
def bof4():
    import __graft_entry__ as entry
    entry.build()
    import paper_2505_06653_b200 as m
    assert torch.cuda.is_available()
    return m


def _data(kind, n, I, rng):
    w = rng.standard_normal(n).astype(np.float32)
    tau = 2.5
    if kind == "at_threshold":      # two magnitudes a block: many weights within one bf16 step of sigma * tau
        w = np.where(rng.random(n) < 0.15, 2.0, 1.0).astype(np.float32) * np.where(rng.random(n) < 0.5, -1, 1)
        v = w[:I].astype(np.float64)
        tau = 2.0 / float(np.std(v, ddof=1))
    elif kind == "large_mean":      # the sum of squares is nearly all mean
        w += 30.0
        tau = 20.0
    elif kind == "mixed":           # zero, tiny, huge and ordinary blocks side by side
        s = rng.choice([0.0, 1e-38, 1e-30, 1.0, 1e18, 1e37], n // I)
        w *= np.repeat(s, I).astype(np.float32)
    elif kind == "crowded":         # more outliers than a tile's staging slots, in every lane
        w[rng.random(n) < 0.2] *= 8.0
        tau = 1.0
    return torch.from_numpy(w).to(torch.bfloat16), float(np.float32(tau))


@pytest.mark.parametrize("kind", ["at_threshold", "large_mean", "mixed", "crowded"])
@pytest.mark.parametrize("I", [32, 64, 1024, 4096])
def test_rows_that_need_care(bof4, kind, I):
    rng = np.random.default_rng(I)
    for n in (I * 3, 12288 // I * I + I, 12288 * 300):
        n = n // I * I
        w, tau = _data(kind, n, I, rng)
        clean, ridx, rval, rk = oracle.opq_split(w, I, tau)
        for norm in (0, 1):
            codes, scales, idx, val, cnt = bof4.bof4_quantize_opq(w.cuda(), I, norm, LV, tau, n)
            rc, rs = oracle.quantize(clean, I, norm, LV)
            assert bof4.bof4_outlier_count(cnt, n) == rk, (n, norm)
            assert np.array_equal(idx[:rk].cpu().numpy().astype(np.int64), ridx), (n, norm)
            assert np.array_equal(val[:rk].view(torch.int16).cpu().numpy().view(np.uint16), rval), (n, norm)
            assert np.array_equal(codes.cpu().numpy(), rc), (n, norm)
            assert np.array_equal(scales.float().cpu().numpy(), rs), (n, norm)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("n", [1 << 23, (1 << 23) + 512, (1 << 23) + (1 << 18) + 64])
def test_list_positions_at_the_chunk_limit(bof4, dtype, n):
    w = workloads.gaussian(n, 0.02, 5, dtype)
    tau = float(np.float32(bof4.bof4_opq_threshold(0.9, 64)))
    _, ridx, rval, rk = oracle.opq_split(w, 64, tau)
    _, idx, val, cnt = bof4.opq_split(w.cuda(), 64, tau, n // 16)
    assert bof4.bof4_outlier_count(cnt, n // 16) == rk
    assert np.array_equal(idx[:rk].cpu().numpy().astype(np.int64), ridx)
    assert np.array_equal(val[:rk].view(torch.int16).cpu().numpy().view(np.uint16), rval)


@pytest.mark.parametrize("threads", [4, 80])    # fewer and more than the slots that wait for a count
def test_counts_read_by_many_threads(bof4, threads):
    counts = [torch.full((1,), 1000 + k, dtype=torch.int64, device="cuda") for k in range(threads)]
    got = [None] * threads
    torch.cuda.synchronize()

    def read(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            got[k] = [bof4.bof4_outlier_count(counts[k], 1 << 20) for _ in range(50)]

    pool = [threading.Thread(target=read, args=(k,)) for k in range(threads)]
    for t in pool:
        t.start()
    for t in pool:
        t.join()
    assert got == [[1000 + k] * 50 for k in range(threads)]
