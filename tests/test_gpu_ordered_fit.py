"""Fits of enough iterations, which put the samples in order once: one sample per weight (fp32,
small bf16) and one per distinct normalised weight (bf16 from 3 * 2^19 weights), against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bof4():
    import __graft_entry__ as entry
    entry.build()
    import paper_2505_06653_b200 as m
    assert torch.cuda.is_available()
    return m


def _weights(n, dtype, seed, kind):
    w = workloads.gaussian(n, 0.02, seed, torch.float32)
    g = torch.Generator().manual_seed(seed + 1)
    if kind == "sparse":       # many exact zeros
        w *= (torch.rand(n, generator=g) < 0.3)
    elif kind == "grid":       # few distinct values
        w = torch.round(w * 200) / 200
    elif kind == "scales":     # block constants over sixty binades
        w *= torch.exp2(torch.randint(-30, 30, ((n + 63) // 64,), generator=g).float()).repeat_interleave(64)[:n]
    elif kind == "subnormal":  # bf16 weights below the normal range
        w *= 1e-37
    return w.to(dtype)


def _check(bof4, ws, I, norm, metric, iters, mask=None):
    lv, m = bof4.bof4_default_init(norm)
    mask = m if mask is None else mask
    dev = [w.cuda() for w in ws]
    cb, log = bof4.bof4_fit_codebook(dev, I, norm, metric, lv, mask, iters)
    again, log2 = bof4.bof4_fit_codebook(dev, I, norm, metric, lv, mask, iters)
    assert torch.equal(cb, again) and torch.equal(log, log2)
    ref, ref_log = oracle.fit(ws, I, norm, metric, lv, mask, iters)
    if metric == bof4.METRIC_MAE:
        assert np.array_equal(cb.cpu().numpy(), ref)
    else:
        np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=1e-5, atol=1e-7)
    np.testing.assert_allclose(log.cpu().numpy(), ref_log, rtol=1e-5, atol=1e-12)


@pytest.mark.parametrize("sizes", [(1,), (31,), (129,), (4096, 33), (8192 * 148 + 5,), (1 << 20, 70001)])
@pytest.mark.parametrize("metric", [0, 1])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_one_sample_per_weight(bof4, sizes, metric, dtype):
    """Lengths around the edges of warps, chunks and tiles of the ordering passes."""
    _check(bof4, [_weights(n, dtype, 100 + k, "plain") for k, n in enumerate(sizes)], 64, sum(sizes) % 2, metric, 4)


@pytest.mark.parametrize("n,I,kind,mask", [((1 << 22), 64, "plain", None), ((1 << 22) + 37, 32, "sparse", 0),
                                           ((1 << 22) + 4095, 4096, "grid", 0), ((1 << 22) + 64, 64, "scales", None),
                                           ((1 << 22) + 1, 1024, "subnormal", None)])
@pytest.mark.parametrize("metric", [0, 1])
@pytest.mark.parametrize("norm", [0, 1])
def test_one_sample_per_distinct_weight(bof4, n, I, kind, mask, metric, norm):
    _check(bof4, [_weights(n, torch.bfloat16, 7, kind)], I, norm, metric, 4, mask)


@pytest.mark.parametrize("sizes", [(8192 * 148 + 5,), (1 << 20, 70001)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_one_sample_per_weight_long(bof4, sizes, dtype):
    """Sizes from which a few iterations are streamed, with more of them."""
    _check(bof4, [_weights(n, dtype, 200 + k, "plain") for k, n in enumerate(sizes)], 64, 1, 0, 10)


@pytest.mark.parametrize("n,I,kind,mask", [((1 << 22), 64, "plain", None), ((1 << 22) + 37, 32, "sparse", 0),
                                           ((1 << 22) + 4095, 4096, "grid", 0), ((1 << 22) + 64, 64, "scales", None),
                                           ((1 << 22) + 1, 1024, "subnormal", None), ((3 << 19), 64, "plain", None)])
@pytest.mark.parametrize("norm", [0, 1])
def test_one_sample_per_distinct_weight_long(bof4, n, I, kind, mask, norm):
    _check(bof4, [_weights(n, torch.bfloat16, 7, kind)], I, norm, 0, 8, mask)


def test_many_tensors_long(bof4):
    ws = [_weights(70000 + 13 * k, torch.bfloat16, k, "plain") for k in range(66)]
    _check(bof4, ws, 128, 0, 0, 8)


@pytest.mark.parametrize("dtype,n,metric,iters", [(torch.float32, 1 << 20, 0, (5, 6)), (torch.float32, 1 << 21, 0, (7, 8)),
                                                  (torch.float32, 1 << 23, 1, (6, 7)), (torch.bfloat16, 1 << 21, 0, (5, 6)),
                                                  (torch.float32, 1 << 23, 0, (12, 13)), (torch.float32, 1 << 24, 0, (16, 17)),
                                                  (torch.float32, 1 << 24, 1, (8, 9)), (torch.float32, 1 << 25, 0, (19, 20))])
def test_both_sides_of_the_switch_over(bof4, dtype, n, metric, iters):
    """One iteration apart, one fit is streamed and the other ordered; the same oracle."""
    from paper_2505_06653_b200 import binding as b
    dt = b.F32 if dtype == torch.float32 else b.BF16
    a, z = (b.bof4_fit_workspace_bytes(n, dt, 64, metric, it) for it in iters)
    assert a < z
    for it in iters:
        _check(bof4, [_weights(n, dtype, 9, "plain")], 64, 0, metric, it)


def test_converged_fit_fills_the_rest_of_the_log(bof4):
    """Three distinct magnitudes: the levels settle at once, and every further entry is the same."""
    w = torch.tensor([1.0, -0.5, 0.25, 0.0] * 4096)
    _check(bof4, [w], 64, 0, 0, 50)


def test_many_tensors(bof4):
    """More tensors than one launch takes, with and without short last blocks."""
    ws = [_weights(70000 + 13 * k, torch.bfloat16, k, "plain") for k in range(70)]
    _check(bof4, ws, 128, 1, 1, 4)
    _check(bof4, ws[:66], 128, 0, 0, 4)


@pytest.mark.parametrize("n", [300, (1 << 20) + 9, 1 << 23])
@pytest.mark.parametrize("kind", ["plain", "grid", "sparse"])
@pytest.mark.parametrize("metric", [0, 1])
def test_thresholds_in_one_bin(bof4, n, kind, metric):
    """Levels so close that several thresholds cut the same bin, a threshold that is exactly zero, regions that
    stay empty, and bins of one, two and many rounds of samples."""
    w = _weights(n, torch.float32, 5, kind)
    lv = np.array([-1.0, -0.4, -0.2000002, -0.2000001, -0.2, -0.1, -0.01, 0.01, 0.1, 0.25, 0.2500001, 0.2500002, 0.2500003, 0.7,
                   0.99999994, 1.0], np.float32)
    cb, log = bof4.bof4_fit_codebook([w.cuda()], 64, 0, metric, lv, 0x8001, 6)
    ref, ref_log = oracle.fit([w], 64, 0, metric, lv, 0x8001, 6)
    if metric == bof4.METRIC_MAE:
        assert np.array_equal(cb.cpu().numpy(), ref)
    else:
        np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=1e-5, atol=1e-7)
    np.testing.assert_allclose(log.cpu().numpy(), ref_log, rtol=1e-5, atol=1e-12)


@pytest.mark.parametrize("n", [(3 << 19) - 1, 3 << 19, (3 << 19) + 4097])
@pytest.mark.parametrize("metric", [0, 1])
def test_length_from_which_samples_are_distinct_weights(bof4, n, metric):
    _check(bof4, [_weights(n, torch.bfloat16, 3, "plain")], 64, 1, metric, 4)


@pytest.mark.parametrize("metric", [0, 1, 2, 3])
def test_zeros_alone(bof4, metric):
    """No weight counts under the metrics of the weights: there is not a single sample, and the levels stay."""
    _check(bof4, [torch.zeros((3 << 19) + 70, dtype=torch.bfloat16)], 64, 0, metric, 12)
    _check(bof4, [torch.zeros(70000, dtype=torch.float32)], 64, 1, metric, 12)


def _crowded(n, kind, seed):
    """fp32 weights whose blocks of 64 start with a one (x is the weight itself) and that share few bins of x, with levels
    whose thresholds lie among them."""
    g = torch.Generator().manual_seed(seed)
    u = torch.rand(n, generator=g)
    if kind == "grid":         # sixteenths: every other threshold is one of the values
        w, lv = torch.round(32 * u - 16) / 16, np.linspace(-1, 1, 16)
    elif kind == "jitter":     # a few neighbouring values in every crowded bin
        w, lv = torch.round(16 * u - 8) / 8 * (1 + torch.randint(0, 4, (n,), generator=g) * 2.0 ** -23), np.linspace(-1, 1, 16)
    elif kind == "octave":     # everything in two bins, all thresholds as well
        w, lv = 2.0 ** -10 * (1 + 0.2 * u), 2.0 ** -10 * (1 + np.arange(16) / 80)
    else:                      # "tiny": the outermost bins on either side of zero
        w, lv = (u - 0.5) * 2.0 ** -39, (np.arange(16) - 7.5) * 2.0 ** -43
    w[::64] = 1.0
    return w, lv.astype(np.float32)


@pytest.mark.parametrize("n", [4096 + 64, 8192 * 2 + 5, 70001, (1 << 20) + 77])
@pytest.mark.parametrize("kind", ["grid", "jitter", "octave", "tiny"])
@pytest.mark.parametrize("metric", [0, 1, 2, 3])
def test_crowded_bins(bof4, n, kind, metric):
    """Bins of more samples than are looked through: windows put in full order and searched."""
    w, lv = _crowded(n, kind, 11)
    iters = 12
    dev = [w.cuda()]
    cb, log = bof4.bof4_fit_codebook(dev, 64, 0, metric, lv, 0x8000, iters)
    again, log2 = bof4.bof4_fit_codebook(dev, 64, 0, metric, lv, 0x8000, iters)
    assert torch.equal(cb, again) and torch.equal(log, log2)
    ref, ref_log = oracle.fit([w], 64, 0, metric, lv, 0x8000, iters)
    if metric in (1, 3):
        assert np.array_equal(cb.cpu().numpy(), ref)
    else:
        np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=1e-5)
    # the squared error is the difference of two sums: their rounding, 2^-50 of the sum of squares, is what remains of it
    np.testing.assert_allclose(log.cpu().numpy(), ref_log, rtol=1e-5, atol=2.0 ** -50 * float((w.double() ** 2).mean()))


def _best_ms(bof4, w, lv, mask, metric, iters):
    """Time of a fit, with the launches queued behind a wait of 10 ms: the host's time is not in it, nor are its pauses, which on a shared
    machine can be longer than any fit here (85 ms were seen)."""
    room = torch.empty(bof4.bof4_fit_workspace_bytes(w.numel(), bof4.F32, 64, metric, iters), dtype=torch.uint8, device="cuda")
    best = 1e9
    for _ in range(9):
        s, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda._sleep(20_000_000)
        s.record()
        bof4.bof4_fit_codebook(w, 64, 0, metric, lv, mask, iters, workspace=room, sync=False)
        e.record()
        torch.cuda.synchronize()
        best = min(best, s.elapsed_time(e))
    return best


def test_crowded_bins_take_bounded_time(bof4):
    """2^22 weights that have been quantised before (sixteen levels, every block with its own constant): 150 000 samples and
    more in a bin.  Looked through by one warp, a fit takes 16 ms (medians) and streaming the data 14."""
    g = torch.Generator().manual_seed(3)
    n = 1 << 22
    q = torch.randint(-7, 9, (n // 64, 64), generator=g).float()
    q[:, 0] = 8
    w = (q * torch.rand(n // 64, 1, generator=g) * 0.01).reshape(-1).cuda()
    lv, mask = bof4.bof4_default_init(0)
    for metric in (0, 1):
        best = _best_ms(bof4, w, lv, mask, metric, 32)
        assert best < 5.0, (metric, best)


@pytest.mark.parametrize("tail", [0, 37])
@pytest.mark.parametrize("unit", [1.0, 2.0 ** -80])
@pytest.mark.parametrize("metric", [0, 1, 2, 3])
def test_normalised_weights_near_zero_keep_their_sign(bof4, tail, unit, metric):
    """Weights below 2^-40 of their block's constant, of either sign, and a threshold that is exactly zero: which side they
    fall on decides the levels beside it.  Their magnitude is known to a factor of two, which is 2^-40 absolute."""
    n = (1 << 21) + tail
    w = workloads.gaussian(n, 0.02, 21, torch.float32)
    g = torch.Generator().manual_seed(22)
    small = torch.rand(n, generator=g) < 0.4
    sign = torch.where(torch.rand(n, generator=g) < 0.8, -1.0, 1.0)
    w = (torch.where(small, sign * 1e-15 * (0.5 + torch.rand(n, generator=g)), w) * unit).to(torch.bfloat16)
    lv = np.linspace(-1, 1, 16).astype(np.float32)
    cb, log = bof4.bof4_fit_codebook(w.cuda(), 64, 0, metric, lv, 0x8001, 8)
    ref, ref_log = oracle.fit([w], 64, 0, metric, lv, 0x8001, 8)
    np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=0 if metric in (1, 3) else 1e-5, atol=2.0 ** -40 if metric in (1, 3) else 1e-7)
    np.testing.assert_allclose(log.cpu().numpy(), ref_log, rtol=1e-5)


@pytest.mark.parametrize("size", [3000, 20])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("metric", [0, 1])
def test_many_small_tensors(bof4, size, dtype, metric):
    """One sample per weight of more tensors than one launch takes; of 20 weights and a few there are short blocks only.  The
    workspace holds what another fit has left."""
    ws = [_weights(size + 13 * k % 11, dtype, k, "plain") for k in range(140)]
    n = sum(w.numel() for w in ws)
    lv, mask = bof4.bof4_default_init(0)
    room = torch.empty(bof4.bof4_fit_workspace_bytes(1 << 20, bof4.F32, 64, metric, 100), dtype=torch.uint8, device="cuda")
    bof4.bof4_fit_codebook(_weights(1 << 20, torch.float32, 1, "grid").cuda() * 1e9, 64, 0, metric, lv, mask, 9, workspace=room)
    cb, log = bof4.bof4_fit_codebook([w.cuda() for w in ws], 64, 0, metric, lv, mask, 9, workspace=room)
    ref, ref_log = oracle.fit(ws, 64, 0, metric, lv, mask, 9)
    assert n < 1 << 20
    if metric == bof4.METRIC_MAE:
        assert np.array_equal(cb.cpu().numpy(), ref)
    else:
        np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=1e-5, atol=1e-7)
    np.testing.assert_allclose(log.cpu().numpy(), ref_log, rtol=1e-5, atol=1e-12)


def _light(n, light, seed):
    """fp32 weights whose blocks of 64 start with their constant: a region of `light` samples whose blocks are 2^-20 of the others', and
    beside it, in the same bins of x or the next ones, the others' samples; seen from every other level it is nothing."""
    g = torch.Generator().manual_seed(seed)
    u = torch.rand(n // 64, 64, generator=g)
    x = torch.where(torch.rand(n // 64, 64, generator=g) < 0.5, 0.49992 + 3e-5 * u, 0.50006 + 3e-5 * u)
    x[:light] = 0.49998 + 5e-5 * u[:light]
    x[:, 0] = 1.0
    m = torch.ones(n // 64, 1)
    m[:light] = 2.0 ** -20
    lv = np.array([-1, -0.5, -0.4, -0.3, -0.2, -0.1, 0, 0.1, 0.2, 0.3, 0.4, 0.4999, 0.50001, 0.5001, 0.7, 1], np.float32)
    return (x * m).reshape(-1), lv


@pytest.mark.parametrize("n,light", [(64 * 300, 1), (1 << 16, 40)])
def test_a_region_that_is_light_beside_its_neighbours(bof4, n, light):
    """Its weight is 2^-40 of what lies in front of it in its group of bins: as the difference of two sums of doubles its level
    would be off by 1e-3 and more."""
    w, lv = _light(n, light, 31)
    cb, log = bof4.bof4_fit_codebook(w.cuda(), 64, 0, 0, lv, 0xffff ^ (1 << 12), 8)
    ref, ref_log = oracle.fit([w], 64, 0, 0, lv, 0xffff ^ (1 << 12), 8)
    assert ref[12] != lv[12]
    np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=1e-7)
    np.testing.assert_allclose(log.cpu().numpy(), ref_log, rtol=1e-5)


def test_an_infinite_weight_reaches_no_other_region(bof4):
    """Its block counts as zeros of infinite weight and one weight that is not a number: the fixed levels' regions."""
    w = _weights(1 << 16, torch.float32, 17, "plain")
    w[(1 << 15) + 5] = float("inf")
    lv, mask = bof4.bof4_default_init(0)
    cb, _ = bof4.bof4_fit_codebook(w.cuda(), 64, 0, 0, lv, mask, 8)
    w[1 << 15:][:64] = 0
    ref, _ = oracle.fit([w], 64, 0, 0, lv, mask, 8)
    np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=1e-5)


@pytest.mark.parametrize("each", [31, 32, 33, 63, 64, 65, 127, 129, 700])
def test_median_among_the_samples_of_one_bin(bof4, each):
    """`each` samples in every occupied bin, near the sizes at which they are looked through in another way; equal samples among
    them, and medians that lie at the first and the last of a bin."""
    g = torch.Generator().manual_seed(each)
    bins = 90
    x = (torch.arange(bins).repeat_interleave(each) * 137 + 800 + (0.05 + 0.9 * torch.rand(bins * each, generator=g))) / 32566
    x = torch.where(torch.rand(x.numel(), generator=g) < 0.2, x.roll(1), x)[torch.randperm(x.numel(), generator=g)]
    x = x[:x.numel() // 31 * 31].view(-1, 31)
    w = torch.cat([torch.ones(len(x), 1), x, x.neg().flip(0)], 1)
    w = torch.nn.functional.pad(w, (0, 1)) * (0.5 + torch.rand(len(x), 1, generator=g))
    _check(bof4, [w.reshape(-1)], 64, 0, bof4.METRIC_MAE, 12)


def test_a_light_region_among_distinct_weights(bof4):
    """The same for bf16 data: quotients near one half of blocks that are 2^-20 of the others', whose own lie just beside the region."""
    n, light = 1 << 21, 200
    g = torch.Generator().manual_seed(5)
    x = torch.where(torch.rand(n // 64, 64, generator=g) < 0.5, 255 / 512, 129 / 256)
    m = torch.ones(n // 64, 1)
    m[:light] = 2.0 ** -20 * (1 + torch.randint(0, 128, (light, 1), generator=g) / 128)
    x[:light] = 0.5005
    x[:, 0] = 1.0
    w = (x * m).to(torch.bfloat16).reshape(-1)
    lv = np.array([-1, -0.5, -0.4, -0.3, -0.2, -0.1, 0, 0.1, 0.2, 0.3, 0.4, 0.498, 0.5004, 0.5039, 0.7, 1], np.float32)
    cb, log = bof4.bof4_fit_codebook(w.cuda(), 64, 0, 0, lv, 0xffff ^ (1 << 12), 8)
    ref, ref_log = oracle.fit([w], 64, 0, 0, lv, 0xffff ^ (1 << 12), 8)
    assert ref[12] != lv[12]
    np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=1e-7)
    np.testing.assert_allclose(log.cpu().numpy(), ref_log, rtol=1e-5)


def _absolute_error(w, lv, I=64):
    """Mean of |m| |x - level| over the weights (whole blocks), absolute normalisation, and the mean of |w|, in long double."""
    b = w.float().numpy().reshape(-1, I)
    m = np.abs(b).max(1, keepdims=True)
    x = np.divide(b, m, out=np.zeros_like(b), where=m > 0)
    lv = np.asarray(lv, np.float32)
    level = lv[np.searchsorted((lv[:-1] + lv[1:]) * np.float32(0.5), x, side="right")]
    m = m.astype(np.longdouble)
    n = np.longdouble(b.size)
    return (np.abs(x.astype(np.longdouble) - level) * m).sum() / n, (np.abs(x.astype(np.longdouble)) * m).sum() / n


@pytest.mark.parametrize("n,dtype", [(1 << 14, torch.float32), (1 << 18, torch.float32), (1 << 20, torch.float32), (1 << 21, torch.bfloat16)])
@pytest.mark.parametrize("kind", ["plain", "levels"])
def test_the_absolute_error_is_added_up_by_regions(bof4, n, dtype, kind):
    """The logged error against sums in long double.  A half region is the difference of two sums in two doubles each, so what is
    left is the rounding of the halves, 2^-53 of each and of random sign: less than 2^-53 of the mean of |w| in all.  (As 32 differences
    of sums over all the data, each in one double, it would be 2^-51 to 2^-50.)  "levels": most weights lie on one."""
    lv, _ = bof4.bof4_default_init(0)
    for seed in range(4):
        w = _weights(n, torch.float32, 40 + seed, "plain")
        if kind == "levels":
            g = torch.Generator().manual_seed(seed)
            w = torch.randint(-1, 9, (n // 64, 64), generator=g).float() / 8
            w = torch.where(w < 0, -1.0, w)
            w[:, 0] = 1.0
            w = (w * (0.5 + torch.rand(n // 64, 1, generator=g))).reshape(-1)
        w = w.to(dtype)
        _, log = bof4.bof4_fit_codebook(w.cuda(), 64, 0, bof4.METRIC_MAE, lv, 0xffff, 12)
        ref, mean = _absolute_error(w, lv)
        assert abs(log[0].item() - ref) <= 2.0 ** -53 * mean, (seed, float((log[0].item() - ref) / mean))
        assert (log == log[0]).all()


def _iteration_us(bof4, w, lv, mask, metric):
    """100 iterations less 20."""
    return (_best_ms(bof4, w, lv, mask, metric, 100) - _best_ms(bof4, w, lv, mask, metric, 20)) / 80 * 1000


@pytest.mark.parametrize("mask", [0x81c1, 0x8141])
def test_a_level_at_zero_costs_what_others_do(bof4, mask):
    """Data that is symmetric about zero, and thresholds that are too: the weighted sum of the region around zero cancels.  An iteration
    takes 1.1 us with any levels; with this region added up by itself it took 2.5, with that level fixed or free."""
    h = _weights(1 << 19, torch.float32, 23, "plain")
    w = torch.cat([h, -h]).cuda()
    lv = np.array([-1, -.75, -.58, -.44, -.32, -.2, -.1, 0, .1, .2, .3, .4, .5, .63, .8, 1], np.float32)
    other = lv.copy()
    other[8] = 0.11
    assert _iteration_us(bof4, w, lv, mask, 0) < 1.35 * _iteration_us(bof4, w, other, 0x81c1, 0)


def _halfway(dtype, seed):
    """Weights with a region of which the level lies exactly halfway between two floats, and sums are exact if they are added up by
    themselves: its blocks' constant is a power of two.  Its weight is 2^-18 of what lies below it in the same group of bins (of
    places), where constants are arbitrary and sums are rounded.  Returns the weights, the levels, the free level's index and value."""
    g = torch.Generator().manual_seed(seed)
    lv = np.linspace(-1, 1, 16).astype(np.float32)
    if dtype == torch.float32:
        u = torch.rand(64, 64, generator=g)
        w = torch.where(torch.rand(64, 64, generator=g) < 0.5, 0.49991 + 2e-5 * u, 0.50007 + 2e-5 * u)
        w[:, 0] = 1.0
        w *= 0.5 + 0.5 * torch.rand(64, 1, generator=g)
        a = np.float32(0.49999) + np.float32(2.0 ** -24) * np.float32(seed)
        b = np.nextafter(a, np.float32(1))
        lv[10:14] = 0.4, 0.4999, 0.50001, 0.5001
        x = torch.zeros(64 * 63)
        x[:1999], x[1999:2 * 1999] = float(a), float(b)     # (the sums have bits that the others' are rounded by)
        light = torch.cat([torch.ones(64, 1), x.view(64, 63)], 1)
        return torch.cat([w, light * 2.0 ** -10]).reshape(-1), lv, 12, np.float32((np.float64(a) + np.float64(b)) / 2)
    blocks, samples = 2081, 1 << 17
    m = torch.randint(192, 256, ((1 << 15) - blocks, 1), generator=g).float()
    w = torch.where(torch.rand(len(m), 64, generator=g) < 0.5, (m - 1) / 2, m / 8)    # (m - 1) / 2 m: from 0.4973 to 0.498
    w[:, :1] = m
    w /= 256
    high = 2 * int(torch.randint(1 << 13, 1 << 15, (1,), generator=g)) + 1
    x = torch.zeros(blocks * 63)
    x[:samples] = 0.5
    x[:high] = 129 / 256
    light = torch.cat([torch.ones(blocks, 1), x[torch.randperm(len(x), generator=g)].view(blocks, 63)], 1)
    lv[10:14] = 0.4, 0.498, 0.5005, 0.51
    return torch.cat([w, light * 2.0 ** -8]).to(dtype).reshape(-1), lv, 12, np.float32(0.5 + high * 2.0 ** -25)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_a_light_region_is_as_exact_as_by_itself(bof4, dtype):
    """As the difference of rounded sums its level would be off by 2^-34, which decides to which side a level halfway between two
    floats is rounded: to the even one if it is exact."""
    for seed in range(16):
        w, lv, free, level = _halfway(dtype, seed)
        cb, _ = bof4.bof4_fit_codebook(w.cuda(), 64, 0, 0, lv, 0xffff ^ (1 << free), 8)
        assert cb[free].item() == level, seed


def test_a_median_in_a_crowded_bin_is_looked_for_between_its_thresholds(bof4):
    """2^20 weights about zero, all thresholds in the outermost bins of it: 18 iterations 1.8 ms.  Among all samples of a bin, whose keys
    span fourteen binades, and from nowhere in particular, they took 3.4."""
    w, lv = _crowded(1 << 20, "tiny", 11)
    assert _best_ms(bof4, w.cuda(), lv, 0x8000, bof4.METRIC_MAE, 18) < 2.6


def _few_values(dtype, seed):
    """Blocks of 64 with one of 24 constants of any significand and twelve weights of its own, from 2^-45 of it on (powers of two below
    2^-40), zeros and the constant's own size among them: a few hundred normalised weights, so that one on the wrong side of a threshold
    shows.  Returns the weights and, by ascending x: x, sum of m^2, sum of |m|."""
    rng = np.random.default_rng(seed)
    blocks = (3 << 19) // 64 if dtype == torch.bfloat16 else 1 << 11
    sig = rng.integers(128, 256, 24)
    m = sig * 2.0 ** rng.integers(-9, -6, 24)
    d = (rng.uniform(0, 45, (24, 12)) ** 1.5 / 45 ** 0.5 * 128).astype(int)       # distances of the bit patterns, small ones more often
    e, a = -(-(d - sig[:, None] + 128) // 128), (sig[:, None] - 128 - d) % 128 + 128
    w = np.where(d < 5120, m[:, None] * (a / sig[:, None]) * 2.0 ** -e, m[:, None] * 2.0 ** -(d // 128))
    w[:, 0], w[:, 1] = 0.0, -m
    w[:, 2:] *= rng.choice([-1, 1], (24, 10))
    which = rng.integers(0, 24, blocks)
    data = np.concatenate([m[which][:, None], w[which[:, None], rng.integers(0, 12, (blocks, 63))]], 1).astype(np.float32)
    assert np.array_equal(torch.from_numpy(data).to(torch.bfloat16).float().numpy(), data)
    x, at = np.unique(data / data[:, :1], return_inverse=True)
    c = np.broadcast_to(data[:, :1].astype(np.float64), data.shape).reshape(-1)
    return torch.from_numpy(data).to(dtype).reshape(-1), x, np.bincount(at.reshape(-1), c * c), np.bincount(at.reshape(-1), c)


def _lloyd(x, s, lv, metric, iters, n):
    """By the definition: a region is what lies between its thresholds, and nothing where they do not ascend."""
    lv, log = lv.copy(), []
    for _ in range(iters):
        t = (lv[:-1] + lv[1:]) * np.float32(0.5)
        lo, hi = np.append(np.float32(-np.inf), t), np.append(t, np.float32(np.inf))
        new, err = lv.copy(), 0.0
        for k in range(16):
            i = (x >= lo[k]) & (x < hi[k])
            v, u = s[i], x[i].astype(np.float64)
            d = np.abs(u - np.float64(lv[k]))
            err += (v * (d if metric == 1 else d * d)).sum()
            if v.sum() > 0:
                new[k] = x[i][np.argmax(2 * np.cumsum(v) >= v.sum())] if metric == 1 else np.float32((v * u).sum() / v.sum())
        log.append(err / n)
        lv = new
    return lv, np.array(log)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("metric", [0, 1])
@pytest.mark.parametrize("ascend", [True, False])
def test_thresholds_at_the_samples(bof4, dtype, metric, ascend):
    """Eight thresholds of every fit are a normalised weight that occurs, the next number below it or above it; and levels that do not
    ascend, whose regions are empty (the log of the squared error is not defined for them)."""
    for seed in range(4):
        w, x, m2, m1 = _few_values(dtype, seed)
        dev, rng = w.cuda(), np.random.default_rng(100 + seed)
        inside = x[(np.abs(x) < 0.99)]
        for _ in range(12):
            p = np.sort(rng.choice(inside[np.abs(inside) > 2.0 ** -60], 8, replace=False))
            p = np.where(rng.random(8) < 0.34, p, np.nextafter(p, np.where(rng.random(8) < 0.5, -9, 9).astype(np.float32)))
            step = np.spacing(np.abs(p)) * 2
            step = np.where(((p - step) + (p + step)) * np.float32(0.5) == p, step, step * np.float32(1.5))     # (beside a power of two)
            lv = np.stack([p - step, p + step], 1).reshape(-1)
            assert np.array_equal((lv[::2] + lv[1::2]) * np.float32(0.5), p)
            if not ascend:
                k = rng.choice(15, 3, replace=False)
                lv[k], lv[k + 1] = lv[k + 1].copy(), lv[k].copy()
                lv[rng.integers(1, 16)] = lv[rng.integers(0, 15)]
            ref, ref_log = _lloyd(x, m1 if metric == 1 else m2, lv, metric, 6, w.numel())
            cb, log = bof4.bof4_fit_codebook(dev, 64, 0, metric, lv, 0, 6)
            if metric == 1:
                assert np.array_equal(cb.cpu().numpy(), ref)
            else:
                np.testing.assert_allclose(cb.cpu().numpy(), ref, rtol=2e-7, atol=1e-30)
            if metric == 1 or ascend:
                np.testing.assert_allclose(log.cpu().numpy(), ref_log, rtol=1e-9, atol=2.0 ** -50 * float((m1 if metric == 1 else m2).sum()) / w.numel())


@pytest.mark.parametrize("metric", [0, 1])
def test_few_weights_take_no_longer_than_many(bof4, metric):
    """1000 weights leave most bins empty: finding the bins' first samples took longer than all else was shorter (86 us against 71; 66 now,
    and 8 % are left for the clocks)."""
    lv, mask = bof4.bof4_default_init(0)
    few, many = (_best_ms(bof4, _weights(n, torch.float32, 3, "plain").cuda(), lv, mask, metric, 6) for n in (1000, 1 << 16))
    assert few < 1.08 * many
