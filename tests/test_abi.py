"""CPU-only checks of the C ABI: the library loads, exports every declared symbol, and the
host-side logic (argument validation, workspace sizes, host helpers) behaves as documented.
No kernel is launched here."""
import ctypes
import os
import re

import numpy as np
import pytest

import __graft_entry__ as entry
import oracle

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def L():
    entry.build()
    from paper_2505_06653_b200 import binding
    return binding.lib()


def _declared():
    src = open(os.path.join(ROOT, "include", "bof4.h")).read()
    return sorted(set(re.findall(r"^BOF4_API\s+[\w\s\*]+?\b(\w+)\s*\(", src, flags=re.M)))


def test_every_declared_symbol_is_exported(L):
    from paper_2505_06653_b200 import binding
    names = _declared()
    assert len(names) >= 10
    for name in names:
        assert hasattr(L, name), name
    assert sorted(binding.EXPORTS) == names


def test_stats_struct_size_matches_header(L):
    from paper_2505_06653_b200 import binding
    assert ctypes.sizeof(binding.EmStats) == 16 * 8 * 3 + 8 + 8 + 16 * 4


def test_opq_threshold_matches_quantile_definition(L):
    # F_M(tau) = (2 G(tau) - 1)^I = q  (App. B.1), checked through the forward formula
    from scipy.special import ndtr
    for I in (32, 64, 128, 256):
        for q in (0.9, 0.95, 0.97, 0.99):
            tau = L.bof4_opq_threshold(q, I)
            assert abs((2 * ndtr(tau) - 1) ** I - q) < 1e-12
            assert abs(tau - oracle.opq_threshold(q, I)) < 1e-10
    assert np.isnan(L.bof4_opq_threshold(1.5, 64))
    assert np.isnan(L.bof4_opq_threshold(0.5, 0))


def test_default_init(L):
    from paper_2505_06653_b200 import binding
    lv, mask = binding.bof4_default_init(binding.NORM_ABS)
    assert mask == (1 | 1 << 7 | 1 << 15)
    assert lv[0] == -1 and lv[7] == 0 and lv[15] == 1 and np.all(np.diff(lv) > 0)
    lv, mask = binding.bof4_default_init(binding.NORM_SIGNED)
    assert mask == (1 << 7 | 1 << 15)
    with pytest.raises(binding.Bof4Error):
        binding.bof4_default_init(7)


def test_workspace_sizes(L):
    from paper_2505_06653_b200 import binding as b
    assert b.bof4_workspace_bytes(b.OP_EM, 1 << 20, 64, b.METRIC_MSE) > 0
    assert b.bof4_workspace_bytes(b.OP_EM, 1 << 20, 64, 5) == 0
    assert b.bof4_workspace_bytes(b.OP_OPQ, 1 << 20, 48, 0) == 0
    assert b.bof4_workspace_bytes(b.OP_OPQ, 1 << 20, 8192, 0) == 0
    assert b.bof4_workspace_bytes(b.OP_OPQ, 1 << 20, 4096, 0) > 0
    assert b.bof4_workspace_bytes(9, 1 << 20, 64, 0) == 0
    small = b.bof4_workspace_bytes(b.OP_OPQ, 1 << 20, 64, 0)
    big = b.bof4_workspace_bytes(b.OP_OPQ, 1 << 24, 64, 0)
    assert 0 < small < big
    assert b.bof4_workspace_bytes(b.OP_OPQ, 0, 64, 0) >= 256


def test_only_a_fit_that_orders_its_samples_asks_for_room_for_them(L):
    """The E step, the joint fit and short fits stream: partial records and candidate lists, whatever the data's
    size and type.  A long fit asks for 16 bytes per fp32 weight up to 2^26, or about 64 MB and 10 bytes per block (bf16)."""
    from paper_2505_06653_b200 import binding as b
    base = b.bof4_workspace_bytes(b.OP_EM, 0, 64, b.METRIC_MSE)
    assert base < 10 << 20
    for metric in range(4):
        for n in (1, 1 << 20, 1 << 24, 1 << 26):
            assert b.bof4_workspace_bytes(b.OP_EM, n, 64, metric) == base
            for dt in (b.F32, b.BF16):
                for iters in (-1, 0, 1, 3):
                    assert b.bof4_fit_workspace_bytes(n, dt, 64, metric, iters) == base
        big = 1 << 28
        stream = b.bof4_workspace_bytes(b.OP_EM, big, 64, metric)
        assert base < stream <= base + big // 8
        assert b.bof4_fit_workspace_bytes(big, b.F32, 64, metric, 1000) == stream      # too large to order: no cell layout either
        for n in (1 << 20, 1 << 24, 1 << 26):
            assert 16 * n < b.bof4_fit_workspace_bytes(n, b.F32, 64, metric, 1000) < 17 * n + (16 << 20)
        for n in (1 << 24, 1 << 26, 1 << 30):
            cells = b.bof4_fit_workspace_bytes(n, b.BF16, 64, metric, 1000)
            assert 10 * (n // 64) + (50 << 20) < max(cells, stream) and cells <= max(10 * (n // 64) + (100 << 20), base + n // 8)
            assert b.bof4_workspace_bytes(b.OP_EM_BF16, n, 64, metric) == cells
    assert b.bof4_fit_workspace_bytes(1 << 20, 7, 64, 0, 10) == 0
    assert b.bof4_fit_workspace_bytes(1 << 20, b.F32, 48, 0, 10) == 0
    assert b.bof4_fit_workspace_bytes(1 << 20, b.F32, 64, 9, 10) == 0
    assert b.bof4_fit_workspace_bytes(-1, b.F32, 64, 0, 10) == 0


# (type, log2 of the weights, metric): iterations that are streamed, iterations that are ordered, by the times measured
ROUTES = [("f32", 20, 0, 4, 8), ("f32", 22, 0, 8, 16), ("f32", 24, 0, 16, 32), ("f32", 26, 0, 32, 60),
          ("f32", 20, 1, 3, 4), ("f32", 22, 1, 3, 4), ("f32", 24, 1, 8, 16), ("f32", 26, 1, 16, 32),
          ("bf16", 21, 0, 4, 8), ("bf16", 22, 0, 4, 8), ("bf16", 24, 0, 3, 6), ("bf16", 26, 0, 3, 4), ("bf16", 30, 0, 3, 4),
          ("bf16", 22, 1, 3, 4), ("bf16", 28, 1, 3, 4)]


@pytest.mark.parametrize("dtype,lg,metric,few,many", ROUTES)
def test_a_fit_is_ordered_where_that_is_faster(L, dtype, lg, metric, few, many):
    """The rule that picks between streaming the data and ordering it once, on either side of where the two cross (seen by
    the workspace a fit asks for)."""
    from paper_2505_06653_b200 import binding as b
    dt = b.F32 if dtype == "f32" else b.BF16
    size = lambda iters: b.bof4_fit_workspace_bytes(1 << lg, dt, 64, metric, iters)  # noqa: E731
    order = [size(it) for it in range(1, 101)]
    assert order == sorted(order)
    assert size(few) == b.bof4_workspace_bytes(b.OP_EM, 1 << lg, 64, metric)
    assert size(many) == size(1000)
    if lg < 30:      # beyond, the candidate lists of a streamed fit are larger than the cells
        assert size(many) > size(few)


# (type, log2 of the weights, metric): what ordering costs and what it gains per iteration, in us
GAINS = [("f32", 20, 0, 66, 15), ("f32", 22, 0, 156, 19), ("f32", 23, 0, 262, 25), ("f32", 24, 0, 502, 34), ("f32", 25, 0, 937, 61),
         ("f32", 26, 0, 1830, 105), ("f32", 23, 1, 264, 71), ("f32", 24, 1, 517, 90), ("f32", 25, 1, 911, 142), ("f32", 26, 1, 1814, 231),
         ("bf16", 21, 0, 43, 16), ("bf16", 24, 0, 65, 31)]


@pytest.mark.parametrize("dtype,lg,metric,cost,gain", GAINS)
def test_a_fit_is_ordered_soon_after_that_pays(L, dtype, lg, metric, cost, gain):
    """The first number of iterations that is ordered gains what ordering costs, and not more than two and a half times that."""
    from paper_2505_06653_b200 import binding as b
    dt = b.F32 if dtype == "f32" else b.BF16
    small = b.bof4_workspace_bytes(b.OP_EM, 1 << lg, 64, metric)
    first = next(it for it in range(1, 100) if b.bof4_fit_workspace_bytes(1 << lg, dt, 64, metric, it) > small)
    assert cost <= first * gain <= 2.5 * cost + gain


def test_argument_validation_happens_before_any_cuda_call(L):
    """Bad shapes / dtypes / pointers are rejected on the host with the documented codes."""
    from paper_2505_06653_b200 import binding as b
    fake = ctypes.c_void_p(0x1000)  # never dereferenced: validation fails first
    # block size and divisibility
    assert L.bof4_quantize(fake, b.BF16, 128, 48, 0, fake, fake, fake, b.BF16, None) == -2
    assert L.bof4_quantize(fake, b.BF16, 128, 8192, 0, fake, fake, fake, b.BF16, None) == -2
    assert L.bof4_quantize(fake, b.BF16, -64, 64, 0, fake, fake, fake, b.BF16, None) == -1
    # dtypes: unknown, and fp32 weights with bf16 scales
    assert L.bof4_quantize(fake, 3, 128, 64, 0, fake, fake, fake, b.BF16, None) == -3
    assert L.bof4_quantize(fake, b.F32, 128, 64, 0, fake, fake, fake, b.BF16, None) == -3
    assert L.bof4_quantize(fake, b.BF16, 128, 64, 2, fake, fake, fake, b.BF16, None) == -1
    assert L.bof4_quantize(None, b.BF16, 128, 64, 0, fake, fake, fake, b.BF16, None) == -1
    # dequantise
    assert L.bof4_dequantize(fake, fake, b.BF16, 96, 24, fake, None, None, None, 0, fake, b.BF16, None) == -2
    assert L.bof4_dequantize(fake, fake, 9, 128, 64, fake, None, None, None, 0, fake, b.BF16, None) == -3
    assert L.bof4_dequantize(fake, fake, b.BF16, 128, 64, fake, fake, None, None, 4, fake, b.BF16, None) == -1
    assert L.bof4_dequantize(fake, fake, b.BF16, 128, 64, fake, fake, fake, fake, -1, fake, b.BF16, None) == -5
    # OPQ: size limit, capacity, workspace
    ws = ctypes.c_void_p(0x10000)
    assert L.opq_split(fake, b.BF16, 1 << 31, 64, 3.0, None, fake, fake, 8, fake, ws, 1 << 40, None) == -2
    assert L.opq_split(fake, b.BF16, 128, 64, 3.0, None, fake, fake, -1, fake, ws, 1 << 40, None) == -5
    assert L.opq_split(fake, b.BF16, 128, 64, 3.0, None, fake, fake, 8, fake, None, 1 << 40, None) == -4
    assert L.opq_split(fake, b.BF16, 128, 64, 3.0, None, fake, fake, 8, fake, ws, 16, None) == -4
    assert L.opq_split(fake, b.BF16, 128, 64, 3.0, None, fake, fake, 8, fake, ctypes.c_void_p(0x10010), 1 << 40, None) == -4
    assert L.opq_split(fake, b.BF16, 128, 64, -1.0, None, fake, fake, 8, fake, ws, 1 << 40, None) == -1
    # the synchronising count check rejects bad arguments before touching the device
    assert L.bof4_outlier_count(None, 8, None, None) == -1
    assert L.bof4_outlier_count(fake, -1, None, None) == -1
    # EM
    ptrs = (ctypes.c_void_p * 1)(0x1000)
    ns = (ctypes.c_int64 * 1)(100)
    assert L.bof4_em_step(ptrs, ns, 1, b.BF16, 48, 0, 0, fake, fake, ws, 1 << 40, None) == -2   # block size
    ns[0] = -1
    assert L.bof4_em_step(ptrs, ns, 1, b.BF16, 64, 0, 0, fake, fake, ws, 1 << 40, None) == -1
    ns[0] = 100                      # a ragged length is accepted; the small workspace is refused next
    assert L.bof4_em_step(ptrs, ns, 1, b.BF16, 64, 0, 0, fake, fake, ws, 8, None) == -4
    assert L.bof4_em_step(ptrs, ns, 1, b.BF16, 64, 0, 4, fake, fake, ws, 1 << 40, None) == -1
    assert L.bof4_em_step(ptrs, ns, 1, 7, 64, 0, 0, fake, fake, ws, 1 << 40, None) == -3
    assert L.bof4_fit_codebook(ptrs, ns, 1, b.BF16, 64, 0, 0, fake, 0, -1, None, ws, 1 << 40, None) == -1
    assert L.bof4_fit_codebook(ptrs, ns, 1, b.BF16, 64, 0, 0, None, 0, 1, None, ws, 1 << 40, None) == -1
    # fused matrix-vector product: shape, dtype, outlier-list and alignment rules
    gv = lambda *a: L.bof4_gemv(*a)
    assert gv(fake, fake, b.BF16, 4, 96, 64, fake, fake, b.BF16, None, None, None, 0, fake, None) == -2
    assert gv(fake, fake, b.BF16, 4, 65536, 64, fake, fake, b.BF16, None, None, None, 0, fake, None) == -2
    assert gv(fake, fake, b.BF16, -1, 64, 64, fake, fake, b.BF16, None, None, None, 0, fake, None) == -1
    assert gv(fake, fake, 5, 4, 64, 64, fake, fake, b.BF16, None, None, None, 0, fake, None) == -3
    assert gv(fake, fake, b.BF16, 4, 64, 64, fake, fake, b.BF16, fake, None, None, 4, fake, None) == -1
    assert gv(fake, fake, b.BF16, 4, 64, 64, fake, fake, b.BF16, fake, fake, fake, -1, fake, None) == -5
    assert gv(fake, fake, b.BF16, 1 << 20, 4096, 64, fake, fake, b.BF16, fake, fake, fake, 4, fake, None) == -2
    assert gv(fake, fake, b.BF16, 4, 64, 64, fake, ctypes.c_void_p(0x1008), b.BF16, None, None, None, 0, fake, None) == -1
    assert b"aligned" in L.bof4_last_error()
    assert gv(ctypes.c_void_p(0x1010), fake, b.BF16, 4, 64, 64, fake, fake, b.BF16, None, None, None, 0, fake, None) == -1
    assert gv(fake, fake, b.BF16, 4, 64, 64, fake, fake, b.BF16, None, None, None, 0, None, None) == -1
    assert gv(None, None, b.BF16, 0, 64, 64, None, None, b.BF16, None, None, None, 0, None, None) == 0
    # theoretical codebook: the outermost levels must be fixed, metric MSE / MAE only
    full = (1 << 0) | (1 << 7) | (1 << 15)
    assert L.bof4_theoretical_codebook(64, 0, 0, fake, 1 << 15, 1, ws, 256, None) == -1   # -1 not fixed (abs)
    assert L.bof4_theoretical_codebook(64, 1, 0, fake, 1 << 7, 1, ws, 256, None) == -1    # +1 not fixed
    assert L.bof4_theoretical_codebook(64, 0, 2, fake, full, 1, ws, 256, None) == -1
    assert L.bof4_theoretical_codebook(1, 0, 0, fake, full, 1, ws, 256, None) == -2
    assert L.bof4_theoretical_codebook(64, 0, 0, fake, full, 1, ws, 8, None) == -4
    one = lambda v, t=ctypes.c_int: (t * 1)(v)
    batch = L.bof4_theoretical_codebook_batch
    assert batch(129, one(64), one(0), one(0), one(full, ctypes.c_uint32), fake, 1, ws, 1 << 20, None) == -2
    assert batch(1, one(64), one(0), one(0), one(1 << 15, ctypes.c_uint32), fake, 1, ws, 256, None) == -1
    assert batch(1, one(64), one(0), one(0), one(full, ctypes.c_uint32), fake, 1, ws, 128, None) == -4
    assert batch(1, None, one(0), one(0), one(full, ctypes.c_uint32), fake, 1, ws, 256, None) == -1
    assert batch(0, None, None, None, None, None, 1, None, 0, None) == 0


def test_native_module_of_another_torch_is_rebuilt_and_not_loaded(L, tmp_path, monkeypatch):
    """The native half of the binding is tied to the torch and Python it was compiled against."""
    from paper_2505_06653_b200 import binding, build
    assert build.host_matches(binding.HOST_PATH) and not build.needs_build()
    other = tmp_path / "_bof4_torch.so"
    data = open(binding.HOST_PATH, "rb").read()
    other.write_bytes(data.replace(build.host_tag().encode(), build.host_tag().replace("torch ", "torch 0").encode()[:len(build.host_tag())]))
    monkeypatch.setattr(build, "HOST_LIB", str(other))
    monkeypatch.setattr(binding, "HOST_PATH", str(other))
    monkeypatch.setattr(binding, "_host", None)
    assert build.needs_build()              # newer than every source, and stale all the same
    with pytest.raises(ImportError, match="not built for this torch"):
        binding._native()


def test_binding_refuses_cpu_tensors(L):
    import torch
    from paper_2505_06653_b200 import binding as b
    with pytest.raises(ValueError, match="no CPU path"):
        b.bof4_quantize(torch.zeros(64), 64, 0, np.linspace(-1, 1, 16))


def test_product_does_not_import_the_oracle():
    pkg = os.path.join(ROOT, "paper_2505_06653_b200")
    for dirpath, _, files in os.walk(pkg):
        for f in files:
            if f.endswith((".py", ".cu", ".cuh", ".h")):
                txt = open(os.path.join(dirpath, f)).read()
                assert "oracle" not in txt, os.path.join(dirpath, f)
