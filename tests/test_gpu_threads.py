"""Other Python threads run while a call of the binding waits for room in the stream's queue."""
import threading
import time

import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


def _quantize(bof4, w, cb):
    codes, scales = bof4.bof4_quantize(w, 64, 1, cb)
    return lambda: bof4.bof4_quantize(w, 64, 1, cb, out=(codes, scales))


def _gemv(bof4, w, cb):
    codes, scales = bof4.bof4_quantize(w, 64, 1, cb)
    x, y = torch.zeros(64, dtype=torch.bfloat16, device="cuda"), torch.empty(w.numel() // 64, device="cuda")
    return lambda: bof4.bof4_gemv(codes, scales, w.numel() // 64, 64, 64, cb, x, out=y)


def _fit(bof4, w, cb):
    out = (cb.clone(), torch.zeros(2, dtype=torch.float64, device="cuda"))
    ws = torch.empty(bof4.bof4_fit_workspace_bytes(w.numel(), bof4.BF16, 64, 0, 2), dtype=torch.uint8, device="cuda")
    return lambda: bof4.bof4_fit_codebook(w, 64, 1, 0, out[0], 0, 2, workspace=ws, sync=False, out=out)


@pytest.mark.parametrize("make", [_quantize, _gemv, _fit])
def test_a_full_queue_stops_no_other_thread(make):
    import __graft_entry__ as entry
    entry.build()
    import paper_2505_06653_b200 as bof4
    w = workloads.gaussian(1 << 12, 0.02, 1, torch.bfloat16).cuda()
    cb = torch.tensor(workloads.BOF4S_MSE_I64, dtype=torch.float32, device="cuda")
    call = make(bof4, w, cb)
    call()
    torch.cuda.synchronize()
    for attempt in range(3):  # a busy machine may stop a thread for a while by itself; the lock does every time
        waited, gap = _longest_gap(call)
        assert waited > 0.4, "the queue did not fill"
        if gap < 0.2:
            return
    raise AssertionError("another thread stood still for %.3f s of %.3f s" % (gap, waited))


def _longest_gap(call):
    """Seconds that 3000 calls behind a kernel of 0.6 s and more take, and the longest that another thread stood still."""
    seen, stop = [], threading.Event()

    def watch():
        while not stop.is_set():
            seen.append(time.perf_counter())
            time.sleep(0.002)

    t = threading.Thread(target=watch)
    t.start()
    time.sleep(0.05)
    torch.cuda._sleep(int(1.2e9))
    start = time.perf_counter()
    for _ in range(3000):
        call()
    waited = time.perf_counter() - start
    stop.set()
    t.join()
    torch.cuda.synchronize()
    return waited, max(b - a for a, b in zip(seen, seen[1:]))
