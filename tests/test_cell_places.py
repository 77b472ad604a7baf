"""The order of the cells by their normalised weight, and the place of a threshold in it, restated from the kernels' integer rules
(em_cells.cuh, em_cells_fit.cu) and compared with the sorted fp32 quotients themselves."""
import numpy as np

PARTS, FRACTIONS, DEEP = 4096, 128 * 128, 88
ONE = 1 + DEEP + 40 * FRACTIONS


def _f32(bits):
    return np.asarray(bits, np.uint32).view(np.float32)


def _rank(a0, b0):
    """fraction_rank: how many of a / b (a >= b) or 2 a / b lie before that of (a0, b0) + 128, equal ones by b."""
    b = b0 + 128
    a = (a0 + 128) << (a0 < b0)
    c = np.arange(128, 256)
    tie = c < b
    q1, q2 = a * c // b, a * c // (2 * b)
    n1 = np.minimum(np.where((a * c % b != 0) | tie, q1, q1 - 1), 255) - c + 1
    n2 = np.minimum(np.where((a * c % (2 * b) != 0) | tie, q2, q2 - 1), c - 1) - 127
    return int(np.maximum(n1, 0).sum() + np.maximum(n2, 0).sum())


def _order():
    value = np.full(FRACTIONS, -1)
    for f in range(FRACTIONS):
        value[_rank(f >> 7, f & 127)] = f
    assert (value >= 0).all()                       # a permutation
    x = np.zeros(ONE + 1, np.float32)
    e = np.arange(DEEP)
    x[1:1 + DEEP] = _f32(np.where(e > 0, e << 23, 0x400000))
    a, b = value >> 7, value & 127
    seen = 0
    for binade in range(40, 0, -1):
        d = 128 * np.where(a >= b, binade, binade - 1) + b - a
        at = 1 + DEEP + (40 - binade) * FRACTIONS
        x[at:at + FRACTIONS] = _f32((0x3f80 + b - d) << 16) / _f32((0x3f80 + b) << 16)
        seen += int((d < 5120).sum())
    x[ONE] = 1
    assert seen == 128 * 5119                       # every distance of every significand but 0 has one place
    return value, np.concatenate([-x[:0:-1], x])


def _place(p, front, a, b):
    """place_of."""
    bits = int(_f32(np.float32(p).view(np.uint32)).view(np.uint32)) & 0x7fffffff
    neg = bool(p < 0)
    q = (bits & 0x7fffff) | 0x800000
    half = 2 * q + (1 if neg else -1)
    n = front[q // (0x800000 // PARTS) - PARTS]
    while n < FRACTIONS and (a[n] << 24) < b[n] * half:
        n += 1
    e = bits >> 23
    if bits >= 0x3f800000:
        below = ONE + 1 if neg or bits > 0x3f800000 else ONE
        if bits > 0x7f800000:
            below = ONE
    elif e >= 87:
        below = 1 + DEEP + (e - 87) * FRACTIONS + n
        if not neg and bits == 87 << 23:
            below = DEEP
    elif e > 0:
        below = 1 + e + int(neg or bits & 0x7fffff != 0)
    else:
        below = 0 if bits == 0 else 1 + int(bits > 0x400000 or (neg and bits == 0x400000))
    return ONE + 1 - below if neg else ONE + below


def test_places_are_those_of_the_sorted_quotients():
    value, x = _order()
    assert len(x) == 2 * ONE + 1 and (np.diff(x) >= 0).all()
    hi, lo = (value >> 7) + 128, (value & 127) + 128
    y = np.where(hi < lo, 2 * hi, hi) / lo
    front = []
    for part in range(PARTS):                       # fractions_below
        c = np.arange(128, 256)
        t = c * (PARTS + part) - 1
        front.append(int(np.maximum(np.minimum(t // PARTS, 255) - c + 1, 0).sum() + np.maximum(np.minimum(t // (2 * PARTS), c - 1) - 127, 0).sum()))
    assert front == [int((y < 1 + part / PARTS).sum()) for part in range(PARTS)]
    a, b = [int(v) for v in np.where(hi < lo, 2 * hi, hi)], [int(v) for v in lo]
    rng = np.random.default_rng(0)
    at = rng.choice(x, 1500)
    ps = np.concatenate([rng.uniform(-1.1, 1.1, 500), at, np.nextafter(at, np.float32(-9)), np.nextafter(at, np.float32(9)),
                         np.exp2(rng.uniform(-149, 1, 500)) * rng.choice([-1, 1], 500), [s * 2.0 ** -k for k in range(150) for s in (1, -1)],
                         [0.0, -0.0, 2, -2, np.inf, -np.inf]]).astype(np.float32)
    for p in ps:
        assert _place(p, front, a, b) == int(np.searchsorted(x, p, side="left")), p
