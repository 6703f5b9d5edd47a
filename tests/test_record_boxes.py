"""The 16-bit boxes of the two-level node records never miss what the exact
box test hits.

The kernels form a plane's distance as fma(2^23 + n, S, C), n the plane's cell
rounded outward, S = inverse direction times cell size, C the constant part
rounded down for the entry plane and up for the exit plane.  Emulated here with
exact rationals and every rounding step, over scales, offsets and directions:
the entry distance is never above, the exit distance never below the distance
fma(plane, inverse, -(o * inverse)) that the exact test computes.
"""
import math
import random
from fractions import Fraction as F

import numpy as np

MAX = float(np.finfo(np.float32).max)


def _rn(x):
    """Nearest float32 (ties to even) of a rational, as a rational."""
    c = np.float32(float(x))  # within an ulp; pick among the neighbours
    best = None
    for d in (np.nextafter(c, np.float32(-np.inf)), c, np.nextafter(c, np.float32(np.inf))):
        if not np.isfinite(d):
            continue
        key = (abs(F(float(d)) - x), int(d.view(np.uint32)) & 1)
        if best is None or key < best[0]:
            best = (key, F(float(d)))
    return best[1]


def _rd(x):
    r = _rn(x)
    if r > x:
        r = F(float(np.nextafter(np.float32(float(r)), np.float32(-np.inf))))
    return r


def _ru(x):
    return -_rd(-x)


def _cell(lo, hi):
    need = _ru(_ru(hi - lo) / 65535)
    need = max(need, F(2) ** -40)
    c = F(2) ** math.floor(math.log2(float(need)))
    while c > need:
        c /= 2
    while c < need:
        c *= 2
    return c


def _cases(rng):
    for _ in range(1500):
        lo, hi = sorted((rng.uniform(-1, 1), rng.uniform(-1, 1)))
        scale = 2.0 ** rng.randint(-20, 30)
        off = rng.choice([0.0, 0.0, 1.0, -1e3, 1e5]) * scale
        root = [float(np.float32(v * scale + off)) for v in (lo, hi)]
        if rng.random() < 0.1:
            root[1] = root[0]
        a, b = sorted(float(np.float32(rng.uniform(*root))) for _ in range(2))
        a, b = max(a, root[0]), min(b, root[1])
        if rng.random() < 0.2:
            a = b = rng.choice(root)
        d = rng.choice([rng.uniform(-1, 1), 2.0 ** -80, -(2.0 ** -80), 1.0, -1.0,
                        2.0 ** rng.randint(-60, 60)])
        o = rng.choice([rng.uniform(-2, 2) * scale + off, 0.0, a, 1e8 * scale, -1e12])
        yield root, (a, b), float(np.float32(d)), float(np.float32(o))


def test_record_boxes_are_conservative():
    n = 0
    for (r0, r1), (a, b), d, o in _cases(random.Random(11)):
        if d == 0.0:
            continue
        inv = _rn(1 / F(d))
        if abs(inv) < F(2) ** -80:
            continue  # walks the binary nodes
        if abs(F(o) * inv) >= F(MAX) / 4 or abs(F(r1) * inv) >= F(MAX) / 2 ** 30:
            continue  # infinite distances: the same on both sides
        no = -_rn(F(o) * inv)
        g0, cell = F(r0), _cell(F(r0), F(r1))
        below = min(max(math.floor(_rd(_rd(F(a) - g0) / cell)), 0), 65535)
        above = min(max(math.ceil(_ru(_ru(F(b) - g0) / cell)), 0), 65535)
        assert g0 + below * cell <= F(a) and g0 + above * cell >= F(b)
        s = inv * cell
        assert s == _rn(s)
        base = s * 2 ** 23
        lo_plane, hi_plane = (a, below), (b, above)
        (xe, ne), (xx, nx) = (lo_plane, hi_plane) if inv > 0 else (hi_plane, lo_plane)
        ce = _rd(_rd(g0 * inv + no) - base)
        cx = _ru(_ru(g0 * inv + no) - base)
        entry, exit_ = _rn((2 ** 23 + ne) * s + ce), _rn((2 ** 23 + nx) * s + cx)
        assert entry <= _rn(F(xe) * inv + no)
        assert exit_ >= _rn(F(xx) * inv + no)
        n += 1
    assert n > 1000
