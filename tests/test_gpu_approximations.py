"""The FP64 functions that stand in for log, sqrt, sincospi and a division, element by element against extended
precision, where their tables and reductions can go wrong: the first and last words, every power of two
and its neighbours, both sides of every table interval and sector, the seam at mantissa 3/2."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# -2 ln u is stated within 3.2e-16 relative (half of it in the root), the root and the product round by
# 2.2e-16 and 1.1e-16, sine and cosine are within 1.9e-16 of the unit circle: 6.8e-16 of the radius together
PAIR = 7e-16


@pytest.fixture(scope="module")
def icm():
    import paper_1212_6427_gb300 as m
    from paper_1212_6427_gb300 import build
    build.build_library()
    m.use_torch_allocator()
    return m


def _around(values):
    v = np.unique(np.concatenate([np.asarray(values, dtype=np.int64) + k for k in (-1, 0, 1)]))
    return v[(v >= 0) & (v < 2 ** 32)]


def _radius_words():
    seams = [(2 ** e * (1024 + i)) // 2048 for e in (32, 31, 30, 21, 12) for i in range(1025)]
    return np.concatenate([_around(2 ** np.arange(33)), _around(3 * 2 ** np.arange(31)), _around(seams)])


def _angle_words():
    return np.concatenate([_around(np.arange(1025) * 2 ** 22), _around(np.arange(1024) * 2 ** 22 + 2 ** 21)])


def test_normal_pairs_element_by_element(icm):
    rng = np.random.default_rng(1)
    a, b = _radius_words(), _angle_words()
    any_word = lambda n: rng.integers(0, 2 ** 32, size=n)
    words = np.concatenate([np.stack([a, any_word(len(a))], 1), np.stack([any_word(len(b)), b], 1),
                            np.stack([any_word(20000), any_word(20000)], 1),
                            [[2 ** 32 - 1, 0], [0, 0], [0, 2 ** 32 - 1], [2 ** 32 - 1, 2 ** 32 - 1]]])
    sim = icm.Simulation((16, 16, 16), 1.0, 1.0, 1.0, 1e-3, 0.05, 3, 1, 64)
    got = icm.icm_op_normal_pairs(sim.handle, words).astype(np.longdouble)
    sim.close()
    u = (words.astype(np.longdouble) + np.longdouble(0.5)) / np.longdouble(2) ** 32
    rad = np.sqrt(np.longdouble(-2) * np.log(u[:, 0]))
    # 2 pi u to the quarter turn next to it, so that the zeros of sine and cosine keep their accuracy
    quarter = np.round(4 * u[:, 1])
    t = (u[:, 1] - quarter / 4) * 2 * np.longdouble("3.14159265358979323846264338327950288")
    c, s = np.cos(t), np.sin(t)
    q = quarter.astype(np.int64) % 4
    cos = np.choose(q, [c, -s, -c, s])
    sin = np.choose(q, [s, c, -s, -c])
    assert float((np.abs(got[:, 0] - rad * cos) / rad).max()) < PAIR
    assert float((np.abs(got[:, 1] - rad * sin) / rad).max()) < PAIR
    assert float((np.abs(np.hypot(got[:, 0], got[:, 1]) - rad) / rad).max()) < PAIR


def test_reciprocals_are_within_an_ulp(icm):
    rng = np.random.default_rng(2)
    mantissa = np.concatenate([1.0 + np.arange(4096) / 4096, np.nextafter(1.0 + np.arange(1, 4097) / 4096, 0.0),
                               rng.uniform(1.0, 2.0, size=20000)])
    x = np.concatenate([mantissa * 2.0 ** e for e in (-960, -300, -13, 0, 4, 300, 960)])
    exact = np.longdouble(1) / x.astype(np.longdouble)
    err = np.abs(icm.icm_op_reciprocals(64, x).astype(np.longdouble) - exact) / exact
    assert float(err.max()) < 2.0 ** -52
    y = np.concatenate([mantissa * 2.0 ** e for e in (-100, -13, 0, 4, 100)]).astype(np.float32).astype(np.float64)
    assert np.abs(icm.icm_op_reciprocals(32, y) * y - 1.0).max() < 2.0 ** -23 * 1.01   # (rounded to FP32, then the product)
