"""The velocity factor of an accepted exchange on the mixed path's fixed-point
words (units of 2^-48), against exact integers: one rounding, halves upward, for
factors in [2^-10, 2); the FP64 product rounded to the nearest word outside.  The
same words whether the factor is applied to what is read, at the next launch's
start, or inside a free-running launch."""
from fractions import Fraction

import numpy as np
import pytest

from paper_0812_1633_gb300 import inputs

pytestmark = pytest.mark.gpu

FACTORS = [2.0 ** -10, np.nextafter(2.0 ** -10, 0), np.nextafter(2.0 ** -10, 1), 2.0 ** -12, 0.1, 1 / 3,
           0.5, np.nextafter(0.5, 0), np.nextafter(1.0, 0), 1.0, np.nextafter(1.0, 2), np.sqrt(1.3), 1.5,
           np.nextafter(2.0, 0), 2.0, np.nextafter(2.0, 3), 3.7]


@pytest.fixture(scope="module")
def re():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0812_1633_gb300 import build
    build.build()
    import paper_0812_1633_gb300 as m
    m.lib()
    return m


def scaled(word, f):
    if f == 1.0:
        return word
    if 2.0 ** -10 <= f < 2.0:
        p = Fraction(f) * word + Fraction(1, 2)
        return p.numerator // p.denominator
    return int(np.rint(float(word) * f))


def test_words(re):
    N, R = 256, len(FACTORS)
    L = inputs.box_length(N)
    rng = np.random.default_rng(8)
    ctx = re.Context(N, L, 2.5, [1.0 + 0.01 * k for k in range(R)], 3, precision="mixed")
    mag = np.exp2(rng.uniform(0, 51, (N * R, 3)))
    words = np.rint(rng.choice([-1, 1], mag.shape) * mag).astype(np.int64)
    words[:3 * R:R // 3] = 0
    words[1], words[2], words[5] = (1, -1, 3), (-3, 2 ** 51 - 1, -2 ** 51 + 1), (2 ** 50 + 1, 1 << 20, -(1 << 20) - 1)
    ctx.set_state(None, words * 2.0 ** -48)
    ctx.apply_exchange(ctx.temps(), np.array(FACTORS))
    want = np.array([[scaled(int(w), FACTORS[a // N]) for w in words[a]] for a in range(N * R)])
    read = ctx.get_state()[1] * 2.0 ** 48
    assert np.array_equal(read, want)
    ctx.advance(np.zeros(R, np.int32))  # the launch applies the factors to the state
    assert np.array_equal(ctx.get_state()[1] * 2.0 ** 48, want)
    ctx.close()


def test_exchange_inside_a_launch(re):
    """A free-running launch against budgets of the same steps with exchanges
    between the launches: equal bit for bit."""
    N, R, nx, A = 256, 8, 6, 5
    L = inputs.box_length(N)
    temps = inputs.geometric_ladder(0.8, 1.6, R)
    a = re.Context(N, L, 2.5, temps, 12, precision="mixed")
    b = re.Context(N, L, 2.5, temps, 12, precision="mixed")
    steps, _, partner, acc = a.run_free(A, nx, log=True)
    prev = np.zeros(R, np.int64)
    for k in range(A):
        b.advance((steps[k] - prev).astype(np.int32))
        po, ao = b.exchange(outputs=True)
        assert np.array_equal(partner[k], po) and np.array_equal(acc[k].astype(bool), ao.astype(bool))
        prev = steps[k].copy()
    assert acc.any()
    for s, t in zip(a.get_state(), b.get_state()):
        np.testing.assert_array_equal(s, t)
    a.close()
    b.close()
