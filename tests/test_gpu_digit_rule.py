"""The digits of P in the D_AB product: each word of its f32 pair is rounded to the last unit u = 2^(e - 7 k),
ties to even, and the digits after the first lie in [-64, 63].

Four one-AO atoms with C on (0, 2) and (1, 3), V on (0, 1) and D on (0, 1) alone leave one term,
Sigma_23 = -sum_al C[al] P[al], P = D Y.  P[0] (near 1, so e = 2) only sets the row's exponent, as C[0] = 0;
P[1] is the value under test.  Every operand but P has at most k exact digits, so the results are exact."""
import numpy as np
import pytest

import paper_2009_12505_gb300 as hfx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _sigma(k, y0, c, d, y1=1.0):
    z = (0, 0, 0)
    ctx = hfx.Context([1, 1, 1, 1], [2, 1, 1, 1])
    ctx.set_block("C", 0, 2, z, [0.0, c])
    ctx.set_block("C", 1, 3, z, [1.0])
    ctx.set_block("V", 0, 1, z, [y0, y1])
    ctx.set_block("D", 0, 1, z, [d])
    ctx.build(0.0, *(("bf16x3", 2) if k == 2 else ("ozaki", k)))
    assert ctx.keys().tolist() == [[2, 3, 0, 0, 0]]
    return float(ctx.sigma()[0])


@pytest.mark.parametrize("k", [4, 5, 6])
@pytest.mark.parametrize("units,rounded", [(2.0 ** 22 + 0.7, 2.0 ** 22), (2.0 ** 22 + 1.3, 2.0 ** 22 + 2),
                                           (-2.0 ** 22 - 0.7, -2.0 ** 22)])
def test_words_round_separately(k, units, rounded):
    """The high word lies on a tie, the low one (0.2 u) rounds to nothing."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    u = 2.0 ** (2 - 7 * k)
    high = float(np.float32(units))
    assert abs(high - units) > 0.1 and high % 1.0 == 0.5  # a pair whose high word is a tie
    assert _sigma(k, 2.0 ** (7 * k - 24), 1.0, units * u) == -rounded * u


@pytest.mark.parametrize("k", [2, 4, 5, 6])
def test_digit_range(k):
    """64 last units are the digits 1, -64: with the second digit of C (2^-12) the 1 is in the kept orders."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    u = 2.0 ** (2 - 7 * k)
    assert _sigma(k, 2.0 ** (7 * k - 8), 1.0 + 2.0 ** -12, 64.0 * u) == -(64.0 + 128.0 * 2.0 ** -12) * u


@pytest.mark.parametrize("k", [4, 5, 6])
@pytest.mark.parametrize("y0,y1,c,d", [(1e30, 1e30, 1e-55, 1e30), (1e30, 1.0, 1e-28, 1e30),
                                       (1e39, 1e39, 1e-38, 1.0), (-1e30, 1.0, 1e-28, 1e30)])
def test_overflow_fails(k, y0, y1, c, d):
    """P beyond the f32 range (its own row's or another, from D Y or already in Y): an error, not a Sigma
    without the row."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    with pytest.raises(hfx.HfxError):
        _sigma(k, y0, c, d, y1)
