"""Blocks whose AOs differ by up to 2^24 in size (as tight and diffuse functions do), in the products of
blocks with more than 16 AOs (k_zcw) and of smaller ones: every element of Sigma against its own scale.

C[al, a, f] is graded by s_a s_f and D either not at all or by 1 / s of its column, so every term of
Sigma_ij is of the order s_i s_j.

Tolerance: B_ij, Sigma of the absolute values (one sign throughout), is the sum of the sizes of an element's
terms.  With k digits an operand is off by at most 2^-7k of the largest in its row (column, for D), which
over the K products of a sum costs 2^-7k K max max; against the sum of their sizes that is (max / mean)^2,
about 25 for normal data, times 27 / 2 where the contracted AOs are graded (about two of 27 carry the sum):
2^8.4.  Both operands of two products in a row: 2^2 more, and 2^0.6 to spare: 2^(11 - 7 k) B_ij."""
import copy

import numpy as np
import pytest

import oracle
import synth
from gpu_common import gpu_build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _grade(blocks, left, right, rows):
    """Blocks (i, j) times left[i] over their AOs of i and right[j] over those of j (rows: ABFs before)."""
    for e, (i, j) in enumerate(blocks.keys[:, :2]):
        x = blocks.data[blocks.offs[e]:blocks.offs[e + 1]].reshape(rows(i), len(left[i]), len(right[j]))
        x *= left[i][:, None] * right[j]


@pytest.mark.parametrize("nao", [[27, 20, 17], [32, 13, 24], [13, 16, 9]])
@pytest.mark.parametrize("columns", [False, True])
@pytest.mark.parametrize("nslices", [6, 5])
def test_graded(nao, columns, nslices):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nabf = [11, 40, 23]
    sys_ = synth.custom("graded", 1.0, 5, [[0, 0, 0], [2, 1, 0], [1, 3, 2]], nao, nabf)
    wl = synth.make_workload(sys_, 3.2, 4.2, 3.0, seed=9)
    s = [np.exp2(-24.0 * np.arange(n) / (n - 1)) for n in nao]
    _grade(wl.C, s, s, lambda i: nabf[i])
    if columns:
        _grade(wl.D, [np.ones(n) for n in nao], [1.0 / x for x in s], lambda i: 1)
    ref = oracle.Oracle.of(wl).build(0.0)
    size = copy.deepcopy(wl)
    for k in "CVD":
        b = getattr(size, k)
        b.data[:] = np.abs(b.data)
    size = np.abs(oracle.Oracle.of(size).build(0.0)["data"])
    _, got = gpu_build(wl, 0.0, "ozaki", nslices)
    np.testing.assert_array_equal(got["keys"], ref["keys"])
    # Sigma's words hold 2^-64: at s_i s_j = 2^-48 the roundings of some 300 terms to them count too
    err = np.abs(got["data"] - ref["data"]) / (2.0 ** (11 - 7 * nslices) * size + 1e3 * 2.0 ** -64)
    assert err.max() <= 1.0, err.max()
