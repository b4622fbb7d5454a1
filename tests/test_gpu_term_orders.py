"""Both product orders of hfx_term_noalloc at the edges of the rule between them, against the same sum
in torch: the smallest sizes, the static array's limit, and blocks of many outputs."""
import pytest

from paper_2009_12505_gb300 import hfx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# nabf_a, nabf_b, nao_i, nao_k, nao_j, nao_l
@pytest.mark.parametrize("sizes", [
    (1, 1, 1, 1, 1, 1), (60, 90, 13, 13, 27, 27), (90, 60, 27, 27, 13, 13), (33, 7, 5, 31, 2, 3),
    (128, 3, 9, 32, 32, 32), (2, 8192, 4, 4, 3, 3), (2, 8193, 4, 4, 3, 3), (2, 3, 256, 2, 257, 1)])
def test_orders(sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pa, pb, ni, nk, nj, nl = sizes
    g = torch.Generator().manual_seed(sum(sizes))
    r = lambda *s: torch.rand(*s, dtype=torch.float64, generator=g) - 0.5  # noqa: E731
    cA, V, cB, D = r(pa, ni, nk), r(pa, pb), r(pb, nj, nl), r(nk, nl)
    ref = torch.einsum("xik,xjk->ij", cA, torch.einsum("xy,yjl,kl->xjk", V, cB, D))
    out = torch.full((ni, nj), float("nan"), dtype=torch.float64, device="cuda")
    hfx.term_noalloc(cA.cuda(), V.cuda(), cB.cuda(), D.cuda(), out)
    # random signs: the rounding of n products of at most 1/16 grows as sqrt(n)
    tol = 2.0 ** -52 * (pa * pb * nk * nl) ** 0.5
    assert (out.cpu() - ref).abs().max() <= tol
