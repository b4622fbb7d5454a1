"""The adjoint with mirror pieces (exactly Hermitian V and D: the B role taken twice, dV written to a
pair and its mirror) against the general path (HFX_NO_MIRROR) on the same inputs, at block sizes around
the tiles of the dV product, with and without the ERI screen."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _grad(wl, theta, eri):
    import paper_2009_12505_gb300 as hfx
    c = hfx.Context(wl.system.nao, wl.system.nabf)
    c.set_eri_screen(eri)
    for k in "CVD":
        c.set_blocks(k, getattr(wl, k))
    c.build(theta)
    return c.stats()["mirror"], *c.grad(wl.C.data.size, wl.V.data.size)


@pytest.mark.parametrize("nao,nabf,theta,eri", [
    ([2, 4, 3], [3, 5, 2], 0.0, None), ([1, 7, 33], [65, 1, 32], 1e-2, None),
    ([5, 2, 16], [31, 33, 128], 1e-2, 1e-2)])
def test_mirror_adjoint(nao, nabf, theta, eri, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    s = synth.custom("odd", 1.0, 5, [[0, 0, 0], [2, 1, 0], [1, 3, 2]], nao, nabf)
    wl = synth.make_workload(s, 3.2, 4.2, 3.0, seed=6)
    on, dC, dV = _grad(wl, theta, eri)
    monkeypatch.setenv("HFX_NO_MIRROR", "1")
    off, rC, rV = _grad(wl, theta, eri)
    assert (on, off) == (1, 0)
    # both are FP64 sums of the same terms in another order: at most some 1e5 terms an element
    for got, ref in ((dC, rC), (dV, rV)):
        np.testing.assert_allclose(got, ref, rtol=0, atol=2.0 ** -52 * 300 * np.abs(ref).max())
