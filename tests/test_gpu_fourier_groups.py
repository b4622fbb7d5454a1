"""The grouped k-space kernels at their edges, against oracle/fourier.py: density keys of one atom
pair in both orientations and in more than one group of eight, band counts around the staged sixteen,
blocks of more elements than threads; Sigma at k points with more keys a pair than are held at once."""
import numpy as np
import pytest

import synth
from oracle import fourier
from paper_2009_12505_gb300 import hfx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("nao,nbands,nk,reach", [([3, 5], 1, 1, 0), ([1, 17], 16, 2, 1),
                                                 ([13, 4], 33, 3, 1), ([64, 2], 15, 2, 1)])
def test_density_groups(nao, nbands, nk, reach):
    rng = np.random.default_rng(nbands)
    kf = rng.uniform(-0.5, 0.5, (nk, 3))
    coef = rng.normal(size=(nk, sum(nao), nbands)) + 1j * rng.normal(size=(nk, sum(nao), nbands))
    occ = rng.uniform(0, 2, (nk, nbands))
    r = range(-reach, reach + 1)
    keys = np.array([(i, j, a, b, c) for i in (0, 1) for j in (1, 0) for a in r for b in r for c in r])
    keys = keys[rng.permutation(len(keys))]  # any order, up to 27 images a pair and orientation
    got, maxim = hfx.Context(nao, [4, 4]).density_from_eigvecs(kf, coef, occ, keys)
    ref = np.concatenate([b.ravel() for b in fourier.density(nao, kf, coef, occ, keys)])
    # sums of nk nbands products of unit size, each rounded a few times
    tol = 8 * np.finfo(float).eps * nk * nbands * np.abs(ref).max()
    np.testing.assert_allclose(got, ref.real, rtol=0, atol=tol)
    assert abs(maxim - np.abs(ref.imag).max()) <= tol


def test_density_overflow_shows_in_max_imag():
    """Finite coefficients whose products overflow: the imaginary part is no number, and says so."""
    coef = np.full((1, 5, 2), 1e200 + 1e200j)
    _, maxim = hfx.Context([2, 3], [4, 4]).density_from_eigvecs(
        np.zeros((1, 3)), coef, np.ones((1, 2)), np.array([(0, 1, 0, 0, 0)]))
    assert not np.isfinite(maxim)


@pytest.mark.parametrize("nao", [2, 17])
def test_sigma_k_many_keys(nao):
    s = synth.custom("one", 1.0, 1, [[0, 0, 0]], [nao], [2])
    wl = synth.make_workload(s, 1.8, 2.3, 2.3, seed=3)
    ctx = hfx.Context(s.nao, s.nabf)
    for k in "CVD":
        ctx.set_blocks(k, getattr(wl, k))
    ctx.build(0.0)
    keys, offs, sig = ctx.keys(), ctx.offsets(), ctx.sigma()
    assert len(keys) > 512
    kf = np.array([[0.0, 0.0, 0.0], [0.1, -0.3, 0.2]])
    ref = fourier.sigma_k(s.nao, keys, [sig[offs[e]:offs[e + 1]] for e in range(len(keys))], kf)
    tol = 8 * np.finfo(float).eps * len(keys) * np.abs(sig).max()
    np.testing.assert_allclose(ctx.sigma_k(kf), ref, rtol=0, atol=tol)
