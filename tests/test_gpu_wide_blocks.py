"""The D_FG / D_FB products of blocks with more than 16 AOs (k_zcw) against the CPU oracle, at the edges
of their row tiles and fragments: AO counts around 16 and 32, one-AO atoms beside 32 (Y read from
global memory), few and many ABFs, with and without the mirror pieces, and with every digit count."""
import pytest

import oracle
import synth
from gpu_common import compare_full, gpu_build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nao,nabf,mirror,nslices", [
    ([17, 16, 5], [9, 33, 20], "1", 6), ([32, 9, 27], [5, 40, 8], "1", 6),
    ([1, 32, 2], [70, 3, 120], "0", 6), ([18, 22, 25], [13, 1, 7], "0", 6),
    ([27, 13, 14], [11, 60, 9], "1", 5), ([3, 31, 11], [64, 4, 17], "1", 4)])
def test_wide_blocks(nao, nabf, mirror, nslices, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    monkeypatch.setenv("HFX_NO_MIRROR", "0" if mirror == "1" else "1")
    s = synth.custom("wide", 1.0, 5, [[0, 0, 0], [2, 1, 0], [1, 3, 2]], nao, nabf)
    wl = synth.make_workload(s, 3.2, 4.2, 3.0, seed=6)
    ref = oracle.Oracle.of(wl).build(1e-2)
    _, g = gpu_build(wl, 1e-2, "ozaki", nslices)
    # the library's bar of 1e-8 Ha with 6 digits; each digit fewer costs 2^7
    scale = max(1.0, abs(ref["data"]).max() / 66.0)
    compare_full(wl, 1e-2, g, ref, 1e-8 * 128.0 ** (6 - nslices) * scale)
