"""Harmonic sums at thresholds that many sums cross: warps whose staged records reach the flush limit
in every tile, part of the lanes appending, up to every sum of the plane.  Crossing sets against the
FP64 oracle; every stored power is within the FP32 summation bound of the oracle's."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -24


@pytest.mark.parametrize("share", [0.002, 0.02, 0.1, 0.5, 1.0])   # of the sums of each level
@pytest.mark.parametrize("m,n,bin0,H", [(85, 20_011, 210, 1), (5, 400_003, 0, 1), (85, 20_011, 210, 2), (85, 20_011, 210, 8),
                                        (129, 9_001, 0, 32)])
def test_dense_crossings(oracle_mod, m, n, bin0, H, share):
    import paper_1805_12280_gb300 as fd
    fd.load()
    P = synth.noise_plane(m, n, seed=n + H)
    S = oracle_mod.harmonic_sums(P, bin0, H)
    levels = np.array(fd.harmonic_levels(H))
    defined = ~np.isnan(S)
    thr = np.array([np.float32(-1.0 if share == 1.0 else np.quantile(s[d], 1.0 - share)) for s, d in zip(S, defined)])
    S = np.where(defined, S, -np.inf)
    bound = (levels - 1) * U / (1 - (levels - 1) * U)
    room = int((S > thr[:, None, None]).sum()) + 4096
    for stored in (room, 1000):   # a list with room for all, and one that is truncated
        buf, count = fd.harmonic_sum(torch.from_numpy(P).cuda(), bin0, H, list(thr), max_cand=stored)
        got = fd.harmonic_to_numpy(buf, count)
        j = np.log2(got["nharm"]).astype(np.int64)
        key = (j * m + got["tpl"]) * n + got["bin"]
        assert np.unique(key).size == got.size == min(int(count.item()), stored)
        ref = S[j, got["tpl"], got["bin"]]
        assert np.all(np.abs(got["power"].astype(np.float64) - ref) <= bound[j] * ref)
        assert np.all(got["power"] > thr[j])
        if stored == room:
            sure = np.zeros(S.shape, dtype=bool)
            sure.reshape(-1)[key] = True
            assert np.all(sure[S > (thr * (1 + 2 * bound))[:, None, None]]) and got.size > 0
