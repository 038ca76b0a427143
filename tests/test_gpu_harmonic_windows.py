"""Harmonic sums where the plane is walked in several slope windows, at the edges of the window
table (one row, as many rows as the table holds, more rows than it holds) and across the tile
sizes of one harmonic: crossing sets against the FP64 oracle."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -24


@pytest.fixture(scope="module")
def fd():
    import paper_1805_12280_gb300 as m
    m.load()
    return m


@pytest.mark.parametrize("m,n,bin0,H", [(85, 260_003, 210, 32),      # two windows, ragged row length
                                        (85, 700_001, 210, 8),       # four windows
                                        (2001, 20_011, 7, 4),        # table room for two windows
                                        (4095, 9_001, 0, 8),         # c = 2047 entries, one window
                                        (4099, 3_001, 0, 2),         # c = 2049: more than the table holds
                                        (1, 70_001, 3, 8), (3, 70_001, 0, 16),
                                        (85, 2_049, 0, 1), (85, 400_000, 210, 1)])   # the two tile sizes of one harmonic
def test_crossing_sets(fd, oracle_mod, m, n, bin0, H):
    P = synth.noise_plane(m, n, seed=n + H)
    levels = np.array(fd.harmonic_levels(H))
    thr = np.array([np.float32(h + 5.0 * np.sqrt(h)) for h in levels], dtype=np.float64)
    ref = oracle_mod.harmonic_candidates(P, bin0, H, thr)
    room = ref["bin"].size + 4096
    buf, count = fd.harmonic_sum(torch.from_numpy(P).cuda(), bin0, H, list(thr), max_cand=room)
    got = fd.harmonic_to_numpy(buf, count)
    assert int(count.item()) == got.size and ref["bin"].size > 0
    # FP32 sums of h non-negative terms: relative error at most gamma_{h-1}
    h = levels[ref["level"]]
    band = (h - 1) * U / (1 - (h - 1) * U) * ref["value"]
    sure = np.abs(ref["value"] - thr[ref["level"]]) > band
    cell = lambda lv, t, b: (lv.astype(np.int64) * m + t) * n + b
    want = cell(ref["level"], ref["row"], ref["bin"])
    have = cell(np.log2(got["nharm"]).astype(np.int64), got["tpl"], got["bin"])
    assert np.unique(have).size == have.size
    assert np.isin(want[sure], have).all()
    # what else crosses lies within its bound below the threshold
    extra = ~np.isin(have, want)
    j = np.log2(got["nharm"][extra]).astype(np.int64)
    assert np.all(got["power"][extra] <= thr[j] * (1 + 2 * H * U))
    both, at_have, at_want = np.intersect1d(have, want, return_indices=True)
    value = ref["value"][at_want]
    h = levels[ref["level"][at_want]]
    assert np.all(np.abs(got["power"][at_have].astype(np.float64) - value) <= (h - 1) * U / (1 - (h - 1) * U) * value)


@pytest.mark.parametrize("m,n,bin0,H", [(4099, 1_025, 0, 32), (4097, 2_000, 3, 8), (20_001, 41, 2, 8),   # rows of |z| > c / H in runs
                                        (8193, 6, 0, 32),             # fewer columns than harmonics
                                        (2_051, 700, 0, 16), (85, 13_000, 210, 2), (3, 3, 0, 2),
                                        (513, 901, 0, 8), (515, 901, 0, 8), (449, 12_000, 1, 32),     # long tables over few tiles
                                        (200_001, 20, 0, 2), (60_001, 257, 1, 1), (60_003, 258, 0, 8)])   # short rows, several per tile
def test_planes_walked_by_rows(fd, oracle_mod, m, n, bin0, H):
    # more rows than the window table takes, and planes beside that limit: every defined sum
    P = synth.noise_plane(m, n, seed=n + H)
    S = oracle_mod.harmonic_sums(P, bin0, H)
    levels = np.array(fd.harmonic_levels(H))
    total = int((~np.isnan(S)).sum())
    buf, count = fd.harmonic_sum(torch.from_numpy(P).cuda(), bin0, H, [-1.0] * levels.size, max_cand=total + 64)
    assert int(count.item()) == total
    got = fd.harmonic_to_numpy(buf, count)
    j = np.log2(got["nharm"]).astype(np.int64)
    assert np.unique((j * m + got["tpl"]) * n + got["bin"]).size == total
    ref = S[j, got["tpl"], got["bin"]]
    h = levels[j]
    assert np.all(np.abs(got["power"].astype(np.float64) - ref) <= (h - 1) * U / (1 - (h - 1) * U) * ref)
