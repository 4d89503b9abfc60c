"""Parity of the event-drawn tiles where their rules change: shifts per row too small for the stepped
form, between one and two columns, and both signs of k; row counts beside a tile's; bins far wider
than a tile (counted without a walk); peak lists in and out of FFT order; bands without peaks.  Every
map cell, candidate and statistic equals the oracle's (whole numbers: no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import (alloc_outputs, assert_candidates_equal, oracle_grid, read_cands, read_stats,
                      to_dev)
from oracle import gfh_oracle as O
from paper_1810_09784_gb300 import synth

pytestmark = pytest.mark.gpu


def fields_of(n, bin_lo, nb, n_fft, n_k, dk_cols=1.0, k_min_rows=0.0, t_first=1.0):
    """A grid whose line moves dk_cols x0 columns per k row at the last FFT."""
    df, t_obs = 0.5, float(n_fft + 1)
    f_max = (bin_lo + nb - 1) * df
    slope = 1.0 if n == 0.0 else n - 1.0
    dx0 = df if n == 0.0 else (n - 1.0) * df / f_max ** n
    dk = dk_cols * dx0 / (slope * t_obs)
    return dict(n=n, df=df, bin_lo=bin_lo, bin_hi=bin_lo + nb - 1, n_fft=n_fft, t_first=t_first, t_hop=1.0,
                t_obs=t_obs, n_k=n_k, k_min=k_min_rows * dk, dk=dk, f_max=0.0,
                ana_lo=bin_lo * df + 1.0, ana_hi=(bin_lo + nb) * df - 3.0, band_hz=1.0, list=0)


CASES = {
    "tiny_shift": fields_of(5.0, 200, 150, 60, 70, dk_cols=0.004),          # S below 2^25 for every FFT
    "small_shift": fields_of(5.0, 200, 150, 200, 129, dk_cols=0.03),        # both forms of the rows
    "one_column": fields_of(4.0, 200, 150, 120, 131, dk_cols=1.0),
    "steep": fields_of(3.0, 200, 150, 120, 67, dk_cols=1.9),                # two events of an edge per row
    "k_min": fields_of(5.0, 220, 130, 120, 40, k_min_rows=300.0),
    "wide_bins": fields_of(7.0, 140, 420, 300, 200),                        # widest bin: 2000 columns
    "both_signs": fields_of(0.0, 300, 90, 150, 65, k_min_rows=-32.0),
    "t0_zero": fields_of(5.0, 200, 100, 130, 9, t_first=0.0),               # the first FFT never moves
    "one_row": fields_of(6.0, 200, 100, 130, 1),
}


def peaks_of(f, seed, shuffle=False, empty=False):
    fi, bj = synth.random_peaklist(f["n_fft"], f["bin_lo"] - 2, f["bin_hi"] + 2, 0.08, seed)
    if empty:                                     # only the outer quarters of the band hold peaks
        nb = f["bin_hi"] - f["bin_lo"] + 1
        keep = (bj < f["bin_lo"] + nb // 4) | (bj > f["bin_hi"] - nb // 4)
        fi, bj = fi[keep], bj[keep]
    if shuffle:
        order = np.lexsort((np.random.default_rng(seed).random(len(fi)), bj))
        fi, bj = fi[order], bj[order]
    return fi, bj


@pytest.mark.parametrize("tile", [None, (8, 256, 256), (32, 640, 1024)], ids=str)
@pytest.mark.parametrize("name", sorted(CASES))
def test_maps_equal_the_oracle(built_lib, gpu_ctx, name, tile):
    f = CASES[name]
    g = built_lib.grid_make(built_lib.Grid(**f))
    og = oracle_grid(f)
    hmap, cands, stats = alloc_outputs(torch, g)
    plan = built_lib.Plan(gpu_ctx, [g], [hmap], [cands], stats, tile=tile)
    for kw in (dict(), dict(shuffle=True), dict(empty=True)):
        fi, bj = peaks_of(f, 11, **kw)
        off = to_dev(torch, np.array([0, len(fi)], np.int64))
        hmap.fill_(-7)
        plan.execute(to_dev(torch, fi), to_dev(torch, bj), off, 1)
        torch.cuda.synchronize()
        assert gpu_ctx.check() == built_lib.GFH_OK
        ref = O.hough_map(og, fi, bj)
        got = hmap.cpu().numpy()
        assert np.array_equal(got[:, : g.n_x0], ref), kw
        assert not got[:, g.n_x0:].any()
        oc, _ = O.select_candidates(og, ref)
        assert_candidates_equal(read_cands(built_lib, cands), oc, g.n_bands)
        st = read_stats(built_lib, stats)[0]
        ana = np.array([b >= 0 for b in built_lib.grid_columns(g)[0]])
        sel = ref[:, ana].astype(np.int64)
        assert (int(st["sum"]), int(st["sum_sq"]), int(st["cells"])) == (sel.sum(), (sel * sel).sum(), sel.size)
    plan.close()
