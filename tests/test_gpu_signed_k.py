"""Maps with k of both signs (n = 0) whose shifts are level on some row: k = 0 on rows that are no power
of two, bin edges on whole columns, tiles that start there.  Every cell, candidate and statistic equals
the oracle's (whole numbers: no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import (alloc_outputs, assert_candidates_equal, oracle_grid, read_cands, read_stats,
                      to_dev)
from oracle import gfh_oracle as O
from paper_1810_09784_gb300 import synth

pytestmark = pytest.mark.gpu


def fields_of(df, bin_lo, nb, n_fft, n_k, zero_row, t_first, t_hop, t_obs, dk):
    return dict(n=0.0, df=df, bin_lo=bin_lo, bin_hi=bin_lo + nb - 1, n_fft=n_fft, t_first=t_first, t_hop=t_hop,
                t_obs=t_obs, n_k=n_k, k_min=-zero_row * dk, dk=dk, f_max=0.0, ana_lo=bin_lo * df + df,
                ana_hi=(bin_lo + nb) * df - df, band_hz=1.0, list=0)


CASES = {
    "centred": fields_of(0.5, 300, 90, 500, 48, 24, 0.0, 1.0, 500.0, 0.5 / 499),
    "centred_18": fields_of(0.5, 300, 90, 500, 37, 18, 1.0, 1.0, 501.0, 0.5 / 500),
    "up_to_zero": fields_of(0.125, 8000, 160, 2519, 289, 288, 4.0, 4.0, 10080.0, 0.125 / 10080.0),
}


@pytest.mark.parametrize("tile", [None, (8, 256, 256), (16, 3072, 512)], ids=str)
@pytest.mark.parametrize("name", sorted(CASES))
def test_maps_equal_the_oracle(built_lib, gpu_ctx, name, tile):
    f = CASES[name]
    g = built_lib.grid_make(built_lib.Grid(**f))
    og = oracle_grid(f)
    hmap, cands, stats = alloc_outputs(torch, g)
    plan = built_lib.Plan(gpu_ctx, [g], [hmap], [cands], stats, tile=tile)
    fi, bj = synth.random_peaklist(f["n_fft"], f["bin_lo"] - 2, f["bin_hi"] + 2, 0.08, 5)
    off = to_dev(torch, np.array([0, len(fi)], np.int64))
    plan.execute(to_dev(torch, fi), to_dev(torch, bj), off, 1)
    torch.cuda.synchronize()
    assert gpu_ctx.check() == built_lib.GFH_OK
    ref = O.hough_map(og, fi, bj)
    got = hmap.cpu().numpy()
    assert np.array_equal(got[:, : g.n_x0], ref)
    assert not got[:, g.n_x0:].any()
    oc, _ = O.select_candidates(og, ref)
    assert_candidates_equal(read_cands(built_lib, cands), oc, g.n_bands)
    st = read_stats(built_lib, stats)[0]
    ana = np.array([b >= 0 for b in built_lib.grid_columns(g)[0]])
    sel = ref[:, ana].astype(np.int64)
    assert (int(st["sum"]), int(st["sum_sq"]), int(st["cells"])) == (sel.sum(), (sel * sel).sum(), sel.size)
    plan.close()
