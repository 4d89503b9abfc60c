"""Sparse maps, whose tiles keep one signed count per cell: tile ends, steep and level lines, both signs
of k, one row, a map's last columns, and sparse and dense maps in one plan.  Every map cell, candidate
and statistic equals the oracle's (whole numbers: no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import alloc_outputs, assert_candidates_equal, oracle_grid, read_cands, read_stats, to_dev
from oracle import gfh_oracle as O
from paper_1810_09784_gb300 import synth

from test_gpu_hough_events import fields_of

pytestmark = pytest.mark.gpu

# few FFTs over wide bins: fewer than two noise peaks per x0 column
CASES = {
    "few_ffts": fields_of(5.0, 150, 300, 24, 150),
    "wide_bins": fields_of(7.0, 140, 420, 60, 129),
    "steep": fields_of(6.0, 150, 300, 30, 67, dk_cols=1.9),
    "tiny_shift": fields_of(5.0, 150, 300, 24, 70, dk_cols=0.004),
    "k_min": fields_of(5.0, 150, 300, 24, 40, k_min_rows=300.0),
    "both_signs": fields_of(0.0, 300, 90, 20, 65, k_min_rows=-31.0),
    "one_row": fields_of(6.0, 150, 300, 30, 1),
    "near_the_line": fields_of(5.0, 200, 150, 120, 70),                     # 1.7 peaks per column
    "t0_zero": fields_of(5.0, 150, 300, 24, 9, t_first=0.0),
}
DENSE = fields_of(5.0, 200, 150, 200, 60)
# small plans take two counts whatever their maps: a map of 8 million cells without peaks beside them
LARGE = fields_of(7.0, 140, 420, 60, 20)


def check(gfh, ctx, fields, tile, seed=11):
    fields = fields + [dict(LARGE, list=len(fields))]
    grids = [gfh.grid_make(gfh.Grid(**f)) for f in fields]
    maps = [torch.full((g.n_k, g.ld_x0), -7, dtype=torch.int32, device="cuda") for g in grids]
    cands = [torch.zeros(g.n_bands * 64, dtype=torch.uint8, device="cuda") for g in grids]
    stats = torch.zeros(24 * len(grids), dtype=torch.uint8, device="cuda")
    plan = gfh.Plan(ctx, grids, maps, cands, stats, tile=tile)
    lists = [synth.random_peaklist(f["n_fft"], f["bin_lo"] - 2, f["bin_hi"] + 2, 0.08, seed + i)
             for i, f in enumerate(fields)]
    lists[-1] = tuple(x[:0] for x in lists[-1])
    off = np.cumsum([0] + [len(l[0]) for l in lists]).astype(np.int64)
    plan.execute(*(to_dev(torch, np.concatenate([l[k] for l in lists])) for k in (0, 1)), to_dev(torch, off),
                 len(lists))
    torch.cuda.synchronize()
    assert ctx.check() == gfh.GFH_OK
    st = read_stats(gfh, stats)
    assert not maps.pop().any()
    for i, (f, g) in enumerate(zip(fields[:-1], grids)):
        ref = O.hough_map(oracle_grid(f), *lists[i])
        got = maps[i].cpu().numpy()
        assert np.array_equal(got[:, : g.n_x0], ref)
        assert not got[:, g.n_x0:].any()
        oc, _ = O.select_candidates(oracle_grid(f), ref)
        assert_candidates_equal(read_cands(gfh, cands[i]), oc, g.n_bands)
        sel = ref[:, np.array([b >= 0 for b in gfh.grid_columns(g)[0]])].astype(np.int64)
        assert (int(st[i]["sum"]), int(st[i]["sum_sq"]), int(st[i]["cells"])) == (sel.sum(), (sel * sel).sum(), sel.size)
    plan.close()


@pytest.mark.parametrize("tile", [None, (8, 256, 256), (16, 3072, 1024)], ids=str)
@pytest.mark.parametrize("name", sorted(CASES))
def test_sparse_maps(built_lib, gpu_ctx, name, tile):
    f = CASES[name]
    g = built_lib.grid_make(built_lib.Grid(**f))
    assert 0.0755 * g.n_fft * (g.bin_hi - g.bin_lo + 1) < 2.0 * g.n_x0
    check(built_lib, gpu_ctx, [f], tile)


@pytest.mark.parametrize("tile", [None, (8, 256, 256)], ids=str)
def test_sparse_and_dense_maps_together(built_lib, gpu_ctx, tile):
    check(built_lib, gpu_ctx, [dict(CASES["few_ffts"], list=0), dict(DENSE, list=1), dict(CASES["steep"], list=2)], tile)
