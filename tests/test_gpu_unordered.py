"""Peak lists in bin order whose FFTs are in no order inside a bin: ordered by blocks of FFTs on the way,
or walked whole where they hold more peaks than there is room to order.  Equal FFTs in a bin, more
FFTs than a block table of 64 each covers, lists of which a map reads a part, lists of both kinds in
one plan, and the x-direction form.  Every cell equals the oracle's (whole numbers: no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import oracle_grid, to_dev
from oracle import gfh_oracle as O
from paper_1810_09784_gb300 import synth

pytestmark = pytest.mark.gpu


def fields_of(n=5.0, bin_lo=200, nb=120, n_fft=500, n_k=60, dk_cols=1.0, lst=0):
    df, t_obs = 0.5, float(n_fft + 1)
    f_max = (bin_lo + nb - 1) * df
    dk = dk_cols * (n - 1.0) * df / f_max ** n / ((n - 1.0) * t_obs)
    return dict(n=n, df=df, bin_lo=bin_lo, bin_hi=bin_lo + nb - 1, n_fft=n_fft, t_first=1.0, t_hop=1.0, t_obs=t_obs,
                n_k=n_k, k_min=0.0, dk=dk, f_max=0.0, ana_lo=bin_lo * df, ana_hi=(bin_lo + nb) * df, band_hz=1.0,
                list=lst)


def shuffled(fi, bj, seed):
    order = np.lexsort((np.random.default_rng(seed).random(len(fi)), bj))
    return fi[order], bj[order]


def run(gfh, ctx, fields, lists, tile=None):
    grids = [gfh.grid_make(gfh.Grid(**f)) for f in fields]
    maps = [torch.full((g.n_k, g.ld_x0), -7, dtype=torch.int32, device="cuda") for g in grids]
    plan = gfh.Plan(ctx, grids, maps, None, None, tile=tile)
    off = np.cumsum([0] + [len(l[0]) for l in lists]).astype(np.int64)
    args = [to_dev(torch, np.concatenate([l[k] for l in lists])) for k in (0, 1)] + [to_dev(torch, off)]
    for _ in range(2):                            # the second run meets the first one's copies
        plan.execute(*args, len(lists))
    torch.cuda.synchronize()
    assert ctx.check() == gfh.GFH_OK
    for f, g, m in zip(fields, grids, maps):
        fi, bj = lists[f["list"]]
        order = np.lexsort((fi, bj))
        ref = O.hough_map(oracle_grid(f), fi[order], bj[order])
        assert np.array_equal(m.cpu().numpy()[:, : g.n_x0], ref)
    plan.close()


@pytest.mark.parametrize("tile", [None, (8, 256, 256)], ids=str)
@pytest.mark.parametrize("density", [0.01, 0.08, 0.3, 0.9])
def test_densities(built_lib, gpu_ctx, density, tile):
    f = fields_of()
    run(built_lib, gpu_ctx, [f], [shuffled(*synth.random_peaklist(500, 195, 330, density, 3), 4)], tile)


def test_equal_ffts_in_a_bin(built_lib, gpu_ctx):
    fi, bj = synth.random_peaklist(500, 198, 322, 0.03, 5)
    order = np.argsort(np.tile(bj, 3), kind="stable")
    run(built_lib, gpu_ctx, [fields_of()], [shuffled(np.tile(fi, 3)[order], np.tile(bj, 3)[order], 6)])


@pytest.mark.parametrize("n_fft", [1, 33, 513, 20000])
def test_fft_counts(built_lib, gpu_ctx, n_fft):
    f = fields_of(nb=12, n_fft=n_fft, n_k=40)
    run(built_lib, gpu_ctx, [f], [shuffled(*synth.random_peaklist(n_fft, 198, 214, 0.08, 7), 8)])


def test_parts_of_lists_of_both_kinds(built_lib, gpu_ctx):
    a, b, c = (synth.random_peaklist(500, 150, 420, 0.08, s) for s in (1, 2, 3))
    fields = [fields_of(bin_lo=200, nb=60, lst=1), fields_of(bin_lo=330, nb=40, n_k=20, lst=1),
              fields_of(n=3.0, bin_lo=250, nb=50, lst=0), fields_of(n=7.0, bin_lo=180, nb=50, lst=2)]
    run(built_lib, gpu_ctx, fields, [a, shuffled(*b, 9), shuffled(*c, 10)])


@pytest.mark.parametrize("tile", [None, (4, 1024, 256), (32, 1024, 1024)], ids=str)
@pytest.mark.parametrize("density", [0.01, 0.08, 0.3])
@pytest.mark.parametrize("order", [True, False])
def test_x_direction(built_lib, gpu_ctx, density, tile, order):
    f = fields_of(n_k=37, dk_cols=5.0)
    lst = synth.random_peaklist(500, 195, 330, density, 3)
    run(built_lib, gpu_ctx, [f], [lst if order else shuffled(*lst, 4)], tile)
