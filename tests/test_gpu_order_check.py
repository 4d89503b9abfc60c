"""The order check over lists of very different lengths, empty ones among them: one descending pair
anywhere flags the input and leaves that list's map undrawn and no other; the step from one list to the
next is no pair.  Maps of the other lists equal the oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import oracle_grid, to_dev
from oracle import gfh_oracle as O
from paper_1810_09784_gb300 import synth

from test_gpu_unordered import fields_of

pytestmark = pytest.mark.gpu

LENGTHS = (0, 1, 30, 20000, 0, 3, 700, 2)


def lists():
    fi, bj = synth.random_peaklist(2000, 198, 322, 0.12, 3)
    out = []
    for n in LENGTHS:                              # every list starts again at the lowest bins
        at = np.sort(np.random.default_rng(n).choice(len(fi), n, replace=False)) if n else np.zeros(0, int)
        out.append((fi[at], bj[at]))
    return out


@pytest.mark.parametrize("where", [None, (3, 1), (3, 19999), (3, 9984), (3, 65), (2, 29), (6, 350), (7, 1)], ids=str)
def test_one_pair(built_lib, gpu_ctx, where):
    gfh = built_lib
    ls = [(f.copy(), b.copy()) for f, b in lists()]
    if where:
        l, p = where
        ls[l][1][p - 1] = ls[l][1][p] + 1          # descends at p (and may at p - 1 too)
    fields = [fields_of(n_fft=2000, n_k=12, lst=i) for i in range(len(ls))]
    grids = [gfh.grid_make(gfh.Grid(**f)) for f in fields]
    maps = [torch.full((g.n_k, g.ld_x0), -7, dtype=torch.int32, device="cuda") for g in grids]
    plan = gfh.Plan(gpu_ctx, grids, maps, None, None)
    off = np.cumsum([0] + [len(f) for f, _ in ls]).astype(np.int64)
    plan.execute(*(to_dev(torch, np.concatenate([x[k] for x in ls])) for k in (0, 1)), to_dev(torch, off), len(ls))
    torch.cuda.synchronize()
    assert gpu_ctx.check() == (gfh.GFH_ERR_INPUT if where else gfh.GFH_OK)
    for i, (g, m) in enumerate(zip(grids, maps)):
        got = m.cpu().numpy()[:, : g.n_x0]
        if where and i == where[0]:
            assert not got.any()
        else:
            assert np.array_equal(got, O.hough_map(oracle_grid(fields[i]), *ls[i]))
    plan.close()


def test_too_many_lists_stay_refused(built_lib, gpu_ctx):
    g = built_lib.grid_make(built_lib.Grid(**fields_of(nb=4, n_fft=8, n_k=4)))
    m = torch.zeros((g.n_k, g.ld_x0), dtype=torch.int32, device="cuda")
    plan = built_lib.Plan(gpu_ctx, [g], [m], None, None)
    z = torch.zeros(65537, dtype=torch.int64, device="cuda")
    w = torch.zeros(16, dtype=torch.int32, device="cuda")
    with pytest.raises(built_lib.GfhError):
        plan.execute(w, w, z, 65536)
    plan.execute(w, w, z, 65535)
    torch.cuda.synchronize()
    assert gpu_ctx.check() == built_lib.GFH_OK
    plan.close()
