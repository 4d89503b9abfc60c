"""FFT indices past a map's last FFT in bins far wider than a tile, whose FFTs are mostly counted without
a walk: the input is flagged, the indices are drawn nowhere, and so the map does not depend on the tile
shape: it equals the oracle's map of the peaks in range (whole numbers: no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import oracle_grid, to_dev
from oracle import gfh_oracle as O
from paper_1810_09784_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [None, (8, 128, 256), (16, 3072, 512), (32, 640, 1024)], ids=str)
@pytest.mark.parametrize("shuffle", [False, True])
def test_indices_past_the_last_fft(built_lib, gpu_ctx, tile, shuffle):
    n_fft = 300
    f = dict(n=7.0, df=0.5, bin_lo=140, bin_hi=399, n_fft=n_fft, t_first=1.0, t_hop=1.0, t_obs=301.0, n_k=60,
             k_min=0.0, dk=0.0, f_max=0.0, ana_lo=71.0, ana_hi=197.0, band_hz=1.0, list=0)
    g = built_lib.grid_make(built_lib.Grid(**f))
    hmap = torch.full((g.n_k, g.ld_x0), -7, dtype=torch.int32, device="cuda")
    plan = built_lib.Plan(gpu_ctx, [g], [hmap], None, None, tile=tile)
    fi, bj = synth.random_peaklist(n_fft + 40, f["bin_lo"] - 2, f["bin_hi"] + 2, 0.08, 9)
    fi[bj == 150] = n_fft + 1                     # a bin without any index in range
    keep = fi < n_fft
    if shuffle:
        order = np.lexsort((np.random.default_rng(2).random(len(fi)), bj))
        fi, bj = fi[order], bj[order]
        keep = keep[order]
    off = to_dev(torch, np.array([0, len(fi)], np.int64))
    plan.execute(to_dev(torch, fi), to_dev(torch, bj), off, 1)
    torch.cuda.synchronize()
    assert gpu_ctx.check() == built_lib.GFH_ERR_INPUT
    order = np.lexsort((fi[keep], bj[keep]))
    ref = O.hough_map(oracle_grid(f), fi[keep][order], bj[keep][order])
    assert np.array_equal(hmap.cpu().numpy()[:, : g.n_x0], ref)
    plan.close()
    assert gpu_ctx.check() == built_lib.GFH_OK
