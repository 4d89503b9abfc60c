"""Maps that read bins of one list far apart, adjacent, overlapping and nested: the index covers the bins
that maps read and not those between.  Every cell equals the oracle's (whole numbers: no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1810_09784_gb300 import synth

from test_gpu_unordered import fields_of, run, shuffled

pytestmark = pytest.mark.gpu

FAR = 2_000_000_000


def far_map(bin_lo, nb, n_k, n_fft, lst=0):
    """n = 0 (x = -f) at the top of the bins' range."""
    df, t_obs = 0.5, float(n_fft + 1)
    dk = df / t_obs
    return dict(n=0.0, df=df, bin_lo=bin_lo, bin_hi=bin_lo + nb - 1, n_fft=n_fft, t_first=1.0, t_hop=1.0, t_obs=t_obs,
                n_k=n_k, k_min=-(n_k // 2) * dk, dk=dk, f_max=0.0, ana_lo=bin_lo * df, ana_hi=(bin_lo + nb) * df,
                band_hz=1.0, list=lst)


@pytest.mark.parametrize("shuffle", [False, True])
def test_runs_of_bins(built_lib, gpu_ctx, shuffle):
    n_fft = 200
    near = synth.random_peaklist(n_fft, 190, 420, 0.08, 3)
    far = synth.random_peaklist(n_fft, FAR - 5, FAR + 70, 0.08, 4)
    lst = tuple(np.concatenate([a, b]) for a, b in zip(near, far))
    if shuffle:
        lst = shuffled(*lst, 5)
    f = lambda lo, nb, n_k=20, ffts=n_fft: fields_of(bin_lo=lo, nb=nb, n_k=n_k, n_fft=ffts)     # noqa: E731
    fields = [far_map(FAR, 60, 17, n_fft), f(200, 40), f(240, 20), f(250, 60, 33), f(270, 5), f(380, 30)]
    run(built_lib, gpu_ctx, fields, [lst])
