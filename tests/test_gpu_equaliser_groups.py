"""The equaliser's peaks where its two kernels meet: bands below, at and beside whole groups of 32 bins,
FFT counts beside whole words, and spectra whose means sit at the edge of float32's range (zeros,
denormals, one infinite bin), all equal to the oracle's (the same float32 operations: no tolerance)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_util import to_dev
from oracle import gfh_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_fft", [1, 31, 33, 70])
@pytest.mark.parametrize("n_bins", [1, 2, 31, 32, 33, 63, 64, 65, 97, 300])
@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e-37, 1e-41, 0.0])
def test_peaks_equal_the_oracle(built_lib, gpu_ctx, n_fft, n_bins, scale):
    rng = np.random.default_rng(n_bins * 1000 + n_fft)
    lo = 140
    P = (rng.exponential(size=(n_fft, lo + n_bins + 3)) * scale).astype(np.float32)
    if scale == 1.0 and n_bins > 20:
        P[n_fft // 2, lo + 5] = np.inf
        P[:, lo + 17] *= 50.0
    cap = n_fft * n_bins + 1
    fo, bo = (torch.empty(cap, dtype=torch.int32, device="cuda") for _ in range(2))
    with np.errstate(all="ignore"):
        ofi, obj = O.peaks_from_power(P, lo, lo + n_bins - 1)
    n = gpu_ctx.peaks_from_power(to_dev(torch, P), lo, lo + n_bins - 1, 2.5, fo, bo)
    assert np.array_equal(bo[:n].cpu().numpy(), obj) and np.array_equal(fo[:n].cpu().numpy(), ofi)
    cnt = torch.empty(1, dtype=torch.int64, device="cuda")
    fo.zero_()
    built_lib.peaks_from_power_static(torch.cuda.current_stream(), to_dev(torch, P), lo, lo + n_bins - 1, 2.5,
                                      fo, bo, cnt)
    assert int(cnt.item()) == n and np.array_equal(fo[:n].cpu().numpy(), ofi)
