"""The bins that a tile reads, on the CPU: every bin of which some FFT meets the tile, for planned tiles
and for those of a plan that is executed once."""
import pytest

from test_fft_windows import check, windows  # noqa: F401


@pytest.mark.parametrize("n", [0.0, 2.0, 5.0, 7.0])
@pytest.mark.parametrize("tile", [(0, 0), (-1, 0)], ids=str)
def test_no_bin_is_left_out(windows, n, tile):  # noqa: F811
    check(windows, [(n, 0.5, lo, lo + nb, n_fft, 1.0, n_k, k_min, dk, *tile)
                    for lo, nb in ((150, 60), (300, 1), (400, 300)) for n_fft, n_k in ((40, 131), (300, 7), (300, 300))
                    for k_min in ((0.0, -20.0) if n == 0.0 else (0.0, 50.0)) for dk in (0.01, 1.0, 2.0)])
