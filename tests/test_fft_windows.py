"""The window of FFTs that a tile reads of a bin, on the CPU: over the planner's own tiles, no FFT with
an edge in a tile is left out and none is taken for a cover of the tile that is not one.  Signed k
(n = 0, k_min < 0) with k = 0 on rows of every kind: there the line that the shifts follow is level and
its slope a difference of nearly equal numbers."""
import pathlib
import subprocess

import pytest

from paper_1810_09784_gb300 import build

HERE = pathlib.Path(__file__).resolve().parent


@pytest.fixture(scope="module")
def windows(tmp_path_factory):
    """Runs cases (n, df, bin_lo, bin_hi, n_fft, t_first, n_k, k_min_rows, dk_cols, rows, cols)."""
    exe = tmp_path_factory.mktemp("windows") / "fft_windows"
    cuda = pathlib.Path(build._nvcc()).resolve().parent.parent / "include"
    # the planner alone: what calls the CUDA runtime is unreachable and dropped
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", str(build.ROOT / "include"), "-I",
                        str(build.CSRC), "-I", str(cuda), str(HERE / "fft_windows.cpp"), "-o", str(exe),
                        "-ffunction-sections", "-Wl,--gc-sections"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(cases):
        text = "\n".join(" ".join(repr(v) for v in c) for c in cases)
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
        rows = [tuple(int(v) for v in line.split()) for line in out.splitlines()]
        assert len(rows) == len(cases)
        return rows
    return run


def check(windows, cases):
    rows = windows(cases)
    bad = [(c, r) for c, r in zip(cases, rows) if r[2] or r[3]]
    assert not bad, bad
    assert all(r[1] > 0 for r in rows)
    return rows


@pytest.mark.parametrize("n_fft", [150, 500, 2519])
@pytest.mark.parametrize("tile", [(0, 0), (8, 128), (16, 1024)], ids=str)
def test_signed_k(windows, n_fft, tile):
    nb = 90 if n_fft <= 500 else 40
    check(windows, [(0.0, 0.5, 300, 299 + nb, n_fft, t_first, n_k, -float(zero), dk, *tile)
                    for zero in (12, 18, 20, 24, 48, 96, 16, 32) for n_k in (zero + 1, 2 * zero)
                    for t_first, dk in ((0.0, 1.0), (1.0, 1.0), (1.0, 0.7))])


@pytest.mark.parametrize("rows", [288, 600, 1120])
def test_k_ending_at_zero(windows, rows):
    check(windows, [(0.0, 0.125, 8000, 8159, 2519, 1.0, rows + 1, -float(rows), 2519 / 2520, *tile)
                    for tile in ((0, 0), (8, 128))])


def test_power_laws(windows):
    rows = check(windows, [(n, 0.5, 200, 349, n_fft, t_first, 131, k_min, dk, *tile)
                           for n in (2.0, 5.0, 7.0) for n_fft in (1, 2, 60, 500) for t_first in (0.0, 1.0)
                           for k_min in (0.0, 300.0) for dk in (0.004, 1.0, 1.9) for tile in ((0, 0), (8, 128))
                           if n_fft > 1 or t_first > 0.0])
    assert sum(r[1] for r in rows) > 0


def test_bins_wider_than_tiles(windows):
    rows = check(windows, [(n, 0.5, lo, lo + 300, 500, 1.0, 200, k_min, 1.0, *tile)
                           for n, lo in ((7.0, 140), (5.0, 100)) for k_min in (0.0, 300.0)
                           for tile in ((0, 0), (8, 128), (16, 256))])
    assert all(r[4] > 0 for r in rows)                   # tiles that some FFT covers
