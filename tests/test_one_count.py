"""The rule for one count per cell, on the CPU: the maps of the GPU parity tests stand on the side they are
there for."""
from host_program import compile_host, run_host


def ask(f):
    t_obs = f["n_fft"] + 1.0
    f_max = f["bin_hi"] * 0.5
    m = 1.0 if f["n"] == 0.0 else f["n"] - 1.0
    dx0 = m * 0.5 / f_max ** f["n"]
    dk_cols = f["dk"] * m * t_obs / dx0
    return (f["n"], f["bin_lo"], f["bin_hi"] - f["bin_lo"] + 1, f["n_fft"], f["n_k"], f["k_min"] / f["dk"], dk_cols)


def test_sides_of_the_line(tmp_path):
    import test_gpu_sparse as sparse
    import test_gpu_x_direction as xdir
    exe = compile_host("one_count.cpp", tmp_path)
    names = sorted(sparse.CASES)
    assert run_host(exe, [ask(sparse.CASES[n]) for n in names]) == [(1, 0)] * len(names)
    assert run_host(exe, [ask(sparse.DENSE), ask(sparse.LARGE)]) == [(0, 0), (1, 0)]
    names = sorted(xdir.CASES)
    got = dict(zip(names, run_host(exe, [ask(xdir.CASES[n]) for n in names])))
    assert all(x == 1 for _, x in got.values())
    assert got["sparse"][0] == 1 and got["far"][0] == 1 and got["dense"][0] == 0 and got["just_over"][0] == 0


def test_peaks_that_share_columns(tmp_path):
    """1.5 peaks per column: one count where neighbouring peaks lie apart, two where they share a column."""
    exe = compile_host("one_count.cpp", tmp_path)
    assert run_host(exe, [(5.0, 200, 150, 106, 70, 0.0, 1.0), (5.0, 200, 150, 106, 70, 0.0, 0.05)]) == [(1, 0), (0, 0)]
