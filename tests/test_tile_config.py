"""Requested tile shapes, on the CPU: the drawing form selects nothing, so the default shape is planned
with either; refused shapes stay refused."""
from host_program import compile_host, run_host
from paper_1810_09784_gb300 import gfh


def test_form_selects_nothing(tmp_path):
    exe = compile_host("tile_config.cpp", tmp_path)
    ask = [(0, 0, 0, 0), (16, 3072, 512, 0), (16, 3072, 512, 1), (0, 0, 0, 1), (16, 3072, 1024, 0), (16, 3072, 1024, 1),
           (8, 256, 256, 1)]
    got = run_host(exe, ask)
    assert [r[0] for r in got] == [gfh.GFH_OK] * len(ask)
    assert [r[4] for r in got] == [0] * len(ask)
    assert [r[5] for r in got] == [1, 1, 1, 1, 0, 0, 0]
    assert got[4] == got[5]


def test_refused_shapes(tmp_path):
    exe = compile_host("tile_config.cpp", tmp_path)
    bad = [(5, 3072, 512, 0), (16, 100, 512, 0), (16, 4224, 512, 0), (16, 3072, 128, 0), (8, 3072, 1024, 0),
           (16, 3072, 512, 2), (16, 3072, 512, -1), (8, -128, 256, 0)]
    assert [r[0] for r in run_host(exe, bad)] == [gfh.GFH_ERR_ARG] * len(bad)
