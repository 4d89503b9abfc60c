"""Compiles a test program that includes the library's host planner (no GPU)."""
import pathlib
import subprocess

from paper_1810_09784_gb300 import build

HERE = pathlib.Path(__file__).resolve().parent


def compile_host(source: str, folder) -> str:
    exe = pathlib.Path(folder) / pathlib.Path(source).stem
    cuda = pathlib.Path(build._nvcc()).resolve().parent.parent / "include"
    # the planner alone: what calls the CUDA runtime is unreachable and dropped
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", str(build.ROOT / "include"), "-I",
                        str(build.CSRC), "-I", str(cuda), str(HERE / source), "-o", str(exe),
                        "-ffunction-sections", "-Wl,--gc-sections"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(exe)


def run_host(exe: str, rows) -> list:
    text = "\n".join(" ".join(repr(v) for v in r) for r in rows)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
    return [tuple(int(v) for v in line.split()) for line in out.splitlines()]
