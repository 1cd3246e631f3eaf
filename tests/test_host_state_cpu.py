"""The library's host-side bookkeeping without a GPU: its objects linked with a
runtime whose device memory is host memory and whose kernels do nothing
(native/fake_cudart.cpp), so that allocations can be counted and made to fail."""
import glob
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
NATIVE = os.path.join(HERE, "native")


def run_check(name, tmp_path, *args):
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    from paper_2511_21198_gb300 import build
    build.build()
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc_path()))), "include")
    exe = str(tmp_path / name)
    src = os.path.join(NATIVE, name + ".cpp")
    if not os.path.exists(src):   # needs the kernels' own structures
        src = str(tmp_path / (name + ".o"))
        subprocess.run([build.nvcc_path(), *build.ARCH, "-std=c++17", "-I" + NATIVE, "-I" + build.CSRC,
                        "-I" + os.path.join(ROOT, "include"), "-c", os.path.join(NATIVE, name + ".cu"), "-o", src],
                       check=True)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", NATIVE, "-I", build.CSRC, "-I", os.path.join(ROOT, "include"),
                    "-isystem", cuda, src, os.path.join(NATIVE, "fake_cudart.cpp"),
                    *sorted(glob.glob(os.path.join(build.BUILD_DIR, "*.o"))), "-o", exe], check=True)
    out = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    return out.stdout


def test_loop_buffers(tmp_path):
    run_check("loop_buffers_check", tmp_path)


def test_batch_tile_widths(tmp_path):
    run_check("batch_tiles_check", tmp_path)


def test_tile_widths(tmp_path):
    from test_gpu_widths import WIDTHS
    out = run_check("tile_widths_check", tmp_path, *(v for n in WIDTHS for v in n))
    got = [[int(v) for v in line.split()] for line in out.splitlines()]
    assert got == [sum(map(list, w), []) for w in WIDTHS.values()]
    for kind in range(3):   # every width of each rule occurs
        assert {v for w in WIDTHS.values() for v in w[kind]} == {64, 128, 256}
