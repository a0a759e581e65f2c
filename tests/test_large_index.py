"""Index arithmetic at the largest lists the C ABI takes (m = 2^31 - 1, 2^32 - 2 entries),
compiled for the CPU from the header that the kernels and the host code share."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1302_4587_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def _run(tmp_path, body):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include <cstdio>\n#include "lm_internal.h"\nusing namespace lm;\n'
                   "int main() {\n" + body + "\nreturn 0;\n}\n")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", os.path.join(CUDA, "include"), str(src), "-o", str(exe)],
                   check=True)
    return subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()


def test_division_rounds_up_for_every_32_bit_number(tmp_path):
    xs = [0, 1, 31, 32, 33, 1023, 1024, 1025, (1 << 32) - 1025, (1 << 32) - 1024, (1 << 32) - 1023, (1 << 32) - 33,
          (1 << 32) - 32, (1 << 32) - 31, (1 << 32) - 2, (1 << 32) - 1]
    ds = [1, 32, 1024, 4096]
    body = "\n".join(f'printf("%u\\n", div_up({x}u, {d}u));' for x in xs for d in ds)
    assert [int(t) for t in _run(tmp_path, body)] == [-(-x // d) for x in xs for d in ds]


def test_tiles_cover_the_largest_lists(tmp_path):
    # round-0 tiles of 2m entries: as many as allocate tmap / rbits, none missing for m >= 2^31 - 511
    ms = [0, 1, 511, 512, 513, (1 << 31) - 513, (1 << 31) - 512, (1 << 31) - 511, (1 << 31) - 1]
    body = "\n".join(f'printf("%u %u\\n", div_up({2 * m}u, TILE0), TILE0);' for m in ms)
    got = [int(t) for t in _run(tmp_path, body)]
    for m, tiles, tile in zip(ms, got[::2], got[1::2]):
        assert (tiles - 1) * tile < max(2 * m, 1) <= max(tiles, 1) * tile, m
    # the build and its launch count them the same way, and a row's first tile too
    for f in ("lm_api.cpp", "lm_kernels.cu"):
        src = open(os.path.join(CSRC, f)).read()
        assert "div_up(" in src and "TILE0 - 1) / TILE0" not in src, f
