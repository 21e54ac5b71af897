"""Index arithmetic of the friends-of-friends kernels for every lattice up to np^3 = 2^31 - 1, on the CPU.

The statements by which the kernels of fof.cu walk the records and particles are taken from the source as they
stand, compiled as host C++ with the built-in variables as arguments, and run for the threads at the ends of the
first and last blocks, on both kinds of grid the launches use: one thread per element, and (loops only) a grid
capped at 152 x 64 blocks.  Every index they produce must lie in [0, n), and a thread must stop."""

import ctypes
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = os.path.join(ROOT, "paper_1507_05329_gb300", "csrc", "fof.cu")

# for (TYPE t = .. blockIdx ..; t < n; t += ..)    and    const TYPE t = .. blockIdx ..;  if (t >= n) return;
LOOP = re.compile(r"for \(((?:long long|int) (\w+) = [^;]*blockIdx[^;]*; \2 < n; [^;{}]*)\)(?= ?\{|\n)")
ONE = re.compile(r"const ((?:long long|int) (\w+) = [^;]*blockIdx[^;]*;)\s*if \(\2 >= n\) return;")

HEAD = """
struct Dim { unsigned x; };
static void put(long long v, long long* out, int* count, int room) { if (*count < room) out[*count] = v; ++*count; }
"""
ARGS = "(int n, Dim gridDim, Dim blockDim, Dim blockIdx, Dim threadIdx, long long* out, int* count, int room)"


def walks():
    with open(SOURCE) as f:
        text = f.read()
    loops = [f"for ({m.group(1)}) {{ put({m.group(2)}, out, count, room); if (*count >= room) return; }}"
             for m in LOOP.finditer(text)]
    ones = [f"const {m.group(1)} if ({m.group(2)} >= n) return; put({m.group(2)}, out, count, room);"
            for m in ONE.finditer(text)]
    # no walk of another form: every use of blockIdx.x but the row walk of k_fof_prepare is one of these
    assert len(loops) + len(ones) == text.count("blockIdx.x") - 1
    return loops + ones, len(loops)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fof_index")
    found, loops = walks()
    body = HEAD + "".join(f'static void walk{i}{ARGS} {{ {w} }}\n' for i, w in enumerate(found))
    body += 'extern "C" void walk(int k, int n, unsigned grid, unsigned block, unsigned thread, long long* out, int* count, int room) {\n'
    body += "  const Dim g{grid}, t{256u}, b{block}, i{thread};\n  *count = 0;\n"
    body += "".join(f"  if (k == {i}) walk{i}(n, g, t, b, i, out, count, room);\n" for i in range(len(found))) + "}\n"
    src, so = d / "walk.cpp", d / "walk.so"
    src.write_text(body)
    # signed overflow wraps, as on the GPU
    subprocess.run(["g++", "-O1", "-fwrapv", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so)), len(found), loops


@pytest.mark.parametrize("n", [1, 255, 257, 64 ** 3, 1024 ** 3, 1080 ** 3, 1152 ** 3, 1200 ** 3, 1250 ** 3, 1280 ** 3, 2 ** 31 - 1])
def test_every_index_is_in_range(lib, n):
    so, count, loops = lib
    assert count >= 8
    room = 4096
    full = (n + 255) // 256
    for k in range(count):
        for grid in (full, min(full, 152 * 64)) if k < loops else (full,):
            for block in {0, grid // 2, max(grid - 2, 0), grid - 1}:
                for thread in (0, 1, 31, 255):
                    out, got = (ctypes.c_longlong * room)(), ctypes.c_int()
                    so.walk(k, n, grid, block, thread, out, ctypes.byref(got), room)
                    first, step = block * 256 + thread, grid * 256
                    want = [first + i * step for i in range(room) if first + i * step < n]
                    assert list(out[:min(got.value, room)]) == want, (k, n, grid, block, thread)
