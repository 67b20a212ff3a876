"""The compiled solver shapes' resources as the kernel takes them: the shared
memory of pgs_smem for every CTA an SM is to hold, aligned tiles, and registers
without heavy spilling (as the compiler reports them)."""
import os
import re
import subprocess

import pytest

from paper_2011_00459_gb300 import autotune, build

SRC = os.path.join(build.CSRC, "tds_solve.cu")
KB = 1024


def constant(name):
    return int(re.search(rf"constexpr \w+ {name} = (\d+);", open(SRC).read()).group(1))


def test_rings_fit():
    stages, row = constant("kStages"), constant("kRowBytes")
    tile = 32 * row
    assert tile % 128 == 0 and (32 * 68) % 128 == 0  # tiles, and the bulk copy's part of one, stay aligned
    src = open(SRC).read()
    # the formula below is the one compiled
    assert "return (size_t)(threads / 32) * ring_tiles(per_thread) * (kTileBytes + 8);" in src
    assert "ring_tiles(int per_thread) { return kStages * per_thread + 1; }" in src
    for threads, per, ctas in autotune.SHAPES:
        smem = (threads // 32) * (stages * per + 1) * (tile + 8)
        assert smem + 8 * KB <= 227 * KB, (threads, per)  # beside the static shared memory
        assert ctas * (smem + 9 * KB) <= 228 * KB, (threads, per)  # and what the system takes of each


@pytest.fixture(scope="module")
def reported(tmp_path_factory):
    out = tmp_path_factory.mktemp("ptxas") / "solve.o"
    r = subprocess.run([build.nvcc(), *build.flags(["-Xptxas", "-v"]), "-c", SRC, "-o", str(out)], capture_output=True,
                       text=True, check=True)
    got = {}
    for shape, spill, regs in re.findall(r"entry function '\S*k_pgsI((?:Li\d+E)+)\S*'.*?(\d+) bytes spill stores.*?Used (\d+) "
                                         r"registers", r.stderr, flags=re.S):
        threads, per, ctas = (int(v) for v in re.findall(r"Li(\d+)E", shape))
        got[threads, per, ctas] = int(spill), int(regs)
    return got


def test_registers(reported):
    """The default shape and 512x3 spill nothing; the others, which have 72 to 96 registers a thread, no more than a
    few values (reading records ahead they spilled up to 750 bytes and lost a third of their speed)."""
    assert sorted(reported) == sorted(autotune.SHAPES)
    for (threads, per, ctas), (spill, regs) in reported.items():
        assert ctas * threads * regs <= 65536
        assert spill == 0 if ctas * threads <= 512 else spill <= 256, (threads, per, spill)
