"""The FP64 form's tile rule (csrc/tile_rule.h), compiled for the host."""
import functools
import os
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2305_00762_gb300", "csrc")
SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "tile_rule.h"
int main(int, char** a)
{
    const gbr::TileShape t = gbr::fixed_tile_rule(atoi(a[1]), atoi(a[2]), atoi(a[3]), atoi(a[4]) != 0, atoi(a[5]) != 0);
    std::printf("%dx%d", t.bx, t.by);
    return 0;
}
"""


@functools.lru_cache(None)
def _program():
    d = tempfile.mkdtemp()
    src, exe = os.path.join(d, "t.cpp"), os.path.join(d, "t")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, src, "-o", exe], check=True)
    return exe


@functools.lru_cache(None)
def shape(nx, ny, sms=152, cons=False, viscous=False):
    """Name of the tile a grid takes, e.g. '16x8'."""
    args = [str(int(v)) for v in (nx, ny, sms, cons, viscous)]
    return subprocess.run([_program()] + args, capture_output=True, text=True, check=True).stdout
