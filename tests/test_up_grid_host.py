"""The grid of the resident-row up phase, over every sector of up to 32 sites: no
more CTAs than asked for, also where one spin is empty or full and the sector has
one row or one column, and lists that fit in shared memory."""
import ctypes
import math
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1204_3425_gb300", "csrc")
MAX_ROW = (1 << 29) - 1                                # longer rows do not take this path


@pytest.fixture(scope="module")
def grid(tmp_path_factory):
    d = tmp_path_factory.mktemp("up_grid")
    (d / "g.cpp").write_text('#include "up_grid.h"\nextern "C" void grid(int64_t Dup, int64_t hops, int W, int64_t nchunk, int ctas, '
                             'int64_t* o) {\n const hub::UpGrid g = hub::make_up_grid(Dup, hops, W, nchunk, ctas);\n'
                             ' o[0] = g.gx; o[1] = g.gy; o[2] = g.cap; o[3] = g.W; o[4] = (int64_t)g.smem;\n}\n')
    so = str(d / "g.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "g.cpp"), "-o", so], check=True)
    f = ctypes.CDLL(so).grid
    f.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_int, ctypes.c_int64, ctypes.c_int, ctypes.c_void_p]

    def call(*a):
        o = (ctypes.c_int64 * 5)()
        f(*a, o)
        return list(o)
    return call


@pytest.mark.parametrize("ctas", [1, 2, 3 * 152, 4 * 152])
def test_no_more_ctas_than_asked_for(grid, ctas):
    for ns in range(1, 33):
        for nup in range(ns + 1):
            Dup = math.comb(ns, nup)
            hops = 2 * ns * math.comb(ns - 2, nup - 1) if ns > 2 and nup else 0        # ring
            W = 2 * min(nup, ns - nup)
            for ndn in range(ns + 1):
                Ddn = math.comb(ns, ndn)
                if Ddn > MAX_ROW:
                    continue
                for cols in (32, 64, 128):
                    nchunk = (Ddn + cols - 1) // cols
                    gx, gy, cap, w, smem = grid(Dup, hops, W, nchunk, ctas)
                    assert gx >= 1 and 1 <= gy <= nchunk and gx <= Dup
                    assert gx * gy <= ctas, (ns, nup, ndn, cols)
                    rounds = -(-nchunk // gy)           # chunks of a CTA: dealt evenly
                    assert gy == -(-nchunk // rounds)
                    assert 1 <= cap <= Dup and w >= max(W, 1)
                    assert smem == cap * (12 + 4 * w) and (cap == 1 or smem <= 24 * 1024)
