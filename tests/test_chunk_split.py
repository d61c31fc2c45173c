"""The acceptance's division of chunks among warps (csrc/chunk_split.h),
compiled for the host and checked over every warp that a launch has."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2505_12728_gb300 import build_lib

SOURCE = """
#include "chunk_split.h"
extern "C" void ranges(int U, int most, int warps, int *nw, int *u0, int *u1) {
  *nw = sf::chunk_warps(U, most);
  for (int g = 0; g < warps; ++g) {
    const sf::ChunkRange r = sf::chunk_range(g, U, *nw);
    u0[g] = r.u0;
    u1[g] = r.u1;
  }
}
extern "C" void owners(int U, int nw, int n, const int *u, int *g) {
  for (int i = 0; i < n; ++i) g[i] = sf::chunk_owner(u[i], U, nw);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("chunk_split")
    src, so = os.path.join(d, "t.cpp"), os.path.join(d, "t.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", build_lib.CSRC, src, "-o", so], check=True)
    return ctypes.CDLL(so)


def split(lib, U, sms):
    most = 2 * sms * 8
    warps = (min(U, most) + 7) // 8 * 8            # whole CTAs of eight warps
    nw = ctypes.c_int()
    u0, u1 = np.empty(warps, np.int32), np.empty(warps, np.int32)
    lib.ranges(U, most, warps, ctypes.byref(nw), u0.ctypes.data_as(ctypes.c_void_p), u1.ctypes.data_as(ctypes.c_void_p))
    return nw.value, u0, u1


@pytest.mark.parametrize("U", [
    1, 7, 8, 9, 66,      # fewer chunks than warps of a CTA, one more, a part-filled last CTA
    745,                 # one sequence, k = 4, V = 152064
    2425, 2431, 2432,    # just below and at two CTAs per SM of 152 SMs
    2433, 2440, 21456,   # above: several chunks to a warp
    2_000_000_011,       # the products need 64 bits
])
@pytest.mark.parametrize("sms", [152, 148])
def test_every_chunk_has_one_owner_and_no_warp_more(lib, U, sms):
    nw, u0, u1 = split(lib, U, sms)
    assert (u0 >= 0).all() and (u1 <= U).all() and (u0 <= u1).all()
    mine = u1 > u0
    assert mine[:nw].all() and not mine[nw:].any()
    assert u0[0] == 0 and u1[nw - 1] == U and (u0[1:nw] == u1[:nw - 1]).all()
    at = np.concatenate([u0[:nw], u1[:nw] - 1]).astype(np.int32)
    g = np.empty_like(at)
    lib.owners(U, nw, len(at), at.ctypes.data_as(ctypes.c_void_p), g.ctypes.data_as(ctypes.c_void_p))
    np.testing.assert_array_equal(g, np.concatenate([np.arange(nw)] * 2))
