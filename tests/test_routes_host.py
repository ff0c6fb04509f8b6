"""The host rules that choose how a call runs (csrc/routes.h), compiled for the
CPU and checked on either side of their lines."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2106_11476_gb300", "csrc")

WRAPPER = r"""
#include "routes.h"
extern "C" int sources_apart(long long h, long long t, long long e, int n) { return fw2::sources_apart(h, t, e, n); }
extern "C" int record_apart(long long l, long long c) { return fw2::record_apart(l, c); }
extern "C" int copy_by_kernel(int c, int h, int b, int a) { return fw2::copy_by_kernel(c, h, b, a); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("routes")
    src, lib = d / "routes.cpp", d / "libroutes.so"
    src.write_text(WRAPPER)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    m = C.CDLL(str(lib))
    m.sources_apart.argtypes = [C.c_longlong, C.c_longlong, C.c_longlong, C.c_int]
    m.record_apart.argtypes = [C.c_longlong, C.c_longlong]
    return m


def test_dense_sources_and_long_chains_run_apart(rules):
    """Arrays and lines stay inside the half steps; a field full of sources, a
    point in every half tile of a large grid, and thousands of entries of one
    cell do not."""
    def apart(nx, ny, targets, extra=0, half_tiles=None):
        tiles = -(-nx // 128) * -(-ny // 8)
        return bool(rules.sources_apart(min(tiles, targets) if half_tiles is None else half_tiles, targets, extra, 152))
    assert not apart(250, 186, 0, half_tiles=0)
    assert not apart(4096, 4096, 1408, half_tiles=17)            # an array of 128 elements of 11 cells
    assert not apart(4096, 4096, 4096, half_tiles=512)           # a line along y
    assert not apart(512, 512, 65536) and apart(512, 512, 512 * 512)
    assert apart(2048, 1024, 2048 * 1024) and apart(2048, 1024, 2048 * 256)
    assert apart(4096, 4096, 20000)                              # scattered over every half tile
    assert not apart(250, 186, 13, extra=3000, half_tiles=3) and apart(250, 186, 13, extra=4000, half_tiles=3)


@pytest.mark.parametrize("longest,cells,apart", [(1, 256, False), (11, 704, False), (384, 6144, False), (385, 385, True),
                                                 (1, 1 << 19, False), (1, (1 << 19) + 1, True),
                                                 (2**31, 2**31, True)])
def test_long_groups_and_dense_sensors_are_recorded_apart(rules, longest, cells, apart):
    assert bool(rules.record_apart(longest, cells)) is apart


@pytest.mark.parametrize("ctx,current,buf,aligned,kernel", [
    (0, 0, 0, 1, True), (1, 1, 1, 1, True),
    (0, 0, 0, 0, False), (0, 0, -1, 1, False),            # odd address, host memory
    (0, 0, 1, 1, False), (1, 0, 1, 1, False),             # a buffer of another device, another device current
    (0, 1, 1, 1, False), (1, 0, 0, 1, False)])            # both: the buffer's device is current, the context's is not
def test_field_copies_take_the_kernel_on_the_contexts_own_device_only(rules, ctx, current, buf, aligned, kernel):
    assert bool(rules.copy_by_kernel(ctx, current, buf, aligned)) is kernel
