"""The launch shape of small arrays, on the host: the rule is compiled from the library's own header.
No GPU."""
import os
import subprocess

import pytest

from paper_2103_00571_gb300 import build

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "su3_internal.h"
int main(int, char** v) {
  su3::LaunchCfg c{atoi(v[1]), atoi(v[2]), 3, 4, 0, atoi(v[3])};
  c.is_default = atoi(v[4]);
  long long ts = c.tile_sites;
  su3::spread_small(&c, &ts, atoll(v[5]), 152, atoll(v[6]), atoi(v[7]), true);
  printf("%lld %d %d\n", ts, c.block, c.threads_per_link);
}
"""


@pytest.fixture(scope="module")
def shape(tmp_path_factory):
    d = tmp_path_factory.mktemp("shape")
    (d / "shape.cpp").write_text(SRC)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-I", build.CSRC, "-I", build.INCLUDE, "-I", cuda, str(d / "shape.cpp"), "-o",
                    str(d / "shape")], check=True)

    def run(block, tile, tpl, default, sites, quantum=1, rows=3):
        out = subprocess.run([str(d / "shape")] + [str(int(x)) for x in (block, tile, tpl, default, sites, quantum, rows)],
                             check=True, capture_output=True, text=True).stdout
        return tuple(int(x) for x in out.split())
    return run


@pytest.mark.parametrize("tpl", [1, 3])
@pytest.mark.parametrize("block", [32, 64, 128, 256])
@pytest.mark.parametrize("sites", [1, 64, 152, 1000, 3333, 4863, 4864, 10 ** 6])
def test_a_set_shape_is_kept(shape, tpl, block, sites):
    ts, b, t = shape(block, 32, tpl, False, sites)
    assert t == tpl and b <= block and 1 <= ts <= 32
    assert (sites + ts - 1) // ts <= max(152, (sites + 31) // 32)
    if sites >= 152 * 32:
        assert (ts, b) == (32, block)


def test_the_default_splits_rows_that_fit_a_cta(shape):
    assert shape(128, 32, 1, True, 64) == (1, 32, 3)
    assert shape(128, 32, 1, True, 152 * 21) == (21, 256, 3)  # 252 rows
    assert shape(128, 32, 1, True, 152 * 21 + 1) == (22, 96, 1)
    assert shape(128, 48, 3, True, 152 * 32, 1, 2) == (32, 256, 3)
    assert shape(128, 32, 1, True, 152 * 32) == (32, 128, 1)
    assert shape(256, 64, 1, True, 100, 8) == (8, 96, 3)  # whole blocks of 32 links
