"""The row kernel's work split (row_split in pair2.cuh, from its source on the CPU): the units cover
every pair of a block and a j-tile, each slot of the partials lies within what a context allocates for its
whole number of blocks, also when it is sharded to fewer, and the tiles hold whole Kahan groups."""
import ctypes
import re

import pytest

import device_source as ds

CTAS = [1, 100, 152 * 8, 1520, 2048, 152 * 8 * 32]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    src = open(ds.CSRC + "/pair2.cuh").read()
    body = src[src.index("struct RowSplit {"):src.index("template <bool KAHAN, bool LINE>\n__global__ void __launch_bounds__(kPairThreads, STEPS_ROW")]
    places = re.search(r"#define STEPS_ROW_MIN_BLOCKS (\d+)", src).group(0)
    lib = ds.compile_host(tmp_path_factory.mktemp("rows"), places, "constexpr int kBJ = 128;", body, """
extern "C" void split(int blocks, int n, int ctas, long long* out) {
  const RowSplit r = row_split(blocks, n, ctas);
  out[0] = r.U; out[1] = r.NT; out[2] = r.jt; out[3] = r.C;
}
extern "C" int ctas(int blocks, int n, int c) { return row_ctas(blocks, n, c); }
""")
    return lib


@pytest.mark.parametrize("n", [2, 31, 33, 129, 500, 1000, 2000, 4863, 4864, 4865, 5000, 10007, 65536])
@pytest.mark.parametrize("ctas", CTAS)
def test_split(lib, n, ctas):
    NB = (n + 127) // 128
    out = (ctypes.c_longlong * 4)()
    slots = NB + lib.ctas(NB, n, ctas)
    for blocks in range(1, NB + 1):
        lib.split(blocks, n, ctas, out)
        U, NT, jt, C = out
        assert jt in (32, 64, 128) and NT == (n + jt - 1) // jt and U == blocks * NT
        assert 1 <= C <= min(U, ctas)
        assert blocks - 1 + C - 1 < slots  # the last slot: the last block's, of the last CTA
