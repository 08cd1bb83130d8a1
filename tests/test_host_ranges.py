"""Index arithmetic of the kernels that host code can run too: compiled from the library's own headers, run without a GPU."""
import ctypes as C
import os
import subprocess

import pytest

from paper_1908_06077_b200 import build as cuda_build

SOURCE = """
#include "nuq_encode_common.cuh"
extern "C" void bucket_of_lane(uint32_t lane, uint32_t spb, uint32_t* out) {
    const nuq::SubBlocks b = nuq::bucket_of_lane(lane, spb);
    out[0] = b.from;
    out[1] = b.to;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    folder = tmp_path_factory.mktemp("ranges")
    (folder / "ranges.cu").write_text(SOURCE)
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")] + cuda_build.NVCC_FLAGS + ["-I", cuda_build.CSRC, "-shared", "-o", str(folder / "ranges.so"),
                    str(folder / "ranges.cu")], check=True)
    return C.CDLL(str(folder / "ranges.so"))


@pytest.mark.parametrize("subs", [32, 8])
def test_norms_are_summed_over_the_tile_s_own_sub_blocks(lib, subs):
    """Every sub-block of a tile, which is of whole buckets or the vector's end, gets the sum of its own bucket's, and finds it within
    the tile's sums; lanes behind the tile's last sub-block may not ask."""
    out = (C.c_uint32 * 2)()
    beyond = 0
    for spb in range(1, subs + 1):
        for lane in range(32):
            lib.bucket_of_lane(lane, spb, out)
            assert tuple(out) == (lane // spb * spb, lane // spb * spb + spb)
            if lane < subs // spb * spb:
                assert out[1] <= subs, (spb, lane)
            else:
                beyond += out[1] > subs
    assert beyond > 0
