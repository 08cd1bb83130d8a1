"""What the library's host code asks of the CUDA runtime, and in which order: the library's own objects linked with a runtime
that runs nothing (fake_cudart.cpp).  No GPU is needed."""
import ctypes as C
import os
import re
import shutil
import subprocess

import pytest

from paper_1908_06077_b200 import build as cuda_build

HERE = os.path.dirname(os.path.abspath(__file__))
STREAM = 0x10                                               # a stream of the caller's own; the fake never looks at it
ERC, FIXED = 0, 1 << 16


@pytest.fixture(scope="module")
def built(tmp_path_factory):
    if not all(os.path.exists(o) for o in cuda_build.OBJECTS):
        cuda_build.build(force=True)
    path = str(tmp_path_factory.mktemp("host") / "libnuq_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I/usr/local/cuda/include", "-Wl,-Bsymbolic", "-o", path,
                    os.path.join(HERE, "fake_cudart.cpp")] + cuda_build.OBJECTS, check=True)
    return path


@pytest.fixture()
def lib(built, tmp_path):
    lib = C.CDLL(shutil.copy(built, tmp_path))              # another file, so another instance of the library, for every test
    lib.nuq_encode.argtypes = [C.c_void_p, C.c_uint64, C.c_uint32, C.c_uint32, C.c_uint32, C.c_uint64, C.c_uint64, C.c_void_p, C.c_void_p, C.c_void_p]
    lib.nuq_encode_static.argtypes = lib.nuq_encode.argtypes
    lib.nuq_decode_accumulate.argtypes = [C.POINTER(C.c_void_p), C.c_uint32, C.c_uint64, C.c_uint32, C.c_uint32, C.c_void_p, C.c_void_p]
    lib.nuq_level_histogram.argtypes = [C.c_void_p, C.c_uint64, C.c_uint32, C.c_uint32, C.c_uint32, C.c_uint64, C.c_uint64, C.c_void_p, C.c_void_p]
    lib.nuq_last_status.argtypes = [C.c_void_p]
    lib.fake_events.restype = C.c_char_p
    lib.fake_last_alloc.restype = C.c_void_p
    return lib


def _encode(lib, d=100000, bucket=1024, s=4, kind=ERC, stream=STREAM):
    return lib.nuq_encode(0x1000, d, bucket, s, kind, 1, 0, 0x2000, None, stream)


def _decode(lib, d=100000, bucket=1024, s=4, stream=STREAM):
    return lib.nuq_decode_accumulate((C.c_void_p * 1)(0x2000), 1, d, bucket, s, 0x3000, stream)


def _launches(lib):
    return [e for e in lib.fake_events().decode().splitlines() if e.startswith("launch")]


@pytest.mark.parametrize("call", [_encode, _decode])
def test_the_first_call_waits_for_the_tables_it_uploads(lib, call):
    """the upload runs on the default stream, which a non-blocking stream's kernels do not wait for"""
    assert call(lib) == 0 and call(lib) == 0
    assert len(_launches(lib)) == 2 and all(e.endswith("unordered 0") for e in _launches(lib))


def test_a_status_is_cleared_in_its_own_stream(lib):
    """a clearing pass on the default stream could wipe out what the next kernel of a non-blocking stream latches"""
    assert _decode(lib) == 0
    status = C.cast(lib.fake_last_alloc(), C.POINTER(C.c_int))      # the workspace begins with it
    status[0] = -3
    assert lib.nuq_last_status(STREAM) == -3 and lib.nuq_last_status(STREAM) == 0
    assert _decode(lib) == 0
    assert all(e.endswith("unordered 0") for e in _launches(lib))


@pytest.mark.parametrize("own,static,want", [(0, 1, 1), (1, 0, 1), (1, 1, 1), (-3, 1, -3), (1, -5, -5), (-3, -5, -5), (0, 0, 0)])
def test_the_static_array_s_status_is_joined_with_the_stream_s(lib, own, static, want):
    """the most negative one wins, a warning shows where there is no error"""
    assert _decode(lib) == 0
    C.cast(lib.fake_last_alloc(), C.POINTER(C.c_int))[0] = own
    assert lib.nuq_encode_static(0x1000, 100000, 1024, 4, ERC, 1, 0, 0x2000, None, STREAM) == 0
    C.cast(lib.fake_last_alloc(), C.POINTER(C.c_int))[0] = static
    assert lib.nuq_last_status(STREAM) == want and lib.nuq_last_status(STREAM) == 0


@pytest.mark.parametrize("call", [_encode, _decode])
def test_a_first_call_is_refused_inside_a_capture_and_works_behind_it(lib, call):
    """tables and workspace come from calls that a capture does not allow; later calls ask for neither"""
    lib.fake_capture(1)
    assert call(lib) == -4 and not _launches(lib)
    lib.fake_capture(0)
    assert call(lib) == 0
    lib.fake_reset()
    lib.fake_capture(1)
    assert call(lib) == 0 and "refused" not in lib.fake_events().decode()


def test_norms_never_lie_where_an_encode_call_keeps_its_scan_state(lib):
    """a replay of a captured call would leave them there, and the host would not know that the next call has to clear"""
    hist = (C.c_uint64 * 8)()
    assert _encode(lib, d=1 << 20, bucket=65536, kind=FIXED) == 0                       # wide buckets with 4-bit fields
    assert lib.nuq_level_histogram(0x1000, 1 << 20, 256, 4, 0, 1, 0, C.addressof(hist), STREAM) == 0
    assert _encode(lib, d=1 << 20, bucket=65536, kind=FIXED) == 0
    where = [e for e in lib.fake_events().decode().splitlines() if e.startswith("norms")]
    assert len(where) == 3 and not any("allocation 0" in e for e in where)              # (0 is the workspace)


@pytest.mark.parametrize("kind", [ERC, FIXED, 2 << 16, 1 << 8])
@pytest.mark.parametrize("bucket", [512, 65536])
def test_every_device_is_told_how_much_shared_memory_the_kernels_take(lib, kind, bucket):
    """the runtime keeps that per device"""
    lengths = (C.c_uint8 * 6)(1, 2, 3, 4, 5, 5)
    assert lib.nuq_set_level_code(lengths, 5) == 0
    for device in (0, 1, 0, 2):
        lib.cudaSetDevice(device)
        for d in (100000, 10000000):
            assert _encode(lib, d=d, bucket=bucket, s=5, kind=kind) == 0 and _decode(lib, d=d, bucket=bucket, s=5) == 0
            assert _decode(lib, d=d, bucket=bucket, s=7) == 0                           # (16-bit symbols)


@pytest.mark.parametrize("kinds", [(ERC,), (FIXED,), (2 << 16,), (ERC, FIXED, 2 << 16)])
@pytest.mark.parametrize("d", [1212417, 2000000, 5000000, 10000000])
def test_a_call_with_fewer_elements_than_the_one_before_never_allocates(lib, d, kinds):
    """whatever its buckets, mode and tiles are: it may be captured, and a graph may hold the workspace's address"""
    assert lib.nuq_set_level_code((C.c_uint8 * 5)(1, 2, 3, 4, 4), 4) == 0
    assert _encode(lib, d=d, bucket=8192) == 0
    lib.fake_capture(1)
    for kind in kinds:
        for bucket in (256, 768, 1024, 1280, 2048, 4352, 8192, 16384):
            if kind == FIXED and bucket > 8192:
                continue                                    # (norms of their own)
            for n in (65536, 148 * 2048, 4 * 148 * 1024, 1200000, 148 * 8192, d):
                assert n > d or _encode(lib, d=n, bucket=bucket, s=4, kind=kind) == 0, (n, bucket)
    assert "refused" not in lib.fake_events().decode()


def test_a_pass_for_norms_over_fewer_elements_than_the_one_before_never_allocates(lib):
    hist = (C.c_uint64 * 8)()
    assert _encode(lib, d=2000000, bucket=65536, kind=FIXED) == 0
    lib.fake_capture(1)
    for bucket in (65536, 32768, 16384):
        assert _encode(lib, d=2000000, bucket=bucket, kind=FIXED) == 0
    for bucket in (256, 1024, 8192, 65536):
        assert lib.nuq_level_histogram(0x1000, 2000000, bucket, 4, 0, 1, 0, C.addressof(hist), STREAM) == 0
    assert "refused" not in lib.fake_events().decode()


def _tile_and_warps(lib, d, bucket, s=4, kind=ERC):
    """elements of a tile and worker warps of the encode kernel that a call launches"""
    lib.fake_reset()
    assert _encode(lib, d=d, bucket=bucket, s=s, kind=kind) == 0
    (name,) = re.findall(r"encode_kernelILj\d+ELj\d+ELb\dELj(\d+)ELj(\d+)E", lib.fake_events().decode())
    return int(name[1]), int(name[0])


SMS = 148                                                   # (of the stand-in)


@pytest.mark.parametrize("bucket,last", [(256, (SMS - 1) * 8192), (768, (SMS - 1) * 7680), (1280, 11 * SMS // 2 * 1280), (1536, (SMS - 1) * 7680), (2048, (SMS - 1) * 8192)])
def test_small_tiles_end_where_sms_would_get_six_or_each_has_a_whole_one(lib, bucket, last):
    assert _tile_and_warps(lib, 256, bucket) == (2048, 8)
    assert _tile_and_warps(lib, last, bucket) == (2048, 8)
    assert _tile_and_warps(lib, last + 1, bucket) == (8192, 16)
    assert _tile_and_warps(lib, SMS * (8192 // bucket * bucket), bucket) == (8192, 16)


@pytest.mark.parametrize("bucket,s,kind,sevenths", [(512, 4, ERC, 17), (8192, 4, ERC, 17), (8192, 2, 1 << 8, 17), (8192, 4, 1 << 8 | 1, 21), (512, 6, 1 << 8, 21),
                                                    (16384, 4, ERC, 14), (32768, 4, ERC, 21), (65536, 4, 1 << 8 | 1, 21)])
def test_sixteen_warps_end_where_an_sm_would_get_four_tiles(lib, bucket, s, kind, sevenths):
    last = sevenths * SMS // 7 * 8192
    assert _tile_and_warps(lib, last, bucket, s, kind) == (8192, 16)
    assert _tile_and_warps(lib, last + 1, bucket, s, kind) == (8192, 8)
