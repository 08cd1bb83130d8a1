"""Edges of the kernels' ranges, against the oracle: streams from 1 to 64 and the units that follow from them, empty and
full sub-blocks, gaps and tokens too long for the decoder's table, chains longer than a lane's copy of them, fields of every
width, norms whose products are not exact, and the encoders' sizes at which another variant takes over."""
import numpy as np
import pytest

import oracle as O
from gpu_util import gpu_decode, gpu_encode, require_cuda

pytestmark = pytest.mark.gpu


def _vector(kind, d, seed):
    rng = np.random.default_rng(seed)
    g = rng.standard_normal(d).astype(np.float32)
    if kind == "sparse":                        # gaps of 128 and more
        g[rng.random(d) > 0.004] = 0.0
    elif kind == "ends":                        # a sub-block's last element alone: gap 256
        keep = np.arange(d) % 256 == 255
        g[~keep] = 0.0
    elif kind == "dense":                       # nearly all symbols high, all tokens long
        g = (np.sign(g) * rng.uniform(0.5, 1.0, d)).astype(np.float32)
    elif kind == "mixed":                       # empty, sparse and dense sub-blocks side by side
        g *= np.repeat(np.float32([0.0, 1e-3, 0.05, 1.0]), 256)[np.arange(d) % 1024]
    elif kind == "tiny":                        # norm times level is not a normal number
        g *= np.float32(1e-38)
    return g


def _container(kind, d, bucket, s, nk, ls, mode, seed):
    return O.encode(_vector(kind, d, seed), bucket, s, O.make_flags(nk, ls, mode), seed=seed, offset=seed)[0]


def _same_sums(streams, d, bucket, s):
    rc, want = O.decode_accumulate(streams, d, bucket, s)
    assert rc == 0
    assert np.array_equal(gpu_decode(streams, d, bucket, s).view(np.uint32), want.view(np.uint32))


@pytest.mark.parametrize("K", [1, 2, 3, 5, 6, 7, 12, 16, 31, 32, 33, 64])
@pytest.mark.parametrize("mode", [O.MODE_ERC, O.MODE_FIXED])
def test_sums_for_every_shape_of_a_unit(K, mode):
    kinds = ["normal", "sparse", "mixed", "dense", "ends"]
    for d, bucket in ((200, 256), (70003, 1024)):
        _same_sums([_container(kinds[k % 5], d, bucket, 4, O.NORM_L2, O.LEVELS_EXP, mode, k) for k in range(K)], d, bucket, 4)


@pytest.mark.parametrize("kind", ["normal", "sparse", "ends", "dense", "mixed", "tiny"])
@pytest.mark.parametrize("d,bucket,s,nk,ls", [
    (30001, 512, 2, O.NORM_LINF, O.LEVELS_EXP), (30001, 8192, 6, O.NORM_LINF, O.LEVELS_EXP),
    (30001, 1024, 14, O.NORM_LINF, O.LEVELS_EXP), (30001, 768, 5, O.NORM_L2, O.LEVELS_UNIFORM),
    (30001, 8192, 6, O.NORM_LINF, O.LEVELS_UNIFORM), (30001, 512, 7, O.NORM_LINF, O.LEVELS_UNIFORM),
    (30001, 1024, 8, O.NORM_LINF, O.LEVELS_UNIFORM), (30001, 1024, 8, O.NORM_LINF, O.LEVELS_EXP)])
def test_sums_of_long_tokens_and_chains(kind, d, bucket, s, nk, ls):
    for mode in (O.MODE_ERC, O.MODE_FIXED):
        _same_sums([_container(kind, d, bucket, s, nk, ls, mode, k) for k in range(3)], d, bucket, s)


@pytest.mark.parametrize("ls,s", [(O.LEVELS_EXP, s) for s in (1, 2, 3, 6, 7, 14)] + [(O.LEVELS_UNIFORM, s) for s in range(1, 9)])
@pytest.mark.parametrize("bucket", [256, 768, 2048])
def test_fields_of_every_width(ls, s, bucket):
    for d in (256, 1023, 8 * bucket + 5, 148 * 16 * 256 + 77):      # the last: more than one sub-block for every warp
        K = 2 if d > 100000 else 9
        _same_sums([_container("normal", d, bucket, s, O.NORM_LINF, ls, O.MODE_FIXED, k) for k in range(K)], d, bucket, s)


def test_sums_of_streams_with_different_codes_and_level_sets():
    d, bucket, s = 20001, 1024, 4
    streams = []
    for k, weights in enumerate(([9, 5, 3, 2, 1], [1, 1, 1, 1, 1], [1, 2, 4, 8, 16])):
        O.set_level_code(O.huffman_lengths(weights))
        streams.append(_container("dense" if k else "sparse", d, bucket, s, O.NORM_LINF, O.LEVELS_EXP, O.MODE_CODED, k))
    _same_sums(streams[1:2] * 3, d, bucket, s)
    _same_sums(streams, d, bucket, s)
    for ls, mode in ((O.LEVELS_EXP, O.MODE_ERC), (O.LEVELS_UNIFORM, O.MODE_ERC), (O.LEVELS_UNIFORM, O.MODE_FIXED)):
        streams.append(_container("mixed", d, bucket, s, O.NORM_LINF, ls, mode, 7))
    _same_sums(streams, d, bucket, s)
    O.set_levels(np.array([0.1, 0.2, 0.5, 0.8], np.float32))
    tables = [_container(kind, d, bucket, s, O.NORM_LINF, O.LEVELS_TABLE, O.MODE_ERC, 8) for kind in ("dense", "tiny")]
    _same_sums(tables, d, bucket, s)
    _same_sums(streams + tables, d, bucket, s)


@pytest.mark.parametrize("kind", ["normal", "sparse", "dense", "mixed", "ends"])
@pytest.mark.parametrize("weights", [[9, 5, 3, 2, 1], [1, 1, 1, 1, 1], [1, 2, 4, 8, 16, 32, 64]])
def test_sums_of_coded_streams_where_warps_have_several_units(kind, weights):
    """A level code's table holds pairs of tokens there (32 streams: a unit is one sub-block)."""
    d, bucket, s = 2500 * 256 + 77, 1024, len(weights) - 1
    O.set_level_code(O.huffman_lengths(weights))
    streams = [_container(kind, d, bucket, s, O.NORM_L2, O.LEVELS_EXP, O.MODE_CODED, k) for k in range(2)]
    _same_sums(streams * 16, d, bucket, s)


@pytest.mark.parametrize("bucket,mode", [(256, O.MODE_ERC), (768, O.MODE_ERC), (1024, O.MODE_ERC), (1024, O.MODE_FIXED), (1280, O.MODE_ERC)])
def test_sums_of_short_blocks_where_warps_have_more_than_two_units(bucket, mode):
    """Buckets of up to 1024 elements have a kernel of their own there; fixed-width streams of unknown origin are a call in it."""
    d, s = 4800 * 256 + 77, 4
    streams = [_container(kind, d, bucket, s, O.NORM_L2, O.LEVELS_EXP, mode, 3) for kind in ("mixed", "normal")]
    _same_sums(streams * 16, d, bucket, s)


@pytest.mark.parametrize("ls,s,less", [(O.LEVELS_EXP, 6, 3), (O.LEVELS_EXP, 5, 4), (O.LEVELS_UNIFORM, 4, 2), (O.LEVELS_UNIFORM, 4, 3)])
def test_symbols_beyond_the_last_level_are_refused(ls, s, less):
    """Containers whose header claims fewer levels than they use: many such symbols follow a good one within a table's prefix."""
    d, bucket = 20001, 1024
    c = _container("normal", d, bucket, s, O.NORM_LINF, ls, O.MODE_ERC, 4)
    c[5] = less
    assert O.decode_accumulate([c], d, bucket, less)[0] != 0
    gpu_decode([c], d, bucket, less, expect_status=-3)


def test_missing_symbols_and_values_that_are_not_finite_in_fixed_width_streams():
    require_cuda()
    d, bucket, s = 5000, 1024, 3                                    # 5 levels in 3 bits: 5, 6 and 7 do not exist
    good = _container("normal", d, bucket, s, O.NORM_LINF, O.LEVELS_EXP, O.MODE_FIXED, 1)
    bad = good.copy()
    bad[16 + 1 + 3] |= np.uint32(0x70000000)
    gpu_decode([good, bad], d, bucket, s, expect_status=-3)
    for norm in (np.inf, np.float32(3e38)):                         # infinite, or a sum that overflows: no error
        big = good.copy()
        big[16] = np.float32(norm).view(np.uint32)
        rc, want = O.decode_accumulate([big] * 3, d, bucket, s)
        got = gpu_decode([big] * 3, d, bucket, s)
        assert rc == 0 and np.array_equal(got, want, equal_nan=True)


@pytest.mark.parametrize("kind", ["normal", "sparse", "dense", "mixed"])
@pytest.mark.parametrize("d,bucket,s,ls", [
    (1, 256, 4, O.LEVELS_EXP), (8191, 8192, 4, O.LEVELS_EXP), (40000, 512, 6, O.LEVELS_EXP), (40000, 768, 5, O.LEVELS_UNIFORM),
    (65536, 65536, 4, O.LEVELS_EXP), (3 * 16384 + 9000, 16384, 4, O.LEVELS_EXP),      # one cluster, several
    (2 * 148 * 8192, 8192, 4, O.LEVELS_EXP), (2 * 148 * 8192 + 1, 8192, 4, O.LEVELS_EXP),       # two tiles per SM, one more
    (3 * 148 * 8192, 8192, 4, O.LEVELS_EXP), (3 * 148 * 8192 + 1, 8192, 4, O.LEVELS_EXP)])      # three tiles per SM, one more
def test_containers_at_the_encoders_edges(kind, d, bucket, s, ls):
    g = _vector(kind, d, 3)
    for mode in (O.MODE_ERC, O.MODE_FIXED) + ((O.MODE_CODED,) if ls == O.LEVELS_EXP else ()):
        if mode == O.MODE_CODED:
            lengths = list(O.huffman_lengths(list(range(1, s + 2))))  # high levels get the short words
            O.set_level_code(lengths)
            require_cuda()[1].set_level_code(lengths)
        flags = O.make_flags(O.NORM_LINF, ls, mode)
        norms = O.bucket_norms(g, bucket, O.NORM_LINF)
        want, want_bits = O.encode(g, bucket, s, flags, seed=5, offset=9, norms=norms)
        got, got_bits = gpu_encode(g, bucket, s, flags, seed=5, offset=9, norms=norms)
        assert got_bits == want_bits and np.array_equal(got, want)
        free, free_bits = gpu_encode(g, bucket, s, flags, seed=5, offset=9)       # (largest magnitudes are exact: the same norms)
        assert free_bits == want_bits and np.array_equal(free, want)


@pytest.mark.parametrize("kind", ["normal", "mixed"])
@pytest.mark.parametrize("tiles,bucket", [(1, 256), (1, 768), (1, 2048), (1, 2304), (3, 512), (3, 8192), (3, 16384)])
def test_containers_where_small_tiles_and_more_warps_end(kind, tiles, bucket):
    """One tile of 8192 elements (whole buckets of it) per SM and one more, three and one more."""
    torch, _ = require_cuda()
    tile = 8192 if bucket > 8192 else 8192 // bucket * bucket
    last = tiles * torch.cuda.get_device_properties(0).multi_processor_count * tile
    for d in (last, last + 1):
        g = _vector(kind, d, 3)
        norms = O.bucket_norms(g, bucket, O.NORM_L2)
        want, want_bits = O.encode(g, bucket, 4, 0, seed=5, offset=9, norms=norms)
        got, got_bits = gpu_encode(g, bucket, 4, 0, seed=5, offset=9, norms=norms)
        assert got_bits == want_bits and np.array_equal(got, want)
        free, _ = gpu_encode(g, bucket, 4, 0, seed=5, offset=9)
        _, _, _, taken = O.decode_symbols(free, d, bucket, 4)
        assert np.array_equal(free, O.encode(g, bucket, 4, 0, seed=5, offset=9, norms=taken)[0])


@pytest.mark.parametrize("ls,s,mode,nk", [(O.LEVELS_EXP, 4, O.MODE_ERC, O.NORM_L2), (O.LEVELS_UNIFORM, 4, O.MODE_ERC, O.NORM_LINF), (O.LEVELS_UNIFORM, 2, O.MODE_ERC, O.NORM_L2),
                                          (O.LEVELS_TABLE, 4, O.MODE_ERC, O.NORM_LINF), (O.LEVELS_EXP, 4, O.MODE_CODED, O.NORM_LINF)])
@pytest.mark.parametrize("bucket", [256, 768, 1024, 1280, 8192])
def test_containers_of_every_kind_at_the_limits_of_small_calls(bucket, ls, s, mode, nk):
    """Small tiles end where every SM has a whole one, or 5.5 small ones; twice the warps at 17/7 tiles per SM or at three."""
    torch, nuq = require_cuda()
    sms, tile, small = torch.cuda.get_device_properties(0).multi_processor_count, 8192 // bucket * bucket, 2048 // bucket * bucket
    limits = [(sms - 1) * tile, 17 * sms // 7 * tile, 3 * sms * tile] + ([11 * sms // 2 * small] if small else [])
    if ls == O.LEVELS_TABLE:
        levels = np.float32([0.6 ** (s + 1 - j) for j in range(1, s + 1)])
        O.set_levels(levels)
        nuq.set_level_table(levels)
    if mode == O.MODE_CODED:
        lengths = list(O.huffman_lengths([9, 5, 3, 2, 1]))
        O.set_level_code(lengths)
        nuq.set_level_code(lengths)
    flags = O.make_flags(nk, ls, mode)
    for d in [n + more for n in limits for more in (0, 1)] + [70001]:
        g = _vector("normal", d, 3)
        free, bits = gpu_encode(g, bucket, s, flags, seed=5, offset=9)
        norms = O.decode_symbols(free, d, bucket, s)[3]
        if nk == O.NORM_LINF:                               # (exact)
            assert np.array_equal(norms, O.bucket_norms(g, bucket, nk))
        want, want_bits = O.encode(g, bucket, s, flags, seed=5, offset=9, norms=norms)
        assert bits == want_bits and np.array_equal(free, want), d


@pytest.mark.parametrize("mode", [O.MODE_ERC, O.MODE_FIXED])
@pytest.mark.parametrize("ls,s,K", [(O.LEVELS_UNIFORM, 4, 3), (O.LEVELS_UNIFORM, 8, 3), (O.LEVELS_TABLE, 5, 3), (O.LEVELS_TABLE, 8, 2), (O.LEVELS_TABLE, 3, 40)])
def test_products_are_rounded_before_they_are_added(ls, s, K, mode):
    """norm times level is a product of its own (one rounding), the sum another: where the product is not exact, an operation
    that rounds once for both gives other last bits.  (The packed multiply and add of two elements were once joined so.)"""
    d, bucket = 60001, 1024
    O.set_levels(np.float32([0.61 ** (s + 1 - j) for j in range(1, s + 1)]))
    streams = [_container("normal", d, bucket, s, O.NORM_LINF, ls, mode, k) for k in range(K)]
    joined = np.zeros(d, np.float32)
    for st in streams:
        rc, sign, sym, norms = O.decode_symbols(st, d, bucket, s)
        level = np.float32([O.level_value(ls, s, j) for j in range(O.num_levels(ls, s))])[sym].astype(np.float64)
        product = np.where(sign != 0, -1.0, 1.0) * level * np.repeat(norms, bucket)[:d].astype(np.float64)      # exact: 48 bits
        joined = (joined.astype(np.float64) + product).astype(np.float32)
    rc, want = O.decode_accumulate(streams, d, bucket, s)
    assert rc == 0 and np.mean(joined != want) > 0.02               # the input tells the two apart
    _same_sums(streams, d, bucket, s)


@pytest.mark.parametrize("bucket", [256, 512, 768, 1024, 8192])
@pytest.mark.parametrize("s", [3, 4, 6])
def test_four_bit_containers_of_dense_and_sparse_symbols(bucket, s):
    """The 4-bit encoder's ways to quantize: by instance (buckets) and, in buckets of 1024 and more, by what a warp's first
    sub-block looks like; kinds change from sub-block to sub-block here, and the last tile ends inside a warp's part."""
    d = 3 * 8192 + 1500
    for kind in ("normal", "sparse", "dense", "mixed", "ends"):
        for nk in (O.NORM_L2, O.NORM_LINF):
            g = _vector(kind, d, s)
            g[5000:9000] *= np.float32(40.0)
            norms = O.bucket_norms(g, bucket, nk)
            flags = O.make_flags(nk, O.LEVELS_EXP, O.MODE_FIXED)
            want, want_bits = O.encode(g, bucket, s, flags, seed=5, offset=9, norms=norms)
            got, got_bits = gpu_encode(g, bucket, s, flags, seed=5, offset=9, norms=norms)
            assert got_bits == want_bits and np.array_equal(got, want), (kind, nk)
