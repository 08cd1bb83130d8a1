"""How calls stand among other work: the first ones of a process, on streams of their own; whole steps captured into graphs."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle as O
from gpu_util import require_cuda

pytestmark = pytest.mark.gpu


FIRST_CALLS = """
import sys
sys.path.insert(0, {root!r})
import numpy as np, torch
import oracle as O
from paper_1908_06077_b200 import nuq
d, bucket, s = 300001, 1024, 4
g = np.random.default_rng(1).standard_normal(d).astype(np.float32)
norms = O.bucket_norms(g, bucket, O.NORM_LINF)
flags = O.make_flags(O.NORM_LINF, O.LEVELS_EXP, O.MODE_ERC)
want, _ = O.encode(g, bucket, s, flags, seed=3, offset=0, norms=norms)
rc, sums = O.decode_accumulate([want], d, bucket, s)
dev = torch.from_numpy(want.view(np.int32)).cuda()
gd = torch.from_numpy(g).cuda()
out = torch.zeros(nuq.encode_bound(d, bucket, s, flags) // 4, dtype=torch.int32, device="cuda")
bits = torch.zeros(1, dtype=torch.int64, device="cuda")
acc = torch.zeros(d, device="cuda")
torch.cuda.synchronize()
side = torch.cuda.Stream()                  # (a non-blocking stream)
with torch.cuda.stream(side):
    if {decode_first}:
        nuq.decode_accumulate([dev], d, bucket, s, acc=acc)
        nuq.encode(gd, bucket, s, flags, seed=3, out=out, out_bits=bits)
    else:
        nuq.encode(gd, bucket, s, flags, seed=3, out=out, out_bits=bits)
        nuq.decode_accumulate([dev], d, bucket, s, acc=acc)
    assert nuq.last_status() == 0
assert np.array_equal(acc.cpu().numpy().view(np.uint32), sums.view(np.uint32))
assert np.array_equal(out.cpu().numpy().view(np.uint32)[: int(bits.item()) // 32], want)
"""


@pytest.mark.parametrize("decode_first", [True, False])
def test_first_calls_of_a_process_on_a_stream_of_its_own(decode_first):
    require_cuda()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    done = subprocess.run([sys.executable, "-c", FIRST_CALLS.format(root=root, decode_first=decode_first)], capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr[-2000:]


@pytest.mark.parametrize("mode", [O.MODE_ERC, O.MODE_FIXED, O.MODE_CODED])
@pytest.mark.parametrize("update", [False, True])
def test_a_step_replayed_from_a_cuda_graph(mode, update):
    """The encode calls of three workers and the decode behind them, captured once and replayed on changing gradients: every
    replay gives what the same calls give outside the graph.  A level code that is set later does not reach the graph."""
    torch, nuq = require_cuda()
    K, d, bucket, s = 3, 400001, 1024, 4
    flags = O.make_flags(O.NORM_L2, O.LEVELS_EXP, mode)
    code = [1, 2, 3, 4, 4]
    nuq.set_level_code(code)
    gen = torch.Generator(device="cuda").manual_seed(5)
    src = [torch.randn(d, generator=gen, device="cuda") for _ in range(5)]
    words = nuq.encode_bound(d, bucket, s, flags) // 4

    class Step:
        def __init__(self):
            self.gs = [torch.zeros(d, device="cuda") for _ in range(K)]
            self.outs = [torch.zeros(words, dtype=torch.int32, device="cuda") for _ in range(K)]
            self.bits = [torch.zeros(1, dtype=torch.int64, device="cuda") for _ in range(K)]
            self.acc, self.w, self.yl = torch.zeros(d, device="cuda"), torch.ones(d, device="cuda"), torch.ones(d, device="cuda")

        def enqueue(self, stream):
            for k in range(K):
                nuq.encode(self.gs[k], bucket, s, flags, seed=k + 1, out=self.outs[k], out_bits=self.bits[k], stream=stream)
            if update:
                nuq.decode_update(self.outs, d, bucket, s, self.w, self.yl, 0.1, 0.9, 1.0, acc=self.acc, stream=stream)
            else:
                nuq.decode_accumulate(self.outs, d, bucket, s, acc=self.acc, stream=stream)

    side, captured, plain = torch.cuda.Stream(), Step(), Step()
    with torch.cuda.stream(side):                            # first use of the stream: workspace and tables
        captured.enqueue(side)
    torch.cuda.synchronize()
    captured.w.fill_(1.0)
    captured.yl.fill_(1.0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        captured.enqueue(side)
    for rnd in range(3):
        for st in (captured, plain):
            for k in range(K):
                st.gs[k].copy_(src[(k + rnd) % 5])
        nuq.set_level_code([4, 4, 3, 2, 1])
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert nuq.last_status(side) == 0
        nuq.set_level_code(code)
        plain.enqueue(None)
        torch.cuda.synchronize()
        assert nuq.last_status() == 0
        for name in ("acc", "w", "yl"):
            assert torch.equal(getattr(captured, name), getattr(plain, name)), (rnd, name)
        for a, b, n in zip(captured.outs, plain.outs, plain.bits):
            assert torch.equal(a[: int(n.item()) // 32], b[: int(n.item()) // 32])


def test_a_replay_between_calls_that_take_norms_apart():
    """A captured encode call is replayed after calls on its stream that keep bucket norms (4-bit fields in wide buckets, a
    histogram), which the graph knows nothing of: they leave its scan state alone."""
    torch, nuq = require_cuda()
    d, bucket, s = 3_000_001, 1024, 4
    g = torch.randn(d, generator=torch.Generator(device="cuda").manual_seed(6), device="cuda")
    want, bits = nuq.encode(g, bucket, s, 0, seed=2)
    n = int(bits.item()) // 32
    out, wide = torch.zeros_like(want), torch.zeros(nuq.encode_bound(d, 65536, s, nuq.MODE_FIXED) // 4, dtype=torch.int32, device="cuda")
    side, hist = torch.cuda.Stream(), torch.zeros(s + 2, dtype=torch.int64, device="cuda")
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        nuq.encode(g, bucket, s, 0, seed=2, out=out, out_bits=bits)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            nuq.encode(g, bucket, s, 0, seed=2, out=out, out_bits=bits)
        for _ in range(3):
            nuq.encode(g, 65536, s, nuq.MODE_FIXED, seed=1, out=wide)
            nuq.level_histogram(g, 256, s, hist=hist)
            out.zero_()
            graph.replay()
            assert nuq.last_status() == 0
            assert torch.equal(out[:n], want[:n])


KINDS = [(O.MODE_ERC, O.LEVELS_EXP, 4), (O.MODE_ERC, O.LEVELS_EXP, 14), (O.MODE_ERC, O.LEVELS_UNIFORM, 4), (O.MODE_ERC, O.LEVELS_UNIFORM, 8),
         (O.MODE_ERC, O.LEVELS_TABLE, 14), (O.MODE_FIXED, O.LEVELS_EXP, 4), (O.MODE_FIXED, O.LEVELS_EXP, 14), (O.MODE_FIXED, O.LEVELS_UNIFORM, 4),
         (O.MODE_FIXED, O.LEVELS_UNIFORM, 8), (O.MODE_FIXED, O.LEVELS_TABLE, 14), (O.MODE_CODED, O.LEVELS_EXP, 4)]


@pytest.mark.parametrize("was", range(len(KINDS)))
@pytest.mark.parametrize("K", [1, 3])
def test_containers_that_lie_where_others_were_encoded(was, K):
    """The library remembers what it encoded where, to choose the decoder's kernel and tables; what lies there now decides."""
    torch, nuq = require_cuda()
    d, bucket = 40001, 1024
    rng = np.random.default_rng(7)
    gs = [rng.standard_normal(d).astype(np.float32) for _ in range(K)]
    words = max(nuq.encode_bound(d, bucket, s, O.make_flags(O.NORM_L2, ls, mode)) // 4 for mode, ls, s in KINDS)
    outs = [torch.zeros(words, dtype=torch.int32, device="cuda") for _ in range(K)]
    for mode, ls, s in KINDS:
        for old, (omode, ols, os_) in enumerate([KINDS[was]] * K if K == 1 else [KINDS[was], KINDS[was], KINDS[(was + 1) % len(KINDS)]]):
            if ols == O.LEVELS_TABLE:
                nuq.set_level_table([0.7 ** (os_ + 1 - j) for j in range(1, os_ + 1)])
            if omode == O.MODE_CODED:
                nuq.set_level_code([1, 2, 3, 4, 4])
            nuq.encode(torch.from_numpy(gs[0]).cuda(), bucket, os_, O.make_flags(O.NORM_L2, ols, omode), out=outs[old])
        if ls == O.LEVELS_TABLE:
            O.set_levels(np.float32([0.6 ** (s + 1 - j) for j in range(1, s + 1)]))
        O.set_level_code([3, 3, 2, 2, 2])
        streams = [O.encode(g, bucket, s, O.make_flags(O.NORM_LINF, ls, mode), seed=k, offset=0)[0] for k, g in enumerate(gs)]
        for out, st in zip(outs, streams):
            out[: st.size].copy_(torch.from_numpy(st.view(np.int32)))
        rc, want = O.decode_accumulate(streams, d, bucket, s)
        acc = nuq.decode_accumulate(outs, d, bucket, s)
        assert rc == 0 and nuq.last_status() == 0
        assert np.array_equal(acc.cpu().numpy().view(np.uint32), want.view(np.uint32)), (mode, ls, s)


@pytest.mark.parametrize("ls,s", [(O.LEVELS_EXP, s) for s in (1, 2, 3, 6, 7, 8, 14)] + [(O.LEVELS_TABLE, s) for s in (2, 5, 8, 14)] +
                         [(O.LEVELS_UNIFORM, s) for s in range(1, 9)])
@pytest.mark.parametrize("bucket", [256, 2048])
@pytest.mark.parametrize("known", [True, False])
def test_fields_of_every_width_where_they_were_encoded_and_elsewhere(ls, s, bucket, known):
    """Sums (into an acc of either alignment) and the fused step of fixed-width streams whose kind the library knows from their
    addresses, and of those it does not know."""
    torch, nuq = require_cuda()
    if ls == O.LEVELS_TABLE:
        levels = np.float32([0.7 ** (s + 1 - j) for j in range(1, s + 1)])
        nuq.set_level_table(levels)
        O.set_levels(levels)
    flags = O.make_flags(O.NORM_LINF, ls, O.MODE_FIXED)
    gen = torch.Generator(device="cuda").manual_seed(s)
    for d, K in ((255, 2), (3 * 2048 + 11, 9), (148 * 16 * 256 + 77, 1), (4 * 148 * 16 * 256 + 4096, 2)):
        gs = [torch.randn(d, generator=gen, device="cuda") for _ in range(K)]
        outs, streams = [], []
        for k, g in enumerate(gs):
            out, bits = nuq.encode(g, bucket, s, flags, seed=k)
            n = int(bits.item()) // 32
            if not known:                                    # (nothing is ever encoded 16 bytes behind the start of a tensor here)
                out = torch.cat([out.new_zeros(4), out])[4:]
            outs.append(out)
            streams.append(out.cpu().numpy().view(np.uint32)[:n].copy())
        rc, want = O.decode_accumulate(streams, d, bucket, s)
        assert rc == 0
        want = torch.from_numpy(want).cuda()
        for shift in (0, 4):                                 # 32-byte or only 16-byte aligned
            buf = torch.full((d + 16,), float("nan"), device="cuda")
            acc = buf[shift:shift + d]
            nuq.decode_accumulate(outs, d, bucket, s, acc=acc)
            assert nuq.last_status() == 0
            assert torch.equal(acc.view(torch.int32), want.view(torch.int32)), (d, K, shift)
            assert buf[:shift].isnan().all() and buf[shift + d:].isnan().all()
        w, yl = torch.ones(d, device="cuda"), torch.ones(d, device="cuda")
        nuq.decode_update(outs, d, bucket, s, w, yl, 0.25, 0.5, 1.0, acc=acc)
        step = torch.tensor(0.25 / K, dtype=torch.float32, device="cuda").double()
        y = (1.0 - step * want.double()).float()             # one fused operation: one rounding
        assert nuq.last_status() == 0 and torch.equal(yl, y)
        assert torch.equal(w, ((y - 1.0).double() * 0.5 + y.double()).float())


@pytest.mark.parametrize("ls,s", [(O.LEVELS_EXP, s) for s in (1, 2, 3, 6, 7, 8, 14)] + [(O.LEVELS_TABLE, s) for s in (2, 5, 8, 14)] +
                         [(O.LEVELS_UNIFORM, s) for s in range(1, 9)])
def test_token_streams_where_fields_of_every_width_were_encoded(ls, s):
    """Each of the kernels for fixed-width streams hands streams of another kind on to the same function: sums and the fused step
    come out right from all of them (short blocks and long ones, one unit for a warp and several)."""
    torch, nuq = require_cuda()
    if ls == O.LEVELS_TABLE:
        levels = np.float32([0.7 ** (s + 1 - j) for j in range(1, s + 1)])
        nuq.set_level_table(levels)
        O.set_levels(levels)
    gen = torch.Generator(device="cuda").manual_seed(s)
    for d, K, bucket in ((3 * 2048 + 11, 9, 2048), (4800 * 256 + 77, 33, 512), (20 * 148 * 256 + 77, 2, 8192)):
        g = torch.randn(d, generator=gen, device="cuda")
        erc = O.encode(g.cpu().numpy(), bucket, s, O.make_flags(O.NORM_LINF, ls, O.MODE_ERC), seed=1, offset=0)[0]
        fixed = O.make_flags(O.NORM_LINF, ls, O.MODE_FIXED)
        words = max(nuq.encode_bound(d, bucket, s, fixed) // 4, erc.size)
        outs = [torch.zeros(words, dtype=torch.int32, device="cuda") for _ in range(K)]
        for out in outs:
            nuq.encode(g, bucket, s, fixed, out=out)
            out[: erc.size].copy_(torch.from_numpy(erc.view(np.int32)))
        rc, want = O.decode_accumulate([erc] * K, d, bucket, s)
        assert rc == 0
        want = torch.from_numpy(want).cuda()
        acc = torch.full((d,), float("nan"), device="cuda")
        nuq.decode_accumulate(outs, d, bucket, s, acc=acc)
        assert nuq.last_status() == 0 and torch.equal(acc.view(torch.int32), want.view(torch.int32)), (d, K)
        w, yl = torch.ones(d, device="cuda"), torch.ones(d, device="cuda")
        nuq.decode_update(outs, d, bucket, s, w, yl, 0.25, 0.5, 1.0, acc=acc)
        step = torch.tensor(0.25 / K, dtype=torch.float32, device="cuda").double()
        y = (1.0 - step * want.double()).float()             # one fused operation: one rounding
        assert nuq.last_status() == 0 and torch.equal(yl, y)
        assert torch.equal(w, ((y - 1.0).double() * 0.5 + y.double()).float())
