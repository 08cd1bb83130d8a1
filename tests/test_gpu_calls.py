"""How calls stand among other work: the first ones of a process, on streams of their own."""
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
