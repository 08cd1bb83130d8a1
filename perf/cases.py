"""The work that a user of this package has it do, as cases to be timed and compared.

A case is one direction of the path on one shape:

    encode   one worker's gradient to its container             (encode)
    decode   the containers of K workers to one summed gradient (decode_accumulate)
    step     one training step of K simulated workers: K gradients encoded, the containers
             decoded and the momentum rule applied to the parameters
             (encode K times, then decode_update; set_level_code first in the coded mode)

with its vector length `d`, bucket size `bucket`, number of levels `s`, number of workers `k`,
container `mode` (erc, fixed, coded), level set `levels` (exp, uniform, table), bucket `norm`
(l2, linf) and the distribution `values` of the gradients, which stands for

    normal    i.i.d. N(0, 1)
    outliers  tensors of a network laid end to end, N(0, sigma^2) with a sigma per tensor and
              one coordinate in a thousand at 50 sigma
    student   tensors laid end to end, Student-t(3) with a scale per tensor (tensor fusion
              mixes scales inside a bucket)
    laplace   flat Laplace(0, 1e-3) with one coordinate in a hundred exactly zero

The shapes are those of the benchmark's configurations (paper_1908_06077_b200/inputs.py) and, where a case
fills a gap between them, generic.
"""
import math

import torch

from paper_1908_06077_b200 import inputs, nuq

LEVELS = {"exp": nuq.LEVELS_EXP, "uniform": nuq.LEVELS_UNIFORM, "table": nuq.LEVELS_TABLE}
NORMS = {"l2": nuq.NORM_L2, "linf": nuq.NORM_LINF}
MODES = {"erc": nuq.MODE_ERC, "fixed": nuq.MODE_FIXED, "coded": nuq.MODE_CODED}

RESNET18, RESNET50 = inputs.RESNET18_NUMEL, inputs.RESNET50_NUMEL
ALPHA, MU, L = 1e-3, 0.9, 1.0                               # learning rate, momentum, Nesterov's method


def _case(name, do, d, bucket, s, k, mode, levels, norm, values):
    c = {"name": name} if name else {}
    c.update(do=do, d=d, bucket=bucket, s=s, k=k, mode=mode, levels=levels, norm=norm, values=values)
    return c


def listed():
    return [
        # a single small tensor, where launches and latency are all there is
        _case("tiny encode", "encode", 65536, 1024, 3, 1, "erc", "exp", "l2", "normal"),
        _case("tiny decode", "decode", 65536, 1024, 3, 1, "erc", "exp", "l2", "normal"),
        # a tensor of odd length sent with coded level indices, small buckets, three workers, a whole step
        _case("odd coded step", "step", 1_000_003, 512, 3, 3, "coded", "exp", "l2", "student"),
        # a ResNet-18 training step with four workers
        _case("resnet18 step", "step", RESNET18, 8192, 4, 4, "erc", "exp", "l2", "outliers"),
        # a ResNet-50 gradient of one of eight workers, both directions, in the two modes the method is run in
        _case("resnet50 encode", "encode", RESNET50, 8192, 4, 1, "erc", "exp", "l2", "student"),
        _case("resnet50 decode", "decode", RESNET50, 8192, 4, 8, "erc", "exp", "l2", "student"),
        _case("resnet50 encode 4-bit", "encode", RESNET50, 8192, 4, 1, "fixed", "exp", "l2", "student"),
        _case("resnet50 decode 4-bit", "decode", RESNET50, 8192, 4, 8, "fixed", "exp", "l2", "student"),
        # the same gradient under the comparison quantizer QSGDinf: dense symbols
        _case("qsgdinf encode", "encode", RESNET50, 8192, 4, 1, "erc", "uniform", "linf", "student"),
        _case("qsgdinf decode", "decode", RESNET50, 8192, 4, 8, "erc", "uniform", "linf", "student"),
        # a billion coordinates
        _case("flat encode", "encode", 1 << 30, 8192, 4, 1, "erc", "exp", "l2", "laplace"),
        _case("flat decode", "decode", 1 << 30, 512, 4, 2, "erc", "exp", "l2", "laplace"),
    ]


def draw(rng):
    do = rng.choice(["encode", "encode", "decode", "decode", "step"])
    levels = rng.choice(["exp"] * 6 + ["uniform"] * 3 + ["table"])
    mode = rng.choice(["erc", "erc", "fixed"] if levels == "uniform" else ["erc", "erc", "erc", "fixed", "fixed", "coded"])
    norm = rng.choice(["l2", "l2", "l2", "linf"])
    s = rng.randint(2, 6)
    k = 1 if do == "encode" else rng.choice([1, 2, 3, 4, 4, 6, 8, 8, 12, 16])
    bucket = 256 * rng.randint(1, 32) if rng.random() < 0.2 else 1 << rng.randint(8, 16)
    # up to the largest listed case; dense symbols and whole steps cost more per coordinate
    most = 1 << (30 if do == "encode" else 29)
    if levels != "exp" or norm != "l2" or bucket < 2048:
        most >>= 2
    if do == "step":
        most >>= 1
    d = int(round(math.exp(rng.uniform(math.log(1 << 12), math.log(most / k)))))
    values = rng.choice(["normal", "outliers", "student", "student", "laplace"])
    return _case(None, do, d, bucket, s, k, mode, levels, norm, values)


def _kind(case):
    return LEVELS[case["levels"]] | NORMS[case["norm"]] | MODES[case["mode"]]


def _tensor_scales(case, low, high, dev):
    """One scale per coordinate, constant over each tensor, log-uniform in [10^low, 10^high]; the same for all workers."""
    d = case["d"]
    if d in (RESNET18, RESNET50):
        sizes = inputs.resnet18_layer_sizes() if d == RESNET18 else inputs.resnet50_layer_sizes()
    else:                                                   # tensors of 64 to a few million coordinates
        sizes, left, i = [], d, 0
        while left:
            n = min(left, (64, 2304, 36864, 512, 262144, 1024, 2359296)[i % 7])
            sizes.append(n)
            left -= n
            i += 1
    gen = torch.Generator().manual_seed(100)
    scale = 10.0 ** (low + (high - low) * torch.rand(len(sizes), generator=gen))
    return torch.repeat_interleave(scale.to(dev), torch.tensor(sizes, device=dev), output_size=d)


def _gradient(case, seed, dev):
    d, values = case["d"], case["values"]
    gen = torch.Generator(device=dev).manual_seed(seed)
    if values == "laplace":
        x = torch.rand(d, generator=gen, device=dev).mul_(2.0).sub_(1.0)
        sign = x.sign()
        x.abs_().clamp_(max=1.0 - 2.0 ** -24).neg_().log1p_().mul_(sign).mul_(-1e-3)
        del sign
        x[torch.randint(d, (max(1, d // 100),), generator=gen, device=dev)] = 0.0
        return x
    x = torch.randn(d, generator=gen, device=dev)
    if values == "outliers":
        hit = torch.randint(d, (max(1, d // 1000),), generator=gen, device=dev)
        x[hit] = 50.0 * x[hit].sign()
        x.mul_(_tensor_scales(case, -4.0, -1.0, dev))
    elif values == "student":
        chi = torch.zeros(d, device=dev)
        for _ in range(3):
            z = torch.randn(d, generator=gen, device=dev)
            chi.addcmul_(z, z)
        x.mul_(chi.div_(3.0).rsqrt_()).mul_(_tensor_scales(case, -5.0, -1.0, dev))
    return x


class _State:
    pass


def prepare(case, seed):
    dev = torch.device("cuda")
    st = _State()
    st.do, st.d, st.bucket, st.s, st.kind = case["do"], case["d"], case["bucket"], case["s"], _kind(case)
    d, bucket, s = st.d, st.bucket, st.s
    if case["levels"] == "table":                           # powers of 0.6, the middle of Sec. 3.3's range
        nuq.set_level_table([0.6 ** (s + 1 - j) for j in range(1, s + 1)])
    words = nuq.encode_bound(d, bucket, s, st.kind) // 4
    st.code, st.grads = None, []
    st.outs = [torch.zeros(words, dtype=torch.int32, device=dev) for _ in range(case["k"])]
    st.bits = [torch.zeros(1, dtype=torch.int64, device=dev) for _ in range(case["k"])]
    for k in range(case["k"]):
        g = _gradient(case, 64 * seed + k, dev)
        if case["mode"] == "coded" and k == 0:              # the code is fitted on a first gradient and then kept
            hist = nuq.level_histogram(g, bucket, s, LEVELS[case["levels"]] | NORMS[case["norm"]], seed=1)
            st.code = nuq.fit_level_code(hist.tolist(), s)
            nuq.set_level_code(st.code)
        if case["do"] == "decode":
            nuq.encode(g, bucket, s, st.kind, seed=k + 1, out=st.outs[k], out_bits=st.bits[k])
        else:
            st.grads.append(g)
    st.acc = torch.zeros(d, device=dev) if case["do"] == "decode" or (case["do"] == "step" and case["k"] <= 2) else None
    if case["do"] == "step":
        gen = torch.Generator(device=dev).manual_seed(64 * seed + 63)
        st.w = torch.randn(d, generator=gen, device=dev).mul_(0.05)
        st.yl = st.w.clone()
    return st


def run(st):
    if st.do == "decode":
        return nuq.decode_accumulate(st.outs, st.d, st.bucket, st.s, acc=st.acc)
    if st.code is not None:                                 # (a program with several models sets the code it needs)
        nuq.set_level_code(st.code)
    for k, g in enumerate(st.grads):
        nuq.encode(g, st.bucket, st.s, st.kind, seed=k + 1, out=st.outs[k], out_bits=st.bits[k])
    if st.do == "encode":
        return {"container": st.outs[0], "bits": st.bits[0]}
    nuq.decode_update(st.outs, st.d, st.bucket, st.s, st.w, yl=st.yl, alpha=ALPHA, mu=MU, l=L, acc=st.acc)
    return {"containers": st.outs, "bits": st.bits, "w": st.w, "yl": st.yl}


def _nonzero_share(case):
    """Expected share of coordinates that keep a nonzero symbol: about E|v| 2^s / norm where that is small."""
    if case["norm"] == "linf":
        return 0.45
    return 1.0 - math.exp(-0.75 * 2.0 ** case["s"] / math.sqrt(case["bucket"]))


def _container_bytes(case):
    d, bucket, s = case["d"], case["bucket"], case["s"]
    norms = 4.0 * math.ceil(d / bucket)
    if case["mode"] == "fixed":
        levels = 2 ** s + 1 if case["levels"] == "uniform" else s + 2
        return norms + d * (1 + math.ceil(math.log2(levels))) / 8
    p = _nonzero_share(case)                                # a token: the run before it, its sign, its level index
    return norms + d * p * (4.2 + 1.2 * math.log2(1.0 / p)) / 8 + d / 256 * 2 + d / min(bucket, 8192) * 8


def work(case):
    d, k, container, p = case["d"], case["k"], _container_bytes(case), _nonzero_share(case)
    enc = {"bytes": 4.0 * d + container, "flops": 10.0 * d}     # square and add, normalise, round
    dec = {"bytes": k * container + 4.0 * d, "flops": 2.0 * k * p * d}
    if case["do"] == "encode":
        return enc
    if case["do"] == "decode":
        return dec
    # the step reads and writes w and y^l; the sum itself is never needed in memory
    return {"bytes": k * enc["bytes"] + k * container + 16.0 * d, "flops": k * enc["flops"] + dec["flops"] + 7.0 * d}


def tolerance(case):
    # containers are the same bits; sums are taken in the order of the workers
    return "exact" if case["do"] == "encode" else {"rel": 1e-6}
