"""Performance cases: what a user of the gradient codec has it do, through its public calls.

Every case is one pass of one kind of call on inputs that stay on the GPU (the last kind: in
pinned host memory):

  roundtrip  compress one gradient, then decode the stream into a cleared dense vector
  compress   compress the gradients of 1..8 workers in one call
  decode     add the streams of 1..8 workers into a dense accumulator
  update     decode the streams and take one Adam step on the decoded coordinates
  kv         compress a gradient that is given as key-value pairs
  host       compress from and decode to host buffers

Inputs are drawn on the GPU from the seed alone, with the distributions of the benchmark
configurations (`paper_2112_04291_b200/workloads.py`): normal values, Student-t or normal values with
per-layer scales, normal values with outliers, and runs of non-zeros in an otherwise zero gradient.
The base b is chosen for the wanted share of kept entries, as there.
"""
import math

import torch

from paper_2112_04291_b200 import binding

SEED_STRIDE = 1_000_003
RUN_MEAN = 32                  # sparse gradients: mean length of a run of non-zeros
SPARSE_KEEP = 0.8              # ... and the share of the non-zeros that is kept


def listed():
    return [
        # the smallest gradients (one layer of a small model): launch latency and host work are all there is
        _case("roundtrip-small", "roundtrip", "normal", 5_003, 1, 0.01),
        # benchmark configuration 1: a million-entry gradient, there and back
        _case("roundtrip-1m", "roundtrip", "normal", 1_048_576, 1, 0.01),
        # configuration 2: a ResNet-50-sized gradient of each of four workers, encoded together
        _case("compress-4x25m", "compress", "layers_t", 25_557_032, 4, 0.005),
        # configuration 4: a BERT-large-sized gradient of each of eight workers
        _case("compress-8x335m", "compress", "layers_normal", 335_141_888, 8, 0.001),
        # configuration 5 at its densest: every tenth entry kept, and an odd length
        _case("compress-67m-dense", "compress", "outliers", 67_108_859, 1, 0.1),
        # group sizes other than the default (larger groups: fewer directory entries)
        _case("compress-16m-groups", "compress", "outliers", 16_777_213, 1, 0.002, group_log2=16),
        # key-value input, configuration 3: a sparse linear model's gradient
        _case("kv-50m", "kv", "sparse", 50_000_000, 1, 0.001),
        # the server's side of configuration 2
        _case("decode-4x25m", "decode", "layers_t", 25_557_032, 4, 0.005),
        # configuration 5: one large stream, its keys scattered over the whole gradient
        _case("decode-268m", "decode", "outliers", 268_435_456, 1, 0.01),
        # the model update of configuration 2, parameters and moments in arrays of their own
        _case("update-4x25m", "update", "layers_t", 25_557_032, 4, 0.005),
        # the update of a model kept as (theta, m, v, g) per coordinate, eight workers
        _case("update-packed-8x67m", "update", "outliers", 67_108_864, 8, 0.01, packed=True),
        # a caller whose buffers live in host memory
        _case("host-1m", "host", "normal", 1_048_576, 1, 0.01),
    ]


def draw(rng):
    kind = rng.choice(["small", "medium", "compress", "compress", "groups", "kv", "decode", "decode", "update", "packed", "host"])
    dist = rng.choice(["normal", "layers_t", "layers_normal", "outliers"])
    flag_bits, tau = rng.choice([1, 2, 2, 2, 3]), rng.choice([64, 128, 128])

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def keep(lo, hi):
        return float("%.3g" % math.exp(rng.uniform(math.log(lo), math.log(hi))))

    opts = {"flag_bits": flag_bits, "tau": tau}
    if kind == "small":
        return _case(None, "roundtrip", "normal", size(1 << 10, 1 << 17), 1, keep(1e-3, 1e-1), **opts)
    if kind == "medium":
        return _case(None, "roundtrip", dist, size(1 << 17, 1 << 23), 1, keep(1e-3, 1e-1), **opts)
    if kind == "compress":
        n = size(1 << 21, 1 << 29)
        return _case(None, "compress", dist, n, rng.randint(1, max(1, min(8, (1 << 30) // n))), keep(1e-4, 1e-1), **opts)
    if kind == "groups":
        return _case(None, "compress", dist, size(1 << 16, 1 << 26), 1, keep(1e-4, 2e-2), group_log2=rng.choice([10, 12, 13, 15, 16, 18]), **opts)
    if kind == "kv":
        return _case(None, "kv", "sparse", size(1 << 20, 1 << 28), 1, keep(1e-4, 4e-3), **opts)
    if kind == "decode":
        n = size(1 << 20, 1 << 28)
        return _case(None, "decode", dist, n, rng.randint(1, max(1, min(8, (1 << 29) // n))), keep(1e-4, 1e-1), **opts)
    if kind == "host":
        return _case(None, "host", dist, size(1 << 12, 1 << 22), 1, keep(1e-3, 1e-1), **opts)
    n = size(1 << 20, 1 << 26)
    return _case(None, "update", dist, n, rng.randint(1, 8), keep(1e-4, 5e-2), packed=kind == "packed", **opts)


def _case(name, op, dist, n, workers, keep, *, group_log2=14, flag_bits=2, tau=128, packed=False):
    c = {"op": op, "dist": dist, "n": n, "workers": workers, "keep": keep, "group_log2": group_log2,
         "flag_bits": flag_bits, "tau": tau, "packed": packed}
    return dict(c, name=name) if name else c


# ---- inputs ---------------------------------------------------------------------------------

def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * SEED_STRIDE + stream)
    return g


def _layer_scales(n, layers, lo, hi, seed):
    """Contiguous layers with heavy-tailed sizes and log-uniform scales: (sizes, scales) on the host."""
    g = torch.Generator()
    g.manual_seed(seed)
    w = torch.exp(6.0 * torch.rand(layers, generator=g, dtype=torch.float64))
    sizes = torch.clamp((w / w.sum() * n).long(), min=1)
    while int(sizes.sum()) > n:                                        # (only when n is not much larger than the number of layers)
        sizes[int(sizes.argmax())] -= int(min(int(sizes.sum()) - n, int(sizes.max()) - 1))
    sizes[-1] += n - int(sizes.sum())
    scales = torch.exp(math.log(lo) + (math.log(hi) - math.log(lo)) * torch.rand(layers, generator=g, dtype=torch.float64))
    return sizes.tolist(), scales.tolist()


def _gradient(case, seed, worker):
    """One worker's dense gradient.  The layers are the model's: shared by the workers."""
    n, dist = case["n"], case["dist"]
    g = _generator(seed, worker)
    v = torch.empty(n, dtype=torch.float32, device="cuda")
    v.normal_(generator=g)
    if dist == "normal":
        v.mul_(1e-3)
    elif dist == "outliers":                                           # a random 1 % of the entries is 100 times larger
        v.mul_(1e-3)
        at = torch.randint(0, n, (max(1, n // 100),), generator=g, device="cuda")
        v[at] *= 100.0
    else:
        if dist == "layers_t":                                         # Student-t with 3 degrees of freedom
            part = 1 << 26
            for lo in range(0, n, part):
                x = v[lo:lo + part]
                chi2 = torch.zeros_like(x)
                for _ in range(3):
                    chi2 += torch.empty_like(x).normal_(generator=g).square_()
                x.div_(chi2.div_(3.0).clamp_(min=1e-12).sqrt_())
            sizes, scales = _layer_scales(n, 161, 1e-4, 1e-1, seed)
        else:
            sizes, scales = _layer_scales(n, 400, 1e-5, 1e-2, seed)
        for x, scale in zip(torch.split(v, sizes), scales):
            x.mul_(scale)
    return v


def _pairs(case, seed):
    """The non-zeros of a sparse model's gradient: ascending keys in runs, Laplace values."""
    n = case["n"]
    g = _generator(seed, 0)
    runs = max(1, int(case["keep"] * n) // RUN_MEAN)
    start = torch.randint(0, n, (runs, 1), generator=g, device="cuda")
    length = torch.poisson(torch.full((runs, 1), float(RUN_MEAN), device="cuda"), generator=g)
    step = torch.arange(3 * RUN_MEAN, device="cuda").unsqueeze(0)
    keys = (start + step)[step < length]
    keys = torch.unique(keys[keys < n])                                # ascending
    u = torch.rand(keys.numel(), generator=g, device="cuda") - 0.5
    values = -1e-2 * torch.sign(u) * torch.log1p(-2.0 * u.abs().clamp(max=0.4999999))
    return keys.to(torch.int32), values


def _base_for(values, keep, tau):
    """b such that about `keep` of the entries reach sum / b^tau."""
    a = values.abs()
    sample = a[:: max(1, a.numel() >> 22)].sort().values               # (the threshold from a regular sample of up to eight million)
    q = float(sample[min(sample.numel() - 1, int(round((1.0 - keep) * sample.numel())))])
    s = float(a.sum(dtype=torch.float64))
    return max((s / q) ** (1.0 / tau), 1.0 + 1e-9) if s > q > 0.0 else 1.1


def _capacity(case, p):
    """Room for the stream: twice the expected number of kept entries at their widest."""
    groups = -(-case["n"] >> case["group_log2"])
    widest = (8 + case["flag_bits"] + case["group_log2"] + 7) // 8
    room = 64 + 12 * groups + 2 * widest * int(case["keep"] * case["n"] + 64)
    return (min(binding.compress_bound(case["n"], p), room) + 255) & ~255


def _checked(rc):
    if rc != binding.OK:
        raise binding.FastSGDError(rc, "perf case")


def prepare(case, seed):
    n, op, workers = case["n"], case["op"], case["workers"]
    state = {"op": op, "n": n, "packed": case["packed"]}

    def params(values, keep):
        return binding.params(_base_for(values, keep, case["tau"]), case["tau"], case["flag_bits"], case["group_log2"])

    if op == "kv":
        state["keys"], state["values"] = _pairs(case, seed)
        p = params(state["values"], SPARSE_KEEP)
        grads = []
    else:
        grads = [_gradient(case, seed, w) for w in range(workers)]
        p = params(grads[0], case["keep"])
    state["p"] = p
    binding.ensure_workspace(n, p)
    cap = _capacity(case, p)
    outs = [torch.zeros(cap, dtype=torch.uint8, device="cuda") for _ in range(workers)]

    if op in ("roundtrip", "compress", "kv"):
        state["grads"], state["outs"], state["sizes"] = grads, outs, [cap] * workers
        if op == "roundtrip":
            state["dense"] = torch.zeros(n, dtype=torch.float32, device="cuda")
    elif op == "host":
        state["grad"] = grads[0].cpu().pin_memory()
        state["out"] = torch.zeros(cap, dtype=torch.uint8).pin_memory()
        state["dense"] = torch.zeros(n, dtype=torch.float32).pin_memory()
        state["scratch"] = torch.empty(binding.host_scratch_bytes(n, p), dtype=torch.uint8, device="cuda")
    else:
        # the streams as they arrive from the workers: exactly as long as they are
        _checked(binding.compress_batch(grads, p, outs))
        state["sizes"] = [binding.stream_info(o)[0] for o in outs]
        state["outs"] = [o[:size].clone() for o, size in zip(outs, state["sizes"])]
        g = _generator(seed, workers)
        if op == "decode":
            state["dense"] = torch.zeros(n, dtype=torch.float32, device="cuda")
        else:
            # a model some steps into its training; g is the library's scratch, all zero between calls
            theta = torch.empty(n, dtype=torch.float32, device="cuda").normal_(generator=g).mul_(0.05)
            m = torch.empty_like(theta).normal_(generator=g).mul_(1e-3)
            v = torch.empty_like(theta).normal_(generator=g).mul_(1e-3).square_()
            arrays = [theta, m, v, torch.zeros_like(theta)]
            state["hyper"] = binding.Adam(1e-3, 0.9, 0.999, 1e-8)
            state["arrays"] = [torch.stack(arrays, dim=1).reshape(-1)] if case["packed"] else arrays
    return state


def run(state):
    op, n, p = state["op"], state["n"], state["p"]
    if op == "roundtrip":
        dense = state["dense"].zero_()
        _checked(binding.compress(state["grads"][0], p, state["outs"][0]))
        _checked(binding.decompress_accumulate(state["outs"][0], state["sizes"][0], n, p, dense))
        return state["outs"][0], dense
    if op == "compress":
        if len(state["grads"]) == 1:
            _checked(binding.compress(state["grads"][0], p, state["outs"][0]))
        else:
            _checked(binding.compress_batch(state["grads"], p, state["outs"]))
        return state["outs"]
    if op == "kv":
        _checked(binding.compress_kv(state["keys"], state["values"], n, p, state["outs"][0]))
        return state["outs"][0]
    if op == "decode":
        _checked(binding.decompress_accumulate_batch(state["outs"], state["sizes"], n, p, state["dense"]))
        return state["dense"]
    if op == "update":
        if state["packed"]:
            _checked(binding.sparse_adam_update_packed_batch(state["outs"], state["sizes"], n, p, state["hyper"], state["arrays"][0]))
        else:
            theta, m, v, g = state["arrays"]
            _checked(binding.sparse_adam_update_batch(state["outs"], state["sizes"], n, p, state["hyper"], g, theta, m, v))
        return state["arrays"]
    rc, size, status = binding.compress_host(state["grad"], p, state["out"], state["scratch"])
    _checked(rc or status)
    rc, status = binding.decompress_accumulate_host([state["out"]], [size], n, p, state["dense"], state["scratch"])
    _checked(rc or status)
    return state["out"], state["dense"]


def work(case):
    """Bytes of the inputs read once and the outputs written once (streams by their expected length)."""
    n, op, workers = case["n"], case["op"], case["workers"]
    kept = case["keep"] * n * (SPARSE_KEEP if op == "kv" else 1.0)
    gap = 4.0 if op == "kv" else 1.0 / case["keep"]
    stream = 64 + 8 * -(-n >> case["group_log2"]) + kept * (8 + case["flag_bits"] + math.log2(gap) + 1) / 8
    if op == "kv":
        return {"bytes": 8 * case["keep"] * n + stream, "flops": 0}
    if op == "compress":
        return {"bytes": workers * (4 * n + stream), "flops": 0}
    if op == "decode":                                                 # every decoded entry is read and written
        return {"bytes": workers * (stream + 8 * kept), "flops": 0}
    if op == "update":                                                 # theta, m and v of every decoded coordinate
        return {"bytes": workers * (stream + 24 * kept), "flops": 0}
    return {"bytes": 4 * n + 2 * stream + 4 * n, "flops": 0}           # gradient in, stream out and in, dense vector out


def tolerance(case):
    """Streams are bytes and the same bit for bit.  Sums of decoded values and the Adam step are fp32."""
    if case["op"] in ("compress", "kv"):
        return "exact"
    return {"rel": 1e-5 if case["op"] == "update" else 1e-6}
