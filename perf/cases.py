"""Workloads of the sum library, as a program meets them.

Every case goes through the public Python binding (which only marshals
arguments to the C ABI).  Five kinds of call:

  sum    one device array, the library choosing the launch (SR_AUTO)
  graph  many small device arrays summed by one replayed CUDA graph
  seg    one call over the CSR segments of a device array
  train  one optimiser step of the small network behind the launch selector
  host   one page-locked host array, result on the host

Values have a non-zero mean (as losses, counts and squared norms do), so a
sum's relative error says something about the summation and not about the
cancellation of the input; the compensated cases take signed lognormal
magnitudes, the input compensation is for.
"""
import math

import torch

import paper_2004_05371_gb300 as sr

DTYPES = {"f32": torch.float32, "i32": torch.int32, "bf16": torch.bfloat16, "fp8": torch.float8_e4m3fn}
ELEM_BYTES = {"f32": 4, "i32": 4, "bf16": 2, "fp8": 1}
FP8_SCALE = 0.0078125  # per-tensor dequantisation factor of the FP8 arrays
OPTIONS = {"": 0, "kahan": sr.F_KAHAN, "kahan_fp64": sr.F_KAHAN | sr.F_FP64_COMBINE, "adaptive": sr.F_ADAPTIVE_SEGMENTS}
GRAPH_DTYPES = ("f32", "bf16", "f32", "i32")  # the tensors of a graph, in turn
NET = (9, 64, 40)  # features, hidden units, candidates of the launch selector
LR = 3e-3

_capture_stream = None


def listed():
    return [
        # a scalar statistic of one small tensor, called eagerly: launch and host latency
        {"name": "sum_f32_2p14", "kind": "sum", "dtype": "f32", "n": 1 << 14, "shift": 0, "option": ""},
        # per-tensor statistics of a step: 48 small tensors of 256 to 262,144 elements, one graph launch
        {"name": "graph_48_small", "kind": "graph", "count": 48, "lo": 1 << 8, "hi": 1 << 18, "salt": 1},
        # an ordinary activation-sized tensor of odd length, not aligned to the vector loads
        {"name": "sum_f32_2p24_odd", "kind": "sum", "dtype": "f32", "n": (1 << 24) + 3, "shift": 1, "option": ""},
        # the device-wide sum over 1 GiB
        {"name": "sum_f32_2p28", "kind": "sum", "dtype": "f32", "n": 1 << 28, "shift": 0, "option": ""},
        # a compensated sum of half-precision data
        {"name": "sum_bf16_kahan_2p28", "kind": "sum", "dtype": "bf16", "n": 1 << 28, "shift": 0, "option": "kahan"},
        # a quantised tensor with its scale, odd length
        {"name": "sum_fp8_2p28_odd", "kind": "sum", "dtype": "fp8", "n": (1 << 28) - 5, "shift": 3, "option": ""},
        # the batched workload: 10,000 arrays of very different lengths
        {"name": "seg_10k_f32", "kind": "seg", "dtype": "f32", "nseg": 10_000, "mean": 26_844, "layout": "lognormal",
         "sigma": 1.94, "shift": 0, "option": ""},
        # a million rows of a few hundred elements, ragged
        {"name": "seg_1m_bf16", "kind": "seg", "dtype": "bf16", "nseg": 1_000_000, "mean": 268, "layout": "ragged",
         "sigma": 0.0, "shift": 1, "option": ""},
        # two million very short rows (0 to 32 elements): counts per key
        {"name": "seg_2m_short_i32", "kind": "seg", "dtype": "i32", "nseg": 1 << 21, "mean": 16, "layout": "ragged",
         "sigma": 0.0, "shift": 0, "option": ""},
        # four million rows of skewed length, empty ones among them, layout unknown to the caller
        {"name": "seg_4m_f32_adaptive", "kind": "seg", "dtype": "f32", "nseg": 1 << 22, "mean": 64,
         "layout": "lognormal", "sigma": 1.5, "shift": 0, "option": "adaptive"},
        # one training step of the launch selector's network
        {"name": "train_256", "kind": "train", "batch": 256},
        # data that starts on the host: 64 MiB of page-locked memory, odd length
        {"name": "host_f32_2p24", "kind": "host", "n": (1 << 24) + 7},
    ]


def draw(rng):
    kind = rng.choice(["sum", "sum", "sum", "sum", "graph", "seg", "seg", "seg", "seg", "train", "host"])
    if kind == "sum":
        dtype = rng.choice(["f32", "f32", "bf16", "fp8", "i32"])
        option = "" if dtype == "i32" else rng.choice(["", "", "kahan", "kahan_fp64"])
        n = int(2.0 ** rng.uniform(10.0, 28.0)) | rng.randint(0, 1)
        return {"kind": "sum", "dtype": dtype, "n": n, "shift": rng.choice([0, 0, 1, 3]), "option": option}
    if kind == "graph":
        return {"kind": "graph", "count": rng.randint(16, 96), "lo": 1 << 8, "hi": int(2.0 ** rng.uniform(14.0, 18.0)),
                "salt": rng.randint(2, 1 << 20)}
    if kind == "seg":
        dtype = rng.choice(["f32", "f32", "bf16", "fp8", "i32"])
        option = rng.choice(["", "", "", "adaptive"]) if dtype == "i32" else rng.choice(["", "", "", "kahan", "adaptive"])
        total = 2.0 ** rng.uniform(18.0, 27.5)
        nseg = max(64, min(1 << 22, int(total / 2.0 ** rng.uniform(4.0, 15.0))))
        layout = rng.choice(["equal", "ragged", "lognormal", "lognormal"])
        return {"kind": "seg", "dtype": dtype, "nseg": nseg, "mean": max(2, int(total / nseg)), "layout": layout,
                "sigma": round(rng.uniform(0.5, 2.0), 2) if layout == "lognormal" else 0.0,
                "shift": rng.choice([0, 0, 1]), "option": option}
    if kind == "train":
        return {"kind": "train", "batch": int(2.0 ** rng.uniform(5.0, 11.0))}
    return {"kind": "host", "n": int(2.0 ** rng.uniform(18.0, 25.0)) | 1}


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _values(n, dtype, signed, gen):
    if dtype == "i32":
        return torch.randint(-1000, 1001, (n,), dtype=torch.int32, device="cuda", generator=gen)
    if signed:
        v = torch.empty(n, dtype=torch.float32, device="cuda").log_normal_(0.0, 2.0, generator=gen)
        v *= torch.randint(0, 2, (n,), dtype=torch.int8, device="cuda", generator=gen).mul_(2).sub_(1)
        v.clamp_(-400.0, 400.0)
    else:
        v = torch.rand(n, dtype=torch.float32, device="cuda", generator=gen)
        v.mul_(1.5).sub_(0.5)
        if dtype == "fp8":
            v.mul_(128.0)
    return v.to(DTYPES[dtype])


def _array(n, dtype, shift, signed, gen):
    """n values that start `shift` elements into their buffer."""
    return _values(n + shift, dtype, signed, gen)[shift:]


def _offsets(case, gen):
    nseg, mean = case["nseg"], case["mean"]
    if case["layout"] == "equal":
        lens = torch.full((nseg,), mean, dtype=torch.int64, device="cuda")
    elif case["layout"] == "ragged":
        lens = torch.randint(0, 2 * mean + 1, (nseg,), dtype=torch.int64, device="cuda", generator=gen)
    else:
        sigma = case["sigma"]
        w = torch.empty(nseg, dtype=torch.float64, device="cuda").log_normal_(0.0, sigma, generator=gen)
        lens = (w * (mean * nseg / float(w.sum()))).floor().to(torch.int64)
    off = torch.zeros(nseg + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=off[1:])
    return off


def _config(case):
    c = sr.make_config(sr.AUTO | OPTIONS[case["option"]])
    if case["dtype"] == "fp8":
        c.scale = FP8_SCALE
    return c


def _graph_sizes(case):
    """Sizes spread over the logarithm of [lo, hi], odd ones among them."""
    state, sizes = case["salt"], []
    for _ in range(case["count"]):
        state = (state * 1103515245 + 12345) % (1 << 31)
        sizes.append(int(case["lo"] * (case["hi"] / case["lo"]) ** (state / float(1 << 31))))
    return sizes


def _graph_arrays(case, gen):
    out = []
    for i, n in enumerate(_graph_sizes(case)):
        dtype = GRAPH_DTYPES[i % len(GRAPH_DTYPES)]
        out.append(_array(n, dtype, 0, False, gen))
    return out


def _net_inputs(case, gen):
    n_in, hidden, n_out = NET
    sizes = [(n_in * hidden, n_in), (hidden, 0), (hidden * hidden, hidden), (hidden, 0), (hidden * n_out, hidden), (n_out, 0)]
    params = torch.cat([torch.randn(k, device="cuda", generator=gen) * (math.sqrt(2.0 / fan) if fan else 0.01)
                        for k, fan in sizes])
    x = torch.randn(case["batch"], n_in, device="cuda", generator=gen)
    q = torch.softmax(4.0 * torch.randn(case["batch"], n_out, device="cuda", generator=gen), dim=1)
    return params, x, q


def _host_values(case, gen):
    return _values(case["n"], "f32", False, gen)


def prepare(case, seed):
    global _capture_stream
    gen = _generator(seed)
    if case["kind"] == "sum":
        x = _array(case["n"], case["dtype"], case["shift"], "kahan" in case["option"], gen)
        return {"kind": "sum", "x": x, "config": _config(case)}
    if case["kind"] == "seg":
        off = _offsets(case, gen)
        x = _array(max(1, int(off[-1])), case["dtype"], case["shift"], "kahan" in case["option"], gen)
        return {"kind": "seg", "x": x, "off": off, "config": _config(case)}
    if case["kind"] == "graph":
        xs = _graph_arrays(case, gen)
        outs = [torch.empty((), dtype=sr.out_dtype(sr.dtype_code(x), 0), device="cuda") for x in xs]
        if _capture_stream is None:
            _capture_stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(_capture_stream):  # the first call on a stream allocates its workspace
            for x, out in zip(xs, outs):
                sr.reduce_sum(x, out=out)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=_capture_stream):
            for x, out in zip(xs, outs):
                sr.reduce_sum(x, out=out)
        return {"kind": "graph", "graph": g, "xs": xs, "outs": outs}
    if case["kind"] == "train":
        params, x, q = _net_inputs(case, gen)
        mlp = sr.MLP(*NET)
        mlp.set_params(params.cpu().numpy())
        return {"kind": "train", "mlp": mlp, "x": x, "q": q,
                "loss": torch.empty((), dtype=torch.float32, device="cuda"),
                "grad": torch.empty(mlp.P, dtype=torch.float32, device="cuda")}
    x = torch.empty(case["n"], dtype=torch.float32, pin_memory=True)
    x.copy_(_host_values(case, gen))
    return {"kind": "host", "x": x, "out": torch.empty(1, dtype=torch.float32, pin_memory=True)}


def run(state):
    kind = state["kind"]
    if kind == "sum":
        return sr.reduce_sum(state["x"], config=state["config"])
    if kind == "seg":
        return sr.reduce_sum_segmented(state["x"], state["off"], config=state["config"])
    if kind == "graph":
        state["graph"].replay()
        return state["outs"]
    if kind == "train":
        state["mlp"].train_step(state["x"], state["q"], LR, loss=state["loss"], grad=state["grad"])
        return {"loss": state["loss"], "grad": state["grad"]}
    sr.check(sr.reduce_sum_host_ptr(state["x"].data_ptr(), state["x"].numel(), sr.F32, state["out"].data_ptr()))
    return state["out"]


# -------------------------------------------------------------------- work
def work(case):
    if case["kind"] == "sum":
        return {"bytes": case["n"] * ELEM_BYTES[case["dtype"]] + 8, "flops": case["n"]}
    if case["kind"] == "seg":
        n = case["nseg"] * case["mean"]
        out = 8 if case["dtype"] == "i32" else 4
        return {"bytes": n * ELEM_BYTES[case["dtype"]] + case["nseg"] * (8 + out), "flops": n}
    if case["kind"] == "graph":
        sizes = _graph_sizes(case)
        return {"bytes": sum(n * ELEM_BYTES[GRAPH_DTYPES[i % len(GRAPH_DTYPES)]] + 8 for i, n in enumerate(sizes)),
                "flops": sum(sizes)}
    if case["kind"] == "train":
        n_in, hidden, n_out = NET
        weights = n_in * hidden + hidden * hidden + hidden * n_out
        params = weights + 2 * hidden + n_out
        # inputs and targets read, parameters and both moments read and written, gradient written;
        # forward, weight gradients, and the backward products of the two upper layers
        return {"bytes": 4 * (case["batch"] * (n_in + n_out) + 7 * params),
                "flops": 2 * case["batch"] * (2 * weights + hidden * hidden + hidden * n_out)}
    return {"bytes": 4 * case["n"] + 4, "flops": case["n"]}


# ------------------------------------------------------------------- exact
def _exact_sum(x, dtype):
    if dtype == "i32":
        return x.to(torch.int64).sum()
    scale = FP8_SCALE if dtype == "fp8" else 1.0
    total = torch.zeros((), dtype=torch.float64, device="cuda")
    for part in x.split(1 << 26):
        total += part.to(torch.float64).sum()
    return total * scale


def _exact_segments(x, off, dtype):
    n = int(off[-1])
    wide = torch.int64 if dtype == "i32" else torch.float64
    out = torch.zeros(off.numel() - 1, dtype=wide, device="cuda")
    row = torch.searchsorted(off, torch.arange(0, n, 1 << 24, device="cuda"), right=True) - 1
    for k, a in enumerate(range(0, n, 1 << 24)):  # pieces: short running sums, little memory
        b = min(n, a + (1 << 24))
        run_sum = torch.zeros(b - a + 1, dtype=wide, device="cuda")
        torch.cumsum(x[a:b].to(wide), 0, out=run_sum[1:])
        first = int(row[k])
        last = int(torch.searchsorted(off, torch.tensor([b], device="cuda"), right=False)[0])
        edges = (off[first:last + 1].clamp(a, b) - a)
        out[first:last] += run_sum[edges[1:]] - run_sum[edges[:-1]]
    return out * FP8_SCALE if dtype == "fp8" else out


def exact(case, seed):
    gen = _generator(seed)
    if case["kind"] == "sum":
        x = _array(case["n"], case["dtype"], case["shift"], "kahan" in case["option"], gen)
        return _exact_sum(x, case["dtype"])
    if case["kind"] == "seg":
        off = _offsets(case, gen)
        x = _array(max(1, int(off[-1])), case["dtype"], case["shift"], "kahan" in case["option"], gen)
        return _exact_segments(x, off, case["dtype"])
    if case["kind"] == "graph":
        return [_exact_sum(x, GRAPH_DTYPES[i % len(GRAPH_DTYPES)]) for i, x in enumerate(_graph_arrays(case, gen))]
    if case["kind"] == "train":
        params, x, q = (t.double() for t in _net_inputs(case, gen))
        n_in, hidden, n_out = NET
        shapes = [(n_in, hidden), (hidden,), (hidden, hidden), (hidden,), (hidden, n_out), (n_out,)]
        parts, at = [], 0
        for s in shapes:
            k = math.prod(s)
            parts.append(params[at:at + k].view(s).clone().requires_grad_(True))
            at += k
        w1, b1, w2, b2, w3, b3 = parts
        z = torch.relu(torch.relu(x @ w1 + b1) @ w2 + b2) @ w3 + b3
        loss = -(q * torch.log_softmax(z, dim=1)).sum(dim=1).mean()
        loss.backward()
        return {"loss": loss.detach(), "grad": torch.cat([p.grad.reshape(-1) for p in parts])}
    return _exact_sum(_host_values(case, gen), "f32").reshape(1)
