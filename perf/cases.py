"""What the library is timed on: attention calls, generations, the 8-bit paths and the calibration pass, as a VAR
image generator calls them.

A case is a dict of plain values; ``kind`` says which entry points it goes through:

  attention    one Plan.forward call per listed step of one layer, or of several layers (``layers``), called one by
               one ("eager") or replayed from a CUDA graph captured beforehand ("graph")
  kv8          the same steps through Plan.forward_kv8 on an 8-bit K/V cache
  qkv8         8-bit Q/K/V without an 8-bit cache: the step's Q and the appended K and V rows go through
               quantize_rows (K and V straight into the cache), then Plan.forward
  quantise     quantize_rows of a whole tensor with codes, scales and zero points
  calibrate    calibrate_windows on saved attention maps

Schedules are written "1-2-3-4"; step k has s_k^2 queries and reads the cache rows of scales 1 .. k.
"""
import math

import numpy as np
import torch

from paper_2411_17178_b200 import binding, workloads as wl

HEAD_DIM = wl.HEAD_DIM
S256, S512, S2K = ("-".join(map(str, s)) for s in (wl.SCALES_256, wl.SCALES_512, wl.SCALES_2K))


def attention_case(name, scales, first_step, last_step, heads, pairs, share, rho="1/4", kind="attention", launch="eager",
                   layers=1, shape="square", sets=1, layout="heads", sharp_keys=False):
    return {"name": name, "kind": kind, "scales": scales, "first_step": first_step, "last_step": last_step,
            "heads": heads, "pairs": pairs, "share": share, "rho": rho, "launch": launch, "layers": layers,
            "shape": shape, "sets": sets, "layout": layout, "sharp_keys": sharp_keys}


def listed():
    return [
        # the smallest call: an early step for one image, where latency and the launch are all there is
        attention_case("256px_step3_one_image", S256, 3, 3, 16, 1, True),
        # the last step for one image: a tensor-core call that does not fill the chip
        attention_case("256px_step10_one_image", S256, 10, 10, 16, 1, False),
        # a whole 256px generation of a 16-layer generator for eight images, replayed from a CUDA graph as a server
        # that has warmed up does: 160 small and middling calls
        attention_case("256px_generation_16_layers", S256, 1, 10, 16, 8, True, launch="graph", layers=16),
        # one layer of a 30-head generator with a full batch of 32 images, called from Python
        attention_case("256px_layer_batch_32", S256, 1, 10, 30, 32, True),
        # one layer at 512px, 36 heads, keys of different sharpness per head
        attention_case("512px_layer", S512, 1, 10, 36, 8, True, sharp_keys=True),
        # one layer of a 2K generation for one image, no sharing: every step from 1 to 16384 queries
        attention_case("2k_layer", S2K, 1, 14, 16, 1, False),
        # the largest call: the last 2K step with full attention (R_0 = 1, the mask the paper starts from)
        attention_case("2k_step14_full_attention", S2K, 14, 14, 16, 1, False, rho="full"),
        # sizes off every tile boundary, two window sets over an odd number of heads, token-major tensors
        attention_case("ragged_layer_head_sets", "1-2-3-5-7-11-17-23-31", 1, 9, 5, 3, False, sets=2, layout="tokens"),
        # the 512px layer on an 8-bit cache
        attention_case("512px_layer_8bit_cache", S512, 1, 10, 36, 8, True, kind="kv8", sharp_keys=True),
        # a 256px layer whose Q, K and V rows are quantised to 8 bits as they are produced
        attention_case("256px_layer_8bit_qkv", S256, 1, 10, 16, 8, True, kind="qkv8", launch="graph"),
        # building an 8-bit cache from a bf16 one: 30 heads, 64 batch rows, a full 256px cache
        {"name": "quantise_cache", "kind": "quantise", "batch": 64, "heads": 30, "tokens": 680, "bits": 8},
        # calibrating the windows of the last 512px step on saved attention maps
        {"name": "calibrate_512px_step10", "kind": "calibrate", "scales": S512, "step": 10, "maps": 64, "r0": 0.95},
    ]


def log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def random_schedule(rng, top):
    """A coarse-to-fine schedule that ends at grid side `top`: 1-2-3 or 1-2-3-4, then growing by 1.2 to 1.6 a step."""
    s = [x for x in (1, 2, 3, 4)[:rng.choice((3, 4))] if x < top]
    while len(s) < 15:
        nxt = max(s[-1] + 1, int(round(s[-1] * rng.uniform(1.2, 1.6))))
        if nxt >= top:
            break
        s.append(nxt)
    return "-".join(map(str, s + [top]))


def draw(rng):
    most = max(work(c)["flops"] for c in listed())
    while True:
        kind = rng.choice(("attention",) * 6 + ("kv8", "qkv8", "quantise", "calibrate"))
        if kind == "quantise":
            c = {"kind": kind, "batch": log_uniform(rng, 2, 64), "heads": rng.randint(4, 36),
                 "tokens": log_uniform(rng, 1, 2240), "bits": rng.choice((4, 6, 8, 8))}
            small = c["batch"] * c["heads"] * c["tokens"] <= 64 * 30 * 680
        elif kind == "calibrate":
            scales = random_schedule(rng, log_uniform(rng, 8, 32))
            c = {"kind": kind, "scales": scales, "step": len(sides(scales)), "maps": log_uniform(rng, 4, 1280),
                 "r0": rng.choice((0.8, 0.9, 0.95))}
            n_k, l_k = step_shape(scales, c["step"])
            small = c["maps"] * n_k * l_k <= 64 * 1024 * 2240
        else:
            bf16 = kind == "attention"
            scales = random_schedule(rng, log_uniform(rng, 4, 128 if bf16 else 32))
            last = len(sides(scales))
            c = attention_case("", scales, rng.choice((1, last)), last, rng.randint(4, 36), log_uniform(rng, 1, 32),
                               rng.random() < 0.6, rho=rng.choice(("1/8", "1/4", "1/4", "1/2", "full")), kind=kind,
                               launch=rng.choice(("eager", "graph")), shape="band" if rng.random() < 0.15 else "square",
                               layout=rng.choice(("heads", "tokens")), sharp_keys=rng.random() < 0.3)
            if c["rho"] != "full" and c["shape"] == "square" and bf16 and rng.random() < 0.25:
                c["sets"] = rng.choice((2, 3))
            del c["name"]
            cache = 2 * c["pairs"] * c["heads"] * sum(s * s for s in sides(scales))
            small = cache <= 64 * 30 * 680 and work(c)["flops"] <= most
        if small:
            return c


# ------------------------------------------------------------------------------------------------- sizes and work
def sides(scales):
    return [int(s) for s in scales.split("-")]


def step_shape(scales, k):
    s = sides(scales)
    return s[k - 1] ** 2, sum(x * x for x in s[:k])


def radius_tables(c):
    """[sets][K][K] window radii: the library's default rule (scales 1 to 3 global, then rho * extent rounded half
    up), set i > 0 with windows 1 / (i + 1) as wide; -1 = the whole part is live."""
    s = sides(c["scales"])
    t = np.full((c["sets"], len(s), len(s)), -1, np.int32)
    if c["rho"] != "full":
        num, den = (int(x) for x in c["rho"].split("/"))
        for i in range(c["sets"]):
            for j in range(3, len(s)):
                extent = s[j] * s[j] if c["shape"] == "band" else s[j]
                t[i, j:, j] = (2 * num * extent + den * (i + 1)) // (2 * den * (i + 1))
    return t


def live_entries(c, k, radius):
    """Live (query, key) pairs of step k under one row of radii."""
    s = sides(c["scales"])
    s_k, total = s[k - 1], 0
    for j in range(k):
        n, m = (s_k * s_k, s[j] * s[j]) if c["shape"] == "band" else (s_k, s[j])
        if radius[j] < 0:
            total += s_k * s_k * s[j] * s[j]
            continue
        ctr = (2 * np.arange(n, dtype=np.int64) + 1) * m // (2 * n)
        per_axis = int((np.minimum(m - 1, ctr + radius[j]) - np.maximum(0, ctr - radius[j]) + 1).sum())
        total += per_axis if c["shape"] == "band" else per_axis * per_axis
    return total


def work(c):
    """Bytes: each input read once, each output written once.  Operations: 4 * 64 per live entry of the map for every
    (batch row, head) that is computed; under CFG sharing only half of the rows are read and computed."""
    if c["kind"] == "quantise":
        rows = c["batch"] * c["heads"] * c["tokens"]
        return {"bytes": rows * (2 * HEAD_DIM * 2 + HEAD_DIM + 8), "flops": 0}
    if c["kind"] == "calibrate":
        n_k, l_k = step_shape(c["scales"], c["step"])
        l_g = sum(x * x for x in sides(c["scales"])[:3])  # the global parts need no reading
        return {"bytes": c["maps"] * n_k * (l_k - l_g) * 4, "flops": 0}
    tables = radius_tables(c)
    rows = 2 * c["pairs"]
    computed = c["pairs"] if c["share"] else rows
    nbytes = flops = 0
    for k in range(c["first_step"], c["last_step"] + 1):
        n_k, l_k = step_shape(c["scales"], k)
        live = [live_entries(c, k, tables[i, k - 1]) for i in range(c["sets"])]
        for h in range(c["heads"]):
            flops += 4 * HEAD_DIM * computed * live[h % c["sets"]]
        kv_row = HEAD_DIM + 8 if c["kind"] == "kv8" else 2 * HEAD_DIM
        nbytes += c["heads"] * (computed * (n_k * 2 * HEAD_DIM + 2 * l_k * kv_row) + rows * n_k * 2 * HEAD_DIM)
        if c["kind"] == "qkv8":  # the step's bf16 rows in, the quantised ones out, for all batch rows
            nbytes += c["heads"] * rows * 3 * n_k * 2 * 2 * HEAD_DIM
    return {"bytes": nbytes * c["layers"], "flops": flops * c["layers"]}


# ------------------------------------------------------------------------------------------------- inputs and passes
def random_rows(gen, batch, heads, tokens, layout="heads", head_scale=None):
    """N(0,1) bf16 rows [batch, heads, tokens, 64]: stored that way, or token-major as a projection leaves them."""
    shape = (batch, heads, tokens, HEAD_DIM) if layout == "heads" else (batch, tokens, heads, HEAD_DIM)
    x = torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)
    x = x if layout == "heads" else x.transpose(1, 2)
    return x if head_scale is None else x.mul_(head_scale.view(1, -1, 1, 1))


def empty_rows(batch, heads, tokens, layout):
    if layout == "heads":
        return torch.empty((batch, heads, tokens, HEAD_DIM), device="cuda", dtype=torch.bfloat16)
    return torch.empty((batch, tokens, heads, HEAD_DIM), device="cuda", dtype=torch.bfloat16).transpose(1, 2)


def prepare(c, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    if c["kind"] == "quantise":
        # rows as after a projection: an offset per head and one channel with outliers
        x = random_rows(gen, c["batch"], c["heads"], c["tokens"])
        x.mul_(0.3).add_(torch.linspace(-2, 2, c["heads"], device="cuda").to(torch.bfloat16).view(1, -1, 1, 1))
        x[..., 5] *= 9.0
        return {"case": c, "x": x, "out": torch.empty_like(x)}
    if c["kind"] == "calibrate":
        n_k, l_k = step_shape(c["scales"], c["step"])
        maps = torch.randn((c["maps"], n_k, l_k), generator=gen, device="cuda").mul_(2.0)
        for m in maps.split(max(1, (1 << 26) // (n_k * l_k))):
            m.copy_(torch.softmax(m, dim=-1))
        return {"case": c, "scales": sides(c["scales"]), "maps": maps}

    s, rows, heads, layout = sides(c["scales"]), 2 * c["pairs"], c["heads"], c["layout"]
    plan = binding.Plan(
        s, n_heads=heads, radius=radius_tables(c), n_sets=c["sets"],
        head_to_set=[h % c["sets"] for h in range(heads)] if c["sets"] > 1 else None,
        share_steps=[1 if c["share"] else 0] * len(s),
        shape=binding.WINDOW_BAND if c["shape"] == "band" else binding.WINDOW_SQUARE)
    sharp = None
    if c["sharp_keys"]:
        sharp = (0.5 + 1.5 * torch.rand(heads, generator=gen, device="cuda")).to(torch.bfloat16)
    steps = range(c["first_step"], c["last_step"] + 1)
    calls, outs = [], []
    tokens = {k: step_shape(c["scales"], k) for k in steps}
    caches = []
    for _ in range(c["layers"]):
        l_max = tokens[c["last_step"]][1]
        kc = random_rows(gen, rows, heads, l_max, layout, sharp)
        vc = random_rows(gen, rows, heads, l_max, layout)
        if c["kind"] == "kv8":
            kc = binding.quantize_rows(kc, want_codes=True)[1:]
            vc = binding.quantize_rows(vc, want_codes=True)[1:]
        caches.append((kc, vc))
    for k in steps:
        n_k, l_k = tokens[k]
        out = torch.empty((c["layers"], rows, heads, n_k, HEAD_DIM) if layout == "heads" else
                          (c["layers"], rows, n_k, heads, HEAD_DIM), device="cuda", dtype=torch.bfloat16)
        outs.append(out)
    for layer, (kc, vc) in enumerate(caches):
        for i, k in enumerate(steps):
            n_k, l_k = tokens[k]
            o = outs[i][layer] if layout == "heads" else outs[i][layer].transpose(1, 2)
            call = {"step": k, "q": random_rows(gen, rows, heads, n_k, layout), "k": kc, "v": vc, "out": o}
            if c["kind"] == "qkv8":
                call.update(k_new=random_rows(gen, rows, heads, n_k, layout), v_new=random_rows(gen, rows, heads, n_k, layout),
                            q_dq=empty_rows(rows, heads, n_k, layout), k_at=kc[:, :, l_k - n_k:l_k], v_at=vc[:, :, l_k - n_k:l_k])
            calls.append(call)
    state = {"case": c, "plan": plan, "calls": calls, "outs": outs, "caches": caches}
    if c["launch"] == "graph":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            issue(state)
        torch.cuda.current_stream().wait_stream(side)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            issue(state)
        state["graph"] = graph
    return state


def issue(state):
    """The calls of one pass, in order, on the current stream."""
    plan, pairs, kind = state["plan"], state["case"]["pairs"], state["case"]["kind"]
    for c in state["calls"]:
        if kind == "attention":
            plan.forward(c["step"], pairs, c["q"], c["k"], c["v"], c["out"])
        elif kind == "kv8":
            (kq, ks, kz), (vq, vs, vz) = c["k"], c["v"]
            plan.forward_kv8(c["step"], pairs, c["q"], kq, ks, kz, vq, vs, vz, c["out"])
        else:
            binding.quantize_rows(c["q"], out=c["q_dq"])
            binding.quantize_rows(c["k_new"], out=c["k_at"])
            binding.quantize_rows(c["v_new"], out=c["v_at"])
            plan.forward(c["step"], pairs, c["q_dq"], c["k"], c["v"], c["out"])


def run(state):
    c = state["case"]
    if c["kind"] == "quantise":
        return binding.quantize_rows(state["x"], c["bits"], out=state["out"], want_codes=True)
    if c["kind"] == "calibrate":
        return binding.calibrate_windows(state["scales"], c["step"], state["maps"], c["r0"], want_ratio=True)
    if "graph" in state:
        state["graph"].replay()
    else:
        issue(state)
    if c["kind"] == "qkv8":
        return {"out": state["outs"], "k_cache": state["caches"][0][0], "v_cache": state["caches"][0][1]}
    return state["outs"]


def tolerance(c):
    if c["kind"] == "quantise":
        return "exact"
    if c["kind"] == "calibrate":
        return {"rel": 1e-6, "max": 1e-5}  # fp32 sums of up to 256 rows in another order, then fp64
    # bf16 probabilities and bf16 results
    return {"rel": 1e-2, "max": 6e-2}
