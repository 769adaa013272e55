"""The work this library is measured on: what a generator of images by next-scale prediction has it do.

A case is a dict of plain values:
  call       how a step is made: "fused" (amskv_append_attend at every scale and layer), "two" (amskv_append, then
             amskv_attend), "density" (amskv_append, then amskv_attend_density), "host" (amskv_step_host from pinned
             host buffers) or "similarity" (amskv_layer_similarity of every adjacent pair of scales)
  layers, heads, head_dim, rows, sides    the shape; rows = 2 x images under classifier-free guidance
  condensed, local, demanding             the policy; `demanding` is the share of cache-demanding layers
  budget     token budgets instead of whole scales (condensed scales + the last one or two scales, in tokens)
  transient  the last scale is never stored (a cache flag)
  layout     "heads": Q, K, V are [rows, heads, T, D] tensors; "packed": views of the [rows, T, 3, heads, D] result
             of one qkv projection, with the output written as [rows, T, heads, D]
  peaked     logits of several units of spread (Q x 6, K of unit variance) instead of N(0, 1) / 8 everywhere
  graph      the pass is captured once into a CUDA graph and replayed; else the calls are made from Python each time

One pass is a whole generation's worth of calls: every scale in order, every layer at each scale.  All layers have
inputs, outputs and cache regions of their own.  Inputs are seeded normal values.
"""
import math
import weakref

import torch

from paper_2511_16047_b200 import binding as B
from paper_2511_16047_b200 import synth

BASE = {"call": "fused", "layers": 1, "heads": 16, "head_dim": 64, "rows": 2, "sides": "", "condensed": 2, "local": 2,
        "demanding": 0.3, "budget": False, "transient": False, "layout": "heads", "peaked": False, "graph": False}
S256, S512, S1024 = (",".join(str(s) for s in x) for x in (synth.SIDES_256, synth.SIDES_512, synth.SIDES_1024))


def _case(name, **kw):
    return dict(BASE, name=name, **kw)


def listed():
    return [
        # one attention layer for one image, called step by step: latency and launches are all there is
        _case("layer_b1", sides=S256, demanding=0.0),
        # one 256x256 image through a depth-30 model, the whole pass a graph: interactive generation
        _case("d30_b1", layers=30, heads=30, sides=S256, layout="packed", graph=True),
        # eight images through a depth-16 model, called step by step
        _case("d16_b8", layers=16, rows=16, sides=S256, demanding=0.5, layout="packed"),
        # a serving batch of 256 images of the depth-30 shape (three of its layers): the benchmark's shape
        _case("d30_b256", layers=3, heads=30, rows=512, sides=S256, graph=True),
        # one 1024x1024 image, 128-channel heads
        _case("t2i_b1", layers=8, head_dim=128, sides=S1024, condensed=3, demanding=0.4, layout="packed", graph=True),
        # eight of them (four of the layers): the largest attention work
        _case("t2i_b8", layers=4, head_dim=128, rows=16, sides=S1024, condensed=3, demanding=0.4, graph=True),
        # 512x512 images of the depth-36 shape (three layers), peaked logits
        _case("d36_512_b32", layers=3, heads=36, rows=64, sides=S512, layout="packed", peaked=True, graph=True),
        # Algorithms 1 and 2 with capacities counted in tokens, as the paper sets them
        _case("budget_b32", layers=10, heads=30, rows=64, sides=S256, budget=True, graph=True),
        # odd sides, an odd number of heads and of images, a window of three scales, append and attend as two calls
        _case("odd_two_calls", call="two", layers=4, heads=15, rows=74, sides="1,3,5,7,9,11,15,19", condensed=1, local=3,
              demanding=0.5, layout="packed"),
        # attention densities beside the outputs, over every layer and scale: the analysis behind the policy
        _case("density_b16", call="density", layers=4, rows=32, sides=S256, demanding=0.5),
        # inter-scale key similarity of every adjacent pair of scales: the classification of the layers
        _case("similarity_b64", call="similarity", layers=4, heads=30, rows=128, sides=S256),
        # inputs and results in pinned host memory
        _case("host_b4", call="host", layers=4, heads=30, rows=8, sides=S256),
    ]


def _sides(case):
    return [int(s) for s in case["sides"].split(",")]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_sides(rng, last):
    """A schedule from 1 x 1 up to about last x last, growing by a random factor from scale to scale."""
    s, growth = [1], rng.uniform(1.15, 1.8)
    while s[-1] < last and len(s) < 20:
        s.append(min(last, max(s[-1] + 1, int(s[-1] * growth * rng.uniform(0.9, 1.1)))))
    return s


# Bounds of a drawn case, under the largest listed ones: about 20 ms of work at 5 TB/s and 700 TFLOP/s, 16 GB of
# tensors, and 0.5 GB over the host link.
_MAX_SECONDS, _MAX_BYTES, _MAX_HOST_BYTES = 0.02, 16e9, 0.5e9


def draw(rng):
    call = rng.choice(["fused"] * 6 + ["two", "density", "similarity", "host"])
    head_dim = rng.choice([64, 64, 64, 128])
    kind = rng.random()
    if kind < 0.35:
        sides = list(synth.SIDES_256)
    elif kind < 0.5:
        sides = list(synth.SIDES_1024 if head_dim == 128 else synth.SIDES_512)
    else:
        sides = _draw_sides(rng, _log_int(rng, 7, 64 if head_dim == 128 else 40))
    c = dict(BASE, call=call, head_dim=head_dim, sides=",".join(str(s) for s in sides),
             layers=rng.randint(1, 12), heads=rng.choice([8, 12, 15, 16, 20, 24, 25, 30, 36]),
             rows=_log_int(rng, 1, 600), condensed=rng.randint(0, 3), local=rng.randint(1, 3),
             demanding=rng.choice([0.0, 0.25, 0.3, 0.5, 1.0]))
    if call in ("fused", "two"):
        c["layout"] = rng.choice(["heads", "packed"])
        c["budget"] = rng.random() < 0.2
        c["peaked"] = rng.random() < 0.25
        c["graph"] = rng.random() < 0.6
    if call == "fused":
        c["transient"] = rng.random() < 0.2
    while True:
        w, mem = work(c), _state_bytes(c)
        over = max(w["bytes"] / 5e12 / _MAX_SECONDS, w["flops"] / 7e14 / _MAX_SECONDS, mem / _MAX_BYTES,
                   mem / _MAX_HOST_BYTES if call == "host" else 0.0)
        if over <= 1.0:
            return c
        if c["layers"] > 1 and (c["rows"] < 8 or over > 8 or rng.random() < 0.5):
            c["layers"] = max(1, min(c["layers"] - 1, int(c["layers"] / over)))
        else:
            c["rows"] = max(1, min(c["rows"] - 1, int(c["rows"] / over)))


# ---------------------------------------------------------------- descriptors
def _policies(case):
    """Spreads the cache-demanding layers evenly over the model."""
    f, n = case["demanding"], case["layers"]
    steps = [math.floor(f * i + 0.5) for i in range(n + 1)]
    return [(case["condensed"], case["local"], steps[i + 1] > steps[i]) for i in range(n)]


def _desc(case, flags=0):
    sides, policies, budgets = _sides(case), _policies(case), None
    if case["budget"]:
        tok = [s * s for s in sides]
        cds = sum(tok[: case["condensed"]])
        c_min = cds + tok[-2 if len(tok) > 1 else -1]
        budgets = [(c_min + tok[-1] if dem else c_min, cds) for _, _, dem in policies]
    if case["transient"]:
        flags |= B.FLAG_TRANSIENT_LAST_SCALE
    return B.make_desc(case["layers"], case["heads"], case["head_dim"], case["rows"], sides, policies, flags=flags,
                       token_budgets=budgets)


def _state_bytes(case):
    desc, _keep = _desc(case)
    tokens = sum(s * s for s in _sides(case))
    tensors = 4 * case["layers"] * case["rows"] * case["heads"] * tokens * case["head_dim"] * 2
    return tensors + B.amskv_cache_required_bytes(desc)


def work(case):
    """Minimum bytes: Q, K and V of the scale and the older attended K and V read once, the output written once, K and
    V stored once where the policy stores them.  Flops: both products over the attended keys."""
    tok = [s * s for s in _sides(case)]
    per = case["rows"] * case["heads"] * case["head_dim"]
    n_layers = case["layers"]
    if case["call"] == "similarity":
        pairs = sum(a + b for a, b in zip(tok, tok[1:]))
        return {"bytes": 2 * per * pairs * n_layers + 8 * n_layers * (len(tok) - 1), "flops": 12 * per * sum(tok[1:]) * n_layers}
    desc, _keep = _desc(case, B.FLAG_PLAN_ONLY)
    plan = B.amskv_cache_create(desc)
    nbytes = flops = 0
    for layer in range(n_layers):
        for k, t in enumerate(tok):
            keys = sum(n for _, _, n in B.amskv_attended_tokens(plan, layer, k))
            stored = sum(n for _, _, n in B.amskv_append_copies(plan, layer, k))
            nbytes += 2 * per * (2 * t + 2 * keys + 2 * stored)
            flops += 4 * per * t * keys
    B.amskv_cache_destroy(plan)
    if case["call"] == "density":
        nbytes += 8 * case["heads"] * n_layers * len(tok)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times what the outputs are off the same computation in fp64: 2.0e-3 to 2.3e-3 in the 2-norm and 1.1e-2 at
    most at a single value (bf16 outputs, and probabilities rounded to bf16), whatever the shape, policy and inputs.
    Similarity: 1.4e-8 measured (fp32 differences and squares, added in fp64); other orders of fp32 sums reach 1e-7."""
    if case["call"] == "similarity":
        return {"rel": 1e-6, "max": 1e-6}
    return {"rel": 8e-3, "max": 4.5e-2}


# ---------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(shape, std, g):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, std, generator=g)


def _qkv(case, t, g):
    """Q, K, V and out of one scale for all layers, each [layers, rows, heads, T, D]; out last."""
    n, r, h, d = case["layers"], case["rows"], case["heads"], case["head_dim"]
    stds = (6.0, 1.0, 1.0) if case["peaked"] else (0.125, 0.125, 0.125)
    if case["layout"] == "packed":
        x = _normal((n, r, t, 3, h, d), stds[1], g)
        x[:, :, :, 0] *= stds[0] / stds[1]
        out = torch.zeros((n, r, t, h, d), dtype=torch.bfloat16, device="cuda")
        return [x[:, :, :, i].transpose(2, 3) for i in range(3)] + [out.transpose(2, 3)]
    return [_normal((n, r, h, t, d), s, g) for s in stds] + [torch.zeros((n, r, h, t, d), dtype=torch.bfloat16, device="cuda")]


def _smooth_keys(case, sides, g):
    """Keys of every scale: samplings of one smooth random map per (row, head, channel), plus noise of each scale."""
    n, d = case["rows"] * case["heads"], case["head_dim"]
    layers = []
    for _ in range(case["layers"]):
        base = torch.empty((n, d, 4, 4), device="cuda").normal_(0.0, 1.0, generator=g)
        keys = []
        for s in sides:
            x = torch.nn.functional.interpolate(base, size=(s, s), mode="bilinear", align_corners=False)
            x = (0.9 * x + 0.43 * torch.empty_like(x).normal_(0.0, 1.0, generator=g)) * 0.125
            keys.append(x.flatten(2).transpose(1, 2).to(torch.bfloat16).reshape(case["rows"], case["heads"], s * s, d).contiguous())
        layers.append(keys)
    return layers


class State:
    """What the caller keeps between passes."""

    def __init__(self, case):
        self.case, self.sides, self.graph = case, _sides(case), None


def prepare(case, seed):
    g = _generator(seed)
    st = State(case)
    sides = st.sides
    if case["call"] == "similarity":
        st.keys = _smooth_keys(case, sides, g)
        st.workspace = torch.empty(B.amskv_similarity_workspace_bytes(), dtype=torch.uint8, device="cuda")
        st.ss = torch.zeros((case["layers"], len(sides) - 1), dtype=torch.float64, device="cuda")
        return st
    desc, _keep = _desc(case)
    n = B.amskv_cache_required_bytes(desc)
    st.arena = torch.empty(n, dtype=torch.uint8, device="cuda")
    st.cache = B.amskv_cache_create(desc, st.arena, n)
    weakref.finalize(st, B.amskv_cache_destroy, st.cache)
    st.steps, st.outs = [], []
    for s in sides:
        tensors = _qkv(case, s * s, g)
        if case["call"] == "host":
            tensors = [x.cpu().pin_memory() for x in tensors]
        st.steps.append(list(zip(*tensors)))
        st.outs.append(tensors[3])
    if case["call"] == "host":
        size = B.amskv_step_staging_bytes(st.cache)
        st.lanes = [(torch.cuda.Stream(), torch.empty(size, dtype=torch.uint8, device="cuda"), size) for _ in range(2)]
    if case["call"] == "density":
        st.density = []
        for k in range(len(sides)):
            sizes = [case["heads"] * len(B.amskv_attended_tokens(st.cache, layer, k)) for layer in range(case["layers"])]
            flat = torch.zeros(sum(sizes), dtype=torch.float64, device="cuda")
            st.density.append(flat.split(sizes))
            st.outs.append(flat)
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _pass(st, side)   # loads the kernels; nothing may be loaded during the capture
        side.synchronize()
        st.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(st.graph, stream=side):
            _pass(st, side)
    return st


# ---------------------------------------------------------------- one pass
def _pass(st, stream):
    call = st.case["call"]
    B.amskv_cache_reset(st.cache)
    for k, scale in enumerate(st.steps):
        for layer, (q, kk, v, o) in enumerate(scale):
            if call == "fused":
                B.amskv_append_attend(st.cache, layer, k, kk, v, q, o, stream)
            elif call == "two":
                B.amskv_append(st.cache, layer, k, kk, v, stream)
                B.amskv_attend(st.cache, layer, k, q, o, stream)
            elif call == "density":
                B.amskv_append(st.cache, layer, k, kk, v, stream)
                d = st.density[k][layer]
                B.amskv_attend_density(st.cache, layer, k, q, o, d, d.numel(), stream)
            else:
                # layers alternate between two streams with a staging buffer each, so that one layer's results go back
                # while the other's inputs come in; a layer stays on its stream, which keeps its steps in order
                lane, staging, size = st.lanes[layer % 2]
                B.amskv_step_host(st.cache, layer, k, kk, v, q, o, staging, size, lane)


def run(st):
    if st.graph is not None:
        st.graph.replay()
        return st.outs
    if st.case["call"] == "similarity":
        case, stream = st.case, torch.cuda.current_stream()
        for layer, keys in enumerate(st.keys):
            for i in range(1, len(st.sides)):
                B.amskv_layer_similarity(keys[i - 1], st.sides[i - 1], keys[i], st.sides[i], case["rows"], case["heads"],
                                         case["head_dim"], st.ss[layer, i - 1], st.workspace, st.workspace.numel(), stream)
        return st.ss
    _pass(st, torch.cuda.current_stream())
    return st.outs
