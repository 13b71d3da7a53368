"""The work that a program has this library do, as cases that can be timed and compared.

Four calls, each through the package's public entry points:

* ``layer``    one MoE layer by ``MoELayer.forward`` (``dmoe_layer_forward``), launched eagerly:
               a step whose shape changes from call to call, a prompt, a test.
* ``step``     the MoE layers of one decoding step, captured once in a CUDA graph and replayed:
               how a serving loop runs the small steady shapes. Every layer has its own weights
               and its own token rows (what the attention between the layers would hand over).
* ``router``   ``dmoe_router`` alone with every output: routing decisions for a program that
               schedules or counts experts itself.
* ``experts``  ``dmoe_dispatch`` and ``dmoe_moe_forward`` on a routing that the program already
               has (its own router, or a replayed one).

Sizes: d_model ``d``, experts ``E`` of intermediate ``I``, shared expert ``Is`` (0: none), top
``k``, blocks of ``B`` tokens, ``nb`` blocks per forward, coreset threshold ``p`` (0: block
top-k), coreset width ``kb`` (0: k), bias scale ``s`` of the Zipf-like expert popularity.
"""
import math

import torch

import paper_2605_30876_gb300 as dmoe
from paper_2605_30876_gb300.layer import MoELayer

_LAYER = {"call": "layer", "d": 2048, "E": 256, "I": 512, "Is": 512, "k": 8, "kb": 0, "B": 32, "nb": 1,
          "mode": "block", "p": 0.0, "s": 0.5, "layers": 1}


def _case(name, **kw):
    return dict(_LAYER, name=name, **kw)


def listed():
    return [
        # the smallest call there is: a unit test's or a toy model's layer, all latency
        _case("tiny", d=256, E=16, I=128, Is=0, k=2, B=8, nb=2, p=0.6, s=0.0),
        # one user decoding: a block of 32 tokens, block top-k; the benchmark's shape
        _case("step_b1", call="step", layers=8),
        # the same with the paper's middle threshold: a coreset of about 17 experts
        _case("step_b1_p06", call="step", layers=8, p=0.6),
        # token-level routing, the baseline that the paper starts from
        _case("step_b1_token", call="step", layers=4, mode="token"),
        # a few short blocks, not a power of two: 5 users with 12 tokens each
        _case("step_b5x12", call="step", layers=8, B=12, nb=5),
        # 8 users: the middle batch, in both kinds of block routing
        _case("layer_b8", nb=8),
        _case("layer_b8_p06", nb=8, p=0.6),
        # blocks that no tile divides, no shared expert
        _case("layer_b5x60", B=60, nb=5, p=0.5, Is=0),
        # 32 users at the middle threshold: bandwidth and tensor work both count
        _case("layer_b32_p06", nb=32, p=0.6),
        # 64 users, block top-k: the tensor-bound end
        _case("layer_b64", nb=64),
        # 64 users with token routing made elsewhere: all 256 experts, the most weight bytes
        _case("experts_b64_token", call="experts", nb=64, mode="token"),
        # the routing of 64 users alone, with coresets and scores
        _case("router_b64_p06", call="router", nb=64, p=0.6),
    ]


def draw(rng):
    """A case of the same ranges: 4 to 64 tokens a block, up to 2048 tokens a forward (64 in a
    captured step), odd counts among them, every routing option, models of half the width or
    with fewer experts."""
    call = rng.choice(["layer", "layer", "layer", "step", "step", "experts", "router"])
    top = 64 if call == "step" else 2048
    B = rng.choice([4, 8, 16, 32, 64, rng.randint(4, 64), rng.randint(4, 64)])
    T = math.exp(rng.uniform(math.log(B), math.log(top)))
    nb = max(1, min(top // B, round(T / B)))
    k = rng.choice([2, 4, 6, 8, 8])
    mode = rng.choice(["block", "block", "block", "token"])
    p = rng.choice([0.0, 0.0, 0.4, 0.5, 0.6, 0.7, 0.8]) if mode == "block" else 0.0
    return {"call": call, "d": rng.choice([1024, 2048, 2048, 128 * rng.randint(6, 16)]),
            "E": rng.choice([64, 128, 256, 256]), "I": rng.choice([256, 512, 512, 384]),
            "Is": rng.choice([0, 512, 512]), "k": k,
            "kb": 8 if mode == "block" and k < 8 and rng.random() < 0.3 else 0,
            "B": B, "nb": nb, "mode": mode, "p": p, "s": rng.choice([0.0, 0.5, 0.5, 1.0]),
            "layers": rng.randint(2, 6) if call == "step" else 1}


def _inputs(c, seed, layer=0, weights=True, device="cuda"):
    """Token rows N(0, 1) in bf16, expert weights N(0, 0.02^2) in bf16, router weight
    N(0, 1/d) in fp32, bias s ln(1/rank) with the ranks a random order of the experts."""
    g = torch.Generator(device=device)
    g.manual_seed(seed * 1009 + layer)

    def normal(shape, std, dtype=torch.bfloat16):
        return torch.empty(shape, dtype=dtype, device=device).normal_(0.0, std, generator=g)

    d, E, I, Is = c["d"], c["E"], c["I"], c["Is"]
    w = {"x": normal((c["B"] * c["nb"], d), 1.0), "w_r": normal((d, E), d ** -0.5, torch.float32)}
    rank = torch.randperm(E, generator=g, device=device) + 1
    w["bias"] = (-c["s"] * torch.log(rank.double())).float()
    if weights:
        w["w_gate"], w["w_up"] = normal((E, I, d), 0.02), normal((E, I, d), 0.02)
        w["w_down"] = normal((E, d, I), 0.02)
        for key, shape in (("ws_gate", (Is, d)), ("ws_up", (Is, d)), ("ws_down", (d, Is))):
            w[key] = normal(shape, 0.02) if Is else None
    return w


def _desc(c):
    mode = dmoe.DMOE_ROUTE_BLOCK if c["mode"] == "block" else dmoe.DMOE_ROUTE_TOKEN
    return dmoe.make_desc(c["d"], c["E"], c["k"], c["I"], c["Is"], c["B"], c["nb"], mode, c["p"],
                          c["kb"])


def prepare(case, seed):
    c, desc = case, _desc(case)
    T, k, E, nb = c["B"] * c["nb"], c["k"], c["E"], c["nb"]

    def empty(shape, dtype=torch.int32):
        return torch.zeros(shape, dtype=dtype, device="cuda")

    if c["call"] in ("layer", "step"):
        layers, xs = [], []
        for l in range(c["layers"]):
            w = _inputs(c, seed, l)
            xs.append(w.pop("x"))
            layers.append(MoELayer(desc, w))
        state = {"call": c["call"], "layers": layers, "x": xs}
        if c["call"] == "step":
            for layer, x in zip(layers, xs):
                layer.forward(x)
            torch.cuda.synchronize()
            state["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(state["graph"]):
                for layer, x in zip(layers, xs):
                    layer.forward(x)
        return state
    w = _inputs(c, seed, weights=c["call"] == "experts")
    state = {"call": c["call"], "desc": desc, "w": w, "ws": dmoe.alloc_workspace(desc)}
    if c["call"] == "router":
        dmoe.dmoe_router_prepare(desc, w["w_r"], state["ws"])
        state["out"] = {"idx": empty((T, k)), "gate": empty((T, k), torch.float32),
                        "coreset": empty((nb, E)), "size": empty(nb),
                        "probs": empty((T, E), torch.float32)}
    else:
        _, idx, gate, _ = _route(c, w)
        state["idx"], state["gate"] = idx.int().contiguous(), gate.float().contiguous()
        state["out"] = {"n_unique": empty(1), "unique_ids": empty(E), "offsets": empty(E + 1),
                        "rows": empty(T * k), "pos": empty(T * k),
                        "y": empty((T, c["d"]), torch.bfloat16)}
    return state


def run(state):
    call = state["call"]
    if call == "layer":
        layer = state["layers"][0]
        y = layer.forward(state["x"][0])
        return {"y": y, "idx": layer.topk_idx, "gate": layer.topk_gate}
    if call == "step":
        state["graph"].replay()
        return [{"y": l.y, "idx": l.topk_idx, "gate": l.topk_gate} for l in state["layers"]]
    w, o = state["w"], state["out"]
    if call == "router":
        dmoe.dmoe_router(state["desc"], w["x"], w["w_r"], w["bias"], o["idx"], o["gate"],
                         o["coreset"], o["size"], o["probs"], workspace=state["ws"])
        return o
    dmoe.dmoe_dispatch(state["desc"], state["idx"], o["n_unique"], o["unique_ids"], o["offsets"],
                       o["rows"], o["pos"], workspace=state["ws"])
    dmoe.dmoe_moe_forward(state["desc"], w["x"], w["w_gate"], w["w_up"], w["w_down"],
                          w["ws_gate"], w["ws_up"], w["ws_down"], state["gate"], o["n_unique"],
                          o["unique_ids"], o["offsets"], o["rows"], o["pos"], o["y"],
                          workspace=state["ws"])
    return o


def _route(c, w):
    """The routing in 64 bits: scores, experts by descending score (ties: lower id), gates and,
    for block routing, which experts each block's coreset holds."""
    s = torch.softmax(w["x"].double() @ w["w_r"].double() + w["bias"].double(), 1)
    T, E = s.shape
    member = None
    masked = s
    if c["mode"] == "block":
        kb = c["kb"] or c["k"]
        val, idx = torch.sort(s, dim=1, descending=True, stable=True)
        hat = torch.zeros_like(s).scatter(1, idx[:, :kb], val[:, :kb])
        S = hat.view(c["nb"], c["B"], E).sum(1)
        S = S / S.sum(1, keepdim=True)
        val, order = torch.sort(S, dim=1, descending=True, stable=True)
        nnz = (val > 0).sum(1)
        short = (val.cumsum(1) < c["p"]).sum(1) + 1
        size = torch.minimum(short, nnz).clamp(min=kb)
        inside = torch.arange(E, device=s.device)[None] < size[:, None]
        member = torch.zeros_like(inside).scatter(1, order, inside)
        masked = torch.where(member.repeat_interleave(c["B"], 0), s, -1.0)
    val, idx = torch.sort(masked, dim=1, descending=True, stable=True)
    val, idx = val[:, :c["k"]], idx[:, :c["k"]]
    return s, idx, val / val.sum(1, keepdim=True), member


def _ffn(x, gate, up, down):
    g = x @ gate.double().T
    return (g * torch.sigmoid(g) * (x @ up.double().T)) @ down.double().T


def _experts(c, w, idx, gate):
    x = w["x"].double()
    y = _ffn(x, w["ws_gate"], w["ws_up"], w["ws_down"]) if c["Is"] else torch.zeros_like(x)
    for e in torch.unique(idx).tolist():
        t, j = torch.nonzero(idx == e, as_tuple=True)
        y[t] += gate[t, j, None].double() * _ffn(x[t], w["w_gate"][e], w["w_up"][e], w["w_down"][e])
    return y


def exact(case, seed):
    c = case
    if c["call"] == "router":
        w = _inputs(c, seed, weights=False)
        s, _, gate, _ = _route(c, w)
        return {"idx": None, "gate": gate, "coreset": None, "size": None, "probs": s}
    out = []
    for l in range(c["layers"]):
        w = _inputs(c, seed, l)
        _, idx, gate, _ = _route(c, w)
        if c["call"] == "experts":   # on the gates as the program holds them, in fp32
            return {"n_unique": None, "unique_ids": None, "offsets": None, "rows": None,
                    "pos": None, "y": _experts(c, w, idx, gate.float())}
        out.append({"y": _experts(c, w, idx, gate), "idx": None, "gate": gate})
        del w
    return out if c["call"] == "step" else out[0]


def work(case):
    """Each unique expert's weights once (the count that one seed's routing gives), the shared
    expert's, the router weight, the token rows in and out, and the routing out; the products
    of the routed (token, expert) pairs, of the shared expert and of the router."""
    c = case
    T, d, E, k, I, Is = c["B"] * c["nb"], c["d"], c["E"], c["k"], c["I"], c["Is"]
    device = "cuda" if torch.cuda.is_available() else "cpu"
    _, idx, _, _ = _route(c, _inputs(c, 0, weights=False, device=device))
    U = len(torch.unique(idx))
    router = {"bytes": 2 * T * d + 4 * d * E + 4 * E + 8 * T * k, "flops": 2 * T * d * E}
    experts = {"bytes": 6 * d * (U * I + Is) + 4 * T * d, "flops": 6 * T * d * (k * I + Is)}
    if c["call"] == "router":
        extra = 4 * T * E + (4 * c["nb"] * (E + 1) if c["mode"] == "block" else 0)
        return {"bytes": router["bytes"] + extra, "flops": router["flops"]}
    if c["call"] == "experts":
        return {"bytes": experts["bytes"] + 16 * T * k + 8 * E, "flops": experts["flops"]}
    n = c["layers"]
    return {"bytes": n * (router["bytes"] + experts["bytes"] - 2 * T * d),   # x is read once
            "flops": n * (router["flops"] + experts["flops"])}


def tolerance(case):
    """Outputs in bf16 from bf16 inputs: rounding the intermediate, the rows and the result
    leaves a relative error of 2.4e-3 against 64 bits; another order of the sums moves single
    roundings only. Scores and gates in fp32. Two experts whose scores agree to the last bits
    may change places when the logits are summed in another order: single values of the
    selected ids."""
    if case["call"] == "router":
        return {"rel": 2e-6, "differ": 2e-3}
    return {"rel": 1e-2, "differ": 0.0 if case["call"] == "experts" else 2e-3}
