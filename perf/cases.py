"""Cases for timing the framework: what its users run, through the package's public calls.

Serving runs the seven linears of a decoder layer (q, k, v, o, gate, up, down) for one to sixteen tokens of decode
or for the tokens of a prompt; the offline part runs the feedback quantiser with the packer, the Gram matrix of the
calibration activations and the reconstruction step.  Sizes are those of Llama-2-7B and -13B layers, as in the
benchmark, plus prompts of other lengths; ``draw`` spreads widths, tokens, ranks and types over the same ranges.

A 7B layer holds about 100 MB of packed weights, so layers that take turns come from HBM, as in a decoder; weights
are random packed words (every bit of both formats belongs to a code, so random words are random codes).
"""
import math

import torch

import paper_2501_16385_b200 as fbq
from paper_2501_16385_b200.accounting import algorithmic_flops

GROUP = 128
RANKS = (0, 16, 32, 64, 96, 128)


def listed():
    return [
        # One projection, one token, called from Python: the smallest call there is.
        dict(name="one linear, 1 token", kind="single", n=4096, k=4096, tokens=1, bits=4, rank=32, dtype="f16"),
        # The decode step of a 7B layer, one request, linear by linear.
        dict(name="7B layer, 1 token", kind="layer", d=4096, ff=11008, tokens=1, bits=3, rank=64, dtype="f16"),
        # The same for a caller that keeps activations in host memory: pinned x in, y out, result awaited.
        dict(name="7B layer, host buffers", kind="host", d=4096, ff=11008, tokens=1, bits=3, rank=64, dtype="f16"),
        # A few requests; the projections that read the same x go to the library as one batch (q k v, gate up).
        dict(name="7B layer, grouped, 4 tokens", kind="grouped", d=4096, ff=11008, tokens=4, bits=4, rank=64, dtype="bf16"),
        # The largest decode batch, on the wider model.
        dict(name="13B layer, 16 tokens", kind="layer", d=5120, ff=13824, tokens=16, bits=4, rank=64, dtype="f16"),
        # A decode step of the whole 7B linear stack, captured once in a CUDA graph and replayed per step, as servers do.
        dict(name="7B stack, graph, 1 token", kind="stack", layers=32, d=4096, ff=11008, tokens=1, bits=4, rank=64, dtype="f16"),
        dict(name="7B stack, graph, 8 tokens", kind="stack", layers=32, d=4096, ff=11008, tokens=8, bits=4, rank=128, dtype="bf16"),
        # Prompts: a short one of odd length, the usual 1024, a long one on the wider model.
        dict(name="7B prompt, 77 tokens", kind="layer", d=4096, ff=11008, tokens=77, bits=3, rank=128, dtype="f16"),
        dict(name="7B prompt, 1024 tokens", kind="layer", d=4096, ff=11008, tokens=1024, bits=4, rank=64, dtype="bf16"),
        dict(name="13B prompt, 4000 tokens", kind="layer", d=5120, ff=13824, tokens=4000, bits=4, rank=64, dtype="bf16"),
        # Offline: weights minus sub-branch to codes, scales and zero points, and the codes packed.
        dict(name="quantise and pack", kind="quantise", n=4096, k=11008, bits=3, rank=64, dtype="f16"),
        # Offline: the Gram matrix of two calibration sequences, then the step that is iterated on it.
        dict(name="Gram and reconstruction", kind="reconstruct", n=4096, k=4096, t=4096, bits=4, rank=128),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["single", "layer", "layer", "host", "grouped", "stack", "prompt", "prompt", "prompt", "quantise", "reconstruct"])
    bits = rng.choice((3, 4))
    if kind == "quantise":
        return dict(kind=kind, n=_log(rng, 500, 4096), k=GROUP * _log(rng, 6, 86), bits=bits, rank=rng.choice(RANKS), dtype=rng.choice(("f16", "bf16")))
    if kind == "reconstruct":
        return dict(kind=kind, n=_log(rng, 500, 4096), k=GROUP * _log(rng, 6, 32), t=_log(rng, 300, 4096), bits=bits, rank=rng.choice(RANKS[1:]))
    case = dict(bits=bits, rank=rng.choice(RANKS), dtype=rng.choice(("f16", "bf16")))
    if kind == "single":
        return dict(case, kind=kind, n=8 * _log(rng, 64, 2048), k=GROUP * _log(rng, 8, 108), tokens=_log(rng, 1, 16))
    # widths of layers between those of a 1B and a 13B model
    most = 32 if kind == "stack" else 40
    d = GROUP * rng.randint(10, most)
    ff = min(11008 if kind == "stack" else 13824, GROUP * int(round(d * rng.uniform(2.2, 3.6) / GROUP)))
    case = dict(case, d=d, ff=ff)
    if kind == "prompt":
        return dict(case, kind="layer", tokens=_log(rng, 17, 4000))
    if kind == "stack":
        return dict(case, kind=kind, layers=rng.randint(4, 32), tokens=_log(rng, 1, 8))
    return dict(case, kind=kind, tokens=_log(rng, 1, 16))


# ---- the linears ---------------------------------------------------------------------------------------------
def _shapes(case):
    """(K, N) of the linears of one pass, and which of them share an input."""
    if case["kind"] == "single":
        return [(case["k"], case["n"])], [[0]]
    d, ff = case["d"], case["ff"]
    return [(d, d)] * 4 + [(d, ff)] * 2 + [(ff, d)], [[0, 1, 2], [3], [4, 5], [6]]


def _act(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float16


def _weights(case, K, N, g):
    G, r, act = K // GROUP, case["rank"], _act(case)
    words = fbq.packed_words(N, K, case["bits"])
    zeros = torch.randint(6, 10, (N, G), device="cuda", generator=g) if case["bits"] == 4 else torch.randint(2, 6, (N, G), device="cuda", generator=g)
    return (torch.randint(-2**31, 2**31, (words,), dtype=torch.int32, device="cuda", generator=g),
            (torch.rand((N, G), device="cuda", generator=g) * 0.015 + 0.005).half(), zeros.half(),
            (torch.randn((r, K), device="cuda", generator=g) * 0.02).to(act) if r else None,
            (torch.randn((N, r), device="cuda", generator=g) * 0.02).to(act) if r else None)


def _activations(case, K, g):
    """x ~ N(0, 1); prompts carry the outlier channels of real activations (1 % of the channels, 20 times as large)."""
    x = torch.randn((case["tokens"], K), device="cuda", generator=g)
    if case["tokens"] > 16:
        x[:, torch.randperm(K, device="cuda", generator=g)[: max(1, K // 100)]] *= 20.0
    return x.to(_act(case))


def _layer(case, g):
    shapes, shared = _shapes(case)
    xs = [None] * len(shapes)
    for members in shared:
        x = _activations(case, shapes[members[0]][0], g)
        for i in members:
            xs[i] = x
    return [(xs[i], *_weights(case, K, N, g)) for i, (K, N) in enumerate(shapes)]


def _prepare_stack(case, g):
    """The linears of all layers write into one output buffer; the calls of a step are captured once."""
    layers = [_layer(case, g) for _ in range(case["layers"])]
    calls = [(l, N) for layer in layers for l, (K, N) in zip(layer, _shapes(case)[0])]
    out = torch.empty(sum(N for _, N in calls) * case["tokens"], dtype=_act(case), device="cuda")
    ys, at = [], 0
    for _, N in calls:
        ys.append(out[at: at + N * case["tokens"]].view(case["tokens"], N))
        at += N * case["tokens"]

    def step():
        for (l, N), y in zip(calls, ys):
            fbq.linear(*l, N, GROUP, case["bits"], y=y)

    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        step()                                   # the library sizes its scratch for the stream before the capture
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            step()
    torch.cuda.current_stream().wait_stream(stream)
    return dict(graph=graph, out=out, layers=layers, stream=stream)


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kind = case["kind"]
    state = dict(case=case, kind=kind)
    if kind == "quantise":
        N, K, r, act = case["n"], case["k"], case["rank"], _act(case)
        state["W"] = torch.randn((N, K), device="cuda", generator=g) * 0.02
        state["A"] = (torch.randn((r, K), device="cuda", generator=g) * 0.02).to(act) if r else None
        state["B"] = (torch.randn((N, r), device="cuda", generator=g) * 0.02).to(act) if r else None
        return state
    if kind == "reconstruct":
        N, K, T, r = case["n"], case["k"], case["t"], case["rank"]
        loud = 1.0 + 4.0 * (torch.rand(K, device="cuda", generator=g) < 0.05)
        state["X"] = torch.randn((T, K), device="cuda", generator=g) * loud
        state["W"] = torch.randn((N, K), device="cuda", generator=g) * 0.05
        # an iteration past the first: B has left its zero initialisation
        state["A"] = torch.randn((r, K), device="cuda", generator=g) * 0.05
        state["B"] = torch.randn((N, r), device="cuda", generator=g) * 0.01
        # step size 0.2 / (largest eigenvalue of X^T X times |A|^2), from the loud channels and the sizes
        top = 25.0 * (math.sqrt(T) + math.sqrt(0.05 * K)) ** 2
        state["lr"] = 0.2 / (top * (0.05 * (math.sqrt(K) + math.sqrt(r))) ** 2)
        state["workspace"] = state["loss"] = None
        return state
    if kind == "stack":
        state.update(_prepare_stack(case, g))
        return state
    layer = _layer(case, g)
    shapes, shared = _shapes(case)
    state["layer"] = layer
    if kind == "host":
        xs = {}
        for x, *_ in layer:                      # linears that share x share its host buffer
            if id(x) not in xs:
                xs[id(x)] = x.cpu().pin_memory()
        state["ys"] = [torch.empty((case["tokens"], N), dtype=_act(case)).pin_memory() for K, N in shapes]
        state["problems"] = [(xs[id(l[0])], *l[1:], y) for l, y in zip(layer, state["ys"])]
        state["batch"] = fbq.make_batch(state["problems"])
    if kind == "grouped":
        state["ys"] = [torch.empty((case["tokens"], N), dtype=_act(case), device="cuda") for K, N in shapes]
        state["groups"] = []
        for members in shared:
            problems = [(*layer[i], state["ys"][i]) for i in members]
            state["groups"].append((problems, fbq.make_batch(problems)))
    return state


def run(state):
    kind, bits = state["kind"], state["case"]["bits"]
    if kind in ("single", "layer"):
        return [fbq.linear(*l, l[2].shape[0], GROUP, bits) for l in state["layer"]]
    if kind == "grouped":
        for problems, batch in state["groups"]:
            if len(problems) > 1:
                fbq.linear_batch(problems, GROUP, bits, batch=batch)
            else:
                *l, y = problems[0]
                fbq.linear(*l, y.shape[1], GROUP, bits, y=y)
        return state["ys"]
    if kind == "host":
        fbq.linear_batch(state["problems"], GROUP, bits, batch=state["batch"], host_io=True)
        torch.cuda.current_stream().synchronize()            # the caller reads y next
        return state["ys"]
    if kind == "stack":
        state["graph"].replay()
        return state["out"]
    if kind == "quantise":
        codes, scales, zeros, _ = fbq.quantize_feedback(state["W"], state["A"], state["B"], GROUP, bits)
        return [codes, scales, zeros, fbq.pack(codes, bits)]
    H = fbq.gram(state["X"])
    state["loss"], state["workspace"] = fbq.reconstruct_step(state["W"], H, state["A"], state["B"], state["lr"], GROUP, bits,
                                                             workspace=state["workspace"], loss=state["loss"])
    return [H, state["A"], state["B"], state["loss"]]


def work(case):
    kind, bits, r = case["kind"], case["bits"], case["rank"]
    if kind == "quantise":
        N, K = case["n"], case["k"]
        return {"bytes": 4 * N * K + 2 * r * (N + K) + N * K + 4 * N * (K // GROUP) + N * K * bits / 8, "flops": 2 * N * K * r + 8 * N * K}
    if kind == "reconstruct":
        # H is symmetric: half of its products; then B.A, Delta.H and the two gradient products
        N, K, T = case["n"], case["k"], case["t"]
        return {"bytes": 4 * (T * K + 2 * K * K + N * K + 2 * r * (N + K)), "flops": T * K * (K + 1) + 2 * N * K * K + 6 * N * K * r}
    shapes, shared = _shapes(case)
    M, layers = case["tokens"], case.get("layers", 1)
    flops = sum(algorithmic_flops(M, N, K, r) for K, N in shapes)
    weights = sum(N * K * bits // 8 + 4 * N * (K // GROUP) + 2 * r * (K + N) for K, N in shapes)
    moved = sum(2 * M * shapes[members[0]][0] for members in shared) + sum(2 * M * N for K, N in shapes)
    return {"bytes": layers * (weights + moved), "flops": layers * flops}


def tolerance(case):
    if case["kind"] == "quantise":
        return "exact"                           # every code is one fixed sequence of single-precision operations
    if case["kind"] == "reconstruct":
        return {"rel": 1e-5, "max": 2e-3}        # fp32 sums in another order; now and then a code falls on the other side
    # one rounding of y and, in prompts, of the dequantised weights and of t to the activation type
    return {"rel": 1e-2, "max": 4e-2} if case["dtype"] == "bf16" else {"rel": 1.5e-3, "max": 6e-3}
