"""The calls whose speed counts: optimizer steps, steps that refresh their subspaces, and steps on host buffers.

A case is a set of weight matrices with the rank, history length and options of one optimizer state, and the way its
user steps it.  Three kinds of pass:

* ``step``: one ``NGaLore.step`` in the steady state of training (history ring full, subspaces set, no refresh due),
  as a plain call or as the replay of a CUDA graph captured from it.
* ``refresh``: one ``NGaLore.step`` at which the refresh is due (T = 1), i.e. new subspaces from the current gradient
  and then the step.  The columns of a new basis that lie in the noise of a gradient are arbitrary, and Adam's
  moments depend on the basis, so that case steps without history and with eps far above the squared gradients
  (projected gradient descent): its result P P^T G depends on the subspace alone.
* ``host``: one ``NGaLore.step_host``, weights and gradients in pinned host memory.

Gradients have the size that clipping at global norm 1 leaves, a falling spectrum along the projector and noise; they
change from pass to pass.
"""
import math
import re

import torch

from paper_2410_16029_b200.ngalore import NGaLore
from paper_2410_16029_b200.workload import WORKLOADS

SWEEPS = 6          # default sweeps of the refresh's subspace iteration
GRADIENT_BYTES = 8e9  # distinct gradient sets a state may hold


def _decoder(layers, hidden, mlp, vocab, kv):
    h = "%dx%d" % (hidden, hidden)
    block = [h, "%dx%d" % (hidden, kv), "%dx%d" % (hidden, kv), h, "%dx%d" % (hidden, mlp), "%dx%d" % (hidden, mlp),
             "%dx%d" % (mlp, hidden)]
    head = "%dx%d" % (vocab, hidden)
    return "%s %d(%s) %s" % (head, layers, " ".join(block), head)


def _encoder(layers, hidden, ffn):
    h = "%dx%d" % (hidden, hidden)
    return "%d(%s %s %s %s %dx%d %dx%d)" % (layers, h, h, h, h, hidden, ffn, ffn, hidden)


def _case(kind, matrices, r, s, **more):
    case = {"kind": kind, "matrices": matrices, "r": r, "s": s, "projection": "left", "history_bf16": False,
            "moments_bf16": False, "graph": False, "wd": 0.0}
    case.update(more)
    return case


def _named(name, case):
    return dict(case, name=name)


def listed():
    w = WORKLOADS
    m60, m130 = _decoder(8, 512, 1376, 32000, 512), _decoder(12, 768, 2048, 32000, 768)
    m350, m1b = _decoder(24, 1024, 2736, 32000, 1024), _decoder(22, 2048, 5632, 32000, 256)
    base = _encoder(12, 768, 3072)
    return [
        # one matrix, e.g. a single adapted layer: launches and latency
        _named("step-one-matrix", _case("step", "512x1376", w[0].r, w[0].s)),
        # pre-training, from the smallest model to the largest
        _named("step-60m", _case("step", m60, w[1].r, w[1].s)),
        # ... replayed from a CUDA graph, as a launch-bound training loop does
        _named("step-130m-graph", _case("step", m130, w[2].r, w[2].s, graph=True)),
        # ... with the reduced-precision state that makes room for a longer history
        _named("step-350m-bf16-state", _case("step", m350, w[3].r, w[3].s, history_bf16=True, moments_bf16=True)),
        _named("step-1.1b", _case("step", m1b, w[4].r, w[4].s)),
        # fine-tuning at small ranks
        _named("step-encoder-r8", _case("step", base, w[5].r, w[5].s, wd=0.01)),
        _named("step-1.1b-r8", _case("step", m1b, w[7].r, w[7].s)),
        # sizes that are no multiples of any tile, GaLore's short-side projection, weight decay
        _named("step-ragged-short-side", _case("step", _decoder(5, 728, 1976, 30011, 184), 100, 5,
                                               projection="short_side", wd=0.1)),
        # the step at which the subspaces are due, every T = 200 steps of pre-training
        _named("refresh-60m", _case("refresh", m60, w[1].r, 0)),
        _named("refresh-130m", _case("refresh", m130, w[2].r, 0)),
        _named("refresh-1.1b", _case("refresh", m1b, w[4].r, 0)),
        # weights and gradients that live in host memory
        _named("host-60m", _case("host", m60, w[1].r, w[1].s)),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _in_reach(case):
    """No dearer than the listed cases of its kind, and of a size that is quickly made."""
    shapes = _shapes(case["matrices"])
    params = sum(M * N for M, N in shapes)
    low_rank = sum(min(case["r"], M, N) * (max(M, N) if case["projection"] == "short_side" else N) for M, N in shapes)
    if case["kind"] == "refresh":
        return params <= 4e8 and sum(M * N * min(case["r"], M, N) for M, N in shapes) <= 1e11
    if case["kind"] == "host":
        return params <= 5.8e7
    return params <= 1.1e9 and low_rank * (4 * case["s"] + 20) <= 1.6e10


def draw(rng):
    while True:
        kind = rng.choice(["step", "step", "step", "refresh", "refresh", "host"])
        form = rng.choice(["decoder", "decoder", "encoder", "loose"])
        hidden = 8 * _log_int(rng, 16, 256)
        if form == "decoder":
            kv = rng.choice([hidden, max(8, hidden // 32 * 8)])
            matrices = _decoder(_log_int(rng, 1, 24), hidden, 8 * int(hidden * rng.uniform(2.0, 4.0) / 8),
                                _log_int(rng, 500, 50000), kv)
        elif form == "encoder":
            matrices = _encoder(_log_int(rng, 1, 24), hidden, 8 * int(hidden * rng.uniform(2.0, 4.0) / 8))
        else:
            matrices = " ".join("%dx%d" % (_log_int(rng, 64, 6000), 8 * _log_int(rng, 8, 700))
                                for _ in range(_log_int(rng, 1, 12)))
        case = _case(kind, matrices, _log_int(rng, 4, 512), rng.randint(0, 20))
        if rng.random() < 0.7 or kind == "refresh":
            case["r"] = (case["r"] + 3) // 4 * 4  # a rank in earnest is mostly a multiple of four
        case["wd"] = rng.choice([0.0, 0.0, 0.01, 0.1])
        option = rng.choice(["none", "none", "short_side", "history", "moments", "both"])
        if kind == "refresh":
            case["s"], case["wd"] = 0, 0.0
        if option == "short_side":
            case["projection"] = "short_side"
        elif kind != "refresh":
            case["history_bf16"] = option in ("history", "both") and case["s"] > 0
            case["moments_bf16"] = option in ("moments", "both")
        case["graph"] = kind == "step" and rng.random() < 0.3
        if _in_reach(case):
            return case


def _shapes(text):
    for group in re.findall(r"\d+\([^)]*\)", text):
        count, inner = group[:-1].split("(")
        text = text.replace(group, " ".join([inner] * int(count)), 1)
    return [tuple(int(x) for x in t.split("x")) for t in text.split()]


def _views(flat, shapes):
    out, at = [], 0
    for M, N in shapes:
        out.append(flat[at: at + M * N].view(M, N))
        at += M * N
    return out


def _right(case, M, N):
    return case["projection"] == "short_side" and M >= N


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) % (2 ** 63))

    def randn(*size):
        return torch.randn(size, generator=gen, device=dev, dtype=torch.float32)

    shapes = _shapes(case["matrices"])
    total = sum(M * N for M, N in shapes)
    refresh = case["kind"] == "refresh"
    norm = 1.0 / math.sqrt(len(shapes))  # per matrix, of a gradient clipped at global norm 1
    if refresh:
        # u = m / sqrt(v + eps) with v negligible: plain projected gradient descent
        rms = norm / math.sqrt(total / len(shapes))
        opt = NGaLore(shapes, case["r"], 0, 1, lr=1e-2, beta1=0.0, beta2=0.999999, eps=rms * rms,
                      projection=case["projection"])
    else:
        opt = NGaLore(shapes, case["r"], case["s"], 0, lr=1e-3, wd=case["wd"], projection=case["projection"],
                      history_bf16=case["history_bf16"], moments_bf16=case["moments_bf16"])
    W_flat = randn(total).mul_(0.02)
    W = _views(W_flat, shapes)

    # projectors: orthonormal columns, one random basis per distinct shape and signs of each matrix's own
    P = []
    if not refresh:
        bases = {}
        for i, (M, N) in enumerate(shapes):
            rows, rank = (N if _right(case, M, N) else M), min(case["r"], M, N)
            if (rows, rank) not in bases:
                bases[rows, rank] = torch.linalg.qr(randn(rows, rank))[0]
            P.append(bases[rows, rank] * torch.sign(randn(rank) + 1e-6))
            opt.set_subspace(i, P[i])

    sets = max(2, min(case["s"] + 1, int(GRADIENT_BYTES // (2 * total))))
    G_flat = [torch.empty(total, dtype=torch.bfloat16, device=dev) for _ in range(sets)]
    G = [_views(f, shapes) for f in G_flat]
    for views in G:
        for i, (M, N) in enumerate(shapes):
            rank = min(case["r"], M, N)
            q = max(1, min(64, rank // 2 if refresh else rank))
            sigma = torch.arange(1, q + 1, device=dev, dtype=torch.float32) ** (-1.0 if refresh else -0.5)
            sigma /= sigma.norm()
            if refresh:
                # the strongest directions lie well above the noise, so that the part of G that a subspace of r'
                # columns keeps is determined
                A, B = randn(M, q) / math.sqrt(M), randn(N, q) / math.sqrt(N)
                noise = 0.02 * float(q ** -1.0) / (math.sqrt(M) + math.sqrt(N))
            else:
                # a slowly moving subspace: the gradient's strong directions lie in the projector's span
                if _right(case, M, N):
                    A, B = randn(M, q) / math.sqrt(M), P[i][:, :q]
                else:
                    A, B = P[i][:, :q], randn(N, q) / math.sqrt(N)
                noise = 1.0 / math.sqrt(M * N)
            g = (A * (norm * sigma)) @ B.T
            views[i].copy_(g.add_(randn(M, N), alpha=norm * noise))
    state = {"opt": opt, "W": W, "G": G, "W_flat": W_flat, "G_flat": G_flat, "at": 0, "graphs": None,
             "kind": case["kind"]}
    if not refresh:
        for k in range(max(case["s"], sets)):  # fill the history
            opt.step(W, G[k % sets])
    if case["graph"]:
        state["graphs"] = []
        torch.cuda.synchronize()
        for views in G:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                opt.step(W, views)
            state["graphs"].append(graph)
    if case["kind"] == "host":
        host = torch.empty(total, dtype=torch.float32, pin_memory=True)
        host.copy_(W_flat)
        G_host = []
        for f in G_flat:
            G_host.append(torch.empty(total, dtype=torch.bfloat16, pin_memory=True))
            G_host[-1].copy_(f)
        state.update(W_flat=host, W=_views(host, shapes), G=[_views(f, shapes) for f in G_host], G_flat=G_host)
    torch.cuda.synchronize()
    return state


def run(state):
    k = state["at"]
    state["at"] = (k + 1) % len(state["G"])
    if state["graphs"] is not None:
        state["graphs"][k].replay()
    elif state["kind"] == "host":
        state["opt"].step_host(state["W"], state["G"][k])
    else:
        state["opt"].step(state["W"], state["G"][k])
    return state["W_flat"]


def work(case):
    """Weights read and written, gradient read; projector, history and moments read, the new gradient of the history
    and the moments written, each once.  A refresh applies the gradient 2 SWEEPS + 2 times to r' columns and writes
    the projector."""
    n_bytes = n_flops = 0
    for M, N in _shapes(case["matrices"]):
        rank = min(case["r"], M, N)
        right = _right(case, M, N)
        rows, low_rank = (N, M * rank) if right else (M, rank * N)
        s = case["s"]
        n_bytes += 10 * M * N
        n_flops += 4 * M * N * rank
        if case["kind"] == "refresh":
            n_bytes += 4 * rows * rank
            n_flops += (2 * SWEEPS + 2) * 2 * M * N * rank
        else:
            hist = 2 if case["history_bf16"] else 4
            moments = 8 if case["moments_bf16"] else 16
            n_bytes += 2 * rows * rank + (hist * s + moments) * low_rank
            n_flops += (4 * s + 12) * low_rank
    return {"bytes": float(n_bytes), "flops": float(n_flops)}


def tolerance(case):
    """About four times what the weights differ by when the same passes run through the plain kernels (other order of
    all sums, fp32 SIMT products): 2.4e-6 (largest difference 6e-5), with bf16 state 4.9e-5 (2e-3: values next to a
    rounding boundary fall to either side); for a refresh, when the random start is another one: 3e-3 (5e-2)."""
    if case["kind"] == "refresh":
        return {"rel": 1.2e-2, "max": 0.2}
    if case["history_bf16"] or case["moments_bf16"]:
        return {"rel": 2e-4, "max": 8e-3}
    return {"rel": 1e-5, "max": 2.5e-4}
