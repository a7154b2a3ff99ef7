"""The work a user of this library has it do, as measurable cases.

Every case is one pass through the public entry points of `paper_2505_07239_b200.binding`, both parties, on inputs
that are resident in GPU memory (shares and triples are uniform 64-bit words whatever they stand for, because an
additive share is).  Four kinds:

  ffn       one secret-shared layer: block mask (host bytes, as the public sparsity distribution arrives) ->
            ffn_up -> truncate -> ffn_down -> truncate, with fresh activations, triples and hidden state and the
            weights kept in the context, as a serving loop runs it; optionally under a per-token mask
  gate      the element-wise step between the projections of a gated layer: Beaver product, truncation with a
            dealer's pair, bias
  shuffle   the oblivious shuffle of the activations before a layer and the unshuffle of its result
  static    the allocation-free dense product
"""
import math

import torch

from paper_2505_07239_b200 import binding as cb

_stream = None


def _on_stream():
    """All passes go to one stream of the caller's own, one layer after the other."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return torch.cuda.stream(_stream)


def _ffn(name, tokens, d_model, d_ff, block, active, stacked=1, frac=16, clusters=0, p_token=0.0):
    case = {"kind": "ffn", "tokens": tokens, "d_model": d_model, "d_ff": d_ff, "block": block, "active": active,
            "stacked": stacked, "frac": frac, "clusters": clusters, "p_token": p_token}
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest layer (16 tokens, 3 of 32 blocks): nothing but latency and launches
        _ffn("ffn tiny", 16, 256, 1024, 32, 3, frac=12),
        # a short prompt on a small model: 128 token rows, 10 of 96 blocks
        _ffn("ffn opt125m prompt", 128, 768, 3072, 32, 10, frac=13),
        # one decode step of a batch of 32 sequences: few rows, large weights
        _ffn("ffn opt6.7b decode", 32, 4096, 16384, 32, 41),
        # one decode step of a handful of sequences on a gated layer
        _ffn("ffn llama7b decode", 7, 4096, 11008, 64, 26, stacked=2),
        # prompts of 512 tokens at the sparsity the models are run with (90 %) ...
        _ffn("ffn opt1.3b prompt", 512, 2048, 8192, 32, 26),
        # ... and with every neuron active, the dense layer that the sparse one replaces
        _ffn("ffn opt1.3b dense", 512, 2048, 8192, 32, 256),
        # a prompt on a gated layer with large blocks
        _ffn("ffn llama7b prompt", 256, 4096, 11008, 64, 26, stacked=2),
        # query / key / value and output projections under a head mask (16 heads of 64, half of them active), a
        # prompt whose length is no multiple of anything
        _ffn("qkv 16 heads", 203, 1024, 1024, 64, 8, stacked=3),
        # a batch that mixes four groups of requests with disjoint active blocks: masks differ from token to token
        _ffn("ffn four groups", 512, 2048, 8192, 32, 26, clusters=4, p_token=0.6),
        # ReLU(gate) times up, rescaled, plus bias, on the hidden state of the gated prompt above
        {"name": "gate product", "kind": "gate", "rows": 256, "cols": 1664, "frac": 16},
        # shuffle and unshuffle of the activations of the 512-token prompt
        {"name": "shuffle", "kind": "shuffle", "rows": 512, "cols": 2048},
        # the allocation-free product near its size limit
        {"name": "static product", "kind": "static", "tokens": 24, "inner": 1024, "cols": 480},
    ]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choices(("ffn", "groups", "gate", "shuffle", "static"), (10, 3, 2, 2, 2))[0]
    if kind == "gate":
        return {"kind": "gate", "rows": _log_int(rng, 1, 512), "cols": 16 * _log_int(rng, 1, 512),
                "frac": rng.choice((12, 13, 16))}
    if kind == "shuffle":
        return {"kind": "shuffle", "rows": _log_int(rng, 16, 4096), "cols": _log_int(rng, 64, 4096)}
    if kind == "static":
        tokens, inner = _log_int(rng, 1, 256), 8 * _log_int(rng, 4, 128)
        most = cb.STATIC_SCRATCH_WORDS // 2 // inner - tokens
        return {"kind": "static", "tokens": tokens, "inner": inner, "cols": 4 * max(1, _log_int(rng, 4, max(4, most // 4)))}
    while True:
        block = rng.choice((16, 32, 32, 64, 128))
        d_model = 16 * _log_int(rng, 16, 256)
        blocks = max(2, int(d_model * rng.uniform(1.0, 4.0)) // block)
        active = min(blocks, max(1, _log_int(rng, max(1, blocks // 20), blocks)))
        stacked = rng.choices((1, 2, 3), (5, 3, 1))[0]
        tokens = _log_int(rng, 40, 512) if kind == "groups" else _log_int(rng, 1, 512)
        clusters = rng.randint(1, 16) if kind == "groups" else 0
        case = _ffn(None, tokens, d_model, block * blocks, block, active, stacked, rng.choice((12, 13, 16)), clusters,
                    round(rng.uniform(0.1, 0.9), 2) if clusters else 0.0)
        largest, mine = work(_ffn(None, 512, 2048, 8192, 32, 256)), work(case)
        # every word of the weights is kept, whether active or not: no more of those than the decode step has
        if (mine["bytes"] <= largest["bytes"] and mine["flops"] <= largest["flops"]
                and (stacked + 1) * d_model * block * blocks <= 2 * 4096 * 16384):
            return case


class _Source:
    """Uniform words, permutations and masks, all from one seed."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)

    def words(self, *shape):
        return torch.randint(-(1 << 63), (1 << 63) - 1, shape, dtype=torch.int64, device="cuda", generator=self.gen)

    def pair(self, *shape):
        return [self.words(*shape) for _ in (0, 1)]

    def permutation(self, n):
        return torch.randperm(n, device="cuda", generator=self.gen)

    def uniform(self, *shape):
        return torch.rand(shape, device="cuda", generator=self.gen)


def _token_mask(src, tokens, blocks, clusters, p_token):
    """Tokens and blocks dealt to `clusters` groups of requests; inside a group a token uses a block with
    probability p_token, and every token has a block and every block a token where its group allows it."""
    tc = src.permutation(tokens) % clusters
    bc = src.permutation(blocks) % clusters
    same = tc[:, None] == bc[None, :]
    u = torch.where(same, src.uniform(tokens, blocks), torch.ones((), device="cuda"))
    mask = u < p_token
    mask.scatter_(1, u.argmin(dim=1, keepdim=True), True)
    mask.scatter_(0, u.argmin(dim=0, keepdim=True), True)
    return (mask & same).to(torch.uint8).contiguous()


def prepare(case, seed):
    src = _Source(seed)
    kind = case["kind"]
    if kind == "gate":
        rows, cols = case["rows"], case["cols"]
        state = {k: src.pair(rows, cols) for k in ("gate", "up", "a", "b", "c", "r", "rp")}
        return dict(state, kind=kind, bias=src.pair(cols), frac=case["frac"])
    if kind == "shuffle":
        rows, cols = case["rows"], case["cols"]
        pi, tau = src.permutation(rows), [src.permutation(rows) for _ in (0, 1)]
        rho = [torch.argsort(tau[1])[pi], torch.argsort(tau[0])[pi]]       # pi = rho_0 o tau_1 = rho_1 o tau_0
        state = {k: src.pair(rows, cols) for k in ("x", "a", "b", "y", "a2", "b2")}
        return dict(state, kind=kind, tau=[t.int() for t in tau], rho=[r.int() for r in rho])
    if kind == "static":
        T, K, N = case["tokens"], case["inner"], case["cols"]
        return {"kind": kind, "X": src.pair(T, K), "A": src.pair(T, K), "Y": src.pair(N, K), "B": src.pair(N, K),
                "C": src.pair(T, N), "Z": [torch.empty((T, N), dtype=torch.int64, device="cuda") for _ in (0, 1)]}
    T, d, D, g = case["tokens"], case["d_model"], case["d_ff"], case["stacked"]
    n = case["active"] * case["block"]
    blocks = D // case["block"]
    with _on_stream():
        ctx = cb.Comet(T, d, D, case["block"], case["frac"], g - 1, torch.cuda.current_device(), n, stream=_stream)
    # the weights live as long as the context: bound once
    weights = {k: src.pair(D, d) for k in ((cb.W1, cb.WG, cb.W3)[:g] if g > 1 else (cb.W1,))}
    weights[cb.W2] = src.pair(d, D)
    torch.cuda.synchronize()
    for tid, shares in weights.items():
        for p in (0, 1):
            ctx.bind_shares(p, tid, shares[p])
    mask = torch.zeros(blocks, dtype=torch.uint8, device="cuda")
    mask[src.permutation(blocks)[:case["active"]]] = 1
    # what is known before the layer starts, and the hidden state that the activation step hands back
    first = {cb.X: src.pair(T, d), cb.A_UP: src.pair(T, d), cb.B_UP: src.pair(g * n, d), cb.C_UP: src.pair(T, g * n),
             cb.A_DN: src.pair(T, n), cb.B_DN: src.pair(d, n), cb.C_DN: src.pair(T, d)}
    state = {"kind": kind, "tokens": T, "ctx": ctx, "weights": weights, "first": first, "hidden": src.pair(T, n),
             "mask": mask.cpu().numpy(), "token_mask": None, "out": {}}
    if case["clusters"]:
        state["token_mask"] = _token_mask(src, T, case["active"], case["clusters"], case["p_token"])
    for name, tid, shape in (("up", cb.Z_UP, (T, g * n)), ("down", cb.Y, (T, d))):
        for p in (0, 1):
            view = ctx.result_view(p, tid, shape)
            view.context = ctx                        # the buffer is the context's: keep it as long as the view
            state["out"][f"{name}{p}"] = view
    return state


def _run_ffn(s):
    ctx, tokens = s["ctx"], s["tokens"]
    ctx.set_mask(s["mask"])
    if s["token_mask"] is not None:
        ctx.set_token_mask(s["token_mask"])
    for tid, shares in s["first"].items():
        ctx.bind_shares(0, tid, shares[0])
        ctx.bind_shares(1, tid, shares[1])
    ctx.ffn_up(tokens)
    ctx.truncate(cb.Z_UP)
    ctx.bind_shares(0, cb.H, s["hidden"][0])
    ctx.bind_shares(1, cb.H, s["hidden"][1])
    ctx.ffn_down(tokens)
    ctx.truncate(cb.Y)
    return s["out"]


def run(state):
    kind = state["kind"]
    with _on_stream():
        if kind == "ffn":
            return _run_ffn(state)
        if kind == "gate":
            d, e, z = cb.beaver_mul(state["gate"], state["up"], state["a"], state["b"], state["c"], stream=_stream)
            m = cb.truncate_pair(z, state["r"], state["rp"], state["frac"], stream=_stream)
            cb.add_bias(z, state["bias"], stream=_stream)
            return {"d": d, "e": e, "m": m, "z": z}
        if kind == "shuffle":
            sent, shuffled = cb.shuffle(state["x"], state["tau"], state["rho"], state["a"], state["b"], stream=_stream)
            tau = [cb.invert_permutation(p, stream=_stream) for p in state["rho"]]
            rho = [cb.invert_permutation(p, stream=_stream) for p in state["tau"]]
            back, plain = cb.shuffle(state["y"], tau, rho, state["a2"], state["b2"], stream=_stream)
            return {"sent": sent, "shuffled": shuffled, "back": back, "plain": plain}
        code = cb.beaver_matmul_static(state["X"], state["A"], state["Y"], state["B"], state["C"], state["Z"],
                                       stream=_stream)
        return {"code": code, "z": state["Z"]}


def work(case):
    """Both parties: every share, triple and mask word read once, every message and result word written once; a
    ring multiply-add counts as two operations."""
    kind = case["kind"]
    if kind == "gate":
        words = case["rows"] * case["cols"]
        # product: five inputs, two messages; pair: two inputs, one message; result
        return {"bytes": 2 * 8 * 11 * words, "flops": 2 * 8 * words}
    if kind == "shuffle":
        # per party and direction: matrix, two masks, message, result; permutations of 4 bytes
        words = case["rows"] * case["cols"]
        return {"bytes": 2 * 2 * (8 * 5 * words + 8 * case["rows"]), "flops": 2 * 2 * 2 * words}
    T = case["tokens"]
    if kind == "static":
        K, N = case["inner"], case["cols"]
        return {"bytes": 2 * 8 * (2 * T * K + 2 * N * K + 2 * T * N), "flops": 2 * 2 * 2 * T * K * N}
    d, n, g = case["d_model"], case["active"] * case["block"], case["stacked"]
    bytes_up = 3 * T * d + 3 * g * n * d + 2 * T * g * n
    bytes_down = 3 * T * n + 3 * n * d + 2 * T * d
    share_up = share_down = 1.0
    if case["clusters"]:
        groups = min(case["clusters"], case["active"], T)
        share_up, share_down = 1.0 / groups, min(1.0, case["p_token"]) / groups
    macs = 2 * T * d * n * (g * share_up + share_down)
    return {"bytes": 2 * 8 * (bytes_up + bytes_down), "flops": 2 * 2 * macs}


def tolerance(case):
    """Ring words: the shares are the same bits in any correct implementation."""
    return "exact"
