"""What the speed of this framework is measured on: decode steps, generations, DS2D rounds and prefills of the models in
``gen.configs``, and the single projections of its kernel-level calls, through the public calls of ``binding``.

A case is a dict of plain values; ``listed()`` names the ones that stand for the framework's use, ``draw()`` gives more
of the same ranges.  Inputs are synthetic and made on the GPU from the seed alone.  All contexts work on one stream that is
not the default one (steps are replayed from CUDA graphs there), as the benchmark does it.

The language models are random except for what a trained one would also show: its greedy token is decided by a clear
margin.  The lm_head column of token ``follow[t]`` is the (scaled) embedding of ``t``, so the token after ``t`` is
``follow[t]``, whatever the order in which an implementation adds up its sums; drafts can be planted and are accepted.
Logits carry everything else that the pass computed (attention over prompt and own rows, adapters, every layer)."""
import functools
import math

import numpy as np
import torch

import gen
from paper_2604_18655_b200 import binding as mb

MODELS = {"tiny": gen.CFG0, "1b": gen.CFG1, "3b": gen.CFG3}


# ----------------------------------------------------------------------------- the cases
def listed():
    return [
        # one decoder layer, hidden states in and out, four streams: the smallest call, all launch latency
        {"name": "tiny_step", "kind": "step_h", "model": "tiny", "streams": 4, "prompt": 128, "rank": 8},
        # one user, the host picks the token itself: one step, logits wanted
        {"name": "1b_step_1", "kind": "step", "model": "1b", "streams": 1, "prompt": 300, "rank": 16},
        # the benchmark's workload: eight streams with an adapter each over one prompt, tokens fed back on the device
        {"name": "1b_generate_8", "kind": "generate", "model": "1b", "streams": 8, "prompt": 512, "rank": 16, "steps": 32},
        # the larger model behind a long shared prompt
        {"name": "3b_generate_8", "kind": "generate", "model": "3b", "streams": 8, "prompt": 2048, "rank": 32, "steps": 8},
        # DS2D rounds with host-made drafts: 16-node trees (128 rows), 32-node trees of the larger model (256 rows)
        {"name": "1b_verify_8x16", "kind": "verify", "model": "1b", "streams": 8, "prompt": 512, "rank": 16, "nodes": 16, "fan": 3},
        {"name": "3b_verify_8x32", "kind": "verify", "model": "3b", "streams": 8, "prompt": 2048, "rank": 32, "nodes": 32, "fan": 4},
        # DS2D rounds drafted on the device: (3,2) trees with two forecast rows under every token, 30 rows a stream
        {"name": "1b_draft_8x30", "kind": "draft", "model": "1b", "streams": 8, "prompt": 512, "rank": 16, "branch": "3,2"},
        # the shared prompt: the benchmark's, and a long one of ragged length on the larger model
        {"name": "1b_prefill_512", "kind": "prefill", "model": "1b", "streams": 8, "prompt": 512, "rank": 16},
        {"name": "3b_prefill_1999", "kind": "prefill", "model": "3b", "streams": 8, "prompt": 1999, "rank": 32},
        # the projection as a call of its own: a decode step's rows, and a batch of rows with adapters picked per row
        {"name": "linear_8", "kind": "linear", "K": 4096, "N": 14336, "rows": 8, "adapters": 8, "rank": 16},
        {"name": "linear_250", "kind": "linear", "K": 14336, "N": 4096, "rows": 250, "adapters": 8, "rank": 16},
        # per-channel INT4 weights x per-tensor INT8 activations (quantised on the way in)
        {"name": "w4a8_8", "kind": "w4a8", "K": 4096, "N": 4096, "rows": 8},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step_h", "step", "generate", "generate", "verify", "verify", "draft", "prefill", "prefill", "linear",
                       "linear", "w4a8"])
    if kind == "w4a8":
        return {"kind": kind, "K": 256 * _log(rng, 4, 56), "N": 16 * _log(rng, 64, 896), "rows": _log(rng, 1, 64)}
    if kind == "linear":
        ad = rng.choice([0, _log(rng, 1, 64)])
        return {"kind": kind, "K": 128 * _log(rng, 8, 112), "N": 16 * _log(rng, 64, 896), "rows": _log(rng, 1, 256), "adapters": ad,
                "rank": rng.choice([8, 16, 32, 64]) if ad else 0}
    if kind == "step_h":
        return {"kind": kind, "model": "tiny", "streams": rng.randint(1, 8), "prompt": _log(rng, 16, 512), "rank": rng.choice([4, 8, 16])}
    model = rng.choice(["1b", "1b", "3b"])
    c = {"kind": kind, "model": model, "streams": rng.randint(1, 8), "prompt": _log(rng, 16, 2048), "rank": rng.choice([8, 16, 32])}
    if kind == "generate":
        c["steps"] = _log(rng, 4, 48 if model == "1b" else 12)
    elif kind == "verify":
        c["nodes"], c["fan"] = _log(rng, 3, 64), rng.randint(1, 4)
    elif kind == "draft":
        c["branch"] = rng.choice(["3,2", "2,2", "4,1", "3", "4", "2,1,1"])
    return c


# ----------------------------------------------------------------------------- inputs
def _gen(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + what)
    return g


def _quantise(w, group):
    """fp32 [K][N] -> the canonical format: nibbles uint8 [K][N/2], scales fp16 [K/group][N] (as gen.quantize_int4)."""
    K, N = w.shape
    wg = w.view(K // group, group, N)
    scale = (wg.abs().amax(dim=1) / 7.0).half()
    scale = torch.where(scale == 0, torch.ones_like(scale), scale)
    q = (wg / scale.float()[:, None, :]).round_().clamp_(-8, 7).add_(8).to(torch.uint8).view(K, N)
    return (q[:, 0::2] | (q[:, 1::2] << 4)).contiguous(), scale.contiguous()


@functools.lru_cache(maxsize=None)
def _stream():
    return torch.cuda.Stream()


class Model:
    """A context with its adapters, prompt and everything that has to stay alive with it."""

    def __init__(self, case, seed, max_suffix, max_tree, prefill=True):
        cfg = MODELS[case["model"]]
        self.cfg, self.ctx, n = cfg, None, case["streams"]
        g = _gen(seed, 1)
        qw, sc = [], []
        for _ in range(cfg.n_layers):
            for p in gen.PROJ_NAMES:
                a, b = _quantise(torch.randn(gen.proj_shape(cfg, p), generator=g, device="cuda") * cfg.w_std, cfg.group_size)
                qw.append(a)
                sc.append(b)
        gains = [(1 + 0.02 * torch.randn(cfg.d_model, generator=g, device="cuda")).half() for _ in range(2 * cfg.n_layers + 1)]
        self.keep, self.embed, self.follow, embed, final = [gains], None, None, None, None
        if cfg.vocab:
            embed = torch.randn(cfg.vocab, cfg.d_model, generator=g, device="cuda").half()
            follow = torch.randperm(cfg.vocab, generator=g, device="cuda")
            head = torch.empty(cfg.vocab, cfg.d_model, device="cuda")
            head[follow] = embed.float() * cfg.w_std
            a, b = _quantise(head.t().contiguous(), cfg.group_size)
            qw.append(a)
            sc.append(b)
            final = gains[-1]
            self.embed, self.follow = embed, follow.cpu().numpy().astype(np.int32)
        torch.cuda.synchronize()
        self.stream = _stream()
        with torch.cuda.stream(self.stream):
            self.ctx = mb.mlora_create(cfg, qw, sc, gains[0:-1:2], gains[1:-1:2], final, embed, max_adapters=n, max_streams=n,
                                       max_prefix=case["prompt"], max_suffix=max_suffix, max_tree=max_tree, lora_rank=case["rank"])
        shapes = [gen.proj_shape(cfg, p) for p in gen.PROJ_NAMES]
        for s in range(n):
            r = case["rank"]
            A, B = [], []
            for _ in range(cfg.n_layers):
                for p, (K, N) in zip(gen.PROJ_NAMES, shapes):
                    on = bool(cfg.lora_targets & gen.PROJ_BITS[p])
                    A.append((torch.randn(r, K, generator=g, device="cuda") / r).half() if on else None)
                    B.append((torch.randn(r, N, generator=g, device="cuda") * cfg.b_std).half() if on else None)
            self.keep.append((A, B))
            torch.cuda.synchronize()
            mb.mlora_set_adapter(self.ctx, s, A, B, cfg.alpha)
        self.adapter_idx = torch.arange(n, dtype=torch.int32, device="cuda")
        if cfg.vocab:
            self.prompt = torch.randint(0, cfg.vocab, (case["prompt"],), generator=g, device="cuda", dtype=torch.int32)
            self.first = torch.randperm(cfg.vocab, generator=g, device="cuda")[:n].to(torch.int32)
            self.last_logits = torch.empty(cfg.vocab, device="cuda")
        else:
            self.prompt = torch.randn(case["prompt"], cfg.d_model, generator=g, device="cuda").half()
        torch.cuda.synchronize()
        if prefill and cfg.vocab:
            mb.mlora_prefill_shared(self.ctx, self.prompt, None)
        elif prefill:
            mb.mlora_prefill_shared_h(self.ctx, self.prompt, None)
        torch.cuda.synchronize()

    def __del__(self):
        if self.ctx is not None:
            mb.mlora_destroy(self.ctx)
            self.ctx = None

    def logits(self, rows):
        return torch.empty(rows, self.cfg.vocab, device="cuda")


def _ints(*shape):
    return torch.zeros(*shape, dtype=torch.int32, device="cuda")


def _planted_trees(model, parent, n, rounds, seed):
    """Draft trees of `rounds` successive rounds: a node's first child carries the greedy continuation six times in ten,
    every other node a random token; a round's root is the token that the round before it ends with."""
    rng = np.random.default_rng(seed)
    T, root, out = len(parent), model.first.cpu().numpy(), []
    for _ in range(rounds):
        tok = rng.integers(0, model.cfg.vocab, size=(n, T), dtype=np.int32)
        tok[:, 0] = root
        end = root.copy()
        for s in range(n):
            at, seen = 0, set()
            for i in range(1, T):
                p = int(parent[i])
                if p not in seen and rng.random() < 0.6:
                    tok[s, i] = model.follow[tok[s, p]]
                seen.add(p)
            for i in range(1, T):
                if parent[i] == at and tok[s, i] == model.follow[tok[s, at]]:
                    at = i
            end[s] = model.follow[tok[s, at]]
        out.append(torch.from_numpy(tok).cuda())
        root = end
    return out


def _prepare_linear(case, seed):
    K, N, M, r = case["K"], case["N"], case["rows"], case["rank"]
    g = _gen(seed, 2)
    s = {"case": case}
    qw, sc = _quantise(torch.randn(K, N, generator=g, device="cuda") * 0.02, 128)
    s["w"] = Weight(mb.mlora_weight_create(qw, sc, K, N, 128))
    s["x"] = torch.randn(M, K, generator=g, device="cuda").half()
    s["y"] = torch.empty(M, N, device="cuda")
    s["ws"] = torch.zeros(mb.mlora_linear_workspace_bytes(s["w"].w, M, max(r, 1)), dtype=torch.uint8, device="cuda")
    s["lora"] = ()
    if case["adapters"]:
        n = case["adapters"]
        A = (torch.randn(n, r, K, generator=g, device="cuda") / r).half()
        B = (torch.randn(n, r, N, generator=g, device="cuda") * 0.01).half()
        rows = torch.randint(0, n, (M,), generator=g, device="cuda", dtype=torch.int32)
        ptr = [torch.tensor([t[i].data_ptr() for i in range(n)], dtype=torch.int64, device="cuda") for t in (A, B)]
        s["keep"] = (A, B)
        s["lora"] = (rows, ptr[0], ptr[1], torch.full((n,), 16.0 / r, device="cuda"), r)
    return s


class Weight:
    def __init__(self, w):
        self.w = w

    def __del__(self):
        mb.mlora_weight_destroy(self.w)


def _prepare_w4a8(case, seed):
    K, N, M = case["K"], case["N"], case["rows"]
    g = _gen(seed, 3)
    w = torch.randn(N, K, generator=g, device="cuda") * 0.02
    scale = (w.abs().amax(dim=1) / 7.0).half()
    q = (w / scale.float()[:, None]).round_().clamp_(-8, 7).add_(8).to(torch.uint8)
    x = torch.randn(M, K, generator=g, device="cuda").half()
    return {"case": case, "qw": (q[:, 0::2] | (q[:, 1::2] << 4)).contiguous(), "ws": scale, "x": x, "x_scale": float(x.float().abs().max()) / 127.0,
            "qx": torch.empty(M, K, dtype=torch.int8, device="cuda"), "y": torch.empty(M, N, device="cuda")}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "linear":
        return _prepare_linear(case, seed)
    if kind == "w4a8":
        return _prepare_w4a8(case, seed)
    n, s = case["streams"], {"case": case}
    if kind in ("step_h", "step", "generate", "prefill"):
        m = s["m"] = Model(case, seed, case.get("steps", 1) + 1, 1, prefill=kind != "prefill")
        if kind == "step_h":
            s["x"] = torch.randn(n, m.cfg.d_model, generator=_gen(seed, 4), device="cuda").half()
            s["out"] = torch.empty(n, m.cfg.d_model, device="cuda")
        elif kind != "prefill":
            s["tokens"], s["next"], s["logits"] = _ints(case.get("steps", 1), n), _ints(n), m.logits(n)
        return s
    rounds = 2
    if kind == "verify":
        T = case["nodes"]
        parent = np.array([-1] + [(i - 1) // case["fan"] for i in range(1, T)], dtype=np.int32)
    else:
        t = gen.ds2d_template(tuple(int(b) for b in case["branch"].split(",")))
        T, parent = t["R"], t["parent"]
    m = s["m"] = Model(case, seed, rounds * T, T)
    s["parent"] = torch.from_numpy(np.stack([parent] * n)).cuda()
    if kind == "verify":
        s["trees"] = _planted_trees(m, parent, n, rounds, seed)
    else:
        # forecast embedding j: a mix of token embeddings, so that its row's most probable ids are set apart, too
        g = _gen(seed, 5)
        ids = torch.randint(0, m.cfg.vocab, (t["m"], 4), generator=g, device="cuda")
        mix = torch.tensor([1.3, 1.0, 0.7, 0.4], device="cuda")
        s["forecast"] = (m.embed[ids].float() * mix[None, :, None]).sum(dim=1).half().contiguous()
        mb.mlora_set_forecast(m.ctx, s["forecast"])
        s["tpl"] = [torch.from_numpy(t[k]).cuda() for k in ("level", "rank", "forecast_of", "widths")] + [int(t["widths"].max())]
        tree = _planted_trees(m, parent[:t["T"]], n, 1, seed)[0]
        first = _ints(n, T)
        first[:, :t["T"]] = tree
        level = torch.from_numpy(t["level"]).cuda()
        first[:, t["T"]:] = m.cfg.vocab - level[t["T"]:] - 1
        s["trees"] = [first] + [_ints(n, T) for _ in range(rounds)]
    s["acc_len"], s["acc_idx"], s["next"] = [_ints(n) for _ in range(rounds)], [_ints(n, T) for _ in range(rounds)], [_ints(n) for _ in range(rounds)]
    s["logits"] = m.logits(n * T)
    torch.cuda.synchronize()
    return s


# ----------------------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "linear":
        mb.mlora_linear(s["w"].w, s["x"], s["y"], s["ws"], *s["lora"])
        return s["y"]
    if kind == "w4a8":
        mb.mlora_quantize_act_int8(s["x"], s["x_scale"], s["qx"])
        mb.mlora_linear_w4a8(s["qw"], s["ws"], s["qx"], s["x_scale"], s["y"])
        return s["qx"], s["y"]
    m = s["m"]
    if kind == "prefill":
        mb.mlora_prefill_shared(m.ctx, m.prompt, m.last_logits)
        return m.last_logits
    mb.mlora_reset_streams(m.ctx)              # a new request over the same prompt
    if kind == "step_h":
        mb.mlora_decode_step_h(m.ctx, m.adapter_idx, s["x"], s["out"])
        return s["out"]
    if kind == "step":
        mb.mlora_decode_step(m.ctx, m.adapter_idx, m.first, s["next"], s["logits"])
        return s["next"], s["logits"]
    if kind == "generate":                     # the steps, then one more whose distribution the caller looks at
        mb.mlora_generate(m.ctx, m.adapter_idx, m.first, s["tokens"])
        mb.mlora_decode_step(m.ctx, m.adapter_idx, s["tokens"][-1], s["next"], s["logits"])
        return s["tokens"], s["next"], s["logits"]
    rounds = len(s["next"])
    for r in range(rounds):
        lg = s["logits"] if r == rounds - 1 else None
        if kind == "verify":
            if r:                              # the root of a tree is the token that the round before it ends with
                with torch.cuda.stream(m.stream):
                    s["trees"][r][:, 0].copy_(s["next"][r - 1])
            mb.mlora_verify_tree(m.ctx, m.adapter_idx, s["trees"][r], s["parent"], s["acc_len"][r], s["acc_idx"][r], s["next"][r], lg)
        else:
            mb.mlora_ds2d_round(m.ctx, m.adapter_idx, s["trees"][r], s["parent"], *s["tpl"], s["acc_len"][r], s["acc_idx"][r],
                                s["next"][r], s["trees"][r + 1], lg)
    out = {"acc_len": s["acc_len"], "acc_idx": s["acc_idx"], "next": s["next"], "logits": s["logits"]}
    if kind == "draft":
        out["trees"] = s["trees"][1:]
    return out


# ----------------------------------------------------------------------------- what a pass cannot do without
def _pass_work(cfg, rank, rows, streams, context, lm_rows, adapters=True):
    """One pass of `rows` rows through the model: every packed weight, the adapters in use, the K/V that `rows` see (the
    shared part once) and the logits; a pass streams the weights once, a later one has to do so again (they are several
    times what the L2 holds)."""
    by, fl = 0.0, 0.0
    for p in gen.PROJ_NAMES:
        K, N = gen.proj_shape(cfg, p)
        by += K * N / 2 + K // cfg.group_size * N * 2
        fl += 2.0 * rows * K * N
        if adapters and cfg.lora_targets & gen.PROJ_BITS[p]:
            by += streams * rank * (K + N) * 2
            fl += 2.0 * rows * rank * (K + N)
    by += (context + rows) * 2 * cfg.n_kv_heads * cfg.head_dim * 2
    fl += 4.0 * rows * context * cfg.n_q_heads * cfg.head_dim
    by, fl = by * cfg.n_layers, fl * cfg.n_layers
    if cfg.vocab and lm_rows:
        by += cfg.d_model * cfg.vocab / 2 + cfg.d_model // cfg.group_size * cfg.vocab * 2 + lm_rows * cfg.vocab * 4
        fl += 2.0 * lm_rows * cfg.d_model * cfg.vocab
    return np.array([by + rows * cfg.d_model * 2, fl])


def work(case):
    kind = case["kind"]
    if kind in ("linear", "w4a8"):
        K, N, M = case["K"], case["N"], case["rows"]
        by, fl = K * N / 2 + M * N * 4, 2.0 * M * K * N
        if kind == "linear":
            used = min(case["adapters"], M)
            by += K // 128 * N * 2 + M * K * 2 + used * case["rank"] * (K + N) * 2
            fl += 2.0 * M * case["rank"] * (K + N)
        else:
            by += N * 2 + M * K * 3
        return {"bytes": by, "flops": fl}
    cfg, n, P, r = MODELS[case["model"]], case["streams"], case["prompt"], case["rank"]
    if kind == "prefill":
        w = _pass_work(cfg, r, P, n, P / 2, 1, adapters=False)
    elif kind == "generate":
        w = sum(_pass_work(cfg, r, n, n, P + n * j, n) for j in range(case["steps"] + 1))
    elif kind in ("step", "step_h"):
        w = _pass_work(cfg, r, n, n, P, n)
    else:
        T = case["nodes"] if kind == "verify" else gen.ds2d_template(tuple(int(b) for b in case["branch"].split(",")))["R"]
        w = 2 * _pass_work(cfg, r, n * T, n, P, n * T)
    return {"bytes": float(w[0]), "flops": float(w[1])}


def tolerance(case):
    """fp16 activations between the layers, 32-bit sums inside a projection; integers throughout in the INT8 path."""
    kind = case["kind"]
    if kind == "w4a8":
        return "exact"
    if kind == "linear":
        return {"rel": 2e-4}
    if kind == "step_h":
        return {"rel": 2e-3}
    return {"rel": 5e-3, "differ": 0.01}
