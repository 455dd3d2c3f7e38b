"""The work that is timed: what a program that decodes with this library has it do.

A case is a dict of plain values.  `prepare` makes what such a program has in hand before the call (weights, a loaded
engine, trees, prompts, filled caches), `run` is one pass through the public entry points of
paper_2410_13344_b200.binding, `work` the bytes and operations the pass cannot do without, `tolerance` how far the
results of another correct implementation may lie from these.

Models are random-init LLaMA decoders of the shapes in synth.py, initialised so that they behave like trained ones
where it matters for the path: output projections are scaled by 1/sqrt(2 x layers) (the residual stream grows slowly
with depth), the LM head scores a token's successor clearly above the rest (decisions are not near-ties), the decoding
heads guess the tokens after it correctly about 70 % of the time each (two to three tokens are accepted per drafting
step), and the last hidden state of seven tokens in ten is peaked enough for the gate to choose parallel decoding.
"""
import math

import torch

from paper_2410_13344_b200 import binding, synth

# name: shape, decoding heads, candidates kept per head
MODELS = {
    "7b": (synth.shape_7b(), 4, [10] * 4),
    "13b": (synth.shape_13b(), 5, [10] * 5),
    "tiny fp32": (synth.tiny_shape("fp32"), 4, [4, 2, 1, 1]),
    "tiny bf16": (synth.tiny_shape("bf16"), 4, [4, 2, 1, 1]),
}
N_LEVELS = 4


def listed():
    return [
        # One whole request as a server handles it: prefill, then decoding steps whose tokens are read one by one.
        # The tiny fp32 decoder is the library's smallest configuration: launches and latency.
        dict(name="request tiny fp32", kind="request", model="tiny fp32", batch=1, prompt=64, nodes=16, steps=12),
        # The benchmark's workload: one 7B conversation, 64-node tree, 70 % of the tokens decoded in parallel.
        dict(name="request 7b", kind="request", model="7b", batch=1, prompt=2048, nodes=64, steps=48),
        # A small batch on the larger model; prompts of unequal length, sequences gated separately (ragged rows).
        dict(name="request 13b x4", kind="request", model="13b", batch=4, prompt=1500, nodes=64, steps=12),
        # Prefill until the first token is known: one long prompt, and a batch of short ragged ones.
        dict(name="prefill 7b 2048", kind="prefill", model="7b", batch=1, prompt=2048),
        dict(name="prefill 7b x8 ragged", kind="prefill", model="7b", batch=8, prompt=437),
        # Tree verification alone, from one auto-regressive row to 2048 rows.
        dict(name="verify 7b one node", kind="verify", model="7b", batch=1, prompt=1000, nodes=1),
        dict(name="verify 7b 64 nodes", kind="verify", model="7b", batch=1, prompt=2048, nodes=64),
        dict(name="verify 7b x8 32 nodes", kind="verify", model="7b", batch=8, prompt=2000, nodes=32),
        dict(name="verify 7b x16 128 nodes", kind="verify", model="7b", batch=16, prompt=512, nodes=128),
        # Drafting for a small batch (batch 1 is part of the requests above).
        dict(name="draft 7b x4", kind="draft", model="7b", batch=4, prompt=40, nodes=64),
        # The attention kernel as a building block of another program: one 7B layer.
        dict(name="attention 64 nodes 1k", kind="attention", dtype="bf16", batch=1, heads=32, head_dim=128, prefix=1024, nodes=64),
        dict(name="attention x16 16 nodes 8k", kind="attention", dtype="bf16", batch=16, heads=32, head_dim=128, prefix=8192, nodes=16),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["request", "verify", "verify", "prefill", "prefill", "draft", "attention", "attention"])
    if kind == "attention":
        dtype = rng.choice(["bf16", "bf16", "bf16", "bf16", "fp32"])
        batch = log_int(1, 16)
        c = dict(kind=kind, dtype=dtype, batch=batch, heads=rng.choice([4, 32, 32, 40]), head_dim=rng.choice([64, 128, 128]),
                 prefix=log_int(16, 8192 if batch <= 8 else 4096), nodes=log_int(1, 192))
        if dtype == "fp32":
            c.update(batch=min(batch, 2), prefix=min(c["prefix"], 300 + c["prefix"] % 700), nodes=min(c["nodes"], 64), heads=4)
        return c
    model = rng.choice(["7b", "7b", "7b", "7b", "13b", "tiny fp32", "tiny bf16"])
    batch = log_int(1, 16) if kind != "request" else log_int(1, 4)
    c = dict(kind=kind, model=model, batch=batch)
    if model.startswith("tiny"):
        c["prompt"] = log_int(8, 256)
        if kind != "prefill":
            c["nodes"] = log_int(2, 20)
    else:
        c["prompt"] = log_int(16, min(4096, 8192 // batch))
        if kind != "prefill":
            c["nodes"] = log_int(2 if kind == "draft" else 1, min(192, 2048 // batch))
        if kind == "draft":
            c["prompt"] = log_int(16, 64)
    if kind == "request":
        c["prompt"] = min(c["prompt"], 1500)
        c["nodes"] = max(2, min(c["nodes"], 151))
        c["steps"] = rng.randint(4, 12)
    return c


def lengths(c):
    """Prompt lengths of the batch: the longest first, the others shorter by odd amounts, down to half of it."""
    p = c["prompt"]
    return [max(1, p - (b * 37) % (p // 2 + 1)) for b in range(c["batch"])]


# ---------------------------------------------------------------------------------------------- inputs


def _model(shape, n_cheads, g):
    dt, dev = shape.torch_dtype, "cuda"
    d, F, V, HD, L = shape.d_model, shape.mlp_dim, shape.vocab, shape.n_heads * shape.head_dim, shape.n_layers

    def normal(size, std, mean=0.0):
        return torch.empty(size, dtype=dt, device=dev).normal_(mean, std, generator=g)

    out_std = 0.02 / math.sqrt(2 * L)
    embed = torch.empty(V, d, dtype=torch.float32, device=dev).normal_(generator=g)
    peaked = (torch.arange(V, device=dev) % 10 < 7).unsqueeze(1)
    spikes = 4.0 * (torch.empty(V, d, device=dev).uniform_(generator=g) < 1 / 16).float()
    embed = torch.where(peaked, spikes, embed)              # unit mean square either way
    m = {"embed": (2.0 * embed).to(dt), "final_norm": normal((d,), 0.1, 1.0), "lm_head": (embed.roll(1, 0) * 0.02).to(dt)}
    for l in range(L):
        m[f"attn_norm.{l}"] = normal((d,), 0.1, 1.0)
        m[f"wqkv.{l}"] = normal((3 * HD, d), 0.02)
        m[f"wo.{l}"] = normal((d, HD), out_std)
        m[f"mlp_norm.{l}"] = normal((d,), 0.1, 1.0)
        m[f"wgu.{l}"] = normal((2 * F, d), 0.02)
        m[f"wd.{l}"] = normal((d, F), out_std)
    layout = synth.cerberus_layout(n_cheads, N_LEVELS)
    widths = layout.widths(d)
    heads = {}
    for h in range(n_cheads):
        for j in range(N_LEVELS):
            w = widths[h][j + 1]
            heads[f"W.{h}.{j}"] = normal((w, w), 0.005)
            heads[f"b.{h}.{j}"] = normal((w,), 0.02)
        fc = normal((V, widths[h][N_LEVELS]), 0.02)
        knows = (torch.empty(V, 1, device=dev).uniform_(generator=g) < 0.7).float()
        fc[:, :d] += (embed.roll(2 + h, 0) * (0.02 * knows)).to(dt)
        heads[f"fc.{h}"] = fc
    return m, layout, heads


def _threshold(shape):
    """Between the entropies of the peaked hidden states (1.3 bits or more below log2 d) and the plain ones (0.5 to 0.95)."""
    return math.log2(shape.d_model) - 1.1


class _State:
    pass


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    s = _State()
    s.case = case
    if case["kind"] == "attention":
        return _prepare_attention(s, case, seed, g)
    shape, n_cheads, topk = MODELS[case["model"]]
    model, layout, heads = _model(shape, n_cheads, g)
    nodes = case.get("nodes", 64)
    grow = 16 + (n_cheads + 1) * case.get("steps", 0)          # tokens a request may add
    s.eng = binding.Cerberus(shape, model, layout, heads, topk, max_tokens=case["prompt"] + grow, max_batch=case["batch"],
                             max_nodes=nodes)
    s.lens = lengths(case)
    s.tokens = torch.randint(0, shape.vocab, (case["batch"], case["prompt"]), dtype=torch.int32, device="cuda", generator=g)
    s.T = _threshold(shape)
    if case["kind"] in ("request", "draft"):
        s.tree = s.eng.tree(synth.best_first_tree(nodes, topk))
    elif case["kind"] == "verify":
        s.tree = s.eng.tree(synth.random_parent_tree(nodes, min(4, nodes), tree_id=seed % 1000, n_heads=n_cheads, kmax=min(topk)))
        s.tree_tok = torch.randint(0, shape.vocab, (case["batch"], nodes), dtype=torch.int32, device="cuda", generator=g)
    if case["kind"] in ("verify", "draft"):
        s.eng.prefill(s.tokens, s.lens)
    return s


def _prepare_attention(s, c, seed, g):
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    B, n, H, Dh = c["batch"], c["nodes"], c["heads"], c["head_dim"]
    s.lens_host = [max(1, c["prefix"] - 7 * b) for b in range(B)]
    s.max_len = max(s.lens_host) + n
    mp = (s.max_len + synth.PAGE - 1) // synth.PAGE

    def normal(size):
        return torch.empty(size, dtype=dt, device="cuda").normal_(generator=g)

    s.q = normal((B, n, H, Dh))
    s.k, s.v = normal((B * mp, H, synth.PAGE, Dh)), normal((B * mp, H, synth.PAGE, Dh))
    s.page_table = torch.randperm(B * mp, generator=g, device="cuda").to(torch.int32).view(B, mp)
    s.lens = torch.tensor(s.lens_host, dtype=torch.int32, device="cuda")
    tree = synth.random_parent_tree(n, 6, tree_id=seed % 1000)
    s.anc = torch.from_numpy(binding.tree_ancestors(tree.parent).view("int64")).cuda()
    _, _, s.scratch = binding.tree_attention(s.q, s.k, s.v, s.page_table, s.lens, s.anc, Dh ** -0.5, s.max_len)
    return s


# ---------------------------------------------------------------------------------------------- one pass


def _cached(eng, spans):
    """Views of the pages that hold the slots begin .. end - 1 of every sequence (the engine's pages lie in order)."""
    out = []
    for b, (begin, end) in enumerate(spans):
        pages = slice(b * eng.max_pages + begin // synth.PAGE, b * eng.max_pages + -(-end // synth.PAGE))
        out += [eng.k_pool[:, pages], eng.v_pool[:, pages]]
    return out


def run(s):
    kind = s.case["kind"]
    if kind == "attention":
        out, lse, _ = binding.tree_attention(s.q, s.k, s.v, s.page_table, s.lens, s.anc, s.q.shape[-1] ** -0.5, s.max_len,
                                             scratch=s.scratch)
        return out, lse
    eng = s.eng
    if kind == "verify":
        outs = eng.verify(s.tree, s.tree_tok, want_logits=True, want_hidden=True)
        return list(outs) + _cached(eng, [(k, k + s.tree.n) for k in s.lens])
    if kind == "draft":
        # (the candidates below the best are picked among near-equal logits; what they are picked from is compared)
        tree_tok, _, logits = eng.draft(s.tree, want_logits=True)
        return tree_tok[:, 0], logits
    eng.prefill(s.tokens, s.lens)
    steps = []
    for _ in range(s.case.get("steps", 0)):
        eng.step(s.tree, s.T)
        torch.cuda.current_stream().synchronize()          # the step's tokens are in the pinned mirrors: send them on
        steps.append((eng.h_mode.clone(), eng.h_n_accept.clone(), eng.h_tokens.clone(), eng.h_S.clone()))
    lens, roots, h_last = eng.read_state()
    outs = [lens, roots, h_last]
    if steps:
        outs += [torch.stack(x) for x in zip(*steps)]
    # the prompt and one token per step are committed for certain; what lies behind the last accepted token is scratch
    return outs + _cached(eng, [(0, (k + len(steps)) // synth.PAGE * synth.PAGE) for k in s.lens])


# ---------------------------------------------------------------------------------------------- bounds


def _forward(shape, rows, kv_read, kv_write, head_rows):
    """(bytes, flops) of one base-model forward: weights once, cached keys and values read and new ones written once,
    `kv_read` being a list of (query rows, keys) per sequence; LM head over head_rows rows."""
    e = 2 if shape.dtype == "bf16" else 4
    d, F, V, HD, L = shape.d_model, shape.mlp_dim, shape.vocab, shape.n_heads * shape.head_dim, shape.n_layers
    per_layer = 4 * HD * d + 3 * F * d
    nbytes = e * (L * per_layer + (V * d if head_rows else 0) + rows * d) + 2 * e * HD * L * (sum(k for _, k in kv_read) + kv_write)
    flops = 2 * (L * per_layer * rows + V * d * head_rows) + 4 * HD * L * sum(q * k for q, k in kv_read)
    return nbytes, flops


def _draft(shape, layout, batch):
    e = 2 if shape.dtype == "bf16" else 4
    widths = layout.widths(shape.d_model)
    n = sum(sum(w * w for w in row[1:]) + shape.vocab * row[-1] for row in widths)
    return e * n, 2 * n * batch


def work(case):
    if case["kind"] == "attention":
        e = 2 if case["dtype"] == "bf16" else 4
        B, n, HD = case["batch"], case["nodes"], case["heads"] * case["head_dim"]
        keys = sum(max(1, case["prefix"] - 7 * b) + n for b in range(B))
        return {"bytes": 2 * e * HD * (keys + B * n) + 4 * B * n * case["heads"], "flops": 4 * HD * n * keys}
    shape, n_cheads, _ = MODELS[case["model"]]
    layout = synth.cerberus_layout(n_cheads, N_LEVELS)
    lens, B, n = lengths(case), case["batch"], case.get("nodes", 0)
    db, df = _draft(shape, layout, B)
    if case["kind"] == "draft":
        return {"bytes": db + 4 * B * n_cheads * shape.vocab, "flops": df}
    if case["kind"] == "verify":
        b, f = _forward(shape, B * n, [(n, k + n) for k in lens], B * n, B * n)
        return {"bytes": b + 4 * B * n * shape.vocab, "flops": f}
    # prefill: a query sees half the prompt on average
    b, f = _forward(shape, sum(lens), [(k, k / 2) for k in lens], sum(lens), B)
    steps = case.get("steps", 0)
    if steps:
        # about half of the steps draft (the rest verify one node), and about two tokens are accepted per step
        rows = (n + 1) / 2
        kv = [(rows, k + steps + n) for k in lens]
        vb, vf = _forward(shape, B * rows, kv, B * rows, B * rows)
        b += steps * (vb + db / 2)
        f += steps * (vf + df / 2)
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times what was measured: attention against float64; the models against themselves with the same
    sequence alone and in a batch (other kernels, row counts and summation orders; 32 and 40 layers of bf16 activations:
    3.9e-3 and 5.2e-3 in the last layer's keys, 1.5e-3 in the drafted logits)."""
    if case["kind"] == "attention":
        return {"rel": 7e-3, "max": 2e-2} if case["dtype"] == "bf16" else {"rel": 1e-5, "max": 1e-4}
    if MODELS[case["model"]][0].dtype == "fp32":
        return {"rel": 1e-5, "max": 1e-4}
    if case["kind"] == "draft":
        return {"rel": 6e-3, "max": 3e-2}
    return {"rel": 2e-2, "max": 0.1}
