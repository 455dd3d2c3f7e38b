"""Prefill forwards of many tokens: windows of 128 query rows side by side, packed rows, several forwards per prompt."""
import pytest
import torch

from oracle import cerberus_oracle as orc
from paper_2410_13344_b200 import binding as cb
from paper_2410_13344_b200 import synth
from tests.helpers import close
from tests.test_gpu_model import TOL, Rig

pytestmark = pytest.mark.gpu

SHAPES = {"fp32": synth.tiny_shape("fp32"), "bf16 head_dim 64": synth.tiny_shape("bf16"),
          "bf16 head_dim 128": synth.ModelShape(2, 256, 2, 128, 512, 1024, "bf16")}


# a window edge on both sides; a chunk that ends one token into a window; prompts of unequal length in one forward; a whole
# forward of 16 sequences; two forwards of about equal size (a forward holds 4096 rows)
@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("lens", [(127, 1, 129), (128, 256, 255), (2049,), (1300, 5, 900), tuple(range(131, 147)), (2100, 1999, 40)],
                         ids=lambda l: "-".join(map(str, l[:3])))
def test_prefill_matches_oracle(shape, lens):
    ms = SHAPES[shape]
    B = len(lens)
    rig = Rig(cb, ms, max_batch=B, max_tokens=max(lens) + 16, max_nodes=16)
    prompts = [[int(t) for t in synth.make_prompt(ms.vocab, n, seq=70 + b)] for b, n in enumerate(lens)]
    tok = torch.zeros(B, max(lens), dtype=torch.int32, device="cuda")
    for b, p in enumerate(prompts):
        tok[b, :len(p)] = torch.tensor(p, dtype=torch.int32)
    rig.eng.prefill(tok, list(lens))
    got_len, got_root, h_last = rig.eng.read_state()
    assert rig.eng.device_status() == 0 and list(got_len) == list(lens)
    tol = TOL[ms.dtype]                              # the repository's bound for a small model against the oracle
    for b in {0, B // 2, B - 1}:
        st = orc.prefill(rig.cmodel, rig.sh, prompts[b], lens[b] + 16)
        assert close(h_last[b], st.h_last, 0) < tol
        for l in range(ms.n_layers):
            k, v = rig.eng.gather_kv(b, l, lens[b])
            assert close(k, st.k[l][:lens[b]], 0) < tol and close(v, st.v[l][:lens[b]], 0) < tol, (b, l)
        if ms.dtype == "fp32":
            assert int(got_root[b]) == st.root


def _long_forward(model, sh, tokens):
    """orc.forward_full with the attention's rows in pieces (the whole score matrix of a long prompt takes too much memory)."""
    pos = list(range(len(tokens)))
    x = orc.f64(model["embed"][torch.as_tensor(tokens)])
    kv = []
    for l in range(sh.n_layers):
        q, k, v = orc._qkv(x, model, l, sh, pos)
        kv.append((k, v))
        a = torch.empty_like(q)
        for r in range(0, len(tokens), 2048):
            e = min(r + 2048, len(tokens))
            seen = torch.arange(e)[None, :] <= torch.arange(r, e)[:, None]
            for h in range(sh.n_heads):
                s = (q[r:e, h] @ k[:e, h].T / sh.head_dim ** 0.5).masked_fill(~seen, float("-inf"))
                a[r:e, h] = torch.softmax(s, -1) @ v[:e, h]
        x = orc._post_attention(x, orc.rb(a, sh.act), model, l, sh)
    return orc._final(x, model, sh, want_logits=False)[0], kv


# A CTA of the attention holds the page numbers of 16384 keys; beyond that the keys of a window have to be split, which a launch
# over many windows does not do.
@pytest.mark.parametrize("head_dim,lens", [(64, (16500,)), (128, (16500, 700))])
def test_prompts_longer_than_a_page_list(head_dim, lens):
    ms = synth.ModelShape(2, 256, 4, head_dim, 256, 512, "bf16")
    rig = Rig(cb, ms, max_batch=len(lens), max_tokens=max(lens) + 16, max_nodes=16)
    tok = torch.zeros(len(lens), max(lens), dtype=torch.int32, device="cuda")
    prompts = [synth.make_prompt(ms.vocab, n, seq=77 + b).to(torch.int32) for b, n in enumerate(lens)]
    for b, p in enumerate(prompts):
        tok[b, :lens[b]] = p
    rig.eng.prefill(tok, list(lens))
    got_len, _, h_last = rig.eng.read_state()
    assert rig.eng.device_status() == 0 and list(got_len) == list(lens)
    for b in range(len(lens)):
        hidden, kv = _long_forward(rig.cmodel, rig.sh, [int(t) for t in prompts[b]])
        assert close(h_last[b], hidden[-1], 0) < TOL["bf16"]
        for l in range(ms.n_layers):
            k, v = rig.eng.gather_kv(b, l, lens[b])
            assert close(k, kv[l][0], 0) < TOL["bf16"] and close(v, kv[l][1], 0) < TOL["bf16"], (b, l)
