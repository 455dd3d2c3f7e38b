"""Decoding heads of bf16 models at every batch size class, on the tensor cores."""
import pytest
import torch

from oracle import cerberus_oracle as orc
from paper_2410_13344_b200 import binding as cb
from paper_2410_13344_b200 import synth
from tests.helpers import close
from tests.test_gpu_model import Rig

pytestmark = pytest.mark.gpu


# one column tile, two, three, four (64 weight rows per CTA) and six; widths that are no multiple of a 32-wide k block
# (264, concatenated 528) and shorter than a pass of all warps; a vocabulary that ends inside a CTA's rows
# (and top-k chunks of less than a warp's lanes, of several lists and, at 140000, of more than the 512 entries a warp holds)
@pytest.mark.parametrize("d,vocab", [(264, 1003), (64, 70), (1024, 2048), (64, 140000)])
@pytest.mark.parametrize("B", [1, 2, 3, 5, 8, 9, 13, 16])
def test_draft_logits_match_oracle(B, d, vocab):
    ms = synth.ModelShape(1, d, 2, 64, 128, vocab, "bf16")
    rig = Rig(cb, ms, n_cheads=3, n_levels=3, topk=(5, 3, 2), concat_level=1, max_batch=B, max_tokens=32, max_nodes=16)
    lens = [3 + b % 5 for b in range(B)]
    tok = torch.stack([synth.make_prompt(vocab, 8, seq=50 + b) for b in range(B)]).to(torch.int32).cuda()
    rig.eng.prefill(tok, lens)
    _, roots, h_last = rig.eng.read_state()
    tree = synth.best_first_tree(12, rig.topk)
    tree_tok, topk, logits = rig.eng.draft(rig.eng.tree(tree), want_logits=True)
    for b in range(B):
        want = orc.heads_forward(h_last[b].double(), rig.cheads, rig.csrc)
        for h in range(3):
            # fp32 states, exact products, fp32 sums over at most 2048 terms: 2048 * 2^-24 per level at the worst
            assert close(logits[b, h], want[h], 0) < 2e-4, (b, h)
            ids = [int(t) for t in orc.topk_ids(logits[b, h].cpu().double(), rig.topk[h])]
            assert [int(t) for t in topk[b, h, :rig.topk[h]]] == ids
        assert [int(t) for t in tree_tok[b]] == [int(roots[b])] + [int(topk[b, tree.head[v], tree.rank[v]]) for v in range(1, tree.n)]


# A sum of w products in fp32 is off by about sqrt(w / 2) * 2^-25 at most when every addition rounds (w = 8192: 1.9e-6), and by
# less where partial sums meet in a tree: FMAs with 32 lanes to a row are 1.6e-7 away.  Sums left in the tensor cores,
# which cut off towards zero at every step, are 7e-7 and more away at these widths.
@pytest.mark.parametrize("B", [1, 3, 8, 9, 11, 16])
def test_draft_logits_are_fp32_sums(B):
    ms = synth.ModelShape(1, 4096, 2, 64, 128, 1024, "bf16")
    rig = Rig(cb, ms, n_cheads=2, n_levels=2, topk=(5, 3), concat_level=1, max_batch=B, max_tokens=32, max_nodes=16)
    tok = torch.stack([synth.make_prompt(1024, 8, seq=60 + b) for b in range(B)]).to(torch.int32).cuda()
    rig.eng.prefill(tok, [3 + b % 5 for b in range(B)])
    _, _, h_last = rig.eng.read_state()
    _, _, logits = rig.eng.draft(rig.eng.tree(synth.best_first_tree(12, rig.topk)), want_logits=True)
    for b in {0, B - 1}:
        for h, want in enumerate(orc.heads_forward(h_last[b].double(), rig.cheads, rig.csrc)):
            got, want = logits[b, h].double().cpu(), want.double()
            assert float((got - want).norm() / want.norm()) < 3e-7, (b, h)


@pytest.mark.parametrize("B", [1, 4])
def test_infinite_states_stay_infinite(B):
    """One infinite component in the last hidden state and weights without a sign: every logit is +inf, and the lowest ids win."""
    ms = synth.ModelShape(1, 64, 2, 64, 128, 300, "bf16")
    rig = Rig(cb, ms, n_cheads=2, n_levels=2, topk=(5, 3), concat_level=1, max_batch=B, max_tokens=32, max_nodes=16)
    tok = synth.make_prompt(300, 8, seq=61).to(torch.int32).cuda().repeat(B, 1)
    rig.eng.prefill(tok, [6] * B)
    c = int(torch.argmax(rig.eng.read_state()[2][0].float()))
    rig.model["final_norm"][c] = float("inf")
    for w in rig.heads.values():
        w.copy_(w.abs() + 0.01)
    rig.eng.prefill(tok, [6] * B)
    assert bool(torch.isinf(rig.eng.read_state()[2][:, c]).all())
    _, topk, logits = rig.eng.draft(rig.eng.tree(synth.best_first_tree(12, rig.topk)), want_logits=True)
    assert bool((logits == float("inf")).all())
    for h in range(2):
        assert topk[:, h, :rig.topk[h]].tolist() == [list(range(rig.topk[h]))] * B
