"""Forwards of 9 to 256 rows whose products arrive as sums of few and of many slots: the kernels that add them up."""
import numpy as np
import pytest
import torch

from oracle import cerberus_oracle as orc
from paper_2410_13344_b200 import synth
from tests.helpers import close

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cb():
    from paper_2410_13344_b200 import binding
    return binding


def _slots(cb, product, M, N, K):
    """Slots that the product leaves in a forward of M rows; 0: its outputs are finished where they are summed."""
    if M > 128 and product == "lm_head":
        return 1
    g = cb.forward_gemm_plan(product, M, N, K)
    if g.rows_kernel:
        return 0 if product == "gate_up" else g.parts
    if M > 128:
        return 0 if product == "gate_up" else 1
    nb = cb.C.c_size_t(0)
    assert cb.lib().cerb_gemm_scratch_bytes(M, N, K, cb.C.byref(nb)) == cb.OK
    return (nb.value - 256) // (4 * M * N)


# Slots of the gate-up product (SwiGLU as a kernel of its own: one, four), of the down product (the norm: one trip to L2 for one to eight, two and more for
# 9 and 16, which only matrices of fewer than 16 rows per SM and part leave; two and four pieces of a row per thread) and of the LM head (one, two, four, eight and more;
# rows of more columns than are on their way at once, and of a length that four does not divide); more rows than SMs (200 and 250).  bf16 storage through one layer: the 2e-2 of every bf16 comparison, with weights of 1 / sqrt(d), so that queries and keys have
# elements of size one: rounding them (2^-9) then moves a score of 128 terms over sqrt(128) by 2^-8 or so, and with it a weight by 0.4 %.
# (With weights of 0.03 at d = 8448 they are 2.8, and scores move by 0.03 x the scores' own spread of 8.)  An argmax is that of the logits.
@pytest.mark.parametrize("d,mlp,vocab,n,slots", [(256, 256, 33000, 9, (1, 1, 1)), (1024, 512, 1000, 33, (4, 2, 4)), (1024, 2304, 1002, 17, (0, 8, 4)),
                                                 (1024, 2560, 1000, 64, (0, 8, 4)), (512, 3584, 520, 17, (0, 8, 2)), (128, 2304, 1000, 17, (0, 9, 1)),
                                                 (128, 4096, 1000, 33, (0, 16, 1)), (2560, 4096, 1000, 17, (0, 8, 10)), (4096, 11008, 1000, 32, (0, 5, 8)),
                                                 (4352, 2304, 1000, 17, (0, 4, 8)), (8448, 2304, 1000, 17, (0, 3, 8)), (8448, 1024, 1000, 17, (0, 2, 8)),
                                                 (256, 256, 1004, 100, (0, 1, 1)), (2048, 5632, 1000, 125, (0, 5, 1))])
def test_forward_over_slots(cb, d, mlp, vocab, n, slots):
    assert (_slots(cb, "gate_up", 2 * n, 2 * mlp, d), _slots(cb, "o_down", 2 * n, d, mlp), _slots(cb, "lm_head", 2 * n, vocab, d)) == slots
    ms = synth.ModelShape(1, d, 4, 128, mlp, vocab, "bf16")
    model = synth.make_model(ms, device="cuda", std=d ** -0.5)
    cmodel = {k: v.cpu() for k, v in model.items()}
    eng = cb.Cerberus(ms, model, None, None, [], max_tokens=64, max_batch=2, max_nodes=n)
    prompts = [[int(t) for t in synth.make_prompt(vocab, k, seq=320 + k)] for k in (19, 6)]
    tok = torch.zeros(2, 19, dtype=torch.int32, device="cuda")
    for b, p in enumerate(prompts):
        tok[b, :len(p)] = torch.tensor(p, dtype=torch.int32)
    eng.prefill(tok, [19, 6])
    tree = synth.random_parent_tree(n, 4, tree_id=9)
    tt = torch.stack([synth.make_prompt(vocab, n, seq=330 + b).to(torch.int32) for b in range(2)]).cuda().contiguous()
    th = eng.tree(tree)
    top, logits, hidden = eng.verify(th, tt, want_hidden=True, want_logits=True)
    assert np.array_equal(top.cpu().numpy(), logits.cpu().numpy().argmax(-1))
    assert torch.equal(eng.verify(th, tt)[0], top)
    sh = orc.Shape(1, d, 4, 128, mlp, vocab, "bf16")
    for b, p in enumerate(prompts):
        st = orc.prefill(cmodel, sh, p, 64 + n)
        want, _ = orc.verify_tree(cmodel, sh, st, [int(t) for t in tt[b]], tree.parent)
        assert close(hidden[b], want, 0) < 2e-2, b
        assert close(logits[b], orc.linear(hidden[b].cpu(), cmodel["lm_head"]), 0) < 1e-4, b
