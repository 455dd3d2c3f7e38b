"""Forwards of 9 to 128 rows whose products arrive as sums of few and of many slots: the kernels that add them up."""
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


def _slots(cb, M, N, K):
    nb = cb.C.c_size_t(0)
    assert cb.lib().cerb_gemm_scratch_bytes(M, N, K, cb.C.byref(nb)) == cb.OK
    return (nb.value - 256) // (4 * M * N)


# Slots of the gate-up product: one trip to L2 (1, 2, 4), more (9, 17).  Slots of the down product: one trip (1, 4, 8), code of their own
# (9, 10, 11), two trips (12, 14), two and four pieces of a row per thread.
# Slots of the LM head: 1, 2, 4 and more; rows of more columns than are on their way at once, and of a length that four does not divide;
# more rows than SMs (those of the last case, 200, leave no slots).  bf16 storage through one layer: the 2e-2 of every bf16 comparison, with weights of 1 / sqrt(d), so that queries and keys have
# elements of size one: rounding them (2^-9) then moves a score of 128 terms over sqrt(128) by 2^-8 or so, and with it a weight by 0.4 %.
# (With weights of 0.03 at d = 8448 they are 2.8, and scores move by 0.03 x the scores' own spread of 8.)  An argmax is that of the logits.
@pytest.mark.parametrize("d,mlp,vocab,n,slots", [(256, 256, 33000, 9, (1, 1, 1)), (1024, 2048, 1000, 17, (4, 8, 4)), (1024, 2304, 1002, 17, (4, 9, 4)),
                                                 (1024, 2560, 1000, 64, (4, 10, 4)), (1024, 2816, 4100, 17, (4, 11, 4)), (1024, 3072, 1000, 33, (4, 12, 4)),
                                                 (512, 3584, 520, 17, (2, 14, 2)), (4352, 2304, 1000, 17, (9, 8, 17)), (8448, 1024, 1000, 17, (17, 4, 33)),
                                                 (256, 256, 1004, 100, None)])
def test_forward_over_slots(cb, d, mlp, vocab, n, slots):
    if slots:
        assert (_slots(cb, 2 * n, 2 * mlp, d), _slots(cb, 2 * n, d, mlp), _slots(cb, 2 * n, vocab, d)) == slots
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
