"""Host results of a step: the acceptance kernel writes pinned ones, pageable ones are copied; both are what the device tensors hold."""
import ctypes as C

import pytest
import torch

from paper_2410_13344_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n", [(1, 1), (3, 1), (3, 16), (2, 64)])
@pytest.mark.parametrize("kind", ["pinned", "pageable", "pinned count", "pinned tokens", "none"])
def test_step_host_results(kind, B, n):
    from paper_2410_13344_b200 import binding as cb
    ms = synth.tiny_shape("bf16")
    layout = synth.cerberus_layout(4, 2)
    eng = cb.Cerberus(ms, synth.make_model(ms, device="cuda"), layout, synth.make_heads(ms, layout, device="cuda"), [10] * 4,
                      max_tokens=128, max_batch=B, max_nodes=64)
    g = torch.Generator().manual_seed(5)
    lens = [7 + 3 * b for b in range(B)]
    eng.prefill(torch.randint(0, ms.vocab, (B, max(lens)), dtype=torch.int32, generator=g).cuda(), lens)
    th = eng.tree(synth.random_parent_tree(n, 4, tree_id=2) if n > 1 else synth.single_node_tree())

    def words(count, pinned):                       # a word ahead and words behind that nothing writes
        t = torch.full((count + 9,), -77, dtype=torch.int32)
        return t.pin_memory() if pinned else t
    count = words(B, kind in ("pinned", "pinned count"))
    toks = words(B * cb.PATH_MAX, kind in ("pinned", "pinned tokens"))
    o = cb.StepOut(eng.S.data_ptr(), eng.mode.data_ptr(), eng.n_accept.data_ptr(), eng.tokens.data_ptr(), None, None,
                   None if kind == "none" else count.data_ptr() + 4, None if kind == "none" else toks.data_ptr() + 4)
    for T in (-1e9, 1e9, 1e9):
        cb._check(cb.lib().cerb_step(eng.ctx, th.handle, T, None, C.byref(o), cb._stream()), "cerb_step")
        torch.cuda.synchronize()
        dev_n, dev_t = eng.n_accept[:B].cpu(), eng.tokens[:B].reshape(-1).cpu()
        assert int(dev_n.min()) >= 1
        if kind == "none":
            dev_n, dev_t = torch.full_like(dev_n, -77), torch.full_like(dev_t, -77)
        assert torch.equal(count[1:1 + B], dev_n) and torch.equal(toks[1:1 + dev_t.numel()], dev_t)
        for t, m in ((count, B), (toks, dev_t.numel())):
            assert t[0] == -77 and bool((t[1 + m:] == -77).all())
    eng.close()
