"""Attention of 65 to 128 query rows with more (sequence, head) items than CTAs: every CTA takes several in turn."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2410_13344_b200 import binding as cb
from paper_2410_13344_b200 import synth
from tests.helpers import close
from tests.test_gpu_kernels import TOL_BF16, _attention_case

pytestmark = pytest.mark.gpu


# a second round of 12 CTAs; two full rounds and part of a third; prefixes from nothing (fewer keys than one ring, an odd and
# an even number of tiles) to several rings; live rows that leave the second softmax group without a tile
@pytest.mark.parametrize("B,n,H,lens,n_active", [
    (16, 65, 10, [0, 1, 63, 64, 127, 128, 300, 17, 640, 5, 200, 90, 33, 450, 12, 70], None),
    (16, 128, 20, [(37 * b) % 500 for b in range(16)], None),
    (16, 100, 12, [0] * 8 + [700] * 8, [1, 64, 65, 100, 3, 99, 17, 40] * 2),
])
def test_items_match_oracle(B, n, H, lens, n_active):
    for got_o, got_l, O, l in _attention_case(cb, "bf16", B, n, H, 128, lens, 6, seed_id=120 + n, n_active=n_active):
        assert close(got_o, O, 0) < TOL_BF16
        assert close(got_l, l, 0) < 2e-3


# Pointers that are aligned no further than a route asks for: up to 16 rows q to 4 bytes, any route's output to 8.
@pytest.mark.parametrize("B,n,q_off,out_off", [(3, 1, 2, 4), (3, 7, 2, 4), (2, 40, 0, 4), (3, 100, 0, 4), (16, 100, 0, 4), (1, 150, 0, 4)])
def test_offset_pointers_give_the_same_bits(B, n, q_off, out_off):
    H, Dh, L = 12, 128, 200
    pages = (L + n + 15) // 16
    tree = synth.random_parent_tree(n, 5, tree_id=4) if n > 1 else synth.single_node_tree()
    flat = synth.normal(14, 1, (B * n * H * Dh + 8,), 1.0, dtype=torch.bfloat16, device="cuda")
    q = flat[q_off:q_off + B * n * H * Dh].view(B, n, H, Dh)
    kp, vp = (synth.normal(14, i, (B * pages, H, 16, Dh), 1.0, dtype=torch.bfloat16, device="cuda") for i in (2, 3))
    pt = torch.arange(B * pages, dtype=torch.int32, device="cuda").view(B, pages)
    lens = torch.full((B,), L, dtype=torch.int32, device="cuda")
    anc = torch.from_numpy(cb.tree_ancestors(tree.parent).view(np.int64)).cuda()
    want, _, scratch = cb.tree_attention(q.clone(), kp, vp, pt, lens, anc, Dh ** -0.5, L + n)
    out = torch.zeros(B * n * H * Dh + 8, dtype=torch.bfloat16, device="cuda")[out_off:out_off + B * n * H * Dh].view(B, n, H, Dh)
    a = cb.AttnArgs(cb.BF16, B, n, H, Dh, pages, q.data_ptr(), kp.data_ptr(), vp.data_ptr(), pt.data_ptr(), lens.data_ptr(), None, anc.data_ptr(),
                    out.data_ptr(), None, Dh ** -0.5, L + n, B * pages, scratch.data_ptr(), scratch.numel())
    assert cb.lib().cerb_tree_attention(C.byref(a), torch.cuda.current_stream().cuda_stream) == cb.OK
    torch.cuda.synchronize()
    assert torch.equal(out, want)
