"""fp32 attention of a forward: committed keys asked for ahead of the kernel in front, in rounds of 32 keys (four per warp), two rounds at a time."""
import numpy as np
import pytest
import torch

from paper_2410_13344_b200 import binding as cb
from paper_2410_13344_b200 import synth
from tests.helpers import close
from tests.test_gpu_model import TOL

pytestmark = pytest.mark.gpu

CHAIN = 6        # nodes of the longest path; the tree's other nodes hang on the root


# up to 1024 (node, head) pairs, 512 at head_dim 128, two rounds in turn; above one
@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("B,n", [(1, CHAIN), (3, 20), (16, 17)])
def test_verified_chain_is_the_prompt_it_spells(B, n, head_dim):
    ms = synth.ModelShape(2, 4 * head_dim, 4, head_dim, 688, 512, "fp32")
    eng = cb.Cerberus(ms, synth.make_model(ms, device="cuda"), max_tokens=160, max_batch=B, max_nodes=32)
    parent = np.zeros(n, np.int32)
    parent[:CHAIN] = np.arange(-1, CHAIN - 1)
    head = np.where(np.arange(n) < CHAIN, np.arange(n) - 1, 0).astype(np.int32)
    th = eng.tree(synth.Tree(parent, head, np.arange(n, dtype=np.int32) - 1))
    g = torch.Generator().manual_seed(3)
    # committed keys at and beside the rounds' edges of a warp's first and second four, and beyond
    edges = [1, 3, 4, 5, 31, 32, 33, 35, 36, 37, 63, 64, 65, 67, 68, 96, 100, 129]
    for i in range(0, len(edges), max(1, B)):
        lens = [edges[(i + b) % len(edges)] for b in range(B)]
        tok = torch.randint(0, ms.vocab, (B, max(lens) + CHAIN), dtype=torch.int32, generator=g)
        tree_tok = torch.randint(0, ms.vocab, (B, n), dtype=torch.int32, generator=g)
        for b, L in enumerate(lens):
            tree_tok[b, :CHAIN] = tok[b, L:L + CHAIN]
        eng.prefill(tok[:, :max(lens)].contiguous().cuda(), lens)
        hidden = eng.verify(th, tree_tok.cuda(), want_hidden=True)[2]
        eng.prefill(tok.cuda(), [L + CHAIN for L in lens])
        h_last = eng.read_state()[2]
        assert close(hidden[:, CHAIN - 1], h_last) < TOL["fp32"], lens
    eng.close()
