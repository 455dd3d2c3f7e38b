"""The fp32 GEMM for few output tiles: ragged rows, columns and k, one piece of k and several."""
import pytest
import torch

from oracle import cerberus_oracle as orc
from paper_2410_13344_b200 import binding as cb
from paper_2410_13344_b200 import synth
from tests.helpers import close
from tests.test_gpu_kernels import _attention_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (16, 16, 256), (17, 33, 255), (5, 700, 257), (64, 1024, 688), (3, 40, 2050),
                                   (1024, 1184, 64)])      # 296 tiles of 64 x 64: the first size that stays on the large kernel
def test_gemm_matches_definition(M, N, K):
    X = synth.normal(13, 1, (M, K), 1.0, dtype=torch.float32, device="cuda")
    W = synth.normal(13, 2, (N, K), 0.05, dtype=torch.float32, device="cuda")
    # products and sums in fp32: sqrt(K) * 2^-24 of the terms' size
    assert close(cb.gemm(X, W), orc.linear(X.cpu(), W.cpu()), 0) < 1e-5


def test_weights_may_be_what_the_previous_call_wrote():
    X = synth.normal(13, 3, (48, 1 << 16), 1.0, dtype=torch.float32, device="cuda")
    V = synth.normal(13, 4, (256, 1 << 16), 1e-4, dtype=torch.float32, device="cuda")
    Y = synth.normal(13, 5, (16, 256), 1.0, dtype=torch.float32, device="cuda")
    W = cb.gemm(X, V)                                        # a long launch (65536 deep) ...
    out = cb.gemm(Y, W)                                      # ... whose output (0.03 in size) is the next one's weights
    assert close(out, orc.linear(Y.cpu(), W.cpu()), 0) < 1e-5


# Operands that start one, two or three values into a buffer: nothing but 4-byte alignment is asked for.
@pytest.mark.parametrize("M,N,K", [(16, 768, 256), (5, 33, 260), (3, 40, 255), (1024, 1184, 64)])
@pytest.mark.parametrize("dx,dw", [(1, 0), (0, 2), (3, 3)])
def test_gemm_takes_operands_at_any_offset(M, N, K, dx, dw):
    fx = synth.normal(13, 6, (M * K + 4,), 1.0, dtype=torch.float32, device="cuda")
    fw = synth.normal(13, 7, (N * K + 4,), 0.05, dtype=torch.float32, device="cuda")
    X, W = fx[dx:dx + M * K].view(M, K), fw[dw:dw + N * K].view(N, K)
    assert close(cb.gemm(X, W), orc.linear(X.cpu(), W.cpu()), 0) < 1e-5


# The list of a node's live ancestors: words of the bitmask full and cut by the number of live nodes, none but the node itself,
# more ancestors than a round of all warps (a chain), no prefix
@pytest.mark.parametrize("n,depth,n_active,lens", [(1, 1, None, [0, 37]), (64, 6, [64, 63], [16, 0]), (65, 6, [65, 64], [5, 300]), (128, 127, [128, 127], [3, 50]),
                                                   (192, 8, [129, 192], [16, 100]), (192, 191, [192, 1], [0, 7])])
@pytest.mark.parametrize("head_dim", [64, 128])
def test_attention_over_listed_ancestors(n, depth, n_active, lens, head_dim):
    for got_o, got_l, O, l in _attention_case(cb, "fp32", 2, n, 2, head_dim, lens, depth, seed_id=170, n_active=n_active):
        assert close(got_o, O, 0) < 1e-5 and close(got_l, l, 0) < 1e-5


# Forwards whose GEMMs take the norm, RoPE, SwiGLU and the residual add in: rows and columns that leave a tile part empty, k below, at and
# above the one round that the norm inside takes, both head sizes, and matrices off the 16-byte boundaries (separate kernels).  Sums of
# up to 688 terms in fp32, 2^-24 each, through three layers: 1e-5 of states of size one.
@pytest.mark.parametrize("d,heads,head_dim,mlp,n,off", [(256, 4, 64, 688, 16, 0), (256, 2, 128, 360, 17, 0), (248, 3, 64, 88, 33, 0), (264, 1, 128, 96, 1, 0),
                                                        (512, 4, 64, 8, 64, 0), (8, 1, 64, 8, 5, 0), (256, 4, 64, 688, 16, 1)])
def test_forward_with_fused_gemms(d, heads, head_dim, mlp, n, off):
    ms = synth.ModelShape(3, d, heads, head_dim, mlp, 512, "fp32")
    model = synth.make_model(ms, device="cuda", std=0.05)
    cmodel = {k: v.cpu() for k, v in model.items()}
    if off:
        model = {k: torch.cat([v.new_zeros(off), v.flatten()])[off:].view(v.shape) if k[0] == "w" else v for k, v in model.items()}
    eng = cb.Cerberus(ms, model, None, None, [], max_tokens=64, max_batch=2, max_nodes=n)
    prompts = [[int(t) for t in synth.make_prompt(512, k, seq=300 + k)] for k in (19, 6)]
    tok = torch.zeros(2, 19, dtype=torch.int32, device="cuda")
    for b, p in enumerate(prompts):
        tok[b, :len(p)] = torch.tensor(p, dtype=torch.int32)
    eng.prefill(tok, [19, 6])
    tree = synth.random_parent_tree(n, 4, tree_id=9) if n > 1 else synth.single_node_tree()
    tt = torch.stack([synth.make_prompt(512, n, seq=310 + b).to(torch.int32) for b in range(2)]).cuda().contiguous()
    hidden = eng.verify(eng.tree(tree), tt, want_hidden=True)[2]
    sh = orc.Shape(3, d, heads, head_dim, mlp, 512, "fp32")
    for b, p in enumerate(prompts):
        st = orc.prefill(cmodel, sh, p, 64 + n)
        want, _ = orc.verify_tree(cmodel, sh, st, [int(t) for t in tt[b]], tree.parent)
        assert close(hidden[b], want, 0) < 1e-5, b
