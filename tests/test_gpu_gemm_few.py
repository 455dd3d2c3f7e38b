"""GEMMs of up to 8 rows (warp MMAs, weights straight from global memory) and what runs in front of and behind them."""
import pytest
import torch

from oracle import cerberus_oracle as orc
from paper_2410_13344_b200 import binding as cb
from paper_2410_13344_b200 import synth
from tests.helpers import close
from tests.test_gpu_model import TOL, Rig

pytestmark = pytest.mark.gpu


# rows: one, an MMA's eight columns less one and exactly, the first one of the next kernel; weight rows: fewer than a tile's 16, one more than
# a whole tile, more tiles than CTAs (296) with a part of a tile last; k: less than a warp's 32, a round (1024) less and more one
# 16-byte load, two rounds and a part, an odd number of rounds
@pytest.mark.parametrize("M", [1, 7, 8, 9])
@pytest.mark.parametrize("N,K", [(5, 8), (17, 1016), (4741, 1032), (256, 2560), (40, 11008)])
def test_gemm_matches_definition(M, N, K):
    X = synth.normal(13, 1, (M, K), 1.0, dtype=torch.bfloat16, device="cuda")
    W = synth.normal(13, 2, (N, K), 0.05, dtype=torch.bfloat16, device="cuda")
    out = cb.gemm(X, W)
    # products of bf16 values are exact in fp32: only the order of the sum differs, K * 2^-24 of its terms' size
    assert close(out, orc.linear(X.cpu(), W.cpu()), 0) < 2e-4


# several tiles per CTA in the QKV and gate-up GEMMs; ... in the O and down GEMMs, where one row's norm still fits the GEMM that
# reads it and two rows' just do, or where it does not; head_dim 64 (RoPE in a kernel of its own)
SHAPES = {"wide": synth.ModelShape(2, 256, 25, 128, 4752, 512, "bf16"), "d 4104": synth.ModelShape(2, 4104, 2, 128, 72, 512, "bf16"),
          "d 4872": synth.ModelShape(2, 4872, 1, 128, 64, 512, "bf16"), "head_dim 64": synth.ModelShape(2, 256, 3, 64, 360, 512, "bf16")}


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("lens", [(1,), (1, 1), (3,), (5, 3), (9,), (2, 13, 1)], ids=lambda l: "-".join(map(str, l)))
def test_forward_matches_oracle(shape, lens):
    ms = SHAPES[shape]
    B = len(lens)
    rig = Rig(cb, ms, max_batch=B, max_tokens=32, max_nodes=16)
    prompts = [[int(t) for t in synth.make_prompt(ms.vocab, n, seq=40 + b)] for b, n in enumerate(lens)]
    tok = torch.zeros(B, max(lens), dtype=torch.int32, device="cuda")
    for b, p in enumerate(prompts):
        tok[b, :len(p)] = torch.tensor(p, dtype=torch.int32)
    rig.eng.prefill(tok, list(lens))
    _, _, h_last = rig.eng.read_state()
    assert rig.eng.device_status() == 0 and rig.eng.last_forward_rows() == sum(lens)
    for b in range(B):
        st = orc.prefill(rig.cmodel, rig.sh, prompts[b], 32)
        assert close(h_last[b], st.h_last, 0) < TOL["bf16"]        # the repository's bound for a small model against the oracle
        for l in range(ms.n_layers):
            k, v = rig.eng.gather_kv(b, l, lens[b])
            assert close(k, st.k[l][:lens[b]], 0) < TOL["bf16"] and close(v, st.v[l][:lens[b]], 0) < TOL["bf16"], (b, l)
