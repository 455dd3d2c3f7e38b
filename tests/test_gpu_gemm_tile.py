"""The GEMM of more than 128 rows (output tiles on CTA pairs): whole and split tiles, partial slots, fused epilogues."""
import pytest
import torch

from oracle import cerberus_oracle as orc
from paper_2410_13344_b200 import binding as cb
from paper_2410_13344_b200 import synth
from tests.helpers import close
from tests.test_gpu_model import TOL, Rig

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (256, 74 * 256, 72),      # exactly one whole tile per pair, ragged last k block
    (129, 74 * 256 + 1, 64),  # one k block; one tile more than pairs: 75 tiles cut along k; 160-row chunk
    (300, 37 * 256 + 130, 320),   # two chunks of 160, 76 tiles, the last one half empty
    (2047, 2400, 136),        # eight chunks, 80 tiles
    (513, 50 * 256, 1000),    # three chunks of 192, 150 tiles: whole tiles after the split ones
    (1100, 1000, 2048),       # fewer tiles than pairs: partial slots
    (131, 40, 4096),          # one tile for all pairs
])
def test_gemm_matches_definition(M, N, K):
    X = synth.normal(12, 1, (M, K), 1.0, dtype=torch.bfloat16, device="cuda")
    W = synth.normal(12, 2, (N, K), 0.05, dtype=torch.bfloat16, device="cuda")
    for _ in range(2):                                       # (tickets are left as they were found)
        out = cb.gemm(X, W)
    rows = torch.arange(0, M, max(1, M // 97))
    # products of bf16 values are exact in fp32: only the order of the sum differs, K * 2^-24 of its terms' size
    assert close(out[rows.cuda()], orc.linear(X.cpu()[rows], W.cpu()), 0) < 2e-4
    # ... and every element through its column sums
    assert close(out.double().sum(0) / M, orc.linear(X.double().mean(0, keepdim=True).cpu(), W.cpu())[0], 0) < 2e-4


# which epilogues run depends on how many tiles the matrices have: (model, prompt lengths)
CASES = {
    "rope, swiglu, residual": (synth.ModelShape(2, 2560, 8, 128, 1168, 512, "bf16"), (1900,)),
    "rope, swiglu, residual, two sequences": (synth.ModelShape(1, 2560, 8, 128, 1168, 512, "bf16"), (1500, 431)),
    "rope, swiglu, 160-row chunks": (synth.ModelShape(2, 256, 25, 128, 4752, 512, "bf16"), (170, 129)),
    "swiglu (head_dim 64)": (synth.ModelShape(1, 256, 50, 64, 4752, 512, "bf16"), (300,)),
    "rope": (synth.ModelShape(1, 256, 25, 128, 688, 512, "bf16"), (290,)),
    "norm of 4104 columns": (synth.ModelShape(1, 4104, 2, 128, 64, 512, "bf16"), (140,)),      # beyond four pieces per thread
    "norm of 8200 columns": (synth.ModelShape(1, 8200, 2, 128, 64, 512, "bf16"), (131,)),      # beyond eight
    "residual": (synth.ModelShape(1, 2560, 4, 128, 688, 512, "bf16"), (1800,)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_fused_epilogues_match_oracle(name):
    ms, lens = CASES[name]
    rig = Rig(cb, ms, max_batch=len(lens), max_tokens=max(lens) + 16, max_nodes=16)
    prompts = [[int(t) for t in synth.make_prompt(ms.vocab, n, seq=90 + b)] for b, n in enumerate(lens)]
    tok = torch.zeros(len(lens), max(lens), dtype=torch.int32, device="cuda")
    for b, p in enumerate(prompts):
        tok[b, :len(p)] = torch.tensor(p, dtype=torch.int32)
    rig.eng.prefill(tok, list(lens))
    _, _, h_last = rig.eng.read_state()
    assert rig.eng.device_status() == 0 and rig.eng.last_forward_rows() == sum(lens)
    for b in range(len(lens)):
        st = orc.prefill(rig.cmodel, rig.sh, prompts[b], lens[b] + 16)
        assert close(h_last[b], st.h_last, 0) < TOL["bf16"]
        for l in range(ms.n_layers):
            k, v = rig.eng.gather_kv(b, l, lens[b])
            assert close(k, st.k[l][:lens[b]], 0) < TOL["bf16"] and close(v, st.v[l][:lens[b]], 0) < TOL["bf16"], (b, l)
