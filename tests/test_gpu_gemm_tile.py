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
    (256, 74 * 256, 72),      # every pair has the same number of whole tiles, ragged last k block
    (129, 74 * 256 + 1, 64),  # one k block; a last weight tile of one row
    (300, 37 * 256 + 130, 320),   # a last weight tile that is half empty
    (2047, 2400, 136),        # ragged chunks of rows, ragged last k block
    (513, 50 * 256, 1000),    # more tiles than two per pair
    (1100, 1000, 2048),       # fewer tiles than pairs: several pairs per tile
    (131, 40, 4096),          # one weight tile of 40 rows, sixteen fills
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


# (model, prompt lengths); every epilogue runs above 128 rows: the residual add always, RoPE at head_dim 128, SwiGLU with mlp_dim a
# multiple of 16, as in all of these
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


# The schedules, each named by the plan that has to come out: (rows, columns, k) -> (cut tiles, pairs per tile, fills of an accumulator).
# Every case runs twice: the counters are left as they were found.
@pytest.mark.parametrize("M,N,K,cut,pairs_per_tile,fills", [
    (150, 9728, 2560, True, 1, 3),       # fewer tiles than pairs, cut into shares of about half a tile
    (300, 9728, 2048, True, 1, 3),       # two tiles more than pairs; two chunks of rows
    (513, 6656, 4096, True, 1, 3),       # three chunks, shares a little longer than a tile
    (400, 19024, 2048, True, 1, 2),      # shares first, whole tiles after them
    (256, 2560, 1168, False, 2, 3),      # two pairs per tile, ragged last k block
    (513, 1024, 2560, False, 4, 3),
    (2048, 1376, 264, False, 1, 2),      # one pair per tile, ragged last fill
    (150, 768, 256, False, 1, 1),        # one fill: nothing waits in registers
])
def test_schedules(M, N, K, cut, pairs_per_tile, fills):
    g = cb.gemm_plan(M, N, K)
    assert (g.cut_tiles > 0, g.pairs_per_tile, g.chains, g.halves) == (cut, pairs_per_tile, fills, 1), g
    X = synth.normal(12, 3, (M, K), 1.0, dtype=torch.bfloat16, device="cuda")
    W = synth.normal(12, 4, (N, K), 0.05, dtype=torch.bfloat16, device="cuda")
    first = cb.gemm(X, W)
    out = cb.gemm(X, W)
    rows = torch.unique(torch.cat([torch.arange(0, M, 37), torch.arange(max(0, M - 17), M)]))
    assert close(out[rows.cuda()], orc.linear(X.cpu()[rows], W.cpu()), 0) < 2e-4
    assert close(out.double().sum(0) / M, orc.linear(X.double().mean(0, keepdim=True).cpu(), W.cpu())[0], 0) < 2e-4
    assert torch.equal(first, out)                           # (one order of summation whoever comes first)


# The tensor cores cut a sum off towards zero at every step, about 6.6e-8 of it (2-norm, random signs) per block of 64 k in a chain.
# A chain is at most as long as the even share of a pair when the product is cut over all 74 of them, in pieces of at least 4 blocks.
@pytest.mark.parametrize("M,N,K", [(129, 1000, 1000), (256, 4096, 4096), (300, 5120, 13824), (777, 5120, 13824), (1500, 4096, 11008),
                                   (2048, 4096, 4096)])
def test_chains_of_accumulations_are_short(M, N, K):
    X = synth.normal(12, 5, (M, K), 1.0, dtype=torch.bfloat16, device="cuda")
    W = synth.normal(12, 6, (N, K), 0.02, dtype=torch.bfloat16, device="cuda")
    rows = torch.arange(0, M, max(1, M // 41)).cuda()
    want = X[rows].double() @ W.double().T
    got = cb.gemm(X, W)[rows].double()
    share = max(4.0, -(-N // 512) * -(-K // 64) * -(-M // 256) / 74)
    assert float((got - want).norm() / want.norm()) < 7e-8 * min(share, K / 64)


# Forwards whose GEMMs take the schedules above with an epilogue: (model, prompt length, GEMM, what its plan has to be)
FORWARDS = {
    "gate-up cut, 76 tiles": (synth.ModelShape(1, 2048, 16, 128, 4864, 512, "bf16"), 300, (9728, 2048), lambda g: g.cut_tiles == 76),
    "gate-up cut, 38 tiles": (synth.ModelShape(1, 3072, 2, 128, 4864, 512, "bf16"), 150, (9728, 3072), lambda g: g.cut_tiles == 38),
    "qkv cut": (synth.ModelShape(1, 4096, 26, 128, 64, 512, "bf16"), 256, (9984, 4096), lambda g: g.cut_tiles > 0),
    "qkv cut, 7B width": (synth.ModelShape(1, 4096, 32, 128, 64, 512, "bf16"), 150, (12288, 4096), lambda g: g.cut_tiles > 0),
    "down on 512-row tiles, several pairs each": (synth.ModelShape(1, 2048, 2, 128, 4096, 512, "bf16"), 1100, (2048, 4096),
                                                  lambda g: g.halves == 2 and g.pairs_per_tile > 1),
}


@pytest.mark.parametrize("name", list(FORWARDS))
def test_scheduled_epilogues_match_oracle(name):
    ms, n, (N, K), right = FORWARDS[name]
    assert right(cb.gemm_plan(n, N, K, fused=True)), cb.gemm_plan(n, N, K, fused=True)
    assert n > 256 or not cb.forward_gemm_plan(name.split()[0].rstrip(",").replace("-", "_"), n, N, K).rows_kernel      # (the plan is the one that runs)
    rig = Rig(cb, ms, max_tokens=n + 16, max_nodes=16)
    prompt = [int(t) for t in synth.make_prompt(ms.vocab, n, seq=97)]
    tok = torch.tensor([prompt], dtype=torch.int32, device="cuda")
    st = orc.prefill(rig.cmodel, rig.sh, prompt, n + 16)
    for _ in range(2):
        rig.eng.prefill(tok, [n])
        _, _, h_last = rig.eng.read_state()
        assert rig.eng.device_status() == 0 and rig.eng.last_forward_rows() == n
        assert close(h_last[0], st.h_last, 0) < TOL["bf16"]
        k, v = rig.eng.gather_kv(0, 0, n)
        assert close(k, st.k[0][:n], 0) < TOL["bf16"] and close(v, st.v[0][:n], 0) < TOL["bf16"]
