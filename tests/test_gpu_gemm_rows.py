"""Gate-up and QKV products of 9 to 256 rows in one tile per SM (or pair of SMs): edges of rows, of weight tiles, of k."""
import ctypes as C

import pytest
import torch

from oracle import cerberus_oracle as orc
from paper_2410_13344_b200 import binding as cb
from paper_2410_13344_b200 import synth
from tests.helpers import close
from tests.test_gpu_model import TOL, Rig

pytestmark = pytest.mark.gpu

# (d_model, heads, mlp_dim): weight rows per SM, k blocks
SHAPES = {
    "16 and 16 rows, one k block": (64, 4, 1184),                # the least of both plans
    "16 and 24 rows, ragged k block": (200, 4, 1192),            # one feature group more than two per SM
    "32 and 152 rows, three MMAs per pair": (1096, 10, 11000),   # odd number of groups; the last tile of SwiGLU half empty; ragged k
    "112 and 168 rows": (1024, 40, 12432),                       # too wide for a pair: above 128 rows gate-up is the output tiles'
    "16 and 144 rows, three MMAs per pair": (1024, 4, 10600),    # the fewest k blocks; an even number of groups
    "16 and 136 rows, three MMAs per pair": (1984, 4, 9504),     # 31 k blocks: the most changes of accumulators; the smallest third MMA
}
# prompt lengths: rows of one accumulator quarter, its edges, all of them; pairs: one row in the second CTA's half and all
CASES = [(n, m) for n in SHAPES for m in (9, 33, 64, 65, 128, 129, 256)]
CASES += [("32 and 152 rows, three MMAs per pair", m) for m in (96, 97, 192, 193)]          # ... and both sides of the other plans' edges


def _prompt_matches_oracle(d, H, F, M):
    ms = synth.ModelShape(1, d, H, 128, F, 512, "bf16")
    rig = Rig(cb, ms, max_tokens=M + 16, max_nodes=16)
    prompt = [int(t) for t in synth.make_prompt(ms.vocab, M, seq=140 + M)]
    tok = torch.tensor([prompt], dtype=torch.int32, device="cuda")
    st = orc.prefill(rig.cmodel, rig.sh, prompt, M + 16)
    for _ in range(2):
        before = rig.eng.launch_count()
        rig.eng.prefill(tok, [M])
        launches = rig.eng.launch_count() - before
        _, _, h_last = rig.eng.read_state()
        assert rig.eng.device_status() == 0 and rig.eng.last_forward_rows() == M
        assert close(h_last[0], st.h_last, 0) < TOL["bf16"]
        k, v = rig.eng.gather_kv(0, 0, M)
        assert close(k, st.k[0][:M], 0) < TOL["bf16"] and close(v, st.v[0][:M], 0) < TOL["bf16"]
    return launches


@pytest.mark.parametrize("name,M", CASES)
def test_prompts_match_oracle(name, M):
    d, H, F = SHAPES[name]
    launches = _prompt_matches_oracle(d, H, F, M)
    # live rows, first norm, seven launches of the layer, commit, LM head, argmax
    if M <= 128:
        assert launches == 1 + 1 + 7 + 3
    # ... of which these are this kernel's
    assert [cb.forward_gemm_plan(p, M, N, d).rows_kernel for p, N in (("gate_up", 2 * F), ("qkv", 384 * H))] == [M <= 128 or F < 12000, M <= 128 or M > 192]


# More accumulators than two per issuer, and numbers of them that the issuers do not divide: (rows, product, issuers, accumulators)
@pytest.mark.parametrize("d,H,F,M,product,issuers,chains", [
    (1024, 8, 2816, 9, "qkv", 3, 6), (1024, 8, 2816, 97, "qkv", 2, 4), (1024, 8, 2816, 256, "qkv", 2, 6), (1536, 12, 4096, 97, "qkv", 2, 6),
    (1024, 8, 2816, 33, "gate_up", 2, 4), (1024, 8, 4096, 128, "gate_up", 3, 6), (2048, 4, 5632, 9, "gate_up", 3, 5), (3584, 4, 9728, 65, "gate_up", 1, 3),
    (1024, 8, 1024, 129, "o_down", 3, 5), (1024, 8, 1024, 250, "o_down", 3, 5), (4096, 32, 1184, 96, "qkv", 3, 4), (1984, 4, 1184, 40, "qkv", 3, 9), (1984, 4, 1184, 200, "qkv", 3, 9),
])
def test_accumulators_in_turn_match_oracle(d, H, F, M, product, issuers, chains):
    N = {"qkv": 384 * H, "gate_up": 2 * F, "o_down": d}[product]
    g = cb.forward_gemm_plan(product, M, N, d)
    assert (g.rows_kernel, g.issuers, g.chains) == (1, issuers, chains), g
    _prompt_matches_oracle(d, H, F, M)


@pytest.mark.parametrize("n,live", [(40, (40, 17, 1)), (70, (1, 70, 33))])
def test_trees_with_dead_nodes_match_oracle(n, live):
    """Three sequences (120 and 210 rows): rows of nodes that are not live write nothing."""
    d, H, F = SHAPES["32 and 152 rows, three MMAs per pair"]
    ms = synth.ModelShape(1, d, H, 128, F, 512, "bf16")
    rig = Rig(cb, ms, max_tokens=128, max_batch=3, max_nodes=n)
    lens = [29, 16, 5]
    prompts = [[int(t) for t in synth.make_prompt(ms.vocab, k, seq=160 + k)] for k in lens]
    tok = torch.zeros(3, max(lens), dtype=torch.int32, device="cuda")
    for b, p in enumerate(prompts):
        tok[b, :len(p)] = torch.tensor(p, dtype=torch.int32)
    rig.eng.prefill(tok, lens)
    tree = synth.random_parent_tree(n, 4, tree_id=6, n_heads=4, kmax=1)
    tt = torch.stack([synth.make_prompt(ms.vocab, n, seq=170 + b).to(torch.int32) for b in range(3)]).cuda().contiguous()
    before = rig.eng.k_pool.clone()
    hidden = rig.eng.verify(rig.eng.tree(tree), tt, n_active=torch.tensor(live, dtype=torch.int32, device="cuda"), want_hidden=True)[2]
    assert rig.eng.device_status() == 0
    for b in range(3):
        st = orc.prefill(rig.cmodel, rig.sh, prompts[b], 200)
        want, _ = orc.verify_tree(rig.cmodel, rig.sh, st, [int(t) for t in tt[b, :live[b]]], tree.parent[:live[b]])
        assert close(hidden[b, :live[b]], want, 0) < TOL["bf16"], b
    # cache slots written: the live nodes' only
    changed = (rig.eng.k_pool != before).any(dim=-1).any(dim=2).sum().item()        # (page, slot) pairs with any head changed
    assert changed <= sum(live)


# residual adds in the products (3, 7) where O and down do not leave parts of k for the norm; SwiGLU a kernel of its own (7) in output tiles of 11000 features
@pytest.mark.parametrize("name,n,B,variant", [("16 and 24 rows, ragged k block", 9, 1, 2), ("16 and 24 rows, ragged k block", 64, 2, 2),
                                              ("16 and 24 rows, ragged k block", 65, 2, 3), ("32 and 152 rows, three MMAs per pair", 65, 2, 2),
                                              ("32 and 152 rows, three MMAs per pair", 128, 2, 2), ("32 and 152 rows, three MMAs per pair", 129, 2, 7)])
def test_launches_of_a_forward_are_the_table(name, n, B, variant):
    d, H, F = SHAPES[name]
    ms = synth.ModelShape(3, d, H, 128, F, 512, "bf16")
    taken = n * B <= 256 and all(cb.forward_gemm_plan("o_down", n * B, d, k).rows_kernel for k in (128 * H, F))
    assert taken == (n * B > 128 and variant == 2)
    rig = Rig(cb, ms, max_tokens=64, max_batch=B, max_nodes=n)
    rig.eng.prefill(torch.zeros(B, 4, dtype=torch.int32, device="cuda"), [4] * B)
    th = rig.eng.tree(synth.random_parent_tree(n, 4, tree_id=3, n_heads=4, kmax=1))
    before = rig.eng.launch_count()
    rig.eng.verify(th, torch.zeros(B, n, dtype=torch.int32, device="cuda"))
    buf = C.create_string_buffer(1 << 14)
    assert cb.lib().cerb_launch_order_table(variant, buf, len(buf)) == cb.OK
    # (a tree of more than 128 nodes: attention in two launches)
    assert rig.eng.launch_count() - before == len(buf.value.decode().strip().split("\n")) + (3 if n > 128 else 0)


# The LM head in one part, straight to the logits: columns that four divides, that eight does not, that four does not; rows of one and of two MMA heights
@pytest.mark.parametrize("vocab,n", [(2400, 9), (2412, 64), (2410, 65), (2398, 128)])
def test_lm_head_sums(vocab, n):
    ms = synth.ModelShape(1, 4096, 2, 128, 64, vocab, "bf16")
    model = synth.make_model(ms, device="cuda")
    eng = cb.Cerberus(ms, model, None, None, [], max_tokens=64, max_batch=1, max_nodes=n)
    eng.prefill(torch.zeros(1, 5, dtype=torch.int32, device="cuda"), [5])
    tree = synth.random_parent_tree(n, 4, tree_id=11)
    tt = synth.make_prompt(vocab, n, seq=3).to(torch.int32).cuda().view(1, n).contiguous()
    top, logits, hidden = eng.verify(eng.tree(tree), tt, want_logits=True, want_hidden=True)
    assert eng.device_status() == 0
    assert close(logits[0], orc.linear(hidden[0].cpu(), model["lm_head"].cpu()), 0) < 1e-4
    assert torch.equal(top[0].long(), logits[0].argmax(-1)) and torch.equal(eng.verify(eng.tree(tree), tt)[0], top)


@pytest.mark.parametrize("M", [64, 256])
def test_a_forward_whose_waits_run_out_comes_back_and_the_next_one_is_correct(M):
    """With the budget of every wait at a thousand cycles the epilogue warps of the gate-up product (11008 features of 16384 columns: over 100 us
    of weights) run out of it by the limit alone, in single CTAs and in pairs, while copies and MMAs are in flight.  The forward must come back
    with CERB_E_TIMEOUT from a wait of this kernel, and the same forward with the default budget must give the bits it gave before."""
    ms = synth.ModelShape(1, 16384, 4, 128, 11008, 512, "bf16")
    eng = cb.Cerberus(ms, synth.make_model(ms, device="cuda", std=0.01), None, None, [], max_tokens=M + 16, max_batch=1, max_nodes=16)
    tok = torch.tensor([[int(t) for t in synth.make_prompt(ms.vocab, M, seq=180)]], dtype=torch.int32, device="cuda")

    def forward():
        eng.prefill(tok, [M])
        return eng.wait_diagnosis(), eng.device_status(), eng.read_state()[2].clone()

    _, status, want = forward()
    assert status == cb.OK
    assert cb.lib().cerb_set_wait_cycles(1000) == cb.OK
    try:
        words, status, _ = forward()
    finally:
        assert cb.lib().cerb_set_wait_cycles(4_000_000_000) == cb.OK
    assert status == cb.E_TIMEOUT and 241 <= words[1] <= 246, words
    _, status, got = forward()
    assert status == cb.OK and torch.equal(got, want)
