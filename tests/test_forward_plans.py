"""Which kernel a product of a forward of 9 to 256 rows goes to, and in which chains of tensor-core accumulations it is summed (host only)."""
import math

import pytest

from paper_2410_13344_b200 import binding as cb

# d_model (heads of 128), mlp_dim
WIDTHS = [(256, 768), (1024, 2816), (1536, 4096), (2048, 5632), (2560, 6912), (3200, 8640), (3584, 9728), (4096, 11008), (4096, 12288), (5120, 13824), (8192, 22016)]
# one row count in each class, and both sides of every edge between two
ROWS = [9, 32, 33, 64, 65, 96, 97, 128, 129, 160, 192, 193, 224, 256]


def _products(d, mlp):
    return (("qkv", 3 * d, d), ("o_down", d, d), ("o_down", d, mlp), ("gate_up", 2 * mlp, d), ("lm_head", 32000, d))


def _stream_k_chains(N, K, sms=148):
    """Of up to 128 rows otherwise: (256 weight rows, 64 k) units in one list, cut into equal shares of four at least; a chain ends with its share or its tile."""
    kb = -(-K // 64)
    total = -(-N // 256) * kb
    per = max(-(-total // sms), min(kb, 4))
    cuts = sorted(set(range(0, total, per)) | set(range(0, total, kb)) | {total})
    lengths = [b - a for a, b in zip(cuts, cuts[1:])]
    return max(lengths), math.sqrt(sum(n ** 3 for n in lengths) / total)


@pytest.mark.parametrize("d,mlp", WIDTHS)
def test_chains_are_no_longer_than_those_of_the_kernel_a_product_goes_to_otherwise(d, mlp):
    """A running sum is cut off towards zero at every step, so a sum's error grows with its chains: as the root mean square of their lengths."""
    for M in ROWS:
        for product, N, K in _products(d, mlp):
            g = cb.forward_gemm_plan(product, M, N, K)
            if M <= 128:
                longest, mean = _stream_k_chains(N, K)
                assert g.other_longest == longest and abs(g.other_mean_length - 100 * mean) < 1, (product, M, g)
            if g.rows_kernel:
                assert g.longest <= g.other_longest and g.mean_length <= 1.005 * g.other_mean_length, (product, M, g)
                kb = -(-K // 64)
                assert 512 >= g.chains >= g.issuers >= 1 and g.longest * g.chains * g.parts >= kb, (product, M, g)


def test_who_takes_what_at_the_model_widths():
    """The routes of the 7B and 13B shapes, at the edges of every class of rows."""
    def taken(d, mlp):
        return {p: [M for M in ROWS if all(cb.forward_gemm_plan(q, M, N, K).rows_kernel for q, N, K in _products(d, mlp) if q == p)]
                for p in ("qkv", "o_down", "gate_up", "lm_head")}

    narrow, pairs, wide = [M for M in ROWS if M <= 128], [M for M in ROWS if M > 128], [M for M in ROWS if M > 192]
    assert taken(4096, 11008) == {"qkv": narrow + wide, "o_down": ROWS, "gate_up": narrow + pairs, "lm_head": narrow}
    assert taken(5120, 13824) == {"qkv": narrow + wide, "o_down": narrow + wide, "gate_up": narrow, "lm_head": narrow}


def test_rows_and_products_without_a_plan_are_refused():
    for args in (("qkv", 8, 3072, 1024), ("qkv", 257, 3072, 1024), ("qkv", 64, 3000, 1024), ("gate_up", 64, 5633, 1024)):
        with pytest.raises(cb.CerbError):
            cb.forward_gemm_plan(*args)
