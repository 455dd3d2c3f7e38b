"""Attention of one query row per sequence: pages to warps, splits to the CTAs of a cluster."""
import pytest

from paper_2410_13344_b200 import binding as cb
from tests.helpers import close
from tests.test_gpu_kernels import TOL_BF16, _attention_case

pytestmark = pytest.mark.gpu


# no prefix; this step's key alone in its page, first and last in a page; fewer pages than warps, one more than a round of all
# of them; eight splits with one page per warp less one key and exactly, and with three; two splits (and a sequence without a row); no splits
@pytest.mark.parametrize("H,lens", [(2, [0]), (2, [1, 15, 16, 17]), (3, [112, 127, 128, 129]), (32, [1007]), (32, [1008]), (32, [3000]),
                                    (4, [2047, 5, 700]), (32, [500, 0, 1000, 64]), (20, [(53 * b) % 400 for b in range(16)])],
                         ids=lambda v: str(v) if isinstance(v, int) else "-".join(map(str, v[:4])))
@pytest.mark.parametrize("head_dim", [64, 128])
def test_one_row_matches_oracle(H, lens, head_dim):
    for got_o, got_l, O, l in _attention_case(cb, "bf16", len(lens), 1, H, head_dim, lens, 1, seed_id=150,
                                            n_active=[1, 0, 1, 1] if lens == [500, 0, 1000, 64] else None):
        assert close(got_o, O, 0) < TOL_BF16
        assert close(got_l, l, 0) < 2e-3
