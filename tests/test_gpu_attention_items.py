"""Attention of 65 to 128 query rows with more (sequence, head) items than CTAs: every CTA takes several in turn."""
import pytest

from paper_2410_13344_b200 import binding as cb
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
