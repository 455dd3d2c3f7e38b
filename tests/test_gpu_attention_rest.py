"""Attention whose (sequence, head) items leave a rest behind full rounds of SMs (a launch of its own, keys split), whose key splits have to fit the GPU
at once, or whose tree takes a second launch that does not wait for the first."""
import pytest

from paper_2410_13344_b200 import binding as cb
from tests.helpers import close
from tests.test_gpu_kernels import TOL_BF16, _attention_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n,H,Dh,lens,n_active", [
    # 148 items and a rest of 12 / 2 / 74 (keys on M); lengths on both sides of the first split, dead nodes, an empty cache
    (5, 24, 32, 128, [800, 760, 0, 129, 790], [24, 1, 7, 24, 3]),
    (15, 17, 10, 128, [900 - 61 * b for b in range(15)], None),
    (6, 33, 37, 128, [770, 10, 500, 127, 128, 769], None),
    # a rest of 12 with queries on M, 65 to 128 rows
    (5, 70, 32, 128, [2600, 31, 64, 1500, 2550], [70, 66, 1, 70, 64]),
    # 20, 24 and 48 items: seven, six and three splits would not be there at once; head_dim 64 and 16 rows, too
    (5, 40, 4, 128, [1700, 900, 3, 640, 1290], None),
    (6, 100, 4, 128, [3100, 60, 1000, 2047, 2048, 9], None),
    (12, 20, 4, 64, [1500 - 100 * b for b in range(12)], None),
    (12, 9, 4, 128, [1500 - 100 * b for b in range(12)], None),
    (12, 1, 4, 128, [3000 - 200 * b for b in range(12)], None),
    # two launches over the rows; the second one with live rows in one sequence only
    (2, 150, 5, 128, [700, 333], [150, 128]),
    (3, 192, 50, 128, [800, 20, 130], [192, 129, 5]),
    # ... whose second one takes fewer splits than would be there at once: 24 items in three, 32 in two, 64 in one; 40 of 3000 keys do not
    (6, 150, 4, 128, [1000 - 7 * b for b in range(6)], None),
    (1, 192, 32, 128, [300], None),
    (2, 150, 32, 128, [310, 2], [150, 131]),
    (1, 150, 40, 128, [3000], None),
])
def test_matches_oracle(B, n, H, Dh, lens, n_active):
    for _ in range(2):
        for got_o, got_l, O, l in _attention_case(cb, "bf16", B, n, H, Dh, lens, 6, seed_id=140 + n, n_active=n_active):
            assert close(got_o, O, 0) < TOL_BF16
            assert close(got_l, l, 0) < 2e-3
