"""The sketches at the edges of their kernels' splits, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import mihs_oracle as o
from paper_1912_03514_gb300 import mihs
from paper_1912_03514_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda"


# n, d, m: one chunk of the counting sort and the first row of a second one, few full buckets (their rows cut
# over several blocks and summed by the reduction), one bucket too full to sort, more buckets than the chunk
# counters hold, each width of a block's column slice with its remainder
@pytest.mark.parametrize("n,d,m", [(2048, 64, 7), (2049, 65, 7), (200000, 33, 3), (140000, 130, 16), (30000, 5, 1),
                                   (20000, 129, 8193), (9000, 257, 8192), (131073, 1025, 40), (1, 1, 1)])
def test_countsketch_splits_are_exact(n, d, m):
    """±1 sums of small integers are exact in fp32, in any order."""
    lda = (d + 3) // 4 * 4
    A = torch.full((n, lda), float("nan"))
    A[:, :d] = W.randint_matrix((n, d), n + d, -8, 8)
    Ad = A.to(DEV).as_strided((n, d), (lda, 1))
    out = torch.full((m, d + 1), float("nan"), device=DEV)[:, :d]  # rows of SA not 16-byte aligned
    SA = mihs.sketch_apply(Ad, o.COUNTSKETCH, m, 31 + m, SA=out)
    SA2 = mihs.sketch_apply(Ad, o.COUNTSKETCH, m, 31 + m)
    h, sign = o.countsketch_hash(n, m, 31 + m)
    ref = np.zeros((m, d))
    np.add.at(ref, h, A[:, :d].numpy().astype(np.float64) * np.asarray(sign, dtype=np.float64)[:, None])
    assert np.array_equal(SA.cpu().numpy().astype(np.float64), ref)
    assert np.array_equal(SA2.cpu().numpy().astype(np.float64), ref)
