"""The sketches at the edges of their kernels' splits, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import mihs_oracle as o
from paper_1912_03514_gb300 import mihs
from paper_1912_03514_gb300 import workloads as W
from tests import test_gpu_mixed as mixed
from tests import test_gpu_parity as parity

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


# n, d, m: a single block of 1024 rows and one row more, fewer rows than a block, the last column pair alone, each
# count of samples per thread and its first extra sample, more samples than one block of threads holds
@pytest.mark.parametrize("n,d,m", [(1024, 16, 128), (1025, 17, 129), (3, 5, 2), (1, 1, 1), (2500, 31, 256),
                                   (2500, 33, 257), (5000, 15, 385), (5000, 48, 513), (4100, 20, 640),
                                   (4100, 20, 641), (9000, 3, 2000), (70001, 100, 64)])
def test_srht_splits_are_exact(n, d, m):
    """±1 sums of small integers are exact in fp32; only the factor 1/√m rounds, and the product with it."""
    lda = (d + 3) // 4 * 4
    A = torch.full((n, lda), float("nan"))
    A[:, :d] = W.randint_matrix((n, d), n + d, -3, 3)
    Ad = A.to(DEV).as_strided((n, d), (lda, 1))
    out = torch.full((m, d + 1), float("nan"), device=DEV)[:, :d]  # rows of SA not 16-byte aligned
    SA = mihs.sketch_apply(Ad, o.SRHT, m, 5 + m, SA=out).cpu().numpy().astype(np.float64)
    ref = o.sketch_apply(o.SRHT, A[:, :d].numpy().astype(np.float64), m, 5 + m)
    sums = np.rint(ref * np.sqrt(m))  # the integers themselves (the oracle's own fp64 rounding dropped)
    assert np.all(np.abs(SA * np.sqrt(m) - sums) <= 2.0 ** -22 * np.abs(sums))


# n, d, m: the samples that a block holds in registers and one more (their sums then lie in shared memory), as many of
# both as one block takes and the first that take two, with an odd last column and with that column alone, units that
# end inside the matrix and that do not
@pytest.mark.parametrize("n,d,m", [(5000, 33, 640), (5000, 33, 641), (4096, 17, 673), (3000, 1, 700), (5000, 15, 1240),
                                   (6000, 16, 1241), (4100, 1023, 1249), (9001, 31, 1300), (20000, 2, 2481)])
def test_srht_samples_past_the_registers(n, d, m):
    test_srht_splits_are_exact(n, d, m)


# n, d, m: the most buckets that the chunk counters hold and the first past them, buckets that a block walks in several
# slices after sorting them once, with a ragged last column group, and rows too few to cut a bucket
@pytest.mark.parametrize("n,d,m", [(30000, 70, 2048), (30000, 70, 2049), (9000, 1501, 4000), (5000, 2047, 2500),
                                   (32768, 512, 1024), (60000, 1030, 1300), (8192, 3, 8192)])
def test_countsketch_many_buckets(n, d, m):
    test_countsketch_splits_are_exact(n, d, m)


# widths on both sides of those whose operands are made ready before their stage is free (clusters of four blocks),
# one and two sketch-row tiles, stages fewer and more than the ring
@pytest.mark.parametrize("n,d,m", [(3000, 768, 129), (3000, 769, 129), (60, 900, 40), (5000, 1023, 300),
                                   (2049, 1024, 128), (2049, 1025, 257)])
def test_gaussian_stage_orders(n, d, m):
    parity.test_sketch_matches_oracle(o.GAUSSIAN, n, d, m)
    mixed.test_gaussian_bf16_sketch_matches_oracle(n, d, m)
    mixed.test_gaussian_fp8_sketch_matches_oracle(n, d, m)


# few buckets in many parts: parts of even and of uneven numbers of chunks, at and past two waves of blocks
@pytest.mark.parametrize("n,d,m", [(131072, 17, 31), (131072, 64, 32), (131072, 33, 39), (81920, 256, 30), (81920, 130, 32),
                                   (10240, 260, 97), (10241, 1027, 100), (131073, 4, 1)])
def test_countsketch_few_buckets(n, d, m):
    test_countsketch_splits_are_exact(n, d, m)


# ragged rows whose last warp holds three column groups and four, of more than 256 columns and fewer, a last slice of
# one and of two groups in blocks that walk all slices and that do not, a matrix that takes four blocks per SM
@pytest.mark.parametrize("n,d,m", [(5000, 139, 100), (5000, 267, 100), (5000, 271, 100), (9000, 517, 502), (9000, 525, 502),
                                   (9000, 1025, 2500), (9000, 1030, 40), (20700, 815, 90)])
def test_countsketch_last_groups(n, d, m):
    test_countsketch_splits_are_exact(n, d, m)
