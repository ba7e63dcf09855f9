"""The passes over A at the edges of their kernels' splits, on integer data: every sum is exact in fp32 in any
order, so a dropped, doubled or misplaced row or column shows up as a difference."""
import numpy as np
import pytest
import torch

from paper_1912_03514_gb300 import mihs
from paper_1912_03514_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _matrix(n, d, seed, lo=-2, hi=2):
    """A (n × d) with NaN between its rows, on the GPU, and its values in fp64."""
    A = torch.full((n, (d + 3) // 4 * 4), float("nan"))
    A[:, :d] = W.randint_matrix((n, d), seed, lo, hi)
    return A.to(DEV)[:, :d], A[:, :d].double().numpy()


# rows: less than a stage, one stage and one row more, more stages than the ring, rows that no block gets; columns:
# one group, each width of the kernel, the last that takes 16 rows a stage and the first that takes 8
@pytest.mark.parametrize("n,d,nl", [(3, 1, 1), (16, 64, 16), (17, 65, 3), (33, 128, 16), (3000, 127, 9),
                                    (5000, 256, 16), (12000, 300, 2), (9000, 512, 16), (2500, 676, 16),
                                    (2500, 700, 16), (2600, 704, 5), (4001, 1021, 16), (20001, 1024, 16)])
def test_path_gradient_is_exact(n, d, nl):
    A, An = _matrix(n, d, n + d)
    b = W.randint_matrix((n,), 3, -9, 9)
    X = W.randint_matrix((nl, d), 4, -1, 1)
    lams = [float(l % 3) for l in range(nl)]
    G = mihs.gradient_path(A, b.to(DEV), X.to(DEV), lams).cpu().double().numpy()
    Xn = X.double().numpy()
    ref = (b.double().numpy()[:, None] - An @ Xn.T).T @ An - np.array(lams)[:, None] * Xn
    assert np.abs(ref).max() < 2 ** 24
    assert np.array_equal(G, ref)
    assert mihs.device_status() == 0


# the last width of each form of the path kernel and the first of the next, with the most iterates that take half of
# it and the first that take both; rows that fill the rings several times, and a last stage of 1 to 3 rows
@pytest.mark.parametrize("n,d,nl", [(60001, 128, 8), (60002, 129, 9), (30003, 256, 9), (30000, 257, 8),
                                    (30001, 512, 8), (30002, 513, 9), (15003, 768, 8), (15000, 769, 8),
                                    (15001, 1024, 8), (2, 768, 16)])
def test_path_gradient_widths_are_exact(n, d, nl):
    A, An = _matrix(n, d, n + d, -1, 1)
    b = W.randint_matrix((n,), 3, -9, 9)
    X = W.randint_matrix((nl, d), 4, -1, 1)
    lams = [float(l % 3) for l in range(nl)]
    G = mihs.gradient_path(A, b.to(DEV), X.to(DEV), lams).cpu().double().numpy()
    Xn = X.double().numpy()
    ref = (b.double().numpy()[:, None] - An @ Xn.T).T @ An - np.array(lams)[:, None] * Xn
    assert np.abs(ref).max() < 2 ** 24
    assert np.array_equal(G, ref)
    assert mihs.device_status() == 0


# one row and less than a warp's of them, each width of the one-launch form, rows that end inside a group of eight, the
# largest matrix it takes and the first it does not; the result over x where x has its shape
@pytest.mark.parametrize("n,d", [(1, 1), (15, 3), (16, 128), (300, 129), (4095, 256), (4099, 257), (1000, 509),
                                 (4096, 512), (8192, 512), (8193, 512), (16384, 128), (16385, 128),
                                 (16383, 256), (16385, 255)])
def test_small_gradient_is_exact(n, d):
    A, An = _matrix(n, d, 7 * n + d, -1, 1)
    b, x = W.randint_matrix((n,), 11, -9, 9), W.randint_matrix((d,), 12, -2, 2)
    bn, xn = b.double().numpy(), x.double().numpy()
    ref = An.T @ (bn - An @ xn) - 3.0 * xn
    assert np.abs(ref).max() < 2 ** 24
    off = torch.zeros(d + 1, device=DEV)  # x not 16-byte aligned
    off[1:] = x.to(DEV)
    bd = b.to(DEV)
    assert np.array_equal(mihs.gradient(A, bd, off[1:], 3.0).cpu().double().numpy(), ref)
    mihs.gradient(A, bd, off[1:], 3.0, g=off[1:])
    assert np.array_equal(off[1:].cpu().double().numpy(), ref)


# rows wider than 1024, whose x is in shared memory for all columns that the kernel covers (1536 or 2048): each number of
# 128-column groups from the first to the last of either, the widths on both sides of a step
@pytest.mark.parametrize("n,d", [(2000, 1025), (2003, 1152), (1999, 1153), (2001, 1280), (700, 1281), (2005, 1408),
                                 (2000, 1409), (2002, 1536), (1997, 1537), (2003, 1664), (2001, 1665), (5, 1792),
                                 (2004, 1793), (2001, 1920), (2002, 1921), (2003, 2047)])
def test_wide_gradient_is_exact(n, d):
    A, An = _matrix(n, d, n + d, -1, 1)
    b, x = W.randint_matrix((n,), 11, -9, 9), W.randint_matrix((d,), 12, -1, 1)
    bn, xn = b.double().numpy(), x.double().numpy()
    ref = An.T @ (bn - An @ xn) - 3.0 * xn
    assert np.abs(ref).max() < 2 ** 24
    assert np.array_equal(mihs.gradient(A, b.to(DEV), x.to(DEV), 3.0).cpu().double().numpy(), ref)
    assert mihs.device_status() == 0


# an infinite x: the rows of a block's last group that do not exist add nothing
@pytest.mark.parametrize("n,d", [(5, 3), (70, 130), (300, 260)])
def test_small_gradient_of_an_infinite_iterate(n, d):
    x = torch.zeros(d)
    x[1] = float("inf")
    A, _ = _matrix(n, d, 1, 1, 1)
    g = mihs.gradient(A, torch.zeros(n, device=DEV), x.to(DEV), 1.0)
    assert torch.equal(g.cpu(), torch.full((d,), -float("inf")))


# n, d: one group of columns and less, each width of the kernel with and without 16-byte rows of dA, staged in two
# halves past 1024 columns, the last row's last group
@pytest.mark.parametrize("n,d", [(1, 1), (5, 3), (64, 4), (33, 127), (100, 129), (257, 255), (300, 512), (301, 510),
                                 (77, 1001), (129, 1024), (65, 1025), (40, 2047), (41, 2048)])
def test_backward_is_exact(n, d):
    A, An = _matrix(n, d, 5 * n + d)
    b, x, v = W.randint_matrix((n,), 6, -9, 9), W.randint_matrix((d,), 7, -2, 2), W.randint_matrix((d,), 8, -2, 2)
    off = torch.zeros(d + 1, device=DEV)  # x not 16-byte aligned
    off[1:] = x.to(DEV)
    bn, xn, vn = (t.double().numpy() for t in (b, x, v))
    r, q = bn - An @ xn, An @ vn
    dA, db, dl = mihs.backward_grads(A, b.to(DEV), off[1:], v.to(DEV))
    assert np.array_equal(dA.cpu().double().numpy(), np.outer(r, vn) - np.outer(q, xn))
    assert np.array_equal(db.cpu().double().numpy(), q)
    assert float(dl) == -float(xn @ vn)
    _, db2, _ = mihs.backward_grads(A, b.to(DEV), off[1:], v.to(DEV), want_dA=False)
    assert torch.equal(db, db2)


# n, d: fewer rows than a split or a quad, a last split that is shorter, one and several column slices, ragged columns
@pytest.mark.parametrize("n,d", [(1, 1), (3, 7), (5, 1030), (33, 4096), (37, 8193), (130, 50001), (513, 20000),
                                 (2048, 2048), (2045, 9001)])
def test_dual_gradient_is_exact(n, d):
    A, An = _matrix(n, d, 9 * n + d, -1, 1)
    b, nu = W.randint_matrix((n,), 10, -9, 9), W.randint_matrix((n,), 11, -1, 1)
    g = mihs.gradient_dual(A, b.to(DEV), nu.to(DEV), 2.0).cpu().double().numpy()
    u = An.T @ nu.double().numpy()
    assert np.array_equal(g, b.double().numpy() - An @ u - 2.0 * nu.double().numpy())
    assert np.array_equal(mihs.dual_recover(A, nu.to(DEV)).cpu().double().numpy(), u)


@pytest.mark.parametrize("n,d", [(1, 1), (9, 8), (40, 9), (3000, 257), (5000, 2048)])
def test_gradients_are_exact(n, d):
    """The split-K reductions: fewer and more partials than groups, columns past the last block."""
    A, An = _matrix(n, d, 13 * n + d)
    b, x = W.randint_matrix((n,), 14, -9, 9), W.randint_matrix((d,), 15, -1, 1)
    ref = An.T @ (b.double().numpy() - An @ x.double().numpy()) - 3.0 * x.double().numpy()
    assert np.array_equal(mihs.gradient(A, b.to(DEV), x.to(DEV), 3.0).cpu().double().numpy(), ref)
    assert np.array_equal(mihs.gradient_refined(A, b.to(DEV), x.double().to(DEV), 3.0).cpu().numpy(), ref)


# rows of dA off 16 bytes: the widths at which the last 128 columns are half full and one fewer, for each count of such
# groups, and past them
@pytest.mark.parametrize("n,d", [(300, 63), (301, 65), (77, 191), (78, 193), (100, 319), (101, 321), (65, 447), (66, 449),
                                 (64, 575), (63, 577), (65, 703), (64, 705), (33, 831), (34, 833), (33, 959), (32, 961),
                                 (40, 1023), (41, 1087), (42, 1089)])
def test_backward_of_unaligned_rows(n, d):
    test_backward_is_exact(n, d)


# n, d: one split that writes A^T nu itself, the first matrix with two, one column slice and more
@pytest.mark.parametrize("n,d", [(256, 1500), (257, 1500), (128, 16384), (129, 16384), (255, 8193), (300, 16381),
                                 (64, 65536), (64, 65540)])
def test_dual_gradient_of_few_rows(n, d):
    test_dual_gradient_is_exact(n, d)


# more than eight iterates on both sides of each width, and each number of rows, at which the pass keeps them in shared
# memory
@pytest.mark.parametrize("n,d,nl", [(13000, 256, 9), (12289, 257, 9), (12288, 300, 16), (12287, 300, 16), (14001, 381, 10),
                                    (14000, 384, 9), (13000, 385, 9), (2001, 512, 12), (2500, 513, 9), (2499, 600, 16),
                                    (37, 640, 11), (3, 540, 13), (2000, 641, 9), (32768, 645, 9), (32767, 700, 16),
                                    (33001, 701, 12), (32769, 832, 9), (33000, 833, 9)])
def test_path_gradient_of_many_iterates(n, d, nl):
    test_path_gradient_is_exact(n, d, nl)
