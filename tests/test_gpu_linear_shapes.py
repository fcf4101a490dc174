"""The INT8 linear layer where its kernels change: the few-token forward product at the ends of its range and of its rule
for warps per CTA, against torch's fp32 product of the same operands."""
import pytest
import torch

from paper_2407_08296_b200 import binding as B

pytestmark = pytest.mark.gpu


def _operands(T, m, n, seed=0):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    w = B.zeros_matrix(m, n, torch.float32)
    w.copy_(0.02 * torch.randn(m, n, device="cuda", generator=gen) + 0.01)
    W = B.quantize_int8(w)
    # what lies past a row may be anything: NaN here
    X, dY = B.empty_matrix(T, n, torch.bfloat16), B.empty_matrix(T, m, torch.bfloat16)
    for t in (X, dY):
        (t._base if t._base is not None else t).fill_(float("nan"))
        t.copy_(torch.randn(t.shape, device="cuda", generator=gen))
    return X, dY, W, B.dequantize(W).to(torch.bfloat16).float()


def _check(got, a, b, status):
    """Products are exact and sums binary32: the error is that of a binary32 sum of K terms in another order (both sides),
    K * 2^-24 of the sum of magnitudes to first order (that bound holds for any order), plus the rounding to bfloat16."""
    want, mag = a @ b, a.abs() @ b.abs()
    tol = 2 * a.shape[1] * 2.0 ** -24 * mag + 2.0 ** -8 * want.abs()
    assert got.shape == want.shape and int(status.item()) == 0
    assert bool(((got.float() - want).abs() <= tol).all())
    assert float((got == want.to(torch.bfloat16)).float().mean()) > 0.98     # rounded the same but for near-ties


@pytest.mark.parametrize("T", [1, 7, 8, 9, 16, 17])
@pytest.mark.parametrize("m,n", [(1, 1), (17, 255), (40, 1025), (2369, 4096), (2368, 4096), (15, 11001)])
def test_forward_of_a_few_tokens(T, m, n):
    torch.backends.cuda.matmul.allow_tf32 = False
    X, _, W, Wd = _operands(T, m, n, seed=m + n)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Y = B.int8_linear_forward(X, W, status=status)
    _check(Y, X.float(), Wd.T, status)


# Tiles of 256 or 512 x 256, one per CTA pair: a few of them shared by clusters of 2 .. 4 pairs along K, whole rounds of persistent
# pairs alone or followed by a remainder in clusters, a tile part of whose rows are empty, extents that end inside a tile, a K
# that ends inside a block.  The last takes 512 rows for all three products.
@pytest.mark.parametrize("T,m,n", [(40, 200, 1500), (300, 1159, 3001), (257, 515, 2100), (4200, 1100, 700), (129, 2100, 4500), (1000, 3001, 640),
                                   (2817, 2100, 1800), (600, 4300, 5000), (257, 256, 65), (4500, 4096, 4090)])
def test_products_whose_tiles_are_split_along_k(T, m, n):
    torch.backends.cuda.matmul.allow_tf32 = False
    X, dY, W, Wd = _operands(T, m, n, seed=T)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    x, d = X.float(), dY.float()
    Y = B.int8_linear_forward(X, W, status=status)
    _check(Y, x, Wd.T, status)
    dX = B.int8_linear_backward_input(dY, W, status=status)
    _check(dX, d, Wd, status)
    # the weight gradient reads whole 64-column slabs: give it zeros past the row
    Xz, dYz = B.zeros_matrix(T, n, torch.bfloat16), B.zeros_matrix(T, m, torch.bfloat16)
    Xz.copy_(X)
    dYz.copy_(dY)
    G = B.int8_linear_backward_weight(dYz, Xz, status=status)
    _check(G, d.T, x, status)
    for again, first in ((B.int8_linear_forward(X, W), Y), (B.int8_linear_backward_input(dY, W), dX), (B.int8_linear_backward_weight(dYz, Xz), G)):
        assert torch.equal(again, first)


# Tiles shared by clusters whose last row ends inside a warp: 1337 = 5 * 256 + 57 rows leave one CTA of a pair 57 and the other
# none; 3001 = 5 * 512 + 441, of which 57 in the second CTA's second row block, after whole rounds of persistent pairs (the forward
# product and the input gradient; the weight gradient of either shape ends its columns and K inside a tile).
@pytest.mark.parametrize("T,m,n", [(1337, 4096, 4096), (3001, 11008, 4096)])
def test_split_products_whose_rows_end_inside_a_warp(T, m, n):
    test_products_whose_tiles_are_split_along_k(T, m, n)


# By the estimates that choose between CTA pairs and single CTAs: the forward product by single CTAs in one round (a K of less than
# a block, columns and rows that end inside a tile) and in several, the weight gradient by single CTAs in one and several rounds,
# and by pairs with 512 rows a tile.
@pytest.mark.parametrize("T,m,n", [(17, 129, 40), (255, 1000, 513), (2000, 4300, 300), (5461, 2049, 130), (8200, 4100, 600), (700, 3000, 4000)])
def test_products_by_single_ctas(T, m, n):
    test_products_whose_tiles_are_split_along_k(T, m, n)


# By the same estimates, the forms of the pairs' kernel: 256 and 512 rows a tile, whole rounds, whole rounds and a shared remainder, and
# tiles that are all shared; first as the forward product takes them, then as the weight gradient does.
@pytest.mark.parametrize("T,m,n", [(261, 5827, 2734), (289, 9710, 2155), (12599, 267, 1920), (272, 4855, 6738), (15229, 516, 3740),
                                   (525, 9887, 828), (2014, 244, 228), (4811, 9965, 267), (8947, 261, 4777), (3927, 3591, 9274), (12426, 8853, 1057)])
def test_products_in_each_form_of_the_pairs(T, m, n):
    test_products_whose_tiles_are_split_along_k(T, m, n)
