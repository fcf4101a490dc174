"""The direct route of the subspace refresh where its kernels change: the row counts at which the tridiagonal reduction and
the back-transformation take another instance, a batch that is reduced in several launches, vectors on the long side,
odd extents, gradients whose eigenvalues coincide, spectra on both sides of what it resolves, and the shapes it leaves to the
iterative route."""
import pytest
import torch

from paper_2407_08296_b200 import binding as B

pytestmark = pytest.mark.gpu


def _gradient(m, n, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    k = 16
    u = torch.randn(m, k, device="cuda", generator=gen) / m ** 0.5 / torch.arange(1, k + 1, device="cuda")
    v = torch.randn(n, k, device="cuda", generator=gen) / n ** 0.5
    G = B.zeros_matrix(m, n, torch.bfloat16)
    G.copy_(u @ v.T + 1e-3 * torch.randn(m, n, device="cuda", generator=gen))
    return G


def _check(G, P, side):
    """Backward error: P holds the leading eigenvectors of a matrix within s * 2^-24 * lambda_1 (s the short side: the
    first-order bound of a Householder reduction in binary32, which also covers the sums of the Gram matrix) of G G^T."""
    X = G.double() if side == "left" else G.double().T
    A, Z = X @ X.T, P.double()
    s, r = min(G.shape), P.shape[1]
    lam = torch.linalg.eigvalsh(A if A.shape[0] == s else X.T @ X).flip(0)
    eps = s * 2.0 ** -24
    assert float((Z.T @ Z - torch.eye(r, device="cuda")).abs().max()) <= max(eps, 1e-5)
    q = (Z * (A @ Z)).sum(0)
    assert float((A @ Z - Z * q).norm(dim=0).max()) <= eps * float(lam[0])
    assert float((q - lam[:r]).abs().max()) <= eps * float(lam[0])
    assert bool((Z.gather(0, Z.abs().argmax(0, keepdim=True)) > 0).all())


@pytest.mark.parametrize("m,n,r,side", [(64, 700, 32, "left"), (130, 128, 32, "left"), (511, 640, 64, "left"), (513, 1025, 128, "left"),
                                        (1025, 1030, 160, "right"), (1100, 769, 96, "left"), (2049, 2100, 288, "left"), (2500, 2047, 256, "left")])
def test_vectors_are_those_of_a_nearby_matrix(m, n, r, side):
    G = _gradient(m, n, seed=m)
    P = torch.zeros((m if side == "left" else n, r), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.refresh_subspace(G, r, P_fp32=P, status=status, side=side)
    assert int(status.item()) == 0
    _check(G, P, side)


def test_a_batch_reduced_in_several_launches():
    m, n, r = 1400, 1600, 352               # eight matrices do not fit the SMs at once
    items = [{"G": _gradient(m, n, seed=i), "seed": i, "P_fp32": torch.zeros((m, r), device="cuda")} for i in range(8)]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.refresh_subspace_batched(items, r, status=status)
    assert int(status.item()) == 0
    for it in (items[0], items[5], items[7]):
        _check(it["G"], it["P_fp32"], "left")


@pytest.mark.parametrize("kind", ["zero", "identity", "zero_rows"])
def test_coinciding_eigenvalues_have_orthogonal_vectors(kind):
    G = B.zeros_matrix(256, 384, torch.bfloat16)
    if kind == "identity":
        G.copy_(torch.eye(256, 384))
    elif kind == "zero_rows":
        G[::5].copy_(torch.randn(52, 384))
    P = torch.zeros((256, 64), device="cuda")
    B.refresh_subspace(G, 64, P_fp32=P)
    assert float((P.T @ P - torch.eye(64, device="cuda")).abs().max()) <= 1e-5


# More tiles of the Gram matrix than CTAs, its last rows inside a warp (1400 = 10 * 128 + 120, 2000 = 15 * 128 + 80), read along
# the gradient's rows (m < n) and along its columns, for vectors of the short side and of the long one.
@pytest.mark.parametrize("m,n,r", [(1400, 1600, 192), (1600, 1400, 192), (2000, 2300, 256), (2300, 2000, 256)])
@pytest.mark.parametrize("side", ["left", "right"])
def test_batches_of_odd_gradients_from_both_sides(m, n, r, side):
    rows = m if side == "left" else n
    items = [{"G": _gradient(m, n, seed=40 + i), "seed": i, "P_fp32": torch.zeros((rows, r), device="cuda")} for i in range(8)]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.refresh_subspace_batched(items, r, status=status, side=side)
    assert int(status.item()) == 0
    for it in items[::3]:
        _check(it["G"], it["P_fp32"], side)


def _with_singular_values(m, n, values, seed):
    """A bf16 gradient with these singular values (and what rounding to bf16 adds: about 1e-3 of its size, spread over all of them)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    u = torch.linalg.qr(torch.randn(m, len(values), device="cuda", dtype=torch.float64, generator=gen))[0]
    v = torch.linalg.qr(torch.randn(n, len(values), device="cuda", dtype=torch.float64, generator=gen))[0]
    G = B.zeros_matrix(m, n, torch.bfloat16)
    G.copy_(((u * values) @ v.T).float())
    return G


def test_vectors_computed_beside_those_wanted_do_not_raise_the_flag():
    # vectors of the long side are computed in whole 64s: 96 wanted, 128 computed, and the spectrum ends with the 96th
    m, n, r = 1025, 768, 96
    G = _with_singular_values(m, n, torch.linspace(1.0, 0.5, r, device="cuda", dtype=torch.float64), seed=3)
    P = torch.zeros((m, r), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.refresh_subspace(G, r, P_fp32=P, status=status)
    assert int(status.item()) == 0
    u = torch.linalg.svd(G.double(), full_matrices=False)[0][:, :r]
    # the subspace is separated by a gap of half the spectrum: it is resolved to some units in the last place of binary32
    assert float((u - P.double() @ (P.double().T @ u)).norm(dim=0).max()) <= 768 * 2.0 ** -24 / 0.25


# Shapes that take the iterative route by themselves, one for each block form of its eigen-iteration: a block that is a small part
# of the short side (64 of 1024 columns: rows of up to 1024), and a short side of more than 4096 rows (a block of 1088).  The
# spectrum falls by ten behind the r-th vector, so that twelve iterations leave 10^-24 of what lies behind it.
@pytest.mark.parametrize("m,n,r", [(1024, 1100, 32), (4224, 4160, 544)])
def test_shapes_of_the_iterative_route(m, n, r):
    s = min(m, n)
    values = torch.full((s,), 0.05, device="cuda", dtype=torch.float64)
    values[:r] = torch.linspace(1.0, 0.5, r, device="cuda", dtype=torch.float64)
    G = _with_singular_values(m, n, values, seed=r)
    P = torch.zeros((m, r), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.refresh_subspace(G, r, P_fp32=P, status=status, seed=5)
    assert int(status.item()) == 0
    _check(G, P, "left")


# The flag is raised where the r-th eigenvalue is below 0.1 * 768 * 2^-24 of the first, a singular value of 2.1e-3 of the first.
# Above it the subspace is the exact one's to the 1e-2 rad asked of every refresh; below, the vectors are still orthonormal.
@pytest.mark.parametrize("ratio,flag", [(1e-2, 0), (3.2e-3, 0), (1.5e-3, B.QG_DEV_BAD_FACTOR), (5e-4, B.QG_DEV_BAD_FACTOR)])
def test_spectra_on_both_sides_of_what_is_resolved(ratio, flag):
    m, n, r = 768, 1100, 128
    values = torch.full((m,), 0.3 * ratio, device="cuda", dtype=torch.float64)
    values[:r] = ratio ** (torch.arange(r, device="cuda", dtype=torch.float64) / (r - 1))
    G = _with_singular_values(m, n, values, seed=9)
    P = torch.zeros((m, r), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.refresh_subspace(G, r, P_fp32=P, status=status)
    assert int(status.item()) == flag
    Z = P.double()
    assert float((Z.T @ Z - torch.eye(r, device="cuda")).abs().max()) <= 768 * 2.0 ** -24
    if flag == 0:
        u = torch.linalg.svd(G.double(), full_matrices=False)[0][:, :r]
        assert float(torch.linalg.matrix_norm(u - Z @ (Z.T @ u), 2)) < 1e-2


# The route is decided by the shape: on either side of its line for each range of short sides.  The seed of the start block enters
# the iterative route only.
@pytest.mark.parametrize("s,b,direct", [(768, 128, True), (768, 64, False), (1024, 128, False), (1088, 192, True), (1536, 256, True), (1600, 256, False),
                                        (2048, 512, True), (2112, 512, False), (2112, 576, True)])
def test_route_of_a_shape(s, b, direct):
    G, r = _gradient(s, s + 8, seed=1), 32
    P = [torch.zeros((s, r), device="cuda") for _ in range(2)]
    for seed in range(2):
        B.refresh_subspace(G, r, oversample_cols=b - r, seed=seed, P_fp32=P[seed])
    assert torch.equal(P[0], P[1]) == direct


# More vectors than one launch finds, whose pivots lie over the matrix that has been reduced: more than half of the short side's, or
# a quarter from 2049 rows on; vectors of the long side and their product go there as well.
@pytest.mark.parametrize("m,n,r", [(512, 640, 320), (700, 512, 416), (2304, 2310, 640)])
def test_vectors_found_in_several_launches(m, n, r):
    G = _gradient(m, n, seed=r)
    P = torch.zeros((m, r), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.refresh_subspace(G, r, P_fp32=P, status=status)
    assert int(status.item()) == 0
    _check(G, P, "left")


def test_a_workspace_of_the_iterative_route_gets_that_route():
    # the direct route asks for more than the iterative one here; a caller with a workspace of the smaller size is served by it
    s, b, r = 3072, 768, 384
    G = _gradient(s, s, seed=2)
    enough = 12 * s * b + 4 * s * b + 8 * b * b + 6 * s * b + 256 * (s + b) + (33 << 20)
    assert enough < B.workspace_bytes(B.QG_OP_REFRESH, s, s, b)
    P = [torch.zeros((s, r), device="cuda") for _ in range(3)]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(enough, dtype=torch.uint8, device="cuda")
    B.refresh_subspace(G, r, oversample_cols=b - r, P_fp32=P[0], workspace=ws, status=status)
    B.debug_set_refresh_direct(False)
    try:
        B.refresh_subspace(G, r, oversample_cols=b - r, P_fp32=P[1], status=status)
    finally:
        B.debug_set_refresh_direct(True)
    B.refresh_subspace(G, r, oversample_cols=b - r, P_fp32=P[2], status=status)
    assert int(status.item()) == 0
    assert torch.equal(P[0], P[1]) and not torch.equal(P[0], P[2])
