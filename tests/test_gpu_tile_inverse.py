"""The block inverses through negf_block_inverse, at the edges of their tiles and thread counts:
FP32 with the matrix in registers (n <= 128) or as column tiles over several CTAs, refined
(NEGF_MIXED), and FP64 as column tiles.

Tolerance: X is FP64-class after the refinement, so I - M X is of the order of the FP64
product's own error, n 2^-53 |M| |X| per row; 8 n 2^-53 ||M||_F ||X||_F bounds it.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_03438_gb300 as P
    P.negf.load_library()
    return P


def _matrix(n, units, seed):
    """Random blocks whose largest entries sit off the diagonal: row interchanges in every panel."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    M = torch.randn(units, n, n, dtype=torch.complex128, device="cuda", generator=g) / n ** 0.5
    for u in range(units):
        perm = torch.randperm(n, device="cuda", generator=g)
        M[u, torch.arange(n, device="cuda"), perm] += 2.0
    return M


@pytest.mark.parametrize("n", [16, 17, 31, 33, 127, 128, 129, 144, 159, 160, 255, 256, 257, 300, 511, 512])
@pytest.mark.parametrize("units", [1, 3])
def test_tile_inverse(P, n, units):
    M = _matrix(n, units, 100 * n + units)
    X = torch.empty_like(M)
    status = torch.full((units,), 7, dtype=torch.int32, device="cuda")
    ctx = P.Context(0, 1 << 28)
    try:
        P.negf.negf_block_inverse(ctx, P.MIXED, M, X, status)
        assert ctx.sync() == 0
    finally:
        ctx.close()
    eye = torch.eye(n, dtype=torch.complex128, device="cuda")
    assert int(status.abs().sum()) == 0
    for u in range(units):
        bound = 8 * n * 2.0 ** -53 * float(M[u].norm()) * float(X[u].norm())
        assert float((eye - M[u] @ X[u]).norm()) <= bound


@pytest.mark.parametrize("n,units", [(32, 400), (48, 3), (64, 1), (65, 2), (96, 200), (97, 5), (128, 160)])
def test_register_inverse_of_many_blocks(P, n, units):
    test_tile_inverse(P, n, units)


@pytest.mark.parametrize("n,units", [(63, 2), (64, 2), (65, 76), (71, 3), (72, 77), (111, 1), (112, 2), (113, 90), (128, 3),
                                     (200, 2), (257, 1)])
def test_fp64_inverse(P, n, units):
    """FP64 Gauss-Jordan: an error of the order of n 2^-53 |M| |X| as well, with pivots that keep
    the growth of these matrices (a permutation of weight 2 plus noise) near one."""
    M = _matrix(n, units, 7 * n + units)
    X = torch.empty_like(M)
    status = torch.full((units,), 7, dtype=torch.int32, device="cuda")
    for ws in (1 << 28, 1 << 20):      # with room for the tiles' scratch, and (small n) without
        ctx = P.Context(0, ws + 16 * n * (n + 1) * units)
        try:
            P.negf.negf_block_inverse(ctx, P.FP64, M, X, status)
            assert ctx.sync() == 0
        finally:
            ctx.close()
        assert int(status.abs().sum()) == 0
        eye = torch.eye(n, dtype=torch.complex128, device="cuda")
        for u in range(units):
            bound = 8 * n * 2.0 ** -53 * float(M[u].norm()) * float(X[u].norm())
            assert float((eye - M[u] @ X[u]).norm()) <= bound


@pytest.mark.parametrize("n,col", [(16, 15), (40, 17), (129, 0), (129, 128), (256, 130), (512, 300)])
def test_zero_column_is_reported(P, n, col):
    M = _matrix(n, 3, n)
    M[1, :, col] = 0.0
    X = torch.empty_like(M)
    status = torch.zeros(3, dtype=torch.int32, device="cuda")
    ctx = P.Context(0, 1 << 28)
    try:
        P.negf.negf_block_inverse(ctx, P.MIXED, M, X, status)
        ctx.sync()
    finally:
        ctx.close()
    assert status.tolist() == [0, P.negf.NEGF_ERR_SINGULAR, 0]
    eye = torch.eye(n, dtype=torch.complex128, device="cuda")
    for u in (0, 2):
        bound = 8 * n * 2.0 ** -53 * float(M[u].norm()) * float(X[u].norm())
        assert float((eye - M[u] @ X[u]).norm()) <= bound


@pytest.mark.parametrize("n,units", [(129, 4), (240, 5), (129, 24), (129, 25), (240, 26), (256, 24), (256, 25)])
def test_tiles_of_few_and_many_blocks(P, n, units):   # one cluster per block up to 4 of them
    test_tile_inverse(P, n, units)


@pytest.mark.parametrize("n,units", [(39, 2), (40, 96), (40, 97), (41, 153), (55, 152), (56, 100), (64, 9), (64, 160)])
def test_fp64_inverse_of_small_tiles(P, n, units):
    test_fp64_inverse(P, n, units)


@pytest.mark.parametrize("n,units", [(96, 153), (97, 152), (97, 153), (112, 160), (128, 153), (128, 304)])
def test_fp32_inverse_past_one_round(P, n, units):   # tiles where the second round of 152 would be far from full
    test_tile_inverse(P, n, units)
