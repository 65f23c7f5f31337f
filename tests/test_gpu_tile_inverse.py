"""The FP32 inverse as column tiles (several CTAs per block), through negf_block_inverse with
NEGF_MIXED, at the edges of its tiles and thread counts.

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
