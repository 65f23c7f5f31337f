"""The byte-digit block product (NEGF_MIXED, 16 <= n <= 512) at the edges of its tiles, passes
and tile widths.

Tolerance per entry, from the scheme: with scales 2^e, |x| < 2^(e-1) <= 2 max|x|, every entry is
rounded to 2^-57 of its scale and the dropped digit products stay below 6 2^14 2^-72 of the
scales each, over 2n real terms: at most 2n (2 2^-58 + 6 2^-58) 2^(eA + eB) < 2n 2^-55 16 max|A row|
max|B column| = n 2^-50 max|A row| max|B column|.  (The comparison product in complex128 rounds
at the same order, n 2^-53.)
"""
from fractions import Fraction

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


def _check(P, A, B, C, op, alpha, beta, ref=None):
    n = A.shape[-1]
    D = torch.empty_like(A)
    H = lambda x, o: x.mH if o else x  # noqa: E731
    a, b = H(A, op[0]), H(B, op[1])
    if ref is None:
        ref = alpha * (a @ b) + (beta * C if C is not None else 0)
    ctx = P.Context(0, 1 << 30)
    try:
        P.negf.negf_block_gemm(ctx, P.MIXED, A, B, D, op[0], op[1], alpha, beta, C)
        assert ctx.sync() == 0
    finally:
        ctx.close()
    big = lambda x, d: torch.maximum(x.real.abs(), x.imag.abs()).amax(d, keepdim=True)  # noqa: E731
    bound = abs(alpha) * n * 2.0 ** -50 * big(a, -1) * big(b, -2)
    if C is not None:
        bound = bound + 2.0 ** -51 * abs(beta) * C.abs()
    assert bool(((D - ref).abs() <= bound).all())


def _rand(shape, seed, spread=0.0):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randn(*shape, dtype=torch.complex128, device="cuda", generator=g)
    if spread:
        x = x * 10.0 ** (spread * (torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g) - 0.5))
    return x


@pytest.mark.parametrize("n,units", [(16, 1), (16, 400), (17, 3), (31, 40), (32, 320), (33, 2), (48, 100), (63, 90), (96, 60),
                                     (113, 5), (127, 45), (128, 1), (128, 80), (129, 2), (144, 30), (200, 3), (255, 9),
                                     (257, 2), (384, 2), (500, 3), (512, 1)])
@pytest.mark.parametrize("op", [(0, 0), (2, 0), (0, 2), (2, 2)])
def test_edges(P, n, units, op):
    A, B, C = _rand((units, n, n), n), _rand((units, n, n), n + 1), _rand((units, n, n), n + 2)
    _check(P, A, B, C, op, -1.0, 1.0)


@pytest.mark.parametrize("n", [40, 128, 300])
def test_scales_and_general_factors(P, n):
    A, B, C = _rand((5, n, n), 1, 12.0), _rand((5, n, n), 2, 12.0), _rand((5, n, n), 3)
    A[1, 3] = 0.0            # a zero row and a zero column
    B[2, :, 5] = 0.0
    _check(P, A, B, None, (0, 0), 0.5 - 2.0j, 0.0)
    _check(P, A, B, C, (0, 2), 1.0, -1.0)


@pytest.mark.parametrize("n", [32, 128, 256])
@pytest.mark.parametrize("value", [254.0 / 255.0, 1.0, 127.0 / 128.0])
def test_equal_entries_fill_the_accumulators(P, n, value):
    """Every digit at its largest with one sign: the largest group sums the scheme admits.  The
    reference is exact (a complex128 product of equal entries rounds every addition one way)."""
    A = torch.full((2, n, n), value, dtype=torch.complex128, device="cuda") * (1 + 1j)
    B = torch.full((2, n, n), value, dtype=torch.complex128, device="cuda") * (1 - 1j)
    _check(P, A, B, None, (0, 0), 1.0, 0.0, ref=complex(float(2 * n * Fraction(value) ** 2), 0.0))


def test_in_place_accumulation(P):
    A, B, C = _rand((3, 100, 100), 4), _rand((3, 100, 100), 5), _rand((3, 100, 100), 6)
    want = A @ B + C
    D = C.clone()
    ctx = P.Context(0, 1 << 28)
    try:
        P.negf.negf_block_gemm(ctx, P.MIXED, A, B, D, 0, 0, 1.0, 1.0, D)
        assert ctx.sync() == 0
    finally:
        ctx.close()
    assert float((D - want).abs().max()) <= 100 * 2.0 ** -50 * float(A.abs().max() * B.abs().max())
