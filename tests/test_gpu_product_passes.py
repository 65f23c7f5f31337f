"""The byte-digit product over several exact passes (n > 128): the passes' 64-bit sums lose nothing.

Exact inputs: op(A)'s small entries are multiples of 2^-31, op(B)'s of 2^-23, all below 2^-5, and one
entry of 0.75 per row and column, which meets zeros, sets the scales.  Their digits reach s + t
<= 5, so no digit product is left out, every sum is a multiple of 2^-54 below 1/2, and both the
kernel and complex128 have to give it exactly.
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


def _product(P, A, B, op):
    D = torch.empty_like(A)
    ctx = P.Context(0, 1 << 29)
    try:
        P.negf.negf_block_gemm(ctx, P.MIXED, A, B, D, op[0], op[1], 1.0, 0.0, None)
        assert ctx.sync() == 0
    finally:
        ctx.close()
    return D


@pytest.mark.parametrize("n", [40, 128, 129, 200, 256, 257, 384, 400, 512])
@pytest.mark.parametrize("op", [(0, 0), (2, 2)])
def test_exact_inputs_give_exact_results(P, n, op):
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    r = lambda bits, unit: torch.randint(-2 ** bits + 1, 2 ** bits, (3, n, n, 2), device="cuda", generator=g).double() * 2.0 ** unit
    A, B = torch.view_as_complex(r(26, -31)), torch.view_as_complex(r(18, -23))
    A[:, :, n // 3], B[:, n // 3] = 0.75, 0.0
    A[:, :, n // 2], B[:, n // 2] = 0.0, 0.75
    want = A @ B
    H = lambda x, o: x.mH.contiguous() if o else x  # noqa: E731
    D = _product(P, H(A, op[0]), H(B, op[1]), op)
    assert float(torch.view_as_real(want).abs().max()) < 0.5
    assert torch.equal(D, want)


@pytest.mark.parametrize("n", [384, 500, 512])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("value", [254.0 / 255.0, 1.0 - 2.0 ** -53])
def test_sums_past_63_bits(P, n, sign, value):
    """Equal entries, every real product of one sign: the passes' sum goes past 2^63 of its units.  The
    tolerance is that of the scheme (n 2^-50 of the largest entries)."""
    A = torch.full((2, n, n), value, dtype=torch.complex128, device="cuda") * (1 + 1j)
    B = torch.full((2, n, n), sign * value, dtype=torch.complex128, device="cuda") * (1 - 1j)
    A[1, 0] = 0.0
    B[1, :, 1] *= -1.0
    D = _product(P, A, B, (0, 0))
    want = torch.full((2, n, n), float(2 * n * sign * Fraction(value) ** 2), dtype=torch.float64, device="cuda")
    want[1, 0] = 0.0
    want[1, :, 1] *= -1.0
    assert float((D - want).abs().max()) <= n * 2.0 ** -50


def test_the_two_names_of_the_wide_tiles_are_timed_once(P):
    import ctypes as C
    ctx = P.Context(0, 1 << 28)
    try:
        for n, names in ((64, (1, 2, 3)), (200, (3,))):
            choice, ms = C.c_int32(), (C.c_double * 4)()
            ctx.check(ctx.lib.negf_tune_products(ctx.h, n, 32, C.byref(choice), ms, None))
            assert [v for v in range(4) if ms[v] > 0.0] == list(names)
            assert ms[choice.value] == min(ms[v] for v in names)
            if n <= 128:
                assert ms[2] == ms[3] and choice.value != 3
    finally:
        ctx.close()
