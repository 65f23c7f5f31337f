"""The lead solver's decisions (end of the decimation, end of the Stein doubling, balancing)
come from the entries' high words, and from the moduli where those leave the answer open or
the entries are very large or very small.

A Hamiltonian, energies and broadening that are all 2^k times larger have self-energies exactly
2^k times larger: every decision is relative and every operation scales with the power of two.
So the step counts are equal and the results agree to the last bits (1e-12 leaves room for
rounding where an intermediate of 2^k times 1e-190 or less goes below the normal range), on
the side of the bounds (k = 0, 100, -300) and on that of the moduli (k = -410, 1e-124).
"""
import dataclasses

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_03438_gb300 as P
    P.negf.load_library()
    return P


def _solve(P, ctx, dev):
    ne, b = len(dev.energy), dev.H_up.shape[-1]
    sys_ = P.upload([dev])
    z = lambda: torch.empty(ne * b * b, dtype=torch.complex128, device="cuda")
    sL, sR = z(), z()
    status = torch.full((ne,), 9, dtype=torch.int32, device="cuda")
    iters = torch.zeros(2 * ne, dtype=torch.int32, device="cuda")
    P.negf_obc(ctx, sys_, sL, sR, iters, status, prec=P.FP64)
    assert ctx.sync() == 0
    return sL.cpu().numpy(), sR.cpu().numpy(), status.cpu().numpy(), iters.cpu().numpy()


@pytest.mark.parametrize("b", [17, 33, 70])   # one partial round of a CTA, and several
def test_lead_solver_scales_with_powers_of_two(P, b):
    dev = W.banded_device(2, b, 3, b, overlap=False)
    rng = np.random.default_rng(b)
    dev.H_up = dev.H_up + 0.3 / np.sqrt(b) * (rng.normal(size=dev.H_up.shape) + 1j * rng.normal(size=dev.H_up.shape))
    dev.eta = 1e-2
    ctx = P.Context(0, 256 << 20)
    try:
        base = _solve(P, ctx, dev)
        assert base[2].tolist() == [0, 0, 0]
        for k in (100, -300, -410):
            f = 2.0 ** k
            got = _solve(P, ctx, dataclasses.replace(dev, H_diag=dev.H_diag * f, H_up=dev.H_up * f, energy=dev.energy * f,
                                                     eta=dev.eta * f))
            assert got[2].tolist() == [0, 0, 0]
            assert got[3].tolist() == base[3].tolist()
            for x, y in zip(got[:2], base[:2]):
                assert np.abs(x / f - y).max() <= 1e-12 * np.abs(y).max(), k
    finally:
        ctx.close()


@pytest.mark.parametrize("b,ne", [(17, 2), (17, 300), (17, 1030), (40, 260)])
def test_masked_products_of_many_units(P, b, ne):
    """Mixed precision against FP64: the products under a mask take a list of its units, in one
    round of 512 flags, in several, and (more than 2048 units) by skipping.  Both sides meet
    the residual target of 1e-13 that the fixed point amplifies by at most 1 / eta^2 = 1e4."""
    dev = W.banded_device(2, b, ne, b, overlap=False)
    rng = np.random.default_rng(b)
    dev.H_up = dev.H_up + 0.3 / np.sqrt(b) * (rng.normal(size=dev.H_up.shape) + 1j * rng.normal(size=dev.H_up.shape))
    dev.eta = 1e-2
    sys_ = P.upload([dev])
    out = []
    ctx = P.Context(0, 3 << 30)
    try:
        for prec in (P.FP64, P.MIXED):
            z = lambda: torch.empty(ne * b * b, dtype=torch.complex128, device="cuda")
            sL, sR = z(), z()
            status = torch.full((ne,), 9, dtype=torch.int32, device="cuda")
            iters = torch.zeros(2 * ne, dtype=torch.int32, device="cuda")
            P.negf_obc(ctx, sys_, sL, sR, iters, status, prec=prec)
            assert ctx.sync() == 0
            assert int(status.abs().sum()) == 0
            out.append(torch.stack([sL, sR]).view(2, ne, -1))
    finally:
        ctx.close()
    size = out[0].abs().amax(dim=2, keepdim=True)
    assert float(((out[1] - out[0]).abs() / size).max()) <= 2e-9
