"""The lead solver's FP64 redo of inverses that the refinement leaves open, where every unit needs it at
the first step: energies within 1e-6 of an eigenvalue of the lead's onsite block, eta = 1e-6, and
four orbitals 1000 above the others, a condition number of 1e9.

Every energy is solved in both precisions, checked by the definition: the fixed point's residual,
formed here in complex128, is within the accepted 1e-10 and the rounding of its own formation.
"""
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


@pytest.mark.parametrize("b,ne", [(48, 40), (100, 30), (128, 3), (128, 40)])
def test_every_inverse_redone(P, b, ne):
    dev = W.banded_device(2, b, ne, b, overlap=False)
    rng = np.random.default_rng(b)
    dev.H_up = dev.H_up + 0.3 / np.sqrt(b) * (rng.normal(size=dev.H_up.shape) + 1j * rng.normal(size=dev.H_up.shape))
    q = np.linalg.qr(rng.normal(size=(b, b)) + 1j * rng.normal(size=(b, b)))[0]
    dev.H_diag = dev.H_diag + 1e3 * (q[:, :4] @ q[:, :4].conj().T)
    dev.energy = np.linalg.eigvalsh(dev.H_diag[0])[b // 2] + np.linspace(-1e-6, 1e-6, ne)
    dev.eta = 1e-6
    sys_ = P.upload(dev)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    Z = (t(dev.energy) + 1j * dev.eta)[:, None, None]
    eye = torch.eye(b, dtype=torch.complex128, device="cuda")
    a00, hop = Z * eye - t(dev.H_diag[0]), t(dev.H_up[0])
    ctx = P.Context(0, 1 << 30)
    try:
        for prec in (P.FP64, P.MIXED):
            z = lambda: torch.empty(ne * b * b, dtype=torch.complex128, device="cuda")
            sL, sR, gL, gR = z(), z(), z(), z()
            status = torch.full((ne,), 9, dtype=torch.int32, device="cuda")
            P.negf_obc(ctx, sys_, sL, sR, None, status, gs_L=gL, gs_R=gR, prec=prec)
            assert ctx.sync() == 0
            g = gL.view(ne, b, b)
            K = a00 - hop.mH @ g @ hop
            res = (K @ g - eye).flatten(1).norm(dim=1) / b ** 0.5
            noise = 2.0 ** -53 * b * K.abs().amax(dim=(1, 2)) * g.abs().amax(dim=(1, 2))
            assert int(status.abs().sum()) == 0
            assert bool((res <= 1e-10 + noise).all())
    finally:
        ctx.close()
