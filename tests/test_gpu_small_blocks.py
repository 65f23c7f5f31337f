"""Small blocks (b <= 16) in one launch: the open boundary (one CTA per lead unit) and the
sweeps, at the edges of their block sizes, against the CPU oracle.

Tolerances, derived from eta = 1e-2: the surface functions meet their residual target of
1e-13 in a Frobenius norm divided by sqrt(b), and the fixed-point equation amplifies a
residual by at most about |g|/eta, |g| <= 1/eta: 1e-13 * 1e4 = 1e-9 of the largest entry.
The sweeps run in FP64 from the same self-energies, b nb operations deep on blocks with
|G| <= 1/eta: 1e-10 of each family's norm.
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import negf_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2602_03438_gb300 as P
    P.negf.load_library()
    return P


def _device(nb, b, ne, seed, overlap):
    dev = W.banded_device(nb, b, ne, seed, overlap=overlap)
    rng = np.random.default_rng(seed)
    dev.H_up = dev.H_up + 0.3 / np.sqrt(b) * (rng.normal(size=dev.H_up.shape) + 1j * rng.normal(size=dev.H_up.shape))
    dev.eta = 1e-2
    return dev


@pytest.mark.parametrize("b", [1, 2, 3, 5, 8, 9, 13, 15, 16])
@pytest.mark.parametrize("overlap,prec", [(False, "FP64"), (True, "MIXED")])
def test_obc_of_small_blocks(P, b, overlap, prec):
    devs = [_device(3, b, 5, 10 * b + k, overlap) for k in range(2)]
    ctx = P.Context(0, 64 << 20)
    try:
        for group in (devs[:1], devs):   # alone, and as a batch of (device, energy) units
            sys_ = P.upload(group)
            n = 5 * len(group) * b * b
            z = lambda: torch.empty(n, dtype=torch.complex128, device="cuda")
            sL, sR, gL, gR = z(), z(), z(), z()
            status = torch.full((5 * len(group),), 9, dtype=torch.int32, device="cuda")
            iters = torch.zeros(10 * len(group), dtype=torch.int32, device="cuda")
            P.negf_obc(ctx, sys_, sL, sR, iters, status, gs_L=gL, gs_R=gR, prec=getattr(P, prec))
            assert ctx.sync() == 0
            assert int(status.abs().sum()) == 0
            assert int(iters.min()) >= 1
            for k, dev in enumerate(group):
                for e in range(5):
                    rL, rR = O.lead_self_energies(dev, dev.energy[e] + 1j * dev.eta)[:2]
                    for got, ref in ((sL, rL), (sR, rR)):
                        g = got.view(-1, b, b)[5 * k + e].cpu().numpy()
                        assert np.abs(g - ref).max() <= 1e-9 * np.abs(ref).max()
    finally:
        ctx.close()


def test_obc_without_convergence_is_reported(P):
    dev = _device(3, 8, 4, 3, False)
    ctx = P.Context(0, 64 << 20)
    try:
        sys_ = P.upload(dev)
        out = P.allocate_outputs(sys_, lesser=False)
        P.negf_obc(ctx, sys_, out["sigma_L"], out["sigma_R"], out["iters"], out["obc_status"], max_iter=1)
        assert ctx.sync() == 0
        assert out["obc_status"].tolist() == [P.negf.NEGF_ERR_NOCONV] * 4
    finally:
        ctx.close()


@pytest.mark.parametrize("b,nb,prec", [(1, 4, "FP64"), (2, 1, "FP64"), (7, 3, "MIXED"), (9, 2, "FP64"), (16, 4, "FP64"),
                                       (16, 4, "MIXED"), (16, 1, "MIXED")])
def test_sweeps_of_small_blocks(P, b, nb, prec):
    dev = W.small_scattering_device(nb, b, 3, 7 * b + nb)
    dev.eta = 1e-2
    rng = np.random.default_rng(b)
    sig = []
    for _ in range(2):
        q = rng.normal(size=(3, b, b)) + 1j * rng.normal(size=(3, b, b))
        sig.append(-0.1j * q @ np.conj(np.swapaxes(q, -1, -2)) / b)
    ctx = P.Context(0, 64 << 20)
    try:
        sys_ = P.upload(dev)
        out = P.allocate_outputs(sys_)
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        P.negf_rgf_lesser(ctx, sys_, getattr(P, prec), t(sig[0]).view(-1), t(sig[1]).view(-1), t(dev.f_L()), t(dev.f_R()),
                          P.Scattering.from_devices(dev), out["GR_diag"], out["GR_up"], out["GR_low"], out["GL_diag"],
                          out["GL_low"], out["status"])
        assert ctx.sync() == 0
        assert int(out["status"].abs().sum()) == 0
    finally:
        ctx.close()
    scat = dev.sigL_scat_full()
    for e in range(3):
        ref = O.greens_dense(dev, dev.energy[e] + 1j * dev.eta, sig[0][e], sig[1][e], dev.f_L()[e], dev.f_R()[e],
                             dev.sigR_scat, scat[e])
        for key in ("GR_diag", "GL_diag") + (("GR_up", "GR_low", "GL_low") if nb > 1 else ()):
            got = out[key].view(3, -1, b, b)[e].cpu().numpy()
            assert np.linalg.norm(got - ref[key]) <= 1e-10 * np.linalg.norm(ref[key]), (key, e)
