"""Sweeps whose workspace holds only some of the energies at a time: every chunk's blocks, statuses and
observables are those of the call in one chunk (the same operations per energy: equal bits)."""
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


def _sweep(P, dev, prec, ws):
    sys_ = P.upload(dev)
    out = P.allocate_outputs(sys_, greater=True)
    ne, b = len(dev.energy), dev.H_up.shape[-1]
    E = torch.from_numpy(dev.energy).cuda()
    sig = ((-0.1j * (2.0 + torch.sin(E)))[:, None, None] * torch.eye(b, dtype=torch.complex128, device="cuda")).reshape(-1)
    f = 0.5 + 0.25 * torch.sin(3.0 * E)
    w = torch.full((ne,), 0.1, dtype=torch.float64, device="cuda")
    ctx = P.Context(0, ws)
    try:
        P.negf.negf_rgf_keldysh(ctx, sys_, prec, sig, sig, f, 1.0 - f, P.Scattering.from_devices(dev), out["GR_diag"],
                                out["GR_up"], out["GR_low"], out["GL_diag"], out["GL_low"], out["GG_diag"], out["GG_low"],
                                out["status"])
        assert ctx.sync() == 0
        P.negf_observables(ctx, sys_, sig, w, out["GR_diag"], out["GR_up"], out["GR_low"], out["GL_diag"], out["GL_low"],
                           out["T"], out["dos"], out["current"], out["density"], prec=prec)
        assert ctx.sync() == 0
    finally:
        ctx.close()
    return out


# workspaces of 3, 3, 2 and 3 energies of the 11
@pytest.mark.parametrize("b,prec,ws", [(8, "FP64", 110 << 10), (16, "MIXED", 450 << 10), (24, "FP64", 450 << 10),
                                       (40, "MIXED", 3 << 20)])
def test_chunks_give_what_one_chunk_gives(P, b, prec, ws):
    dev = W.small_scattering_device(5, b, 11, b)
    dev.eta = 1e-2
    one, some = _sweep(P, dev, getattr(P, prec), 256 << 20), _sweep(P, dev, getattr(P, prec), ws)
    assert int(one["status"].abs().sum()) == 0
    for k in ("GR_diag", "GR_up", "GR_low", "GL_diag", "GL_low", "GG_diag", "GG_low", "status", "T", "dos", "current", "density"):
        assert torch.equal(one[k], some[k]), k
