"""The sweeps of small blocks in workspaces below what the one launch needs for one energy: b < 16 is
refused (NEGF_ERR_NOMEM), b = 16 in NEGF_MIXED runs step by step, as in a workspace with room to 1e-9 (a
different order of operations on blocks with |G| <= 1 / eta = 100, and products of FP64 class).
"""
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
    out = P.allocate_outputs(sys_)
    ne, b = len(dev.energy), dev.H_up.shape[-1]
    sig = (-0.1j * torch.eye(b, dtype=torch.complex128, device="cuda")).repeat(ne, 1, 1).view(-1)
    f = torch.full((ne,), 0.5, dtype=torch.float64, device="cuda")
    ctx = P.Context(0, ws)
    try:
        P.negf_rgf_lesser(ctx, sys_, prec, sig, sig, f, f, None, out["GR_diag"], out["GR_up"], out["GR_low"],
                          out["GL_diag"], out["GL_low"], out["status"])
        assert ctx.sync() == 0
    finally:
        ctx.close()
    return out


def _device(b):
    dev = W.banded_device(40, b, 3, b, overlap=True)
    dev.eta = 1e-2
    return dev


# one energy of 40 blocks takes about 200 blocks in the one launch and 47 step by step
@pytest.mark.parametrize("b,prec", [(8, "FP64"), (8, "MIXED"), (15, "MIXED"), (16, "FP64")])
def test_too_small_a_workspace_is_refused(P, b, prec):
    with pytest.raises(P.negf.NegfError) as e:
        _sweep(P, _device(b), getattr(P, prec), 100 * 16 * b * b)
    assert e.value.code == P.negf.NEGF_ERR_NOMEM


def test_blocks_of_16_in_mixed_precision_still_run(P):
    dev = _device(16)
    a, b = _sweep(P, dev, P.MIXED, 64 << 20), _sweep(P, dev, P.MIXED, 700 << 10)
    for k in ("GR_diag", "GR_up", "GR_low", "GL_diag", "GL_low"):
        assert float((a[k] - b[k]).abs().max()) <= 1e-9 * float(a[k].abs().max())
