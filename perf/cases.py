"""Performance cases of the library: what a transport calculation has it do.

Every case is one call (or the short call sequence of one energy batch) through the public
entry points of ``paper_2602_03438_gb300`` on inputs that ``prepare`` makes on the GPU from
a seed: block-tridiagonal devices of the workloads' recipe (random Hermitian blocks with
entries decaying as exp(-|r - r'|/4), S = I + 0.05 R, the flat / linear / flat potential
of a 0.2 V drop, eta = 1e-6) with a dense inter-slice coupling of 0.3 / sqrt(b) so that
current flows, on uniform energy grids in [-3, 3].

A case is a dict of plain values with a ``kind``:

  product      negf_block_gemm, the batched complex block product
  inverse      negf_block_inverse
  obc          negf_obc: lead self-energies and surface functions
  transport    negf_rgf_lesser + negf_observables on stored blocks
  retarded     negf_rgf_retarded of one device or of an uneven batch of devices
  partitioned  negf_rgf_partitioned: few energies of a long device
  observables  negf_rgf_observables: the observables without stored blocks
  scba         negf_scba: sweeps of the self-consistent scattering loop
  network      negf_mlp_train_step: forward, backward and Adam update of the warm start

``exact`` recomputes a case's outputs in complex128 with plain torch.
"""
import math

import torch

import paper_2602_03438_gb300 as P

PREC = {"fp64": P.FP64, "mixed": P.MIXED}
ETA = 1e-6
KT, MU = 0.025, 0.1
Z = torch.complex128
DEV = "cuda"


def listed():
    return [
        # the open boundary of the small ballistic device (16 blocks of 8, 64 energies): the
        # smallest call a user makes, bound by launches and read-backs
        dict(name="obc_small", kind="obc", prec="fp64", b=8, ne=64, overlap=False),
        # the sweeps and observables of that device, in FP64
        dict(name="transport_small", kind="transport", prec="fp64", nb=16, b=8, ne=64, overlap=False),
        # the block product at the headline block size, one unit per energy, accumulating
        dict(name="product_128", kind="product", prec="mixed", b=128, units=1024, op_a="N", op_b="H", beta=1.0),
        # the diagonal-block inverse of the sweeps
        dict(name="inverse_128", kind="inverse", prec="mixed", b=128, units=512),
        # the open boundary at the headline block size
        dict(name="obc_128", kind="obc", prec="mixed", b=128, ne=192, overlap=True),
        # the headline step: G^R and G^< sweeps and observables, with scattering
        dict(name="transport_128", kind="transport", prec="mixed", nb=12, b=128, ne=256, overlap=True),
        # the full-precision sweeps at a middle block size
        dict(name="transport_fp64", kind="transport", prec="fp64", nb=8, b=40, ne=96, overlap=True),
        # an uneven batch of devices in one call, ragged block sizes among them
        dict(name="retarded_uneven", kind="retarded", prec="mixed",
             devices="9x32x40,13x32x24,11x64x48,8x100x33,10x128x20,14x64x16,8x200x12,9x256x8", overlap=True),
        # few energies of a long device, split over partitions
        dict(name="partitioned_64", kind="partitioned", prec="mixed", nb=64, b=128, ne=4, parts=8, overlap=True),
        # the largest blocks: observables of a scattering device without stored blocks
        dict(name="observables_512", kind="observables", prec="mixed", nb=6, b=512, ne=16, overlap=True),
        # two sweeps of the self-consistent scattering loop
        dict(name="scba_16", kind="scba", prec="mixed", nb=8, b=16, ne=256, steps=8, sweeps=2, overlap=True),
        # one training step of the open boundary's warm-start network on a minibatch
        dict(name="network_64", kind="network", b=64, hidden=512, n=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: each kind over its range, block sizes odd and ragged included."""
    kind = rng.choice(["product", "product", "inverse", "obc", "obc", "transport", "transport", "retarded",
                       "partitioned", "observables", "scba", "network"])
    prec = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    if kind in ("product", "inverse"):
        b = _log_int(rng, 8, 96 if prec == "fp64" else 512)
        units = max(1, min(2048, int(_log_int(rng, 2 ** 14, 2 ** 24) / (b * b))))
        if kind == "inverse":
            return dict(kind=kind, prec=prec, b=min(b, 256), units=min(units, 1024))
        return dict(kind=kind, prec=prec, b=b, units=units, op_a=rng.choice("NH"), op_b=rng.choice("NH"),
                    beta=rng.choice([0.0, 1.0]))
    if kind == "obc":
        b = _log_int(rng, 4, 16 if prec == "fp64" else 160)
        return dict(kind=kind, prec=prec, b=b, ne=max(8, min(256, int(_log_int(rng, 2 ** 14, 2 ** 21) / (b * b)))),
                    overlap=rng.random() < 0.5)
    if kind in ("transport", "observables"):
        b = _log_int(rng, 4, 48 if prec == "fp64" else 288)
        nb = rng.randint(3, 16)
        ne = max(4, min(256, int(_log_int(rng, 2 ** 16, 2 ** 25) / (b * b * nb))))
        return dict(kind=kind, prec=prec, nb=nb, b=b, ne=ne, overlap=rng.random() < 0.7)
    if kind == "retarded":
        devs = []
        for _ in range(rng.randint(1, 6)):
            b = rng.choice([32, 64, 96, 128, 192, 256, 100, 24])
            devs.append("%dx%dx%d" % (rng.randint(4, 16), b, max(2, min(64, _log_int(rng, 2 ** 13, 2 ** 18) // (b * b)))))
        return dict(kind=kind, prec="mixed", devices=",".join(devs), overlap=True)
    if kind == "partitioned":
        parts = rng.choice([2, 4, 8])
        return dict(kind=kind, prec="mixed", nb=parts * rng.randint(2, 8), b=_log_int(rng, 24, 160), ne=rng.randint(1, 6),
                    parts=parts, overlap=True)
    if kind == "scba":
        return dict(kind=kind, prec=rng.choice(["mixed", "fp64"]), nb=rng.randint(3, 10), b=rng.choice([8, 12, 16, 24]),
                    ne=rng.randint(64, 300), steps=rng.randint(3, 16), sweeps=rng.randint(1, 3), overlap=True)
    return dict(kind="network", b=rng.choice([8, 16, 32, 64]), hidden=rng.choice([128, 256, 512]), n=rng.randint(64, 512))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _cn(g, *shape):
    return torch.randn(*shape, dtype=Z, device=DEV, generator=g)   # E|x|^2 = 1


def _herm(x):
    return 0.5 * (x + x.mH)


def _potential(nb, dv=0.2):
    q = nb / 4.0
    v = []
    for i in range(nb):
        x = i + 0.5
        v.append(0.5 * dv if x <= q else -0.5 * dv if x >= nb - q else 0.5 * dv - dv * (x - q) / (nb - 2.0 * q))
    return torch.tensor(v, dtype=Z, device=DEV)


def _device(g, nb, b, overlap):
    """H and S blocks of one device: [nb][b][b] and [nb-1][b][b]."""
    r = torch.arange(b, device=DEV, dtype=torch.float64)
    d0 = torch.exp(-(r[:, None] - r[None, :]).abs() / 4.0) / math.sqrt(b)
    d1 = torch.exp(-(b + r[None, :] - r[:, None]) / 4.0) / math.sqrt(b)
    eye = torch.eye(b, dtype=Z, device=DEV)
    Hd = _herm(_cn(g, nb, b, b)) * d0 + _potential(nb)[:, None, None] * eye
    Hu = _cn(g, nb - 1, b, b) * d1 + 0.3 / math.sqrt(b) * _cn(g, nb - 1, b, b)
    if not overlap:
        return Hd, Hu, None, None
    return Hd, Hu, eye + 0.05 * _herm(_cn(g, nb, b, b)) * d0, 0.05 * _cn(g, nb - 1, b, b) * d1


def _lead_sigma(g, E, b):
    """A retarded lead self-energy per energy, of a contact with a smooth spectrum:
    0.1 R - i 0.2 Q Q^H / b scaled smoothly over the energy."""
    R, Q = _herm(_cn(g, b, b)) / math.sqrt(b), _cn(g, b, b)
    S = 0.1 * R - 0.2j * (Q @ Q.mH) / b
    return ((1.0 + 0.3 * torch.sin(E))[:, None, None] * S).contiguous()


def _fermi(E, mu):
    return 0.5 * (1.0 - torch.tanh(0.5 * (E - mu) / KT))


def _scattering(g, E, nb, b):
    """Block-diagonal scattering of strength 0.01: Sigma^R = 0.01 R - i P, Sigma^< = 2 i f P."""
    R, Q = _herm(_cn(g, nb, b, b)) / math.sqrt(b), _cn(g, nb, b, b)
    Pm = 0.01 * (Q @ Q.mH) / b
    mu = MU - 2 * MU * (torch.arange(nb, device=DEV, dtype=torch.float64) + 0.5) / nb
    return 0.01 * R - 1j * Pm, 2j * Pm, _fermi(E[:, None], mu[None, :]).contiguous()


def _grid(ne, lim=3.0):
    return torch.linspace(-lim, lim, ne, dtype=torch.float64, device=DEV)


def _weights(E):
    w = torch.full_like(E, float(E[1] - E[0]) if E.numel() > 1 else 1.0)
    if E.numel() > 1:
        w[0] *= 0.5
        w[-1] *= 0.5
    return w


def _shapes(case):
    if "devices" in case:
        return [tuple(int(x) for x in d.split("x")) for d in case["devices"].split(",")]
    return [(case.get("nb", 2), case["b"], case["ne"])]


def _inputs(case, seed):
    """Tensors of a case, made from the seed alone (both sides of a comparison and exact use them)."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    kind, b = case["kind"], case.get("b")
    if kind == "product":
        n, u = b, case["units"]
        return dict(A=_cn(g, u, n, n), B=_cn(g, u, n, n) / math.sqrt(n),
                    C=_cn(g, u, n, n) if case["beta"] else None)
    if kind == "inverse":
        n, u = b, case["units"]
        E = torch.rand(u, 1, 1, dtype=torch.float64, device=DEV, generator=g) * 6.0 - 3.0
        Q = _cn(g, u, n, n)
        eye = torch.eye(n, dtype=Z, device=DEV)
        return dict(M=(E + 1j * ETA) * eye - _herm(_cn(g, u, n, n)) / math.sqrt(n) + 0.1j * (Q @ Q.mH) / n)
    if kind == "network":
        d = P.negf.negf_mlp_get_dims(b, case["hidden"])
        n, rows, hid = case["n"], P.negf.mlp_rows(case["n"]), case["hidden"]
        f = dict(device=DEV, generator=g)
        p = torch.zeros(d.n_params, device=DEV)
        W1 = (torch.rand(hid, d.k0p, **f) * 2 - 1) * math.sqrt(6.0 / d.k0)
        W1[:, d.k0:] = 0
        p[d.off_W1:d.off_c1] = W1.reshape(-1)
        p[d.off_W2:d.off_c2] = ((torch.rand(hid * hid, **f) * 2 - 1) * math.sqrt(6.0 / hid))
        p[d.off_W3:d.off_c3] = ((torch.rand(d.nout * hid, **f) * 2 - 1) * 0.1 * math.sqrt(6.0 / hid))
        X = torch.zeros(rows, d.k0p, dtype=torch.bfloat16, device=DEV)
        X[:n, :d.k0] = torch.randn(n, d.k0, **f).to(torch.bfloat16)
        return dict(params=p, m=1e-5 * torch.randn(d.n_params, **f), v=1e-8 * (0.1 + torch.rand(d.n_params, **f)),
                    X=X, G=_cn(g, n, b, b), dims=d)
    out = []
    for nb, bb, ne in _shapes(case):
        E = _grid(ne, 4.5 if kind == "scba" else 3.0)
        Hd, Hu, Sd, Su = _device(g, nb, bb, case["overlap"])
        one = dict(nb=nb, b=bb, ne=ne, E=E, Hd=Hd, Hu=Hu, Sd=Sd, Su=Su)
        if kind != "obc":
            one["sL"], one["sR"] = _lead_sigma(g, E, bb), _lead_sigma(g, E, bb)
            one["fL"], one["fR"], one["w"] = _fermi(E, MU), _fermi(E, -MU), _weights(E)
            if kind in ("transport", "observables"):
                one["scR"], one["scL"], one["scale"] = _scattering(g, E, nb, bb)
        out.append(one)
    return dict(devs=out)


def _kernel(case, E):
    """An Einstein boson of ``steps`` grid steps: (w_less, w_great), entry 0 is m = -steps."""
    st, g2 = case["steps"], 0.01
    n = 1.0 / math.expm1(st * float(E[1] - E[0]) / KT)
    wl, wg = [0.0] * (2 * st + 1), [0.0] * (2 * st + 1)
    wl[2 * st], wl[0] = g2 * n, g2 * (n + 1.0)
    wg[2 * st], wg[0] = g2 * (n + 1.0), g2 * n
    return wl, wg


def prepare(case, seed):
    """The device-resident inputs, outputs and library context a program holds."""
    i = _inputs(case, seed)
    kind = case["kind"]
    s = dict(case=case, i=i, prec=PREC.get(case.get("prec")))
    if kind == "product":
        s.update(ctx=P.Context(0, _product_bytes(case)), D=torch.empty_like(i["A"]),
                 op=tuple(2 if case[k] == "H" else 0 for k in ("op_a", "op_b")))
        return s
    if kind == "inverse":
        s.update(ctx=P.Context(0, 2 * _product_bytes(case)), X=torch.empty_like(i["M"]),
                 status=torch.zeros(case["units"], dtype=torch.int32, device=DEV))
        return s
    if kind == "network":
        need = P.negf.negf_mlp_workspace_bytes(i["dims"], case["n"])
        s.update(ctx=P.Context(0, need + (1 << 20)), grad=torch.empty_like(i["params"]),
                 p=i["params"].clone(), m=i["m"].clone(), v=i["v"].clone(),
                 loss=torch.zeros(1, dtype=torch.float64, device=DEV))
        return s
    devs = i["devs"]
    cat = lambda k: None if devs[0].get(k) is None else torch.cat([d[k].reshape(-1) for d in devs])  # noqa: E731
    sy = P.System([d["nb"] for d in devs], [d["b"] for d in devs], [d["ne"] for d in devs], cat("Hd"), cat("Hu"),
                  cat("Sd"), cat("Su"), cat("E"), ETA)
    s.update(sys=sy, out=P.allocate_outputs(sy, lesser=kind not in ("obc", "retarded", "partitioned"),
                                            greater=kind == "scba"))
    for k in ("sL", "sR", "fL", "fR", "w"):
        s[k] = cat(k)
    blk = max(16 * d["b"] ** 2 * d["ne"] * (d["nb"] + 24) for d in devs)
    if kind == "obc":
        s.update(gL=torch.empty_like(s["out"]["sigma_L"]), gR=torch.empty_like(s["out"]["sigma_L"]))
        ws = 2 * 40 * blk // 26
    elif kind == "observables":
        s["out"] = {k: v for k, v in s["out"].items() if k in ("T", "dos", "current", "density", "status")}
        ws = 8 * blk
    else:
        ws = 6 * blk
    if kind in ("transport", "observables"):
        s["scat"] = P.Scattering(cat("scR"), cat("scL"), cat("scale"), False)
    if kind == "scba":
        wl, wg = _kernel(case, devs[0]["E"])
        n = sum(d["ne"] * d["nb"] * d["b"] ** 2 for d in devs)
        s.update(w_lesser=wl, w_greater=wg, sig=[torch.zeros(n, dtype=Z, device=DEV) for _ in range(3)])
        ws += 64 * n
    s["ctx"] = P.Context(0, max(64 << 20, min(24 << 30, ws)))
    return s


def _product_bytes(case):
    n, u = case["b"], case["units"]
    n = (n + 127) // 128 * 128
    return (64 << 20) + u * n * n * 16 * 6


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    case, i, ctx, prec = s["case"], s["i"], s["ctx"], s["prec"]
    kind = case["kind"]
    if kind == "product":
        P.negf.negf_block_gemm(ctx, prec, i["A"], i["B"], s["D"], s["op"][0], s["op"][1], 1.0, case["beta"], i["C"])
        return s["D"]
    if kind == "inverse":
        P.negf.negf_block_inverse(ctx, prec, i["M"], s["X"], s["status"])
        return [s["X"], s["status"]]
    if kind == "network":
        for k, src in (("p", "params"), ("m", "m"), ("v", "v")):
            s[k].copy_(i[src])
        P.negf.negf_mlp_train_step(ctx, i["dims"], s["p"], s["m"], s["v"], s["grad"], 3, 1e-3, case["n"], i["X"],
                                   i["G"], s["loss"])
        return dict(loss=s["loss"], grad=s["grad"], params=s["p"], m=s["m"], v=s["v"])
    sy, o = s["sys"], s["out"]
    if kind == "obc":
        P.negf_obc(ctx, sy, o["sigma_L"], o["sigma_R"], status=o["obc_status"], gs_L=s["gL"], gs_R=s["gR"], prec=prec)
        return dict(sigma_L=o["sigma_L"], sigma_R=o["sigma_R"], gs_L=s["gL"], gs_R=s["gR"], status=o["obc_status"])
    if kind == "transport":
        P.negf_rgf_lesser(ctx, sy, prec, s["sL"], s["sR"], s["fL"], s["fR"], s["scat"], o["GR_diag"], o["GR_up"],
                          o["GR_low"], o["GL_diag"], o["GL_low"], o["status"])
        P.negf_observables(ctx, sy, s["sL"], s["w"], o["GR_diag"], o["GR_up"], o["GR_low"], o["GL_diag"], o["GL_low"],
                           o["T"], o["dos"], o["current"], o["density"], prec=prec)
        return {k: o[k] for k in ("GR_diag", "GR_up", "GR_low", "GL_diag", "GL_low", "T", "dos", "current", "density",
                                  "status")}
    if kind == "retarded":
        P.negf_rgf_retarded(ctx, sy, prec, s["sL"], s["sR"], None, o["GR_diag"], o["GR_up"], o["GR_low"], o["status"])
    elif kind == "partitioned":
        P.negf_rgf_partitioned(ctx, sy, prec, case["parts"], s["sL"], s["sR"], None, o["GR_diag"], o["GR_up"],
                               o["GR_low"], o["status"])
    if kind in ("retarded", "partitioned"):
        return {k: o[k] for k in ("GR_diag", "GR_up", "GR_low", "status")}
    if kind == "observables":
        P.negf.negf_rgf_observables(ctx, sy, prec, s["sL"], s["sR"], s["fL"], s["fR"], s["scat"], s["w"], o["T"],
                                    o["dos"], o["current"], o["density"], o["status"])
        return dict(o)
    for t in s["sig"]:   # a cold start of the loop
        t.zero_()
    it, change = P.negf.negf_scba(ctx, sy, prec, s["sL"], s["sR"], s["fL"], s["fR"], s["w_lesser"], s["w_greater"],
                                  s["sig"][0], s["sig"][1], s["sig"][2], o["GR_diag"], o["GL_diag"], o["GG_diag"],
                                  o["GR_up"], o["GR_low"], o["GL_low"], o["GG_low"], o["status"], mixing=0.5,
                                  tol=1e-30, max_iter=case["sweeps"])
    return dict(sigR=s["sig"][0], sigL=s["sig"][1], sigG=s["sig"][2], GR_diag=o["GR_diag"], GL_diag=o["GL_diag"],
                GG_diag=o["GG_diag"], GL_low=o["GL_low"], GG_low=o["GG_low"], sweeps=it, change=change)


def work(case):
    """Bytes in and out once, and the useful real operations (8 n^3 per complex block product
    or inverse; the textbook block recursions)."""
    kind = case["kind"]
    if kind in ("product", "inverse"):
        n, u = case["b"], case["units"]
        ops = 3 if kind == "product" and case["beta"] else 2 if kind == "product" else 1
        return dict(bytes=16.0 * n * n * u * (ops + 1), flops=8.0 * n ** 3 * u)
    if kind == "network":
        b, h, n = case["b"], case["hidden"], case["n"]
        k0, nout = 3 * b * b + 65, 2 * b * b
        p = h * k0 + h * h + nout * h
        return dict(bytes=4.0 * p * 7 + 2.0 * n * k0 + 16.0 * n * b * b, flops=2.0 * n * (3 * p - h * k0))
    by = fl = 0.0
    for nb, b, ne in _shapes(case):
        blk, n3 = 16.0 * b * b, 8.0 * b ** 3
        if kind == "obc":
            by += blk * (4 + 4 * ne)
            fl += n3 * ne * 2 * 7 * 12       # about a dozen decimation steps of six products and an inverse
            continue
        src = blk * (4 * nb + 2 * ne)
        if kind in ("retarded", "partitioned"):
            by += src + blk * ne * (3 * nb)
            fl += n3 * ne * nb * 7
        elif kind == "transport":
            by += src + blk * (2 * nb + ne * 5 * nb)
            fl += n3 * ne * nb * 16
        elif kind == "observables":
            by += src + blk * 2 * nb
            fl += n3 * ne * nb * 16
        else:
            by += src + blk * ne * nb * 8 * case["sweeps"]
            fl += n3 * ne * nb * 25 * case["sweeps"]
    return dict(bytes=by, flops=fl)


# ---------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ---------------------------------------------------------------------------

def _sweep(d, scR=None, sig=()):
    """G^R blocks and, per Sigma^x in ``sig`` ([ne][nb][b][b], block-diagonal, leads included),
    the diagonal and lower blocks of G^x: the block recursions over all energies at once."""
    nb, z = d["nb"], (d["E"] + 1j * ETA)[:, None, None]
    eye = torch.eye(d["b"], dtype=Z, device=DEV)
    S = (lambda i: eye) if d["Sd"] is None else (lambda i: d["Sd"][i])
    A = []
    for i in range(nb):
        a = z * S(i) - d["Hd"][i]
        if scR is not None:
            a = a - (scR[i] if scR.dim() == 3 else scR[:, i])
        if i == 0:
            a = a - d["sL"]
        if i == nb - 1:
            a = a - d["sR"]
        A.append(a)
    up = [(0 if d["Su"] is None else z * d["Su"][i]) - d["Hu"][i] for i in range(nb - 1)]
    lo = [(0 if d["Su"] is None else z * d["Su"][i].mH) - d["Hu"][i].mH for i in range(nb - 1)]
    g, gx = [torch.linalg.inv(A[0])], [[] for _ in sig]
    for x, s in enumerate(sig):
        gx[x].append(g[0] @ s[:, 0] @ g[0].mH)
    for i in range(1, nb):
        g.append(torch.linalg.inv(A[i] - lo[i - 1] @ g[i - 1] @ up[i - 1]))
        for x, s in enumerate(sig):
            gx[x].append(g[i] @ (s[:, i] + lo[i - 1] @ gx[x][i - 1] @ lo[i - 1].mH) @ g[i].mH)
    G, U, L = [None] * nb, [None] * (nb - 1), [None] * (nb - 1)
    X = [([None] * nb, [None] * (nb - 1)) for _ in sig]
    G[-1] = g[-1]
    for x in range(len(sig)):
        X[x][0][-1] = gx[x][-1]
    for i in range(nb - 2, -1, -1):
        gu, lg = g[i] @ up[i], lo[i] @ g[i]
        U[i], L[i] = -gu @ G[i + 1], -G[i + 1] @ lg
        G[i] = g[i] - U[i] @ lg
        for x in range(len(sig)):
            q, pl = lo[i] @ gx[x][i], X[x][0][i + 1] @ gu.mH
            w = U[i] @ q
            X[x][0][i] = gx[x][i] + gu @ pl - w + w.mH
            X[x][1][i] = -G[i + 1] @ q - pl
    st = lambda v: torch.stack(v, 1) if v else None  # noqa: E731
    return st(G), st(U), st(L), [(st(a), st(c)) for a, c in X]


def _lead_terms(d, greater=False):
    """The leads' Sigma^< (or Sigma^>) on the block diagonal."""
    s = torch.zeros(d["ne"], d["nb"], d["b"], d["b"], dtype=Z, device=DEV)
    for i, sg, f in ((0, d["sL"], d["fL"]), (d["nb"] - 1, d["sR"], d["fR"])):
        f = (1.0 - f) if greater else -f
        s[:, i] += f[:, None, None] * (sg - sg.mH)
    return s


def _transport(d):
    sig = _lead_terms(d) + d["scale"][:, :, None, None] * d["scL"][None]
    G, U, L, ((Gl, Ll),) = _sweep(d, d["scR"], (sig,))
    z = (d["E"] + 1j * ETA)[:, None, None, None]
    tr = lambda a, c: (a * c.transpose(-1, -2)).sum((-1, -2))  # noqa: E731  Tr[a c]
    gam, g0 = 1j * (d["sL"] - d["sL"].mH), G[:, 0]
    T = (tr(gam, 1j * (g0 - g0.mH)) - tr(gam @ g0, gam @ g0.mH)).real
    if d["Sd"] is None:
        dos, lap = torch.diagonal(G, dim1=-2, dim2=-1).sum((-1, -2)), torch.diagonal(Gl, dim1=-2, dim2=-1)
    else:
        dos = tr(G, d["Sd"][None]).sum(1) + (tr(U, d["Su"].mH[None]) + tr(L, d["Su"][None])).sum(1)
        lap = torch.diagonal(Gl @ d["Sd"], dim1=-2, dim2=-1).clone()
        lap[:, 1:] += torch.diagonal(Ll @ d["Su"], dim1=-2, dim2=-1)
        lap[:, :-1] += torch.diagonal(-Ll.mH @ d["Su"].mH, dim1=-2, dim2=-1)
    cur = 2.0 * tr((d["Hu"] - (0 if d["Su"] is None else z * d["Su"])).expand(d["ne"], -1, -1, -1), Ll).real
    den = (d["w"][:, None, None] * (-1j * lap).real).sum(0) / (2.0 * math.pi)
    return G, U, L, Gl, Ll, T, -dos.imag / math.pi, cur, den


def _surface(a00, al, be):
    """Surface Green's function by decimation and two Newton steps, in complex128."""
    inv = torch.linalg.inv
    e, s, a, c = a00, a00, al, be
    for _ in range(40):
        g = inv(e)
        ag, cg = a @ g, c @ g
        x = ag @ c
        s, e, a, c = s - x, e - x - cg @ a, ag @ a, cg @ c
        if max(float(a.abs().max()), float(c.abs().max())) < 1e-16:
            break
    g = inv(s)
    for _ in range(2):
        k = a00 - al @ g @ be
        ki = inv(k)
        p, q = ki @ al, be @ g
        d = -(g - ki)
        for _ in range(30):
            d, p, q = d + p @ d @ q, p @ p, q @ q
        g = g + d
    return g


def _adam(p, m, v, g, t, lr):
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    return p - lr * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8), m, v


def exact(case, seed):
    i, kind = _inputs(case, seed), case["kind"]
    if kind == "product":
        h = lambda k, x: x.mH if case[k] == "H" else x  # noqa: E731
        r = h("op_a", i["A"]) @ h("op_b", i["B"])
        return r + i["C"] if i["C"] is not None else r
    if kind == "inverse":
        return [torch.linalg.inv(i["M"]), None]
    if kind == "network":
        d, n = i["dims"], case["n"]
        p = i["params"].double().requires_grad_()
        at = lambda a, c, *sh: p[a:c].view(*sh)  # noqa: E731
        X = i["X"][:n].double()
        h = torch.relu(X @ at(d.off_W1, d.off_c1, d.hidden, d.k0p).T + p[d.off_c1:d.off_W2])
        h = torch.relu(h @ at(d.off_W2, d.off_c2, d.hidden, d.hidden).T + p[d.off_c2:d.off_W3])
        y = h @ at(d.off_W3, d.off_c3, d.nout, d.hidden).T + p[d.off_c3:]
        G = i["G"].reshape(n, -1)
        loss = ((y - torch.cat([G.real, G.imag], 1)) ** 2).mean()
        (gr,) = torch.autograd.grad(loss, p)
        p2, m, v = _adam(p.detach(), i["m"].double(), i["v"].double(), gr, 3, 1e-3)
        return dict(loss=loss.detach().view(1), grad=gr, params=p2, m=m, v=v)
    devs = i["devs"]
    if kind == "obc":
        (d,) = devs
        z = (d["E"] + 1j * ETA)[:, None, None]
        o = {}
        for side, cd, cu in (("L", 0, 0), ("R", -1, -1)):
            S = torch.eye(d["b"], dtype=Z, device=DEV) if d["Sd"] is None else d["Sd"][cd]
            a00 = z * S - d["Hd"][cd]
            a01 = (0 if d["Su"] is None else z * d["Su"][cu]) - d["Hu"][cu].expand(d["ne"], -1, -1)
            a10 = (0 if d["Su"] is None else z * d["Su"][cu].mH) - d["Hu"][cu].mH.expand(d["ne"], -1, -1)
            al, be = (a10, a01) if side == "L" else (a01, a10)
            gs = _surface(a00, al, be)
            o["gs_" + side], o["sigma_" + side] = gs.reshape(-1), (al @ gs @ be).reshape(-1)
        return dict(o, status=None)
    flat = lambda v: torch.cat([x.reshape(-1) for x in v])  # noqa: E731
    if kind in ("retarded", "partitioned"):
        r = [_sweep(d)[:3] for d in devs]
        return dict(GR_diag=flat([x[0] for x in r]), GR_up=flat([x[1] for x in r]), GR_low=flat([x[2] for x in r]),
                    status=None)
    (d,) = devs
    if kind in ("transport", "observables"):
        names = ("GR_diag", "GR_up", "GR_low", "GL_diag", "GL_low", "T", "dos", "current", "density")
        r = {k: x.reshape(-1) for k, x in zip(names, _transport(d))}
        if kind == "observables":
            r = {k: r[k] for k in ("T", "dos", "current", "density")}
        return dict(r, status=None)
    wl, wg = _kernel(case, d["E"])
    st, ne = case["steps"], d["ne"]
    sl = torch.zeros(ne, d["nb"], d["b"], d["b"], dtype=Z, device=DEV)
    sg, sr = sl.clone(), sl.clone()

    def conv(x, w):
        y = torch.zeros_like(x)
        y[st:] += w[2 * st] * x[:ne - st]
        y[:ne - st] += w[0] * x[st:]
        return y

    for _ in range(case["sweeps"]):
        sc_g = sl + sr - sr.mH
        G, _, _, ((Gl, Ll), (Gg, Lg)) = _sweep(d, sr, (_lead_terms(d) + sl, _lead_terms(d, True) + sc_g))
        nl, ng = conv(Gl, wl), conv(Gg, wg)
        ch = max(float((nl - sl).abs().max()), float((ng - sg).abs().max())) / max(float(nl.abs().max()),
                                                                                  float(ng.abs().max()))
        sl, sg = sl + 0.5 * (nl - sl), sg + 0.5 * (ng - sg)
        sr = 0.5 * (sg - sl)
    f = lambda x: x.reshape(-1)  # noqa: E731
    return dict(sigR=f(sr), sigL=f(sl), sigG=f(sg), GR_diag=f(G), GL_diag=f(Gl), GG_diag=f(Gg), GL_low=f(Ll),
                GG_low=f(Lg), sweeps=None, change=ch)
