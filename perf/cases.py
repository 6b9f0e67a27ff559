"""Workloads of the NTU library whose speed and accuracy matter to its users.

Each case is one call form of the public binding (``paper_2107_06635_gb300.ntu``):

* ``cell``    one second-order Trotter step of the two-site unit cell
              (``Context.set_state / step / measure / get_state``), the loop
              body of a quench or thermal run: latency of four bond updates
              that depend on one another;
* ``su``      the same step with the simple update (``Context.su_step``);
* ``batch``   independent bond updates of one kind (D, r) on device arrays
              (``Context.batch_update_dev``);
* ``uneven``  independent bond updates of mixed kinds on host arrays, replayed
              as one CUDA graph (``UnevenBatch.update``).

``exact`` is the same mathematics in plain 64-bit torch, without the library.
"""
import math

import numpy as np
import torch

from paper_2107_06635_gb300 import inputs as I
from paper_2107_06635_gb300 import ntu

PRECISION = {"fp64": ntu.NTU_FP64, "fp32": ntu.NTU_MIXED_FP32, "bf16x3": ntu.NTU_MIXED_BF16X3}
# candidate pseudo-inverse tolerances 10^-k: the full grid in FP64, and the
# grid that the single-precision metrics can resolve
TAU_KMAX = {"fp64": 15, "fp32": 8, "bf16x3": 8}
SWEEPS = 10
UNEVEN_SWEEPS = 8

_stream = None


def listed():
    return [
        # the smallest call: one Trotter step at D = 3 in the default precision
        {"name": "cell_d3_fp64", "kind": "cell", "model": "zz", "D": 3, "precision": "fp64"},
        # a step of a transverse-field quench with the observable read back, mixed precision
        {"name": "cell_quench_d6_bf16x3", "kind": "cell", "model": "quench", "D": 6, "precision": "bf16x3"},
        # a step of an imaginary-time purification run (ancilla dimension 2), FP64
        {"name": "cell_thermal_d5_fp64", "kind": "cell", "model": "thermal", "D": 5, "precision": "fp64"},
        # a step of a real iPEPO thermal run: physical dimension 4, gate rank 4
        {"name": "cell_ipepo_d4_bf16x3", "kind": "cell", "model": "ipepo", "D": 4, "precision": "bf16x3"},
        # a simple-update step, the cheap preparation of an initial state at the largest D
        {"name": "su_d8_fp64", "kind": "su", "model": "quench", "D": 8, "precision": "fp64"},
        # a handful of rank-4 updates in FP64 (K = 20, no multiple of any tile)
        {"name": "batch7_d5_r4_fp64", "kind": "batch", "D": 5, "r": 4, "n": 7, "precision": "fp64"},
        # a small batch at the largest D in FP64
        {"name": "batch48_d8_fp64", "kind": "batch", "D": 8, "r": 2, "n": 48, "precision": "fp64"},
        # an odd D and batch with the single-precision environment
        {"name": "batch101_d7_fp32", "kind": "batch", "D": 7, "r": 2, "n": 101, "precision": "fp32"},
        # the throughput workloads: many independent bonds, split-BF16 environment
        {"name": "batch912_d6_bf16x3", "kind": "batch", "D": 6, "r": 2, "n": 912, "precision": "bf16x3"},
        {"name": "batch912_d8_bf16x3", "kind": "batch", "D": 8, "r": 2, "n": 912, "precision": "bf16x3"},
        # rank-4 gates at the largest bond the library takes (K = 32)
        {"name": "batch45_d8_r4_bf16x3", "kind": "batch", "D": 8, "r": 4, "n": 45, "precision": "bf16x3"},
        # the mixed batch: D uniform in 3..8, r in {2, 4}, host arrays in and out
        {"name": "uneven512_bf16x3", "kind": "uneven", "n": 512, "precision": "bf16x3"},
    ]


def draw(rng):
    kind = rng.choices(["cell", "su", "batch", "uneven"], [3, 1, 5, 1])[0]
    precision = rng.choice(["fp64", "fp32", "bf16x3", "bf16x3"])
    if kind == "uneven":
        return {"kind": "uneven", "n": round(math.exp(rng.uniform(math.log(24), math.log(500)))),
                "precision": "bf16x3"}
    if kind == "su":
        return {"kind": "su", "model": rng.choice(["quench", "thermal"]), "D": rng.randint(2, 8), "precision": "fp64"}
    if kind == "cell":
        model = rng.choice(["zz", "quench", "thermal", "ipepo"])
        # the product-state part makes the metric of larger D too ill-conditioned
        # for outputs that can be compared
        D = rng.randint(3, {"zz": 8, "quench": 6, "thermal": 5, "ipepo": 4}[model])
        return {"kind": "cell", "model": model, "D": D, "precision": precision}
    D, r = rng.randint(3, 8), rng.choice([2, 2, 4])
    most = {"fp64": 0.2e12, "fp32": 4e12, "bf16x3": 4e12}[precision] / _env_flops(D, r, 2)
    most = min(912.0, most, 32e9 / (16.0 * 20 * (D * r) ** 4))
    n = round(math.exp(rng.uniform(0.0, math.log(max(most, 2.0)))))
    return {"kind": "batch", "D": D, "r": r, "n": n, "precision": precision}


# ------------------------------------------------------------------ the calls
def _shared_stream():
    """The one stream a user's program queues its batches on."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream.cuda_stream


def _model(case):
    """(d, d_anc, r, bond gates, site gate, observable) of a cell case."""
    m = case["model"]
    if m == "zz":
        return 2, 1, 2, [I.zz_gate(0.01)] * 4, None, I.pauli("Z")
    if m == "quench":
        return (2, 1, 2, *I.tfim_real_time_gates(2.5, 0.01), I.pauli("X"))
    if m == "thermal":
        return (2, 2, 2, *I.tfim_imag_time_gates(2.5, 0.005), I.pauli("X"))
    return (4, 1, 4, *I.ipepo_thermal_gates(2.5, 0.005), I.ipepo_observable(I.pauli("X")))


def _cell_state(case, seed):
    """Site tensors part-way into a run: the model's product start and a
    random part of the same norm."""
    D, m = case["D"], case["model"]
    if m == "zz":
        return I.random_pair(seed, 2, D)
    if m == "quench":
        return I.quench_start(D, 1.0, seed)
    if m == "ipepo":
        A, B = I.ipepo_start(D, 1.0, seed)
        return A.astype(np.complex128), B.astype(np.complex128)
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(2):
        t = I.purification_state(D) + I.random_site_tensor(rng, 4, D)
        out.append(t / np.linalg.norm(t))
    return out


def _lambdas(case, seed):
    return np.random.default_rng(seed + 77).uniform(0.2, 1.0, (4, case["D"]))


def _batch_inputs(case, seed):
    """Normalised complex Gaussian site tensors on the GPU and one gate each."""
    D, n = case["D"], case["n"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    gen = torch.Generator(device=dev).manual_seed(seed)
    out = []
    for _ in range(2):
        t = torch.randn((n, 2 * D ** 4), dtype=torch.complex128, device=dev, generator=gen)
        t /= torch.linalg.vector_norm(t, dim=1, keepdim=True)
        out.append(t.view(n, 2, D, D, D, D))
    g = I.zz_gate(0.01) if case["r"] == 2 else I.heisenberg_gate(0.01)
    out.append(torch.from_numpy(g).to(dev).expand(n, 2, 2, 2, 2).contiguous())
    return out


def _uneven_items(case, seed):
    """Items (D, r, Ta, Tb, gate) as ``inputs.uneven_batch`` makes them, with the
    kinds D in 3..8, r in {2, 4} drawn from the batch size alone."""
    pick, rng = np.random.default_rng(case["n"]), np.random.default_rng(seed)
    items = []
    for _ in range(case["n"]):
        D, r = int(pick.integers(3, 9)), int(pick.choice([2, 4]))
        ta, tb = (I.random_site_tensor(rng, 2, D, np.complex64).astype(np.complex128) for _ in range(2))
        items.append((D, r, ta, tb, I.zz_gate(0.01) if r == 2 else I.heisenberg_gate(0.01)))
    return items


def prepare(case, seed):
    precision, kmax = PRECISION[case["precision"]], TAU_KMAX[case["precision"]]
    if case["kind"] == "uneven":
        items = _uneven_items(case, seed)
        kinds = sorted({(it[0], it[1]) for it in items})
        counts = [sum((it[0], it[1]) == k for it in items) for k in kinds]
        return {"case": case, "items": items,
                "ub": ntu.UnevenBatch(kinds, counts, sweeps=UNEVEN_SWEEPS, precision=precision, tau_kmax=kmax)}
    if case["kind"] == "batch":
        Ta, Tb, G = _batch_inputs(case, seed)
        ctx = ntu.Context(case["D"], r=case["r"], sweeps=SWEEPS, precision=precision, tau_kmax=kmax,
                          max_batch=case["n"], stream=_shared_stream())
        return {"case": case, "ctx": ctx, "in": (Ta, Tb, G), "Ta": torch.empty_like(Ta), "Tb": torch.empty_like(Tb),
                "info": torch.empty((case["n"], 4), dtype=torch.float64, device=Ta.device)}
    d, d_anc, r, gates, gate1, op = _model(case)
    ctx = ntu.Context(case["D"], d, d_anc, r, SWEEPS, precision, tau_kmax=kmax, stream=_shared_stream())
    A, B = _cell_state(case, seed)
    return {"case": case, "ctx": ctx, "A": A, "B": B, "gates": gates, "gate1": gate1, "op": op,
            "lam": _lambdas(case, seed)}


def run(state):
    case = state["case"]
    if case["kind"] == "uneven":
        Ta, Tb, info = state["ub"].update(state["items"], use_graph=True)
        # the items' results are views, in item order, of one flat array per site
        return {"Ta": Ta[0].base, "Tb": Tb[0].base, "info": info}
    ctx = state["ctx"]
    if case["kind"] == "batch":
        ctx.batch_update_dev(case["n"], *state["in"], state["Ta"], state["Tb"], state["info"])
        return {"Ta": state["Ta"], "Tb": state["Tb"], "info": state["info"]}
    ctx.set_state(state["A"], state["B"])
    if case["kind"] == "su":
        ctx.su_set_lambdas(state["lam"])
        deltas = ctx.su_step(state["gates"], state["gate1"])
        lam = ctx.su_get_lambdas()
    else:
        deltas, lam = ctx.step(state["gates"], state["gate1"]), None
    value = ctx.measure(0, state["op"])
    A, B = ctx.get_state()
    out = {"A": A, "B": B, "deltas": deltas, "value": np.array([value.real, value.imag])}
    return out if lam is None else {**out, "lam": lam}


# ------------------------------------------------------------ algorithmic work
def _env_flops(D, r, d_p):
    """Complex multiply-adds of the exact eight-site environment x 8."""
    macs = d_p * (2 * D ** 5 + 4 * D ** 6) + 2 * (d_p * D ** 5 * r + d_p * D ** 7 * r ** 2 + 2 * D ** 8 * r ** 2) \
        + D ** 8 * r ** 4
    return 8.0 * macs


def _update_work(D, r, d, d_anc, sweeps):
    """(bytes, flops) of one bond update: sites and gate in, sites and the four
    figures out; environment, gate + QR, and the ALS reduced problems."""
    d_p, K = d * d_anc, D * r
    als = sweeps * 2 * (K ** 4 * D + K ** 3 * D ** 2)
    qr = 2 * 2 * d_p * D ** 3 * K ** 2
    return 16.0 * (4 * d_p * D ** 4 + d ** 4 + 2), _env_flops(D, r, d_p) + 8.0 * (als + qr)


def work(case):
    if case["kind"] == "uneven":
        # the expected batch: every kind equally likely
        parts = [_update_work(D, r, 2, 1, UNEVEN_SWEEPS) for D in range(3, 9) for r in (2, 4)]
        return {"bytes": case["n"] * sum(p[0] for p in parts) / 12, "flops": case["n"] * sum(p[1] for p in parts) / 12}
    if case["kind"] == "batch":
        b, f = _update_work(case["D"], case["r"], 2, 1, SWEEPS)
        return {"bytes": case["n"] * b, "flops": case["n"] * f}
    d, d_anc, r = _model(case)[:3]
    D, K, d_p = case["D"], case["D"] * r, d * d_anc
    b, f = _update_work(D, r, d, d_anc, SWEEPS)
    if case["kind"] == "su":
        f = 8.0 * (2 * 2 * d_p * D ** 3 * K ** 2 + 20 * K ** 3)
    return {"bytes": 16.0 * 4 * d_p * D ** 4, "flops": 4 * f}


# ---------------------------------------------------- the same in 64-bit torch
def _svd(X):
    """X = U diag(s) Vh over a stack of small matrices; the first entry of each
    left vector within 1e-10 of its largest modulus is real and positive."""
    U, s, Vh = torch.linalg.svd(X.cpu(), full_matrices=False)
    a = U.abs()
    at = (a >= (1 - 1e-10) * a.amax(dim=1, keepdim=True)).to(torch.int8).argmax(dim=1, keepdim=True)
    u = torch.gather(U, 1, at)
    ph = u.conj() / u.abs()
    return (U * ph).to(X.device), s.to(X.device), (Vh * ph.conj().transpose(1, 2)).to(X.device)


def _split(G, r):
    """G[n, a', b', a, b] into its operator-Schmidt halves of rank r."""
    n, d = G.shape[:2]
    X = G.permute(0, 1, 3, 2, 4).reshape(n, d * d, d * d)
    U, s, _ = _svd(X)
    k = (s > 1e-15 * s[:, :1])[:, None, :r]
    rs = torch.where(k, s[:, None, :r].sqrt(), torch.ones_like(s[:, None, :r]))
    GA = torch.where(k, U[:, :, :r] * rs, 0)
    GB = torch.where(k, (U.mH @ X).transpose(1, 2)[:, :, :r] / rs, 0)
    return GA.view(n, d, d, r), GB.view(n, d, d, r)


def _qr(M):
    Q, R = torch.linalg.qr(M)
    p = torch.diagonal(R, dim1=1, dim2=2)
    p = p / p.abs()
    return Q * p[:, None, :], R * p.conj()[:, :, None]


def _gate_qr(Ta, Tb, G, d_anc, r):
    n, d_p, D = Ta.shape[:3]
    GA, GB = _split(G, r)
    Ta6, Tb6 = (t.view(n, d_p // d_anc, d_anc, D, D, D, D) for t in (Ta, Tb))
    K, m = D * r, d_p * D ** 3
    MA = torch.einsum("ztsk,zscluwx->ztcluxwk", GA, Ta6).reshape(n, m, K)
    MB = torch.einsum("ztsk,zscluwx->ztcwuxlk", GB, Tb6).reshape(n, m, K)
    return (*_qr(MA), *_qr(MB))


def _half(Q, side, top, bot, d_p, D):
    n, _, K = Q.shape
    Q5 = Q.view(n, d_p, D, D, D, K)
    Y = torch.einsum("zpeunk,zef->zpfunk", Q5, side)
    T = torch.einsum("zpfunk,zpfvml->zunkvml", Y, Q5.conj())
    T = torch.einsum("zunkvml,zhujv->zhjnkml", T, top)
    return torch.einsum("zhjnkml,zanbm->zabhjkl", T, bot)


def _metric(Ta, Tb, QA, QB):
    """The eight-site metric, Hermitian, non-negative, of unit trace."""
    n, d_p, D = Ta.shape[:3]
    K = QA.shape[2]
    a, b = Ta.conj(), Tb.conj()
    e = torch.einsum
    HL = _half(QA, e("zpluxn,zpluyn->zxy", Tb, b), e("zpluhv,zplujw->zhvjw", Tb, b), e("zplvhn,zplwjn->zhvjw", Tb, b), d_p, D)
    HR = _half(QB, e("zpxurn,zpyurn->zxy", Ta, a), e("zphurv,zpjurw->zhvjw", Ta, a), e("zphvrn,zpjwrn->zhvjw", Ta, a), d_p, D)
    g = e("zabhikl,zabhijm->zlmkj", HL, HR).reshape(n, K * K, K * K)
    g = (g + g.mH) / 2
    for i in torch.linalg.cholesky_ex(g)[1].nonzero().flatten().tolist():
        w, V = torch.linalg.eigh(g[i])
        g[i] = (V * w.clamp(min=0)) @ V.mH
    return g / torch.diagonal(g, dim1=1, dim2=2).real.sum(1)[:, None, None]


def _solve(gA, J, eps0, kmax):
    """pinv_tau(gA) J with the largest tolerance 10^-4 .. 10^-kmax that
    minimises the error; (M, tau)."""
    n, N, _ = gA.shape
    M, tau = torch.empty_like(J), torch.full((n,), 1e-4, dtype=torch.float64)
    top = gA.abs().sum(2).amax(1)
    eye = torch.eye(N, dtype=gA.dtype, device=gA.device)
    # a Cholesky factor of gA - 1e-4 B, B >= lambda_max: every tolerance keeps all
    ok = torch.linalg.cholesky_ex(gA - (1e-4 * top)[:, None, None] * eye)[1] == 0
    if ok.any():
        M[ok] = torch.linalg.solve(gA[ok], J[ok][..., None])[..., 0]
    for i in (~ok).nonzero().flatten().tolist():
        w, V = torch.linalg.eigh(gA[i])
        y = V.mH @ J[i]
        taus = [float("1e-%d" % k) for k in range(4, kmax + 1)]
        eps = [float(eps0[i]) - float((y[w > t * w[-1]].abs() ** 2 / w[w > t * w[-1]]).sum()) for t in taus]
        j = next(q for q, x in enumerate(eps) if x <= min(eps) + 1e-14 * float(eps0[i]))
        keep = w > taus[j] * w[-1]
        M[i], tau[i] = V[:, keep] @ (y[keep] / w[keep]), taus[j]
    return M, tau


def _tilt(Y, Z):
    """Y to an isometry Q, Y = Q R, and Z to Z R^T: the same Z Y^T."""
    for _ in range(2):
        R = torch.linalg.cholesky(Y.mH @ Y).mH
        Y = torch.linalg.solve_triangular(R, Y, upper=True, left=False)
        Z = Z @ R.transpose(1, 2)
    return Y, Z


def _balanced(X, D):
    U, s, Vh = _svd(X)
    rs = s[:, None, :D].sqrt()
    return U[:, :, :D] * rs, Vh[:, :D].transpose(1, 2) * rs


def _als(g, RA, RB, D, sweeps, kmax):
    n, K, _ = RA.shape
    X0 = RA @ RB.transpose(1, 2)
    x0 = X0.reshape(n, K * K, 1)
    gx0 = (g @ x0).view(n, K, K)
    eps0 = (x0.conj() * gx0.view(n, K * K, 1)).sum((1, 2)).real
    g4 = g.view(n, K, K, K, K)
    MA, MB = _balanced(X0, D)
    tau = torch.full((n,), math.nan, dtype=torch.float64)
    for _ in range(sweeps):
        MB, MA = _tilt(MB, MA)
        gA = torch.einsum("zya,zxywb->zxawb", MB.conj(), torch.einsum("zxywv,zvb->zxywb", g4, MB))
        J = torch.einsum("zya,zxy->zxa", MB.conj(), gx0)
        v, tau = _solve(gA.reshape(n, K * D, K * D), J.reshape(n, K * D), eps0, kmax)
        MA, MB = _tilt(v.view(n, K, D), MB)
        gB = torch.einsum("zxa,zxywb->zyawb", MA.conj(), torch.einsum("zxyvw,zvb->zxywb", g4, MA))
        J = torch.einsum("zxa,zxy->zya", MA.conj(), gx0)
        v, tau = _solve(gB.reshape(n, K * D, K * D), J.reshape(n, K * D), eps0, kmax)
        MB = v.view(n, K, D)
    MA, MB = _balanced(MA @ MB.transpose(1, 2), D)
    x = (MA @ MB.transpose(1, 2)).reshape(n, K * K, 1) - x0
    eps = (x.conj() * (g @ x)).sum((1, 2)).real
    return MA, MB, torch.stack([eps, eps / eps0, eps0, tau.to(eps.device)], dim=1)


def _unit(T):
    return T / torch.linalg.vector_norm(T.flatten(1), dim=1).view(-1, 1, 1, 1, 1, 1)


def _recompose(QA, QB, MA, MB, d_p, D):
    n = QA.shape[0]
    A = (QA @ MA).view(n, d_p, D, D, D, D).permute(0, 1, 2, 3, 5, 4)
    B = (QB @ MB).view(n, d_p, D, D, D, D).permute(0, 1, 5, 3, 2, 4)
    return _unit(A), _unit(B)


def _update(Ta, Tb, G, d_anc, r, sweeps, kmax):
    """Bond updates of a stack of items, in slices that fit the card."""
    n, d_p, D = Ta.shape[:3]
    chunk = max(1, int(6e9 / (16.0 * (D * r) ** 2 * (D ** 4 + (D * r) ** 2))))
    out = []
    for i in range(0, n, chunk):
        ta, tb, gg = Ta[i:i + chunk], Tb[i:i + chunk], G[i:i + chunk]
        QA, RA, QB, RB = _gate_qr(ta, tb, gg, d_anc, r)
        MA, MB, info = _als(_metric(ta, tb, QA, QB), RA, RB, D, sweeps, kmax)
        out.append((*_recompose(QA, QB, MA, MB, d_p, D), info))
    return [torch.cat(x) for x in zip(*out)]


def _update_su(Ta, Tb, G, d_anc, r):
    n, d_p, D = Ta.shape[:3]
    QA, RA, QB, RB = _gate_qr(Ta, Tb, G, d_anc, r)
    X0 = RA @ RB.transpose(1, 2)
    s = _svd(X0)[1]
    A, B = _recompose(QA, QB, *_balanced(X0, D), d_p, D)
    return A, B, s[0, :D], float((s[0, D:] ** 2).sum() / (s[0] ** 2).sum())


def _weighted(T, lam, bonds, skip, power):
    for leg, b in enumerate(bonds):
        if b != skip:
            shape = [1] * 6
            shape[leg + 2] = -1
            T = T * (lam[b] ** power).view(shape)
    return T


def _site_gate(T, U, d_anc):
    n, d_p, D = T.shape[:3]
    t = torch.einsum("ts,zsclurn->ztclurn", U, T.reshape(n, d_p // d_anc, d_anc, D, D, D, D))
    return _unit(t.reshape(T.shape))


def _estimator(T, N, O, d_anc):
    """Cluster estimator of O on T among four neighbours N."""
    T, N, e = T[0], N[0], torch.einsum
    n = N.conj()
    ends = (e("pluxn,pluyn->xy", N, n), e("plurx,plury->xy", N, n), e("pxurn,pyurn->xy", N, n), e("plxrn,plyrn->xy", N, n))
    W = T
    for leg, E in enumerate(ends):
        W = torch.movedim(torch.tensordot(W, E, dims=([leg + 1], [0])), -1, leg + 1)
    full = torch.kron(O, torch.eye(d_anc, dtype=O.dtype, device=O.device))
    return complex((T.conj() * torch.tensordot(full, W, dims=([1], [0]))).sum() / (T.conj() * W).sum())


def _exact_cell(case, seed):
    d, d_anc, r, gates, gate1, op = _model(case)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    up = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to(dev)  # noqa: E731
    A, B = (up(t)[None] for t in _cell_state(case, seed))
    lam = up(_lambdas(case, seed))
    turn = lambda t: t.permute(0, 1, 5, 2, 3, 4)  # noqa: E731
    back = lambda t: t.permute(0, 1, 3, 4, 5, 2)  # noqa: E731
    su, deltas = case["kind"] == "su", []
    if gate1 is not None:
        A, B = (_site_gate(t, up(gate1), d_anc) for t in (A, B))
    for b in range(4):
        G = up(gates[b])[None]
        a2, b2 = A, B
        if su:
            a2, b2 = _weighted(a2, lam, (2, 1, 0, 3), b, 0.5), _weighted(b2, lam, (0, 3, 2, 1), b, 0.5)
        if b in (1, 3):
            a2, b2 = turn(a2), turn(b2)
        left, right = (a2, b2) if b < 2 else (b2, a2)
        G = G if b < 2 else G.permute(0, 2, 1, 4, 3)
        left, right = left.contiguous(), right.contiguous()
        if su:
            left, right, s, delta = _update_su(left, right, G, d_anc, r)
        else:
            left, right, info = _update(left, right, G, d_anc, r, SWEEPS, TAU_KMAX[case["precision"]])
            delta = float(info[0, 1])
        deltas.append(delta)
        a2, b2 = (left, right) if b < 2 else (right, left)
        if b in (1, 3):
            a2, b2 = back(a2), back(b2)
        if su:
            a2, b2 = _weighted(a2, lam, (2, 1, 0, 3), b, -0.5), _weighted(b2, lam, (0, 3, 2, 1), b, -0.5)
            lam = lam.clone()
            lam[b] = s / torch.linalg.vector_norm(s)
        A, B = _unit(a2), _unit(b2)
    if gate1 is not None:
        A, B = (_site_gate(t, up(gate1), d_anc) for t in (A, B))
    v = _estimator(A, B, up(op), d_anc)
    # the halves of a rank-4 gate with equal Schmidt values are not unique: the
    # phases of the bond basis, and so the tensors, have no one value
    A, B = (None, None) if r == 4 else (A[0], B[0])
    out = {"A": A, "B": B, "deltas": torch.tensor(deltas, dtype=torch.float64), "value": np.array([v.real, v.imag])}
    return {**out, "lam": lam} if su else out


def exact(case, seed):
    kmax = TAU_KMAX[case["precision"]]
    if case["kind"] in ("cell", "su"):
        return _exact_cell(case, seed)
    if case["kind"] == "batch":
        Ta, Tb, G = _batch_inputs(case, seed)
        A, B, info = _update(Ta, Tb, G, 1, case["r"], SWEEPS, kmax)
        return {"Ta": A if case["r"] == 2 else None, "Tb": B if case["r"] == 2 else None, "info": info}
    items = _uneven_items(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    info = np.empty((case["n"], 4))
    for k in sorted({(it[0], it[1]) for it in items}):
        at = [i for i, it in enumerate(items) if (it[0], it[1]) == k]
        stack = [torch.from_numpy(np.stack([items[i][q] for i in at])).to(dev) for q in (2, 3, 4)]
        info[at] = _update(*stack, 1, k[1], UNEVEN_SWEEPS, kmax)[2].cpu().numpy()
    # the tensors of the rank-4 items have no one value (see above)
    return {"Ta": None, "Tb": None, "info": info}
