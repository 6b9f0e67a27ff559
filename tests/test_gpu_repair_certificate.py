"""Metrics that the Gershgorin discs leave open, with one diagonal entry next to
the shift of the FP32 certificate (6 (n_g + 3) 2^-24 of the trace): definite ones
are kept whichever factorisation proves it, indefinite ones clipped."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _metric(rng, n):
    """Definite, eigenvalues in [0.5, 1.5], not diagonally dominant."""
    w, _ = np.linalg.qr(rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)))
    g = (w * np.linspace(0.5, 1.5, n)) @ w.conj().T
    return 0.5 * (g + g.conj().T)


@pytest.mark.parametrize("D,r", [(4, 2), (6, 2), (4, 4), (5, 4)])
def test_smallest_diagonal_next_to_the_shift(D, r):
    import torch

    from paper_2107_06635_gb300 import ntu

    n = (D * r) ** 2
    rng = np.random.default_rng(n)
    shift = 6.0 * (n + 3) * 2.0 ** -24 * n
    G = []
    for i, f in enumerate((1e-9, 0.5, 0.99, 1.01, 2.0, 1e3)):
        s = np.ones(n)
        s[(7 * i) % n] = np.sqrt(f * shift)                  # a congruence: still definite
        G.append(s[:, None] * _metric(rng, n) * s)
    bad = _metric(rng, n)
    bad[3, 3] = -0.2                                         # indefinite
    G = np.stack([*G, bad])
    g = torch.from_numpy(G).cuda()
    diag = torch.empty((len(G), 3), dtype=torch.float64, device="cuda")
    with ntu.Context(D, r=r, max_batch=len(G)) as ctx:
        ctx.solver_paths()
        ctx.batch_repair_dev(len(G), g, diag)
        ctx.sync()
        paths = ctx.solver_paths()
    assert (paths["repair_gershgorin"], paths["repair_cholesky"], paths["repair_eigen"]) == (0, len(G) - 1, 1)
    out = g.cpu().numpy()
    for i in range(len(G) - 1):                              # scaled to unit trace, one rounding an entry
        ref = G[i] / np.trace(G[i]).real
        assert np.abs(out[i] - ref).max() <= n * 2.0 ** -52 * np.abs(ref).max()
    lam, W = np.linalg.eigh(bad)
    ref = (W * np.maximum(lam, 0)) @ W.conj().T
    assert np.linalg.norm(out[-1] - ref / np.trace(ref).real) <= n * 2.0 ** -50 * np.linalg.norm(out[-1])


@pytest.mark.parametrize("D,r", [(1, 1), (2, 1), (2, 2), (5, 1), (3, 2), (7, 1), (4, 2), (3, 3), (6, 2)])
def test_metrics_that_the_discs_decide(D, r):
    """n_g = 1 to 144, on either side of the sizes that one block takes alone:
    Hermitised, of unit trace, and the diagnostics; beside them one metric that
    a factorisation decides and, from n_g = 4 on, one to be clipped."""
    import torch

    from paper_2107_06635_gb300 import ntu

    n = (D * r) ** 2
    rng = np.random.default_rng(10 * D + r)
    noise = rng.standard_normal((3, n, n)) + 1j * rng.standard_normal((3, n, n))
    G = [np.diag(rng.uniform(1, 2, n)) + x * (0.3 / (n + 1)) for x in noise]
    if n > 1:
        h = 0.5 * np.full((n, n), 1.9 / n) + np.eye(n)       # discs reach past zero from n = 21 on, definite
        bad = np.eye(n) + 0j
        bad[0, 1] = bad[1, 0] = 2.0                          # eigenvalue -1
        G += [h + 0j, bad]
    G = np.stack(G)
    g = torch.from_numpy(G).cuda()
    diag = torch.empty((len(G), 3), dtype=torch.float64, device="cuda")
    with ntu.Context(D, r=r, max_batch=len(G)) as ctx:
        ctx.solver_paths()
        ctx.batch_repair_dev(len(G), g, diag)
        ctx.sync()
        paths = ctx.solver_paths()
    assert paths["repair_eigen"] == (1 if n > 1 else 0)
    assert paths["repair_gershgorin"] + paths["repair_cholesky"] == len(G) - paths["repair_eigen"]
    assert paths["repair_gershgorin"] >= 3
    out, diag = g.cpu().numpy(), diag.cpu().numpy()
    for i, x in enumerate(G):
        h = 0.5 * (x + x.conj().T)
        defect = np.linalg.norm(x - x.conj().T) / np.linalg.norm(x)
        assert abs(diag[i, 0] - defect) <= n * n * 2.0 ** -52 * max(defect, 1e-300)
        lam, W = np.linalg.eigh(h)
        ref = (W * np.maximum(lam, 0)) @ W.conj().T if i == 4 else h
        tr = np.trace(ref).real
        assert np.linalg.norm(out[i] - ref / tr) <= n * 2.0 ** -50 * np.linalg.norm(out[i])
        assert abs(diag[i, 2] - np.log(tr)) <= n * 2.0 ** -50
        assert np.isnan(diag[i, 1]) == (i != 4)


@pytest.mark.parametrize("D,r", [(3, 2), (6, 2)])
@pytest.mark.parametrize("n", [4, 170])
def test_result_does_not_depend_on_the_batch(D, r, n):
    """Flat and graded metrics in one batch (below and above the number of items
    that run at once, which decides whether the certificate is tried): every
    result has the bits it has alone."""
    import torch

    from paper_2107_06635_gb300 import ntu

    m = (D * r) ** 2
    rng = np.random.default_rng(m)
    shift = 6.0 * (m + 3) * 2.0 ** -24 * m
    kinds = []
    for f in (1e-6, 2.9, 3.1, 1e3):
        s = np.ones(m)
        s[1] = np.sqrt(f * shift)
        kinds.append(s[:, None] * _metric(rng, m) * s)
    which = np.arange(n) % 4

    def repair(x):
        g = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        diag = torch.empty((len(x), 3), dtype=torch.float64, device="cuda")
        with ntu.Context(D, r=r, max_batch=len(x)) as ctx:
            ctx.batch_repair_dev(len(x), g, diag)
            ctx.sync()
            assert ctx.solver_paths()["repair_cholesky"] == len(x)
        return g.cpu().numpy()

    alone = [repair(k[None])[0] for k in kinds]
    out = repair(np.stack([kinds[w] for w in which]))
    for i in range(n):
        assert np.array_equal(out[i], alone[which[i]])
