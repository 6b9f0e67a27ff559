"""ALS solves of the FP64 contexts that the Gershgorin discs do not decide
(selection by factorisations, and through the spectrum of the tridiagonal
form), against the oracle on the same metric, at the sizes where the working
matrix changes place (n_A = 77 and below: packed in shared memory) and at the
smallest and largest n_A = D^2 r."""
import numpy as np
import pytest

from oracle import ntu_oracle as O

pytestmark = pytest.mark.gpu


def _metric(rng, ng, lam):
    a = rng.standard_normal((ng, ng)) + 1j * rng.standard_normal((ng, ng))
    w, _ = np.linalg.qr(a)
    g = (w * lam) @ w.conj().T
    return 0.5 * (g + g.conj().T)


def _compare(D, r, lam_of, kmax, sweeps, seed, tol):
    import torch

    from paper_2107_06635_gb300 import ntu

    K, ng = D * r, (D * r) ** 2
    rng = np.random.default_rng(seed)
    g = _metric(rng, ng, lam_of(ng))
    RA, RB = (rng.standard_normal((K, K)) + 1j * rng.standard_normal((K, K)) for _ in range(2))
    cfg = O.Config(D=D, r=r, sweeps=sweeps, tau_exponents=tuple(range(4, kmax + 1)))
    ma, mb, eps, delta, eps0, tau = O.als_truncate(g, RA, RB, D, sweeps, cfg.taus)
    with ntu.Context(D, r=r, sweeps=sweeps, tau_kmax=kmax) as ctx:
        dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)[None]).cuda()  # noqa: E731
        MA, MB = (torch.empty((1, K, D), dtype=torch.complex128, device="cuda") for _ in range(2))
        info = torch.empty((1, 4), dtype=torch.float64, device="cuda")
        ctx.solver_paths()
        ctx.batch_als_dev(1, dev(g), dev(RA), dev(RB), MA, MB, info)
        ctx.sync()
        paths = ctx.solver_paths()
    inf = info[0].cpu().numpy()
    assert inf[3] == tau
    assert abs(inf[2] - eps0) <= 1e-12 * eps0
    assert abs(inf[1] - delta) <= tol
    X = MA[0].cpu().numpy() @ MB[0].cpu().numpy().T
    assert np.linalg.norm(X - ma @ mb.T) <= tol * np.linalg.norm(ma @ mb.T)
    return paths


@pytest.mark.parametrize("D,r", [(2, 1), (3, 2), (6, 2), (4, 4), (5, 3), (5, 4), (8, 2), (8, 4)])
@pytest.mark.parametrize("spread", [30.0, 1e6])
def test_graded_metrics(D, r, spread):
    """lambda geometric on [1, spread]: every tolerance keeps all, or the
    selection decides.  The solution's condition is at most the spread:
    1e6 x 2e-16 x n_A x sweeps, 1e-7, bounds the rounding of either side."""
    paths = _compare(D, r, lambda n: np.geomspace(1.0, spread, n), 15, 2, 91 + D, 1e-7)
    assert paths["als_gershgorin"] + paths["als_cholesky"] + paths["als_eigen"] == 4


@pytest.mark.parametrize("D,r", [(3, 2), (6, 2), (5, 4)])
def test_null_modes_are_dropped(D, r):
    """A metric of rank n_A / 2 plus 1e-30 of the rest: the reduced metric has
    n_A / 2 rounding-level eigenvalues that every tolerance drops.  The kept
    part's condition is some 1e4 (a random projection of a unit spectrum)."""
    n = D * D * r
    paths = _compare(D, r, lambda ng: np.where(np.arange(ng) < n // 2, 1.0, 1e-30), 12, 1, 17, 1e-7)
    assert paths["als_eigen"] == 2
