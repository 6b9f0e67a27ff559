"""The tolerance selection of the FP64 contexts against the oracle on metrics
whose reduced spectrum is known: with r = 1 the isometric factor is unitary, so
the reduced metric has the eigenvalues of g.  The branches are the ones where
the selection can go wrong: every pair kept although no factorisation proves
it, and an isolated eigenvalue next to a tolerance."""
import numpy as np
import pytest

from oracle import ntu_oracle as O

pytestmark = pytest.mark.gpu


def _items(D, lam, n, seed):
    """n metrics of the spectrum lam on random eigenvectors, and random R."""
    K = D
    rng = np.random.default_rng(seed)
    g, R = [], []
    for _ in range(n):
        w, _ = np.linalg.qr(rng.standard_normal((K * K, K * K)) + 1j * rng.standard_normal((K * K, K * K)))
        x = (w * lam) @ w.conj().T
        g.append(0.5 * (x + x.conj().T))
        R.append([rng.standard_normal((K, K)) + 1j * rng.standard_normal((K, K)) for _ in range(2)])
    return np.stack(g), np.array(R)


def _check(D, lam, n, kmin, kmax, seed, tol):
    """One sweep of n items; X = M_A M_B^T and the tolerance against the oracle."""
    import torch

    from paper_2107_06635_gb300 import ntu

    g, R = _items(D, lam, n, seed)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    MA, MB = (torch.empty((n, D, D), dtype=torch.complex128, device="cuda") for _ in range(2))
    info = torch.empty((n, 4), dtype=torch.float64, device="cuda")
    with ntu.Context(D, r=1, sweeps=1, tau_kmin=kmin, tau_kmax=kmax, max_batch=n) as ctx:
        ctx.batch_als_dev(n, dev(g), dev(R[:, 0]), dev(R[:, 1]), MA, MB, info)
        ctx.sync()
        paths = ctx.solver_paths()
    taus = O.Config(D=D, r=1, tau_exponents=tuple(range(kmin, kmax + 1))).taus
    X = MA.cpu().numpy() @ MB.cpu().numpy().transpose(0, 2, 1)
    tau = info[:, 3].cpu().numpy()
    for i in range(n):
        ma, mb, _, _, _, want = O.als_truncate(g[i], R[i, 0], R[i, 1], D, 1, taus)
        assert tau[i] == want, (i, tau[i], want)
        assert np.linalg.norm(X[i] - ma @ mb.T) <= tol * np.linalg.norm(ma @ mb.T)
    return paths


@pytest.mark.parametrize("D", [2, 4, 7, 8])
@pytest.mark.parametrize("kmax", [4, 5])
def test_nothing_dropped_through_the_spectrum(D, kmax):
    """lambda_min 0.3% above the smallest tolerance: no certified bound on
    lambda_max is that close, so the spectrum decides, and keeps every pair
    (kmax 5: after looking at those below the larger tolerance).  A solve of
    condition 1 / tau is good to n_A 2^-53 / tau, and there are two a side:
    64 x 1.1e-16 x 1e5 x 4 = 3e-9."""
    n = D * D
    lam = np.concatenate([np.geomspace(1.003 * 10.0 ** -kmax, 0.3, n - 1), [1.0]])
    paths = _check(D, lam, 48, 4, kmax, 5 * D + kmax, 3e-9)
    assert paths["als_eigen"] == 2 * 48


@pytest.mark.parametrize("D", [2, 4, 7, 8])
@pytest.mark.parametrize("k", [7, 8, 9, 10])
@pytest.mark.parametrize("fac", [0.3, 3.0])
@pytest.mark.parametrize("kmin", [4, None])
def test_isolated_eigenvalue_next_to_a_tolerance(D, k, fac, kmin):
    """One eigenvalue at fac 10^-k lambda_max, the others above 10^-2: the
    largest tolerance that keeps it is 10^-k or 10^-(k+1), and a certificate at
    10^-k is right only for fac > 1.  kmin None: 10^-k is the first candidate.
    Dropping the pair costs at least 3e-11 / n_A of eps0, far above 1e-14.  Two
    solves a side of condition 1 / lambda_min, each good to n_A 2^-53 times it."""
    n = D * D
    lam = np.concatenate([[fac * 10.0 ** -k], np.geomspace(1e-2, 1.0, n - 1)])
    _check(D, lam, 20, k if kmin is None else kmin, k + 2, 1000 * k + D, 4.0 * n * 2.0 ** -53 / lam[0])
