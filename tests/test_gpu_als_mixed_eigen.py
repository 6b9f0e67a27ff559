"""The eigen path of the mixed contexts' ALS solves against the oracle on the
same metric, at the smallest and largest n_A = D^2 r, at odd ones, and on the
tensor-core builds' sizes (K = 16 and 32)."""
import numpy as np
import pytest

from oracle import ntu_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,r", [(2, 1), (3, 1), (3, 2), (5, 3), (6, 2), (8, 2), (8, 4)])
def test_null_modes_are_dropped(D, r):
    """A metric of rank n_A / 2 (and 1e-30 of the rest): every tolerance drops the
    rounding-level half of the reduced metric's eigenvalues.  The double-FP32
    metric is good to 2^-46 and the kept part's condition some 1e4 (a random
    projection of a unit spectrum): 1e4 x 2^-46 x n_A x 2 solves < 1e-7; 1e-6."""
    import torch

    from paper_2107_06635_gb300 import ntu

    K, ng, n = D * r, (D * r) ** 2, D * D * r
    rng = np.random.default_rng(170 + D)
    a = rng.standard_normal((ng, ng)) + 1j * rng.standard_normal((ng, ng))
    w, _ = np.linalg.qr(a)
    g = (w * np.where(np.arange(ng) < max(n // 2, 1), 1.0, 1e-30)) @ w.conj().T
    g = 0.5 * (g + g.conj().T)
    RA, RB = (rng.standard_normal((K, K)) + 1j * rng.standard_normal((K, K)) for _ in range(2))
    cfg = O.Config(D=D, r=r, sweeps=1, tau_exponents=tuple(range(4, 9)))
    ma, mb, eps, delta, eps0, tau = O.als_truncate(g, RA, RB, D, 1, cfg.taus)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)[None]).cuda()  # noqa: E731
    with ntu.Context(D, r=r, sweeps=1, precision=ntu.NTU_MIXED_FP32, tau_kmax=8) as ctx:
        MA, MB = (torch.empty((1, K, D), dtype=torch.complex128, device="cuda") for _ in range(2))
        info = torch.empty((1, 4), dtype=torch.float64, device="cuda")
        ctx.solver_paths()
        ctx.batch_als_dev(1, dev(g), dev(RA), dev(RB), MA, MB, info)
        ctx.sync()
        paths = ctx.solver_paths()
    assert paths["als_eigen"] == 2
    inf = info[0].cpu().numpy()
    assert inf[3] == tau
    assert abs(inf[1] - delta) <= 1e-6
    X = MA[0].cpu().numpy() @ MB[0].cpu().numpy().T
    assert np.linalg.norm(X - ma @ mb.T) <= 1e-6 * np.linalg.norm(ma @ mb.T)
