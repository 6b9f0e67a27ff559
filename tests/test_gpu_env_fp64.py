"""The sliced FP64 environment (tensor cores) against the oracle at the edges
of its tiles: one row and column, sums shorter than a stage, remainders of the
64-wide tiles, rows longer and shorter than 64 terms, and several passes."""
import numpy as np
import pytest

from oracle import ntu_oracle as O
from paper_2107_06635_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _env(ctx, n, Ta, Tb, QA, QB):
    import torch

    ng = ctx.K ** 2
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    g = torch.empty((n, ng, ng), dtype=torch.complex128, device="cuda")
    ctx.batch_env_dev(n, dev(Ta), dev(Tb), dev(QA), dev(QB), g)
    ctx.sync()
    return g.cpu().numpy()


def _q(rng, n, m, K):
    out = []
    for _ in range(n):
        q, _ = np.linalg.qr(rng.standard_normal((m, K)) + 1j * rng.standard_normal((m, K)))
        out.append(q)
    return np.stack(out)


# D, r, d, d_anc: K = D r
@pytest.mark.parametrize("D,r,d,d_anc", [(1, 1, 2, 1), (2, 1, 2, 1), (2, 4, 2, 1), (3, 2, 2, 2), (4, 4, 4, 1),
                                         (5, 4, 2, 1), (7, 4, 2, 1), (8, 1, 2, 1), (8, 3, 2, 4), (8, 4, 2, 1)])
def test_matches_oracle(D, r, d, d_anc):
    """Both sides sum in FP64 accuracy over at most D^4 = 4096 complex terms:
    4096 x 2^-53 = 5e-13 bounds either side's relative error of g."""
    from paper_2107_06635_gb300 import ntu

    n, d_p, K = 2, d * d_anc, D * r
    rng = np.random.default_rng(100 * D + r)
    Ta, Tb = (np.stack([I.random_site_tensor(rng, d_p, D) for _ in range(n)]) for _ in range(2))
    Ta[1] *= 2.0 ** 70                  # scales far apart within a batch
    Tb[1] *= 2.0 ** -90
    QA, QB = _q(rng, n, d_p * D ** 3, K), _q(rng, n, d_p * D ** 3, K)
    with ntu.Context(D, d, d_anc, r, max_batch=n) as ctx:
        g = _env(ctx, n, Ta, Tb, QA, QB)
    for i in range(n):
        ref = O.metric_raw(Ta[i], Tb[i], QA[i], QB[i], d_p, D)
        assert np.linalg.norm(g[i] - ref) <= 5e-13 * np.linalg.norm(ref)


def test_passes_agree():
    """More items than one pass holds: each equals its value alone, bit for bit."""
    from paper_2107_06635_gb300 import ntu

    D, r, n = 8, 4, 13
    rng = np.random.default_rng(5)
    Ta, Tb = (np.stack([I.random_site_tensor(rng, 2, D) for _ in range(n)]) for _ in range(2))
    QA, QB = _q(rng, n, 2 * D ** 3, D * r), _q(rng, n, 2 * D ** 3, D * r)
    with ntu.Context(D, r=r, max_batch=n) as ctx:
        g = _env(ctx, n, Ta, Tb, QA, QB)
    with ntu.Context(D, r=r, max_batch=1) as ctx:
        for i in (0, 10, 11, 12):
            assert np.array_equal(_env(ctx, 1, Ta[i:i + 1], Tb[i:i + 1], QA[i:i + 1], QB[i:i + 1])[0], g[i])


def test_non_finite_rows_stay_in_their_item():
    from paper_2107_06635_gb300 import ntu

    D, r, n = 4, 2, 3
    rng = np.random.default_rng(6)
    Ta, Tb = (np.stack([I.random_site_tensor(rng, 2, D) for _ in range(n)]) for _ in range(2))
    QA, QB = _q(rng, n, 2 * D ** 3, D * r), _q(rng, n, 2 * D ** 3, D * r)
    with ntu.Context(D, r=r, max_batch=n) as ctx:
        good = _env(ctx, n, Ta, Tb, QA, QB)
        QA[1, 5, 3] = np.inf
        g = _env(ctx, n, Ta, Tb, QA, QB)
    assert not np.isfinite(g[1]).all()
    assert np.array_equal(g[0], good[0]) and np.array_equal(g[2], good[2])
