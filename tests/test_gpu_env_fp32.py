"""The FP32 environment's products, whose tile follows the sizes and the number
of items: an item's metric has the same bits in every tile, and agrees with the
oracle within the rounding of its sums."""
import numpy as np
import pytest

from oracle import ntu_oracle as O
from paper_2107_06635_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _env(D, r, d, d_anc, n, Ta, Tb, QA, QB):
    import torch

    from paper_2107_06635_gb300 import ntu

    ng = (D * r) ** 2
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    g = torch.empty((n, ng, ng), dtype=torch.complex128, device="cuda")
    with ntu.Context(D, d, d_anc, r, precision=ntu.NTU_MIXED_FP32, tau_kmax=8, max_batch=n) as ctx:
        ctx.batch_env_dev(n, dev(Ta), dev(Tb), dev(QA), dev(QB), g)
        ctx.sync()
    return g.cpu().numpy()


# D, r, d, d_anc, items: rows D^2 and (D r)^2 around the tiles' 16 to 64 rows,
# sums of d_p D, D^2 and D^4 terms around the 16 terms of a stage
@pytest.mark.parametrize("D,r,d,d_anc,n", [(1, 1, 2, 1, 2), (2, 2, 2, 1, 700), (3, 4, 2, 1, 90), (4, 2, 2, 2, 200),
                                           (5, 2, 2, 1, 150), (6, 2, 2, 1, 90), (7, 2, 2, 1, 40), (8, 2, 4, 1, 20),
                                           (8, 4, 2, 1, 3)])
def test_tiles_agree_and_match_oracle(D, r, d, d_anc, n):
    """Three chained sums of at most 64, 64 and 4096 complex terms in FP32, each
    term four roundings: 4 x 4224 x 2^-24 = 1.0e-3 bounds the relative error."""
    d_p, K = d * d_anc, D * r
    rng = np.random.default_rng(10 * D + r)
    Ta, Tb = (np.stack([I.random_site_tensor(rng, d_p, D) for _ in range(2)]) for _ in range(2))
    QA, QB = (np.stack([np.linalg.qr(rng.standard_normal((d_p * D ** 3, K))
                                     + 1j * rng.standard_normal((d_p * D ** 3, K)))[0] for _ in range(2)])
              for _ in range(2))
    alone = [_env(D, r, d, d_anc, 1, *(x[i:i + 1] for x in (Ta, Tb, QA, QB)))[0] for i in range(2)]
    which = np.arange(n) % 2
    g = _env(D, r, d, d_anc, n, *(x[which] for x in (Ta, Tb, QA, QB)))
    for i in {0, 1, n // 2, n - 1}:
        assert np.array_equal(g[i], alone[i % 2])
    for i in range(2):
        ref = O.metric_raw(Ta[i], Tb[i], QA[i], QB[i], d_p, D)
        assert np.linalg.norm(alone[i] - ref) <= 1.0e-3 * np.linalg.norm(ref)
