"""The FP64 environment does not depend on how the legs of a bond are scaled: a
floating-point sum is as accurate when one side of its index grows as the
other falls, and so must the sliced products be.  Against the oracle in
extended precision on the same Q."""
import numpy as np
import pytest

from oracle import ntu_oracle as O
from paper_2107_06635_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# legs (of Ta, of Tb) of the three bonds that the neighbourhood contracts: A.u - B.dn,
# A.l - B.r (the edges of the two halves as well), A.dn - B.u
BONDS = [(2, 4), (1, 3), (4, 2)]


def _env(ctx, n, Ta, Tb, QA, QB):
    import torch

    ng = ctx.K ** 2
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    g = torch.empty((n, ng, ng), dtype=torch.complex128, device="cuda")
    ctx.batch_env_dev(n, dev(Ta), dev(Tb), dev(QA), dev(QB), g)
    ctx.sync()
    return g.cpu().numpy()


def _scaled(Ta, Tb, bonds, s):
    for la, lb in bonds:
        shape = [1] * 5
        shape[la] = -1
        Ta = Ta * s.reshape(shape)
        shape = [1] * 5
        shape[lb] = -1
        Tb = Tb / s.reshape(shape)
    return Ta, Tb


@pytest.mark.parametrize("D,r,d_anc", [(3, 2, 1), (2, 4, 2), (4, 2, 1)])
@pytest.mark.parametrize("bonds", [[0], [1], [2], [0, 1, 2]])
def test_scaled_legs(D, r, d_anc, bonds):
    """Legs scaled by 1 .. 10^-q and their partners by the inverse, rising and
    falling, on a random and on a nearly-product pair.  5e-13 bounds the
    rounding of sums of up to D^4 terms with room (the existing bound of the
    unscaled metric); without the balance q = 2 is 1e-10 off, q = 8 has no digit."""
    from paper_2107_06635_gb300 import ntu

    d_p = 2 * d_anc
    rng = np.random.default_rng(7 * D + len(bonds))
    GA, GB = O.gate_split(I.random_gate(rng), r)
    items, refs = [], []
    for q in (0, 1, 2, 4, 6, 8):
        for eps in (1.0, 1e-3):
            T = [eps * I.random_site_tensor(rng, d_p, D) for _ in range(2)]
            if eps < 1:
                for t in T:
                    t[:, 0, 0, 0, 0] += rng.standard_normal(d_p)
            for s in (10.0 ** np.linspace(0, -q, D), 10.0 ** np.linspace(-q, 0, D)):
                Ta, Tb = _scaled(*T, [BONDS[b] for b in bonds], s)
                QA, _ = O.qr_positive(O.gated_matrix(Ta, GA, d_anc, "left"))
                QB, _ = O.qr_positive(O.gated_matrix(Tb, GB, d_anc, "right"))
                items.append((Ta, Tb, QA, QB))
                refs.append(O.metric_raw(*(x.astype(np.clongdouble) for x in items[-1]), d_p, D))
    n = len(items)
    with ntu.Context(D, 2, d_anc, r, max_batch=n) as ctx:
        g = _env(ctx, n, *(np.stack([it[k] for it in items]) for k in range(4)))
    for i in range(n):
        ref = refs[i].astype(np.complex128)
        assert np.linalg.norm(g[i] - ref) <= 5e-13 * np.linalg.norm(ref), i


def test_scaled_legs_with_long_rows():
    """D = 6: rows of more than 64 terms, whose largest entries come from a pass
    of their own; the crossing bond's legs (A.l, B.r) scaled by powers of two
    down to 2^-200.  Against the FP64 oracle: sums of up to 1296 terms are good
    to 1296 x 2^-53 = 1.5e-13 on either side."""
    from paper_2107_06635_gb300 import ntu

    D, r = 6, 2
    K, m = D * r, 2 * D ** 3
    rng = np.random.default_rng(3)
    Ta, Tb = (I.random_site_tensor(rng, 2, D) for _ in range(2))
    QA, QB = (np.linalg.qr(rng.standard_normal((m, K)) + 1j * rng.standard_normal((m, K)))[0] for _ in range(2))
    batch = []
    for q in (0, 4, 12, 40):
        s = 2.0 ** (-q * np.arange(D))
        a, b = _scaled(Ta, Tb, [BONDS[1]], s)
        e = s.reshape(1, D, 1, 1, 1)                        # the leg as the rows of either Q have it
        qa, qb = QA.reshape(2, D, D, D, K) * e, QB.reshape(2, D, D, D, K) / e
        batch.append((a, b, qa.reshape(m, K), qb.reshape(m, K)))
    n = len(batch)
    with ntu.Context(D, r=r, max_batch=n) as ctx:
        g = _env(ctx, n, *(np.stack([it[k] for it in batch]) for k in range(4)))
    for i in range(n):
        ref = O.metric_raw(*batch[i], 2, D)
        assert np.linalg.norm(g[i] - ref) <= 5e-13 * np.linalg.norm(ref), i
