"""The sliced FP64 environment where every digit product has one sign: all entries
of a tensor equal, so that nothing cancels in any level's sum.  The metric is
known exactly."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_equal_entries():
    """D = 8, the longest sums (4096 complex terms in the join): the levels that
    accumulate in FP32 add at most 2^-45 of such a sum, 2.9e-14; the side edges,
    sums of 1024 terms in four chains on the FP64 pipe, 260 x 2^-53 each and enter
    twice, 5.8e-14; the other roundings are a few 2^-53: 9e-14 in all."""
    import torch

    from paper_2107_06635_gb300 import ntu

    D, r, d_p, n = 8, 2, 2, 24
    K, m, ng = D * r, d_p * D ** 3, (D * r) ** 2
    rng = np.random.default_rng(2)
    digits = [[63] + [127] * 6] * 4 + [[64 - i] + [126] * 6 for i in range(4, 8)]
    digits += [[rng.integers(33, 63), *rng.integers(60, 128, 6)] for _ in range(n - 8)]
    t = np.array([sum(int(x) * 256.0 ** -j for j, x in enumerate(d)) for d in digits])
    q = t[::-1].copy()
    full = lambda x, *s: torch.from_numpy(x.astype(np.complex128)).cuda().view(n, *[1] * len(s)).expand(n, *s).contiguous()  # noqa: E731
    T, Q = full(t, d_p, D, D, D, D), full(q, m, K)
    g = torch.empty((n, ng, ng), dtype=torch.complex128, device="cuda")
    with ntu.Context(D, r=r, max_batch=n) as ctx:
        ctx.batch_env_dev(n, T, T, Q, Q, g)
        ctx.sync()
    g = g.cpu().numpy()
    for i in range(n):
        a, b = Fraction(t[i]), Fraction(q[i])
        y = D * b * (d_p * D ** 3 * a * a)                   # side edge on Q
        edge = d_p * D ** 2 * a * a
        h = (D * D * edge) ** 2 * (d_p * D * y * b)
        want = D ** 4 * h * h
        for x in (g[i].real.min(), g[i].real.max()):
            assert abs(Fraction(x) - want) <= Fraction(9e-14) * want, i
        assert abs(g[i].imag).max() <= 9e-14 * float(want)
