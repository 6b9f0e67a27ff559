"""The FP64 QR and recomposition, on a cluster of CTAs for a few items and on
one CTA each for many: both against the gated matrices' own QR at the smallest
and largest row counts, with columns whose reflectors are trivial and scales
far apart."""
import numpy as np
import pytest

from paper_2107_06635_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _qr(D, r, d, d_anc, Ta, Tb, G):
    import torch

    from paper_2107_06635_gb300 import ntu

    n, m, K = len(Ta), d * d_anc * D ** 3, D * r
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    Q = [torch.empty((n, m, K), dtype=torch.complex128, device="cuda") for _ in range(2)]
    R = [torch.empty((n, K, K), dtype=torch.complex128, device="cuda") for _ in range(2)]
    with ntu.Context(D, d, d_anc, r, max_batch=n) as ctx:
        ctx.batch_gate_qr_dev(n, dev(Ta), dev(Tb), dev(G), Q[0], R[0], Q[1], R[1])
        ctx.sync()
    return [x.cpu().numpy() for x in (Q[0], R[0], Q[1], R[1])]


@pytest.mark.parametrize("D,r,d,d_anc", [(4, 2, 2, 1), (4, 4, 4, 1), (5, 3, 2, 1), (7, 2, 2, 1), (8, 2, 2, 1), (8, 4, 2, 4)])
@pytest.mark.parametrize("scale", [1.0, 1e-170])
def test_cluster_and_single_cta_agree(D, r, d, d_anc, scale):
    """QR is unique with a positive diagonal; both sides' errors are at most
    m K 2^-53 times the condition of a random matrix (< 1e3): 1e-9 at the
    largest.  Orthogonality needs no condition: K m 2^-53 < 1e-10."""
    rng = np.random.default_rng(31 * D + r)
    n = 40                                               # one CTA each
    Ta, Tb = (np.stack([I.random_site_tensor(rng, d * d_anc, D) for _ in range(n)]) for _ in range(2))
    Ta[1] *= scale
    G = np.stack([I.random_gate(rng, d) for _ in range(n)])
    many = _qr(D, r, d, d_anc, Ta, Tb, G)
    few = _qr(D, r, d, d_anc, Ta[:2], Tb[:2], G[:2])     # on clusters
    for i in range(2):
        for s in (0, 2):
            up = 1.0 / scale if (i, s) == (1, 0) else 1.0
            Q, R, Q1, R1 = few[s][i], few[s + 1][i] * up, many[s][i], many[s + 1][i] * up
            K = R.shape[0]
            assert np.linalg.norm(Q.conj().T @ Q - np.eye(K)) <= 1e-10
            assert np.allclose(np.tril(R, -1), 0, atol=0) and (np.diagonal(R).real >= 0).all()
            assert np.linalg.norm(R - R1) <= 1e-9 * np.linalg.norm(R1)
            assert np.linalg.norm(Q @ R - Q1 @ R1) <= 1e-9 * np.linalg.norm(R1)


def test_trivial_reflectors():
    """A site tensor whose gated columns are already triangular (identity gate,
    unit entries): every reflector is trivial and R is diagonal."""
    D = 4
    T = np.zeros((1, 2, D, D, D, D), dtype=np.complex128)
    for k in range(D):
        T[0, 0, 0, 0, k, k] = 1.0 + k                    # right leg k, row k
    few = _qr(D, 1, 2, 1, T, T.transpose(0, 1, 4, 3, 2, 5), I.identity_gate()[None])
    Q, R = few[0][0], few[1][0]
    ref = np.abs(np.diagonal(R))
    assert np.allclose(np.abs(R), np.diag(ref), atol=1e-14)
    assert np.allclose(ref / ref[0], 1.0 + np.arange(D), atol=1e-13)
    assert np.linalg.norm(Q.conj().T @ Q - np.eye(D)) <= 1e-13
