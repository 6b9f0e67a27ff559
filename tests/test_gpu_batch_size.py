"""An item's result in an FP64 context does not depend on how many items go with
it: few items run their QR and recomposition on clusters of CTAs, many on one CTA
each, and both give the same bits (so the uneven modes agree, and the
allocation-free entry with the context's)."""
import numpy as np
import pytest

from paper_2107_06635_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _stages(D, r, d, d_anc, max_batch, Ta, Tb, G, MA, MB):
    """gate_qr and recompose of the given items."""
    import torch

    from paper_2107_06635_gb300 import ntu

    n, m, K = len(Ta), d * d_anc * D ** 3, D * r
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    new = lambda *s: torch.empty((n, *s), dtype=torch.complex128, device="cuda")  # noqa: E731
    QA, QB, RA, RB = new(m, K), new(m, K), new(K, K), new(K, K)
    Ta, Tb, G, MA, MB = (dev(x) for x in (Ta, Tb, G, MA, MB))
    oa, ob = torch.empty_like(Ta), torch.empty_like(Tb)
    torch.cuda.synchronize()
    with ntu.Context(D, d, d_anc, r, max_batch=max_batch) as ctx:
        ctx.batch_gate_qr_dev(n, Ta, Tb, G, QA, RA, QB, RB)
        ctx.batch_recompose_dev(n, QA, QB, MA, MB, oa, ob)
        ctx.sync()
    return [x.cpu().numpy() for x in (QA, RA, QB, RB, oa, ob)]


# m = d_p D^3 from 128 (the smallest on clusters), odd columns, K = 32
@pytest.mark.parametrize("D,r,d,d_anc", [(4, 2, 2, 1), (4, 4, 4, 1), (5, 1, 2, 1), (5, 3, 2, 1), (7, 2, 2, 1), (7, 3, 3, 1),
                                         (8, 2, 2, 1), (8, 4, 2, 4)])
def test_few_items_have_the_bits_of_many(D, r, d, d_anc):
    rng = np.random.default_rng(17 * D + r)
    n, K = 24, D * r
    Ta, Tb = (np.stack([I.random_site_tensor(rng, d * d_anc, D) for _ in range(n)]) for _ in range(2))
    Ta[1] *= 1e-170
    Tb[2, :, 1:] = 0                                     # columns of zeros: trivial reflectors
    G = np.stack([I.random_gate(rng, d) for _ in range(n)])
    MA, MB = (rng.standard_normal((n, K, D)) + 1j * rng.standard_normal((n, K, D)) for _ in range(2))
    many = _stages(D, r, d, d_anc, n, Ta, Tb, G, MA, MB)
    for max_batch in (3, n):
        few = _stages(D, r, d, d_anc, max_batch, *(x[:3] for x in (Ta, Tb, G, MA, MB)))
        for a, b in zip(few, many):
            assert np.array_equal(a, b[:3])


def test_uneven_modes_agree_in_fp64():
    from paper_2107_06635_gb300 import ntu

    rng = np.random.default_rng(9)
    kinds, caps = [(4, 2), (5, 2)], [12, 11]
    items = []
    for k, (D, r) in enumerate(kinds):
        for _ in range(caps[k]):
            ta, tb = (I.random_site_tensor(rng, 2, D) for _ in range(2))
            items.append((D, r, ta, tb, I.random_gate(rng)))
    ub = ntu.UnevenBatch(kinds, caps, sweeps=2)
    ub.stage(items)
    res = {}
    for mode in (ub.GROUPED, ub.GRAPH, ub.PER_ITEM):
        ub.run(mode)
        ub.sync()
        res[mode] = ub.fetch(items)
    ub.close()
    for mode in (ub.GRAPH, ub.PER_ITEM):
        for a, b in zip(res[mode], res[ub.GROUPED]):
            assert all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("D,r", [(4, 4), (8, 2)])
def test_noalloc_has_the_context_bits(D, r):
    import torch

    from paper_2107_06635_gb300 import ntu

    rng = np.random.default_rng(D)
    m, K = 2 * D ** 3, D * r
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    ta, tb = (dev(I.random_site_tensor(rng, 2, D)) for _ in range(2))
    gg = dev(I.random_gate(rng))
    shapes = ((m, K), (K, K), (m, K), (K, K))
    ref, out = ([torch.empty(s, dtype=torch.complex128, device="cuda") for s in shapes] for _ in range(2))
    with ntu.Context(D, r=r) as ctx:
        ctx.batch_gate_qr_dev(1, ta, tb, gg, *ref)
        ctx.sync()
    assert ntu.load().ntu_gate_qr_noalloc(D, 2, 1, r, ta.data_ptr(), tb.data_ptr(), gg.data_ptr(),
                                          *(o.data_ptr() for o in out), None) == 0
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(out, ref))
