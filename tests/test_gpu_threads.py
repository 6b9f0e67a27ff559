"""Contexts of different sizes used by a host thread each at the same time: what
one sets on a kernel must not be what another launches with."""
import threading

import numpy as np
import pytest

from paper_2107_06635_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["NTU_MIXED_FP32", "NTU_FP64"])
def test_threads_with_their_own_contexts(precision):
    """The FP32 products of D = 2 (sums of one stage) and D = 6 (of one and of
    three) run in the same tile.  Every call succeeds and every thread's last
    metric equals its first, taken alone."""
    import torch

    from paper_2107_06635_gb300 import ntu

    errors, sizes = [], (2, 6, 2, 6)
    gate = threading.Barrier(len(sizes))

    def inputs(D):
        rng = np.random.default_rng(D)
        dev = lambda x: torch.from_numpy(np.ascontiguousarray(x[None])).cuda()  # noqa: E731
        q = lambda: np.linalg.qr(rng.standard_normal((2 * D ** 3, 2 * D)) + 0j)[0]  # noqa: E731
        return [dev(I.random_site_tensor(rng, 2, D)) for _ in range(2)] + [dev(q()) for _ in range(2)]

    def work(D, args, first, last, calls):
        try:
            with ntu.Context(D, precision=getattr(ntu, precision), tau_kmax=8) as ctx:
                ctx.batch_env_dev(1, *args, first)
                ctx.sync()
                gate.wait()
                for _ in range(calls):
                    ctx.batch_env_dev(1, *args, last)
                ctx.sync()
        except Exception as e:  # noqa: BLE001
            errors.append((D, repr(e)))
            gate.abort()

    state = []
    for D in sizes:
        g = [torch.zeros((1, 4 * D * D, 4 * D * D), dtype=torch.complex128, device="cuda") for _ in range(2)]
        state.append((D, inputs(D), *g, 1500))
    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=s) for s in state]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for _, _, first, last, _ in state:
        assert torch.equal(first, last) and torch.isfinite(torch.view_as_real(first)).all()
