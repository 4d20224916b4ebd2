"""Contexts of different orders on two host threads: what they share (kernels' limits, tables) does not
depend on who comes first."""
import threading

import pytest

from paper_1405_2255_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1405_2255_gb300 import build
    build.build()
    from paper_1405_2255_gb300 import gb3fmm
    gb3fmm.load()
    return gb3fmm


@pytest.mark.parametrize("n,rounds,prm", [(150, 1500, dict(precision=0)), (3000, 100, dict(precision=0)),
                                          (150, 800, dict(precision=1, m2l_rot=0)), (12_000, 100, dict(leaf_size=8))])
def test_two_orders_on_four_threads(g, n, rounds, prm):
    """Every thread gets the bits of its first call, made alone, and no launch is refused (a launch falls
    between another thread's setting of a limit and its launch a few times in a thousand calls)."""
    import torch
    x, mu = (torch.from_numpy(a).to("cuda:0") for a in inputs.plummer(n, 19))
    work = []
    for p in (6, 18, 7, 17):
        ctx = g.Context(**{**dict(p=p, eps=1e-3, leaf_size=4, p2p_c=0.0), **prm})
        work.append((ctx, torch.cuda.Stream(), [t.clone() for t in ctx.fmm_evaluate_active(x, mu, tidal=True)]))
    torch.cuda.synchronize()
    errors = []

    def loop(ctx, stream, ref):
        try:
            with torch.cuda.stream(stream):
                T = torch.empty_like(ref[2])
                psi, acc = torch.empty_like(ref[0]), torch.empty_like(ref[1])
                for k in range(rounds):
                    out = ctx.fmm_evaluate_active(x, mu, psi=psi, acc=acc, tidal=T)
                    if k % 20 == 19:
                        stream.synchronize()
                        if not all(torch.equal(a, b) for a, b in zip(out, ref)):
                            errors.append("different bits")
                            return
        except Exception as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=loop, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for ctx, _, _ in work:
        ctx.close()
    assert not errors, errors
