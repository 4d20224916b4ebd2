"""The mixed-precision P2P of small systems, whose pieces are cut into parts at tile boundaries, at the
edges of that cut, against plain FP64 sums; and an ensemble against its systems alone (the cut depends
on a system's own size)."""
import numpy as np
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


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


@pytest.mark.parametrize("n,leaf", [(1100, 2000), (3000, 1), (4097, 7), (6000, 33), (9001, 64), (12000, 130),
                                    (16384, 48), (16385, 48)])
def test_mixed_p2p_parts(g, n, leaf):
    """With eps near 0 every pair is direct.  A pair's FP32 term is good to 3 times the rsqrt
    approximation's 2^-22 and a few roundings (1.2e-6), an FP32 sum of at most 64 of them adds at most
    64 x 2^-24: 6e-6 of the sum of the terms' magnitudes bounds both."""
    x, mu = inputs.plummer(n, 990 + n)
    x[20] = x[21]
    ctx = g.Context(p=3, eps=1e-30, leaf_size=leaf, p2p_c=1.0, precision=g.FMM_PREC_MIXED)
    psi, acc, st = ctx.fmm_evaluate(_dev(x), _dev(mu), stats=True)
    assert st["n_m2l"] == 0
    p, a, f = ctx.fmm_direct(_dev(x), _dev(mu), want_f=True)
    ctx.close()
    assert float(((psi - p).abs() / p).max()) < 6e-6
    assert float(((acc - a).abs() / f[:, None]).max()) < 6e-6


def test_parts_alone_and_in_an_ensemble(g):
    import torch
    sizes = [16384, 16385, 3000, 1, 9000]
    sys_ = [inputs.plummer(k, 70 + k) for k in sizes]
    prm = dict(p=10, eps=1e-6, leaf_size=40, p2p_c=1.0)
    ctx = g.Context(**prm)
    alone = [ctx.fmm_evaluate(_dev(x), _dev(mu)) for x, mu in sys_]
    off = np.concatenate([[0], np.cumsum(sizes)])
    psi, acc = ctx.fmm_evaluate_batch(off, _dev(np.concatenate([x for x, _ in sys_])),
                                      _dev(np.concatenate([m for _, m in sys_])), np.ones(len(sizes)))
    ctx.close()
    for k, (p, a) in enumerate(alone):
        assert torch.equal(psi[off[k]:off[k + 1]], p) and torch.equal(acc[off[k]:off[k + 1]], a)
