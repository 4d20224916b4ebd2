"""The shifts of the expansions (P2M, M2M, L2L, L2P) at every number of warps per cell: the FP64 ones against
the oracle, the mixed ones of a system in a wide batch (a block per parent) against the system alone (a cluster
per parent)."""
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


@pytest.mark.parametrize("p", [4, 6, 7, 9, 10, 13, 14, 15, 19, 20])
@pytest.mark.parametrize("leaf", [3, 40])
def test_fp64_orders(g, orc, p, leaf):
    """1e-10 of the sum of the magnitudes of a sink's terms: the FP64 rounding of some 1e4 terms of an
    expansion, each good to (p + 10) 2^-53, is below 1e-11."""
    x, mu = inputs.plummer(2500, inputs.BASE_SEED + 57)
    prm = dict(p=p, mac=2, theta_crit=0.7, leaf_size=leaf, p2p_c=0.0)
    ctx = g.Context(precision=g.FMM_PREC_FP64, **prm)
    psi, acc, _ = ctx.fmm_evaluate(_dev(x), _dev(mu), stats=True)
    ctx.close()
    run = orc.fmm(x, mu, **prm)
    f = orc.direct(x, mu)[2]
    assert np.max(np.linalg.norm(acc.cpu().numpy() - run.acc, axis=1) / f) <= 1e-10
    assert np.max(np.abs(psi.cpu().numpy() - run.psi) / run.psi) <= 1e-10


@pytest.mark.parametrize("p", [3, 6, 7, 9, 10, 14, 16, 20])
def test_mixed_batch_of_wide_levels(g, p):
    """60 systems of 2000 with leaves of at most 4: more than 6 x 152 parents on a level."""
    ns = 60
    parts = [inputs.plummer(2000, 3000 + i) for i in range(ns)]
    x, mu = np.concatenate([a[0] for a in parts]), np.concatenate([a[1] for a in parts])
    off = np.arange(ns + 1, dtype=np.int64) * 2000
    ctx = g.Context(p=p, mac=2, theta_crit=0.6, leaf_size=4, p2p_c=0.0)
    psi, acc = ctx.fmm_evaluate_batch(off, _dev(x), _dev(mu), np.ones(ns), stats=True)[:2]
    psi, acc = psi.cpu().numpy(), acc.cpu().numpy()
    for i in (0, 31, 59):
        p1, a1 = ctx.fmm_evaluate(_dev(parts[i][0]), _dev(parts[i][1]), 1.0, stats=True)[:2]
        assert np.array_equal(psi[off[i]:off[i + 1]], p1.cpu().numpy())
        assert np.array_equal(acc[off[i]:off[i + 1]], a1.cpu().numpy())
    ctx.close()
