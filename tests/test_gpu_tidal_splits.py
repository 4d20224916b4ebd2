"""The mixed-precision tidal tensor at the edges of its work split (slots, groups, tiles and batches of
tiles, pieces) and orders of its far part, against plain FP64 sums and the FP64 mode."""
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


@pytest.mark.parametrize("n,leaf", [(2, 1), (33, 1), (500, 3), (777, 17), (1500, 33), (2000, 65), (5001, 64),
                                    (4000, 130), (3000, 1000), (4096, 4096)])
def test_mixed_near_tidal_splits(g, n, leaf):
    """With eps near 0 every pair is direct.  A pair's FP32 term is good to about 2^-20 of its magnitude
    (r^-5 of an r good to 2^-23) and a tile sums at most 32 of them: 4e-6 of the sum of the terms'
    magnitudes (3 mu / r^3) bounds both.  A coincident pair is skipped."""
    x, mu = inputs.plummer(n, 970 + n)
    if n > 300:
        x[20] = x[21]
    ctx = g.Context(p=3, eps=1e-30, leaf_size=leaf, p2p_c=1.0, precision=g.FMM_PREC_MIXED)
    psi, acc, T, st = ctx.fmm_evaluate_active(_dev(x), _dev(mu), tidal=True, stats=True)
    ctx.close()
    assert st["n_m2l"] == 0
    T = T.cpu().numpy()
    ref, mag = np.zeros((n, 6)), np.zeros(n)
    for b in range(0, n, 500):
        d = x[None] - x[b:b + 500, None]
        r2 = (d * d).sum(2)
        q3 = np.where(r2 > 0, mu / np.where(r2 > 0, r2, 1.0) ** 1.5, 0.0)
        q5 = np.where(r2 > 0, q3 / np.where(r2 > 0, r2, 1.0), 0.0)
        mag[b:b + 500] = 3 * q3.sum(1)
        for k, (i, j) in enumerate([(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]):
            ref[b:b + 500, k] = (3 * q5 * d[:, :, i] * d[:, :, j] - (q3 if i == j else 0.0)).sum(1)
    assert np.max(np.abs(T - ref) / mag[:, None]) < 4e-6


def _near_ref(x, mu):
    """Plain FP64 sums over all pairs, and the sums of the terms' magnitudes."""
    d = x[None] - x[:, None]
    r2 = (d * d).sum(2)
    q3 = np.where(r2 > 0, mu / np.where(r2 > 0, r2, 1.0) ** 1.5, 0.0)
    q5 = np.where(r2 > 0, q3 / np.where(r2 > 0, r2, 1.0), 0.0)
    ref = [(3 * q5 * d[:, :, i] * d[:, :, j] - (q3 if i == j else 0.0)).sum(1)
           for i, j in [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]]
    return np.stack(ref, 1), 3 * q3.sum(1)


@pytest.mark.parametrize("r", [2.0 ** k for k in (-62, -64, -68, -71, -74, -77)])
@pytest.mark.parametrize("leaf", [1, 9, 17, 40])
def test_mixed_near_tidal_at_the_origin(g, leaf, r):
    """A particle so near the origin that its squared distance from it is an FP32 subnormal (or 0): the
    fillers of short tiles add nothing wherever it lies (bound as in test_mixed_near_tidal_splits)."""
    x, mu = inputs.plummer(1200, 41)
    x[7] = (r, 0.0, 0.0)
    ctx = g.Context(p=3, eps=1e-30, leaf_size=leaf, p2p_c=1.0, precision=g.FMM_PREC_MIXED)
    T = ctx.fmm_evaluate_active(_dev(x), _dev(mu), tidal=True)[2].cpu().numpy()
    ctx.close()
    ref, mag = _near_ref(x, mu)
    assert np.max(np.abs(T - ref) / mag[:, None]) < 4e-6


@pytest.mark.parametrize("n", [1, 2, 5])
@pytest.mark.parametrize("at", [1e15, 1e19, 1e20, 1e30, 3e38])
def test_mixed_near_tidal_of_one_place(g, n, at):
    """All particles at one place (no extent to scale by): the tensor is 0 at any coordinates."""
    x, mu = np.full((n, 3), at), np.ones(n)
    ctx = g.Context(p=3, leaf_size=8, precision=g.FMM_PREC_MIXED)
    T = ctx.fmm_evaluate_active(_dev(x), _dev(mu), tidal=True)[2].cpu().numpy()
    ctx.close()
    assert np.array_equal(T, np.zeros((n, 6)))


@pytest.mark.parametrize("n", [1, 3, 20])
@pytest.mark.parametrize("at", [2.0 ** 127, 1e39, -1e100, 1e300])
def test_one_place_beyond_fp32(g, n, at):
    """The same where the coordinates have no FP32 value: every result is 0."""
    x, mu = np.full((n, 3), at), np.full(n, 0.5)
    ctx = g.Context(p=3, leaf_size=8, precision=g.FMM_PREC_MIXED)
    out = ctx.fmm_evaluate_active(_dev(x), _dev(mu), tidal=True)
    ctx.close()
    for t in out:
        assert np.array_equal(t.cpu().numpy(), np.zeros(tuple(t.shape)))


@pytest.mark.parametrize("p", [1, 2, 3, 7, 14, 18])
def test_far_tidal_orders(g, orc, p):
    """The far part alone differs from the oracle's only by FP64 rounding (FP64 mode, 1e-10 of the
    largest entry; lists of the geometric criterion)."""
    x, mu = inputs.plummer(2500, inputs.BASE_SEED + 33)
    prm = dict(p=p, mac=2, theta_crit=0.6, leaf_size=13, p2p_c=0.0)
    ctx = g.Context(precision=g.FMM_PREC_FP64, **prm)
    _, _, T = ctx.fmm_evaluate_active(_dev(x), _dev(mu), tidal=True)
    ctx.close()
    run = orc.fmm(x, mu, tidal=True, **prm)
    scale = np.maximum(np.abs(run.tidal).max(axis=1, keepdims=True), 1e-300)  # (p = 1: 0 without near sources)
    assert np.max(np.abs(T.cpu().numpy() - run.tidal) / scale) < 1e-10
