"""The FP64 direct sum, the FP64 P2P and the FP64 M2L and M2M at the edges of their work splits (sinks per block, slices
of the sources, slots and replicas of a leaf, pieces of a long item) against plain FP64 sums."""
import numpy as np
import pytest

from paper_1405_2255_gb300 import inputs

pytestmark = pytest.mark.gpu

# a sum of up to 6000 FP64 terms in any order, each term good to a few ulp: (6000 + 10) 2^-53 of the
# sum of the terms' magnitudes is 7e-13
TOL = 1e-12


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


def _sums(x, mu, sinks):
    """psi, acc, f and the sums of the magnitudes of acc's terms, by numpy."""
    psi, acc, f = np.zeros(len(sinks)), np.zeros((len(sinks), 3)), np.zeros(len(sinks))
    for b in range(0, len(sinks), 500):
        d = x[None] - x[sinks[b:b + 500], None]
        r2 = (d * d).sum(2)
        ri = np.where(r2 > 0, 1.0 / np.sqrt(np.where(r2 > 0, r2, 1.0)), 0.0)
        psi[b:b + 500] = (mu * ri).sum(1)
        f[b:b + 500] = (mu * ri * ri).sum(1)
        acc[b:b + 500] = ((mu * ri ** 3)[:, :, None] * d).sum(1)
    return psi, acc, f


def _check(psi, acc, ref):
    p, a, f = ref
    scale = np.maximum(f, 1e-300)  # sum of |terms| of each component of acc is at most f
    assert np.max(np.abs(psi - p) / np.maximum(p, 1e-300)) < TOL
    assert np.max(np.abs(acc - a) / scale[:, None]) < TOL


@pytest.mark.parametrize("n,ns", [(1, 1), (31, 1), (257, 3), (1000, 33), (999, 250), (2049, 1217), (300, 9728),
                                  (257, 38912), (130, 40001)])
@pytest.mark.parametrize("want_f", [False, True])
def test_direct_splits(g, n, ns, want_f):
    x, mu = inputs.plummer(n, 900 + n)
    if n > 300:
        mu[::7] = 0.0
        x[11] = x[12]  # a coincident pair
    sinks = (np.arange(ns) * 7919) % n
    ctx = g.Context()
    out = ctx.fmm_direct(_dev(x), _dev(mu), 1.0, sinks=_dev(sinks.astype(np.int64)), want_f=want_f)
    ref = _sums(x, mu, np.arange(n))
    ref = tuple(v[sinks] for v in ref)
    _check(out[0].cpu().numpy(), out[1].cpu().numpy(), ref)
    if want_f:
        assert np.max(np.abs(out[2].cpu().numpy() - ref[2]) / np.maximum(ref[2], 1e-300)) < TOL
    ctx.close()


@pytest.mark.parametrize("n", [2, 8, 112, 113, 224, 225, 448, 449, 897])
@pytest.mark.parametrize("ns", [1, 40])
def test_direct_slices_of_few_sources(g, n, ns):
    """One, two, four and eight slices of the sources, warps without any among them."""
    x, mu = inputs.plummer(n, 940 + n)
    sinks = (np.arange(ns) * 7919) % n
    ctx = g.Context()
    out = ctx.fmm_direct(_dev(x), _dev(mu), 1.0, sinks=_dev(sinks.astype(np.int64)), want_f=True)
    ctx.close()
    ref = tuple(v[sinks] for v in _sums(x, mu, np.arange(n)))
    _check(out[0].cpu().numpy(), out[1].cpu().numpy(), ref)
    assert np.max(np.abs(out[2].cpu().numpy() - ref[2]) / np.maximum(ref[2], 1e-300)) < TOL


@pytest.mark.parametrize("n,leaf", [(2, 1), (33, 1), (500, 3), (777, 17), (1500, 33), (2000, 65), (5001, 64),
                                    (4000, 130), (3000, 1000), (700, 4096)])
@pytest.mark.parametrize("mac", [0, 1])
def test_fp64_p2p_splits(g, n, leaf, mac):
    """With eps near 0 every pair is summed directly, so the evaluation is the direct sum: leaves of
    1 to 4096 sinks, items with and without pieces, a coincident pair."""
    x, mu = inputs.plummer(n, 950 + n)
    if n > 300:
        x[20] = x[21]
    ctx = g.Context(p=3, eps=1e-30, leaf_size=leaf, p2p_c=1.0, mac=mac, precision=g.FMM_PREC_FP64)
    psi, acc, st = ctx.fmm_evaluate(_dev(x), _dev(mu), stats=True)
    assert st["n_m2l"] == 0
    _check(psi.cpu().numpy(), acc.cpu().numpy(), _sums(x, mu, np.arange(n)))
    ctx.close()


@pytest.mark.parametrize("m", [0.0, 1e-20])
def test_subnormal_squared_distance(g, m):
    """Two light particles whose squared distance is subnormal (1e-310, with a dozen digits) and one of
    mass 1: a massless source adds nothing, and mu / r^2 is finite where its value is."""
    x = np.zeros((3, 3))
    x[1, 0], x[2, 0] = 1e-155, 1.0
    mu = np.array([m, m, 1.0])
    near = m * 1e155 * 1e155  # mu / r^2
    ctx = g.Context(p=3, leaf_size=8, mac=1, precision=g.FMM_PREC_FP64)
    psi, acc, f = (t.cpu().numpy() for t in ctx.fmm_direct(_dev(x), _dev(mu), want_f=True))
    psi2, acc2 = (t.cpu().numpy() for t in ctx.fmm_evaluate(_dev(x), _dev(mu)))
    d = ctx.fmm_debug_dump()
    f2 = np.empty(3)
    f2[d["perm"]] = d["scale"]
    ctx.close()
    for p, a, ff in ((psi, acc, f), (psi2, acc2, f2)):
        assert np.allclose(p, [1.0 + m * 1e155, 1.0 + m * 1e155, 2 * m], rtol=1e-12, atol=0)
        assert np.allclose(ff, [1.0 + near, 1.0 + near, 2 * m], rtol=1e-12, atol=0)
        assert np.allclose(a[2], [-2 * m, 0, 0], rtol=1e-12, atol=0)
        if m == 0.0:
            assert np.array_equal(a[:2], [[1.0, 0, 0], [1.0, 0, 0]])


@pytest.mark.parametrize("p", [1, 2, 3, 9, 16, 17, 18])
@pytest.mark.parametrize("shape", ["plummer", "z axis", "x axis", "plane"])
def test_fp64_m2l_orders_and_directions(g, orc, p, shape):
    """Every order class of the rotated M2L, with interaction directions along the axes (where the
    rotation angle about z is undefined) among them: tree, lists and forces equal the oracle's
    to 1e-10 of the sum of the magnitudes of a sink's terms (f of eq. 6; on a line neighbours on both
    sides cancel).  The geometric criterion gives lists of all lengths."""
    x, mu = inputs.plummer(3000, inputs.BASE_SEED + 31)
    if shape == "z axis":
        x[:, :2] = 0.0
    elif shape == "x axis":
        x[:, 1:] = 0.0
    elif shape == "plane":
        x[:, 2] = 0.0
    prm = dict(p=p, mac=2, theta_crit=0.6, leaf_size=12, p2p_c=0.0)
    ctx = g.Context(precision=g.FMM_PREC_FP64, **prm)
    psi, acc, st = ctx.fmm_evaluate(_dev(x), _dev(mu), stats=True)
    ctx.close()
    run = orc.fmm(x, mu, **prm)
    assert st["n_m2l"] == run.stats["n_m2l"] > 1000
    f = orc.direct(x, mu)[2]
    assert np.max(np.linalg.norm(acc.cpu().numpy() - run.acc, axis=1) / f) <= 1e-10
    assert np.max(np.abs(psi.cpu().numpy() - run.psi) / run.psi) <= 1e-10
