"""The device sorts at the edges of their tiles (2048 items): the particle order against a stable sort
of the Morton keys, and the interaction lists in strict (sink, source) order."""
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


def _morton(x):
    lo = x.min(0)
    side = (x - lo).max() * (1 + 2.0 ** -20)
    q = np.clip(np.floor((x - lo) / side * 2097152.0).astype(np.int64), 0, 2097151).astype(np.uint64)
    key = np.zeros(len(x), np.uint64)
    for b in range(21):
        for d in range(3):
            key |= ((q[:, d] >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + 2 - d)
    return key


@pytest.mark.parametrize("n", [2, 31, 2047, 2048, 2049, 4097, 16385, 70001, 300007])
def test_order_and_lists(g, n):
    x, mu = inputs.plummer(n, 300 + n)
    if n > 1000:
        x[5:400] = x[5]  # equal keys keep the caller's order
    ctx = g.Context(p=6, eps=1e-5, leaf_size=32, p2p_c=1.0)
    ctx.fmm_evaluate(_dev(x), _dev(mu))
    d = ctx.fmm_debug_dump()
    ctx.close()
    assert np.array_equal(d["perm"], np.argsort(_morton(x), kind="stable"))
    for lst in (d["m2l"], d["p2p"]):
        key = lst[:, 1] * (1 << 32) + lst[:, 0]
        assert np.all(np.diff(key) > 0)


@pytest.mark.parametrize("n", [8191, 8192, 8193, 16384, 16385, 32768, 32769, 65536, 65537])
@pytest.mark.parametrize("leaf", [16, 256])
def test_order_and_lists_in_one_cluster(g, n, leaf):
    """Sizes at the edges of the sort in one cluster (items per thread 1, 2, 4, 8, then the passes as
    launches); lists of about 1e4 to 1e6 pairs."""
    x, mu = inputs.plummer(n, 400 + n)
    x[7:900] = x[7]
    ctx = g.Context(p=6, eps=1e-5, leaf_size=leaf, p2p_c=1.0)
    ctx.fmm_evaluate(_dev(x), _dev(mu))
    d = ctx.fmm_debug_dump()
    ctx.close()
    assert np.array_equal(d["perm"], np.argsort(_morton(x), kind="stable"))
    for lst in (d["m2l"], d["p2p"]):
        key = lst[:, 1] * (1 << 32) + lst[:, 0]
        assert np.all(np.diff(key) > 0)
