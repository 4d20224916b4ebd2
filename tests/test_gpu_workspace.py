"""The workspace stays within fmm_footprint_bytes where work plans hold partial sums of split items, and a
system's pieces do not depend on the systems beside it."""
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


SHAPES = [(64, 8, 8.0), (64, 6, 1.0), (96, 10, 4.0), (256, 10, 8.0), (512, 8, 8.0), (1024, 8, 8.0), (4096, 8, 8.0)]


@pytest.mark.parametrize("model,n", [("plummer", 200_000), ("dehnen", 200_000), ("plummer", 16_384), ("dehnen", 50_000)])
@pytest.mark.parametrize("leaf,p,c", SHAPES)
@pytest.mark.parametrize("mac", [0, 1])
def test_fp64_workspace_within_footprint(g, model, n, leaf, p, c, mac):
    if n * leaf > 200_000 * 1024:
        pytest.skip("near the direct sum: seconds")
    x, mu = getattr(inputs, model)(n, 77)
    prm = dict(p=p, eps=1e-6, leaf_size=leaf, p2p_c=c, mac=mac, precision=g.FMM_PREC_FP64)
    ctx = g.Context(**prm)
    ctx.fmm_evaluate(_dev(x), _dev(mu))
    assert ctx.fmm_workspace_bytes() <= g.fmm_footprint_bytes(n, **prm)
    ctx.close()


@pytest.mark.parametrize("model", ["plummer", "dehnen"])
@pytest.mark.parametrize("leaf,p", [(8, 4), (16, 5), (32, 5)])
def test_fp64_workspace_of_long_lists(g, model, leaf, p):
    """Low orders: the P2P lists are long, and so are the plan's ranges."""
    n = 50_000
    x, mu = getattr(inputs, model)(n, 77)
    prm = dict(p=p, eps=1e-6, leaf_size=leaf, p2p_c=1.0, precision=g.FMM_PREC_FP64)
    ctx = g.Context(**prm)
    ctx.fmm_evaluate(_dev(x), _dev(mu))
    assert ctx.fmm_workspace_bytes() <= g.fmm_footprint_bytes(n, **prm)
    ctx.close()


@pytest.mark.parametrize("leaf,p,c", SHAPES[:4])
@pytest.mark.parametrize("mac", [0, 1])
def test_tidal_workspace_within_footprint(g, leaf, p, c, mac):
    """Mixed mode: the tidal plan and the f estimate's (the bound itself, made for forces, holds here too)."""
    n = 200_000
    x, mu = inputs.plummer(n, 77)
    prm = dict(p=p, eps=1e-6, leaf_size=leaf, p2p_c=c, mac=mac, precision=g.FMM_PREC_MIXED)
    ctx = g.Context(**prm)
    ctx.fmm_evaluate_active(_dev(x), _dev(mu), tidal=True)
    assert ctx.fmm_workspace_bytes() <= g.fmm_footprint_bytes(n, **prm)
    ctx.close()


@pytest.mark.parametrize("model", ["plummer", "dehnen"])
@pytest.mark.parametrize("n", [9_000, 16_384])
@pytest.mark.parametrize("leaf,p,c", [(8, 6, 1.0), (16, 6, 1.0), (32, 5, 1.0), (32, 6, 1.0), (48, 14, 1.0),
                                      (512, 8, 8.0)])
def test_small_mixed_workspace_within_footprint(g, model, n, leaf, p, c):
    """Systems whose pieces are shared by several warps (the parts have records of their own)."""
    x, mu = getattr(inputs, model)(n, 77)
    prm = dict(p=p, eps=1e-6, leaf_size=leaf, p2p_c=c, precision=g.FMM_PREC_MIXED)
    ctx = g.Context(**prm)
    ctx.fmm_evaluate(_dev(x), _dev(mu))
    assert ctx.fmm_workspace_bytes() <= g.fmm_footprint_bytes(n, **prm)
    ctx.close()


@pytest.mark.parametrize("mac", [0, 1])
def test_pieces_in_an_ensemble_as_alone(g, mac):
    """Systems whose pieces have the least length and longer ones, together and alone: the same bits."""
    sizes = [20_000, 700, 0, 40_000, 5_000, 1]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    parts = [inputs.plummer(s, 50 + k) if s else (np.zeros((0, 3)), np.zeros(0)) for k, s in enumerate(sizes)]
    x, mu = np.concatenate([q[0] for q in parts]), np.concatenate([q[1] for q in parts])
    ctx = g.Context(p=8, eps=1e-6, leaf_size=512, p2p_c=8.0, mac=mac, precision=g.FMM_PREC_FP64)
    psi, acc = (t.cpu().numpy() for t in ctx.fmm_evaluate_batch(off, _dev(x), _dev(mu), 1.0))
    for k, s in enumerate(sizes):
        if s:
            p1, a1 = (t.cpu().numpy() for t in ctx.fmm_evaluate(_dev(parts[k][0]), _dev(parts[k][1])))
            assert np.array_equal(p1, psi[off[k]:off[k + 1]]) and np.array_equal(a1, acc[off[k]:off[k + 1]])
    ctx.close()
