"""The FP64 front elimination on the tensor cores (exact integer digit products)
and the panel over a thread-block cluster, against the CUDA-core sweep and
the shared-memory panel.

Tolerances.  Both sides are float64 eliminations of the same fronts in another
blocking; a block's relative difference is c kappa u64.  On the parity
problems c kappa is below 1e3 (7e-6 measured at u = 4.8e-7 in FP32); 1e-11
allows 1e5, and 1e-10 for A_ii^{-1}, whose entries carry one more factor of
the condition number.  Scaling the matrix by a power of two scales every
intermediate value exactly (nothing under- or overflows at 2^+-700 here), so
that comparison is bit for bit.
"""
import numpy as np
import pytest

from ndhss_inputs import helmholtz_impedance, poisson_dirichlet
from closeness import rel as _rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def nd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_07791_gb300 import build, ndhss
    build.build()
    ndhss.load()
    return ndhss


def _problem(kind, N, p):
    return poisson_dirichlet(N, p=p, seed=2) if kind == "poisson" else helmholtz_impedance(N, p, 0.2 * N * p, seed=2)


def _factor(nd, tree, A, **kw):
    M = nd.DeviceCSR(A)
    return nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(prec=0, **kw))


def _compare(nd, tree, fa, fb, top):
    info = nd.ndhss_tree_export(tree)["node_info"]
    for s in np.argsort(-info[:, 5], kind="stable")[:top]:
        mi, mb = int(info[s, 5]), int(info[s, 7])
        for w in range(4 if mb else 1):
            a = nd.ndhss_factor_get_block(fa, int(s), w, mi, mb)
            b = nd.ndhss_factor_get_block(fb, int(s), w, mi, mb)
            assert _rel(a, b) <= (1e-10 if w == 0 else 1e-11), (s, w, mi, mb, _rel(a, b))


# leaves of 16 and 64 unknowns put the switch between both sweeps on different
# levels; the odd grids give interior blocks off the 16- and 64-pivot blocks;
# width 4 panels leave partly filled operands
@pytest.mark.parametrize("kind,N,p,leaf,panel", [("poisson", 53, 1, 16, 0), ("poisson", 61, 2, 64, 0),
                                                 ("helmholtz", 47, 1, 64, 0), ("helmholtz", 45, 2, 64, 4),
                                                 ("helmholtz", 100, 2, 64, 0)])
def test_fp64_tensor_core_sweep_matches_cuda_core_sweep(nd, kind, N, p, leaf, panel, monkeypatch):
    P = _problem(kind, N, p)
    tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, leaf)
    fa = _factor(nd, tree, P.A, panel=panel)
    monkeypatch.setenv("NDHSS_FRONT_UPDATE", "simt")
    fb = _factor(nd, tree, P.A, panel=panel)
    assert nd.ndhss_factor_stats_get(fa)["tc_flops"] > 0 and nd.ndhss_factor_stats_get(fb)["tc_flops"] == 0
    _compare(nd, tree, fa, fb, 40)


@pytest.mark.parametrize("kind,e", [("poisson", 700), ("helmholtz", -700)])
def test_fp64_factor_scales_exactly(nd, kind, e):
    P = _problem(kind, 40, 2)
    tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, 64)
    fa = _factor(nd, tree, P.A)
    fb = _factor(nd, tree, P.A * 2.0 ** e)
    x = torch.from_numpy(np.random.default_rng(0).standard_normal(P.n).astype(P.A.dtype)).cuda()
    ya = nd.ndhss_apply(fa, x, torch.empty_like(x))
    yb = nd.ndhss_apply(fb, x, torch.empty_like(x)) * 2.0 ** e
    assert torch.equal(ya, yb)


def test_fp64_cluster_panel_matches_shared_memory_panel(nd, monkeypatch):
    """A root front of ~600 complex interior unknowns: panels over up to eight
    CTAs against the panel in one CTA's shared memory (same pivots)."""
    P = _problem("helmholtz", 100, 2)
    tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, 64)
    fa = _factor(nd, tree, P.A)
    monkeypatch.setenv("NDHSS_PANEL", "smem")
    fb = _factor(nd, tree, P.A)
    _compare(nd, tree, fa, fb, 15)
