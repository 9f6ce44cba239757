"""HSS compression where its row ID and its tables change shape: every number
of lanes per column and entries per lane (5 to 8, from 40 to 256 samples),
ranks up to the sample count, blocks that take a cluster of 16 CTAs, and more
tables than a call's staging memory holds.

Bounds: the sampling stops at an estimated error of eps relative to the block,
and the blocks are compared at 50 eps, as in the other tests of the compressed
tier.  A preconditioner whose blocks are good to eps and whose problem has a
condition number of 1e4 leaves a residual of eps x 1e4 after one apply, and
GMRES gains as much per step.
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


@pytest.fixture(scope="module", params=["poisson", "helmholtz"])
def case(request, nd):
    P = poisson_dirichlet(200, seed=3) if request.param == "poisson" else helmholtz_impedance(160, 1, 24.0, seed=3)
    tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, 64)
    info = nd.ndhss_tree_export(tree)["node_info"]
    M = nd.DeviceCSR(P.A)
    return P, tree, info, M, {}


def _factor(nd, case, prec, **kw):
    _, tree, _, M, _ = case
    return nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(prec=prec, **kw))


@pytest.mark.parametrize("prec,eps", [(0, 1e-6), (0, 1e-11), (1, 1e-6)])
@pytest.mark.parametrize("p", [40, 48, 56, 64, 65, 80, 96, 112, 128, 129, 160, 192, 224, 256])
def test_every_lane_and_entry_count(nd, case, prec, eps, p):
    P, _, info, M, dense = case
    level = 2
    if prec not in dense:
        dense[prec] = _factor(nd, case, prec, hss_levels=-1)
    f = _factor(nd, case, prec, hss_levels=int(info[:, 0].max()) - level, eps_hss=eps, k0=p - 16, r=16, seed=5)
    for s in np.flatnonzero(info[:, 0] == level):
        mi, mb = int(info[s, 5]), int(info[s, 7])
        assert mb > 128
        assert _rel(nd.ndhss_factor_get_block(f, int(s), 3, mi, mb),
                    nd.ndhss_factor_get_block(dense[prec], int(s), 3, mi, mb)) <= 50 * eps
    b = torch.from_numpy(np.random.default_rng(p).standard_normal(P.n).astype(P.A.dtype)).cuda()
    st = nd.ndhss_gmres(f, M.rowptr, M.col, M.vals, b, torch.empty_like(b), tol=1e-9)
    assert st["iters"] <= 8


def test_blocks_that_take_a_cluster_of_sixteen(nd):
    """An interior block of 422 rows with 256 samples in complex128: 105 KB per
    CTA with 16 of them, more than a CTA holds with eight."""
    P = helmholtz_impedance(420, 1, 60.0, seed=1)
    tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, 64)
    info = nd.ndhss_tree_export(tree)["node_info"]
    assert 390 <= info[info[:, 0] == 1, 5].max() <= 780
    M = nd.DeviceCSR(P.A)
    f = nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(
        prec=0, hss_levels=int(info[:, 0].max()) - 2, eps_hss=1e-9, k0=240, r=16))
    b = torch.from_numpy(np.random.default_rng(0).standard_normal(P.n).astype(np.complex128)).cuda()
    y = nd.ndhss_apply(f, b, torch.empty_like(b))
    r = P.A @ y.cpu().numpy() - b.cpu().numpy()
    assert np.linalg.norm(r) <= 1e-5 * np.linalg.norm(b.cpu().numpy())
    assert nd.ndhss_gmres(f, M.rowptr, M.col, M.vals, b, y, tol=1e-10)["iters"] <= 4


def test_more_tables_than_the_staging_memory_holds(nd):
    """4096 fronts of some 40 boundary unknowns in HSS leaves of eight: over
    7 MB of node records in one round, page-locked staging has 4."""
    P = poisson_dirichlet(512, seed=1)
    tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, 64)
    M = nd.DeviceCSR(P.A)
    f = nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(
        prec=0, hss_levels=1, eps_hss=1e-8, beta=8, k0=8, r=8))
    b = torch.from_numpy(np.random.default_rng(0).standard_normal(P.n)).cuda()
    y = nd.ndhss_apply(f, b, torch.empty_like(b))
    r = P.A @ y.cpu().numpy() - b.cpu().numpy()
    assert np.linalg.norm(r) <= 1e-2 * np.linalg.norm(b.cpu().numpy())
    assert nd.ndhss_gmres(f, M.rowptr, M.col, M.vals, b, y, tol=1e-10)["iters"] <= 10
