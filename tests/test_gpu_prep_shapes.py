"""Exact factorizations whose levels take every shape of the panel's second
step: fronts below and above the row count from which a whole CTA packs a pivot
column, levels of so many fronts that a CTA walks over many columns, ragged
last column batches, panels narrower than the pivot block.

One application of an exact factor solves the system up to rounding.  The
interior blocks are inverted explicitly, so the residual is bounded by the
condition number (below 1e5 in the 1-norm here) x the unit roundoff: 6e-3 in
FP32, rounded up to 1e-2; 1e-11 in FP64, with a factor of 100 for the length of
the sums.  A wrong or missing row or column leaves a residual of order 1.
"""
import numpy as np
import pytest

from ndhss_inputs import helmholtz_impedance, poisson_dirichlet

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


@pytest.mark.parametrize("prec,tol", [(0, 1e-9), (1, 1e-2)])
@pytest.mark.parametrize("kind,N,leaf", [("poisson", 23, 8), ("poisson", 190, 16), ("poisson", 330, 8),
                                         ("helmholtz", 17, 8), ("helmholtz", 90, 12), ("helmholtz", 134, 64)])
def test_exact_factor_solves(nd, kind, N, leaf, prec, tol):
    P = poisson_dirichlet(N, seed=2) if kind == "poisson" else helmholtz_impedance(N, 2, 8.0, seed=2)
    A = P.A.tocsr()
    tree = nd.ndhss_build_tree(P.coords, A.indptr, A.indices, leaf)
    M = nd.DeviceCSR(A)
    f = nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(prec=prec))
    rng = np.random.default_rng(N)
    b = rng.standard_normal(P.n) + (1j * rng.standard_normal(P.n) if kind != "poisson" else 0.0)
    bd = torch.from_numpy(b).cuda()
    y = nd.ndhss_apply(f, bd, torch.empty_like(bd)).cpu().numpy()
    assert np.linalg.norm(b - A @ y) <= tol * np.linalg.norm(b)
