"""The applies at the sizes where their tilings can go wrong: fronts smaller
than one tile, ragged rows, right-hand sides off the column groups.

Tolerance: both sides of each comparison read the same FP64 factor and sum
the same products in another order, so they differ by at most the summation
length (< 1000 terms here) x 2^-53 x the growth through the levels: 1e-11.
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


def _rand(shape, cplx, seed):
    rng = np.random.default_rng(seed)
    v = rng.standard_normal(shape)
    return v + 1j * rng.standard_normal(shape) if cplx else v


@pytest.mark.parametrize("nrhs", [1, 4, 5, 31, 32])
@pytest.mark.parametrize("kind,N,leaf", [("poisson", 4, 64), ("poisson", 41, 16), ("helmholtz", 3, 64),
                                         ("helmholtz", 29, 24), ("helmholtz", 52, 16)])
def test_fp64_multi_apply_matches_single_applies(nd, kind, N, leaf, nrhs):
    P = poisson_dirichlet(N, seed=1) if kind == "poisson" else helmholtz_impedance(N, 2, 6.0, seed=1)
    tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, leaf)
    M = nd.DeviceCSR(P.A)
    f = nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(prec=0))
    X = torch.from_numpy(_rand((P.n, nrhs), kind != "poisson", nrhs)).cuda()
    Y = nd.ndhss_apply_multi(f, X, torch.full_like(X, float("nan")))
    for c in range(nrhs):
        x = X[:, c].contiguous()
        y = nd.ndhss_apply(f, x, torch.empty_like(x))
        assert _rel(Y[:, c].cpu().numpy(), y.cpu().numpy()) <= 1e-11, c
