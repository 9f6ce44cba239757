"""The applies where their task shapes change: FP64 levels whose tasks are
narrower and wider than the columns from which 16-row tasks are taken, FP32
multi applies in levels with fewer and with more tiles than SMs whose sums are
up to two chunks and longer.

The queue and one launch per level add the same products in the same order:
bit for bit.  One right-hand side and many read the same factor and sum the same
products in another order: the summation length (< 1000) x the unit roundoff x
the growth through the levels, 1e-11 in FP64, 1e-3 in FP32.
"""
import numpy as np
import pytest

from ndhss_inputs import helmholtz_batch, helmholtz_impedance, poisson_dirichlet
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


def _check(nd, tree, M, n, cplx, prec, monkeypatch):
    f = nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(prec=prec))
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 5)) + (1j * rng.standard_normal((n, 5)) if cplx else 0.0)
    X = torch.from_numpy(X).cuda()
    Y = nd.ndhss_apply_multi(f, X, torch.empty_like(X))
    for c in (0, 4):
        x = X[:, c].contiguous()
        y = nd.ndhss_apply(f, x, torch.empty_like(x))
        assert _rel(Y[:, c].cpu().numpy(), y.cpu().numpy()) <= (1e-11 if prec == 0 else 1e-3)
        monkeypatch.setenv("NDHSS_APPLY_SCHEDULE", "levels")
        assert torch.equal(nd.ndhss_apply(f, x, torch.empty_like(x)), y)
        monkeypatch.delenv("NDHSS_APPLY_SCHEDULE")


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kind,N,leaf", [("poisson", 17, 64), ("poisson", 33, 12), ("poisson", 121, 32), ("poisson", 121, 150),
                                         ("helmholtz", 12, 64), ("helmholtz", 40, 12), ("helmholtz", 70, 150)])
def test_one_problem(nd, kind, N, leaf, prec, monkeypatch):
    P = poisson_dirichlet(N, seed=1) if kind == "poisson" else helmholtz_impedance(N, 1, 0.15 * N, seed=1)
    tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, leaf)
    _check(nd, tree, nd.DeviceCSR(P.A), P.n, kind == "helmholtz", prec, monkeypatch)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("count,lo,hi,leaf", [(200, 6, 10, 24), (150, 6, 10, 64), (40, 12, 20, 24), (20, 20, 30, 64)])
def test_forest(nd, count, lo, hi, leaf, prec, monkeypatch):
    probs = helmholtz_batch(count, seed=1, nmin=lo, nmax=hi, nsrc=1, mb=4)
    tree = nd.ndhss_build_tree_batched([(P.coords, P.A.indptr, P.A.indices) for P in probs], leaf)
    A = nd.batch_csr([P.A for P in probs])[0]
    _check(nd, tree, nd.DeviceCSR(A), A.shape[0], True, prec, monkeypatch)
