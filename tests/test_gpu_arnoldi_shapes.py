"""GMRES where its reductions change shape: fewer rows than a block takes, rows
just past one and past all blocks, more rows than threads, and cycles long
enough for several chunks of basis vectors, ragged last chunks included.

The preconditioner is the exact factor of A + D with D of rank r, so
P^{-1} A = I - (rank r) and GMRES ends after at most r + 1 steps in exact
arithmetic; the factor's rounding (about condition x 2^-53, far above the
tolerance's square) can cost one more.  A wrong or missing partial sum costs
the basis its orthogonality, and with it that bound; the true residual is
recomputed on the host.
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


# n: 9, 121, 144, 19321, 89401 real; 49, 169, 19881, 80089 complex
@pytest.mark.parametrize("kind,N", [("poisson", 4), ("poisson", 12), ("poisson", 13), ("poisson", 140),
                                    ("poisson", 300), ("helmholtz", 3), ("helmholtz", 6), ("helmholtz", 70),
                                    ("helmholtz", 141)])
@pytest.mark.parametrize("rank", [2, 5, 13])
def test_cycle_ends_within_rank_plus_two_steps(nd, kind, N, rank):
    P = poisson_dirichlet(N, seed=1) if kind == "poisson" else helmholtz_impedance(N, 2, 6.0, seed=1)
    A = P.A.tocsr()
    rank = min(rank, P.n // 2)
    rng = np.random.default_rng(rank)
    d = np.zeros(P.n)
    d[rng.choice(P.n, rank, replace=False)] = abs(A.diagonal()).mean() * (0.5 + rng.random(rank))
    B = A.copy()
    B.setdiag(A.diagonal() + d)
    assert np.array_equal(B.indptr, A.indptr) and np.array_equal(B.indices, A.indices)
    b = rng.standard_normal(P.n) + (1j * rng.standard_normal(P.n) if kind != "poisson" else 0.0)
    tree = nd.ndhss_build_tree(P.coords, A.indptr, A.indices, 64)
    MA, MB = nd.DeviceCSR(A), nd.DeviceCSR(B)
    f = nd.ndhss_factor(tree, MB.vtype, MB.rowptr, MB.col, MB.vals, nd.make_factor_opts(prec=0))
    bd = torch.from_numpy(b).cuda()
    x = torch.empty_like(bd)
    st = nd.ndhss_gmres(f, MA.rowptr, MA.col, MA.vals, bd, x, restart=30, maxit=60, tol=1e-10)
    assert st["iters"] <= rank + 2 and st["cycles"] == 1
    xh = x.cpu().numpy()
    assert np.linalg.norm(b - A @ xh) <= 1.001e-10 * np.linalg.norm(b)
