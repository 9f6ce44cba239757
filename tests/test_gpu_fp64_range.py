"""FP64 factors of matrices near the ends of the float64 range: the block
exchanges on the tensor cores form their results from integers and a power of
two, which has to be right wherever the result itself is a float64 number.

Tolerance: scaling by 2^e is exact but for results that become subnormal,
at most 2^-1074 each against values of 2^(e - 12) and more: 2^-57 relative at
e = -1005, times the condition number (below 2^17 here), 2^-40 = 1e-12.
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


@pytest.mark.parametrize("kind", ["poisson", "helmholtz"])
@pytest.mark.parametrize("e", [-1000, -960, 960, 1005])
def test_factor_of_a_matrix_scaled_to_the_ends_of_the_range(nd, kind, e, monkeypatch):
    monkeypatch.setenv("NDHSS_TC_MIN_MI", "24")       # small levels too, real and complex
    P = poisson_dirichlet(40, p=2, seed=2) if kind == "poisson" else helmholtz_impedance(40, 2, 16.0, seed=2)
    tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, 64)
    x = torch.from_numpy(np.random.default_rng(0).standard_normal(P.n).astype(P.A.dtype)).cuda()
    y = []
    for A in (P.A, P.A * 2.0 ** e):
        M = nd.DeviceCSR(A)
        f = nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(prec=0))
        y.append(nd.ndhss_apply(f, x, torch.empty_like(x)).cpu().numpy())
    assert _rel(y[1] * 2.0 ** e, y[0]) <= 1e-12
