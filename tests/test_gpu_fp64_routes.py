"""Which FP64 levels exchange their blocks on the tensor cores: real fronts only
where a level's updates fill the FP64 pipes or its pivots go in several blocks.

Every route eliminates the same fronts in float64: rounding (2^-53) times the
condition number (2^20 at most here).  The sizes lie on both sides of the rule:
few fronts of up to 95 and from 96 interior unknowns, many small fronts, slabs
that fill the GPU and slabs that do not.
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


@pytest.mark.parametrize("kind,N,p,leaf,route", [
    ("poisson", 16, 1, 64, "none"), ("poisson", 48, 1, 64, "none"), ("poisson", 49, 1, 64, "some"),
    ("poisson", 16, 1, 300, "some"), ("poisson", 130, 1, 64, "some"), ("poisson", 130, 1, 16, "some"),
    ("poisson", 260, 1, 64, "some"), ("poisson", 100, 2, 64, "some"), ("poisson", 100, 2, 150, "some"),
    ("helmholtz", 12, 1, 64, "all"), ("helmholtz", 40, 1, 64, "all")])
def test_routes_agree(nd, kind, N, p, leaf, route, monkeypatch):
    P = poisson_dirichlet(N, p=p, seed=2) if kind == "poisson" else helmholtz_impedance(N, p, 0.2 * N * p, seed=2)
    tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, leaf)
    M = nd.DeviceCSR(P.A)
    x = torch.from_numpy(np.random.default_rng(0).standard_normal(P.n).astype(P.A.dtype)).cuda()
    y, flops = {}, {}
    for name, var, val in (("rule", None, None), ("all", "NDHSS_TC_MIN_MI", "24"), ("simt", "NDHSS_FRONT_UPDATE", "simt")):
        if var:
            monkeypatch.setenv(var, val)
        f = nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(prec=0))
        y[name] = nd.ndhss_apply(f, x, torch.empty_like(x)).cpu().numpy()
        flops[name] = nd.ndhss_factor_stats_get(f)["tc_flops"]
        assert np.linalg.norm(P.A @ y[name] - x.cpu().numpy()) <= 1e-9 * np.linalg.norm(x.cpu().numpy())
    assert flops["simt"] == 0 < flops["all"]
    assert (flops["rule"] == 0) if route == "none" else (0 < flops["rule"] <= flops["all"])
    if route == "all":
        assert flops["rule"] == flops["all"]
    for name in ("rule", "all"):
        assert np.linalg.norm(y[name] - y["simt"]) <= 2.0 ** -33 * np.linalg.norm(y["simt"])
