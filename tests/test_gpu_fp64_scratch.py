"""The FP64 exchanges' packed operands are work space on top of the factor: a
factorization whose factor fits the device memory must not fail for them.

A fresh process leaves the device the memory that the same factorization keeps
(as its statistics give it), 5 % and 1.2 GB for the other work space of a level
and the context, under the 2.5 GB that the leaf level's operands take in one
piece.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

from ndhss_inputs import helmholtz_impedance, poisson_dirichlet
from closeness import rel as _rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys
import numpy as np, torch
sys.path.insert(0, sys.argv[1])
from ndhss_inputs import helmholtz_impedance
from paper_2105_07791_gb300 import ndhss as nd
P = helmholtz_impedance(512, 1, 60.0, seed=1)
tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, 64)
M = nd.DeviceCSR(P.A)
x = torch.ones(P.n, dtype=torch.complex128, device="cuda")
y = torch.empty_like(x)
keep = int(sys.argv[2])
if keep:
    keep = int(1.05 * keep) + 1200 * 2 ** 20
    hold = torch.empty(torch.cuda.mem_get_info()[0] - keep, dtype=torch.uint8, device="cuda")
f = nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(prec=0))
nd.ndhss_apply(f, x, y)
np.save(sys.argv[3], y.cpu().numpy())
print("bytes", nd.ndhss_factor_stats_get(f)["factor_bytes"])
"""


def test_factor_that_fits_does_not_fail_for_the_packed_operands(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")

    def run(keep, out):
        r = subprocess.run([sys.executable, "-c", CHILD, ROOT, str(keep), str(out)], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        return int(r.stdout.split("bytes")[1])

    need = run(0, tmp_path / "a.npy")
    run(need, tmp_path / "b.npy")
    # smaller batches give the same products; a front without packed operands
    # takes them in float64: rounding (2^-53) times the condition number (2^20)
    assert _rel(np.load(tmp_path / "b.npy"), np.load(tmp_path / "a.npy")) <= 1e-9


@pytest.fixture(scope="module")
def nd():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2105_07791_gb300 import build, ndhss
    build.build()
    ndhss.load()
    return ndhss


# limits that hold every front, most of them, only the smaller ones, and none
@pytest.mark.parametrize("kind,p", [("poisson", 1), ("poisson", 2), ("helmholtz", 1), ("helmholtz", 2)])
@pytest.mark.parametrize("limit", [10 ** 7, 10 ** 6, 2 * 10 ** 5, 0])
def test_smaller_batches_and_fronts_without_packed_operands(nd, kind, p, limit, monkeypatch):
    """Batches change no product (bit for bit, as long as every front fits one);
    fronts without packed operands take float64 ones: rounding times the
    condition number (2^17 at most here)."""
    monkeypatch.setenv("NDHSS_TC_MIN_MI", "24")       # small levels too, real and complex
    N = 96 // p + 5
    P = poisson_dirichlet(N, p=p, seed=2) if kind == "poisson" else helmholtz_impedance(N, p, 12.0, seed=2)
    tree = nd.ndhss_build_tree(P.coords, P.A.indptr, P.A.indices, 64)
    M = nd.DeviceCSR(P.A)
    x = torch.from_numpy(np.random.default_rng(0).standard_normal(P.n).astype(P.A.dtype)).cuda()
    y, flops = [], []
    for env in (None, str(limit)):
        if env:
            monkeypatch.setenv("NDHSS_TC64_SCRATCH", env)
        f = nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(prec=0))
        y.append(nd.ndhss_apply(f, x, torch.empty_like(x)).cpu().numpy())
        flops.append(nd.ndhss_factor_stats_get(f)["tc_flops"])
    assert (flops[1] == flops[0]) if limit == 10 ** 7 else (flops[1] == 0) if limit == 0 else (0 < flops[1] <= flops[0])
    if flops[1] == flops[0]:
        assert np.array_equal(y[1], y[0])
    else:
        assert limit < 10 ** 7 and np.linalg.norm(y[1] - y[0]) <= 2.0 ** -36 * np.linalg.norm(y[0])
