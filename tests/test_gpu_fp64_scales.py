"""One block exchange of an FP64 front against the same products in extended
precision on the host, on evenly and on unevenly scaled unknowns.

Nodes with at most 64 interior unknowns have one exchange of all pivots with
their boundary columns.  From the factor's own blocks (every bit of A_ii^{-1}
and L, the children's S) the host forms S = A_bb + L A_ib and R = -A_ii^{-1}
A_ib again.

Bounds, K real products per entry (two per complex one).  Even scales: two
roundings to float64, and for what eight 8-bit digits leave out 7 terms of
2^14 x 2^-76 of the product of the two rows' largest entries (as powers of two:
up to 4 times it) per product, 2^-59 K with the later digits; a lost digit sum
would leave 2^-51.  Scales D A D and D A E with entries of D and E over 2^s:
the bound of a float64 product of that length, K 2^-53, against the largest
sum of magnitudes among the entries divided by their scales.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from ndhss_inputs import helmholtz_impedance, poisson_dirichlet
from oracle.frontal import assemble_front
from oracle.tree import build_tree

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


def _problem(kind):
    if kind == "poisson":
        return poisson_dirichlet(61, seed=2), 64
    if kind == "poisson_p2":
        return poisson_dirichlet(40, p=2, seed=2), 40
    return helmholtz_impedance(48, 1, 9.0, seed=2), 64


def _wide(a):
    return a.astype(np.clongdouble if np.iscomplexobj(a) else np.longdouble)


def _cabs(a):
    return np.maximum(np.abs(a.real), np.abs(a.imag)) if np.iscomplexobj(a) else np.abs(a)


@pytest.mark.parametrize("kind", ["poisson", "poisson_p2", "helmholtz"])
@pytest.mark.parametrize("s,both", [(0, True), (24, True), (48, True), (80, True), (40, False)])
def test_exchange_matches_extended_precision(nd, kind, s, both, monkeypatch):
    monkeypatch.setenv("NDHSS_TC_MIN_MI", "24")       # small levels too, real and complex
    P, leaf = _problem(kind)
    rng = np.random.default_rng(s)
    Dr = np.exp2(rng.uniform(0, s, P.n))
    Dc = Dr if both else np.exp2(rng.uniform(0, s, P.n))
    A = sp.csr_matrix(P.A)
    if s:
        A = sp.csr_matrix((A.data * np.repeat(Dr, np.diff(A.indptr)) * Dc[A.indices], A.indices, A.indptr), A.shape)
    T = build_tree(P.coords, A.indptr, A.indices, leaf)
    M = nd.DeviceCSR(A)
    tree = nd.ndhss_build_tree(P.coords, A.indptr, A.indices, leaf)
    f = nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(prec=0))
    mimax = {l: max(T.node_info[q, 5] for q in np.flatnonzero(T.node_info[:, 0] == l)) for l in range(T.depth + 1)}
    block = lambda q, w: nd.ndhss_factor_get_block(f, int(q), w, int(T.node_info[q, 5]), int(T.node_info[q, 7]))
    seen = 0
    for q in range(T.nnodes):
        mi, mb = int(T.node_info[q, 5]), int(T.node_info[q, 7])
        if not (16 <= mi <= 64 and mb and mimax[T.node_info[q, 0]] >= 24):
            continue
        F = assemble_front(T, q, A, {c: block(c, 3) for c in T.children(q)})
        Ai, R, L, S = (block(q, w) for w in range(4))
        Aib, Abb = F[:mi, mi:], F[mi:, mi:]
        K = mi * (2 if np.iscomplexobj(F) else 1)
        rI, rB, cB = Dc[T.perm][T.I(q)], Dr[T.perm][T.B(q)], Dc[T.perm][T.B(q)]
        for left, out, add, ro in ((L, S, Abb, rB), (-Ai, R, 0.0, 1.0 / rI)):
            prod = _wide(left) @ _wide(Aib)
            d = np.abs(out - (add + prod))
            if s == 0:
                rows, cols = _cabs(left).max(1), _cabs(Aib).max(0)
                tol = 2.0 ** -53 * 2 * (np.abs(prod) + np.abs(add + prod)) + K * 2.0 ** -59 * 4 * np.outer(rows, cols)
            else:
                sc = np.outer(ro, cB)
                big = np.max((np.abs(left) @ np.abs(Aib) + np.abs(add)) / sc)
                tol = K * 2.0 ** -53 * big * sc
            assert np.all(d <= tol), (q, mi, mb, float(np.max(d / np.maximum(tol, 1e-300))))
        seen += 1
    assert seen >= 8


@pytest.mark.parametrize("kind", ["poisson", "helmholtz"])
@pytest.mark.parametrize("bad,diag", [(np.nan, True), (np.nan, False), (np.inf, True), (np.inf, False)])
def test_entries_that_are_not_finite_end_as_in_the_cuda_core_sweep(nd, kind, bad, diag, monkeypatch):
    """One such entry: the same status from both sweeps, or results that are not
    finite in both, or (an infinite pivot has the inverse zero) finite ones that
    agree to rounding (2^-53) times the condition number (2^17 here)."""
    monkeypatch.setenv("NDHSS_TC_MIN_MI", "24")
    P, leaf = _problem(kind)
    A = sp.csr_matrix(P.A).copy()
    row = P.n // 2
    at = np.flatnonzero((A.indices[A.indptr[row]:A.indptr[row + 1]] == row) == diag)[0]
    A.data[A.indptr[row] + at] = bad
    tree = nd.ndhss_build_tree(P.coords, A.indptr, A.indices, leaf)
    M = nd.DeviceCSR(A)
    x = torch.ones(P.n, dtype=torch.complex128 if kind == "helmholtz" else torch.float64, device="cuda")
    out = []
    for update in (None, "simt"):
        if update:
            monkeypatch.setenv("NDHSS_FRONT_UPDATE", update)
        try:
            f = nd.ndhss_factor(tree, M.vtype, M.rowptr, M.col, M.vals, nd.make_factor_opts(prec=0))
            y = nd.ndhss_apply(f, x, torch.empty_like(x)).cpu().numpy()
            out.append(y if np.isfinite(y).all() else "not finite")
        except nd.NdhssError as err:
            out.append(err.code)
    if isinstance(out[1], np.ndarray):
        assert isinstance(out[0], np.ndarray), out[0]
        assert np.linalg.norm(out[0] - out[1]) <= 2.0 ** -36 * np.linalg.norm(out[1])
    else:
        assert out[0] == out[1]
