"""Recompute of the walker tables at the edges of its launches: both sides of the FP64 form's line between
G by multiply-adds and G by digit products (n_sigma = 24), and walker counts and odd orbital counts that do
not fill the walker pairs, walker groups and orbital pairs of the Fock and Jastrow sums."""
import numpy as np
import pytest

from paper_1807_10633_gb300 import systems as S
from test_gpu_refresh import _expected, _tables, vmc  # noqa: F401  (vmc: the module's fixture)

pytestmark = pytest.mark.gpu

CASES = [(7, 3, 2, 1), (9, 5, 4, 3), (27, 23, 12, 2), (30, 24, 23, 5), (33, 25, 24, 18), (49, 32, 33, 17)]


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("M,na,nb,W", CASES)
def test_recompute_edges(vmc, M, na, nb, W, precision):  # noqa: F811
    """G and C_occ^-1 against FP64 inverses (the bounds of the register refresh's test), and every walker's
    tables, the Fock and Jastrow sums among them, bit-identical to those it has alone."""
    sys_ = S.hubbard(M, n_alpha=na, n_beta=nb)
    prm = S.make_params(sys_, seed=M + 1)
    occ = S.init_occupations(sys_, prm, W, seed=M + 2)
    eng = vmc.Engine(sys_, prm, occ, eps=0.0, precision=precision)
    try:
        got = dict(_tables(eng), F=eng.walkers.F.cpu().numpy().copy())
    finally:
        eng.close()
    G, A = _expected(sys_, prm, occ)
    tol = 1e-10 if precision == 0 else 2e-4
    assert np.abs(got["G"][:G.size] - G).max() / max(1.0, np.abs(G).max()) < tol
    assert np.abs(got["AinvT"][:A.size] - A).max() / max(1.0, np.abs(A).max()) < tol
    for w in sorted({0, W // 2, W - 1}):
        one = vmc.Engine(sys_, prm, occ[w:w + 1], eps=0.0, precision=precision)
        try:
            alone = dict(_tables(one), F=one.walkers.F.cpu().numpy().copy())
        finally:
            one.close()
        for k in ("G", "AinvT", "S", "F"):
            n = alone[k].size
            assert np.array_equal(got[k].ravel()[w * n:(w + 1) * n], alone[k].ravel()), (k, w)
