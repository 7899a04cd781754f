"""Local energy, residence time and CTMC choice from the rows of free-entry bits, against the walker's
move set element by element (Sec. II.A-B), at the sizes where tiles of walkers, words of entries, blocks
of words and batches of 32 begin and end (needs a GB300).

Reference: vmc_screened_moves walks the lists unit by unit, without the bits; its codes, ratios and
contributions are checked against the oracle elsewhere.  From them this test forms E_L and 1/sum r in
FP64 and the choice in exact integers (floor(r 2^64), Philox from numpy).
Tolerances: t is one rounding of an exact sum, 1e-13; E_L of the FP64 form differs in summation order
alone, 1e-13 of sum |contributions|; the mixed form adds n FP32 terms, each lane at most n / 32 + 6 of
them in sequence: (n / 32 + 6) 2^-24 of sum |contributions|.
"""
import numpy as np
import pytest

from paper_1807_10633_gb300 import systems as S
from tests.gpu_common import make_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vmc():
    from paper_1807_10633_gb300 import vmc as v
    v.lib()
    return v


def _fixed(r):
    """floor(r 2^64) of a non-negative float, exactly."""
    n, d = float(r).as_integer_ratio()
    return (n << 64) // d


# system, eps, walkers: empty double lists and rows of one block; groups of several blocks (eps = 0);
# odd orbital counts; tiles of 64 walkers and their neighbours
CASES = [("hubbard10", 0.0, 1), ("hubbard6x6", 0.0, 65), ("H7", 0.0, 63), ("H20", 0.0, 33), ("H20", 1e-6, 64),
         ("H33", 1e-6, 130), ("H33", 1e-3, 31), ("H40", 0.0, 8)]


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("name,eps,W", CASES)
def test_energy_time_choice(vmc, form, name, eps, W):
    sys_, prm, occ = make_case(name, W, seed=S.MASTER_SEED + W)
    eng = vmc.Engine(sys_, prm, occ, eps=eps, precision=form)
    moves, count, _ = eng.screened_moves()
    e_diag = eng.walkers.e_diag.cpu().numpy()
    e, t = (x.cpu().numpy() for x in eng.local_energy())
    seed = 77
    picked = eng.ctmc_step(seed).cpu().numpy().astype(np.uint64)
    eng.sync()
    for w in range(W):
        code, ratio, contrib = moves[w]
        n, scale = len(code), np.abs(contrib).sum()
        tol = (1e-13 if form == vmc.VMC_FP64 else (n / 32 + 6) * 2.0 ** -24) * scale + 1e-13 * abs(e_diag[w])
        assert abs(e[w] - (e_diag[w] + contrib.sum())) <= tol
        q = [_fixed(abs(r)) for r in ratio]
        Q = sum(q)
        assert abs(t[w] * (Q / 2 ** 64) - 1.0) <= 1e-13
        # numpy's generator raises its counter before a block: 2^256 - 1 gives counter 0
        U = int(np.random.Philox(key=np.array([seed, w], dtype=np.uint64),
                                 counter=np.array([2 ** 64 - 1] * 4, dtype=np.uint64)).random_raw())
        T, k, acc = (U * Q) >> 64, 0, 0
        while acc + q[k] <= T:
            acc += q[k]
            k += 1
        assert picked[w] == code[k], (w, k)


def test_several_launches(vmc):
    """More walkers than one launch's rows hold (1 GiB): the same values as in a small call, bit for bit,
    and a choice made without the rows."""
    W = 2600                                     # 2.4 M doubles at eps = 0: about 0.45 MB per row
    sys_, prm, occ = make_case("H40", W)
    eng = vmc.Engine(sys_, prm, occ, eps=0.0, precision=vmc.VMC_MIXED)
    e, t = (x.cpu().numpy() for x in eng.local_energy())
    pick = eng.ctmc_step(5).cpu().numpy()
    eng.sync()
    for a in (0, W - 40):
        sub = vmc.Engine(sys_, prm, occ[a:a + 40], eps=0.0, precision=vmc.VMC_MIXED)
        es, ts = (x.cpu().numpy() for x in sub.local_energy())
        assert np.array_equal(e[a:a + 40], es) and np.array_equal(t[a:a + 40], ts)
        if a == 0:                               # the Philox key holds the walker's index
            assert np.array_equal(pick[:40], sub.ctmc_step(5).cpu().numpy())
        sub.sync()
