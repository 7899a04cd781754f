"""FP64 form's G by digit products on the tensor cores, at sizes where the recompute takes them (n_sigma above 24; the
smaller cases of test_gpu_refresh.test_fp64_g_digit_products form G by multiply-adds either way): the shortest row, and
three tiles of virtual orbitals with odd n_sigma.  Bound as there: n 2^-42 of the two rows' power-of-two scales.
Needs a GB300."""
import numpy as np
import pytest

from paper_1807_10633_gb300 import systems as S
from test_gpu_refresh import _digit_bound, _g_system, _tables, vmc  # noqa: F401  (vmc: the module's fixture)

pytestmark = pytest.mark.gpu


# virtual orbitals per spin: 25 / 26, 55 / 57, 171 / 173
@pytest.mark.parametrize("name,W", [("ring50_25_24", 40), ("ring84_29_27", 9), ("ring200_29_27", 8)])
def test_digit_products(vmc, name, W):  # noqa: F811
    sys_ = _g_system(name)
    prm = S.make_params(sys_, seed=31)
    occ = S.init_occupations(sys_, prm, W, seed=32)
    eng = vmc.Engine(sys_, prm, occ, eps=1e-6, precision=0)
    try:
        tables, launches = {}, {}
        for tc in (1, 0):
            vmc.vmc_set_option(eng.ctx, vmc.VMC_OPT_G_TENSOR_CORES, tc)
            a = vmc.vmc_launch_count(eng.ctx)
            eng.refresh()
            launches[tc] = vmc.vmc_launch_count(eng.ctx) - a
            tables[tc] = _tables(eng)
        assert launches[1] > launches[0]                 # the digit kernels ran
        for k in ("AinvT", "occ_bits", "virt_list", "pos", "S"):
            assert np.array_equal(tables[1][k], tables[0][k]), k
        bound = _digit_bound(sys_, prm, tables[0], W)
        err = np.abs(tables[1]["G"][:bound.size] - tables[0]["G"][:bound.size])
        assert np.all(err <= bound), float((err / bound).max())
        assert err.max() > 0.0
    finally:
        eng.close()
