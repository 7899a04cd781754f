"""More walkers than one launch's free-entry rows hold (1 GiB): several launches, and in a batch several rounds over
all systems, give the same values as one system's launches alone, bit for bit, and the choice is made without the rows
(Sec. II.A-B; needs a GB300)."""
import numpy as np
import pytest
import torch

from tests.gpu_common import make_case

pytestmark = pytest.mark.gpu


def test_rounds():
    from paper_1807_10633_gb300 import vmc
    # H40 at eps = 0: about 0.45 MB a row; the ring's 40 walkers are all in the first rounds
    cases = [("H40", 0.0, 2600), ("hubbard10", 0.0, 40)]
    single, batched = [], []
    for name, eps, W in cases:
        sys_, prm, occ = make_case(name, W)
        for out in (single, batched):
            out.append(vmc.Engine(sys_, prm, occ, eps=eps, precision=vmc.VMC_MIXED))
    b = vmc.Batch(batched)
    for step in range(2):
        a = vmc.vmc_launch_count(b.ctx)
        b.local_energy()
        rounds = (vmc.vmc_launch_count(b.ctx) - a) // 2
        assert rounds >= 2
        for k, e in enumerate(single):
            a = vmc.vmc_launch_count(e.ctx)
            e.local_energy()
            n = vmc.vmc_launch_count(e.ctx) - a
            assert n >= 4 if k == 0 else n == 1
            e.ctmc_step(17)
        b.ctmc_step(17)
        torch.cuda.synchronize()
        for e1, e2 in zip(single, batched):
            assert torch.equal(e1.e_loc, e2.e_loc) and torch.equal(e1.t_res, e2.t_res), step
            assert torch.equal(e1.moves, e2.moves), step
    for e1, e2 in zip(single, batched):
        assert np.array_equal(e1.occupations(), e2.occupations())
        e1.sync()
        e2.sync()
    for e in single + batched:
        e.close()
