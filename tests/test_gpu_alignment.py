"""Walker arrays that start at any of their elements (a caller may pack them into one buffer): the tables, gradient
sums and moves equal those of arrays on allocation boundaries, bit for bit (needs a GB300).  G and AinvT stay on their
boundaries: the update's kernel for other addresses rounds its sums in another order."""
import pytest
import torch

from tests.gpu_common import make_case

pytestmark = pytest.mark.gpu


def _off(t, k):
    """The same tensor k elements into a buffer of its own."""
    out = torch.zeros(t.numel() + k, dtype=t.dtype, device=t.device)[k:]
    out.copy_(t)
    return out


# H24: pos is read as 16-byte vectors (M a multiple of 8); H7: an odd number of orbital pairs; both forms
@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("name,W,k", [("H7", 9, 1), ("H24", 70, 1), ("H64", 5, 3)])
def test_unaligned_walker_arrays(form, name, W, k):
    from paper_1807_10633_gb300 import vmc
    got = []
    for shift in (0, k):
        sys_, prm, occ = make_case(name, W)
        eng = vmc.Engine(sys_, prm, occ, eps=1e-6, precision=form)
        if shift:
            for f in ("S", "pos", "occ_list", "virt_list", "occ_bits"):
                setattr(eng.walkers, f, _off(getattr(eng.walkers, f), shift))
            assert eng.walkers.S.data_ptr() % 16 and eng.walkers.pos.data_ptr() % 16
        eng.init()
        out = [eng.walkers.S.clone()]
        for seed in (1, 2):
            e, t = eng.local_energy()
            out += [e.clone(), t.clone(), *eng.grad_logpsi(t)]
            out.append(eng.ctmc_step(seed).clone())
        eng.refresh()
        out += [getattr(eng.walkers, f).clone() for f in ("S", "G", "AinvT", "pos")]
        eng.sync()
        got.append(out)
        eng.close()
    for a, b in zip(*got):
        assert torch.equal(a, b)
