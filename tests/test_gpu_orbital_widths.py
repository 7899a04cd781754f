"""Orbital block of the walker sums in the FP64 form for odd n_sigma above 32: single elements, a CTA of up to 32 warps
(needs a GB300).  Reference and tolerance as in test_gpu_orbital_sums: n u sum |terms|, u = 2^-53."""
import numpy as np
import pytest

from test_gpu_orbital_sums import _engine, vmc  # noqa: F401  (vmc: the module's fixture)

pytestmark = pytest.mark.gpu


# M, n_alpha, n_beta, W: 9 and 32 warps of single elements; an odd and an even spin together
@pytest.mark.parametrize("M,na,nb,W", [(40, 35, 33, 70), (130, 127, 97, 20), (72, 66, 65, 33)])
def test_odd_widths(vmc, M, na, nb, W):  # noqa: F811
    import torch
    prm, occ, eng = _engine(vmc, M, na, nb, W, 0, 7 * M + W)
    w = torch.as_tensor(np.random.default_rng(W).normal(size=W), device="cuda")
    _, dCa, dCb = eng.grad_logpsi(w)
    eng.sync()
    A = eng.walkers.AinvT.cpu().numpy().reshape(W, -1)
    cols = eng.walkers.occ_list.cpu().numpy().astype(int).reshape(W, -1)
    c = w.cpu().numpy()
    for got, n, o, off in ((dCa, na, 0, 0), (dCb, nb, na, na * na)):
        a = A[:, off:off + n * n].reshape(W, n, n)
        ref, mag = np.zeros((M, n)), np.zeros((M, n))
        for k in range(W):
            ref[cols[k, o:o + n]] += c[k] * a[k]
            mag[cols[k, o:o + n]] += np.abs(c[k] * a[k])
        assert (np.abs(got.cpu().numpy() - ref) <= 2.0 ** -53 * W * mag + 1e-300).all()
    eng.close()
