"""ln|psi| (Sec. III.A) at the ends of its range: pivots whose reciprocals are no normal numbers, and the largest
determinant that an SM's shared memory holds (needs a GB300).

Reference: slogdet in FP64 of the occupied rows, the scaled column taken back to order one exactly (powers of two;
the subnormal elements are rounded before, in both).  Tolerance of LU with partial pivoting as in
test_gpu_orbital_sums: 1e-11."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _log_psi(M, na, nb, W, Ca, Cb, J, occ):
    """vmc_log_psi alone: it reads occ_list and the parameters, and no table."""
    from paper_1807_10633_gb300 import vmc
    ctx = vmc.vmc_create(0, torch.cuda.current_stream())
    wk = vmc.Walkers.allocate(W, M, na, nb, None)
    wk.occ_list.copy_(torch.from_numpy(occ.astype(np.int16).reshape(-1)))
    dev = [torch.as_tensor(x, dtype=torch.float64, device="cuda").contiguous() for x in (J, Ca, Cb)]
    out = torch.zeros(W, dtype=torch.float64, device="cuda")
    vmc.vmc_log_psi(ctx, wk.struct(), vmc.params_struct(*dev), out)
    vmc.vmc_sync(ctx)
    vmc.vmc_destroy(ctx)
    return out.cpu().numpy()


# n on both sides of 16 and 32 (a warp's rows in registers, a CTA's in shared memory); pivots of a scaled first
# column near 2^-1030 (subnormal) and 2^1022; n = 169, where rows and lists fill the shared memory
@pytest.mark.parametrize("M,na,nb,W,ex", [(12, 5, 4, 5, -1030), (40, 20, 17, 3, -1030), (80, 40, 33, 3, -1030),
                                          (12, 5, 4, 5, 1021), (80, 40, 20, 3, 1021), (40, 20, 32, 2, 0),
                                          (172, 169, 33, 2, 0)])
def test_range(M, na, nb, W, ex):
    rng = np.random.default_rng(M + na)
    Ca, Cb = rng.uniform(0.6, 1.9, (M, na)) * rng.choice((-1.0, 1.0), (M, na)), rng.normal(size=(M, nb))
    J = 0.01 * rng.normal(size=(2 * M, 2 * M))
    Ca[:, 0] = np.ldexp(Ca[:, 0], ex)
    occ = np.concatenate([np.argsort(rng.random((W, M)), axis=1)[:, :n] for n in (na, nb)], axis=1)
    got = _log_psi(M, na, nb, W, Ca, Cb, J, occ)
    Ca[:, 0] = np.ldexp(Ca[:, 0], -ex)
    for w in range(W):
        so = np.sort(np.concatenate([occ[w, :na], M + occ[w, na:]]))
        ref = np.triu(J)[np.ix_(so, so)].sum() + ex * np.log(2.0)
        ref += np.linalg.slogdet(Ca[occ[w, :na]])[1] + np.linalg.slogdet(Cb[occ[w, na:]])[1]
        assert abs(got[w] - ref) <= 1e-11 * max(1.0, abs(ref)), (got[w], ref)
