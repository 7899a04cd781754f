"""Orbital block of the walker sums and ln|psi| (Sec. III.A-B) where their kernels change: row widths of 16, 8
and 4 or 8 bytes, ranges of orbitals over several CTAs, chunks of walkers, determinants of 1 to 64
columns on both sides of 16 and 32 (needs a GB300).

References in FP64 with plain PyTorch from the walker tables: sum_w c_w AinvT_w[col(k)] over the occupied k,
and slogdet of the occupied rows plus the Jastrow sum.
Tolerances: a sum of n terms is off by at most n u sum |terms|, with u = 2^-53 (FP64 form) or, within a chunk of
64 walkers, 2^-24 (mixed form; its weights are rounded to FP32 too, one more u); ln|det| by LU with partial pivoting: 1e-11.
"""
import numpy as np
import pytest

from paper_1807_10633_gb300 import systems as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vmc():
    from paper_1807_10633_gb300 import vmc as v
    v.lib()
    return v


def _engine(vmc, M, na, nb, W, form, seed):
    sys_ = S.hubbard(M, 1, n_alpha=na, n_beta=nb)
    rng = np.random.default_rng(seed)
    prm = S.Params(S.random_jastrow(M, rng), rng.normal(size=(M, na)), rng.normal(size=(M, nb)))
    occ = np.concatenate([np.argsort(rng.random((W, M)), axis=1)[:, :n] for n in (na, nb)], axis=1)
    return prm, occ, vmc.Engine(sys_, prm, occ.astype(np.uint16), eps=1e-6, precision=form)


# M, n_alpha, n_beta, W: widths 16 / 8 / 4 (mixed) and 16 / 8 bytes (FP64), n on both sides of 24 (the mixed form's
# rule), several ranges of orbitals (n = 60 of 64), one beta electron, chunks of 1, 64 and 65 walkers
SUMS = [(10, 5, 5, 1), (12, 4, 8, 64), (13, 6, 2, 65), (15, 8, 1, 130), (49, 24, 24, 70), (51, 25, 26, 70), (64, 60, 40, 200)]


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("M,na,nb,W", SUMS)
def test_orbital_sums(vmc, form, M, na, nb, W):
    import torch
    prm, occ, eng = _engine(vmc, M, na, nb, W, form, 5 * M + W)
    rng = np.random.default_rng(W)
    t, e = rng.exponential(size=W), rng.normal(size=W)
    dev = lambda x: torch.as_tensor(x, dtype=torch.float64, device="cuda")  # noqa: E731
    z = lambda: [torch.zeros_like(x) for x in (eng.J, eng.Ca, eng.Cb)]  # noqa: E731
    AO, AEO, one, sums = z(), z(), z(), torch.zeros(2, dtype=torch.float64, device="cuda")
    vmc.vmc_accumulate_gradient(eng.ctx, eng.walkers.struct(), dev(t), dev(e), AO, AEO, sums)
    eng.grad_logpsi(dev(e), *one)
    eng.sync()
    A = eng.walkers.AinvT.cpu().double().numpy().reshape(W, -1)
    cols = eng.walkers.occ_list.cpu().numpy().astype(int).reshape(W, -1)
    u = 2.0 ** -53 * W if form == vmc.VMC_FP64 else 2.0 ** -24 * 66
    for s, (n, o, off) in enumerate(((na, 0, 0), (nb, na, na * na))):
        if n == 0:
            continue
        a = A[:, off:off + n * n].reshape(W, n, n)
        for got, c in ((AO[1 + s], t), (AEO[1 + s], t * e), (one[1 + s], e)):
            ref, mag = np.zeros((M, n)), np.zeros((M, n))
            for w in range(W):
                ref[cols[w, o:o + n]] += c[w] * a[w]
                mag[cols[w, o:o + n]] += np.abs(c[w] * a[w])
            assert (np.abs(got.cpu().numpy() - ref) <= u * mag + 1e-300).all()


@pytest.mark.parametrize("M,na,nb,W", [(4, 1, 1, 3), (9, 8, 1, 1), (20, 16, 15, 5), (24, 17, 9, 6), (40, 32, 31, 9),
                                       (48, 33, 20, 4), (70, 64, 40, 3)])
def test_log_psi(vmc, M, na, nb, W):
    import torch
    prm, occ, eng = _engine(vmc, M, na, nb, W, 0, 11 * M)
    got = eng.log_psi().cpu().numpy()
    eng.sync()
    J = np.triu(prm.J)
    for w in range(W):
        so = np.concatenate([occ[w, :na], M + occ[w, na:]])
        ref = J[np.ix_(np.sort(so), np.sort(so))].sum()
        for C, o in ((prm.C_alpha, occ[w, :na]), (prm.C_beta, occ[w, na:])):
            if len(o):
                ref += float(torch.linalg.slogdet(torch.as_tensor(C[o]))[1])
        assert abs(got[w] - ref) <= 1e-11 * max(1.0, abs(ref))


@pytest.mark.parametrize("n", [5, 20, 40])
def test_log_psi_singular(vmc, n):
    """A column of zeros in the alpha orbitals: -inf for every walker, the status latched once."""
    prm, occ, eng = _engine(vmc, 2 * n, n, n, 3, 0, n)
    eng.Ca[:, n // 2] = 0.0
    got = eng.log_psi().cpu().numpy()
    with pytest.raises(vmc.VmcError) as e:
        eng.sync()
    assert e.value.status == 4 and np.all(np.isneginf(got))
    eng.sync()
