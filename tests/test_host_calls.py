"""Host side of the library's calls on a CUDA runtime without a device (CPU only): what is refused before a launch,
what the context's rate store holds, and when it is allocated."""
import pytest

from paper_1807_10633_gb300 import systems as S
from paper_1807_10633_gb300 import vmc
from tests import fake_cudart


@pytest.fixture(scope="module")
def runtime(tmp_path_factory):
    path = fake_cudart.build(tmp_path_factory.mktemp("fake"))
    keep = vmc.LIB, vmc._lib
    vmc.LIB, vmc._lib = path, None
    yield fake_cudart.Runtime(vmc.lib())
    vmc.LIB, vmc._lib = keep


@pytest.fixture
def ctx(runtime):
    runtime.limit()
    c = vmc.vmc_create(0, 0)
    runtime.launches()
    yield c
    runtime.limit()
    vmc.vmc_destroy(c)


def _refused(call, *args, **kw):
    with pytest.raises(vmc.VmcError) as e:
        call(*args, **kw)
    assert e.value.status == 1, e.value                  # VMC_ERR_ARG
    return str(e.value)


@pytest.mark.parametrize("precision,shift", [(0, 8), (1, 4), (1, 8)])
def test_moves_need_aligned_fock_sums(runtime, ctx, precision, shift):
    """The update reads F as 16-byte vectors: a misaligned F is refused before any kernel, alone and in a batch; the
    other arrays may start at any of their elements."""
    sys_ = S.named_system("H6")
    bad = fake_cudart.System(ctx, sys_, 5, 1e-6, precision, {"F": shift})
    bad.energy()
    runtime.launches()
    assert "16-byte" in _refused(bad.step)
    items = fake_cudart.batch([bad])
    vmc.vmc_local_energy_batch(ctx, items)
    runtime.launches()
    assert "16-byte" in _refused(vmc.vmc_ctmc_step_batch, ctx, items, 3)
    assert runtime.launches() == []
    real = 8 if precision == 0 else 4
    ok = fake_cudart.System(ctx, sys_, 5, 1e-6, precision, {"S": real, "G": real, "AinvT": real, "pos": 2, "occ_list": 2})
    ok.energy()
    ok.step()
    assert any("k_ctmc_apply" in x for x in runtime.launches())
    for s in (bad, ok):
        s.close()


def test_moves_refuse_rates_of_other_lists(runtime, ctx):
    """Rates and rows are laid out by the lists of the local energy: other lists of the same size, or more walkers than
    it had, are refused; a second build of the same lists is the same lists."""
    s = fake_cudart.System(ctx, S.named_system("H12"), 700, 1e-4)
    same = fake_cudart.System(ctx, S.named_system("H12"), 1, 1e-4)
    other = fake_cudart.System(ctx, S.named_system("H12"), 1, 1e-6)
    s.energy()
    runtime.launches()
    assert "lists" in _refused(s.step, other.lists)
    s.walkers.W = 701
    assert "walkers" in _refused(s.step)
    assert runtime.launches() == []
    s.walkers.W = 700
    s.step(same.lists)
    assert any("k_ctmc_select" in x for x in runtime.launches())
    for x in (s, same, other):
        x.close()


def test_moves_use_the_threshold_of_their_rates(runtime, ctx):
    """Another context may run the same lists at another eps_run in between: the choice is made at the rates' own."""
    s = fake_cudart.System(ctx, S.named_system("H12"), 700, 1e-6)
    c2 = vmc.vmc_create(0, 0)
    s.energy(1e-5)
    s.energy(1e-3, c2)
    s.step()
    before = runtime.counts()["uploads"]
    s.energy(1e-5)                                       # the lists stand at 1e-5 again: nothing to upload
    assert runtime.counts()["uploads"] == before
    vmc.vmc_destroy(c2)
    s.close()


def _two(ctx, W=700):
    return [fake_cudart.System(ctx, S.named_system("H12"), W, 1e-6), fake_cudart.System(ctx, S.named_system("H6"), 40, 1e-6)]


@pytest.mark.parametrize("between", ["energy", "refresh", "init"])
def test_batched_moves_need_their_own_energies(runtime, ctx, between):
    """A local energy or a rebuild of the tables on the context takes the batch's rates with it, as it does those of a
    single system."""
    two = _two(ctx)
    items = fake_cudart.batch(two)
    vmc.vmc_local_energy_batch(ctx, items)
    if between == "energy":
        two[1].energy()
    else:
        call = vmc.vmc_walkers_refresh if between == "refresh" else vmc.vmc_walkers_init
        call(ctx, two[0].lists, two[0].params, two[0].walkers)
    runtime.launches()
    assert "must precede" in _refused(vmc.vmc_ctmc_step_batch, ctx, items, 3)
    assert runtime.launches() == []
    vmc.vmc_local_energy_batch(ctx, items)
    vmc.vmc_ctmc_step_batch(ctx, items, 3)
    for s in two:
        s.close()


def _store_bytes(runtime, call):
    a = runtime.counts()["live"]
    call()
    return runtime.counts()["live"] - a


@pytest.mark.parametrize("later", [0, None])
def test_batched_moves_keep_the_rate_store(runtime, ctx, later):
    """Too little memory for every walker's rows: the energies run in rounds, and the moves read the store as it is,
    whether or not there is more memory by then."""
    two = _two(ctx)
    items = fake_cudart.batch(two)
    full = _store_bytes(runtime, lambda: vmc.vmc_local_energy_batch(ctx, items))
    c2 = vmc.vmc_create(0, 0)
    runtime.launches()
    runtime.limit(full * 3 // 4)
    vmc.vmc_local_energy_batch(c2, items)
    assert sum("k_local_energy" in x for x in runtime.launches()) == 2
    runtime.limit(later)
    before = runtime.counts()
    vmc.vmc_ctmc_step_batch(c2, items, 3)
    assert runtime.counts() == before
    assert sum("k_ctmc" in x for x in runtime.launches()) == 2
    vmc.vmc_destroy(c2)
    for s in two:
        s.close()


def test_moves_refuse_other_batch_items(runtime, ctx):
    two = _two(ctx)
    other = fake_cudart.System(ctx, S.named_system("H6"), 1, 1e-2)
    vmc.vmc_local_energy_batch(ctx, fake_cudart.batch(two))
    two[0].walkers.W += 1
    assert "must precede" in _refused(vmc.vmc_ctmc_step_batch, ctx, fake_cudart.batch(two), 3)
    two[0].walkers.W -= 1
    keep, two[1].lists = two[1].lists, other.lists
    assert "must precede" in _refused(vmc.vmc_ctmc_step_batch, ctx, fake_cudart.batch(two), 3)
    two[1].lists = keep
    vmc.vmc_ctmc_step_batch(ctx, fake_cudart.batch(two), 3)
    for s in (*two, other):
        s.close()


@pytest.mark.parametrize("batched", [False, True])
def test_short_memory_is_remembered(runtime, ctx, batched):
    """Rows that did not fit are not asked for again: later calls allocate, free and wait for nothing, so that they can
    be captured; rates that are needed are still asked for when there may be memory again."""
    two = _two(ctx)
    items = fake_cudart.batch(two)

    def energy(c):
        vmc.vmc_local_energy_batch(c, items) if batched else two[0].energy(ctx=c)
    full = _store_bytes(runtime, lambda: energy(ctx))
    big = fake_cudart.System(ctx, S.named_system("H6"), 100000, 1e-6)
    c2 = vmc.vmc_create(0, 0)
    runtime.limit(full * 3 // 4)
    energy(c2)
    before = runtime.counts()
    runtime.limit(0, capturing=True)
    energy(c2)
    assert runtime.counts() == before
    runtime.limit(0)
    with pytest.raises(vmc.VmcError) as e:
        big.energy(ctx=c2)
    assert e.value.status == 3                           # VMC_ERR_OOM
    runtime.limit()
    big.energy(ctx=c2)
    for s in (*two, big):
        s.close()
    vmc.vmc_destroy(c2)


def test_a_failed_allocation_is_reported_once(runtime, ctx):
    """The runtime keeps an allocation's error until it is asked for: the call after it must not report it again."""
    s = fake_cudart.System(ctx, S.named_system("H6"), 64, 1e-6)
    out = [s._array(8 * k) for k in (144, 18, 18)]
    runtime.limit(0)
    with pytest.raises(vmc.VmcError) as e:
        vmc.vmc_grad_logpsi(ctx, s.walkers, s.t, *out)
    assert e.value.status == 3                           # VMC_ERR_OOM
    vmc.vmc_log_psi(ctx, s.walkers, s.params, s.e)
    runtime.limit()
    s.close()



def test_batch_table_that_could_not_grow(runtime, ctx):
    """A failed allocation of the batch's table leaves none: the next call uploads one or reports the same, it does not
    launch on the table that was freed."""
    two = _two(ctx)
    big, small = fake_cudart.batch(two), fake_cudart.batch(two[:1])
    vmc.vmc_local_energy_batch(ctx, big)
    c2 = vmc.vmc_create(0, 0)
    two[0].energy(ctx=c2)
    two[0].walkers.W = 1                                 # (the store is large enough)
    vmc.vmc_local_energy_batch(c2, small)
    runtime.launches()
    for items in (big, small):
        runtime.limit(0)
        with pytest.raises(vmc.VmcError) as e:
            vmc.vmc_local_energy_batch(c2, items)
        assert e.value.status == 3                       # VMC_ERR_OOM
    assert runtime.launches() == []
    runtime.limit()
    vmc.vmc_local_energy_batch(c2, small)
    assert len(runtime.launches()) == 2
    vmc.vmc_destroy(c2)
    for s in two:
        s.close()
