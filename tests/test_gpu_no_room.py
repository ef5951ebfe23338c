"""Calls that find no device memory: allocations refused on the host above a size
(KMC_FAULT=alloc_over:<bytes>), nothing faults. A refused call leaves the context
as it was, and what does without the room gives the same bits.
"""
import numpy as np
import pytest

from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1407_2737_gb300 import build as kbuild
    kbuild.build()


def _runs(kind, refuse, monkeypatch):
    ly = inputs.make_lysosome(77, 12e-9, 0.05, seed=2)
    ctx = kmc.kmc_create([ly], kmc.KMC_FP32_MIXED, center=np.zeros(3))
    if kind == "cluster":
        monkeypatch.setenv("KMC_TUNE_CLUSTER", "1")
    else:
        kmc.kmc_targets_per_lane(ctx, 1)
        kmc.kmc_persistent(ctx, 2)
        kmc.kmc_tuning(ctx, 4, 64, 0)
    kmc.kmc_run(ctx, 0.02, 1e5, 40, 1, 0, 3)
    kmc.kmc_sync(ctx)
    if refuse:  # a longer period's table of cosines finds no room
        monkeypatch.setenv("KMC_FAULT", "alloc_over:20000")
        with pytest.raises(kmc.KmcError) as e:
            kmc.kmc_run(ctx, 0.02, 1e5, 4000, 1, 1, 3)
        assert e.value.status == kmc.KMC_ENOMEM
        monkeypatch.delenv("KMC_FAULT")
    kmc.kmc_run(ctx, 0.02, 1e5, 40, 1, 0, 3)
    kmc.kmc_sync(ctx)
    out = [kmc.kmc_read(ctx, w, 0) for w in (kmc.KMC_READ_LOOP_M, kmc.KMC_READ_MOMENTS)]
    kmc.kmc_destroy(ctx)
    return out


@pytest.mark.parametrize("kind", ["cluster", "persistent"])
def test_a_refused_period_leaves_the_shorter_ones_table(kind, monkeypatch):
    want = _runs(kind, False, monkeypatch)
    got = _runs(kind, True, monkeypatch)
    assert all(np.array_equal(w, g) for w, g in zip(want, got))
    assert np.ptp(got[0]) > 0.1  # the field was applied


def _quiet(call):
    """What call returns, and that it leaves no message of an allocation or a shape that
    it did without."""
    with pytest.raises(kmc.KmcError):
        kmc._check(kmc.lib().kmc_sync(None))
    before = kmc.kmc_last_error()
    out = call()
    # (a call may clear the message; the binding asks for the size of phi with no room)
    assert kmc.kmc_last_error() in ("", before, "output needs 3000 elements")
    return out


def test_local_concentration_without_its_grid(monkeypatch):
    ly = inputs.lattice_nodes_lysosome(3000, 14e-9, 0.1, seed=1)
    ly.pos = ly.pos + 1e-9 * np.random.default_rng(1).normal(size=ly.pos.shape)
    out = []
    for limit in (None, 60000):  # the grid takes 137 KB, the arrays before it 48 KB at most
        ctx = kmc.kmc_create([ly], kmc.KMC_FP64_PLAIN, center=np.zeros(3))
        if limit:
            monkeypatch.setenv("KMC_FAULT", "alloc_over:%d" % limit)
        out += [_quiet(lambda: kmc.kmc_local_concentration(ctx, 0, N)) for N in (1, 20)]
        kmc.kmc_destroy(ctx)
    assert np.array_equal(out[0], out[2]) and np.array_equal(out[1], out[3])


def test_mean_mode_in_less_room(monkeypatch):
    ly = inputs.lattice_nodes_lysosome(500, 14e-9, 0.1, Keff=2e4, seed=1)
    run = lambda: kmc.kmc_mean_run([ly], 0.03, 1e5, 200, 2, 0)  # 6.8 MB of wells at once
    want = _quiet(run)
    monkeypatch.setenv("KMC_FAULT", "alloc_over:1000000")
    assert np.array_equal(_quiet(run), want)
    monkeypatch.setenv("KMC_FAULT", "alloc_over:50000")  # not even one step's
    with pytest.raises(kmc.KmcError) as e:
        run()
    assert e.value.status == kmc.KMC_ENOMEM
    assert "cudaMalloc" in str(e.value)


def test_tuning_leaves_the_last_error():
    # (shapes that cannot run are tried and passed over)
    lyss = [inputs.make_lysosome(n, 12e-9, 0.05, seed=n) for n in (333, 222)]
    ctx = kmc.kmc_create(lyss, kmc.KMC_FP32_MIXED, center=np.zeros(3))
    _quiet(lambda: kmc.kmc_run(ctx, 0.02, 1e5, 10, 1, 0, 5))
    kmc.kmc_destroy(ctx)
