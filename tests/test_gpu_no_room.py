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
