"""kmc_sync, kmc_read and kmc_save wait for everything on the context's stream, also
what a caller put on its own stream after the context's last work."""
import numpy as np
import pytest

from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["sync", "read loop", "read moments", "save"])
def test_waits_for_the_callers_work(call, tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    ly = inputs.make_lysosome(60, 12e-9, 0.05, seed=3)
    ctx = kmc.kmc_create([ly], kmc.KMC_FP32_MIXED, center=np.zeros(3))
    st = torch.cuda.Stream()
    kmc.kmc_set_stream(ctx, st.cuda_stream)
    kmc.kmc_run(ctx, 0.02, 1e5, 10, 1, 0, 5)
    kmc.kmc_sync(ctx)
    x = torch.zeros(1 << 28, device="cuda")
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        for _ in range(200):  # 2 GB each: tens of milliseconds
            y.copy_(x)
    assert not st.query()  # the work is still on its way
    if call == "sync":
        kmc.kmc_sync(ctx)
    elif call == "save":
        kmc.kmc_save(ctx, str(tmp_path / "state"))
    else:
        kmc.kmc_read(ctx, kmc.KMC_READ_LOOP_M if call == "read loop" else kmc.KMC_READ_MOMENTS, 0)
    assert st.query()
    kmc.kmc_set_stream(ctx, 0)
    kmc.kmc_destroy(ctx)
