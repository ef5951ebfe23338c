"""kmc_dipolar_field_noalloc at the edges of its groups of 32 (up to 448 NPs) and 64
targets (two per lane) and of the source ranges that it cuts by size: one and two
groups, ragged second targets, odd counts, ranges of a few records, the largest number of blocks.
Tolerance: the FP32 field's, 1e-5 of the rms field, as in the other tests. The
outputs of every NP are checked, the values beyond them stay as they were."""
import numpy as np
import pytest

import oracle
from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 31, 33, 63, 64, 65, 97, 128, 129, 333, 448, 449, 600, 2047, 4097, 8191])
def test_group_edges(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1407_2737_gb300 import build as kbuild
    kbuild.build()
    d = 12e-9
    ly = inputs.lattice_nodes_lysosome(n, d, 0.08, seed=n)
    rng = np.random.default_rng(n)
    pos = inputs.snap_to_float32(ly.pos + inputs.random_axes(n, rng) * rng.uniform(0, 0.2 * d, (n, 1)), d)
    m = inputs.random_axes(n, rng).astype(np.float32).astype(np.float64)
    ref = oracle.dipolar_field(pos, ly.vol, ly.Ms, m)
    dev = [torch.tensor(x, dtype=torch.float64, device="cuda") for x in (pos, m, ly.vol)]
    B = torch.full((n + 64, 3), 7.0, dtype=torch.float64, device="cuda")
    for status in (torch.full((1,), -1, dtype=torch.int32, device="cuda"), None):
        B[:n] = float("nan")
        kmc.kmc_dipolar_field_noalloc(n, dev[0].data_ptr(), dev[1].data_ptr(), dev[2].data_ptr(),
                                      ly.Ms, np.zeros(3), d, B.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream,
                                      status.data_ptr() if status is not None else 0)
        g = B.cpu().numpy()
        err = np.max(np.linalg.norm(g[:n] - ref, axis=1))
        assert err <= 1e-5 * np.sqrt(np.mean(np.sum(ref ** 2, axis=1)))
        assert np.all(g[n:] == 7.0)
        if status is not None:
            assert int(status.item()) == kmc.KMC_OK
