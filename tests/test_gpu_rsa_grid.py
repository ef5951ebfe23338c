"""Random sequential addition with cell lists and rounds of decisions, against the
oracle's one-at-a-time loop: sizes about a batch, one sphere, dilute samples
(cells wider than the spheres), dense ones (long chains of conflicts, more
conflicts than a candidate lists), and a candidate bound that cuts a batch.
Positions are the same draws and the same decisions on both sides; the tolerance
is the existing tests' (1e-15 of the radius, a rounding of the angle functions).
"""
import numpy as np
import pytest

import oracle
from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu
D = 14e-9


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1407_2737_gb300 import build as kbuild
    kbuild.build()


@pytest.mark.parametrize("n,c", [(1, 0.05), (2, 0.1), (33, 0.2), (127, 0.1), (128, 0.1),
                                 (129, 0.3), (1000, 1e-4), (1000, 0.3), (1500, 0.28), (5000, 0.2)])
def test_the_sequential_rule(n, c):
    ly = inputs.lattice_nodes_lysosome(n, D, 0.1, seed=n)
    R = inputs.lysosome_radius(n, D, c) if n > 1 else D
    ctx = kmc.kmc_create([ly], kmc.KMC_FP64_PLAIN, center=np.zeros(3))
    for seed in (1, 2):
        used = kmc.kmc_regenerate_rsa(ctx, 0, R, D, seed, 5)
        o, ou = oracle.rsa(n, R, D, seed, 5, 0)
        assert used == ou
        g = kmc.kmc_read(ctx, kmc.KMC_READ_POSITIONS, 0)
        assert np.max(np.abs(g - o)) <= 1e-15 * R
    # the bound on candidates: enough to the last one, one short
    kmc.kmc_regenerate_rsa(ctx, 0, R, D, 2, 5, max_candidates=ou)
    if n > 1:
        with pytest.raises(kmc.KmcError) as e:
            kmc.kmc_regenerate_rsa(ctx, 0, R, D, 2, 5, max_candidates=ou - 1)
        assert e.value.status == kmc.KMC_ESTATE
    kmc.kmc_destroy(ctx)
