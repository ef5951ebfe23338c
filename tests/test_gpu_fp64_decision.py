"""Steps v-vii of an FP64 step where its FP32 shortcuts end: rates beyond FP32's
range in the draw u < P (only kmc_run takes that shortcut, kmc_debug_step returns P
itself, so whole runs are compared with the oracle's), and the arc that holds the
moment.

Tolerances: those of an FP64 run (moments 1e-9 after some dozens of steps, which a
single other decision breaks by far) and of an FP64 step (moments 1e-12).
"""
import math

import numpy as np
import pytest

import oracle
from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1407_2737_gb300 import build as kbuild
    kbuild.build()


@pytest.mark.parametrize("ratio", [1e37, 3e38, 1e39, 1e45, 1e-37, 1e-45])
def test_step_lengths_beyond_fp32(ratio):
    # barriers of 0 to 6 kT: nu0 t_step of 1e39 puts one rate, both or their sum
    # above FP32's largest number, and 1e-45 puts both below its smallest
    S, periods, tau0 = 20, 2, 1e-10
    ly = inputs.make_lysosome(200, 5e-9, 0.02, Ms=1e6, Keff=1.6e5, T=300.0, tau0=tau0, seed=4)
    f = 1.0 / (S * ratio * tau0)
    o = oracle.run(ly, 0, 0.15, f, S, periods, 0, 11, nthreads=4)
    ctx = kmc.kmc_create([ly], kmc.KMC_FP64_PLAIN, center=np.zeros(3))
    kmc.kmc_run(ctx, 0.15, f, S, periods, 0, 11)
    jumps, near = kmc.kmc_read(ctx, kmc.KMC_READ_COUNTERS, 0)[:2]
    m = kmc.kmc_read(ctx, kmc.KMC_READ_MOMENTS, 0)
    loop = kmc.kmc_read(ctx, kmc.KMC_READ_LOOP_M, 0)
    kmc.kmc_destroy(ctx)
    assert near == 0 and jumps == o["counters"]["flips"]
    assert jumps > 500 if ratio > 1 else jumps == 0
    assert np.max(np.abs(m - o["m"])) <= 1e-9
    np.testing.assert_allclose(loop, o["loop_M"], rtol=0, atol=1e-9)


def _plane(t, H, K=2e4, Ms=1e6):
    """An axis at 45 degrees to the field, and the unit vector of its plane with the field
    at the angle t from it."""
    a = np.array([math.sqrt(0.5), 0.0, math.sqrt(0.5)])
    e = np.array([-math.sqrt(0.5), 0.0, math.sqrt(0.5)])
    return a, math.cos(t) * a + math.sin(t) * e


def _same_basins(moments, H, K=2e4):
    """One NP per moment, all with the axis of _plane: the step's basins (the barriers
    are those of the well the moment fell into) and new moments are the oracle's."""
    a, _ = _plane(0.0, H)
    lyss = [inputs.Lysosome(pos=np.zeros((1, 3)), axis=a[None], vol=np.array([math.pi * (14e-9) ** 3
            / 6]), Ms=1e6, Keff=K, T=300.0, tau0=1e-10) for _ in moments]
    ctx = kmc.kmc_create(lyss, kmc.KMC_FP64_PLAIN, center=np.zeros(3))
    g = kmc.kmc_debug_step(ctx, np.full(len(lyss), H), 5e-8, 3, 9, np.array(moments))
    kmc.kmc_destroy(ctx)
    o = [oracle.step(l, q, moments[q][None], H, 5e-8, 3, 9) for q, l in enumerate(lyss)]
    dE = np.concatenate([x["dE"] for x in o])
    assert np.all(g["n_min"] == 2) and len(set((dE[:, 0] > dE[:, 1]).tolist())) == 2
    np.testing.assert_allclose(g["dE"], dE, rtol=1e-11)
    assert np.abs(g["m_out"] - np.concatenate([x["m_out"] for x in o])).max() <= 1e-12


@pytest.mark.parametrize("scale", [0.5, 1e-20, 1e-37, 1e-40, 1e-46, 1e-60])
def test_moments_normal_to_the_plane(scale):
    # maxima at 105.8 and 259.9 degrees
    H = 0.3 * 2 * 2e4 / 1e6
    _same_basins([scale * _plane(math.radians(t), H)[1] + [0.0, math.sqrt(1 - scale ** 2), 0.0]
                  for t in (95, 104, 107, 180, 255, 262, 268, 350)], H)
