"""kmc_local_concentration's grid search against the oracle where it can go
wrong: the sizes at which it takes over from the all-pairs kernel, ranks from 1
to the largest, equal distances (lattices: more pairs in the FP32 error band
than a warp has lanes), flat and clustered samples, NPs far from the frame's
origin, and coinciding NPs.

The oracle takes the frame coordinates that the device holds (positions over the
diameter of the mean volume), so both form r_N^2 from the same FP64 numbers in the
same order and differ by the rounding of a root, a cube and a quotient: 1e-13
relative leaves two orders of magnitude.
"""
import dataclasses
import math

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


def _sample(kind, n):
    rng = np.random.default_rng(n)
    ly = inputs.lattice_nodes_lysosome(n, D, 0.1, seed=n)
    a = inputs.lattice_spacing(D, 0.1)
    if kind == "random":
        pos = ly.pos + inputs.random_axes(n, rng) * rng.uniform(0, 0.3 * D, (n, 1))
    elif kind == "lattice":
        pos = ly.pos
    elif kind == "plane":
        m = int(np.ceil(np.sqrt(n)))
        pos = a * np.stack([np.arange(n) % m, np.arange(n) // m, np.zeros(n)], 1)
    elif kind == "line":
        pos = a * np.stack([np.arange(n), np.zeros(n), np.zeros(n)], 1) * 0.3
    elif kind == "two balls":
        pos = np.where(np.arange(n)[:, None] < n // 2, ly.pos, ly.pos + 60 * a)
    elif kind == "outlier":
        pos = ly.pos.copy()
        pos[0] += 500 * a
    elif kind == "far":
        pos = ly.pos + 700 * a
    else:  # pairs at one point
        pos = ly.pos.copy()
        pos[1::2] = pos[0:2 * (n // 2):2]
    vol = ly.vol * np.linspace(0.8, 1.2, n)
    return dataclasses.replace(ly, pos=pos, vol=vol)


def _oracle(ly, N):
    total = 0.0
    for v in ly.vol.tolist():
        total += v
    length = math.cbrt(6.0 * (total / ly.n) / math.pi)
    with np.errstate(divide="ignore"):
        return oracle.local_concentration(ly.pos / length, ly.vol / length ** 3, N)


@pytest.mark.parametrize("kind,n,N", [
    ("random", 1023, 20), ("random", 1024, 20), ("random", 1025, 1), ("random", 3001, 64),
    ("lattice", 2000, 20), ("lattice", 2000, 64), ("lattice", 5000, 57), ("plane", 1500, 20),
    ("line", 1200, 7), ("two balls", 1100, 64), ("outlier", 1400, 20), ("far", 1300, 20),
    ("pairs", 1200, 1), ("pairs", 1200, 20)])
@pytest.mark.parametrize("prec", [kmc.KMC_FP64_PLAIN, kmc.KMC_FP32_MIXED])
def test_against_the_oracle(kind, n, N, prec):
    ly = _sample(kind, n)
    ctx = kmc.kmc_create([ly], prec, center=np.zeros(3))
    g = kmc.kmc_local_concentration(ctx, 0, N)
    kmc.kmc_destroy(ctx)
    o = _oracle(ly, N)
    fin = np.isfinite(o)
    assert np.array_equal(fin, np.isfinite(g))
    np.testing.assert_allclose(g[fin], o[fin], rtol=1e-13)


def test_lysosomes_of_a_batch():
    # the grid's scratch is the largest lysosome's; the others use part of it
    lyss = [_sample("random", n) for n in (100, 1500, 4000)]
    ctx = kmc.kmc_create(lyss, kmc.KMC_FP32_MIXED, center=np.zeros(3))
    for q in (1, 0, 2, 1):
        np.testing.assert_allclose(kmc.kmc_local_concentration(ctx, q, 20), _oracle(lyss[q], 20),
                                   rtol=1e-13)
    kmc.kmc_destroy(ctx)


@pytest.mark.parametrize("n", [2, 7, 8, 9, 33, 65])
@pytest.mark.parametrize("prec", [kmc.KMC_FP64_PLAIN, kmc.KMC_FP32_MIXED])
def test_small_samples(n, prec):
    """About the size from which the grid serves (8 NPs): few cells, and ranks up to all
    other NPs, which need the whole box."""
    ly = _sample("random", n)
    ctx = kmc.kmc_create([ly], prec, center=np.zeros(3))
    for N in {1, max(1, n // 2), min(n - 1, 64)}:
        np.testing.assert_allclose(kmc.kmc_local_concentration(ctx, 0, N), _oracle(ly, N),
                                   rtol=1e-13)
    kmc.kmc_destroy(ctx)
