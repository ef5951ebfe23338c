"""The FP64 search for the extrema of Eq. 2 (FP32 sign pass with FP64 inside its
error bound, Newton from an FP32 root) and the mean mode's two kernels, at the
places where they can go wrong: roots on the nodes of the scan, profiles near
switching, a flat or single-term profile, magnitudes outside FP32's range, and
runs cut into several spans of steps.

Tolerances: those of the FP64 step (moments 1e-12) and of the mean mode (1e-12),
which rest on a few ulp per operation; cut runs are compared bit for bit.
"""
import math

import numpy as np
import pytest

import oracle
from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu
V = math.pi * (14e-9) ** 3 / 6
MS = 1e6


@pytest.fixture(scope="module", autouse=True)
def _built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1407_2737_gb300 import build as kbuild
    kbuild.build()


def _lone(phis, K, T=300.0):
    """One-NP lysosomes whose axes make the angles phis with z."""
    return [inputs.Lysosome(pos=np.zeros((1, 3)), axis=np.array([[math.sin(p), 0.0, math.cos(p)]]),
                            vol=np.array([V]), Ms=MS, Keff=K, T=T, tau0=1e-10) for p in phis]


def _check(lyss, H, t_step=5e-8):
    m = np.concatenate([oracle.initial_moments(l.axis) for l in lyss])
    ctx = kmc.kmc_create(lyss, kmc.KMC_FP64_PLAIN, center=np.zeros(3))
    g = kmc.kmc_debug_step(ctx, np.full(len(lyss), H), t_step, 3, 9, m)
    o = [oracle.step(l, q, m[q:q + 1], H, t_step, 3, 9) for q, l in enumerate(lyss)]
    same = np.array([x["near"][0] == 0 for x in o])
    assert np.array_equal(g["n_min"], [x["n_min"][0] for x in o])
    assert np.array_equal(g["flipped"][same], np.array([x["flipped"][0] for x in o])[same])
    d = np.abs(g["m_out"] - np.concatenate([x["m_out"] for x in o]))[same]
    assert d.max() <= 1e-12


@pytest.mark.parametrize("h", [0.2, 0.6, 1.5])
def test_roots_on_scan_nodes(h):
    # k sin 2 theta_j = b sin(phi - theta_j): theta_j is an extremum to rounding
    K = 2e4
    H = h * 2 * K / MS
    th = 2 * math.pi * (np.arange(200) + 0.5) / 200
    s = np.sin(2 * th) / (2 * h)
    th, s = th[np.abs(s) <= 1], s[np.abs(s) <= 1]
    phi = (th + np.arcsin(s)) % (2 * math.pi)
    _check(_lone([p for p in phi if p <= math.pi], K), H)


@pytest.mark.parametrize("K,H", [(0.0, 0.01), (2e4, 0.0), (2e4, 1e-30), (1e-30, 0.02),
                                 (1e-27, 1e-33), (2e4, 1e6)])
def test_ends_of_the_range(K, H):
    _check(_lone([0.3, 1.1, math.pi / 2 - 1e-3, 2.0], K), H)


@pytest.mark.parametrize("eps", [1e-3, 1e-6, -1e-6, -1e-3])
def test_near_switching(eps):
    # the astroid h = (sin^2/3 phi + cos^2/3 phi)^-3/2, a little inside and outside
    for p in (0.2, 0.7, 1.3):
        h = (math.sin(p) ** (2 / 3) + math.cos(p) ** (2 / 3)) ** -1.5
        _check(_lone([math.pi - p], 2e4), h * (1 + eps) * 2 * 2e4 / MS)


@pytest.mark.parametrize("n,S,periods", [(10000, 200, 1), (10000, 200, 2), (40000, 400, 2)])
def test_mean_mode_in_spans(n, S, periods):
    # the first and the last exceed the workspace (64 MB; 1 GB for several periods), so
    # a period is solved in spans, anew in each period; the others fit and are solved once
    big = inputs.lattice_nodes_lysosome(n, 14e-9, 0.1, Keff=2e4, seed=1)
    small = inputs.lattice_nodes_lysosome(33, 14e-9, 0.1, Keff=2e4, seed=2)
    one = _lone([1.0], 2e4, T=0.0)[0]
    g = kmc.kmc_mean_run([small, big, one], 0.03, 1e5, S, periods, 0)
    assert np.array_equal(kmc.kmc_mean_run([small, one], 0.03, 1e5, S, periods, 0), g[[0, 2]])
    for q, ly in ((0, small), (2, one)):
        o = oracle.mean_run(ly.axis, ly.vol, ly.Ms, ly.Keff, ly.T, ly.tau0, 0.03, 1e5, S, periods,
                            0)
        np.testing.assert_allclose(g[q], o, rtol=0, atol=1e-12)


@pytest.mark.parametrize("S,H,K", [(1, 0.02, 2e4), (7, 0.0, 2e4), (7, 0.0, 0.0)])
def test_mean_mode_small(S, H, K):
    ly = inputs.lattice_nodes_lysosome(3, 14e-9, 0.1, Keff=K, seed=3)
    g = kmc.kmc_mean_run([ly], H, 1e5, S, 2, 1)
    o = oracle.mean_run(ly.axis, ly.vol, ly.Ms, ly.Keff, ly.T, ly.tau0, H, 1e5, S, 2, 1)
    np.testing.assert_allclose(g[0], o, rtol=0, atol=1e-12)
