"""Steps v-vii of an FP64 step where its FP32 shortcuts end: rates beyond FP32's
range in the draw u < P and draws close to P (only kmc_run takes that shortcut,
kmc_debug_step returns P itself, so runs are compared with the oracle's), and the
arc that holds the moment; and the square roots and inverse distances of its own.

Tolerances: those of an FP64 run (moments 1e-9 after some dozens of steps, which a
single other decision breaks by far) and of an FP64 step (moments 1e-12); where a
quantity stands alone, the units in the last place that its operations can lose.
"""
import math

import numpy as np
import pytest

import oracle
from paper_1407_2737_gb300 import inputs, kmc

pytestmark = pytest.mark.gpu
V0 = math.pi * (14e-9) ** 3 / 6


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


@pytest.mark.parametrize("delta", [1e-3, 2e-5, 1e-5, 1e-6, 1e-7, 1e-9, 1e-12])
def test_moments_at_the_ends_of_the_basins(delta):
    # within 1e-5 rad of a maximum FP64 settles the basin
    H, K = 0.3 * 2 * 2e4 / 1e6, 2e4
    ends = [t for t, _, is_min in oracle.extrema(K, 1e6, math.pi * (14e-9) ** 3 / 6, H, math.pi / 4)
            if not is_min]
    assert len(ends) == 2
    _same_basins([_plane(t + s * delta, H)[1] for t in ends for s in (-1, 1)], H)


@pytest.mark.parametrize("eps", [1e-2, 1e-4, 1e-5, 5e-6, 3e-6, 1e-6, 1e-7, 1e-8])
def test_draws_at_their_probabilities(eps):
    """One-NP lysosomes in the upper well, whose tau0 puts P a little above or below the
    first draw, inside and outside the band (4e-6 of P) in which FP64 decides."""
    a, _ = _plane(0.0, 0.0)
    H, t_step, seed, lyss, want = -0.014, 1e-6, 21, [], {}
    for q in range(64):
        ly = inputs.Lysosome(pos=np.zeros((1, 3)), axis=a[None], vol=np.array([math.pi * (12e-9) ** 3
                             / 6]), Ms=1e6, Keff=2e4, T=300.0, tau0=1e-10)
        lyss.append(ly)
        m, u = oracle.initial_moments(ly.axis), oracle.uniform(seed, 0, 0, q)
        if u > 0.95:  # above the equilibrium value of P
            continue
        aim = u * (1 + eps if q & 1 else 1 - eps)
        lo, hi = math.log(1e-25), math.log(1e3)  # P falls as tau0 grows
        for _ in range(100):
            ly.tau0 = math.exp(0.5 * (lo + hi))
            p = oracle.step(ly, q, m, H, t_step, seed, 0)["P"][0]
            lo, hi = (0.5 * (lo + hi), hi) if p > aim else (lo, 0.5 * (lo + hi))
        assert abs(p - aim) <= 1e-3 * eps * aim
        want[q] = float(q & 1)
    assert len(want) > 50
    ctx = kmc.kmc_create(lyss, kmc.KMC_FP64_PLAIN, center=np.zeros(3))
    kmc.kmc_run(ctx, H, 1 / t_step, 1, 1, 0, seed)
    got = {q: kmc.kmc_read(ctx, kmc.KMC_READ_COUNTERS, q)[kmc.CNT_JUMPS] for q in want}
    kmc.kmc_destroy(ctx)
    assert got == want


def test_inverse_distances():
    """The field of one NP on another, 1/r^3 from the symmetric form's own 1/r, at distances
    over 90 orders of magnitude. Roundings: the two coordinates, their
    difference, r^2 (3), 1/r (one or two units), its powers, the dot product and the sum:
    some 20 units of 1.1e-16 in a field of 1 to 2 times the scale, so 4e-15."""
    rng = np.random.default_rng(6)
    V, Ms, lyss, exact, moments = math.pi * (14e-9) ** 3 / 6, 1e6, [], [], []
    L = (6 * V / math.pi) ** (1 / 3)
    for r in np.exp(rng.uniform(math.log(1e-45), math.log(1e45), 400)).tolist() + [1.0, 2.0, 0.5]:
        e = inputs.random_axes(1, rng)[0]
        pos = np.stack([-0.5 * r * L * e, 0.5 * r * L * e])
        m = inputs.random_axes(2, rng)
        lyss.append(inputs.Lysosome(pos=pos, axis=m, vol=np.full(2, V), Ms=Ms, Keff=2e4, T=300.0,
                                    tau0=1e-10))
        moments.append(m)
        x, v = pos.astype(np.longdouble), m.astype(np.longdouble)
        d = x[1] - x[0]
        rr = np.sqrt((d * d).sum())
        d /= rr
        k = np.longdouble(1e-7) * Ms * V / rr ** 3  # mu0 / 4 pi
        exact.append(np.stack([k * (3 * (v[1 - i] @ d) * d - v[1 - i]) for i in (0, 1)]))
    ctx = kmc.kmc_create(lyss, kmc.KMC_FP64_PLAIN, center=np.zeros(3))
    kmc.kmc_launch_shape(ctx, dict(dict.fromkeys(kmc.SHAPE_KEYS, 0), warps=4, tile=32, tpl=1, rpl=1,
                                   fp64_parts=1))
    try:
        g = kmc.kmc_debug_step(ctx, np.zeros(len(lyss)), 5e-8, 3, 9, np.concatenate(moments))
    finally:
        kmc.kmc_destroy(ctx)
    exact = np.concatenate(exact)
    err = np.linalg.norm((g["B_dip"] - exact).astype(float) / np.linalg.norm(
        exact.astype(float), axis=1, keepdims=True), axis=1)
    print("largest relative error of a pair's field: %.2e" % err.max())
    assert err.max() <= 4e-15


def test_planes_of_lone_moments():
    """Without anisotropy the moment falls along the field: steps iii-v reduce to the
    plane's square roots and divisions and the sines of one root. cos phi, the
    normal part and the root err by some ten units of 1.1e-16 each: 3e-15. Fields down to
    where the square of the reduced field leaves sqrt_inv's own range and beyond it."""
    axes = inputs.random_axes(200, np.random.default_rng(8))
    lyss = [inputs.Lysosome(pos=np.zeros((1, 3)), axis=a[None], vol=np.array([V0]), Ms=1e6, Keff=0.0,
                            T=0.0, tau0=1e-10) for a in axes]
    for H in (0.02, 1.0, 1e-20, 1e-100, 1e-143, 1e-147, 1e100, 1e143, 1e147):
        ctx = kmc.kmc_create(lyss, kmc.KMC_FP64_PLAIN, center=np.zeros(3))
        g = kmc.kmc_debug_step(ctx, np.full(len(lyss), H), 5e-8, 3, 9,
                               np.concatenate([oracle.initial_moments(l.axis) for l in lyss]))
        kmc.kmc_destroy(ctx)
        assert np.abs(g["m_out"] - [0.0, 0.0, 1.0]).max() <= 3e-15, H
