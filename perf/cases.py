"""Performance cases: what a program that uses this package has it do, through
its public entry points, from the smallest calls to the largest.

    listed()            the named cases
    draw(rng)           one more case from the same ranges
    prepare(case, seed) a program's state before the call: inputs and handles
    run(state)          one pass of the call, with its outputs
    work(case)          the bytes and operations the path cannot do without
    exact(case, seed)   run()'s outputs for these inputs, in 64 bits, by torch
                        and numpy alone

Kinds of case:

    run    kmc_run of one or several lysosomes over one field period, then the
           reads of its results (the M(H) loop, the moments, and in FP64 the
           energy of each NP: for NPs that do not jump it is the small
           difference of large terms, which float32 moments do not hold)
    field  kmc_dipolar_field_noalloc: the dipolar field on device buffers
    phi    kmc_local_concentration: Eq. 8 for every NP
    mean   kmc_mean_run: the mode of Ref. [8]
    rsa    kmc_regenerate_rsa: random sequential addition, then the positions

Samples are the paper's: monodisperse NPs displaced at random about the nodes
of a cubic lattice as far as they can be without touching (Sec. II.4), easy
axes uniform on the sphere, a field along z at 100 kHz. The FP32-mixed runs
take magnetically hard, dilute NPs in a weak field (d = 20 nm, K_eff = 5e4 J/m^3,
1 %, 10 to 20 mT: inside the batch workload's ranges), which seldom jump: FP32
barriers put a relative rounding noise of about 1e-5 on the jump probability P, so
that in a sample whose NPs all jump some draw u < P falls within it every few
periods, and from there on two correct runs are different realisations. A step
costs the same there: two wells, four extrema, rates and a draw for nearly every
NP. The FP64 runs take the workloads' own materials.

Results of the FP32-mixed path come back from the library in float64 buffers
but hold float32 values (moments) or sums of them; run() returns them as the
float32 they are.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_1407_2737_gb300 import inputs, kmc

MU0 = 4.0e-7 * math.pi
KB = 1.380649e-23
FREQ = 1e5            # Hz, of every workload
MAT_SMALL = (12e-9, 1.3e4, 0.05, 0.020)  # d (m), K_eff, concentration, mu0 Hmax (T)
MAT_SINGLE = (14e-9, 2.0e4, 0.10, 0.020)
MAT_HARD = (20e-9, 5.0e4, 0.01, 0.020)


def listed():
    return [
        # the 100-NP workload, all in FP64: the smallest run, the reference
        # that a user checks the mixed path against
        {"name": "run f64 100", "kind": "run", "fp32": False, "n": 100, "k": 1, "S": 200},
        # the same size in FP32-mixed: a step is a few microseconds of latency
        {"name": "run f32 100", "kind": "run", "fp32": True, "n": 100, "k": 1, "S": 200},
        # FP64 where the pair sum rules; 2000 NPs, the usual lysosome
        {"name": "run f64 2000", "kind": "run", "fp32": False, "n": 2000, "k": 1, "S": 50},
        # eight seeds of one 2000-NP sample: the benchmark's workload
        {"name": "run f32 8x2000", "kind": "run", "fp32": True, "n": 2000, "k": 8, "S": 100},
        # one lysosome of the concentration sweep's size
        {"name": "run f32 8000", "kind": "run", "fp32": True, "n": 8000, "k": 1, "S": 100},
        # a batch of different lysosomes, NP counts lognormal (ragged)
        {"name": "batch f32 96", "kind": "batch", "n": 1500, "k": 96, "S": 100},
        # the largest workload: one lysosome of 50 000 NPs
        {"name": "run f32 50000", "kind": "run", "fp32": True, "n": 50000, "k": 1, "S": 20},
        # the field alone, called on another framework's device buffers: a small
        # odd size, where launches count, and the largest the call takes
        {"name": "field 333", "kind": "field", "n": 333},
        {"name": "field 8192", "kind": "field", "n": 8192},
        # Eq. 8 at the paper's N = 20 on the large lysosome
        {"name": "phi 50000", "kind": "phi", "n": 50000, "N": 20},
        # the mode of Ref. [8] on the usual lysosome, a period of 200 steps
        {"name": "mean 2000", "kind": "mean", "n": 2000, "S": 200},
        # a fresh random placement of a large lysosome at the highest
        # concentration the workloads place at random
        {"name": "rsa 20000", "kind": "rsa", "n": 20000, "c": 0.10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run32", "run32", "run32", "run64", "batch", "field", "phi", "mean", "rsa"])
    if kind == "run32":
        n = _log_int(rng, 50, 45000)
        k = rng.choice([1, 1, 2, 3, 4, 8]) if n <= 4000 else 1
        S = max(10, min(rng.choice([40, 75, 100, 200]), int(4e10 / (k * n * n))))
        return {"kind": "run", "fp32": True, "n": n, "k": k, "S": S}
    if kind == "run64":
        n = _log_int(rng, 40, 2000)
        return {"kind": "run", "fp32": False, "n": n, "k": 1,
                "S": max(10, min(rng.choice([50, 100, 200]), int(4e8 / (n * n))))}
    if kind == "batch":
        return {"kind": "batch", "n": rng.randint(300, 1500), "k": rng.randint(12, 96),
                "S": rng.choice([40, 60, 100])}
    if kind == "field":
        return {"kind": "field", "n": _log_int(rng, 7, 8192)}
    if kind == "phi":
        return {"kind": "phi", "n": _log_int(rng, 500, 50000), "N": rng.randint(1, 64)}
    if kind == "mean":
        return {"kind": "mean", "n": _log_int(rng, 100, 4000), "S": rng.choice([50, 100, 150])}
    return {"kind": "rsa", "n": _log_int(rng, 300, 20000), "c": round(rng.uniform(0.01, 0.15), 4)}


# ---------------------------------------------------------------------------
# Inputs.

def _sample(n, mat, seed):
    d, K, c, _ = mat
    rng = np.random.Generator(np.random.PCG64(seed))
    ly = inputs.lattice_nodes_lysosome(n, d, c, Keff=K)
    pos = ly.pos + (inputs.random_axes(n, rng) * rng.uniform(0, inputs.max_disorder(d, c), (n, 1)))
    return dataclasses.replace(ly, pos=inputs.snap_to_float32(pos, d), axis=inputs.random_axes(n, rng))


def _lysosomes(case, seed):
    """The lysosomes of a run and their field amplitudes."""
    if case["kind"] == "batch":
        rng = np.random.Generator(np.random.PCG64(1000 * case["n"] + case["k"]))
        sizes = np.clip(np.round(case["n"] * np.exp(0.5 * rng.standard_normal(case["k"]))),
                        100, 10 * case["n"]).astype(int)  # the case's, whatever the seed
        rng = np.random.Generator(np.random.PCG64(seed))
        out, H = [], []
        for q, n in enumerate(sizes):
            mat = (rng.uniform(18e-9, 20e-9), rng.uniform(4.5e4, 5e4), rng.uniform(0.008, 0.012), 0)
            out.append(_sample(int(n), mat, seed * 1009 + q))
            H.append(rng.integers(10, 21) * 1e-3)
        return out, np.array(H)
    if case["fp32"]:
        mat = MAT_HARD
    else:
        mat = MAT_SMALL if case["n"] < 1000 else MAT_SINGLE
    ly = _sample(case["n"], mat, seed)
    return inputs.replicate(ly, case["k"]), np.array([mat[3]])


def _field_inputs(case, seed):
    ly = _sample(case["n"], MAT_SINGLE, seed)
    m = inputs.random_axes(case["n"], np.random.Generator(np.random.PCG64(seed + 1)))
    return ly, m


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": seed, "kind": kind}
    if kind in ("run", "batch"):
        lys, s["H"] = _lysosomes(case, seed)
        s["fp32"] = kind == "batch" or case["fp32"]
        s["ctx"] = kmc.kmc_create(
            lys, kmc.KMC_FP32_MIXED if s["fp32"] else kmc.KMC_FP64_PLAIN, center=np.zeros(3))
    elif kind == "field":
        ly, m = _field_inputs(case, seed)
        dev = torch.device("cuda")
        s["pos"] = torch.tensor(ly.pos, dtype=torch.float64, device=dev)
        s["m"] = torch.tensor(m, dtype=torch.float64, device=dev)
        s["vol"] = torch.tensor(ly.vol, dtype=torch.float64, device=dev)
        s["B"] = torch.empty_like(s["pos"])
        s["status"] = torch.empty(1, dtype=torch.int32, device=dev)
        s["Ms"], s["d"] = ly.Ms, ly.d
    elif kind == "phi":
        s["ctx"] = kmc.kmc_create([_sample(case["n"], MAT_SINGLE, seed)], center=np.zeros(3))
    elif kind == "mean":
        s["lys"] = [_sample(case["n"], MAT_SINGLE, seed)]
        s["H"] = np.array([MAT_SINGLE[3]])
    else:
        d, K, _, _ = MAT_SINGLE
        s["ctx"] = kmc.kmc_create([_sample(case["n"], (d, K, case["c"], 0), seed)],
                                  center=np.zeros(3))
        s["radius"], s["d"] = inputs.lysosome_radius(case["n"], d, case["c"]), d
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind in ("run", "batch"):
        ctx = s["ctx"]
        kmc.kmc_run(ctx, s["H"], FREQ, case["S"], 1, 0, s["seed"])
        dt = np.float32 if s["fp32"] else np.float64
        k = len(ctx.sizes)
        out = {"loop": np.concatenate([kmc.kmc_read(ctx, kmc.KMC_READ_LOOP_M, q)
                                       for q in range(k)]).astype(dt),
               "m": np.concatenate([kmc.kmc_read(ctx, kmc.KMC_READ_MOMENTS, q)
                                    for q in range(k)]).astype(dt)}
        if not s["fp32"]:
            out["energy"] = np.concatenate([kmc.kmc_read(ctx, kmc.KMC_READ_NP_ENERGY, q)
                                            for q in range(k)])
        return out
    if kind == "field":
        kmc.kmc_dipolar_field_noalloc(case["n"], s["pos"].data_ptr(), s["m"].data_ptr(),
                                      s["vol"].data_ptr(), s["Ms"], np.zeros(3), s["d"],
                                      s["B"].data_ptr(),
                                      stream_handle=torch.cuda.current_stream().cuda_stream,
                                      status_dev=s["status"].data_ptr())
        return {"B": s["B"].float(), "status": s["status"]}
    if kind == "phi":
        return kmc.kmc_local_concentration(s["ctx"], 0, case["N"])
    if kind == "mean":
        return kmc.kmc_mean_run(s["lys"], s["H"], FREQ, case["S"], 1, 0)
    used = kmc.kmc_regenerate_rsa(s["ctx"], 0, s["radius"], s["d"], s["seed"], 0)
    return {"used": used, "pos": kmc.kmc_read(s["ctx"], kmc.KMC_READ_POSITIONS)}


# ---------------------------------------------------------------------------
# Work. Of Eq. 1 per unordered pair: separation 3, r^2 5, reciprocal square
# root 1, its powers 2, and for each of the two NPs m.d 5, scaling 1, direction
# and moment 6, sum 6; so 23.5 flops per ordered pair. Steps iii-vii per NP and
# step: 200 nodes of dE/dtheta (5 each) and about 500 for the rest.

_PAIR, _UPDATE = 23.5, 1500.0


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "run":
        w = 4 if case["fp32"] else 8
        N = n * case["k"]
        return {"bytes": N * (10 * w + 24) + 8 * case["S"] * case["k"],
                "flops": case["S"] * (case["k"] * _PAIR * n * n + _UPDATE * N)}
    if kind == "batch":  # mean and mean square of the lognormal sizes
        N, N2 = case["k"] * n * math.exp(0.125), case["k"] * n * n * math.exp(0.5)
        return {"bytes": N * 64 + 8 * case["S"] * case["k"],
                "flops": case["S"] * (_PAIR * N2 + _UPDATE * N)}
    if kind == "field":
        return {"bytes": n * 80, "flops": _PAIR * n * n}
    if kind == "phi":  # each NP's list, and the distances to a few times N neighbours
        return {"bytes": n * 40, "flops": n * 8.0 * 4 * case["N"]}
    if kind == "mean":
        return {"bytes": n * 40, "flops": case["S"] * _UPDATE * n}
    return {"bytes": n * 48, "flops": n * 200.0}


# ---------------------------------------------------------------------------
# The same in 64 bits, by torch and numpy alone.

def _philox(c, key):
    """Philox4x32-10: words of the counters c (four arrays) under `key`."""
    mask, sh = np.uint64(0xFFFFFFFF), np.uint64(32)
    c = [np.asarray(x, dtype=np.uint64) & mask for x in c]
    k0, k1 = key & 0xFFFFFFFF, (key >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> sh) ^ c[1] ^ np.uint64(k0), p1 & mask, (p0 >> sh) ^ c[3] ^ np.uint64(k1),
             p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _u53(hi, lo):
    return ((hi << np.uint64(21)) ^ (lo >> np.uint64(11))).astype(np.float64) * 2.0 ** -53


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _pair_sum(pos, mv):
    """sum_j 3 (mv_j . d) d / r^5 - mv_j / r^3 for every NP (Eq. 1)."""
    n = pos.shape[0]
    step = max(1, int(3e7) // n)
    out = torch.empty_like(pos)
    for a in range(0, n, step):
        d = pos[None, :, :] - pos[a:a + step, None, :]
        r2 = d.square().sum(-1)
        r2[torch.arange(d.shape[0]), torch.arange(a, a + d.shape[0])] = math.inf
        q3 = r2.pow(-1.5)
        s = 3.0 * torch.einsum("ijk,jk->ij", d, mv) * q3 / r2
        out[a:a + step] = torch.einsum("ij,ijk->ik", s, d) - q3 @ mv
    return out


def _pair_matrix(pos):
    """Eq. 1 as a matrix [3n, 3n] acting on the moments (small n)."""
    n = pos.shape[0]
    T = torch.empty(n, 3, n, 3, dtype=pos.dtype, device=pos.device)
    step = max(1, int(3e7) // n)
    eye = torch.eye(3, dtype=pos.dtype, device=pos.device)
    for a in range(0, n, step):
        d = pos[None, :, :] - pos[a:a + step, None, :]
        r2 = d.square().sum(-1)
        r2[torch.arange(d.shape[0]), torch.arange(a, a + d.shape[0])] = math.inf
        q3 = r2.pow(-1.5)
        t = 3.0 * (q3 / r2)[..., None, None] * d[..., :, None] * d[..., None, :]
        T[a:a + step] = (t - q3[..., None, None] * eye).permute(0, 2, 1, 3)
    return T.reshape(3 * n, 3 * n)


def _extrema(K, bc, bs):
    """Extrema of K sin^2 th - bc cos th - bs sin th per NP (K, bc, bs: [n]), by
    the 200-node scan and bisection: count and, in grid order, up to four
    (angle, energy, is a minimum)."""
    n, dev = bc.shape[0], bc.device
    th = 2.0 * math.pi * (torch.arange(200, dtype=torch.float64, device=dev) + 0.5) / 200

    def d1(k, c, s, t):
        return k * torch.sin(2 * t) + c * torch.sin(t) - s * torch.cos(t)

    neg = d1(K[:, None], bc[:, None], bs[:, None], th[None, :]) < 0
    chg = neg != torch.roll(neg, -1, dims=1)
    np_i, node = torch.nonzero(chg, as_tuple=True)
    rank = (torch.cumsum(chg, dim=1) - 1)[np_i, node]
    lo = th[node].clone()
    hi = lo + 2.0 * math.pi / 200
    left = neg[np_i, node]
    k, c, s = K[np_i], bc[np_i], bs[np_i]
    for _ in range(56):
        x = 0.5 * (lo + hi)
        same = (d1(k, c, s, x) < 0) == left
        lo, hi = torch.where(same, x, lo), torch.where(same, hi, x)
    x = 0.5 * (lo + hi)
    e = k * torch.sin(x).square() - c * torch.cos(x) - s * torch.sin(x)
    t4 = torch.zeros(n, 4, dtype=torch.float64, device=dev)
    e4, m4 = torch.zeros_like(t4), torch.zeros(n, 4, dtype=torch.bool, device=dev)
    t4[np_i, rank], e4[np_i, rank], m4[np_i, rank] = x % (2 * math.pi), e, left
    cnt = chg.sum(1)
    if int(cnt.max()) > 4:
        raise ValueError("more than four extrema")
    return cnt, t4, e4, m4


def _wells(cnt, t4, e4, m4):
    """Per NP: two wells?, angle and energy of each minimum and maximum in grid
    order (the second repeats the first where there is one)."""
    two = cnt == 4
    idx = torch.arange(4, device=cnt.device)[None, :]
    ok = idx < cnt[:, None]
    mins = torch.argsort(torch.where(m4 & ok, idx, idx + 8), dim=1)[:, :2]
    maxs = torch.argsort(torch.where(~m4 & ok, idx, idx + 8), dim=1)[:, :2]
    mins[:, 1] = torch.where(two, mins[:, 1], mins[:, 0])
    maxs[:, 1] = torch.where(two, maxs[:, 1], maxs[:, 0])
    return two, t4.gather(1, mins), e4.gather(1, mins), t4.gather(1, maxs), e4.gather(1, maxs)


def _on_arc(x, a, b):
    tp = 2 * math.pi
    dx, dt = (x - a) % tp, (b - a) % tp
    return (dx > 0) & (dx <= dt)


def _exact_run(ly, index, H, S, seed):
    """One period of the method for one lysosome, from the moments along the axes."""
    dev, n = _dev(), ly.n
    t64 = lambda v: torch.tensor(np.asarray(v), dtype=torch.float64, device=dev)  # noqa: E731
    a, vol = t64(ly.axis), t64(ly.vol)
    a = a / a.norm(dim=1, keepdim=True)
    m = torch.where(a[:, 2:] >= 0, a, -a)
    pos, w = t64(ly.pos) / ly.d, MU0 * ly.Ms * vol / (4 * math.pi * ly.d ** 3)
    T = _pair_matrix(pos) if n <= 6000 else None
    loop, E = np.zeros(S), torch.zeros(n, dtype=torch.float64, device=dev)
    lognu, beta = math.log(1.0 / (FREQ * S) / ly.tau0), 1.0 / (KB * ly.T)
    ids = np.arange(n)
    for k in range(S):
        Hk = H * math.cos(2 * math.pi * k / S)
        mv = w[:, None] * m
        B = (T @ mv.reshape(-1)).reshape(n, 3) if T is not None else _pair_sum(pos, mv)
        B = B + torch.tensor([0.0, 0.0, Hk], dtype=torch.float64, device=dev)
        b = B.norm(dim=1)
        h = B / b[:, None]
        cphi = (a * h).sum(1)
        perp = h - cphi[:, None] * a
        sphi = perp.norm(dim=1)
        e = perp / sphi[:, None]
        th0 = torch.atan2((m * e).sum(1), (m * a).sum(1)) % (2 * math.pi)
        MV = ly.Ms * vol
        two, tmin, emin, tmax, emax = _wells(*_extrema(ly.Keff * vol, MV * b * cphi, MV * b * sphi))
        first = _on_arc(th0, tmax[:, 0], tmax[:, 1]) == _on_arc(tmin[:, 0], tmax[:, 0], tmax[:, 1])
        wa = torch.where(two & ~first, 1, 0)[:, None]
        e3 = emax.min(dim=1).values
        ea, eb = emin.gather(1, wa)[:, 0], emin.gather(1, 1 - wa)[:, 0]
        na, nb = torch.exp(lognu - beta * (e3 - ea)), torch.exp(lognu - beta * (e3 - eb))
        P = na / (na + nb) * -torch.expm1(-(na + nb))
        step = np.full(n, k)
        c = _philox([step, np.zeros(n), ids, np.full(n, index)], seed)
        jump = two & (t64(_u53(c[0], c[1])) < P)
        th = tmin.gather(1, torch.where(jump[:, None], 1 - wa, wa))
        new = torch.cos(th) * a + torch.sin(th) * e
        E += Hk * (new[:, 2] - m[:, 2])
        m = new
        loop[k] = float((vol * m[:, 2]).sum() / vol.sum())
    return loop, m.cpu().numpy(), (ly.Ms * vol * E).cpu().numpy()


def _exact_mean(ly, H, S):
    dev = _dev()
    a = torch.tensor(ly.axis, dtype=torch.float64, device=dev)
    a = a / a.norm(dim=1, keepdim=True)
    vol = torch.tensor(ly.vol, dtype=torch.float64, device=dev)
    sp = torch.sqrt((1 - a[:, 2] ** 2))
    phz, az, epz = torch.atan2(sp, a[:, 2]), a[:, 2], sp
    thw = torch.stack([torch.where(az >= 0, 0.0, math.pi).double()] * 2, 1)
    pw = torch.stack([torch.ones_like(az), torch.zeros_like(az)], 1)
    lognu, beta, MV = math.log(1.0 / (FREQ * S) / ly.tau0), 1.0 / (KB * ly.T), ly.Ms * vol
    loop = np.zeros(S)
    for k in range(S):
        Hk = H * math.cos(2 * math.pi * k / S)
        phi = phz + math.pi if Hk < 0 else phz
        two, tmin, emin, tmax, emax = _wells(*_extrema(
            ly.Keff * vol, MV * abs(Hk) * torch.cos(phi), MV * abs(Hk) * torch.sin(phi)))
        arcA = _on_arc(tmin[:, 0], tmax[:, 0], tmax[:, 1])
        inA = torch.stack([_on_arc(thw[:, q], tmax[:, 0], tmax[:, 1]) == arcA for q in (0, 1)], 1)
        pA = (pw * inA).sum(1)
        e3 = emax.min(dim=1).values
        nA, nB = torch.exp(lognu - beta * (e3 - emin[:, 0])), torch.exp(lognu - beta * (e3 - emin[:, 1]))
        inf = nB / (nA + nB)
        pA = inf + (pA - inf) * torch.exp(-(nA + nB))
        p0 = torch.where(two, pA, torch.ones_like(pA))
        thw, pw = tmin, torch.stack([p0, 1 - p0], 1)
        mz = (pw * (torch.cos(thw) * az[:, None] + torch.sin(thw) * epz[:, None])).sum(1)
        loop[k] = float((vol * mz).sum() / vol.sum())
    return loop[None, :]


def _exact_rsa(n, radius, d, seed):
    """Candidates in order, each kept unless a kept one is closer than d."""
    Rb, kept, grid, used, c0 = radius - 0.5 * d, [], {}, 0, 0

    def uni(sub, ids):
        c = _philox([np.zeros(len(ids)), np.full(len(ids), 0x80000000 | sub), ids, np.zeros(len(ids))], seed)
        return _u53(c[0], c[1]), _u53(c[2], c[3])

    while len(kept) < n:
        ids = np.arange(c0, c0 + 2 * n)
        z, az = uni(3, ids)
        z = 1.0 - 2.0 * z
        rho = np.sqrt(np.maximum(1.0 - z * z, 0.0))
        x = np.maximum(np.maximum(*uni(4, ids)), uni(5, ids)[0])
        p = (Rb * x)[:, None] * np.stack([rho * np.cos(2 * math.pi * az),
                                          rho * np.sin(2 * math.pi * az), z], 1)
        cell = np.floor(p / d).astype(int).tolist()
        pts = p.tolist()
        for i, ((cx, cy, cz), (px, py, pz)) in enumerate(zip(cell, pts)):
            ok = True
            for ix in (cx - 1, cx, cx + 1):
                for iy in (cy - 1, cy, cy + 1):
                    for iz in (cz - 1, cz, cz + 1):
                        for qx, qy, qz in grid.get((ix, iy, iz), ()):
                            if (px - qx) ** 2 + (py - qy) ** 2 + (pz - qz) ** 2 < d * d:
                                ok = False
            if ok:
                grid.setdefault((cx, cy, cz), []).append((px, py, pz))
                kept.append((px, py, pz))
                if len(kept) == n:
                    used = c0 + i + 1
                    break
        c0 += 2 * n
    return {"used": used, "pos": np.array(kept)}


def exact(case, seed):
    kind, dev = case["kind"], _dev()
    if kind in ("run", "batch"):
        lys, H = _lysosomes(case, seed)
        if sum(ly.n ** 2 for ly in lys) * case["S"] > 1.5e10:
            return None
        got = [_exact_run(ly, q, float(H[q % len(H)]), case["S"], seed)
               for q, ly in enumerate(lys)]
        out = {"loop": np.concatenate([g[0] for g in got]), "m": np.concatenate([g[1] for g in got])}
        if kind == "run" and not case["fp32"]:
            out["energy"] = np.concatenate([g[2] for g in got])
        return out
    if kind == "field":
        ly, m = _field_inputs(case, seed)
        pos = torch.tensor(ly.pos, dtype=torch.float64, device=dev) / ly.d
        w = MU0 * ly.Ms * torch.tensor(ly.vol, dtype=torch.float64, device=dev) / (4 * math.pi * ly.d ** 3)
        return {"B": _pair_sum(pos, w[:, None] * torch.tensor(m, dtype=torch.float64, device=dev)),
                "status": None}
    if kind == "phi":
        ly, N = _sample(case["n"], MAT_SINGLE, seed), case["N"]
        pos = torch.tensor(ly.pos, dtype=torch.float64, device=dev) / ly.d
        r = torch.empty(ly.n, dtype=torch.float64, device=dev)
        step = max(1, int(3e7) // ly.n)
        for a in range(0, ly.n, step):
            d2 = (pos[None, :, :] - pos[a:a + step, None, :]).square().sum(-1)
            r[a:a + step] = d2.topk(N + 1, dim=1, largest=False).values[:, -1].sqrt() * ly.d
        return (3.0 * N * torch.tensor(ly.vol, device=dev) / (4 * math.pi * r ** 3)).cpu().numpy()
    if kind == "mean":
        return _exact_mean(_sample(case["n"], MAT_SINGLE, seed), MAT_SINGLE[3], case["S"])
    d = MAT_SINGLE[0]
    return _exact_rsa(case["n"], inputs.lysosome_radius(case["n"], d, case["c"]), d, seed)
