// kmc_mean.cuh -- the Ref. [8] mode on the device (Sec. II.3): the mean
// magnetisation of non-interacting NPs, obtained by carrying the probability of
// each energy well instead of sampling jumps. Included only by kmc_step.cu,
// which owns the grid tables and the Eq. 2 helpers it uses.
//
// With no dipolar field the total field stays along z, so each NP keeps one
// working plane for the whole run: the plane of its easy axis a and z, with
// e_perp the unit vector of z normal to a (or a fallback when a is along z).
// The field enters Eq. 2 at the angle phi_z between a and z, or phi_z + pi
// when the field is negative. At every step, per NP, in FP64:
//   * extrema of Eq. 2 by the 200-node scan and Newton (as in the kMC step);
//   * with one minimum all probability sits in it; with two, the probability
//     of each old well moves to the new minimum whose basin (the arc between
//     the two maxima) contains the old well's angle;
//   * Eqs. 3-5 relax the two-well occupation towards its equilibrium over
//     t_step: p_A <- p_A,inf + (p_A - p_A,inf) e^{-(nu_A + nu_B) t_step},
//     p_A,inf = nu_B / (nu_A + nu_B), the barrier top being the lower maximum;
//   * <m_z> = sum_w p_w (cos th_w a_z + sin th_w e_perp,z), added volume-
//     weighted to the lysosome's loop record in 64-bit fixed point.
//
// The extrema of a step depend on its field alone, not on the occupations, and
// the field of step k is the same in every period. So the work is cut in two:
// kmc_mean_wells solves every (NP, step) of a span of steps at once, one thread
// each, and kmc_mean_carry, one thread per NP, carries the probabilities
// through the span's steps from those results. Where the whole period fits the
// workspace it is solved once for all periods. Bound: the FP64 pipe (a warp
// instruction every 16 cycles and SM), so the scan runs in FP32 with FP64 for
// the nodes within its error (SignProfile) and Newton starts from an FP32 root
// (root_in_cell). 2000 NPs, 200 steps: 75.4 ms with one
// thread per NP for the whole run (63 warps on 152 SMs, every step a serial chain
// of about 1.7e4 FP64 instructions), 0.65 ms now, of which the wells take 0.29 ms
// and the carry 0.09 ms.
#pragma once

namespace kmc {

constexpr int kMeanWarps = 4;

// The NP's fixed working plane: phi_z (the angle between axis and z, as its sine
// and cosine) and the z component of e_perp = normalise(z - (z.a) a).
__device__ __forceinline__ void mean_plane(const dbl4 &ax, double &epz, double &sphz,
                                           double &cphz) {
  double px = -ax.z * ax.x, py = -ax.z * ax.y, pz = 1.0 - ax.z * ax.z;
  double sp = sqrt(px * px + py * py + pz * pz);
  if (sp >= 1e-12) {
    const double r = 1.0 / sqrt(sp * sp + ax.z * ax.z);
    sphz = sp * r;
    cphz = ax.z * r;
  } else {  // a along z: any normal will do
    if (fabs(ax.x) > 0.9) {
      px = -ax.z;
      py = 0.0;
      pz = ax.x;
    } else {
      px = 0.0;
      py = ax.z;
      pz = -ax.y;
    }
    sp = sqrt(px * px + py * py + pz * pz);
    sphz = 0.0;
    cphz = (ax.z >= 0.0) ? 1.0 : -1.0;
  }
  epz = pz / sp;
}

// Block (x, y): item x (32 NPs, one per lane), steps k0 + 4 y + warp.
__global__ void __launch_bounds__(kMeanWarps * 32)
    kmc_mean_wells(const MeanArgs a, int k0, int k1) {
  __shared__ GridTables<double> tab;
  tab.load();
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = k0 + blockIdx.y * kMeanWarps + warp;
  if (k >= k1) return;  // the whole warp
  const MeanItem it = a.items[blockIdx.x];
  const MeanLysDev L = a.lys[it.l];
  const int i = L.off + it.t0 + min(lane, it.nt - 1);
  const dbl4 ax = a.axis[i];
  double epz, sphz, cphz;
  mean_plane(ax, epz, sphz, cphz);
  const double H = L.bmax * a.cos_k[k];
  const double b = fabs(H);
  Profile<double> pf;
  pf.k = L.k;
  pf.k2 = 2.0 * L.k;
  pf.bc = H < 0.0 ? -(b * cphz) : b * cphz;
  pf.bs = H < 0.0 ? -(b * sphz) : b * sphz;
  // step iv: brackets in grid order (node j of bracket q in byte q of nodes,
  // bit q of left_neg: de/dth < 0 there)
  const SignProfile sp(pf.k2, pf.bc, pf.bs);
  unsigned nodes = 0, left_neg = 0;
  int cnt = 0;
#pragma unroll 1
  for (int j0 = 0; j0 < kGrid; j0 += kMaxSeg) {
    const unsigned long long neg = fp64_signs(tab, pf, sp, j0, kMaxSeg);
    unsigned long long chg = (neg ^ (neg >> 1)) & ((1ull << kMaxSeg) - 1);
    while (chg) {
      const int q = __ffsll(static_cast<long long>(chg)) - 1;
      chg &= chg - 1;
      if (cnt < 4) {
        nodes |= static_cast<unsigned>(j0 + q) << (8 * cnt);
        left_neg |= static_cast<unsigned>((neg >> q) & 1) << cnt;
      }
      ++cnt;
    }
  }
  // Newton; the two minima (angle, energy, mean m_z) and maxima in grid order
  const double h = tab.th[1] - tab.th[0];
  double tmin0 = 0.0, tmin1 = 0.0, emin0 = 0.0, emin1 = 0.0, g0 = 0.0, g1 = 0.0;
  double tmax0 = 0.0, tmax1 = 0.0, e3 = 0.0;
  int nmin = 0, nmax = 0;
#pragma unroll 1
  for (int q = 0; q < min(cnt, 4); ++q) {
    const int j = (nodes >> (8 * q)) & 255;
    const bool is_min = (left_neg >> q) & 1;
    double s, c;
    double t = tab.th[j] + root_in_cell(pf, tab.sc[j].x, tab.sc[j].y, tab.ss[j], tab.cc[j], h,
                                        is_min, s, c);
    if (t >= Prec<double>::two_pi) t -= Prec<double>::two_pi;
    const double e = pf.e(s, c);
    if (is_min) {
      const double g = c * ax.z + s * epz;
      if (nmin == 0) {
        tmin0 = t;
        emin0 = e;
        g0 = g;
      } else {
        tmin1 = t;
        emin1 = e;
        g1 = g;
      }
      ++nmin;
    } else {
      if (nmax == 0) {
        tmax0 = t;
        e3 = e;
      } else {
        tmax1 = t;
        e3 = fmin(e3, e);
      }
      ++nmax;
    }
  }
  int flag = nmin;
  if (cnt > 4 || nmin > 2 || nmax > 2) flag = kMeanSkip;
  double pinf = 0.0, decay = 1.0;
  if (flag == 2) {
    if (on_arc<double>(tmin0, tmax0, tmax1)) flag |= kMeanArc;
    if (!L.t_zero) {
      // Eqs. 3-5 with nu t_step = exp(ln(t_step / tau0) - beta dE)
      const double beta = a.beta[i];
      const double nuA = exp(L.lognu0t - beta * (e3 - emin0));
      const double nuB = exp(L.lognu0t - beta * (e3 - emin1));
      const double sum = nuA + nuB;
      if (sum > 0.0) {
        flag |= kMeanRelax;
        decay = exp(-sum);
        pinf = nuB / sum;
      }
    }
  }
  if (lane < it.nt) {
    double *w = a.wells + static_cast<size_t>(k - k0) * kMeanFields * a.n;
    w[i] = tmin0;
    w[i + a.n] = tmin1;
    w[i + 2ll * a.n] = tmax0;
    w[i + 3ll * a.n] = tmax1;
    w[i + 4ll * a.n] = pinf;
    w[i + 5ll * a.n] = decay;
    w[i + 6ll * a.n] = g0;
    w[i + 7ll * a.n] = g1;
    a.flags[static_cast<size_t>(k - k0) * a.n + i] = flag;
  }
}

// on_arc by FP32 angles (all within 1e-6 rad of the FP64 ones) unless x lies within
// 1e-5 rad of an end. The ends are maxima of different brackets, 0.03 rad apart at least.
__device__ __forceinline__ bool on_arc_fast(double x, double from, double to) {
  const float t = static_cast<float>(x), f = static_cast<float>(from), e = static_cast<float>(to);
  const float d1 = fabsf(t - f), d2 = fabsf(t - e);
  const float near = fminf(fminf(d1, Prec<float>::two_pi - d1), fminf(d2, Prec<float>::two_pi - d2));
  return near > 1e-5f ? on_arc<float>(t, f, e) : on_arc<double>(x, from, to);
}

// One block per item of 32 NPs: the probabilities through steps k0 .. k1 - 1 of
// period p, from and to the state of the NPs (a.state; first: the start of the
// run), in tiles of kCarryTile steps. Warp 0 runs the chain of a tile, which is
// all that is serial: occupations of a step from those before it, four dependent
// FP64 operations. Meanwhile the helper warps, one per step of a tile, load the
// next tile into shared memory, find for its steps which basin holds the wells of
// the step before (on_arc_fast; a span's first step and one that follows a step
// without wells are left to the chain) and reduce the previous tile's
// contributions to the loop. 200 steps of 2000 NPs: one warp doing all of it 242 us, with
// four helpers and the basins in the chain 182, now 87.
constexpr int kCarryTile = 8, kCarryHelpers = 8;

__global__ void __launch_bounds__(32 * (1 + kCarryHelpers))
    kmc_mean_carry(const MeanArgs a, int k0, int k1, int p, int first) {
  __shared__ double s_well[2][kCarryTile][kMeanFields][32];
  __shared__ double s_mz[2][kCarryTile][32];
  __shared__ int s_flag[2][kCarryTile][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const MeanItem it = a.items[blockIdx.x];
  const MeanLysDev L = a.lys[it.l];
  const bool active = lane < it.nt;
  const int i = L.off + it.t0 + min(lane, it.nt - 1);
  const int steps = k1 - k0, tiles = (steps + kCarryTile - 1) / kCarryTile;
  // helpers: the wells of tile t, and where those of the step before went
  auto load = [&](int t) {
    for (int q = warp - 1; q < kCarryTile; q += kCarryHelpers) {
      const int r = t * kCarryTile + q;
      if (r >= steps) break;
      const double *src = a.wells + static_cast<size_t>(r) * kMeanFields * a.n + i;
      double v[kMeanFields];
#pragma unroll
      for (int f = 0; f < kMeanFields; ++f) v[f] = src[static_cast<size_t>(f) * a.n];
      int flag = a.flags[static_cast<size_t>(r) * a.n + i];
      double t0 = 0.0, t1 = 0.0;
      int before = 0;
      if (r > 0) {
        t0 = src[-static_cast<long long>(kMeanFields) * a.n];
        t1 = src[-static_cast<long long>(kMeanFields) * a.n + a.n];
        before = a.flags[static_cast<size_t>(r - 1) * a.n + i];
      }
      if ((flag & 3) == 2 && (before & 3) != 0 && !(before & kMeanSkip)) {
        const bool arcA = (flag & kMeanArc) != 0;
        flag |= kMeanKnown;
        if (on_arc_fast(t0, v[2], v[3]) == arcA) flag |= kMeanIn0;
        if (on_arc_fast(t1, v[2], v[3]) == arcA) flag |= kMeanIn1;
      }
#pragma unroll
      for (int f = 0; f < kMeanFields; ++f) s_well[t & 1][q][f][lane] = v[f];
      s_flag[t & 1][q][lane] = flag;
    }
  };
  // helpers: the volume-weighted sums of tile t into the loop record
  auto reduce = [&](int t) {
    if (p < a.discard) return;
    for (int q = warp - 1; q < kCarryTile; q += kCarryHelpers) {
      const int r = t * kCarryTile + q;
      if (r >= steps) break;
      double c = s_mz[t & 1][q][lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
      if (lane == 0) {
        const long long rec = static_cast<long long>(p - a.discard) * a.S + k0 + r;
        atomicAdd(reinterpret_cast<unsigned long long *>(
                      &a.loop[static_cast<long long>(it.l) * a.n_rec + rec]),
                  static_cast<unsigned long long>(__double2ll_rn(c * kLoopScale)));
      }
    }
  };
  // warp 0: the wells as of the last step that had any: angles, probabilities (0
  // for a well that does not exist) and mean m_z
  double th0 = 0.0, th1 = 0.0, p0 = 1.0, p1 = 0.0, g0 = 0.0, g1 = 0.0, vfrac = 0.0;
  double *st = a.state + i;
  bool bad = false;
  if (warp == 0) {
    vfrac = active ? a.vfrac[i] : 0.0;
    if (first) {  // all probability in the well along +-a with m_z >= 0
      const double az = a.axis[i].z;
      th0 = (az >= 0.0) ? 0.0 : 0.5 * Prec<double>::two_pi;
      g0 = fabs(az);
    } else {
      th0 = st[0];
      th1 = st[a.n];
      p0 = st[2ll * a.n];
      p1 = st[3ll * a.n];
      g0 = st[4ll * a.n];
      g1 = st[5ll * a.n];
    }
  } else {
    load(0);
  }
  __syncthreads();
  for (int t = 0; t < tiles; ++t) {
    if (warp == 0) {
      const int cnt = min(kCarryTile, steps - t * kCarryTile);
#pragma unroll 2
      for (int q = 0; q < cnt; ++q) {
        const double(&w)[kMeanFields][32] = s_well[t & 1][q];
        const int flag = s_flag[t & 1][q][lane];
        const int nmin = flag & 3;
        const bool skip = (flag & kMeanSkip) != 0;
        bad = bad || (active && skip);
        if (nmin == 1) {
          p0 = 1.0;
          p1 = 0.0;
        } else if (nmin == 2) {
          const double pinf = w[4][lane];
          bool in0 = (flag & kMeanIn0) != 0, in1 = (flag & kMeanIn1) != 0;
          if (!(flag & kMeanKnown)) {
            const double M1 = w[2][lane], M2 = w[3][lane];
            const bool arcA = (flag & kMeanArc) != 0;
            in0 = on_arc<double>(th0, M1, M2) == arcA;
            in1 = on_arc<double>(th1, M1, M2) == arcA;
          }
          double pA = (in0 ? p0 : 0.0) + (in1 ? p1 : 0.0);
          double pB = (in0 ? 0.0 : p0) + (in1 ? 0.0 : p1);
          if (flag & kMeanRelax) {
            pA = pinf + (pA - pinf) * w[5][lane];
            pB = 1.0 - pA;
          }
          p0 = pA;
          p1 = pB;
        }
        if (nmin != 0 && !skip) {
          th0 = w[0][lane];
          th1 = w[1][lane];
          g0 = w[6][lane];
          g1 = w[7][lane];
        }
        s_mz[t & 1][q][lane] = skip ? 0.0 : vfrac * (p0 * g0 + p1 * g1);
      }
    } else {
      if (t > 0) reduce(t - 1);
      if (t + 1 < tiles) load(t + 1);
    }
    __syncthreads();
  }
  if (warp != 0) {
    if (tiles > 0) reduce(tiles - 1);
    return;
  }
  if (active) {
    st[0] = th0;
    st[a.n] = th1;
    st[2ll * a.n] = p0;
    st[3ll * a.n] = p1;
    st[4ll * a.n] = g0;
    st[5ll * a.n] = g1;
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(a.err, kErrExtrema);
}

}  // namespace kmc
