// kmc_field_f64.cuh -- the FP64-plain step in the symmetric pair form: a field
// kernel that forms every unordered pair of NPs once for both of them, and an
// update kernel that adds the partial sums and runs steps iii-vii. Included
// only by kmc_step.cu, which owns block_update.
//
// Bound: the FP64 pipe, one warp instruction per 16 cycles and SM (1/64 of the
// FP32 rate); shuffles, loads and integer work are free beside it. Per
// unordered pair it takes 33 FP64 instructions: separation 3, r^2 3, 1/r 5 (below),
// its powers 2, and for each of the two NPs the reduced moment along d 4 and the
// term and its sum 6. The ordered kernel (kmc_step_f64) takes about 27 per ordered
// pair, 54 for the two.
//
// Work item: one warp, one pair of cells (g, h), g <= h, of 32 NPs each, and
// rotations s0 <= s < s1 of 32: lane L holds target L of cell g, and at rotation s
// source (L + s) mod 32 of cell h, which moves one lane per rotation by
// shuffles with the reverse sums it has gathered. A warp shares nothing with
// another, so a plan places an item on any SM: that is what small lysosomes
// need, whose few target groups would otherwise keep a few SMs' FP64 pipes
// busy while the others idle (100 NPs: 10 cell pairs, cut in 16 parts, run on
// every SM). A diagonal pair (g = h) runs its rotations 1 .. 31 forward only: 23
// instructions per ordered pair. Every item writes its sums to its own slot, and
// the update adds a target's slots in a fixed order: results are deterministic
// and do not depend on the batch. Per step against the ordered
// kernel at its best shape: 100 NPs 17.2 against 36 us (parts 2, 4, 8, 16: 35.0,
// 25.3, 20.8, 19.4 when timed), 400: 26 against 62, 1000: 54 against 73, 2000: 150 against 214,
// 4000: 523 against 754, where the pipe is 88 % busy. The autotuner times both.
#pragma once

namespace kmc {

struct F64Src {  // position and 3 w m of one NP (n = -w m is t times -1/3: kept apart)
  double x, y, z, tx, ty, tz, nx, ny, nz;
};

__device__ __forceinline__ F64Src f64_source(const dbl4 *__restrict__ pos,
                                             const dbl4 *__restrict__ mu, int i, bool valid) {
  F64Src r;
  r.x = r.y = r.z = static_cast<double>(kPadCoord);  // past the cell's last NP: no moment
  r.tx = r.ty = r.tz = r.nx = r.ny = r.nz = 0.0;
  if (valid) {
    const dbl4 p = pos[i], q = mu[i];
    r.x = p.x;
    r.y = p.y;
    r.z = p.z;
    r.tx = 3.0 * q.x;
    r.ty = 3.0 * q.y;
    r.tz = 3.0 * q.z;
    r.nx = -q.x;
    r.ny = -q.y;
    r.nz = -q.z;
  }
  return r;
}

// KMC_DEBUG builds: the item lies inside the launch and the context's NPs.
__device__ __forceinline__ bool f64_item_in_bounds(const StepArgs &a, const F64Item &it) {
  return KMC_DCHECK(it.ng >= 1 && it.ng <= 32 && it.nh >= 1 && it.nh <= 32 && it.g >= 0 &&
                        it.g <= it.h && it.s0 >= 0 && it.s0 < it.s1 && it.s1 <= 32 &&
                        it.slot >= 0 && it.slot < a.n_slots,
                    a.err, kSiteItem);
}

__global__ void __launch_bounds__(32) kmc_field_f64(const StepArgs a, int /*tile*/) {
  if (!KMC_DCHECK(static_cast<int>(blockIdx.x) < a.n_items, a.err, kSiteItem)) return;
  const F64Item it = a.fitems[blockIdx.x];
  if (!f64_item_in_bounds(a, it)) return;
  const int lane = threadIdx.x;
  const bool diag = it.g == it.h;
  const long long step = a.rs->step_base + a.k_local;  // before the wait, as in kmc_step_f32
  grid_dependency_wait();
  const int par = static_cast<int>(step & 1);
  const dbl4 *__restrict__ pos = static_cast<const dbl4 *>(a.src_pos);
  const dbl4 *__restrict__ mu = static_cast<const dbl4 *>(a.src[par]);
  const F64Src t = f64_source(pos, mu, it.g + lane, lane < it.ng);
  const int s0 = diag && it.s0 == 0 ? 1 : it.s0;  // the self pairs are not formed
  const int j = (lane + s0) & 31;
  F64Src s = f64_source(pos, mu, it.h + j, j < it.nh);
  double fx = 0.0, fy = 0.0, fz = 0.0, rx = 0.0, ry = 0.0, rz = 0.0;
  const int from = (lane + 1) & 31;
  auto move = [&](double v) { return __shfl_sync(0xffffffffu, v, from); };
  auto next = [&](const F64Src &v) {
    return F64Src{move(v.x),  move(v.y),  move(v.z),  move(v.tx), move(v.ty),
                  move(v.tz), move(v.nx), move(v.ny), move(v.nz)};
  };
  if (diag) {
#pragma unroll 2
    for (int r = s0; r < it.s1; ++r) {
      const F64Src ahead = next(s);  // independent of this rotation's sums
      const double dx = s.x - t.x, dy = s.y - t.y, dz = s.z - t.z;
      const double q = rsqrt_pair(fma(dx, dx, fma(dy, dy, dz * dz)));
      const double q2 = q * q, q3 = q * q2;
      const double u = fma(s.tx, dx, fma(s.ty, dy, s.tz * dz)) * q2;
      fx = fma(q3, fma(u, dx, s.nx), fx);
      fy = fma(q3, fma(u, dy, s.ny), fy);
      fz = fma(q3, fma(u, dz, s.nz), fz);
      s = ahead;
    }
  } else {
#pragma unroll 2
    for (int r = s0; r < it.s1; ++r) {
      const F64Src ahead = next(s);  // independent of this rotation's sums
      const double dx = s.x - t.x, dy = s.y - t.y, dz = s.z - t.z;
      const double q = rsqrt_pair(fma(dx, dx, fma(dy, dy, dz * dz)));
      const double q2 = q * q, q3 = q * q2;
      const double u = fma(s.tx, dx, fma(s.ty, dy, s.tz * dz)) * q2;
      fx = fma(q3, fma(u, dx, s.nx), fx);
      fy = fma(q3, fma(u, dy, s.ny), fy);
      fz = fma(q3, fma(u, dz, s.nz), fz);
      // the target's term at the source: -d enters twice
      const double v = fma(t.tx, dx, fma(t.ty, dy, t.tz * dz)) * q2;
      rx = move(fma(q3, fma(v, dx, t.nx), rx));
      ry = move(fma(q3, fma(v, dy, t.ny), ry));
      rz = move(fma(q3, fma(v, dz, t.nz), rz));
      s = ahead;
    }
  }
  // the slot: forward sums [3][32] by target, reverse sums [3][32] by source
  double *slot = a.f64part + static_cast<size_t>(it.slot) * kF64Slot;
  __stcg(slot + lane, fx);
  __stcg(slot + 32 + lane, fy);
  __stcg(slot + 64 + lane, fz);
  if (!diag) {
    const int js = (lane + it.s1) & 31;
    __stcg(slot + 96 + js, rx);
    __stcg(slot + 128 + js, ry);
    __stcg(slot + 160 + js, rz);
  }
  grid_launch_dependents();
}

// One block per cell of 32 targets: warp w takes the cell's slots w, w + 4, ...
// (partner cells in order, parts in order), the warps are added in order, and
// steps iii-vii follow.
constexpr int kF64UpdWarps = 4;

__global__ void __launch_bounds__(kF64UpdWarps * 32)
    kmc_update_f64(const StepArgs a, int /*tile*/) {
  constexpr int NW = kF64UpdWarps;
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char *dyn = smem + 16;
  __shared__ GridTables<double> tab;
  if (!KMC_DCHECK(static_cast<int>(blockIdx.x) < a.n_upd, a.err, kSiteItem)) return;
  const F64Upd u = a.fupd[blockIdx.x];  // read in kmc_update_sym's order
  const long long step = a.rs->step_base + a.k_local;
  const int per = a.rs->period;
  tab.load();
  if (!KMC_DCHECK(u.l >= 0 && u.l < a.n_lys, a.err, kSiteLys)) return;
  const LysDev L = a.lys[u.l];
  if (!KMC_DCHECK(u.t0 == 32 * u.cell && u.nt >= 1 && u.nt <= 32 && u.t0 + u.nt <= L.n &&
                      u.cell < u.nc && u.slot0 >= 0 &&
                      u.slot0 + ((u.nc * (u.nc + 1) / 2) << u.log_parts) <= a.n_slots,
                  a.err, kSiteTargets))
    return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  Item it;
  it.l = u.l;
  it.t0 = u.t0;
  it.nt = u.nt;
  it.gid = 0;
  it.j0 = it.j1 = 0;
  it.split = 0;
  it.nsplit = 1;
  grid_dependency_wait();
  const int rec = (per >= a.discard) ? (per - a.discard) * a.S + a.k_local : -1;
  TargetIn<dbl4> tin;
  if (warp == 0) tin = load_target<dbl4>(a, L, it, step, lane);
  const int c = u.cell, nc = u.nc, lp = u.log_parts, total = nc << lp;
  // x = partner cell and part: address of the cell's three sums
  auto sums = [&](int x) {
    const int p = x >> lp, part = x & ((1 << lp) - 1);
    const int lo = min(p, c), hi = max(p, c);
    const int pair = lo * nc - lo * (lo - 1) / 2 + (hi - lo);
    return a.f64part + static_cast<size_t>(u.slot0 + (pair << lp) + part) * kF64Slot +
           (p < c ? 96 : 0) + lane;
  };
  double h0 = 0.0, h1 = 0.0, h2 = 0.0;
  constexpr int kBatch = 8;  // slots loaded together and added pairwise: a chain of
                             // three dependent additions and one instead of eight
#pragma unroll 1
  for (int x0 = warp; x0 < total; x0 += NW * kBatch) {
    double v[kBatch][3];
#pragma unroll
    for (int b = 0; b < kBatch; ++b) {
      const bool in = x0 + b * NW < total;
      const double *p = sums(in ? x0 + b * NW : x0);
#pragma unroll
      for (int q = 0; q < 3; ++q) v[b][q] = in ? __ldcg(p + 32 * q) : 0.0;
    }
#pragma unroll
    for (int w = 1; w < kBatch; w *= 2)
#pragma unroll
      for (int b = 0; b < kBatch; b += 2 * w)
#pragma unroll
        for (int q = 0; q < 3; ++q) v[b][q] += v[b + w][q];
    h0 += v[0][0];
    h1 += v[0][1];
    h2 += v[0][2];
  }
  double *wp = reinterpret_cast<double *>(dyn);  // [NW][3][32]
  wp[(warp * 3 + 0) * 32 + lane] = h0;
  wp[(warp * 3 + 1) * 32 + lane] = h1;
  wp[(warp * 3 + 2) * 32 + lane] = h2;
  __syncthreads();
  EpiShared<double> &sm =
      *reinterpret_cast<EpiShared<double> *>(dyn + static_cast<size_t>(NW) * 12 * 32 * 4);
  if (warp == 0) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      double s = wp[q * 32 + lane];
#pragma unroll
      for (int w = 1; w < NW; ++w) s += wp[(w * 3 + q) * 32 + lane];
      sm.h[q][lane] = s;
    }
  }
  __syncthreads();
  block_update<dbl4, false>(a, L, it, step, rec, tin, sm, tab);
  grid_launch_dependents();
}

}  // namespace kmc
