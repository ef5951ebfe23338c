// kmc_local.cu -- local volume concentration phi_N (Eq. 8, Sec. III.5) on the
// device: for every NP i of one lysosome, r_N = distance to its N-th nearest
// neighbour and phi_N,i = 3 N V_i / (4 pi r_N^3).
//
// Squared distances are formed as (dx^2 + dy^2) + dz^2 without contraction, the
// order the oracle uses, and r_N^2 is the N-th smallest of them, whatever the way to
// it: phi does not depend on which of the two kernels below ran, bit for bit.
//
// Grid search (kPhiGridMin NPs and more). The NPs are binned into cubic cells of
// about half the expected r_N and sorted by cell; a warp takes one target and the
// block of 5 x 5 x 5 cells about its own, each lane a row of cells (contiguous in
// the sorted order), and widens the block until it provably holds the N nearest.
// FP32 squared distances select: the N-th smallest, T, by bisection on its bits,
// then the pairs within the error band about T (usually one) are formed in FP64
// and the exact order statistic is taken among them. About 5 N candidates per
// target instead of n: bound by the warps' instructions, not by memory (the
// positions stay in L2). The call,
// with its copies and host work, against all pairs: 50 000 NPs (N = 20) 0.365
// against 55.7 ms, of which the search takes 0.146 ms; 5000 NPs 95 us against 6.3
// ms; 200 NPs 70 against 445 us, so it serves all but the smallest sizes. At 50 000
// and N = 64 0.59 ms against 266.
//
// All pairs (fewer NPs; no device memory for the grid; NPs so unevenly spread that
// a cell holds more than kPhiMaxCell; coordinates outside FP32's range): one thread
// per target keeps the N smallest squared FP64 distances seen so far in ascending order. FP32 copies of
// the source positions are staged through shared memory tile by tile, and an
// FP32 pre-screen skips a pair whose FP32 squared distance exceeds the current
// N-th by more than a bound on the FP32 error.
//
// FP32 error: with coordinates of magnitude at most rmax (converted to FP32 with
// error <= u rmax, u = 2^-24), the FP32 squared distance errs by at most
// 4 sqrt(3) u rmax D + 12 u^2 rmax^2 + 5 u D^2; the margin used is
// 64 u (rmax D + D^2 + u rmax^2), over five times that.
#include <cuda_runtime.h>
#include <math.h>

#include "kmc_local.h"

namespace kmc {

namespace {

// one warp per block: many small blocks spread the targets evenly over the SMs
// (50 000 NPs, before the FP32 pre-screen: 46.9 ms against 50.9 ms with
// 128-thread blocks; splitting a target's sources over 4 warps was slower,
// since each warp's threshold then tightens on a quarter of them)
constexpr int kPhiThreads = 32;
constexpr int kPhiTile = 512;

// Grid search: smallest n, largest cell, warps per block (a warp keeps up to
// kPhiCand candidates in shared memory, a template argument; more are read again
// from global memory)
constexpr int kPhiGridMin = 8;
constexpr int kPhiMaxCell = 32;
constexpr int kPhiWarps = 4;

struct PhiGrid {
  float lox, loy, loz;  // corner of the box
  float s, inv_s;       // cell edge and its inverse
  float slack;          // bound on the rounding of a cell boundary
  int nx, ny, nz;
};

__device__ __forceinline__ int phi_cell(float x, float lo, float inv_s, int n) {
  return min(max(static_cast<int>((x - lo) * inv_s), 0), n - 1);
}

__device__ __forceinline__ float screen_limit(double thr, double rmax) {
  if (!(thr < INFINITY)) return INFINITY;
  const double u = 0x1.0p-24;
  return static_cast<float>(thr + 64.0 * u * (rmax * sqrt(thr) + thr + u * rmax * rmax));
}

// FP32 copy of the positions, made once per call.
__global__ void positions_f32_kernel(const dbl4 *__restrict__ pos, int n, float4 *__restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n)
    out[i] = make_float4(static_cast<float>(pos[i].x), static_cast<float>(pos[i].y),
                         static_cast<float>(pos[i].z), 0.0f);
}

__global__ void __launch_bounds__(kPhiThreads)
    local_concentration_kernel(const dbl4 *__restrict__ pos, const float4 *__restrict__ posf,
                               int n, int N, double rmax, const int *__restrict__ max_cell,
                               double *__restrict__ phi) {
  if (max_cell && *max_cell <= kPhiMaxCell) return;  // the grid search has the answer
  __shared__ float sx[kPhiTile], sy[kPhiTile], sz[kPhiTile];
  const int i = blockIdx.x * kPhiThreads + threadIdx.x;
  const bool active = i < n;
  const dbl4 p = pos[active ? i : 0];
  const float4 pf = posf[active ? i : 0];
  double best[kPhiMaxN];
  for (int q = 0; q < N; ++q) best[q] = INFINITY;
  double thr = INFINITY;  // best[N - 1]
  float lim = INFINITY;   // FP32 squared distances above it cannot enter the list
  for (int t0 = 0; t0 < n; t0 += kPhiTile) {
    const int cnt = min(kPhiTile, n - t0);
    __syncthreads();
    for (int j = threadIdx.x; j < cnt; j += kPhiThreads) {
      const float4 s = posf[t0 + j];
      sx[j] = s.x;
      sy[j] = s.y;
      sz[j] = s.z;
    }
    __syncthreads();
    if (!active) continue;
    for (int j = 0; j < cnt; ++j) {
      const float dxf = sx[j] - pf.x, dyf = sy[j] - pf.y, dzf = sz[j] - pf.z;
      if (fmaf(dzf, dzf, fmaf(dyf, dyf, dxf * dxf)) > lim) continue;
      // a pair that could enter the list: its distance as the oracle forms it
      const dbl4 s = pos[t0 + j];
      const double dx = __dsub_rn(s.x, p.x);
      const double dy = __dsub_rn(s.y, p.y);
      const double dz = __dsub_rn(s.z, p.z);
      const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
      if (d2 < thr && t0 + j != i) {
        int k = N - 1;
        while (k > 0 && best[k - 1] > d2) {
          best[k] = best[k - 1];
          --k;
        }
        best[k] = d2;
        thr = best[N - 1];
        lim = screen_limit(thr, rmax);
      }
    }
  }
  if (active) {
    const double r = sqrt(thr);
    phi[i] = (3.0 * static_cast<double>(N) * p.w) / (r * r * r);
  }
}

// FP32 copies, each NP's cell and its place within it (atomic: the order inside a
// cell varies, the result does not).
__global__ void phi_bin_kernel(const dbl4 *__restrict__ pos, int n, PhiGrid g,
                               float4 *__restrict__ posf, int *__restrict__ cell,
                               int *__restrict__ rank, int *__restrict__ count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float x = static_cast<float>(pos[i].x), y = static_cast<float>(pos[i].y),
              z = static_cast<float>(pos[i].z);
  posf[i] = make_float4(x, y, z, __int_as_float(i));
  const int c = (phi_cell(z, g.loz, g.inv_s, g.nz) * g.ny + phi_cell(y, g.loy, g.inv_s, g.ny)) *
                    g.nx + phi_cell(x, g.lox, g.inv_s, g.nx);
  cell[i] = c;
  rank[i] = atomicAdd(&count[c], 1);
}

// One block: count[0 .. cells) (padded with zeros to a multiple of 8192) to
// exclusive prefix sums in place, start[cells] = n, and the largest count.
__global__ void __launch_bounds__(1024) phi_scan_kernel(int *__restrict__ count, int padded,
                                                        int *__restrict__ max_cell) {
  __shared__ int s_sum[32], s_max[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int base = 0, big = 0;
  int4 *v = reinterpret_cast<int4 *>(count) + 2 * threadIdx.x;
  int4 a = v[0], b = v[1];
  for (int t0 = 0; t0 < padded / 4; t0 += 2048) {
    int4 an = a, bn = b;
    if (t0 + 2048 < padded / 4) {  // the next tile's loads ahead of this one's sums
      an = v[t0 + 2048];
      bn = v[t0 + 2049];
    }
    big = max(big, max(max(max(a.x, a.y), max(a.z, a.w)), max(max(b.x, b.y), max(b.z, b.w))));
    const int own = a.x + a.y + a.z + a.w + b.x + b.y + b.z + b.w;
    int inc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    if (lane == 31) s_sum[warp] = inc;
    __syncthreads();
    int sums = s_sum[lane];  // every warp scans the warps' sums
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, sums, o);
      if (lane >= o) sums += x;
    }
    const int before = __shfl_sync(0xffffffffu, sums, warp == 0 ? 0 : warp - 1);
    int run = base + (warp == 0 ? 0 : before) + inc - own;
    base += __shfl_sync(0xffffffffu, sums, 31);
    int4 c, d;
    c.x = run;
    c.y = run += a.x;
    c.z = run += a.y;
    c.w = run += a.z;
    d.x = run += a.w;
    d.y = run += b.x;
    d.z = run += b.y;
    d.w = run += b.z;
    v[t0] = c;
    v[t0 + 1] = d;
    a = an;
    b = bn;
    __syncthreads();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) big = max(big, __shfl_xor_sync(0xffffffffu, big, o));
  if (lane == 0) s_max[warp] = big;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 32; ++w) big = max(big, s_max[w]);
    *max_cell = big;
  }
}

__global__ void phi_scatter_kernel(const float4 *__restrict__ posf, int n,
                                   const int *__restrict__ cell, const int *__restrict__ rank,
                                   const int *__restrict__ start, float4 *__restrict__ sorted) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) sorted[start[cell[i]] + rank[i]] = posf[i];
}

// The squared distance of the definition, as the oracle forms it.
__device__ __forceinline__ double phi_d2(const dbl4 &p, const dbl4 &s) {
  const double dx = __dsub_rn(s.x, p.x);
  const double dy = __dsub_rn(s.y, p.y);
  const double dz = __dsub_rn(s.z, p.z);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// One warp per target (in cell order): out[i] = r_N^2. FP64 instructions issue at
// 1/64 of the FP32 rate whether one lane needs them or 32, so a target's warp
// forms only the band's distances in FP64; r_N^2 becomes phi in phi_finish_kernel.
template <int kPhiCand>
__global__ void __launch_bounds__(kPhiWarps * 32)
    phi_grid_kernel(const dbl4 *__restrict__ pos, const float4 *__restrict__ sorted, int n,
                    int N, float rmax, PhiGrid g, const int *__restrict__ start,
                    const int *__restrict__ max_cell, double *__restrict__ out) {
  if (*max_cell > kPhiMaxCell) return;  // the all-pairs kernel takes it
  __shared__ float s_d[kPhiWarps][kPhiCand];
  __shared__ int s_j[kPhiWarps][kPhiCand];
  __shared__ int s_band[kPhiWarps][32];
  constexpr unsigned kAll = 0xffffffffu;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * kPhiWarps + warp;
  if (k >= n) return;
  const float4 t = sorted[k];
  const int cx = phi_cell(t.x, g.lox, g.inv_s, g.nx), cy = phi_cell(t.y, g.loy, g.inv_s, g.ny),
            cz = phi_cell(t.z, g.loz, g.inv_s, g.nz);
  float *cd = s_d[warp];
  int *cj = s_j[warp];
  int x0, x1, y0, y1, z0, z1;
  // every other NP of the block: f(valid, FP32 squared distance, place in sorted),
  // the warp together, lane by lane a row of cells each
  auto each = [&](auto f) {
    const int wy = y1 - y0 + 1, rows = wy * (z1 - z0 + 1);
    for (int r0 = 0; r0 < rows; r0 += 32) {
      const int r = r0 + lane;
      int j = 0, je = 0;
      if (r < rows) {
        const int row = ((z0 + r / wy) * g.ny + y0 + r % wy) * g.nx;
        j = start[row + x0];
        je = start[row + x1 + 1];
      }
      while (__any_sync(kAll, j < je)) {
        const bool in = j < je;
        const float4 s = in ? sorted[j] : t;
        const float dx = s.x - t.x, dy = s.y - t.y, dz = s.z - t.z;
        f(in && j != k, fmaf(dz, dz, fmaf(dy, dy, dx * dx)), j);
        ++j;
      }
    }
  };
  int m = 0;  // candidates
  for (int R = 2;; ++R) {
    x0 = max(cx - R, 0);
    x1 = min(cx + R, g.nx - 1);
    y0 = max(cy - R, 0);
    y1 = min(cy + R, g.ny - 1);
    z0 = max(cz - R, 0);
    z1 = min(cz + R, g.nz - 1);
    // every NP nearer than `reach` lies in the block: sides at the box's faces
    // have nothing beyond them
    float reach = INFINITY;
    if (x0 > 0) reach = fminf(reach, t.x - (g.lox + x0 * g.s));
    if (y0 > 0) reach = fminf(reach, t.y - (g.loy + y0 * g.s));
    if (z0 > 0) reach = fminf(reach, t.z - (g.loz + z0 * g.s));
    if (x1 < g.nx - 1) reach = fminf(reach, g.lox + (x1 + 1) * g.s - t.x);
    if (y1 < g.ny - 1) reach = fminf(reach, g.loy + (y1 + 1) * g.s - t.y);
    if (z1 < g.nz - 1) reach = fminf(reach, g.loz + (z1 + 1) * g.s - t.z);
    const bool whole = !(reach < INFINITY);
    reach = fmaxf(reach - g.slack, 0.0f);
    const float reach2 = whole ? INFINITY : reach * reach;
    m = 0;
    int near = 0;
    each([&](bool ok, float d, int j) {
      const unsigned mask = __ballot_sync(kAll, ok);
      const int at = m + __popc(mask & ((1u << lane) - 1));
      if (ok && at < kPhiCand) {
        cd[at] = d;
        cj[at] = j;
      }
      m += __popc(mask);
      near += __popc(__ballot_sync(kAll, ok && d <= reach2));
    });
    if (whole || near >= N) break;
  }
  __syncwarp();
  const bool kept = m <= kPhiCand;
  auto cand = [&](auto f) {  // the candidates: f(valid, squared distance, place)
    if (!kept) {
      each(f);
      return;
    }
    for (int q0 = 0; q0 < m; q0 += 32) {
      const int q = q0 + lane;
      const bool ok = q < m;
      f(ok, ok ? cd[q] : 0.0f, ok ? cj[q] : 0);
    }
  };
  // T = the N-th smallest FP32 squared distance (non-negative floats order as
  // their bits): the least value that N candidates do not exceed
  unsigned lo = 0, hi = 0x7f800000u;
  while (lo < hi) {
    const unsigned mid = (lo + hi) >> 1;
    int c = 0;
    cand([&](bool ok, float d, int) { c += ok && __float_as_uint(d) <= mid; });
    c = __reduce_add_sync(kAll, c);
    if (c >= N)
      hi = mid;
    else
      lo = mid + 1;
  }
  const float T = __uint_as_float(lo);
  const float u = 0x1.0p-24f;
  const float margin = 129.0f * u * (rmax * sqrtf(T) + T + u * rmax * rmax);
  const float below = T - margin - u * T, above = T + margin + u * T;
  // pairs under the band are nearer than the N-th for certain, pairs above it
  // farther; the N-th is the rank-th smallest of the band in FP64
  int rank = 0, band = 0;
  cand([&](bool ok, float d, int) {
    rank += __popc(__ballot_sync(kAll, ok && d < below));
    band += __popc(__ballot_sync(kAll, ok && d >= below && d <= above));
  });
  rank = N - rank;
  const dbl4 p = pos[__float_as_int(t.w)];
  unsigned long long l = 0, h = 0x7ff0000000000000ull;
  if (band <= 32) {
    // one pair per lane, by a list of the warp's
    int at0 = 0;
    cand([&](bool ok, float d, int j) {
      const bool in = ok && d >= below && d <= above;
      const unsigned mask = __ballot_sync(kAll, in);
      if (in) s_band[warp][at0 + __popc(mask & ((1u << lane) - 1))] = j;
      at0 += __popc(mask);
    });
    __syncwarp();
    const int mine = lane < band ? s_band[warp][lane] : -1;
    double d2 = INFINITY;
    if (mine >= 0) d2 = phi_d2(p, pos[__float_as_int(sorted[mine].w)]);
    // non-negative doubles order as their bits
    const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(d2));
    int less = 0, same = 0;
    for (int b = 0; b < band; ++b) {
      const unsigned long long v = __shfl_sync(kAll, bits, b);
      less += v < bits;
      same += v == bits;
    }
    const unsigned hit = __ballot_sync(kAll, lane < band && less < rank && rank <= less + same);
    h = __shfl_sync(kAll, bits, hit ? __ffs(hit) - 1 : 0);
  } else {
    // a lattice's many equal distances: bisection on the FP64 bits
    while (l < h) {
      const unsigned long long mid = (l + h) >> 1;
      int c = 0;
      cand([&](bool ok, float d, int j) {
        if (ok && d >= below && d <= above)
          c += static_cast<unsigned long long>(__double_as_longlong(
                   phi_d2(p, pos[__float_as_int(sorted[j].w)]))) <= mid;
      });
      c = __reduce_add_sync(kAll, c);
      if (c >= rank)
        h = mid;
      else
        l = mid + 1;
    }
  }
  if (lane == 0) out[__float_as_int(t.w)] = __longlong_as_double(static_cast<long long>(h));
}

__global__ void phi_finish_kernel(const dbl4 *__restrict__ pos, int n, int N,
                                  const int *__restrict__ max_cell, double *__restrict__ phi) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || *max_cell > kPhiMaxCell) return;
  const double r = sqrt(phi[i]);
  phi[i] = (3.0 * static_cast<double>(N) * pos[i].w) / (r * r * r);
}

// The grid for n NPs in the box [lo, hi] and rank N: cells of about half the r_N
// of a uniform density (1.5 times that of the box, which a ball fills by half),
// at most 2 n + 64 of them. False where FP32 coordinates will not do.
bool phi_grid(int n, int N, double rmax, const double *lo, const double *hi, PhiGrid *g) {
  double ext[3], big = 0.0;
  for (int q = 0; q < 3; ++q) {
    ext[q] = hi[q] - lo[q];
    big = ext[q] > big ? ext[q] : big;
  }
  if (!(big > 1e-12) || !(rmax < 1e12)) return false;
  double vol = 1.0;
  for (int q = 0; q < 3; ++q) vol *= ext[q] > 1e-3 * big ? ext[q] : 1e-3 * big;
  double s = 0.54 * cbrt(3.0 * N * vol / (4.0 * 3.14159265358979323846 * 1.5 * n));
  double c[3];
  for (;;) {  // widen the cells until their number is in bounds
    for (int q = 0; q < 3; ++q) c[q] = floor(ext[q] / s) + 1.0;
    if (c[0] * c[1] * c[2] <= 2.0 * n + 64.0) break;
    s *= 1.1;
  }
  g->lox = static_cast<float>(lo[0]);
  g->loy = static_cast<float>(lo[1]);
  g->loz = static_cast<float>(lo[2]);
  g->s = static_cast<float>(s);
  g->inv_s = static_cast<float>(1.0 / s);
  // boundaries and coordinates are FP32 values and products of magnitude up to
  // rmax + big: 64 roundings' worth
  g->slack = static_cast<float>(64.0 * 0x1.0p-24 * (rmax + big));
  g->nx = static_cast<int>(c[0]);
  g->ny = static_cast<int>(c[1]);
  g->nz = static_cast<int>(c[2]);
  return true;
}

int phi_padded_cells(int cells) { return (cells + 1 + 8191) / 8192 * 8192; }

}  // namespace

size_t local_concentration_scratch(int n) {
  // [n] float4 sorted, [n] cell, [n] rank, the cells' starts, the largest count
  return n < kPhiGridMin ? 0
                         : static_cast<size_t>(n) * (sizeof(float4) + 2 * sizeof(int)) +
                               sizeof(int) * (static_cast<size_t>(phi_padded_cells(2 * n + 64)) + 4);
}

cudaError_t launch_local_concentration(const dbl4 *pos, int n, int N, double rmax,
                                       const double *lo, const double *hi, float4 *posf,
                                       void *scratch, double *phi, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  PhiGrid g;
  const int *max_cell = nullptr;
  if (scratch && n >= kPhiGridMin && n <= (1 << 28) && phi_grid(n, N, rmax, lo, hi, &g)) {
    float4 *sorted = static_cast<float4 *>(scratch);
    const int padded = phi_padded_cells(g.nx * g.ny * g.nz);
    int *start = reinterpret_cast<int *>(sorted + n);  // 16-byte aligned
    int *most = start + padded, *cell = most + 4, *rank = cell + n;
    cudaError_t e = cudaMemsetAsync(start, 0, sizeof(int) * padded, st);
    if (e != cudaSuccess) return e;
    phi_bin_kernel<<<(n + 255) / 256, 256, 0, st>>>(pos, n, g, posf, cell, rank, start);
    phi_scan_kernel<<<1, 1024, 0, st>>>(start, padded, most);
    phi_scatter_kernel<<<(n + 255) / 256, 256, 0, st>>>(posf, n, cell, rank, start, sorted);
    const int blocks = (n + kPhiWarps - 1) / kPhiWarps;
    const float rm = static_cast<float>(rmax) * 1.000001f;
    if (N <= 24)
      phi_grid_kernel<512><<<blocks, kPhiWarps * 32, 0, st>>>(pos, sorted, n, N, rm, g, start,
                                                              most, phi);
    else
      phi_grid_kernel<1280><<<blocks, kPhiWarps * 32, 0, st>>>(pos, sorted, n, N, rm, g, start,
                                                               most, phi);
    phi_finish_kernel<<<(n + 255) / 256, 256, 0, st>>>(pos, n, N, most, phi);
    max_cell = most;
  } else {
    positions_f32_kernel<<<(n + 255) / 256, 256, 0, st>>>(pos, n, posf);
  }
  const int blocks = (n + kPhiThreads - 1) / kPhiThreads;
  local_concentration_kernel<<<blocks, kPhiThreads, 0, st>>>(pos, posf, n, N, rmax, max_cell, phi);
  return cudaGetLastError();
}

}  // namespace kmc
