// kmc_cluster.cuh -- a whole field period of small lysosomes (up to 512 NPs) in
// one launch, FP32-mixed: each lysosome is one thread-block cluster, which keeps
// its source records in shared memory. Included only by kmc_step.cu, which owns
// the pair loop and the parts of the update.
//
// A step of a small lysosome is latency: 100 NPs took 7.0 us per step, of which the
// pair sums are 0.3 us and steps iii-vii about 3.5; the rest was the launch
// boundary, the loads of the targets' state and of the sources behind it, and
// their way back through the L2. Here block r of the cluster keeps targets
// 32 r .. 32 r + 31 in registers and a copy of all source records (positions and
// moments, double buffered) in shared memory for the whole period. After a step it
// writes its new moments into every block's next buffer (distributed shared
// memory), and one cluster barrier ends the step: a block can be one step ahead
// at most, so nobody reads the buffer that is being written. What is not on the way
// from one step's moments to the next is done by warps 1 to 3 while warp 0 adds the
// sums up and sets the working planes: the previous step's loop record and energy
// (FP64 chains of a thousand cycles) and this step's draw. Per step against
// the per-step launches: 100 NPs 4.7 against 6.9 us, 32: 4.3 against 6.5, 256: 6.0
// against 8.1, 512: 8.5 against 9.4; 32 lysosomes of 300 NPs 11 against 9.9 (their
// clusters exceed the SMs). The autotuner times both.
//
// Each target's sums are kmc_step_f32's at the same warps with all records in one
// tile: the same operations in the same order, so the same bits.
#pragma once

namespace kmc {

constexpr int kClusterMaxBlocks = 16;  // 512 NPs (above 8: the non-portable size)
constexpr int kClusterWarps = 8;

__device__ __forceinline__ void st_cluster(float *p, uint32_t rank, float v) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_addr(p)), "r"(rank));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(remote), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The pair loop of kmc_step_f32 over all records, the same operations in the same
// order. A copy of its own, inlined: as one more caller of pair_tile_f32 this
// kernel moved that function's schedule, and kmc_step_f32 ran 3 to 7 % slower.
template <int NW>
__device__ __forceinline__ AccF32 cluster_pairs(const ulonglong2 *__restrict__ sp, int cnt,
                                                int first, f2 X, f2 Y, f2 Z) {
  AccF32 acc;
  acc.x = acc.y = acc.z = 0ull;
#pragma unroll 4
  for (int r = first; r < cnt; r += NW) {
    ulonglong2 a, b, c, d;
    f2 e;
    load_record(sp, r, a, b, c, d, e);
    pair_record<true>(a, b, c, d, e, X, Y, Z, acc);
  }
  return acc;
}

// Dynamic shared memory: two buffers of source records.
constexpr size_t cluster_smem(int max_n) {
  return 2 * static_cast<size_t>((max_n + 1) / 2) * sizeof(SrcPair);
}

// Grid: n_lys clusters of `blocks` blocks; a.S steps from step_base. The cosine of
// step k is a.cosk[k], or a.cos_k without a table.
template <int NW>
__global__ void __launch_bounds__(NW * 32) kmc_cluster_f32(const StepArgs a, int blocks) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ GridTables<float> tab;
  __shared__ EpiShared<float> sm;
  __shared__ float s_wp[NW][3][32];
  __shared__ float s_m[3][kTargets];  // the step's new moments
  __shared__ double s_u[kTargets];    // its draws
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l = blockIdx.x / blocks, rank = blockIdx.x % blocks;
  const LysDev L = a.lys[l];
  const int nrec = (L.n + 1) / 2;
  SrcPair *buf[2] = {reinterpret_cast<SrcPair *>(smem),
                     reinterpret_cast<SrcPair *>(smem) + nrec};
  tab.load();
  const float4 *gpos = static_cast<const float4 *>(a.pos) + L.off;
  float4 *gm = static_cast<float4 *>(a.m) + L.off;
  for (int j = threadIdx.x; j < 2 * nrec; j += NW * 32) {
    float4 p = make_float4(kPadCoord, kPadCoord, kPadCoord, 0.f), m = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j < L.n) {
      p = gpos[j];
      m = gm[j];
    }
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      SrcPair &r = buf[b][j >> 1];
      const int h = j & 1;
      r.x[h] = p.x;
      r.y[h] = p.y;
      r.z[h] = p.z;
      set_source_moment(r, h, p.w, m.x, m.y, m.z);
    }
  }
  // this block's targets (none in the last blocks of a lysosome smaller than the
  // batch's largest: they only keep the barriers)
  const int t0 = rank * kTargets, nt = min(kTargets, L.n - t0);
  const bool mine = nt > 0;
  const int il = mine ? t0 + min(lane, nt - 1) : 0, i = L.off + il;
  const bool active = warp == 0 && lane < nt;
  const float4 pt = gpos[il];
  const f2 X = pk(pt.x, pt.x), Y = pk(pt.y, pt.y), Z = pk(pt.z, pt.z);
  const long long base = a.rs->step_base;
  const int per = a.rs->period;
  const bool record = per >= a.discard;
  float4 ax = make_float4(0.f, 0.f, 1.f, 0.f), m4 = ax;
  double beta = 0.0;
  // warp 1: V / sum V; warp 3: the energies, and m_z of the step before
  double vfrac = 0.0, eacc = 0.0;
  float mz_prev = 0.f;
  int count[kCntNonFinite + 1];  // the lane's counts of the period
#pragma unroll
  for (int q = 0; q <= kCntNonFinite; ++q) count[q] = 0;
  int bad = 0;
  if (warp == 0) {
    ax = static_cast<const float4 *>(a.axis)[i];
    m4 = gm[il];
    beta = a.beta[i];
    sm.k[lane] = static_cast<float>(L.k);
    sm.k2[lane] = 2.0f * static_cast<float>(L.k);
  }
  if (warp == 1 && lane < nt) vfrac = a.vfrac[i];
  if (warp == 3) {
    eacc = a.e_acc[i];
    mz_prev = gm[il].z;
  }
  // step k's loop record (warp 1) and energies (warp 3), from its new m_z
  auto records = [&](int k, double bext, float mz) {
    if (warp == 1) {
      double c = lane < nt ? vfrac * static_cast<double>(mz) : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
      if (lane == 0)
        atomicAdd(reinterpret_cast<unsigned long long *>(
                      &a.loop_m[static_cast<long long>(l) * a.n_rec + (per - a.discard) * a.S + k]),
                  static_cast<unsigned long long>(__double2ll_rn(c * kLoopScale)));
    } else if (warp == 3) {
      eacc += bext * (static_cast<double>(mz) - static_cast<double>(mz_prev));
      mz_prev = mz;
    }
  };
  __syncwarp();
  // every block's buffers are filled (and every block runs) before another one
  // writes into them
  cluster_arrive();
  cluster_wait();
  double cos_next = a.cosk ? a.cosk[0] : a.cos_k, bext_prev = 0.0;
  float mz_new = 0.f;  // warps 1 and 3: the last step's m_z
#pragma unroll 1
  for (int k = 0; k < a.S; ++k) {
    const double bext = L.bmax * cos_next;
    if (a.cosk && k + 1 < a.S) cos_next = a.cosk[k + 1];  // ahead of its use
    const SrcPair *src = buf[k & 1];
    if (mine) {
      const AccF32 acc = cluster_pairs<NW>(reinterpret_cast<const ulonglong2 *>(src), nrec, warp, X,
                                           Y, Z);
      s_wp[warp][0][lane] = hsum(acc.x);
      s_wp[warp][1][lane] = hsum(acc.y);
      s_wp[warp][2][lane] = hsum(acc.z);
      __syncthreads();
      TargetState<float> st;
      if (warp == 0) {
        float h[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float s = 0.f, e = 0.f;
#pragma unroll
          for (int w = 0; w < NW; ++w) neumaier_add(s, e, s_wp[w][c][lane]);
          h[c] = s + e;
          sm.h[c][lane] = h[c];
        }
        // Eq. 6: the dipolar field along the applied field at its two extremes
        if (record && active && (k == 0 || k == a.S / 2)) {
          double d = a.dh_acc[i];
          if (k == 0) d += static_cast<double>(h[2]);
          if (k == a.S / 2) d -= static_cast<double>(h[2]);
          a.dh_acc[i] = d;
        }
        st = setup_plane<float>(ax.x, ax.y, ax.z, m4.x, m4.y, m4.z, h[0], h[1],
                                h[2] + static_cast<float>(bext));
        sm.bc[lane] = st.bmag * st.cphi;
        sm.bs[lane] = st.bmag * st.sphi;
        sm.cnt[lane] = 0;
      } else if (warp == 2) {
        s_u[lane] = kmc_uniform(a.seed, base + k, il, l);
      } else if (record && k > 0) {
        records(k - 1, bext_prev, mz_new);
      }
      __syncthreads();
      segment_scan<float>(sm, tab, warp, NW, lane, nt);
      __syncthreads();
      const bool noisy = lane < nt && (sm.cnt[lane] > 4 || a.force_rescan);
      if (__any_sync(0xffffffffu, noisy)) {  // the same in every warp
        __syncthreads();
        if (warp == 0 && noisy) rescan_fp64(sm, lane);
        __syncthreads();
      }
      for (int x = threadIdx.x; x < 4 * nt; x += NW * 32) {
        const int t = x >> 2, q = x & 3, nb = min(sm.cnt[t], 4);
        if (q < nb) refine_bracket<float>(sm, tab, t, q, nb, a.err);
      }
      __syncthreads();
      if (warp == 0) {
        float sn, cn;
        const double u = s_u[lane];
        const Decision r = decide<float, true>(sm, min(lane, nt - 1), st, beta, L.lognu0t,
                                               L.t_zero != 0, u, a.debug != 0, sn, cn);
        const bool finite = isfinite(sm.h[0][lane]) && isfinite(sm.h[1][lane]) &&
                            isfinite(sm.h[2][lane]) && isfinite(r.dEa) && isfinite(r.dEb) &&
                            isfinite(r.P);
        if (finite) {
          m4.x = fmaf(cn, st.ax, sn * st.ex);
          m4.y = fmaf(cn, st.ay, sn * st.ey);
          m4.z = fmaf(cn, st.az, sn * st.ez);
        }
        s_m[0][lane] = m4.x;
        s_m[1][lane] = m4.y;
        s_m[2][lane] = m4.z;
        const bool jumped = finite && r.flipped;
        if (active) {
          count[kCntJumps] += jumped;
          count[kCntNear] += r.near;
          count[kCntOneMin] += r.nmin == 1;
          count[kCntFallback] += st.degenerate;
          count[kCntRescan] += noisy;
          count[kCntPolish] += r.polished;
          count[kCntNonFinite] += !finite;
          bad |= r.bad;
        }
        if (a.debug && active) {
          a.dbg.bdip[3 * i + 0] = static_cast<double>(sm.h[0][lane]);
          a.dbg.bdip[3 * i + 1] = static_cast<double>(sm.h[1][lane]);
          a.dbg.bdip[3 * i + 2] = static_cast<double>(sm.h[2][lane]);
          a.dbg.dE[2 * i + 0] = r.dEa;
          a.dbg.dE[2 * i + 1] = r.dEb;
          a.dbg.P[i] = r.P;
          a.dbg.u[i] = u;
          a.dbg.flags[i] = r.nmin | (jumped ? kFlagJumped : 0) | (r.near ? kFlagNear : 0) |
                           (st.degenerate ? kFlagFallback : 0) | (noisy ? kFlagRescan : 0) |
                           (r.polished ? kFlagPolish : 0) | (finite ? 0 : kFlagNonFinite);
        }
      }
      __syncthreads();
      mz_new = s_m[2][lane];
      // the new moments into every block's next buffer, a block per warp
      if (lane < nt) {
        SrcPair *next = buf[(k & 1) ^ 1] + (il >> 1);
        const int h = il & 1;
        SrcPair v;
        set_source_moment(v, 0, pt.w, s_m[0][lane], s_m[1][lane], s_m[2][lane]);
        for (int to = warp; to < blocks; to += NW) {
          st_cluster(&next->tx[h], to, v.tx[0]);
          st_cluster(&next->ty[h], to, v.ty[0]);
          st_cluster(&next->tz[h], to, v.tz[0]);
          st_cluster(&next->nx[h], to, v.nx[0]);
          st_cluster(&next->ny[h], to, v.ny[0]);
          st_cluster(&next->nz[h], to, v.nz[0]);
        }
      }
    }
    bext_prev = bext;
    __syncwarp();
    cluster_arrive();
    cluster_wait();
  }
  if (mine && record) records(a.S - 1, bext_prev, mz_new);
  if (warp == 3 && record && lane < nt) a.e_acc[i] = eacc;
  if (!mine || warp != 0) return;
  if (active) gm[il] = m4;
  unsigned long long *cn = a.counters + static_cast<long long>(kCounters) * l;
#pragma unroll
  for (int q = 0; q <= kCntNonFinite; ++q) {
    const unsigned total = __reduce_add_sync(0xffffffffu, static_cast<unsigned>(count[q]));
    if (lane == 0 && total) atomicAdd(cn + q, static_cast<unsigned long long>(total));
    if (q == kCntNonFinite && lane == 0 && total) atomicOr(a.err, kErrNonFinite);
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(a.err, kErrExtrema);
}

}  // namespace kmc
