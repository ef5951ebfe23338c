// kmc_regen.cuh -- sample regeneration between loops on the device (Sec. II.4).
// Included only by kmc_step.cu, which owns the Philox generator.
//
// Between loops the paper draws fresh easy axes and, around fixed mean
// positions (the nodes of a cubic lattice), fresh positions. One thread per NP
// draws from Philox4x32-10 with key (seed lo, seed hi) and counter
// (loop, 0x80000000 | sub, NP, lysosome); the top bit of word 1 keeps these
// counters apart from those of the kMC draws, whose word 1 is the high half of
// a step index below 2^31. Two 53-bit uniforms come from each call, made like
// the kMC draw from words (0, 1) and (2, 3).
//   axes (sub 0): uniform on the sphere, z = 1 - 2 u0, azimuth 2 pi u1;
//   positions: node + rho e, e uniform on the sphere from sub 1 and
//     rho = disorder * (first uniform of sub 2), uniform on [0, disorder];
//   random sequential addition: candidate c (NP slot of the counter = c) is
//     uniform in the ball of centres, direction from sub 3 and radius
//     Rb max(u0, u1, u2) from subs 4 and 5.
// The NP's arrays are then rewritten as creation builds them (unit axis,
// position in the lysosome's frame, moment along the axis with m_z >= 0).
#pragma once

namespace kmc {

__device__ __forceinline__ void regen_uniforms(unsigned long long seed, uint32_t loop,
                                               uint32_t sub, int np, int lys, double u[2]) {
  const uint4 w = philox4x32_10(
      make_uint4(loop, 0x80000000u | sub, static_cast<uint32_t>(np), static_cast<uint32_t>(lys)),
      make_uint2(static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32)));
  u[0] = static_cast<double>((static_cast<unsigned long long>(w.x) << 21) ^
                             static_cast<unsigned long long>(w.y >> 11)) * 0x1.0p-53;
  u[1] = static_cast<double>((static_cast<unsigned long long>(w.z) << 21) ^
                             static_cast<unsigned long long>(w.w >> 11)) * 0x1.0p-53;
}

// Uniform point on the unit sphere. Roundings are spelled out so that no
// product is fused into a subtraction: near the poles 1 - z^2 cancels, and a
// fused form would differ from the plain one by many ulps.
__device__ __forceinline__ void sphere_point(const double u[2], double &x, double &y, double &z) {
  z = __dsub_rn(1.0, __dmul_rn(2.0, u[0]));
  const double r2 = __dsub_rn(1.0, __dmul_rn(z, z));
  const double r = r2 > 0.0 ? sqrt(r2) : 0.0;
  double s, c;
  sincos(__dmul_rn(Prec<double>::two_pi, u[1]), &s, &c);
  x = __dmul_rn(r, c);
  y = __dmul_rn(r, s);
}

__global__ void kmc_regen_kernel(const RegenArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  const int g = a.off + i;
  double ax, ay, az;
  if (a.what & kRegenAxes) {
    double u[2];
    regen_uniforms(a.seed, a.loop, 0u, i, a.lys, u);
    sphere_point(u, ax, ay, az);
    const double an = sqrt(__dadd_rn(__dadd_rn(__dmul_rn(ax, ax), __dmul_rn(ay, ay)),
                                     __dmul_rn(az, az)));
    ax /= an;
    ay /= an;
    az /= an;
  } else if (a.fp32) {
    const float4 v = static_cast<const float4 *>(a.axis)[g];
    ax = v.x;
    ay = v.y;
    az = v.z;
  } else {
    const dbl4 v = static_cast<const dbl4 *>(a.axis)[g];
    ax = v.x;
    ay = v.y;
    az = v.z;
  }
  if (a.what & (kRegenPositions | kRegenGiven)) {
    double px, py, pz;
    if (a.what & kRegenPositions) {
      double u[2], v[2], ex, ey, ez;
      regen_uniforms(a.seed, a.loop, 1u, i, a.lys, u);
      regen_uniforms(a.seed, a.loop, 2u, i, a.lys, v);
      sphere_point(u, ex, ey, ez);
      const double rho = __dmul_rn(a.disorder, v[0]);
      px = __dadd_rn(a.nodes[3 * g], __dmul_rn(rho, ex));
      py = __dadd_rn(a.nodes[3 * g + 1], __dmul_rn(rho, ey));
      pz = __dadd_rn(a.nodes[3 * g + 2], __dmul_rn(rho, ez));
      a.pos_si[3 * g] = px;
      a.pos_si[3 * g + 1] = py;
      a.pos_si[3 * g + 2] = pz;
    } else {
      px = a.pos_si[3 * g];
      py = a.pos_si[3 * g + 1];
      pz = a.pos_si[3 * g + 2];
    }
    const double x = (px - a.cx) / a.len, y = (py - a.cy) / a.len, z = (pz - a.cz) / a.len;
    if (a.fp32) {
      float4 &p4 = static_cast<float4 *>(a.pos)[g];
      p4 = make_float4(static_cast<float>(x), static_cast<float>(y), static_cast<float>(z), p4.w);
      dbl4 &q4 = static_cast<dbl4 *>(a.pos64)[g];
      q4.x = x;
      q4.y = y;
      q4.z = z;
    } else {
      dbl4 &p4 = static_cast<dbl4 *>(a.pos)[g];
      p4.x = x;
      p4.y = y;
      p4.z = z;
    }
  }
  const double sgn = az >= 0.0 ? 1.0 : -1.0;
  if (a.fp32) {
    const float fx = static_cast<float>(ax), fy = static_cast<float>(ay), fz = static_cast<float>(az);
    if (a.what & kRegenAxes) static_cast<float4 *>(a.axis)[g] = make_float4(fx, fy, fz, 0.0f);
    const float fs = static_cast<float>(sgn);
    static_cast<float4 *>(a.m)[g] = make_float4(fs * fx, fs * fy, fs * fz, 0.0f);
  } else {
    dbl4 v;
    v.w = 0.0;
    if (a.what & kRegenAxes) {
      v.x = ax;
      v.y = ay;
      v.z = az;
      static_cast<dbl4 *>(a.axis)[g] = v;
    }
    v.x = sgn * ax;
    v.y = sgn * ay;
    v.z = sgn * az;
    static_cast<dbl4 *>(a.m)[g] = v;
  }
}

// Candidate c of the random sequential addition, about the lysosome centre.
__device__ __forceinline__ void rsa_candidate(double Rb, unsigned long long seed, uint32_t loop,
                                              long long c, int lys, double *p) {
  double u[2], v[2], w[2], ex, ey, ez;
  const int slot = static_cast<int>(static_cast<uint32_t>(c));
  regen_uniforms(seed, loop, 3u, slot, lys, u);
  regen_uniforms(seed, loop, 4u, slot, lys, v);
  regen_uniforms(seed, loop, 5u, slot, lys, w);
  sphere_point(u, ex, ey, ez);
  double x = v[0] > v[1] ? v[0] : v[1];
  if (w[0] > x) x = w[0];
  const double r = __dmul_rn(Rb, x);
  p[0] = __dmul_rn(r, ex);
  p[1] = __dmul_rn(r, ey);
  p[2] = __dmul_rn(r, ez);
}

// Squared distance, rounded as the definition reads it.
__device__ __forceinline__ double rsa_d2(const double *p, const double *q) {
  const double dx = __dsub_rn(p[0], q[0]), dy = __dsub_rn(p[1], q[1]), dz = __dsub_rn(p[2], q[2]);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// Spheres p (pf in FP32) and q closer than d. The FP32 squared distance settles
// the pair unless it falls within the margin [d2_lo, d2_hi] around d^2, which
// bounds its error for centres inside the ball; there the FP64 test of the
// definition decides.
__device__ __forceinline__ bool rsa_close(const RsaArgs &a, const double *p, const float4 &pf,
                                          const double *q, const float4 &qf) {
  const float dx = pf.x - qf.x, dy = pf.y - qf.y, dz = pf.z - qf.z;
  const float d2f = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
  return d2f < a.d2_lo || (d2f <= a.d2_hi && rsa_d2(p, q) < a.d2);
}

// Cubic cells of edge at least d over the ball's box: spheres closer than d lie
// in the same or in touching cells. Each cell heads a linked list of the kept
// spheres in it and one of the batch's candidates; the order inside a list
// varies, what is found in it does not.
__device__ __forceinline__ int3 rsa_cell(const RsaArgs &a, const double *p) {
  auto at = [&](double x) {
    return min(max(static_cast<int>((x + a.Rb) * a.inv_edge), 0), a.dim - 1);
  };
  return make_int3(at(p[0]), at(p[1]), at(p[2]));
}

// f(j) for every entry j of the lists about cell c, until f returns true.
template <typename F>
__device__ __forceinline__ bool rsa_around(const RsaArgs &a, const int3 &c, const int32_t *head,
                                           const int32_t *next, F f) {
  for (int z = max(c.z - 1, 0); z <= min(c.z + 1, a.dim - 1); ++z)
    for (int y = max(c.y - 1, 0); y <= min(c.y + 1, a.dim - 1); ++y)
      for (int x = max(c.x - 1, 0); x <= min(c.x + 1, a.dim - 1); ++x)
        for (int j = head[(z * a.dim + y) * a.dim + x]; j >= 0; j = next[j])
          if (f(j)) return true;
  return false;
}

__device__ __forceinline__ int rsa_index(const RsaArgs &a, const int3 &c) {
  return (c.z * a.dim + c.y) * a.dim + c.x;
}

// Candidate k of the batch: drawn, and checked against the spheres that earlier
// batches kept; if it clears them it joins its cell's list of candidates.
__global__ void rsa_candidates_kernel(const RsaArgs a) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.B) return;
  double p[3];
  rsa_candidate(a.Rb, a.seed, a.loop, a.c0 + k, a.lys, p);
  const float4 pf = make_float4(static_cast<float>(p[0]), static_cast<float>(p[1]),
                                static_cast<float>(p[2]), 0.0f);
  for (int q = 0; q < 3; ++q) a.cand[3 * k + q] = p[q];
  a.candf[k] = pf;
  const int3 c = rsa_cell(a, p);
  const bool clash = rsa_around(a, c, a.head_k, a.next_k, [&](int j) {
    return rsa_close(a, p, pf, a.pos + 3 * j, a.posf[j]);
  });
  a.clear[k] = clash ? 0 : 1;
  if (!clash) a.next_b[k] = atomicExch(a.head_b + rsa_index(a, c), k);
}

// The earlier candidates of the batch that candidate k clashes with (counted;
// the first kRsaMaxConf listed).
__global__ void rsa_conflicts_kernel(const RsaArgs a) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.B || !a.clear[k]) return;
  const double *p = a.cand + 3 * k;
  const float4 pf = a.candf[k];
  int n = 0;
  rsa_around(a, rsa_cell(a, p), a.head_b, a.next_b, [&](int j) {
    if (j < k && rsa_close(a, p, pf, a.cand + 3 * j, a.candf[j])) {
      if (n < kRsaMaxConf) a.conf[k * kRsaMaxConf + n] = j;
      ++n;
    }
    return false;
  });
  a.nconf[k] = n;
}

// The sequential rule over the batch, by one block: a candidate that cleared the
// earlier batches is kept unless one kept earlier in this batch lies closer
// than d. Its fate is known once those of its earlier conflicts are: in rounds,
// each decides every candidate whose conflicts are decided (the first undecided
// one always is), until none is left. The rounds follow chains of conflicts,
// a dozen or so, where a walk in candidate order took as many steps as
// candidates. The kept ones' places follow from a scan in candidate order.
__global__ void __launch_bounds__(1024) rsa_resolve_kernel(const RsaArgs a) {
  extern __shared__ unsigned char s_state[];  // per candidate: 0 undecided, 1 kept, 2 not
  __shared__ int s_sum[32];
  volatile unsigned char *state = s_state;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // bit i of todo: this thread's candidate threadIdx.x + 1024 i is undecided
  static_assert(kRsaMaxBatch <= 32 * 1024, "a thread's candidates are bits of one word");
  unsigned todo = 0;
  for (int i = 0, k = threadIdx.x; k < a.B; ++i, k += 1024) {
    const int st = !a.clear[k] ? 2 : (a.nconf[k] == 0 ? 1 : 0);
    state[k] = static_cast<unsigned char>(st);
    todo |= static_cast<unsigned>(st == 0) << i;
  }
  __syncthreads();
  for (;;) {
    for (unsigned left = todo; left;) {
      const int i = __ffs(left) - 1;
      left &= left - 1;
      const int k = threadIdx.x + 1024 * i;
      bool wait = false, out = false;
      auto meet = [&](int j) {
        const unsigned char s = state[j];
        out = out || s == 1;
        wait = wait || s == 0;
      };
      const int nc = a.nconf[k];
      if (nc <= kRsaMaxConf) {
        for (int q = 0; q < nc && !out; ++q) meet(a.conf[k * kRsaMaxConf + q]);
      } else {
        const double *p = a.cand + 3 * k;
        const float4 pf = a.candf[k];
        rsa_around(a, rsa_cell(a, p), a.head_b, a.next_b, [&](int j) {
          if (j < k && rsa_close(a, p, pf, a.cand + 3 * j, a.candf[j])) meet(j);
          return out;
        });
      }
      if (out || !wait) {
        state[k] = out ? 2 : 1;
        todo &= ~(1u << i);
      }
    }
    if (!__syncthreads_or(todo != 0)) break;
  }
  // places in candidate order: thread t counts a run of consecutive candidates
  const int per = (a.B + 1023) / 1024, k0 = threadIdx.x * per, k1 = min(a.B, k0 + per);
  int own = 0;
  for (int k = k0; k < k1; ++k) own += state[k] == 1;
  int inc = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += x;
  }
  if (lane == 31) s_sum[warp] = inc;
  const int kept = *a.kept;
  __syncthreads();
  int before = 0, all = 0;
  for (int w = 0; w < 32; ++w) {
    before += w < warp ? s_sum[w] : 0;
    all += s_sum[w];
  }
  int slot = kept + before + inc - own;
  for (int k = k0; k < k1; ++k) {
    const bool in = state[k] == 1 && slot < a.n;
    a.clear[k] = in ? 1 + slot : 0;  // for rsa_place_kernel
    if (in && ++slot == a.n) *a.used = a.c0 + k + 1;
  }
  if (threadIdx.x == 0) *a.kept = min(a.n, kept + all);
}

// The kept candidates into their places and into the lists of kept spheres.
__global__ void rsa_place_kernel(const RsaArgs a) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.B || a.clear[k] == 0) return;
  const int slot = a.clear[k] - 1;
  const double *p = a.cand + 3 * k;
  for (int q = 0; q < 3; ++q) a.pos[3 * slot + q] = p[q];
  a.posf[slot] = a.candf[k];
  a.next_k[slot] = atomicExch(a.head_k + rsa_index(a, rsa_cell(a, p)), slot);
}

}  // namespace kmc
