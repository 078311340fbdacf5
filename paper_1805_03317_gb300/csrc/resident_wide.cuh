// HMC trajectory with the subsample resident in shared memory for BF16 rows of 41 to 64 covariates
// (Algorithm 1 step 2), in the arithmetic of the streamed kernel (k_hmc, estimator.cuh).
//
// The rows are those of resident.cuh (gathered once per particle, L + 1 passes over shared memory),
// but a lane per row would need 4 p registers of rows and gradient partials. The sums are those that
// one warp with T = 4 lanes per row and 16 slots per lane forms (k_hmc's tile at these widths), every
// one of them in the same order, so theta comes out bit for bit as the streamed kernel has it. That
// matters because one last bit of theta is 1e-5 of theta - theta_bar where |theta| is a few units,
// and sigma2_hat goes with about the sixth power of that: sums in another order moved sigma2_hat by
// 2e-5 on the Student-t problem. The work of that warp is spread over WARPS row warps and a lead warp
// without touching an order:
//   1. D and the row terms: a row's D is the streamed one's (16 slots per lane, four lanes), rows are
//      independent, so warp w takes sweeps (32 rows) w, w + WARPS, .. and leaves (d, r) in shared
//      memory. The lead warp forms C delta.
//   2. Gradient partials: sum r x and sum e r x of slot c over the rows 4 g .. 4 g + 3 of every sweep
//      (g = 0..7) are 512 independent chains; a lane takes 64 / WARPS / 4 slots of one g and runs down
//      the rows. Three shuffles add the eight chains of a slot, in k_hmc's tree. The lead warp sums e.
//   3. The lead warp alone has theta, rho and the gradient (columns lane, lane + 32): leapfrog update.
// e = d - K with K the d of the particle's first row. Rows past m are copies of row m - 1 and count
// as zero. Block sums of the last pass: a block per warp.
//
// Bound by latency and issue: eight row warps and the lead at 0.41 instructions per cycle and scheduler
// (1250 rows leave room for one CTA per SM), a fifth of the stalls at the three barriers of a pass. us
// per trajectory of L = 20, streamed and here, Student-t p = 50: 770 and 262 for 280 particles of
// m = 1250, 510 and 340 for 1024 of 512, 3320 and 3350 for 4096 of 1250, 824 and 820 for 4096 of 100
// (four row warps: 294, 374, 3780 and 743). So every size that fits takes it.
//
// Row j is eight 16-byte units; unit u lies at u ^ wide_pos(j), which makes the 128-bit reads of step 1
// (four lanes x 32 bytes of two rows), the narrow reads of step 2 (32 bytes of four rows, or 16 of
// eight) and the reads of the constants (one unit of eight rows) free of bank conflicts.
#pragma once

#include "resident.cuh"

namespace subsmc {

__host__ __device__ inline int wide_pos(int j) {
  const int g = (j >> 2) & 7, t = j & 3;
  return (((g & 3) * 2 + (g & 1)) ^ (g >> 2)) ^ (t & 1) ^ ((t & 2) << 1);
}

// Shared-memory plan of one CTA (NV units of covariates per row; with NV = 7 the row's constants are
// its eighth unit, with NV = 8 they lie apart).
struct WidePlan {
  int off_consts, off_dr, off_mat, off_vec, off_blk, off_k, off_draws, total;
};
inline __host__ __device__ int round32(int v) { return (v + 31) & ~31; }
template <int NV> inline WidePlan wide_plan(int m, int G) {
  constexpr int CP = 8 * NV;
  const int mp = round32(m);
  WidePlan P;
  int off = mp * 128;
  P.off_consts = off;
  if (NV == 8) off += mp * (int)sizeof(RowC<float>);
  P.off_dr = off;  // (d, r) of every row; between trajectories the next rows' indices
  off += mp * 8;
  P.off_mat = off;  // C and Sigma, zero-padded to CP x CP
  off += 2 * CP * CP * 4;
  P.off_vec = off;  // 64 each: delta, rho, z, G1, G2; eight units of zeros
  off += 5 * 64 * 4 + 128;
  P.off_blk = off;
  off += G * 2 * (int)sizeof(double);
  P.off_k = off;
  off = round16(off + (int)sizeof(ResK<float>));
  P.off_draws = off;  // the next particles' draws
  off += kDraws<8> * (int)sizeof(Draws);
  P.total = off;
  return P;
}

// The row warps' gather of a particle's rows: the indices (wide_stage_u), then, after a wait and a
// barrier of the row warps, the rows and their constants at the centre (the packed row's tail).
// Invalid indices are flagged and their rows zeroed.
template <int WARPS>
__device__ __forceinline__ void wide_stage_u(const EstArgs &a, int i, int32_t *us) {
  const int32_t *u = a.u + (int64_t)i * a.m;
  for (int j = threadIdx.x; j < a.m; j += WARPS * 32) cp_async4(us + j, u + j);
  cp_async_wait_all();
  asm volatile("bar.sync 1, %0;\n" ::"n"(WARPS * 32) : "memory");
}
template <int NV, int WARPS>
__device__ __forceinline__ void wide_gather(const EstArgs &a, const WidePlan &P, const int32_t *us,
                                            unsigned char *rows, unsigned char *consts) {
  const int m = a.m, mp = round32(m), nvec = round16(a.p * 2) / 16;
  const int64_t pitch = (int64_t)a.S * 2;
  const unsigned char *Xp = reinterpret_cast<const unsigned char *>(a.Xp);
  auto unit = [&](int j, bool tail, int u, unsigned char *dst) {
    const uint32_t k = (uint32_t)us[min(j, m - 1)];
    const bool bad = k >= (uint32_t)a.n;  // n < 2^31
    if (bad || (!tail && u >= nvec)) {
      *reinterpret_cast<uint4 *>(dst) = make_uint4(0u, 0u, 0u, 0u);
      if (bad && u == 0) set_err(a.st, kErrIndex);
    } else {
      cp_async16(dst, Xp + (int64_t)k * pitch + (tail ? a.Yo * 2 : 16 * u));
    }
  };
  for (int t = threadIdx.x; t < 8 * mp; t += WARPS * 32) {
    const int j = t >> 3, u = t & 7;
    unit(j, u == NV, u, rows + j * 128 + ((u ^ wide_pos(j)) << 4));
  }
  if (NV == 8)
    for (int j = threadIdx.x; j < mp; j += WARPS * 32) unit(j, true, 8, consts + 16 * j);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// One particle's trajectory (the steps of hmc_body, estimator.cuh). Its rows are already on their way;
// an, in: the CTA's next particle (an null: none), whose rows are gathered as soon as this
// trajectory has read its own for the last time. reload: the CTA's previous particle belonged to
// another problem, or there was none.
template <int NV, int WARPS>
__device__ __forceinline__ void wide_particle(const EstArgs &a, int i, bool reload, const WidePlan &P,
                                              const Draws &draws, const EstArgs *an, int in) {
  constexpr int CP = 8 * NV, NT = (WARPS + 1) * 32;
  constexpr int SPL = 32 / WARPS;        // bytes of a row that a lane takes in step 2: 8 or 4
  constexpr int NS = SPL / 4;            // its slot pairs
  static_assert(WARPS == 4 || WARPS == 8, "row warps");
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (warp-uniform to the compiler)
  const bool lead = warp == WARPS;
  const int p = a.p, m = a.m, G = a.G, nsw = (m + 31) >> 5;
  const unsigned char *rows = smem;
  float2 *dr = reinterpret_cast<float2 *>(smem + P.off_dr);
  float *Cs = reinterpret_cast<float *>(smem + P.off_mat), *Sgs = Cs + CP * CP;
  float *vdl = reinterpret_cast<float *>(smem + P.off_vec), *vrho = vdl + 64, *vz = vrho + 64,
        *G1s = vz + 64, *G2s = G1s + 64;
  double *blks = reinterpret_cast<double *>(smem + P.off_blk);
  ResK<float> *ks = reinterpret_cast<ResK<float> *>(smem + P.off_k);
  const float inv_s2 = (float)a.inv_s2;
  const int fam = a.fam, cv1 = a.cv_order == 1;
  const int g = lane >> 2, q = lane & 3;  // group of rows, lane of the group

  const uint32_t smv = stage_move(a.stage_dev ? a.st->stage : a.stage, a.move);
  if (reload) {
    __syncthreads();  // the lead warp has decided on the previous particle
    if (tid == 0) {
      ResK<float> k;
      k.temp = a.st->a;
      k.nm = (double)a.n / (double)m;
      k.inv_m = 1.0 / (double)m;
      k.ta = (float)k.temp;
      k.ta2 = (float)(k.temp * k.temp * k.nm * k.nm);
      k.tnm = (float)(k.temp * k.nm);
      *ks = k;
    }
    if (tid < 32) G2s[64 + tid] = 0.f;
    for (int e = tid; e < CP * CP; e += NT) {
      const int r = e / CP, c = e - r * CP;
      const bool in_ = r < p && c < p;
      Cs[e] = in_ ? ldg_ct<float>(a.C_ct, r * p + c) : 0.f;
      Sgs[e] = in_ ? ldg_ct<float>(a.Sigma_ct, r * p + c) : 0.f;
    }
    __syncthreads();
  }
  const ResK<float> kc = *ks;
  const double temp = kc.temp, nm = kc.nm;
  float *thg = reinterpret_cast<float *>(a.theta_out) + (int64_t)i * p;
  // the lead warp's columns lane, lane + 32
  float th[2] = {0.f, 0.f}, rho[2] = {0.f, 0.f}, gr[2], cd[2] = {0.f, 0.f};
  float Bc[2], muc[2], ivc[2], tbc[2];
  bool col[2];
  float eps = 0.f;
  double logU = 0.0, lp0 = 0.0, kin0 = 0.0, like0 = 0.0, qlin = 0.0;
  auto log_prior = [&](const float *t, const float *mu, const float *iv) -> double {
    double lp = 0.0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const double rr = (double)t[h] - (double)mu[h];
      if (col[h]) lp += -0.5 * rr * rr * (double)iv[h];
    }
    return warp_sum(lp) + a.log_prior_const;
  };
  // y[c] = sum_k M[k, c] x_k, k ascending, for x in shared memory
  auto matvec = [&](const float *Ms, const float *x, float *y) {
    const int c1 = lane + 32 < CP ? lane + 32 : 0;
    float s0 = 0.f, s1 = 0.f;
#pragma unroll 2
    for (int k0 = 0; k0 < CP; k0 += 8) {
      float xv[8];
      load_vec<8>(x + k0, xv);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        s0 = fmaf(Ms[(k0 + k) * CP + lane], xv[k], s0);
        s1 = fmaf(Ms[(k0 + k) * CP + c1], xv[k], s1);
      }
    }
    y[0] = s0;
    y[1] = s1;
  };
  auto kinetic = [&]() -> double {  // rho' Sigma rho / 2
    float v[2];
    __syncwarp();
    vrho[lane] = rho[0];
    vrho[lane + 32] = rho[1];
    __syncwarp();
    matvec(Sgs, vrho, v);
    double k = 0.0;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (col[h]) k += (double)rho[h] * (double)v[h];
    return 0.5 * warp_sum(k);
  };
  auto set_delta = [&]() {
#pragma unroll
    for (int h = 0; h < 2; ++h) vdl[lane + 32 * h] = col[h] ? th[h] - tbc[h] : 0.f;
  };
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c = lane + 32 * h;
    col[h] = c < p;
    if (lead) {
      Bc[h] = col[h] ? ldg_ct<float>(a.B_ct, c) : 0.f;
      muc[h] = col[h] ? ldg_ct<float>(a.mu_ct, c) : 0.f;
      ivc[h] = col[h] ? ldg_ct<float>(a.ivar_ct, c) : 0.f;
      tbc[h] = col[h] ? ldg_ct<float>(a.tb_ct, c) : 0.f;
    }
  }
  // momentum draws and the prior at the start while the rows arrive
  if (lead) {
#pragma unroll
    for (int h = 0; h < 2; ++h) th[h] = col[h] ? thg[lane + 32 * h] : 0.f;
    eps = (float)draws.eps;
    logU = draws.logU;
    set_delta();
    lp0 = log_prior(th, muc, ivc);
  } else if (warp < 2) {
    const Stream smom(a.seed, kMomentum, smv, (uint32_t)i);
    const int c = lane + 32 * warp;
    vz[c] = c < p ? (float)stream_normal(smom, (uint32_t)c) : 0.f;
  }
  if (!lead) cp_async_wait_all();
  __syncthreads();  // the row warps' copies have landed; delta and z are there
  if (lead) {  // rho_r = sum_{c >= r} Linv[c, r] z_c, c ascending
#pragma unroll 8
    for (int c = 0; c < p; ++c) {
      const float zc = vz[c];
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (col[h] && c >= lane + 32 * h)
          rho[h] = fmaf(ldg_ct<float>(a.Linv_ct, c * p + lane + 32 * h), zc, rho[h]);
    }
    kin0 = kinetic();
  }
  float K = 0.f, cdbar = 0.f;
  // estimates and target (without the prior) from a pass's shifted sums, as eval_particle has them
  auto like = [&](double S, double Q, double &ell, double &sig) -> double {
    ell = (a.A_dev ? __ldg(a.A_dev) : a.A) + qlin + nm * fma((double)m, (double)K, S);
    sig = nm * nm * fmax(0.0, Q - S * S / (double)m);
    return temp * ell - 0.5 * temp * temp * sig;
  };
  // byte offsets of this lane's reads within a sweep. A lane whose second unit is the constants'
  // (NV = 7: slots 56 to 63) reads zeros there.
  const bool none = NV == 7 && q == 3;
  uint32_t o0[4], o1[4], o2[4];
  const int u2 = warp * SPL / 4 + (WARPS == 4 ? q >> 1 : 0);  // step 2's unit
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int j = 4 * g + t, x = wide_pos(j);
    o0[t] = j * 128 + (((2 * q) ^ x) << 4);
    o1[t] = none ? (uint32_t)(P.off_vec + 5 * 64 * 4) + ((7 ^ x) << 4) : j * 128 + (((2 * q + 1) ^ x) << 4);
    o2[t] = j * 128 + ((u2 ^ x) << 4) + (WARPS == 4 ? 8 * (q & 1) : 4 * q);
  }
  const uint32_t st1 = none ? 0u : 4096u;
  const uint32_t oc = NV == 7 ? lane * 128 + ((7 ^ wide_pos(lane)) << 4) : P.off_consts + lane * 16;
  constexpr uint32_t stc = NV == 7 ? 4096u : 512u;
  double ell1 = 0.0, sig1 = 0.0, S = 0.0, Q = 0.0;

  // One estimator pass at the current delta; ends with the gradient at the lead warp's columns.
  auto pass = [&](bool first, bool final) {
    if (!lead) {  // 1. D, d and r
      float dl[16];
      load_vec<16>(vdl + 16 * q, dl);
      auto sweeps = [&](auto famc) {
        constexpr int F = decltype(famc)::value;
        for (int s = warp; s < nsw; s += WARPS) {
          float pd[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            float x[16];
            Store<__nv_bfloat16>::unpack(*reinterpret_cast<const uint4 *>(rows + o0[t] + s * 4096u), x);
            Store<__nv_bfloat16>::unpack(*reinterpret_cast<const uint4 *>(rows + o1[t] + s * st1),
                                         x + 8);
            pd[t] = dot_slots<16>(x, dl);
          }
          int base = 0;
          reduce_scatter<4, 2, float>(pd, lane, base);
          const RowC<float> c = *reinterpret_cast<const RowC<float> *>(rows + oc + s * stc);
          float d, r;
          row_incr<F, float>(c, pd[0], inv_s2, d, r,
                             __all_sync(0xffffffffu, fabsf(pd[0]) <= 0.05f));
          if (cv1) to_first_order(row_l2<F, float>(c, inv_s2), pd[0], d, r);
          const int j = 32 * s + lane;
          dr[j] = j < m ? make_float2(d, r) : make_float2(0.f, 0.f);
        }
      };
      switch (fam) {
        case 0: sweeps(std::integral_constant<int, 0>{}); break;
        case 1: sweeps(std::integral_constant<int, 1>{}); break;
        case 2: sweeps(std::integral_constant<int, 2>{}); break;
        case 3: sweeps(std::integral_constant<int, 3>{}); break;
        default: sweeps(std::integral_constant<int, 4>{}); break;
      }
    } else {
      matvec(Cs, vdl, cd);
      if (first || final) {  // the linear and quadratic part of l_hat
        double ql = 0.0;
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (col[h]) ql += (double)((th[h] - tbc[h]) * (Bc[h] + 0.5f * cd[h]));
        qlin = warp_sum(ql);
      }
    }
    __syncthreads();
    K = dr[0].x;
    if (!lead) {  // 2. gradient partials
      if (warp * (64 / WARPS) < p) {
        float g1[2 * NS], g2[2 * NS];
#pragma unroll
        for (int e = 0; e < 2 * NS; ++e) g1[e] = g2[e] = 0.f;
#pragma unroll 4
        for (int s = 0; s < nsw; ++s) {
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            uint32_t w[NS];
            const unsigned char *src = rows + o2[t] + s * 4096u;
            if constexpr (NS == 2) {
              const uint2 v = *reinterpret_cast<const uint2 *>(src);
              w[0] = v.x;
              w[1] = v.y;
            } else {
              w[0] = *reinterpret_cast<const uint32_t *>(src);
            }
            const float2 v = dr[32 * s + 4 * g + t];
            const float er = __fmul_rn(v.x - K, v.y);
#pragma unroll
            for (int e = 0; e < NS; ++e) {  // (scalar: a packed FMA would need (r, r) and (e r, e r))
              const float x0 = __uint_as_float(w[e] << 16), x1 = __uint_as_float(w[e] & 0xFFFF0000u);
              g1[2 * e] = fmaf(v.y, x0, g1[2 * e]);
              g1[2 * e + 1] = fmaf(v.y, x1, g1[2 * e + 1]);
              g2[2 * e] = fmaf(er, x0, g2[2 * e]);
              g2[2 * e + 1] = fmaf(er, x1, g2[2 * e + 1]);
            }
          }
        }
#pragma unroll
        for (int o = 4; o < 32; o <<= 1)
#pragma unroll
          for (int e = 0; e < 2 * NS; ++e) {
            g1[e] += __shfl_xor_sync(0xffffffffu, g1[e], o);
            g2[e] += __shfl_xor_sync(0xffffffffu, g2[e], o);
          }
        if (g == 0)
#pragma unroll
          for (int e = 0; e < 2 * NS; ++e) {
            const int c = warp * (64 / WARPS) + 2 * NS * q + e;
            G1s[c] = g1[e];
            G2s[c] = g2[e];
          }
      }
    } else if (!final) {  // sums of e, e^2 by lane, then over the lanes in FP64
      float sd = 0.f, sd2 = 0.f;
#pragma unroll 4
      for (int s = 0; s < nsw; ++s) {
        const int j = 32 * s + lane;
        const float e = j < m ? dr[j].x - K : 0.f;
        sd += e;
        sd2 = fmaf(e, e, sd2);
      }
      S = warp_sum((double)sd);
      cdbar = (float)(S / (double)m);
      if (first) {
        double e0, s0;
        like0 = like(S, warp_sum((double)sd2), e0, s0);
      }
    }
    if (final) {  // block sums of e, e^2 (floor partition of u into G blocks)
      for (int b = warp; b < G; b += WARPS + 1) {
        const int j0 = block_start(b, m, G), j1 = block_start(b + 1, m, G);
        double bs = 0.0, bq = 0.0;
        for (int s = j0 >> 5; 32 * s < j1; ++s) {  // a tree per sweep, as the streamed rows
          const int j = 32 * s + lane;
          const float e = j >= j0 && j < j1 ? dr[j].x - K : 0.f;
          bs += (double)warp_sum(e);
          bq += (double)warp_sum(__fmul_rn(e, e));
        }
        if (lane == 0) {
          blks[2 * b] = bs;
          blks[2 * b + 1] = bq;
        }
      }
    }
    __syncthreads();
    if (lead) {  // 3. the gradient of a l_hat - a^2/2 sigma2_hat + log p(theta)
      if (final) {
        S = Q = 0.0;
        for (int b = lane; b < G; b += 32) {
          S += blks[2 * b];
          Q += blks[2 * b + 1];
        }
        S = warp_sum(S);
        Q = warp_sum(Q);
        cdbar = (float)(S / (double)m);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        gr[h] = target_grad(kc.ta, kc.tnm, kc.ta2, Bc[h], cd[h], G1s[c], G2s[c], cdbar, th[h] - muc[h],
                            ivc[h]);
        if (!col[h]) gr[h] = 0.f;
      }
    }
  };

  pass(true, false);
  for (int l = 0; l < a.L; ++l) {
    if (lead) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        rho[h] += 0.5f * eps * gr[h];
        vrho[lane + 32 * h] = rho[h];
      }
      __syncwarp();
      float v[2];
      matvec(Sgs, vrho, v);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (col[h]) th[h] += eps * v[h];
      set_delta();
    }
    __syncthreads();
    pass(false, l == a.L - 1);
    if (lead) {
#pragma unroll
      for (int h = 0; h < 2; ++h) rho[h] += 0.5f * eps * gr[h];
    }
  }
  // Metropolis-Hastings in the lead warp; the rows and (d, r) have been read for the last time, so the
  // row warps fetch the next particle's
  if (lead) {
    const double like1 = like(S, Q, ell1, sig1);
    const double H0 = -(like0 + lp0) + kin0;
    const double H1 = -(like1 + log_prior(th, muc, ivc)) + kinetic();
    if (logU < H0 - H1) {  // log U < H0 - H1; false when H1 is NaN
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (col[h]) thg[lane + 32 * h] = th[h];
      // the cache holds FP64 (sum d, sum d^2) per block: rebuilt from the shifted sums
      double *blk = a.blk + (int64_t)i * G * 2;
      const double k = (double)K;
      for (int b = lane; b < G; b += 32) {
        const double ng = (double)(block_start(b + 1, m, G) - block_start(b, m, G));
        const double se = blks[2 * b], qe = blks[2 * b + 1];
        blk[2 * b] = fma(ng, k, se);
        blk[2 * b + 1] = qe + k * fma(ng, k, 2.0 * se);
      }
      if (lane == 0) {
        a.ell[i] = ell1;
        a.sig2[i] = sig1;
        atomicAdd(&a.st->acc_theta, 1ull);
      }
    }
  } else if (an) {
    wide_stage_u<WARPS>(*an, in, reinterpret_cast<int32_t *>(dr));
    wide_gather<NV, WARPS>(*an, P, reinterpret_cast<const int32_t *>(dr), smem, smem + P.off_consts);
  }
}

// The first particle's rows of a CTA.
template <int NV, int WARPS>
__device__ __forceinline__ void wide_first(const EstArgs &a, int i, const WidePlan &P,
                                           unsigned char *smem) {
  if (threadIdx.x >= WARPS * 32) return;
  int32_t *us = reinterpret_cast<int32_t *>(smem + P.off_dr);
  wide_stage_u<WARPS>(a, i, us);
  wide_gather<NV, WARPS>(a, P, us, smem, smem + P.off_consts);
}

template <int NV, int WARPS>
__global__ void __launch_bounds__((WARPS + 1) * 32, 2) k_hmc_wide(EstArgs a, WidePlan P) {
  extern __shared__ __align__(16) unsigned char smem[];
  Draws *dr = reinterpret_cast<Draws *>(smem + P.off_draws);
  if ((int)blockIdx.x < a.B) wide_first<NV, WARPS>(a, a.i0 + (int)blockIdx.x, P, smem);
  int k = 0;
  for (int il = blockIdx.x; il < a.B; il += gridDim.x, ++k) {
    if (k % kDraws<8> == 0) {
      if (k) __syncthreads();
      const int64_t nx = il + (int64_t)threadIdx.x * gridDim.x;
      if (threadIdx.x < kDraws<8> && nx < a.B) dr[threadIdx.x] = theta_draws(a, a.i0 + (int)nx);
      __syncthreads();
    }
    const bool more = (int64_t)il + gridDim.x < a.B;
    wide_particle<NV, WARPS>(a, a.i0 + il, k == 0, P, dr[k % kDraws<8>], more ? &a : nullptr,
                             a.i0 + il + (int)gridDim.x);
  }
}

// All particles of the problems of a batch that share one tile (k_hmc_res_batch, resident.cuh).
template <int NV, int WARPS>
__global__ void __launch_bounds__((WARPS + 1) * 32, 2) k_hmc_wide_batch(BatchArgs b, WidePlan P) {
  extern __shared__ __align__(16) unsigned char smem[];
  Draws *dr = reinterpret_cast<Draws *>(smem + P.off_draws);
  int qcur = -1, k = 0, pr = 0;
  if ((int)blockIdx.x < b.total) {
    pr = batch_problem(b.offsets, b.nprob, blockIdx.x);
    wide_first<NV, WARPS>(b.probs[pr], (int)blockIdx.x - b.offsets[pr], P, smem);
  }
  for (int gi = blockIdx.x; gi < b.total; gi += gridDim.x, ++k) {
    if (k % kDraws<8> == 0) {
      if (k) __syncthreads();
      const int64_t gx = gi + (int64_t)threadIdx.x * gridDim.x;
      if (threadIdx.x < kDraws<8> && gx < b.total) {
        const int px = batch_problem(b.offsets, b.nprob, (int)gx);
        dr[threadIdx.x] = theta_draws(b.probs[px], (int)gx - b.offsets[px]);
      }
      __syncthreads();
    }
    const int64_t gn = (int64_t)gi + gridDim.x;
    const int pn = gn < b.total ? batch_problem(b.offsets, b.nprob, (int)gn) : pr;
    wide_particle<NV, WARPS>(b.probs[pr], gi - b.offsets[pr], pr != qcur, P, dr[k % kDraws<8>],
                             gn < b.total ? &b.probs[pn] : nullptr, (int)gn - b.offsets[pn]);
    qcur = pr;
    pr = pn;
  }
}

// Resident CTAs per SM of a kernel with `smem` bytes of dynamic shared memory (0: it does not fit).
template <typename K> inline int resident_blocks(K *kernel, int threads, int smem) {
  int per_sm = 0;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem) !=
          cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return per_sm;
}

template <int NV, int WARPS>
inline int launch_wide(const EstArgs &a, cudaStream_t s, int sms, bool dry) {
  if (a.p > 8 * NV) return -2;
  const WidePlan P = wide_plan<NV>(a.m, a.G);
  const int per_sm = resident_blocks(k_hmc_wide<NV, WARPS>, (WARPS + 1) * 32, P.total);
  if (per_sm < 1) return -2;
  if (dry || a.B <= 0) return 0;
  const int grid = a.B < per_sm * sms ? a.B : per_sm * sms;
  k_hmc_wide<NV, WARPS><<<grid, (WARPS + 1) * 32, P.total, s>>>(a, P);
  return (int)cudaGetLastError();
}

template <int NV, int WARPS>
inline int launch_wide_batch(const BatchArgs &b, int p_max, int m_max, int G_max, cudaStream_t s,
                             int sms, bool dry) {
  if (p_max > 8 * NV) return -2;
  const WidePlan P = wide_plan<NV>(m_max, G_max);
  prefer_shared(k_hmc_wide_batch<NV, WARPS>);
  const int per_sm = resident_blocks(k_hmc_wide_batch<NV, WARPS>, (WARPS + 1) * 32, P.total);
  if (per_sm < 1) return -2;
  if (dry || b.total <= 0) return 0;
  const int grid = b.total < per_sm * sms ? b.total : per_sm * sms;
  k_hmc_wide_batch<NV, WARPS><<<grid, (WARPS + 1) * 32, P.total, s>>>(b, P);
  return (int)cudaGetLastError();
}

}  // namespace subsmc
