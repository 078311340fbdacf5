// HMC trajectory with the particle's subsample resident in shared memory (Algorithm 1 step 2).
//
// u is fixed for the whole trajectory, so the m rows x_{u_j} are gathered once per particle
// (cp.async, 16-byte copies) and kept in shared memory, together with each row's stored
// control-variate constants (its tail: they depend on eta_bar_j and y_j only). The L + 1 estimator passes
// then read shared memory: one lane per row, D_j = x_j'(theta - theta_bar) and the increment terms
// d_j, r_j (device.cuh), gradient partials in registers, a shuffle reduce-scatter per warp and one
// CTA barrier per pass (partials double-buffered). Every warp then assembles the totals and the
// gradient and runs the leapfrog update itself, with theta, rho and the gradient held one column
// per lane (lane l also holds column l + 32 in tiles wider than 32 slots), so no warp waits for
// another between passes. One CTA handles one particle at a time and loops over particles
// (persistent grid).
//
// Sums over rows are of e_j = d_j - K with a CTA-uniform shift K near the subsample mean of d: the
// cached mean for the first pass, then the previous pass's mean (shifted data: Chan, Golub &
// LeVeque 1983). sigma2_hat = (n/m)^2 (sum e^2 - (sum e)^2/m) then stays accurate in FP32 partial
// sums where the d_j share a large mean (particles far from the centre), and the gradient's
// sum (d_j - dbar) r_j x_j is formed as sum e_j r_j x_j - ebar sum r_j x_j without that cancellation.
// The block cache keeps FP64 (sum d, sum d^2), rebuilt from the shifted block sums.
#pragma once

#include "estimator.cuh"

namespace subsmc {

// A particle's scalar draws of the theta move: the log of its MH uniform and its step size. FP64, and
// a warp-wide FP64 instruction holds its pipe for tens of cycles, so a CTA draws them for its next
// few particles at once, one per lane, instead of one particle at a time in every lane.
struct Draws {
  double logU, eps;
};
template <int WARPS> constexpr int kDraws = WARPS >= 8 ? 8 : WARPS == 4 ? 3 : 2;
__device__ __forceinline__ Draws theta_draws(const EstArgs &a, int i) {
  const uint32_t smv = stage_move(a.stage_dev ? a.st->stage : a.stage, a.move);
  Draws o;
  o.logU = log(draw_uniform(Stream(a.seed, kMhTheta, smv, (uint32_t)i).draw(0)));
  o.eps = jittered_eps(a.st->eps, a.eps_jitter, a.seed, smv, (uint32_t)i);
  return o;
}

// FP64 parts of a particle's Hamiltonians, from the warps that form them to the one that decides.
struct HamSums {
  double lp0, lp1, like0, S1, S2;  // log priors; a l_hat - a^2/2 sigma2_hat at the start; block sums
};

// First row of block b of the floor partition of m rows (b m < 2^32: m rows fit shared memory).
__device__ __forceinline__ int block_start(int b, int m, int G) {
  return (int)(((uint32_t)b * (uint32_t)m) / (uint32_t)G);
}

// A vector of CPL values (a multiple of 4) from 16-byte aligned shared memory.
template <int CPL> __device__ __forceinline__ void load_vec(const float *v, float *x) {
#pragma unroll
  for (int k = 0; k < CPL; k += 4) {
    const float4 w = *reinterpret_cast<const float4 *>(v + k);
    x[k] = w.x;
    x[k + 1] = w.y;
    x[k + 2] = w.z;
    x[k + 3] = w.w;
  }
}
template <int CPL> __device__ __forceinline__ void load_vec(const double *v, double *x) {
#pragma unroll
  for (int k = 0; k < CPL; k += 2) {
    const double2 w = *reinterpret_cast<const double2 *>(v + k);
    x[k] = w.x;
    x[k + 1] = w.y;
  }
}

// Shared-memory plan of one CTA.
struct ResPlan {
  int rb;    // bytes per resident row (covariates only): an odd multiple of 16 (conflict-free LDS.128)
  int nvl;   // 16-byte vectors the tile's CPL slots read (those past the covariates are zero-filled)
  int off_consts, off_d, off_red, off_redd, off_blk, off_mat, off_k, off_h, total;
};

// Constants of one launch of a problem (temperature, n/m, stage counter), computed once per
// problem by one thread instead of once per particle by every thread.
template <typename CT> struct alignas(16) ResK {
  double temp, nm, inv_m;
  CT ta, ta2, tnm;
};

inline __host__ __device__ int round16(int v) { return (v + 15) & ~15; }

template <typename CT>
inline ResPlan res_plan(int p, int m, int G, int esz, int warps, int cpl) {
  ResPlan P;
  const int xl = round16(cpl * esz);
  P.nvl = xl / 16;
  P.rb = ((xl / 16) % 2 == 0) ? xl + 16 : xl;
  int off = m * P.rb;
  P.off_consts = off;
  off = round16(off + m * (int)sizeof(RowC<CT>));
  P.off_d = off;
  off = round16(off + m * (int)sizeof(CT));
  P.off_red = off;  // two buffers of [warps][2 cpl] gradient partials
  off = round16(off + 2 * warps * 2 * cpl * (int)sizeof(CT));
  P.off_redd = off;  // two buffers of [2][warps] sums of e, e^2
  off = round16(off + 2 * warps * 2 * (int)sizeof(CT));
  P.off_blk = off;
  off = round16(off + G * 2 * (int)sizeof(double));
  P.off_mat = off;  // C and Sigma, zero-padded to [cpl, cpl], state type
  off = round16(off + 2 * cpl * cpl * (int)sizeof(CT));
  P.off_k = off;
  off = round16(off + (int)sizeof(ResK<CT>));
  P.off_h = off;  // HamSums, then the next particles' draws
  off = round16(off + (int)sizeof(HamSums) +
                (warps >= 8 ? kDraws<8> : warps == 4 ? kDraws<4> : kDraws<1>) * (int)sizeof(Draws));
  P.total = off;
  return P;
}

__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// CPL covariate slots of a resident row; CPL need not be a multiple of the 16-byte vector width
// (the row holds whole vectors, zero-padded, and the unused tail of the last one is dropped).
template <typename XT, int CPL>
__device__ __forceinline__ void load_res_row(const unsigned char *row,
                                             typename Store<XT>::CT *x) {
  using SD = Store<XT>;
  using CT = typename SD::CT;
  constexpr int NV = CPL / SD::VEC, REM = CPL % SD::VEC;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    const uint4 w = *reinterpret_cast<const uint4 *>(row + 16 * v);
    SD::unpack(w, x + v * SD::VEC);
  }
  if constexpr (REM > 0) {
    CT t[SD::VEC];
    SD::unpack(*reinterpret_cast<const uint4 *>(row + 16 * NV), t);
#pragma unroll
    for (int e = 0; e < REM; ++e) x[NV * SD::VEC + e] = t[e];
  }
}

// The gather of a particle's rows: the indices into us, then (after a wait and a barrier) x_{u_j}
// and the row's constants at the centre (its tail) with 16-byte copies; invalid indices are flagged
// and their rows zeroed. Vectors the tile reads beyond the row's covariates (a tile wider than p)
// are zero-filled. The indices are staged in shared memory first (the buffer of the e_j is free
// until the last pass), so no copy waits on a global load.
template <int WARPS>
__device__ __forceinline__ void res_stage_u(const EstArgs &a, int i, int32_t *us) {
  const int32_t *u = a.u + (int64_t)i * a.m;
  for (int j = threadIdx.x; j < a.m; j += WARPS * 32) cp_async4(us + j, u + j);
}
template <typename XT, int WARPS>
__device__ __forceinline__ void res_gather(const EstArgs &a, const ResPlan &P, const int32_t *us,
                                           unsigned char *rows, unsigned char *consts) {
  using CT = typename Store<XT>::CT;
  constexpr int NT = WARPS * 32, NTV = (int)sizeof(RowC<CT>) / 16;
  const int m = a.m, tid = threadIdx.x;
  const int nvec = round16(a.p * (int)sizeof(XT)) / 16;  // 16-byte vectors of this problem's rows
  const int64_t pitch = (int64_t)a.S * (int)sizeof(XT);
  const unsigned char *Xp = reinterpret_cast<const unsigned char *>(a.Xp);
  const int nvr = P.nvl + NTV;
  // copy t = j nvr + q (vector q of row j); each thread steps by NT = dj nvr + dq
  const int dj = NT / nvr, dq = NT - dj * nvr;
  int j = tid / nvr, q = tid - (tid / nvr) * nvr;
  while (j < m) {
    const uint32_t k = (uint32_t)us[j];
    const bool bad = k >= (uint32_t)a.n;  // n < 2^31
    unsigned char *dst = q < P.nvl ? rows + j * P.rb + 16 * q
                                   : consts + j * (int)sizeof(RowC<CT>) + 16 * (q - P.nvl);
    const int qs = q < P.nvl ? q : nvec + (q - P.nvl);  // 16-byte vector of the packed row
    if (bad || (q >= nvec && q < P.nvl)) {
      *reinterpret_cast<uint4 *>(dst) = make_uint4(0u, 0u, 0u, 0u);
      if (q == 0 && bad) set_err(a.st, kErrIndex);
    } else {
      cp_async16(dst, Xp + (int64_t)k * pitch + 16 * qs);
    }
    j += dj;
    q += dq;
    if (q >= nvr) {
      q -= nvr;
      ++j;
    }
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// One particle's trajectory: particle i of the problem described by a, whose rows are already on
// their way (res_gather). reload: the CTA's previous particle belonged to another problem (or there
// was none), so the C and Sigma tiles are loaded. an, in: the CTA's next particle (an null: none).
// Its rows are gathered as soon as this trajectory has read its own for the last time, so they
// arrive during the FP64 work of this particle's acceptance test (before, a particle waited for its
// indices, then its rows, then log U: about 16 us of latency per particle and CTA at p = 20,
// m = 1000, which the other CTAs of the SM hid only in part).
// Lane l of every warp holds columns l, l + 32, .. of theta, rho and the gradient (NC per lane).
template <typename XT, int CPL, int WARPS>
__device__ __forceinline__ void res_particle(const EstArgs &a, int i, bool reload,
                                             const ResPlan &P, const Draws &draws,
                                             const EstArgs *an, int in) {
  using SD = Store<XT>;
  using CT = typename SD::CT;
  constexpr int NC = (CPL + 31) / 32, NT = WARPS * 32;
  static_assert(NC <= 2, "at most two columns per lane");
  // the warps that form the log priors, the first pass's likelihood term and the block totals
  // (warp 0: the kinetic energies and the decision)
  constexpr int kWarpP = WARPS > 1 ? 1 : 0, kWarpL = WARPS > 2 ? 2 : kWarpP,
                kWarpB = WARPS > 3 ? 3 : 0;
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (warp-uniform to the compiler)
  const int p = a.p, m = a.m, G = a.G;
  unsigned char *rows = smem;
  RowC<CT> *cst = reinterpret_cast<RowC<CT> *>(smem + P.off_consts);
  CT *dv = reinterpret_cast<CT *>(smem + P.off_d);
  int32_t *us = reinterpret_cast<int32_t *>(dv);
  CT *red = reinterpret_cast<CT *>(smem + P.off_red);       // [2][WARPS][2 CPL]
  CT *redd = reinterpret_cast<CT *>(smem + P.off_redd);     // [2][2][WARPS]
  double *blks = reinterpret_cast<double *>(smem + P.off_blk);  // [G][2]
  CT *Cs = reinterpret_cast<CT *>(smem + P.off_mat);  // [CPL, CPL] zero-padded
  CT *Sgs = Cs + CPL * CPL;                            // [CPL, CPL] zero-padded
  ResK<CT> *ks = reinterpret_cast<ResK<CT> *>(smem + P.off_k);
  HamSums *hs = reinterpret_cast<HamSums *>(smem + P.off_h);
  const CT inv_s2 = (CT)a.inv_s2;
  const int fam = a.fam;
  const int cv1 = a.cv_order == 1;
  // per-lane column constants (slot h of lane l is column l + 32 h)
  bool col[NC];
  int cl[NC];  // the column's index into the [CPL, CPL] tiles (0 past CPL: a padded read)
  CT Bc[NC], muc[NC], ivc[NC], tbc[NC];
#pragma unroll
  for (int h = 0; h < NC; ++h) {
    const int c = lane + 32 * h;
    col[h] = c < p;
    cl[h] = c < CPL ? c : 0;
    Bc[h] = col[h] ? ldg_ct<CT>(a.B_ct, c) : CT(0);
    muc[h] = col[h] ? ldg_ct<CT>(a.mu_ct, c) : CT(0);
    ivc[h] = col[h] ? ldg_ct<CT>(a.ivar_ct, c) : CT(0);
    tbc[h] = col[h] ? ldg_ct<CT>(a.tb_ct, c) : CT(0);
  }
  const uint32_t smv = stage_move(a.stage_dev ? a.st->stage : a.stage, a.move);
  if (reload) {
    if (tid == 0) {
      ResK<CT> k;
      k.temp = a.st->a;
      k.nm = (double)a.n / (double)m;
      k.inv_m = 1.0 / (double)m;
      k.ta = (CT)k.temp;
      k.ta2 = (CT)(k.temp * k.temp * k.nm * k.nm);
      k.tnm = (CT)(k.temp * k.nm);
      *ks = k;
    }
    for (int e = tid; e < CPL * CPL; e += NT) {
      const int r = e / CPL, c = e - r * CPL;
      const bool in_ = r < p && c < p;
      Cs[e] = in_ ? ldg_ct<CT>(a.C_ct, r * p + c) : CT(0);
      Sgs[e] = in_ ? ldg_ct<CT>(a.Sigma_ct, r * p + c) : CT(0);
    }
    __syncthreads();
  }
  const ResK<CT> kc = *ks;
  const double temp = kc.temp, nm = kc.nm, inv_m = kc.inv_m;
  const CT ta = kc.ta, ta2 = kc.ta2, tnm = kc.tnm;
  // 1. initial momentum rho = Linv' z, in every warp (while the rows arrive)
  CT *thg = reinterpret_cast<CT *>(a.theta_out) + (int64_t)i * p;
  const CT eps = (CT)draws.eps;
  const double logU = draws.logU;
  CT th[NC], rho[NC], gr[NC];
  {
    const Stream smom(a.seed, kMomentum, smv, (uint32_t)i);
    CT z[NC];
#pragma unroll
    for (int h = 0; h < NC; ++h) {
      z[h] = col[h] ? stream_normal_ct<CT>(smom, (uint32_t)(lane + 32 * h)) : CT(0);
      rho[h] = CT(0);
    }
#pragma unroll
    for (int hz = 0; hz < NC; ++hz)  // rho_r = sum_{c >= r} Linv[c, r] z_c, c ascending
#pragma unroll 4
      for (int cc = 0; cc < 32 && 32 * hz + cc < p; ++cc) {
        const int c = 32 * hz + cc;
        const CT zc = __shfl_sync(0xffffffffu, z[hz], cc);
#pragma unroll
        for (int h = 0; h < NC; ++h) {
          const int r = lane + 32 * h;
          if (col[h] && c >= r) rho[h] = fma(ldg_ct<CT>(a.Linv_ct, c * p + r), zc, rho[h]);
        }
      }
#pragma unroll
    for (int h = 0; h < NC; ++h) {
      th[h] = col[h] ? thg[lane + 32 * h] : CT(0);
      gr[h] = CT(0);
    }
  }
  // every warp carries the trajectory in its lanes: theta_c, rho_c, grad_c at lane c mod 32. A vector
  // that all lanes need entry by entry goes through the warp's own part of the partials' buffer
  // that the next pass will fill: every warp has read that buffer before the last pass's barrier.
  CT dr[CPL];
  int buf = 0;
  auto share = [&](const CT *v, CT *all) {
    CT *vec = red + (buf * WARPS + warp) * 2 * CPL;
    __syncwarp();  // the previous vector has been read
#pragma unroll
    for (int h = 0; h < NC; ++h)
      if (lane + 32 * h < CPL) vec[lane + 32 * h] = v[h];
    __syncwarp();
    load_vec<CPL>(vec, all);
  };
  auto set_delta = [&]() {
    CT dl[NC];
#pragma unroll
    for (int h = 0; h < NC; ++h) dl[h] = col[h] ? th[h] - tbc[h] : CT(0);
    share(dl, dr);
  };
  auto sigma_rho = [&](CT *vs) {  // (Sigma rho)_c at the lane's columns
    CT rk[CPL];
    share(rho, rk);
#pragma unroll
    for (int h = 0; h < NC; ++h) vs[h] = CT(0);
#pragma unroll
    for (int k = 0; k < CPL; ++k)
#pragma unroll
      for (int h = 0; h < NC; ++h) vs[h] = fma(Sgs[k * CPL + cl[h]], rk[k], vs[h]);
  };
  auto kinetic = [&]() -> double {  // rho' Sigma rho / 2 (every lane of the warp)
    CT v[NC];
    sigma_rho(v);
    double t = 0.0;
#pragma unroll
    for (int h = 0; h < NC; ++h) t += col[h] ? (double)rho[h] * (double)v[h] : 0.0;
    return 0.5 * warp_sum(t);
  };
  auto log_prior = [&]() -> double {
    double t = 0.0;
#pragma unroll
    for (int h = 0; h < NC; ++h) {
      const double rr = (double)th[h] - (double)muc[h];
      t += col[h] ? -0.5 * rr * rr * (double)ivc[h] : 0.0;
    }
    return warp_sum(t) + a.log_prior_const;
  };
  double kin0 = 0.0;
  if (warp == 0) kin0 = kinetic();
  if (warp == kWarpP) {
    const double lp = log_prior();
    if (lane == 0) hs->lp0 = lp;
  }
  set_delta();
  // shift of the row sums (identical in every warp): the cached subsample mean of d at this
  // particle's current theta and u, in FP64: its last bit is one of e's
  CT Ksh = CT(0);
  if (a.blk) {
    const double *bc = a.blk + (int64_t)i * G * 2;
    double s0 = 0.0;
    for (int g = lane; g < G; g += 32) s0 += bc[2 * g];
    Ksh = (CT)(warp_sum(s0) * inv_m);
    if (!isfinite(Ksh)) Ksh = CT(0);
  }
  cp_async_wait_all();
  __syncthreads();  // every warp's copies have landed
  CT qlin = CT(0), sum0 = CT(0), qlin0 = CT(0), Ksh0 = CT(0);  // (.. 0: the first pass's, warp kWarpL)
  // a l_hat - a^2/2 sigma2_hat, and both estimates, from the shifted sums of a pass (FP64)
  auto like = [&](double S1, double S2, double ql, double shift, double &ell,
                  double &sig) -> double {
    ell = (a.A_dev ? __ldg(a.A_dev) : a.A) + ql + nm * fma((double)m, shift, S1);
    sig = nm * nm * fmax(0.0, S2 - S1 * S1 * inv_m);
    return temp * ell - 0.5 * temp * temp * sig;
  };
  // One estimator pass at the current delta (dr). Every warp ends with the gradient at its lanes.
  // FULL (first and last pass): the sums that l_hat and sigma2_hat need; the last pass also fills the
  // block sums blks.
  auto pass = [&](auto full_c, bool final) {
    constexpr bool FULL = decltype(full_c)::value;
    CT v[2 * CPL];
#pragma unroll
    for (int s = 0; s < 2 * CPL; ++s) v[s] = CT(0);
    CT sd = CT(0), sd2 = CT(0);
    // the row loop, specialised per family (the dispatch is taken once per pass, not per row)
    auto row_loop = [&](auto famc) {
      constexpr int F = decltype(famc)::value;
      for (int j = warp * 32 + lane; j < m; j += NT) {
        CT x[CPL];
        load_res_row<XT, CPL>(rows + j * P.rb, x);
        const CT D = dot_slots<CPL>(x, dr);
        const RowC<CT> c = cst[j];
        CT d, r;
        row_incr<F, CT>(c, D, inv_s2, d, r);
        if (cv1) to_first_order(row_l2<F, CT>(c, inv_s2), D, d, r);
        const CT e = d - Ksh;
        axpy_slots<CPL>(r, x, v);
        axpy_slots<CPL>(e * r, x, v + CPL);
        sd += e;
        if (FULL) sd2 = fma(e, e, sd2);
        if (FULL && final) dv[j] = e;
      }
    };
    switch (fam) {
      case 0: row_loop(std::integral_constant<int, 0>{}); break;
      case 1: row_loop(std::integral_constant<int, 1>{}); break;
      case 2: row_loop(std::integral_constant<int, 2>{}); break;
      case 3: row_loop(std::integral_constant<int, 3>{}); break;
      default: row_loop(std::integral_constant<int, 4>{}); break;
    }
    int base = 0;
    reduce_scatter<2 * CPL, 16, CT>(v, lane, base);
    constexpr int KF = kfinal<2 * CPL, 16>();
    CT *rb = red + buf * WARPS * 2 * CPL;  // [warp][sum r x, sum e r x]
    CT *rd = redd + buf * WARPS * 2;       // [sum e, sum e^2][warp]
#pragma unroll
    for (int q = 0; q < KF; ++q) rb[warp * 2 * CPL + base + q] = v[q];
    const CT s1 = warp_sum(sd);
    if (lane == 0) rd[warp] = s1;
    if (FULL) {
      const CT s2 = warp_sum(sd2);
      if (lane == 0) rd[WARPS + warp] = s2;
    }
    __syncthreads();  // all warps' partial sums of this pass are in buffer buf
    // sum of e over the subsample (the gradient needs only its mean)
    CT S1f = CT(0);
#pragma unroll
    for (int w = 0; w < WARPS; ++w) S1f += rd[w];
    if (FULL && final) {  // shifted block sums of e (floor partition of u into G blocks)
      for (int g = warp; g < G; g += WARPS) {
        const int j0 = block_start(g, m, G), j1 = block_start(g + 1, m, G);
        CT bs = CT(0), bq = CT(0);
        for (int j = j0 + lane; j < j1; j += 32) {
          const CT dj = dv[j];
          bs += dj;
          bq = fma(dj, dj, bq);
        }
        bs = warp_sum(bs);
        bq = warp_sum(bq);
        if (lane == 0) {
          blks[2 * g] = (double)bs;
          blks[2 * g + 1] = (double)bq;
        }
      }
      __syncthreads();
    }
    // gradient of a l_hat - a^2/2 sigma2_hat + log p(theta) at the lane's columns (every warp)
    const CT dbar = S1f * (CT)inv_m;  // mean of e
    CT cd[NC];
#pragma unroll
    for (int h = 0; h < NC; ++h) cd[h] = CT(0);
#pragma unroll
    for (int k = 0; k < CPL; ++k)
#pragma unroll
      for (int h = 0; h < NC; ++h) cd[h] = fma(Cs[k * CPL + cl[h]], dr[k], cd[h]);
#pragma unroll
    for (int h = 0; h < NC; ++h) {
      CT G1 = CT(0), G2 = CT(0);
#pragma unroll
      for (int w = 0; w < WARPS; ++w) {
        G1 += rb[w * 2 * CPL + cl[h]];
        G2 += rb[w * 2 * CPL + CPL + cl[h]];
      }
      gr[h] = col[h] ? ta * (Bc[h] + cd[h]) + tnm * G1 - ta2 * (G2 - dbar * G1) -
                           (th[h] - muc[h]) * ivc[h]
                     : CT(0);
    }
    if (FULL && warp == (final ? 0 : kWarpL)) {  // the linear and quadratic part of l_hat
      CT ql = CT(0);
#pragma unroll
      for (int h = 0; h < NC; ++h)
        if (col[h]) ql += (th[h] - tbc[h]) * (Bc[h] + CT(0.5) * cd[h]);
      qlin = warp_sum(ql);
      if (!final) {  // the first pass's sums, for the FP64 work at the end
        sum0 = lane < 2 * WARPS ? rd[lane] : CT(0);
        qlin0 = qlin;
        Ksh0 = Ksh;
      }
    }
    if (!FULL || !final) Ksh += dbar;  // the next pass is shifted by this pass's mean of d
    buf ^= 1;
  };

  // 2. trajectory
  pass(std::true_type{}, false);
  for (int l = 0; l < a.L; ++l) {
    CT vs[NC];
#pragma unroll
    for (int h = 0; h < NC; ++h) rho[h] += CT(0.5) * eps * gr[h];
    sigma_rho(vs);
#pragma unroll
    for (int h = 0; h < NC; ++h)
      if (col[h]) th[h] += eps * vs[h];
    set_delta();
    if (l == a.L - 1)
      pass(std::true_type{}, true);
    else
      pass(std::false_type{}, false);
#pragma unroll
    for (int h = 0; h < NC; ++h) rho[h] += CT(0.5) * eps * gr[h];
  }
  // 3. Metropolis-Hastings. The rows have been read for the last time: the next particle's are
  // fetched under the FP64 terms (slow on this part: a warp-wide FP64 instruction holds its
  // sub-partition's pipe for tens of cycles), which are split over warps on different sub-partitions.
  if (an) res_stage_u<WARPS>(*an, in, us);
  double kin1 = 0.0;
  const double lp0 = hs->lp0;  // (the next particle's may be written during the decision)
  if (warp == 0) kin1 = kinetic();
  if (warp == kWarpP) {
    const double lp = log_prior();
    if (lane == 0) hs->lp1 = lp;
  }
  if (warp == kWarpL) {
    double S1 = 0.0, S2 = 0.0, e0, s0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
      S1 += (double)__shfl_sync(0xffffffffu, sum0, w);
      S2 += (double)__shfl_sync(0xffffffffu, sum0, WARPS + w);
    }
    const double v = like(S1, S2, (double)qlin0, (double)Ksh0, e0, s0);
    if (lane == 0) hs->like0 = v;
  }
  if (warp == kWarpB) {
    double S1 = 0.0, S2 = 0.0;
    for (int g = lane; g < G; g += 32) {
      S1 += blks[2 * g];
      S2 += blks[2 * g + 1];
    }
    S1 = warp_sum(S1);
    S2 = warp_sum(S2);
    if (lane == 0) {
      hs->S1 = S1;
      hs->S2 = S2;
    }
  }
  cp_async_wait_all();
  __syncthreads();
  if (an) res_gather<XT, WARPS>(*an, P, us, rows, smem + P.off_consts);
  if (warp == 0) {
    double ell, sig;
    const double like1 = like(hs->S1, hs->S2, (double)qlin, (double)Ksh, ell, sig);
    const double H0 = -(hs->like0 + lp0) + kin0;
    const double H1 = -(like1 + hs->lp1) + kin1;
    const bool acc = logU < H0 - H1;  // log U < H0 - H1; false when H1 is NaN
    if (acc) {
#pragma unroll
      for (int h = 0; h < NC; ++h)
        if (col[h]) thg[lane + 32 * h] = th[h];
      // the cache holds FP64 (sum d, sum d^2) per block: rebuilt from the shifted sums
      double *blk = a.blk + (int64_t)i * G * 2;
      const double k = (double)Ksh;
      for (int g = lane; g < G; g += 32) {
        const double ng = (double)(block_start(g + 1, m, G) - block_start(g, m, G));
        const double se = blks[2 * g], qe = blks[2 * g + 1];
        blk[2 * g] = fma(ng, k, se);
        blk[2 * g + 1] = qe + k * fma(ng, k, 2.0 * se);
      }
      if (lane == 0) {
        a.ell[i] = ell;
        a.sig2[i] = sig;
        atomicAdd(&a.st->acc_theta, 1ull);
      }
    }
  }
}

// The first particle's rows of a CTA.
template <typename XT, int WARPS>
__device__ __forceinline__ void res_first(const EstArgs &a, int i, const ResPlan &P,
                                          unsigned char *smem) {
  int32_t *us = reinterpret_cast<int32_t *>(smem + P.off_d);
  res_stage_u<WARPS>(a, i, us);
  cp_async_wait_all();
  __syncthreads();
  res_gather<XT, WARPS>(a, P, us, smem, smem + P.off_consts);
}

template <typename XT, int CPL, int WARPS>
__global__ void __launch_bounds__(WARPS * 32) k_hmc_res(EstArgs a, ResPlan P) {
  extern __shared__ __align__(16) unsigned char smem[];
  Draws *dr = reinterpret_cast<Draws *>(smem + P.off_h + sizeof(HamSums));
  if ((int)blockIdx.x < a.B) res_first<XT, WARPS>(a, a.i0 + (int)blockIdx.x, P, smem);
  int k = 0;
  for (int il = blockIdx.x; il < a.B; il += gridDim.x, ++k) {
    if (k % kDraws<WARPS> == 0) {
      if (k) __syncthreads();
      const int64_t nx = il + (int64_t)threadIdx.x * gridDim.x;
      if (threadIdx.x < kDraws<WARPS> && nx < a.B) dr[threadIdx.x] = theta_draws(a, a.i0 + (int)nx);
      __syncthreads();
    }
    const bool more = (int64_t)il + gridDim.x < a.B;
    res_particle<XT, CPL, WARPS>(a, a.i0 + il, k == 0, P, dr[k % kDraws<WARPS>], more ? &a : nullptr,
                                 a.i0 + il + (int)gridDim.x);
  }
}

// All particles of a batch of independent posteriors (the problems of one resident tile): the
// global particle index picks the problem from the prefix offsets; the shared-memory plan is the
// largest over those problems.
template <typename XT, int CPL, int WARPS>
__global__ void __launch_bounds__(WARPS * 32) k_hmc_res_batch(BatchArgs b, ResPlan P) {
  extern __shared__ __align__(16) unsigned char smem[];
  Draws *dr = reinterpret_cast<Draws *>(smem + P.off_h + sizeof(HamSums));
  int qcur = -1, k = 0, pr = 0;
  if ((int)blockIdx.x < b.total) {
    pr = batch_problem(b.offsets, b.nprob, blockIdx.x);
    res_first<XT, WARPS>(b.probs[pr], (int)blockIdx.x - b.offsets[pr], P, smem);
  }
  for (int g = blockIdx.x; g < b.total; g += gridDim.x, ++k) {
    if (k % kDraws<WARPS> == 0) {
      if (k) __syncthreads();
      const int64_t gx = g + (int64_t)threadIdx.x * gridDim.x;
      if (threadIdx.x < kDraws<WARPS> && gx < b.total) {
        const int px = batch_problem(b.offsets, b.nprob, (int)gx);
        dr[threadIdx.x] = theta_draws(b.probs[px], (int)gx - b.offsets[px]);
      }
      __syncthreads();
    }
    const int64_t gn = (int64_t)g + gridDim.x;
    const int pn = gn < b.total ? batch_problem(b.offsets, b.nprob, (int)gn) : pr;
    res_particle<XT, CPL, WARPS>(b.probs[pr], g - b.offsets[pr], pr != qcur, P, dr[k % kDraws<WARPS>],
                                 gn < b.total ? &b.probs[pn] : nullptr, (int)gn - b.offsets[pn]);
    qcur = pr;
    pr = pn;
  }
}

// dry: only check that the plan fits (no launch).
template <typename XT, int CPL, int WARPS>
inline int launch_res(const EstArgs &a, cudaStream_t s, int sms, bool dry) {
  using CT = typename Store<XT>::CT;
  if (a.p > CPL) return -2;
  const ResPlan P = res_plan<CT>(a.p, a.m, a.G, (int)sizeof(XT), WARPS, CPL);
  cudaError_t e = cudaFuncSetAttribute(k_hmc_res<XT, CPL, WARPS>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, P.total);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return -2;
  }
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_hmc_res<XT, CPL, WARPS>,
                                                    WARPS * 32, P.total);
  if (e != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    return -2;
  }
  if (dry || a.B <= 0) return 0;
  const int grid = a.B < per_sm * sms ? a.B : per_sm * sms;
  k_hmc_res<XT, CPL, WARPS><<<grid, WARPS * 32, P.total, s>>>(a, P);
  return (int)cudaGetLastError();
}

// The groups of a batch run side by side, and an SM takes CTAs of two kernels only if both ask for the
// same division of its memory. By default that follows from each kernel's own CTAs, so the groups
// of three small problems ran one after the other or not by a few bytes of a plan: 430 or 485 us
// per stage (186 particles, p = 5 to 23). All of them ask for the largest shared memory.
template <typename K> inline void prefer_shared(K *kernel) {
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                           cudaSharedmemCarveoutMaxShared) != cudaSuccess)
    cudaGetLastError();  // (a hint)
}

// Batched launch over the problems in b (their largest p, m and G size the plan). dry: check the
// fit only. Returns a cudaError_t or -2 when the plan does not fit.
template <typename XT, int CPL, int WARPS>
inline int launch_res_batch(const BatchArgs &b, int p_max, int m_max, int G_max, cudaStream_t s,
                            int sms, bool dry) {
  using CT = typename Store<XT>::CT;
  if (p_max > CPL) return -2;
  const ResPlan P = res_plan<CT>(p_max, m_max, G_max, (int)sizeof(XT), WARPS, CPL);
  cudaError_t e = cudaFuncSetAttribute(k_hmc_res_batch<XT, CPL, WARPS>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, P.total);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return -2;
  }
  prefer_shared(k_hmc_res_batch<XT, CPL, WARPS>);
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_hmc_res_batch<XT, CPL, WARPS>,
                                                    WARPS * 32, P.total);
  if (e != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    return -2;
  }
  if (dry || b.total <= 0) return 0;
  const int grid = b.total < per_sm * sms ? b.total : per_sm * sms;
  k_hmc_res_batch<XT, CPL, WARPS><<<grid, WARPS * 32, P.total, s>>>(b, P);
  return (int)cudaGetLastError();
}

}  // namespace subsmc
