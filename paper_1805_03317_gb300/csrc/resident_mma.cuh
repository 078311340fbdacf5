// HMC trajectory with the subsample resident in shared memory and both per-row contractions on the
// warp-level tensor-core path (BF16 storage; Algorithm 1 step 2). One CTA per particle, as in
// resident.cuh: the m rows are gathered once and the L + 1 estimator passes read shared memory.
//
// Why mma.sync and not tcgen05: a particle's contractions are [m x p].[p x 1] and [p x m].[m x 2]
// with other rows for every particle, so there is no shared operand and no wide N. tcgen05 needs
// 128-row tiles, a CTA-wide hand-over through tensor memory and an accumulator load per tile; the
// kernel built on it (resident_tc.cuh) is bound by that chain. Here each warp runs its own rows from
// ldmatrix to the gradient sums in registers, with one CTA barrier per pass.
//
// A warp takes 64 rows at a time.
//   D = X delta: delta is split by truncation into three BF16 terms (8 + 8 + 8 bits: exact), which
//   are columns of the 8-wide B operand. The columns are placed so that the four 16-row tiles land
//   in two accumulators with every lane owning two rows: lane 4g + q owns rows g and g + 8 of tile
//   q, tiles 0 and 2 use columns {2q, 2q+1, 2q+2} of accumulator A for (delta1, delta2, delta3),
//   tiles 1 and 3 columns {2q, 2q+1, 2q-2} of accumulator B, zero elsewhere; one shuffle with the
//   neighbouring lane brings the third term.
//   Row terms d, r on the lane's two rows (FP32, device.cuh).
//   [sum r x, sum e r x] = X' Q: Q holds (r, e r) as three BF16 terms each, split by truncation
//   again, 16 bytes per row, and passes through a 1 KB buffer of the warp into the B operand; X' is
//   read from the same rows by ldmatrix.trans. The FP32 accumulators carry the gradient partials
//   across all of the warp's rows, so no per-lane partials have to be reduce-scattered at the end.
// Row j of a 64-row group, 32 h + 8 q + ((g + 2 q) & 7), belongs to slot h of lane 4 g + q: with a row
// pitch of an odd number of 16-byte units this makes the ldmatrix reads of both contractions, the
// constants' 128-bit loads and the writes of Q free of bank conflicts.
//
// Used for 41 to 64 covariates, where the CUDA-core form of resident.cuh would need more than 255
// registers (4 p gradient partials and rows per lane) and the trajectories were streamed through one
// warp per particle: p = 50, m = 1250, L = 20, 280 particles (Student-t) 850 us streamed, 230 us here;
// 1024 particles, m = 512: 505 and 334 us. Bound by shared-memory bandwidth (X is read once per
// contraction; 70% of the wavefront rate) and by two CTAs of four warps at most to hide each pass's
// chain. At p <= 40 it was no better than the CUDA-core form once that one fetched its rows ahead
// (p = 20, m = 1000, 4096 particles: 699 against 682 us), which also takes the other storage types.
#pragma once

#include "resident.cuh"

namespace subsmc {

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void ldsm4(uint32_t a, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t a, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void mma16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%0, %1, %2, %3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma1688(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, "
      "{%0, %1, %2, %3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

// The same with a zero accumulator on entry.
__device__ __forceinline__ void mma16816_0(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                           uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, "
      "{%8, %9}, {%10, %10, %10, %10};\n"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void mma1688_0(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, "
      "{%7, %7, %7, %7};\n"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a0), "r"(a1), "r"(b0), "f"(0.f));
}

// The upper halves of two floats as a BF16 pair (lo in the lower half).
__device__ __forceinline__ uint32_t hi_pair(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}
__device__ __forceinline__ float hi_part(float v) {
  return __uint_as_float(__float_as_uint(v) & 0xFFFF0000u);
}

// FP64 parts of a particle's Hamiltonians, from the warps that form them to the one that decides.
struct MmaSums {
  double lp0, lp1, like0, S1, S2;  // log priors; a l_hat - a^2/2 sigma2_hat at the start; block sums
  float save[2 * 8 + 2];           // the first pass's sums of e, e^2 by warp, its linear part, shift
  float pad[2];
};

// Shared-memory plan of one CTA (NV 16-byte units of covariates per resident row).
struct MmaPlan {
  int off_consts, off_q, off_warp, off_red, off_reds, off_blk, off_mat, off_k, off_h, total;
};
template <int NV> struct MmaShape {
  static constexpr int CP = 8 * NV;                        // covariate slots
  static constexpr int RB = 16 * (NV % 2 ? NV : NV + 1);   // row pitch: an odd number of units
  static constexpr int NC = (CP + 31) / 32;                // columns per lane
  static constexpr int MT = (NV + 1) / 2;                  // 16-column tiles of the gradient
  // the B operand of D in shared memory: 4 terms (the last one zero) x 4 lanes of a quad x one
  // 32-bit word per unit, padded to whole 128-bit vectors
  static constexpr int BW = (NV + 3) / 4 * 4;
  static constexpr int WB = 4 * 4 * BW * 4 + 8 * CP;  // a warp's operand terms, then delta and rho
};
inline __host__ __device__ int round32(int v) { return (v + 31) & ~31; }

template <int NV> inline MmaPlan mma_plan(int m, int G, int warps) {
  using Sh = MmaShape<NV>;
  MmaPlan P;
  const int mp = round32(m);
  int off = mp * Sh::RB;
  P.off_consts = off;
  off += mp * (int)sizeof(RowC<float>);
  P.off_q = off;  // 64 rows of Q per warp; between trajectories the next rows' indices
  off += warps * 1024;
  P.off_warp = off;
  off += warps * Sh::WB;
  P.off_red = off;  // two buffers of [warps][2][16 MT] gradient partials
  off += 2 * warps * 2 * 16 * Sh::MT * 4;
  P.off_reds = off;  // two buffers of [warps][2] sums of e, e^2
  off = round16(off + 2 * warps * 2 * 4);
  P.off_blk = off;
  off += G * 2 * (int)sizeof(double);
  P.off_mat = off;
  off += 2 * Sh::CP * Sh::CP * 4;  // C and Sigma, zero-padded
  P.off_k = off;
  off = round16(off + (int)sizeof(ResK<float>));
  P.off_h = off;  // MmaSums, then the next particles' draws
  off += (int)sizeof(MmaSums) + kDraws<4> * (int)sizeof(Draws);
  P.total = off;
  return P;
}

// The particle's column constants, one column per lane; loaded when the CTA's problem changes.
template <int NV> struct MmaCols {
  using Sh = MmaShape<NV>;
  bool col[Sh::NC];
  float B[Sh::NC], mu[Sh::NC], iv[Sh::NC], tb[Sh::NC];
  __device__ __forceinline__ void load(const EstArgs &a) {
#pragma unroll
    for (int h = 0; h < Sh::NC; ++h) {
      const int c = (threadIdx.x & 31) + 32 * h;
      col[h] = c < a.p;
      B[h] = col[h] ? ldg_ct<float>(a.B_ct, c) : 0.f;
      mu[h] = col[h] ? ldg_ct<float>(a.mu_ct, c) : 0.f;
      iv[h] = col[h] ? ldg_ct<float>(a.ivar_ct, c) : 0.f;
      tb[h] = col[h] ? ldg_ct<float>(a.tb_ct, c) : 0.f;
    }
  }
};

// The gather of a particle's rows, in chunks of the index buffer (WARPS * 256 indices): the indices
// of rows c0 .. c0 + cap - 1 into us, then (after a wait and a barrier) the rows and their constants
// at the centre (the packed row's tail). Invalid indices are flagged and their rows zeroed. The
// indices are staged first, so no copy waits on a global load.
template <int WARPS>
__device__ __forceinline__ void mma_stage_u(const EstArgs &a, int i, int c0, int32_t *us) {
  const int32_t *u = a.u + (int64_t)i * a.m;
  const int n = min(a.m - c0, WARPS * 256);
  for (int j = threadIdx.x; j < n; j += WARPS * 32) cp_async4(us + j, u + c0 + j);
}
template <int NV, int WARPS>
__device__ __forceinline__ void mma_copy_rows(const EstArgs &a, int c0, const int32_t *us,
                                              unsigned char *rows, RowC<float> *cst) {
  constexpr int RB = MmaShape<NV>::RB, NT = WARPS * 32, nvr = NV + 1;
  constexpr int dj = NT / nvr, dq = NT - dj * nvr;
  const int tid = threadIdx.x;
  const int nvec = round16(a.p * 2) / 16;  // 16-byte units of this problem's rows
  const int n = min(a.m - c0, WARPS * 256);
  const unsigned char *Xp = reinterpret_cast<const unsigned char *>(a.Xp);
  const int64_t pitch = (int64_t)a.S * 2;
  int j = tid / nvr, v = tid - (tid / nvr) * nvr;
  while (j < n) {
    const uint32_t k = (uint32_t)us[j];
    const bool bad = k >= (uint32_t)a.n;  // n < 2^31
    const unsigned char *src = Xp + (int64_t)(bad ? 0u : k) * pitch;
    unsigned char *dst = v < NV ? rows + (c0 + j) * RB + 16 * v
                                : reinterpret_cast<unsigned char *>(cst + c0 + j);
    if (bad || (v >= nvec && v < NV)) {
      *reinterpret_cast<uint4 *>(dst) = make_uint4(0u, 0u, 0u, 0u);
      if (v == 0 && bad) set_err(a.st, kErrIndex);
    } else {  // (the tail follows the covariates)
      cp_async16(dst, src + 16 * (v < NV ? v : nvec));
    }
    j += dj;
    v += dq;
    if (v >= nvr) {
      v -= nvr;
      ++j;
    }
  }
}
// The rest of the gather once the first chunk's indices are visible to the CTA. zero: the CTA's
// problem has changed, so the rows and constants past m (zero for all of its particles) are written.
template <int NV, int WARPS>
__device__ __forceinline__ void mma_gather(const EstArgs &a, int i, bool zero, int32_t *us,
                                           unsigned char *rows, RowC<float> *cst) {
  constexpr int RB = MmaShape<NV>::RB, NT = WARPS * 32;
  const int m = a.m, tid = threadIdx.x;
  mma_copy_rows<NV, WARPS>(a, 0, us, rows, cst);
  for (int c0 = WARPS * 256; c0 < m; c0 += WARPS * 256) {
    __syncthreads();
    mma_stage_u<WARPS>(a, i, c0, us);
    cp_async_wait_all();
    __syncthreads();
    mma_copy_rows<NV, WARPS>(a, c0, us, rows, cst);
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  if (zero) {
    for (int e = m * (RB / 16) + tid; e < round32(m) * (RB / 16); e += NT)
      reinterpret_cast<uint4 *>(rows)[e] = make_uint4(0u, 0u, 0u, 0u);
    for (int e = m + tid; e < round32(m); e += NT) cst[e] = RowC<float>{0.f, 0.f, 0.f, 0.f};
  }
}

// Sum of the W warps' consecutive partials at v (16-byte aligned for W >= 4), in warp order.
template <int W> __device__ __forceinline__ float sum_warps(const float *v) {
  if constexpr (W % 4 == 0) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < W; w += 4) {
      const float4 x = *reinterpret_cast<const float4 *>(v + w);
      s = s + x.x + x.y + x.z + x.w;
    }
    return s;
  } else if constexpr (W == 2) {
    const float2 x = *reinterpret_cast<const float2 *>(v);
    return x.x + x.y;
  } else {
    return v[0];
  }
}

// One particle's trajectory (the steps are those of res_particle, resident.cuh). Its rows are already
// on their way (mma_gather); `an`, `in`, `newp`: the CTA's next particle (an null: none) and whether
// it belongs to another problem. Its rows are gathered as soon as this trajectory has read its
// own for the last time, so they arrive during the FP64 work of this particle's acceptance test.
template <int NV, int WARPS>
__device__ __forceinline__ void mma_particle(const EstArgs &a, int i, bool reload,
                                             const MmaPlan &P, const Draws &draws,
                                             MmaCols<NV> &K, const EstArgs *an, int in,
                                             bool newp) {
  using Sh = MmaShape<NV>;
  constexpr int CP = Sh::CP, RB = Sh::RB, NC = Sh::NC, MT = Sh::MT;
  constexpr int NT = WARPS * 32;
  // the warps that form the log priors, the first pass's likelihood term and the block totals
  // (warp 0: the kinetic energies and the decision)
  constexpr int kWarpP = WARPS > 1 ? 1 : 0, kWarpL = WARPS > 2 ? 2 : kWarpP,
                kWarpB = WARPS > 3 ? 3 : 0;
  extern __shared__ __align__(16) unsigned char smem[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // (warp-uniform to the compiler)
  const int p = a.p, m = a.m, G = a.G;
  RowC<float> *cst = reinterpret_cast<RowC<float> *>(smem + P.off_consts);
  unsigned char *qb = smem + P.off_q + warp * 1024;
  int32_t *us = reinterpret_cast<int32_t *>(smem + P.off_q);
  constexpr int BW = Sh::BW;
  uint32_t *dsp = reinterpret_cast<uint32_t *>(smem + P.off_warp + warp * Sh::WB);
  float *dfl = reinterpret_cast<float *>(dsp + 16 * BW);  // delta of the warp
  float *rfl = dfl + CP;                                  // rho of the warp
  float *red = reinterpret_cast<float *>(smem + P.off_red);
  float *reds = reinterpret_cast<float *>(smem + P.off_reds);
  double *blks = reinterpret_cast<double *>(smem + P.off_blk);
  float *Cs = reinterpret_cast<float *>(smem + P.off_mat);
  float *Sgs = Cs + CP * CP;
  ResK<float> *ks = reinterpret_cast<ResK<float> *>(smem + P.off_k);
  MmaSums *hs = reinterpret_cast<MmaSums *>(smem + P.off_h);
  const float inv_s2 = (float)a.inv_s2;
  const int fam = a.fam;
  const int cv1 = a.cv_order == 1;
  const int g = lane >> 2, q = lane & 3;
  const bool (&col)[NC] = K.col;
  const float (&Bc)[NC] = K.B, (&muc)[NC] = K.mu, (&ivc)[NC] = K.iv, (&tbc)[NC] = K.tb;
  // ldmatrix offsets of this lane within a 64-row group. Rows: tile qq of D (owner lanes q = qq);
  // K-steps (t & 1) of the gradient, and both of a 32-row half for a last single unit.
  uint32_t offD[4], offG[2], offGo;
#pragma unroll
  for (int qq = 0; qq < 4; ++qq) {
    const int row = 32 * ((lane >> 3) & 1) + 8 * qq + (((lane & 7) + 2 * qq) & 7);
    offD[qq] = row * RB + 16 * (lane >> 4);
  }
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int e = (lane & 7) + 8 * (lane >> 4), gg = 4 * t + (e >> 2), qq = e & 3;
    offG[t] = (8 * qq + ((gg + 2 * qq) & 7)) * RB + 16 * ((lane >> 3) & 1);
  }
  {
    const int e = lane & 15, gg = 4 * (lane >> 4) + (e >> 2), qq = e & 3;
    offGo = (8 * qq + ((gg + 2 * qq) & 7)) * RB + 16 * (NV - 1);
  }
  const uint32_t offDo0 = (lane < 16 ? offD[0] : offD[1] - 16) + 16 * (NV - 1);
  const uint32_t offDo1 = (lane < 16 ? offD[2] : offD[3] - 16) + 16 * (NV - 1);
  const uint32_t rows_u = smem_u32(smem), qb_u = smem_u32(qb);
  const int myrow = 8 * q + ((g + 2 * q) & 7);  // + 32 h: the lane's rows of a group
  const int ngrp = (m + 63) >> 6;
  // where this lane's quad sum goes: column g (+ 8) of a 16-column tile
  const int redoff = ((g + 4 * (q & 2)) * 2 + (q & 1)) * WARPS + warp;

  const uint32_t smv = stage_move(a.stage_dev ? a.st->stage : a.stage, a.move);
  if (reload) {
    K.load(a);
    if (tid == 0) {
      ResK<float> k;
      k.temp = a.st->a;
      k.nm = (double)a.n / (double)m;
      k.inv_m = 1.0 / (double)m;
      k.ta = (float)k.temp;
      k.ta2 = (float)(k.temp * k.temp * k.nm * k.nm);
      k.tnm = (float)(k.temp * k.nm);
      k.smv = smv;
      *ks = k;
    }
    for (int e = tid; e < CP * CP; e += NT) {
      const int r = e / CP, c = e - r * CP;
      const bool in_ = r < p && c < p;
      Cs[e] = in_ ? ldg_ct<float>(a.C_ct, r * p + c) : 0.f;
      Sgs[e] = in_ ? ldg_ct<float>(a.Sigma_ct, r * p + c) : 0.f;
    }
    for (int e = lane; e < 16 * BW; e += 32) dsp[e] = 0u;
    __syncthreads();
  }
  const ResK<float> kc = *ks;
  const double temp = kc.temp, nm = kc.nm, inv_m = kc.inv_m;
  const float ta = kc.ta, ta2 = kc.ta2, tnm = kc.tnm;
  // initial momentum rho = Linv' z, in every warp (while the rows arrive)
  float *thg = reinterpret_cast<float *>(a.theta_out) + (int64_t)i * p;
  const float eps = (float)draws.eps;
  const double logU = draws.logU;
  float th[NC], rho[NC], gr[NC], cd[NC];
  {
    const Stream smom(a.seed, kMomentum, smv, (uint32_t)i);
    float z[NC];
#pragma unroll
    for (int h = 0; h < NC; ++h) {
      z[h] = col[h] ? stream_normal_f32(smom, (uint32_t)(lane + 32 * h)) : 0.f;
      rho[h] = 0.f;
    }
#pragma unroll
    for (int hz = 0; hz < NC; ++hz)  // rho_r = sum_{c >= r} Linv[c, r] z_c, c ascending
#pragma unroll 8
      for (int cc = 0; cc < 32 && 32 * hz + cc < p; ++cc) {
        const int c = 32 * hz + cc;
        const float zc = __shfl_sync(0xffffffffu, z[hz], cc);
#pragma unroll
        for (int h = 0; h < NC; ++h) {
          const int r = lane + 32 * h;
          if (col[h] && c >= r) rho[h] = fma(ldg_ct<float>(a.Linv_ct, c * p + r), zc, rho[h]);
        }
      }
#pragma unroll
    for (int h = 0; h < NC; ++h) {
      const int c = lane + 32 * h;
      th[h] = col[h] ? thg[c] : 0.f;
      gr[h] = cd[h] = 0.f;
    }
  }
  // y[c] = sum_k M[k, c] x_k for the warp's vector x in shared memory, even and odd k apart
  auto matvec = [&](const float *Ms, const float *x, float *y) {
    float2 s[NC];
#pragma unroll
    for (int h = 0; h < NC; ++h) s[h] = make_float2(0.f, 0.f);
#pragma unroll
    for (int k0 = 0; k0 < CP; k0 += 4) {
      const float4 xv = *reinterpret_cast<const float4 *>(x + k0);
#pragma unroll
      for (int k = 0; k < 4; k += 2) {
        const float2 xs = k ? make_float2(xv.z, xv.w) : make_float2(xv.x, xv.y);
#pragma unroll
        for (int h = 0; h < NC; ++h) {
          const int c = lane + 32 * h < CP ? lane + 32 * h : 0;
          s[h] = __ffma2_rn(make_float2(Ms[(k0 + k) * CP + c], Ms[(k0 + k + 1) * CP + c]), xs,
                            s[h]);
        }
      }
    }
#pragma unroll
    for (int h = 0; h < NC; ++h) y[h] = s[h].x + s[h].y;
  };
  uint32_t bA0[NV], bA1[NV], bB0[NV], bB1[NV];  // B operand of D: tiles 0, 2 (A) and 1, 3 (B)
  // delta and its three BF16 terms into the warp's buffer; the B operand and C delta from there
  auto set_delta = [&]() {
#pragma unroll
    for (int h = 0; h < NC; ++h) {
      const int c = lane + 32 * h;
      if (c < CP) {
        const float dl = col[h] ? th[h] - tbc[h] : 0.f;
        const float d2 = dl - hi_part(dl), d3 = d2 - hi_part(d2);
        dfl[c] = dl;
        // column c = 8 v + 2 qq + e is half e of word v of quad lane qq
        uint16_t *w = reinterpret_cast<uint16_t *>(dsp) + ((c >> 1 & 3) * BW + (c >> 3)) * 2 +
                      (c & 1);
        w[0] = (uint16_t)(__float_as_uint(dl) >> 16);
        w[8 * BW] = (uint16_t)(__float_as_uint(d2) >> 16);
        w[16 * BW] = (uint16_t)(__float_as_uint(d3) >> 16);
      }
    }
    __syncwarp();
    // operand column n = g: term n & 3 (A) or (n & 3) ^ 2 (B), 3 being zero; tiles 0 and 1 use the
    // columns below 4, tiles 2 and 3 the others
    const int tA = g & 3, tB = tA ^ 2;
    const uint32_t *rA0 = dsp + ((g < 4 ? tA : 3) * 4 + q) * BW;
    const uint32_t *rA1 = dsp + ((g < 4 ? 3 : tA) * 4 + q) * BW;
    const uint32_t *rB0 = dsp + ((g < 4 ? tB : 3) * 4 + q) * BW;
    const uint32_t *rB1 = dsp + ((g < 4 ? 3 : tB) * 4 + q) * BW;
    auto words = [&](const uint32_t *src, uint32_t *dst) {
#pragma unroll
      for (int v = 0; v < NV; v += 4) {
        const uint4 x = *reinterpret_cast<const uint4 *>(src + v);
        dst[v] = x.x;
        if (v + 1 < NV) dst[v + 1] = x.y;
        if (v + 2 < NV) dst[v + 2] = x.z;
        if (v + 3 < NV) dst[v + 3] = x.w;
      }
    };
    words(rA0, bA0);
    words(rA1, bA1);
    words(rB0, bB0);
    words(rB1, bB1);
    matvec(Cs, dfl, cd);
  };
  auto sigma_rho = [&](float *vs) {  // (Sigma rho)_c at the lane's columns
#pragma unroll
    for (int h = 0; h < NC; ++h)
      if (lane + 32 * h < CP) rfl[lane + 32 * h] = rho[h];
    __syncwarp();
    matvec(Sgs, rfl, vs);
    __syncwarp();
  };
  auto kinetic = [&]() -> double {  // rho' Sigma rho / 2 (every lane of the warp)
    float v[NC];
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
  set_delta();
  int buf = 0;
  // shift of the row sums (identical in every warp): the cached subsample mean of d
  float Ksh = 0.f;
  if (a.blk) {
    const double *bc = a.blk + (int64_t)i * G * 2;
    float s0 = 0.f;  // any value near the mean serves
    for (int b = lane; b < G; b += 32) s0 += (float)bc[2 * b];
    Ksh = warp_sum(s0) * (float)inv_m;
    if (!isfinite(Ksh)) Ksh = 0.f;
  }
  double kin0 = 0.0;
  if (warp == 0) kin0 = kinetic();
  if (warp == kWarpP) {
    const double lp = log_prior();
    if (lane == 0) hs->lp0 = lp;
  }
  cp_async_wait_all();
  __syncthreads();  // every warp's copies have landed
  // X delta of the 64-row group at `base`, as the accumulators A (tiles 0, 2) and B (tiles 1, 3)
  auto row_dots = [&](uint32_t base, float (&A)[4], float (&B)[4]) {
#pragma unroll
    for (int kk = 0; kk < NV / 2; ++kk) {
#pragma unroll
      for (int qq = 0; qq < 4; ++qq) {
        uint32_t x[4];
        ldsm4(base + offD[qq] + 32 * kk, x);
        const uint32_t b0 = qq == 0 ? bA0[2 * kk] : qq == 2 ? bA1[2 * kk]
                            : qq == 1 ? bB0[2 * kk] : bB1[2 * kk];
        const uint32_t b1 = qq == 0 ? bA0[2 * kk + 1] : qq == 2 ? bA1[2 * kk + 1]
                            : qq == 1 ? bB0[2 * kk + 1] : bB1[2 * kk + 1];
        if (kk == 0 && qq < 2)
          mma16816_0(qq % 2 ? B : A, x[0], x[1], x[2], x[3], b0, b1);
        else
          mma16816(qq % 2 ? B : A, x[0], x[1], x[2], x[3], b0, b1);
      }
    }
    if constexpr (NV % 2) {  // the last unit of two tiles in one load
#pragma unroll
      for (int hq = 0; hq < 2; ++hq) {
        uint32_t x[4];
        const uint32_t o = hq ? offDo1 : offDo0;
        ldsm4(base + o, x);
        if (NV == 1 && hq == 0) {
          mma1688_0(A, x[0], x[1], bA0[NV - 1]);
          mma1688_0(B, x[2], x[3], bB0[NV - 1]);
        } else {
          mma1688(A, x[0], x[1], hq ? bA1[NV - 1] : bA0[NV - 1]);
          mma1688(B, x[2], x[3], hq ? bB1[NV - 1] : bB0[NV - 1]);
        }
      }
    }
  };
  // D of the lane's two rows: main terms in its own accumulator, the third with its neighbour
  auto own_rows = [&](const float (&A)[4], const float (&B)[4]) -> float2 {
    const bool odd = q & 1;
    const float r0 = __shfl_xor_sync(0xffffffffu, odd ? A[0] : B[0], 1);
    const float r1 = __shfl_xor_sync(0xffffffffu, odd ? A[2] : B[2], 1);
    return make_float2((odd ? B[0] + B[1] : A[0] + A[1]) + r0,
                       (odd ? B[2] + B[3] : A[2] + A[3]) + r1);
  };
  float qlin = 0.f;
  // a l_hat - a^2/2 sigma2_hat, and both estimates, from the shifted sums of a pass (FP64)
  auto like = [&](double S1, double S2, float ql, float shift, double &ell, double &sig) -> double {
    ell = (a.A_dev ? __ldg(a.A_dev) : a.A) + (double)ql + nm * fma((double)m, (double)shift, S1);
    sig = nm * nm * fmax(0.0, S2 - S1 * S1 * inv_m);
    return temp * ell - 0.5 * temp * temp * sig;
  };
  // One estimator pass at the current delta. Every warp ends with the gradient at its lanes; FINAL
  // also fills the block sums blks, and leaves e_j in the constants' first word.
  auto pass = [&](auto full_c, bool final) {
    constexpr bool FULL = decltype(full_c)::value;  // first or last pass: totals wanted
    float acc[MT][4];
#pragma unroll
    for (int t = 0; t < MT; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[t][e] = 0.f;
    float sd = 0.f, sd2 = 0.f;
    auto row_loop = [&](auto famc) {
      constexpr int F = decltype(famc)::value;
      // D of the next group is formed while the current group's terms are evaluated
      float A[4] = {0.f, 0.f, 0.f, 0.f}, B[4] = {0.f, 0.f, 0.f, 0.f};
      if (warp < ngrp) row_dots(rows_u + (uint32_t)(warp * 64) * RB, A, B);
      for (int grp = warp; grp < ngrp; grp += WARPS) {
        const uint32_t base = rows_u + (uint32_t)(grp * 64) * RB;
        const int j0 = grp * 64 + myrow, j1 = j0 + 32;
        const RowC<float> c0 = cst[j0], c1 = cst[j1];
        const float2 D = own_rows(A, B);
        const float D0 = D.x;
        const bool half = grp * 64 + 32 >= m;  // no second half: what lies past the rows is not read
        const float D1 = half ? 0.f : D.y;
        if (grp + WARPS < ngrp) row_dots(base + (uint32_t)(WARPS * 64) * RB, A, B);
        float d0, d1, q0, q1;  // d and r of the two rows
        row_incr<F, float>(c0, D0, inv_s2, d0, q0);
        row_incr<F, float>(c1, D1, inv_s2, d1, q1);
        if (cv1) {
          to_first_order(row_l2<F, float>(c0, inv_s2), D0, d0, q0);
          to_first_order(row_l2<F, float>(c1, inv_s2), D1, d1, q1);
        }
        float e0 = d0 - Ksh, e1 = d1 - Ksh;
        if (grp == ngrp - 1) {  // rows past the subsample
          if (j0 >= m) e0 = q0 = 0.f;
          if (j1 >= m) e1 = q1 = 0.f;
        }
        const float w0 = e0 * q0, w1 = e1 * q1;
        __syncwarp();  // the previous group's Q has been read
        {
          const float a2 = q0 - hi_part(q0), a3 = a2 - hi_part(a2);
          const float b2 = w0 - hi_part(w0), b3 = b2 - hi_part(b2);
          *reinterpret_cast<uint4 *>(qb + 16 * lane) =
              make_uint4(hi_pair(q0, w0), hi_pair(a2, b2), hi_pair(a3, b3), 0u);
          const float f2 = q1 - hi_part(q1), f3 = f2 - hi_part(f2);
          const float h2 = w1 - hi_part(w1), h3 = h2 - hi_part(h2);
          *reinterpret_cast<uint4 *>(qb + 512 + 16 * lane) =
              make_uint4(hi_pair(q1, w1), hi_pair(f2, h2), hi_pair(f3, h3), 0u);
        }
        sd += e0 + e1;
        if (FULL) sd2 = fma(e1, e1, fma(e0, e0, sd2));
        if (FULL && final) {
          if (j0 < m) cst[j0].c0 = e0;
          if (j1 < m) cst[j1].c0 = e1;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t y[4], x[2][NV / 2 + 1][4];
          const uint32_t bh = base + 32 * h * RB;
          if (h == 1 && half) break;
#pragma unroll
          for (int mt = 0; mt < NV / 2; ++mt) {
            ldsm4t(bh + offG[0] + 32 * mt, x[0][mt]);
            ldsm4t(bh + offG[1] + 32 * mt, x[1][mt]);
          }
          if constexpr (NV % 2) ldsm4t(bh + offGo, x[0][NV / 2]);
          if (h == 0) __syncwarp();  // Q is written
          ldsm4t(qb_u + 512 * h + 16 * lane, y);
#pragma unroll
          for (int t = 0; t < 2; ++t)
#pragma unroll
            for (int mt = 0; mt < NV / 2; ++mt)
              mma16816(acc[mt], x[t][mt][0], x[t][mt][1], x[t][mt][2], x[t][mt][3], y[2 * t],
                       y[2 * t + 1]);
          if constexpr (NV % 2) {
            mma16816(acc[MT - 1], x[0][NV / 2][0], 0u, x[0][NV / 2][1], 0u, y[0], y[1]);
            mma16816(acc[MT - 1], x[0][NV / 2][2], 0u, x[0][NV / 2][3], 0u, y[2], y[3]);
          }
        }
      }
    };
    switch (fam) {
      case 0: row_loop(std::integral_constant<int, 0>{}); break;
      case 1: row_loop(std::integral_constant<int, 1>{}); break;
      case 2: row_loop(std::integral_constant<int, 2>{}); break;
      case 3: row_loop(std::integral_constant<int, 3>{}); break;
      default: row_loop(std::integral_constant<int, 4>{}); break;
    }
    // the three terms of (r, e r) are columns (0, 1), (2, 3), (4, 5): sum over the quad, each lane
    // keeping one of the four values (sum r x, sum e r x) x (columns g, g + 8) of a tile
    float *rb = red + buf * WARPS * 2 * 16 * MT;  // [column][sum r x, sum e r x][warp]
    float *rd = reds + buf * WARPS * 2;           // [sum e, sum e^2][warp]
#pragma unroll
    for (int t = 0; t < MT; ++t) {
      const bool hi = q & 2, od = q & 1;
      float k0 = hi ? acc[t][2] : acc[t][0], k1 = hi ? acc[t][3] : acc[t][1];
      k0 += __shfl_xor_sync(0xffffffffu, hi ? acc[t][0] : acc[t][2], 2);
      k1 += __shfl_xor_sync(0xffffffffu, hi ? acc[t][1] : acc[t][3], 2);
      const float v = (od ? k1 : k0) + __shfl_xor_sync(0xffffffffu, od ? k0 : k1, 1);
      rb[redoff + 16 * t * 2 * WARPS] = v;
    }
    const float s1 = warp_sum(sd);
    if (lane == 0) rd[warp] = s1;
    if (FULL) {
      const float s2 = warp_sum(sd2);
      if (lane == 0) rd[WARPS + warp] = s2;
    }
    __syncthreads();  // all warps' partial sums of this pass are in buffer buf
    // sum of e over the subsample (the gradient needs only its mean)
    const float S1f = sum_warps<WARPS>(rd);
    if (FULL && final) {  // shifted block sums of e (floor partition of u into G blocks)
      for (int b = warp; b < G; b += WARPS) {
        const int j0 = block_start(b, m, G), j1 = block_start(b + 1, m, G);
        float bs = 0.f, bq = 0.f;
        for (int j = j0 + lane; j < j1; j += 32) {
          const float ej = cst[j].c0;
          bs += ej;
          bq = fma(ej, ej, bq);
        }
        bs = warp_sum(bs);
        bq = warp_sum(bq);
        if (lane == 0) {
          blks[2 * b] = (double)bs;
          blks[2 * b + 1] = (double)bq;
        }
      }
      __syncthreads();
    }
    // gradient of a l_hat - a^2/2 sigma2_hat + log p(theta) at the lane's columns (every warp)
    const float dbar = S1f * (float)inv_m;  // mean of e
#pragma unroll
    for (int h = 0; h < NC; ++h) {
      const int c = lane + 32 * h;
      const int cr = c < CP ? c : 0;
      const float G1 = sum_warps<WARPS>(rb + cr * 2 * WARPS);
      const float G2 = sum_warps<WARPS>(rb + cr * 2 * WARPS + WARPS);
      gr[h] = col[h] ? ta * (Bc[h] + cd[h]) + tnm * G1 - ta2 * (G2 - dbar * G1) -
                           (th[h] - muc[h]) * ivc[h]
                     : 0.f;
    }
    if (FULL && warp == (final ? 0 : kWarpL)) {  // the linear and quadratic part of l_hat
      float ql = 0.f;
#pragma unroll
      for (int h = 0; h < NC; ++h)
        if (col[h]) ql += (th[h] - tbc[h]) * (Bc[h] + 0.5f * cd[h]);
      qlin = warp_sum(ql);
      if (!final) {  // the first pass's sums, for the FP64 work at the end
        if (lane < 2 * WARPS) hs->save[lane] = rd[lane];
        if (lane == 0) {
          hs->save[16] = qlin;
          hs->save[17] = Ksh;
        }
      }
    }
    if (!FULL || !final) Ksh += dbar;  // the next pass is shifted by this pass's mean of d
    buf ^= 1;
  };

  // trajectory
  pass(std::true_type{}, false);
  for (int l = 0; l < a.L; ++l) {
    float vs[NC];
#pragma unroll
    for (int h = 0; h < NC; ++h) rho[h] += 0.5f * eps * gr[h];
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
    for (int h = 0; h < NC; ++h) rho[h] += 0.5f * eps * gr[h];
  }
  // Metropolis-Hastings. The rows have been read for the last time: the next particle's are fetched
  // under the FP64 terms (slow on this part: a warp-wide FP64 instruction holds its sub-partition's
  // pipe for tens of cycles), which are split over warps on different sub-partitions.
  if (an) mma_stage_u<WARPS>(*an, in, 0, us);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
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
      S1 += (double)hs->save[w];
      S2 += (double)hs->save[WARPS + w];
    }
    const double v = like(S1, S2, hs->save[16], hs->save[17], e0, s0);
    if (lane == 0) hs->like0 = v;
  }
  if (warp == kWarpB) {
    double S1 = 0.0, S2 = 0.0;
    for (int b = lane; b < G; b += 32) {
      S1 += blks[2 * b];
      S2 += blks[2 * b + 1];
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
  if (an) mma_gather<NV, WARPS>(*an, in, newp, us, smem, cst);
  if (warp == 0) {
    double ell, sig;
    const double like1 = like(hs->S1, hs->S2, qlin, Ksh, ell, sig);
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
      for (int b = lane; b < G; b += 32) {
        const double ng = (double)(block_start(b + 1, m, G) - block_start(b, m, G));
        const double se = blks[2 * b], qe = blks[2 * b + 1];
        blk[2 * b] = fma(ng, k, se);
        blk[2 * b + 1] = qe + k * fma(ng, k, 2.0 * se);
      }
      if (lane == 0) {
        a.ell[i] = ell;
        a.sig2[i] = sig;
        atomicAdd(&a.st->acc_theta, 1ull);
      }
    }
  }
}

// CTAs per SM that the registers must leave room for (shared memory sets the same limit at the
// sizes a tile serves by default).
template <int NV, int WARPS> constexpr int mma_min_blocks() { return WARPS >= 8 ? 1 : 2; }

// The first particle's rows of a CTA.
template <int NV, int WARPS>
__device__ __forceinline__ void mma_first(const EstArgs &a, int i, const MmaPlan &P,
                                          unsigned char *smem) {
  int32_t *us = reinterpret_cast<int32_t *>(smem + P.off_q);
  mma_stage_u<WARPS>(a, i, 0, us);
  cp_async_wait_all();
  __syncthreads();
  mma_gather<NV, WARPS>(a, i, true, us, smem,
                        reinterpret_cast<RowC<float> *>(smem + P.off_consts));
}

template <int NV, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, mma_min_blocks<NV, WARPS>())
    k_hmc_mma(EstArgs a, MmaPlan P) {
  extern __shared__ __align__(16) unsigned char smem[];
  Draws *dr = reinterpret_cast<Draws *>(smem + P.off_h + sizeof(MmaSums));
  MmaCols<NV> K;
  if ((int)blockIdx.x < a.B) mma_first<NV, WARPS>(a, a.i0 + (int)blockIdx.x, P, smem);
  int k = 0;
  for (int il = blockIdx.x; il < a.B; il += gridDim.x, ++k) {
    if (k % kDraws<WARPS> == 0) {
      if (k) __syncthreads();
      const int64_t nx = il + (int64_t)threadIdx.x * gridDim.x;
      if (threadIdx.x < kDraws<WARPS> && nx < a.B) dr[threadIdx.x] = theta_draws(a, a.i0 + (int)nx);
      __syncthreads();
    }
    const bool more = (int64_t)il + gridDim.x < a.B;
    mma_particle<NV, WARPS>(a, a.i0 + il, k == 0, P, dr[k % kDraws<WARPS>], K, more ? &a : nullptr,
                            a.i0 + il + (int)gridDim.x, false);
  }
}

// All particles of the problems of a batch that share one tile (k_hmc_res_batch, resident.cuh).
template <int NV, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, mma_min_blocks<NV, WARPS>())
    k_hmc_mma_batch(BatchArgs b, MmaPlan P) {
  extern __shared__ __align__(16) unsigned char smem[];
  Draws *dr = reinterpret_cast<Draws *>(smem + P.off_h + sizeof(MmaSums));
  MmaCols<NV> K;
  int qcur = -1, k = 0, pr = 0;
  if ((int)blockIdx.x < b.total) {
    pr = batch_problem(b.offsets, b.nprob, blockIdx.x);
    mma_first<NV, WARPS>(b.probs[pr], (int)blockIdx.x - b.offsets[pr], P, smem);
  }
  for (int gi = blockIdx.x; gi < b.total; gi += gridDim.x, ++k) {
    if (k % kDraws<WARPS> == 0) {
      if (k) __syncthreads();
      const int64_t gn = gi + (int64_t)threadIdx.x * gridDim.x;
      if (threadIdx.x < kDraws<WARPS> && gn < b.total) {
        const int pn = batch_problem(b.offsets, b.nprob, (int)gn);
        dr[threadIdx.x] = theta_draws(b.probs[pn], (int)gn - b.offsets[pn]);
      }
      __syncthreads();
    }
    const int64_t gn = (int64_t)gi + gridDim.x;
    const int pn = gn < b.total ? batch_problem(b.offsets, b.nprob, (int)gn) : pr;
    mma_particle<NV, WARPS>(b.probs[pr], gi - b.offsets[pr], pr != qcur, P, dr[k % kDraws<WARPS>], K,
                            gn < b.total ? &b.probs[pn] : nullptr, (int)gn - b.offsets[pn],
                            pn != pr);
    qcur = pr;
    pr = pn;
  }
}

// Resident grid of a kernel with `smem` bytes of dynamic shared memory (0: it does not fit).
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
inline int launch_mma(const EstArgs &a, cudaStream_t s, int sms, bool dry) {
  if (a.p > 8 * NV) return -2;
  const MmaPlan P = mma_plan<NV>(a.m, a.G, WARPS);
  const int per_sm = resident_blocks(k_hmc_mma<NV, WARPS>, WARPS * 32, P.total);
  if (per_sm < 1) return -2;
  if (dry || a.B <= 0) return 0;
  const int grid = a.B < per_sm * sms ? a.B : per_sm * sms;
  k_hmc_mma<NV, WARPS><<<grid, WARPS * 32, P.total, s>>>(a, P);
  return (int)cudaGetLastError();
}

template <int NV, int WARPS>
inline int launch_mma_batch(const BatchArgs &b, int p_max, int m_max, int G_max, cudaStream_t s,
                            int sms, bool dry) {
  if (p_max > 8 * NV) return -2;
  const MmaPlan P = mma_plan<NV>(m_max, G_max, WARPS);
  const int per_sm = resident_blocks(k_hmc_mma_batch<NV, WARPS>, WARPS * 32, P.total);
  if (per_sm < 1) return -2;
  if (dry || b.total <= 0) return 0;
  const int grid = b.total < per_sm * sms ? b.total : per_sm * sms;
  k_hmc_mma_batch<NV, WARPS><<<grid, WARPS * 32, P.total, s>>>(b, P);
  return (int)cudaGetLastError();
}

}  // namespace subsmc
