// recon_fixed.cuh -- the FP64 path's reconstruction (steps 1-6 of recon.cuh, conserved variables)
// with its inner products in integer arithmetic.
//
// The FP64 pipe of this GPU retires about 2 lanes per clock and SM, the integer multiply-add
// (32 x 32 + 64 bits) 60: an inner product of 57-bit integers costs three of those, a tenth of the
// FP64 time. The products with the central least-squares operators and with the face-point basis are
// therefore taken over block fixed-point numbers: both factors are integers of 57 bits and a sign
// relative to the largest of their block, x = h 2^29 + l with |h| <= 2^28, |l| <= 2^28, and
//   sum x y = 2^58 sum h h' + 2^29 sum (h l' + l h') + sum l l',
// whose first two sums fit 64-bit accumulators exactly for up to 56 terms. The last one, below
// 2^-58 of the block maxima per term, is dropped: an FP64 product rounds at 2^-53 of itself.
//   operators   the central ones, per row (unknown) of a cell, scaled by the set-up kernel to the row's largest entry;
//   U_m - U_0   exact differences of the FP64 means (modulo 2^64) in units of 2^-57 of a bound of the
//               variable's range over the stencil, which a first pass takes from the high words;
//   face values the coefficients against the largest |a_k| max|phi_k|, the table per basis function.
// Ranges and coefficients keep their places from 2^-950 on, lose them one by one below and are zero below 2^-1007.
// The coefficients are those of a basis orthonormal in the smoothness form (O = L L^T, b = L^T a,
// phi' = L^-1 phi, folded into the operators at set-up), so that an indicator (eq. 15) is a sum of K-1
// squares instead of (K-1)(K+2)/2 products. p_1 and U_0 + p stay FP64.
//
// The directional products stay FP64 too. A cell beside a jump drops the central stencil and keeps directional
// ones on its own side, whose differences may be any fraction of the central stencil's range: in its unit they
// lost their last places, 3e-11 of the low side's means at a jump of 1e6 and 3e-7 at 1e10 (2D degree 3; now 2e-16 at
// both, as without a jump). Where the central polynomial is kept, its values are three times as close to exact sums as
// FP64 products are, of the largest mean of the stencil (up to 2.8 times as far, at most 5e-16 of it, if only the
// stencil's least weighted member is across a jump). The FP64 directional products cost 0 to 4 us a launch of those below,
// most at degree 5, where each of 150 takes the FP64 pipe for 64 clocks of a lone warp.
//
// The selection (eqs. 19-23) and the positivity test only yield decisions: they are taken in FP32
// where they hold by a margin far above its error, and in FP64 as printed elsewhere.
//
// Schedule: variable per lane, as recon_lane, one tile per warp. The operators stream through the warp's
// ring of shared-memory stages, one bulk copy per chunk (tiles.h), issued before the previous kernel has
// ended: read from global memory they cost twice the time, at 8 to 16 warps per SM. The
// FP64 differences of the directional members (the first slots of the stencil list) wait in shared
// memory between the two products.
//
// Measured per launch against the FP64 schedules it replaced (bound by the FP64 pipe, 61 to 86 % of its
// rate): 2D degree 3, 131 072 cells 534 -> 121 us; 3D degree 3, 24 576 cells 432 (553 in blocks of 128) -> 131
// us; 2D degree 5, 4200 cells 81 -> 41 us; 2D degree 2, 2048 cells 19 (51 in blocks of 128) -> 11 us. It is
// now bound by the integer pipe (shifts and 64-bit sums of the conversions, 63 % busy at 2D degree 3), the
// small meshes by the length of a warp's chain.
#pragma once

#include "recon.cuh"
#include "tiles.h"

namespace cteno {

// acc += a b, 32 x 32 + 64 bits (one instruction; from C++ the widened operands can become a 64 x 64
// product of several).
__device__ __forceinline__ void fx_mac(int64_t &acc, const int a, const int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}
// x = h 2^29 + l, |l| <= 2^28, from x + 2^28.
__device__ __forceinline__ int2 fx_split(const int64_t t) {
  return make_int2((int)(t >> 29), (int)((uint32_t)t & 0x1FFFFFFFu) - (1 << 28));
}

// u in units of 2^(e - 1079) less `base`, e the biased exponent of the unit's block, modulo 2^64, truncated
// (a value far below the unit gives 0; e >= 64, so zeros and subnormals do).
__device__ __forceinline__ int64_t fx_of(const double u, const int e, const int64_t base) {
  const int hi = __double2hiint(u);
  const uint64_t m = ((uint64_t)((hi & 0xFFFFF) | 0x100000) << 32) | (uint32_t)__double2loint(u);
  const int s = ((hi >> 20) & 0x7FF) - e + 4;
  uint64_t f;
  asm("shl.b64 %0, %1, %2;" : "=l"(f) : "l"(m), "r"(max(s, 0)));
  asm("shr.u64 %0, %1, %2;" : "=l"(f) : "l"(f), "r"(max(-s, 0)));
  const int64_t sg = hi >> 31;
  return (int64_t)(f ^ (uint64_t)sg) - sg - base;
}

// (A1 2^29 + A2) 2^x rounded to FP64, from its integer part in units of 2^(x + 29) (what lies below is less
// than the last places of the factors' integers); 0 outside the normal numbers.
__device__ __forceinline__ double fx_to_double(int64_t A1, const int64_t A2, const int x) {
  A1 += A2 >> 29;
  const uint32_t sg = (uint32_t)(A1 >> 63);
  uint32_t w1 = (uint32_t)(A1 >> 32) ^ sg, w0 = (uint32_t)A1 ^ sg;  // the magnitude, less one unit when negative
  int e = 63 + 29 + 1022 + x;  // biased exponent less one of a leading bit 31 of w1
  if (w1 == 0u) w1 = w0, w0 = 0u, e -= 32;
  const int c = __clz((int)w1);
  const uint32_t mh = __funnelshift_l(w0, w1, c), ml = w0 << (c & 31);
  e -= c;
  const uint64_t b = ((((uint64_t)mh << 32) | ml) >> 11) + ((ml >> 10) & 1u) + ((uint64_t)(uint32_t)e << 52);
  const bool ok = (uint32_t)e <= 2045u && mh != 0u;
  return __hiloint2double(ok ? (int)((uint32_t)(b >> 32) | (sg & 0x80000000u)) : 0, ok ? (int)(uint32_t)b : 0);
}

// x truncated to FP32, 0 below its normal range, infinite above it (and for non-finite x).
__device__ __forceinline__ float fx_float(const double x) {
  const uint32_t H = (uint32_t)__double2hiint(x), e = (H >> 20) & 0x7FFu;
  uint32_t b = __funnelshift_l((uint32_t)__double2loint(x), H, 3) - (384u << 23);
  b = (e < 897u) ? 0u : (e > 1150u) ? 0x7F800000u : b;
  return __uint_as_float(b | (H & 0x80000000u));
}

// The decisions of select_fp64 from FP32 indicators (sums of squares, good to 4e-6), where every
// chi_s is off C_T by more than 3 %: the base-2 logarithms of gamma_s (as in select_fp32) are good to
// 5e-4 (2^-22 of at most 127, times 6), those of CTENOZ where the mean difference of the indicators
// is known to 0.2 %, or gamma_s - 1 is below 2^-12 either way. False where that does not hold, or
// near the limits of FP32: select_fp64 then decides.
template <int NF, int SCHEME>
__device__ __forceinline__ bool select_sure(const KArgs &a, const float SI0, const float (&SId)[NF],
                                            const uint32_t adm, const int stn, uint32_t &bits) {
  const float log2lams = pick<NF>(a.log2_lams_f, stn - 1), eps = (float)a.eps;
  float l0 = SI0 + eps, ld[NF], top = l0, low = l0;
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    ld[f] = SId[f] + eps;
    if ((adm >> f) & 1u) top = fmaxf(top, ld[f]), low = fminf(low, ld[f]);
    ld[f] = lg2_approx(ld[f]);
  }
  l0 = lg2_approx(l0);
  bool sure = top < 1e37f && low > 1e-30f;
  float L0, Ld[NF];
  if constexpr (SCHEME == 0) {
    L0 = -6.0f * l0;
#pragma unroll
    for (int f = 0; f < NF; ++f) Ld[f] = -6.0f * ld[f];
  } else {
    float acc = 0.0f, sum = 0.0f;
#pragma unroll
    for (int f = 0; f < NF; ++f)
      if ((adm >> f) & 1u) acc += fabsf(SId[f] - SI0), sum += SId[f] + SI0;
    const float err = 4e-6f * sum;
    const float lt6 = 6.0f * lg2_approx((acc + err) * pick<NF>(a.inv_stm1_f, stn - 1));
    float xmax = -INFINITY;
    auto l1p = [](float x) {
      return (x > 0.0f) ? x + lg2_approx(1.0f + ex2_approx(-x)) : lg2_approx(1.0f + ex2_approx(x));
    };
    auto gam = [&](float ls) {
      const float x = a.ctenoz_form == 0 ? lt6 - ls : lt6 - 6.0f * ls;
      xmax = fmaxf(xmax, x);
      return l1p(x);
    };
    L0 = gam(l0);
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      Ld[f] = 0.0f;
      if ((adm >> f) & 1u) Ld[f] = gam(ld[f]);
    }
    sure = sure && (err <= 0.002f * acc || xmax < -12.0f);
  }
  if (a.lam_gamma) {
    L0 += a.log2_lam1;
#pragma unroll
    for (int f = 0; f < NF; ++f) Ld[f] += log2lams;
  }
  float Lmax = L0;
#pragma unroll
  for (int f = 0; f < NF; ++f)
    if ((adm >> f) & 1u) Lmax = fmaxf(Lmax, Ld[f]);
  const float e0 = ex2_approx(L0 - Lmax);
  float ed[NF], sum = e0;
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    ed[f] = ex2_approx(Ld[f] - Lmax);
    if ((adm >> f) & 1u) sum += ed[f];
  }
  const float cut = a.C_T32 * sum, below = cut > 1e-35f ? 0.97f * cut : -1.0f, above = 1.03f * cut;
  bits = (e0 > above) ? 1u : 0u;
  sure = sure && (e0 < below || e0 > above);
#pragma unroll
  for (int f = 0; f < NF; ++f)
    if ((adm >> f) & 1u) {
      sure = sure && (ed[f] < below || ed[f] > above);
      bits |= (ed[f] > above) ? 2u << f : 0u;
    }
  return sure;
}

template <int D, int R, int SCHEME>
__global__ void __launch_bounds__(128, TileShape<D, R, 8>::BLOCKS) recon_fixed_kernel(const KArgs a) {
  using S = TileShape<D, R, 8>;
  constexpr int NV = S::NV, NVP = S::NVP, NF = S::NF, NK = S::NK, M = S::M, NQ = S::NQ, NP = S::NP;
  constexpr int KD = S::KD, ND = S::ND, PDS = S::PDS, G = S::G, SLOTS = S::SLOTS, CPW = S::CPW;
  constexpr int MC = S::MC, NCH = S::NCH, NST = S::NST, NKP = S::NKP;
  extern __shared__ __align__(128) unsigned char smem[];
  const int4 *const sPhi = reinterpret_cast<const int4 *>(smem);
  uint64_t *const tbar = reinterpret_cast<uint64_t *>(smem + S::PHI_BYTES);  // the block's: face table
  unsigned char *const wmem = smem + S::PHI_BYTES + 16 + (threadIdx.x >> 5) * S::WARP_BYTES;
  double *const sdel = reinterpret_cast<double *>(wmem + S::HDR + NST * S::STAGE) + (threadIdx.x & 31);
  uint64_t *const bar = reinterpret_cast<uint64_t *>(wmem + S::HDR + NST * S::STAGE + S::DELTA);  // header, stages, test hook
  const int lane = threadIdx.x & 31, grp = lane / NV, v = lane - grp * NV, base = grp * NV;
  const int64_t N = a.N;
  const int64_t tile = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), c0 = tile * CPW;
  const int n = (int)max((int64_t)0, min((int64_t)CPW, N - c0));  // the warp's cells
  auto issue = [&](int c) {  // lane 0: chunk c of the warp's tile
    uint64_t *b = &bar[1 + c % NST];
    mbar_arrive_expect_tx(b, S::STAGE);
    bulk_copy_g2s(wmem + S::HDR + (c % NST) * S::STAGE, (const unsigned char *)a.Pc + (tile * NCH + c) * S::STAGE,
                  S::STAGE, b);
  };
  // the operators do not depend on the previous kernel: their copies start here
  if (lane == 0) {
    for (int b = 0; b < 2 + NST; ++b) mbar_init(&bar[b], 1);
    if (threadIdx.x == 0) mbar_init(tbar, 1);
    fence_barrier_init();
    if (S::PHI_BYTES && threadIdx.x == 0) {
      mbar_arrive_expect_tx(tbar, S::PHI_BYTES);
      bulk_copy_g2s(smem, a.phifx, S::PHI_BYTES, tbar);
    }
    if (n > 0) {
      mbar_arrive_expect_tx(&bar[0], (uint32_t)(CPW * M * 4 + n * NF * PDS * 8));
      bulk_copy_g2s(wmem + S::HPD, a.st + c0 * M, (uint32_t)(CPW * M * 4), &bar[0]);
      bulk_copy_g2s(wmem, (const double *)a.Pd + c0 * (NF * PDS), (uint32_t)(n * NF * PDS * 8), &bar[0]);
      for (int c = 0; c < NST; ++c) issue(c);
    }
  }
  __syncthreads();
  const bool active = grp < n;
  const int slot = active ? grp : max(n, 1) - 1;  // spare lanes shadow a valid cell and store nothing
  const int64_t i = min(c0 + slot, N - 1);
  const uint32_t info = __ldg(a.cinfo + i);
  const int8_t *__restrict__ ei = a.Pe + i * kFixExp;
  pdl_wait(a);  // the state written by the previous stage's update
  if (a.dt_swap && blockIdx.x == 0)  // the CFL step: dt[next] -> dt[cur]
    for (int t = threadIdx.x; t < a.nmesh; t += blockDim.x) {
      a.dt[t] = a.dt[a.nmesh + t];
      a.dt[a.nmesh + t] = 1e300;
    }
  // a bounded wait of the whole warp for its copies; on a timeout the warp reports it, gives the
  // copies in flight (chunks c up to `last`) a second bounded wait and stops
  auto arrived = [&](uint64_t *b, uint32_t parity, int c, int last, uint64_t limit_ns = kStageWaitNs) {
    const bool ok = mbar_wait(b, parity, limit_ns);
    if (!__any_sync(0xffffffffu, !ok)) return true;
    if (lane == 0) {
      atomicOr(a.err, kErrTimeout);
      if (S::PHI_BYTES) mbar_wait(tbar, 0, kStageWaitNs);
      if (n > 0) mbar_wait(&bar[0], 0, kStageWaitNs);
      for (; n > 0 && c < last; ++c) mbar_wait(&bar[1 + c % NST], (uint32_t)((c / NST) & 1), kStageWaitNs);
    }
    __syncwarp();
    return false;
  };
  if (n == 0) {  // a warp past the last cell; the block's copy may be its own
    if (S::PHI_BYTES) arrived(tbar, 0, 0, 0);
    return;
  }
  // test hook: a bounded wait on a barrier that nothing completes runs out
  if (a.test_wait_ns && !arrived(&bar[1 + NST], 0, 0, NST, a.test_wait_ns)) return;
  const double *__restrict__ Uv = after_wait(a.U) + v;
  const int32_t *__restrict__ sti = reinterpret_cast<const int32_t *>(wmem + S::HPD) + slot * M;
  const double U0 = __ldg(Uv + i * NVP);
  auto ids_of = [&](int m, int (&j)[G]) {
    if constexpr (G == 4) {
      const int4 t = *reinterpret_cast<const int4 *>(sti + m);
      j[0] = t.x, j[1] = t.y, j[2] = t.z, j[3] = t.w;
    } else {
#pragma unroll
      for (int g = 0; g < G; g += 2) {
        const int2 t = *reinterpret_cast<const int2 *>(sti + m + g);
        j[g] = t.x, j[g + 1] = t.y;
      }
    }
  };

  if (!arrived(&bar[0], 0, 0, NST)) return;
  // the range of variable v over the stencil, from the high words in the order of the values
  auto key = [](int h) { return h ^ ((h >> 31) & 0x7FFFFFFF); };
  int kmax = key(__double2hiint(U0)), kmin = kmax;
#pragma unroll (M <= 20 ? M / G : 3)
  for (int m = 0; m < M; m += G) {
    int j[G];
    ids_of(m, j);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const int k = key(__ldg(reinterpret_cast<const int *>(Uv + (int64_t)j[g] * NVP) + 1));
      kmax = max(kmax, k);
      kmin = min(kmin, k);
    }
  }
  double range = __hiloint2double(key(kmax), kmax < 0 ? 0 : -1) - __hiloint2double(key(kmin), kmin < 0 ? -1 : 0);
  // where the range is so small that the high words overestimate it by more than 2^-8, from the whole means: the
  // decisions depend on ratios of indicators, so the differences need their own relative accuracy
  const int eu = (max(kmax, ~kmin) >> 20) & 0x7FF;
  const bool near = ((__double2hiint(range) >> 20) & 0x7FF) < eu - 12;
  if (__any_sync(0xffffffffu, near)) {
    auto key64 = [](double u) {
      const long long b = __double_as_longlong(u);
      return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFll);
    };
    long long lmax = key64(U0), lmin = lmax;
#pragma unroll 1
    for (int m = 0; m < M; m += G) {
      int j[G];
      ids_of(m, j);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const long long k = key64(__ldg(Uv + (int64_t)j[g] * NVP));
        lmax = max(lmax, k);
        lmin = min(lmin, k);
      }
    }
    auto value = [](long long k) { return __longlong_as_double(k ^ ((k >> 63) & 0x7FFFFFFFFFFFFFFFll)); };
    if (near) range = value(lmax) - value(lmin);  // a lane's unit depends on its own stencil only
  }
  const int er = max((__double2hiint(range) >> 20) & 0x7FF, 64);  // |U_m - U_0| < 2^(er - 1022)
  // a non-finite member makes every central coefficient NaN
  const bool finite = kmax < 0x7FF00000 && kmin > (int)0x800FFFFF && er < 0x7FF;
  // means near the largest numbers: central coefficients in units of 2^200, taken back by `scale`, so that what does
  // not fit becomes infinite in a face value (the guard's case) and not zero in a coefficient
  const bool top_range = finite && er > 1900;
  const int64_t F0 = fx_of(U0, er, 1 << 28);

  // central coefficients b = P_c (U_m - U_0)
  double ao[NK];
  {
    int64_t A1[NK], A2[NK];
#pragma unroll
    for (int k = 0; k < NK; ++k) A1[k] = A2[k] = 0;
    const int4 *pc = nullptr;
    double un[G];  // the next group's means
    {
      int j[G];
      ids_of(0, j);
#pragma unroll
      for (int g = 0; g < G; ++g) un[g] = __ldg(Uv + (int64_t)j[g] * NVP);
    }
#pragma unroll 1
    for (int m = 0; m < M; m += G) {
      const int c = m / MC;
      int2 dx[G];
#pragma unroll
      for (int g = 0; g < G; ++g) {
        dx[g] = fx_split(fx_of(un[g], er, F0));
        if (m + g < SLOTS) sdel[(m + g) * 32] = un[g] - U0;
      }
      if (m + G < M) {
        int j[G];
        ids_of(m + G, j);
#pragma unroll
        for (int g = 0; g < G; ++g) un[g] = __ldg(Uv + (int64_t)j[g] * NVP);
      }
      if (m % MC == 0) {
        if (!arrived(&bar[1 + c % NST], (uint32_t)((c / NST) & 1), c, min(c + NST, NCH))) return;
        pc = reinterpret_cast<const int4 *>(wmem + S::HDR + (c % NST) * S::STAGE + slot * (MC * NK * 8));
      }
#pragma unroll
      for (int e = 0; e < G * NK / 2; ++e) {
        const int4 p = *pc++;
        const int ph[2] = {p.x, p.z}, pl[2] = {p.y, p.w};
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const int k = (2 * e + t) % NK, g = (2 * e + t) / NK;
          fx_mac(A1[k], ph[t], dx[g].x);
          fx_mac(A2[k], ph[t], dx[g].y);
          fx_mac(A2[k], pl[t], dx[g].x);
        }
      }
      if (NST < NCH && (m + G) % MC == 0 && c + NST < NCH) {
        __syncwarp();  // every lane is done with this stage
        if (lane == 0) {
          fence_proxy_async_shared();
          issue(c + NST);
        }
      }
    }
    // P = h 2^29 + l in units of 2^(E_k - 57), the differences in units of 2^(er - 1079)
#pragma unroll
    for (int k = 0; k < NK; ++k) ao[k] = fx_to_double(A1[k], A2[k], 29 - 57 - 1079 - (top_range ? 200 : 0) + er + __ldg(ei + k));
  }
  // directional coefficients: the members of face f are the next slots of the list
  const uint32_t adm = (info >> kInfoAdmShift) & 0xFu;
  const double *__restrict__ Pdi = reinterpret_cast<const double *>(wmem) + slot * (NF * PDS);
  double ad[NF][KD];
  {
    int off = 0;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const int nm = (info >> (4 * f)) & 15u;
#pragma unroll
      for (int k = 0; k < KD; ++k) ad[f][k] = 0.0;
      if ((adm >> f) & 1u) {
#pragma unroll
        for (int jj = 0; jj < ND; jj += 2) {
          if (jj < nm) {
            const double d0 = sdel[(off + jj) * 32], d1 = jj + 1 < nm ? sdel[(off + jj + 1) * 32] : 0.0;
#pragma unroll
            for (int c = 0; c < KD; ++c) {
              const double2 p = reinterpret_cast<const double2 *>(Pdi + f * PDS + jj * KD)[c];
              const int k = (2 * c) % KD, l = (2 * c + 1) % KD;
              ad[f][k] = fma(p.x, 2 * c / KD ? d1 : d0, ad[f][k]);
              ad[f][l] = fma(p.y, (2 * c + 1) / KD ? d1 : d0, ad[f][l]);
            }
          }
        }
      }
      off += nm;
    }
  }
  if (!finite) {
#pragma unroll
    for (int k = 0; k < NK; ++k) ao[k] = __longlong_as_double(0x7FF8000000000000ll);
  }

  // p_1 (eq. 17) without its factor 1 / lambda_1, which goes to the face values (`scale`)
  const int stn = 1 + __popc(adm);
  const bool split = stn > 1 && a.central_split;
  if (split) {
    const double lams = pick<NF>(a.lams_d, stn - 1) * (top_range ? 0x1p-200 : 1.0);
#pragma unroll
    for (int k = 0; k < KD; ++k) {
      double s = ad[0][k];
#pragma unroll
      for (int f = 1; f < NF; ++f) s += ad[f][k];
      ao[k] -= lams * s;
    }
  }
  double scale = split ? a.inv_lam1 : 1.0;
  if (top_range) scale *= 0x1p200;
  // the indicators (eq. 15) and the selection (eqs. 19-23) or the weights (eq. 14)
  uint32_t bits = 0u;
  bool sure = false;
  if (!a.cweno && !top_range) {
    float s0 = 0.0f, sd[NF];
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const float x = fx_float(ao[k]);
      s0 += x * x;
    }
    if (split) s0 *= a.inv_lam1_32 * a.inv_lam1_32;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      sd[f] = 0.0f;
#pragma unroll
      for (int k = 0; k < KD; ++k) {
        const float x = fx_float(ad[f][k]);
        sd[f] += x * x;
      }
    }
    sure = select_sure<NF, SCHEME>(a, s0, sd, adm, stn, bits);
  }
  if (!sure) {
    double SI0 = 0.0, SId[NF];
#pragma unroll
    for (int k = 0; k < NK; ++k) SI0 += ao[k] * ao[k];
    SI0 *= scale * scale;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      SId[f] = 0.0;
#pragma unroll
      for (int k = 0; k < KD; ++k) SId[f] += ad[f][k] * ad[f][k];
    }
    const double lams = pick<NF>(a.lams_d, stn - 1);
    if (a.cweno) {
      double w0, wd[NF];
      cweno_weights<NF>(SI0, SId, adm, a.lam1, lams, a.eps, w0, wd);
#pragma unroll
      for (int k = 0; k < NK; ++k) ao[k] *= w0 * scale;
#pragma unroll
      for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int k = 0; k < KD; ++k) ao[k] += wd[f] * ad[f][k];
      scale = 1.0;
      bits = 1u | (adm << 1);
    } else {
      bits = select_fp64<NF>(SI0, SId, adm, stn, SCHEME, a.ctenoz_form, a.lam_gamma, a.lam1, lams, a.eps, a.C_T);
    }
  }
  if (!(bits & 1u)) {  // the mean of the selected directional polynomials (none selected: p = 0)
    scale = bits ? 1.0 / (double)__popc(bits >> 1) : 1.0;
#pragma unroll
    for (int k = 0; k < NK; ++k) ao[k] = 0.0;
#pragma unroll
    for (int f = 0; f < NF; ++f)
      if ((bits >> (1 + f)) & 1u) {
#pragma unroll
        for (int k = 0; k < KD; ++k) ao[k] += ad[f][k];
      }
  } else if (!a.cweno) {
    bits = 1u;
  }
  if (a.flags && active) a.flags[v * N + i] = (uint8_t)bits;

  // face values U_0 + sum_k b_k phi'_k: the coefficients in units of the largest |b_k| max |phi'_k|, which keep all
  // their places from 2^-950 on (phi_exp is 1 at most)
  int ef = 72;
#pragma unroll
  for (int k = 0; k < NK; ++k) ef = max(ef, ((__double2hiint(ao[k]) >> 20) & 0x7FF) + a.phi_exp[k]);
  bool nan = false;
  int2 bx[NK];
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    nan = nan || ((__double2hiint(ao[k]) >> 20) & 0x7FF) == 0x7FF;
    bx[k] = fx_split(fx_of(ao[k], ef - a.phi_exp[k], -(1 << 28)));
  }
  const uint32_t perm = info >> kInfoPermShift;
  double *__restrict__ Ufi = (double *)a.Uf + i * (int64_t)(NF * NQ * NV) + v;
  auto slot_of = [&](int f, int q) {  // 2D: edge points in sorted-vertex order
    return (f * NQ + ((D == 2 && ((perm >> (3 * f)) & 7u)) ? NQ - 1 - q : q)) * NV;
  };
  float low = INFINITY;  // bounds of the face values in FP32: the smallest, the bits of the largest magnitude
  uint32_t top = 0u;
  if (S::PHI_BYTES && !arrived(tbar, 0, NCH, NCH)) return;
#pragma unroll 1  // straight-line code for every face would not fit the instruction cache
  for (int f = 0; f < NF; ++f) {
    const int p = D == 3 ? (perm >> (3 * f)) & 7u : 0;
    const int4 *__restrict__ ph = (S::PHI_BYTES ? sPhi : reinterpret_cast<const int4 *>(a.phifx)) + (f * NP + p) * (NQ * NKP / 2);
    int64_t A1[NQ], A2[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) A1[q] = A2[q] = 0;
#pragma unroll
    for (int k = 0; k < NK; k += 2)
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        int4 x;
        if constexpr (S::PHI_BYTES > 0) x = ph[(q * NKP + k) / 2];
        else x = __ldg(ph + (q * NKP + k) / 2);
        fx_mac(A1[q], x.x, bx[k].x);
        fx_mac(A2[q], x.x, bx[k].y);
        fx_mac(A2[q], x.y, bx[k].x);
        if (k + 1 < NK) {
          fx_mac(A1[q], x.z, bx[k + 1].x);
          fx_mac(A2[q], x.z, bx[k + 1].y);
          fx_mac(A2[q], x.w, bx[k + 1].x);
        }
      }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double val = fx_to_double(A1[q], A2[q], 29 - 57 - 1079 + ef);
      if (nan) val = __longlong_as_double(0x7FF8000000000000ll);
      val = fma(val, scale, U0);
      if (active) Ufi[slot_of(f, q)] = val;
      const float x = fx_float(val);
      low = fminf(low, x);
      top = max(top, __float_as_uint(x) & 0x7FFFFFFFu);
    }
  }
  // positivity of every point from those bounds, rho E - |m|^2 / 2 >= min rho min E - max |m|^2 / 2, with a margin
  // of 1e-5 of rho E (its rounding: 1e-6)
  const float rho = __shfl_sync(0xffffffffu, low, base), E = __shfl_sync(0xffffffffu, low, base + NV - 1);
  float ke = 0.0f;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const float m = __uint_as_float(__shfl_sync(0xffffffffu, top, base + 1 + j));
    ke += m * m;
  }
  const float rE = rho * E;
  const bool doubt = !(top < 0x7F800000u && rho > 1e-30f && E > 0.0f && rE > 1e-30f && rE - 0.5f * ke > 1e-5f * rE);
  if (a.guard_on && __any_sync(0xffffffffu, doubt && active)) {
    bool bad = false;
    for (int f = 0; f < NF; ++f)
      for (int q = 0; q < NQ; ++q) {
        const double val = active ? Ufi[slot_of(f, q)] : U0;  // this lane's own store
        const bool pb = lane_point_bad<D, double>(a, val, base);  // every lane shuffles
        bad = bad || pb;
      }
    if (bad && active) {
      for (int f = 0; f < NF; ++f)
        for (int q = 0; q < NQ; ++q) Ufi[slot_of(f, q)] = U0;
      if (v == 0) atomicAdd(a.guard, 1ull);
    }
  }
}

}  // namespace cteno
