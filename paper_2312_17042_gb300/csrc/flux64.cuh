// flux64.cuh -- the flux and stage update of the FP64 path (included by flux.cu after boundary_state,
// the time-step reduction and TwoSum helpers).
//
// Both kernels are bound by the FP64 pipe, which takes a warp instruction every 64 clocks per
// scheduler whatever its other load, so they keep that pipe to the formulas and spread them over as many warps as
// the mesh gives:
//   face_flux64    one lane per face Gauss point (not per face): HLLC once per face in its owner's
//                  orientation, comparisons and selections on integers, square roots from the hardware estimate
//                  (sqrt64.cuh); the points of a face are exchanged by shuffles and summed in order;
//   cell_update64  one lane per conserved variable: the cell's face fluxes, signed, in face order,
//                  the Runge-Kutta update and, over the same lanes, the CFL step (IEEE division and root).
// The per-cell schedules of the mixed path evaluate every face twice; in FP64 they took three times
// as long and are not built.
//
// Measured, both kernels, against the per-cell schedule (the default then) and the face-based one with
// a lane per face: 131 072 triangles, 2 points an edge 499 / 165 -> 146 us; 24 576 tetrahedra 362 / 122
// -> 89 us; 4200 triangles, 3 points 123 / 49 -> 17 us; 2048 triangles 80 / 33 -> 14 us. The large
// ones run at 80 % of the FP64 pipe. Small meshes want many small blocks (4200 triangles: 16.7 us in blocks
// of 32 threads, 20.4 in blocks of 128), large ones do not care (146.7 / 146.3 us): 32 by default.
#pragma once

#include "sqrt64.cuh"

namespace cteno {
namespace {

// x > 0, and fmin(a, b), fmax(a, b) with their rule for NaN (the other operand: a side with a negative pressure has
// no speed of sound, and the wave speeds are then those of the other side and of the Roe average), on integers.
__device__ __forceinline__ bool positive64(const double x) {
  const int h = __double2hiint(x);
  return (h > 0 && h <= 0x7FF00000) || (h == 0 && __double2loint(x) != 0);
}
__device__ __forceinline__ bool nan64(const double x) {  // of a result: its quiet bit is in the high word
  return (__double2hiint(x) & 0x7FFFFFFF) > 0x7FF00000;
}
__device__ __forceinline__ bool less64(const double a, const double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return (x ^ ((x >> 63) & 0x7FFFFFFFFFFFFFFFll)) < (y ^ ((y >> 63) & 0x7FFFFFFFFFFFFFFFll));
}
__device__ __forceinline__ double lower64(const double a, const double b) {
  return (less64(a, b) || nan64(b)) && !nan64(a) ? a : b;
}
__device__ __forceinline__ double higher64(const double a, const double b) {
  return (less64(b, a) || nan64(b)) && !nan64(a) ? a : b;
}

// HLLC flux as hllc() (eqs. 24-29), in its order, with IEEE division and the roots of sqrt64: the states ahead of a
// wave, whose selection hangs on differences of 1e-11, then round as those of any other FP64 evaluation of the
// printed formulas does (taking common factors once and reciprocals one unit off saved a third of the time and
// moved a 200-step shock tube by 5e-12 of its largest momentum, through selections of that size).
template <int D>
__device__ __forceinline__ void hllc64(const double *uL, const double *uR, const double *n, const double g, double *F) {
  constexpr int NV = D + 2;
  const double rL = uL[0], rR = uR[0];
  const double iL = 1.0 / rL, iR = 1.0 / rR;
  double vL[D], vR[D], unL = 0, unR = 0, kL = 0, kR = 0;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    vL[j] = uL[1 + j] * iL;
    vR[j] = uR[1 + j] * iR;
    unL += vL[j] * n[j];
    unR += vR[j] * n[j];
    kL += vL[j] * uL[1 + j];
    kR += vR[j] * uR[1 + j];
  }
  const double pL = (g - 1) * (uL[NV - 1] - 0.5 * kL);
  const double pR = (g - 1) * (uR[NV - 1] - 0.5 * kR);
  const double cL = sqrt64(g * pL * iL), cR = sqrt64(g * pR * iR);
  const double HL = (uL[NV - 1] + pL) * iL, HR = (uR[NV - 1] + pR) * iR;
  const double Dr = sqrt64(rR * iL);
  const double idn = 1.0 / (1 + Dr);
  double ut2 = 0, utn = 0;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const double ut = (vL[j] + vR[j] * Dr) * idn;
    ut2 += ut * ut;
    utn += ut * n[j];
  }
  const double Ht = (HL + HR * Dr) * idn;
  const double ct = sqrt64((g - 1) * (Ht - 0.5 * ut2));
  const double SL = lower64(unL - cL, utn - ct);
  const double SR = higher64(unR + cR, utn + ct);
  const double SM = (rR * unR * (SR - unR) - rL * unL * (SL - unL) + pL - pR) /
                    (rR * (SR - unR) - rL * (SL - unL));
  // The four cases, tested in the order SL > 0 (left state), SM > 0 (left star state), SR > 0
  // (right star state), else (right state), evaluated without branches (neighbouring faces of a
  // warp take different cases): the operands of side k are selected, the star correction is
  // dropped in the two supersonic cases. Each case's arithmetic is the same as written out alone.
  const bool left = positive64(SL) || positive64(SM);
  const bool sup = positive64(SL) || (!positive64(SM) && !positive64(SR));
  double uk[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) uk[v] = left ? uL[v] : uR[v];
  const double pk = left ? pL : pR, unk = left ? unL : unR, Sk = left ? SL : SR, rk = uk[0];
  F[0] = uk[0] * unk;
#pragma unroll
  for (int j = 0; j < D; ++j) F[1 + j] = uk[1 + j] * unk + pk * n[j];
  F[NV - 1] = (uk[NV - 1] + pk) * unk;
  const double ps = rL * (unL - SL) * (unL - SM) + pL;
  const double fct = 1.0 / (Sk - SM), a = Sk - unk;
  double G[NV];
  G[0] = F[0] + Sk * (rk * a * fct - uk[0]);
#pragma unroll
  for (int j = 0; j < D; ++j) G[1 + j] = F[1 + j] + Sk * ((a * uk[1 + j] + (ps - pk) * n[j]) * fct - uk[1 + j]);
  G[NV - 1] = F[NV - 1] + Sk * ((a * uk[NV - 1] - pk * unk + ps * SM) * fct - uk[NV - 1]);
#pragma unroll
  for (int v = 0; v < NV; ++v) F[v] = sup ? F[v] : G[v];
}

// Local CFL step |V_i| / sum_f |A_f| (|u_i . n_f| + c_i) of the FP64 path: the velocity and the speed
// of sound of a state, a face's term, and the step from their sum in face order. Every rounding is
// written out: the set-state kernels and the stage update must give the same bits.
template <int D>
__device__ __forceinline__ void speeds64(const double *u, const double g, double (&vel)[D], double &c) {
  const double ir = 1.0 / u[0];
  double ke = 0.0;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    vel[j] = __dmul_rn(u[1 + j], ir);
    ke = fma(u[1 + j], vel[j], ke);
  }
  c = sqrt(__dmul_rn(__dmul_rn(g, __dmul_rn(g - 1.0, fma(-0.5, ke, u[D + 1]))), ir));
}
template <int D>
__device__ __forceinline__ double face_speed64(const double *gf, const double (&vel)[D], const double c) {
  double un = 0.0;
#pragma unroll
  for (int j = 0; j < D; ++j) un = fma(vel[j], gf[j], un);
  return __dmul_rn(gf[3], __dadd_rn(fabs(un), c));
}
template <int D>
__device__ __forceinline__ double local_dt64(const KArgs &a, const int64_t i, const double *u) {
  double vel[D], c, s = 0.0;
  speeds64<D>(u, a.gamma, vel, c);
#pragma unroll
  for (int f = 0; f <= D; ++f) s = __dadd_rn(s, face_speed64<D>(a.geo + (i * (D + 1) + f) * 4, vel, c));
  return 1.0 / __dmul_rn(s, a.vol[i]);
}

template <int D, int NQ>
__global__ void __launch_bounds__(256) face_flux64_kernel(const KArgs a) {
  constexpr int NV = D + 2, NVP = Lay<D>::NVP, NF = D + 1, NFP = (NV + 3) & ~3;
  constexpr int FPW = 32 / NQ;  // faces of a warp; two spare lanes with three points a face
  pdl_wait(a);                  // face states of the reconstruction
  const int lane = threadIdx.x & 31, grp = lane / NQ, q = lane - grp * NQ, base = grp * NQ;
  const int64_t face = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * FPW + grp;
  const bool active = grp < FPW && face < a.nfaces;
  const int64_t e = active ? face : a.nfaces - 1;  // spare lanes shadow a face and store nothing
  const int2 codes = __ldg(reinterpret_cast<const int2 *>(a.face) + e);  // owner, neighbour side
  const int64_t i = codes.x >> 2;
  const int f = codes.x & 3;
  const double *__restrict__ Uf = (const double *)after_wait((double *)a.Uf);
  auto state = [&](int64_t cell, int face_of, double *u) {
    const double *p = Uf + ((cell * NF + face_of) * NQ + q) * NV;
    if constexpr (D == 2) {
      load16<double, NV>(p, u);
    } else {
#pragma unroll
      for (int v = 0; v < NV; ++v) u[v] = __ldg(p + v);
    }
  };
  double gf[4], uI[NV], uO[NV], F[NV];
  load16<double, 4>(a.geo + (i * NF + f) * 4, gf);
  state(i, f, uI);
  if (codes.y >= 0) {
    state(codes.y >> 2, codes.y & 3, uO);
  } else {  // boundary face: its kind's outside state
    double um[NVP];
#pragma unroll
    for (int v = 0; v < NVP; ++v) um[v] = a.U[i * NVP + v];
    boundary_state<D, double, 1>(a, i, (__ldg(a.fmeta + i) >> (kMetaKindShift + 2 * f)) & 3u, gf, uI, um, uO);
  }
  hllc64<D>(uI, uO, gf, a.gamma, F);
  double out[NFP];  // |A| sum_q w_q F_q, in the order of the points
#pragma unroll
  for (int v = 0; v < NFP; ++v) {
    double x = 0.0;
    if (v < NV) {
      x = a.fw[0] * __shfl_sync(0xffffffffu, F[v], base);
#pragma unroll
      for (int t = 1; t < NQ; ++t) x = fma(a.fw[t], __shfl_sync(0xffffffffu, F[v], base + t), x);
      x *= gf[3];
    }
    out[v] = x;
  }
  if (active && q == 0) store16<double, NFP>((double *)a.Ff + e * NFP, out);
}

template <int D>
__global__ void __launch_bounds__(256) cell_update64_kernel(const KArgs a) {
  constexpr int NV = D + 2, NVP = Lay<D>::NVP, NF = D + 1, NFP = (NV + 3) & ~3, CPW = 32 / NV;
  pdl_wait(a);  // the face fluxes of this stage
  const int lane = threadIdx.x & 31, grp = lane / NV, v = lane - grp * NV, base = grp * NV;
  const int64_t N = a.N;
  const int64_t first = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * CPW;
  const bool active = grp < CPW && first + grp < N;
  // spare lanes shadow the warp's last cell and store nothing: in 3D two lanes of every warp are spare, and one
  // atomic minimum takes the warp's time steps only where all its lanes have the same mesh (16 meshes of 12^3
  // cubes, degree 2: 474 us a flux launch, 617 when the spare lanes shadow the last cell of the batch)
  const int64_t i = min(first + min(grp, CPW - 1), N - 1);
  const int4 cf4 = __ldg(reinterpret_cast<const int4 *>(a.cellface) + i);
  const int cf[4] = {cf4.x, cf4.y, cf4.z, cf4.w};
  const int64_t at = i * NVP + v;
  const double *__restrict__ Ff = after_wait((const double *)a.Ff);
  const double u = a.U[at];
  double acc = 0.0;  // sum_f |A_f| sum_q w_q F_q, signed for this cell
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const double x = __ldg(Ff + (int64_t)(cf[f] & 0x7FFFFFFF) * NFP + v);
    acc += cf[f] < 0 ? -x : x;
  }
  const int mesh = (a.nmesh > 1) ? mesh_of(a, i) : 0;
  const double dtv = a.dt[mesh] * a.vol[i];  // dt / |V_i|
  double r, ac = 0.0;
  if (!a.rk4) {  // SSP-RK3 (Shu-Osher), as stage_tail
    r = fma(-dtv, acc, u);
    if (a.stage == 1) r = 0.75 * a.Un[at] + 0.25 * r;
    else if (a.stage == 2) r = (1.0 / 3.0) * a.Un[at] + (2.0 / 3.0) * r;
  } else {       // classical RK4 with its running sum, as stage_tail
    const double F = -dtv * acc;  // dt k_s
    const double w = (a.stage == 0 || a.stage == 3) ? 1.0 / 6.0 : 1.0 / 3.0;
    ac = fma(F, w, a.stage == 0 ? u : a.Acc[at]);
    r = a.stage == 3 ? ac : (a.stage == 0 ? u : a.Un[at]) + (a.stage == 2 ? F : 0.5 * F);
  }
  const bool finite = finite64(r);
  if (active) {
    if (a.stage == 0) a.Un[at] = u;
    if (a.rk4 && a.stage < 3) a.Acc[at] = ac;
    a.U[at] = r;
    if (!finite) atomicOr(a.err, kErrNonFinite);
  }
  if (a.stage == a.last_stage) {  // the CFL step of the next step: lane f takes face f
    double full[NV], vel[D], c, s = 0.0;
    bool fin = active;
#pragma unroll
    for (int t = 0; t < NV; ++t) {
      full[t] = __shfl_sync(0xffffffffu, r, base + t);
      fin = fin && finite64(full[t]);
    }
    speeds64<D>(full, a.gamma, vel, c);
    double gf[4];
    load16<double, 4>(a.geo + (i * NF + min(v, NF - 1)) * 4, gf);
    const double x = face_speed64<D>(gf, vel, c);
#pragma unroll
    for (int f = 0; f < NF; ++f) s = __dadd_rn(s, __shfl_sync(0xffffffffu, x, base + f));
    const double dt = a.cfl * (1.0 / __dmul_rn(s, a.vol[i]));
    warp_min_to(a.dt, a.nmesh + mesh, fin ? dt : 1e300);
  }
}

}  // namespace
}  // namespace cteno
