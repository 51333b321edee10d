// recon_tile.cuh -- the mixed path's reconstruction at degrees 2 and 3 (steps 1-6 of recon.cuh, conserved
// variables), one tile of cells per warp and VPL variables per lane.
//
// A group of LPC lanes reconstructs a cell: d+2 lanes with a variable each (VPL = 1), or 2 (2D) and 3 (3D)
// lanes with two each (VPL = 2; 3D: the sixth is the record's zero padding). Every sum keeps its order: the
// results are those of the other lane schedules, bit for bit. The tile's records go to shared memory with
// bulk copies issued before the previous kernel has ended: stencil ids and directional operators, and
// the central records, in 2D whole, in 3D through a ring of two chunks of 4 members (one copy per cell
// and chunk, each by a lane of its own). The differences of the directional members wait in shared memory
// for the second product; the face values go through it to 16-byte stores. The positivity guard tests the
// bounds of a cell's face values first (min rho min E against max |m|, one exchange per cell instead of
// one per point); only where that leaves a doubt are the points tested.
//
// What bounds it: each warp is a chain of copies, gathers and dependent sums of some 10 us, so the
// number of warps an SM holds decides, until the shared-memory pipe does: 128 bytes a clock and SM whether
// or not the lanes of a cell ask for the same value. One variable per lane takes few registers (20 to 32
// warps an SM) and reads every operator value d+2 times; two per lane halve that (10 to 16 warps). Measured
// per launch against the best earlier schedule: 3D degree 3, 663 552 cells 676 (streamed lanes) -> 568 us with
// one, 596 with two (one at 16 instead of 20 warps an SM 606, chunks of 8 members 610); shared memory then 88 %
// busy, memory 58 %. 3D degree 2, 196 608 cells 114 (gather-staged) -> 91 us (chunks of 20 members 97, two
// variables 110). 2D degree 2, 131 072 cells 20.6 -> 19.7 us, a batch of 752 644 103 -> 93 us (chunks of 4: 113).
#pragma once

#include <type_traits>

#include "recon.cuh"

namespace cteno {

template <int D, int R, int VPL>
struct TileDims {
  using S = Shape<D, R>;
  using L = Lay<D>;
  static constexpr int LPC = (L::NV + VPL - 1) / VPL, CPW = 32 / LPC;
  static constexpr int MC = D == 2 ? S::M : 4;                // members per chunk
  static constexpr int NCH = S::M / MC, NST = NCH < 2 ? 1 : 2;
  static constexpr int ROW = MC * S::NK * 4, STAGE = CPW * ROW;
  static constexpr int HPD = CPW * L::NF * L::PDS * 4, HDR = HPD + CPW * S::M * 4;
  static constexpr int SLOTS = S::M < L::NF * L::ND ? S::M : L::NF * L::ND;
  static constexpr int REC = L::NF * L::NQ * L::NV;           // face values of a cell
  static constexpr int DELTA = SLOTS * 32 * 4 * VPL > CPW * REC * 4 ? SLOTS * 32 * 4 * VPL : CPW * REC * 4;
  static constexpr int BARS = (2 + NST + 1) / 2 * 16;         // header, stages, test hook
  static constexpr int WARP_BYTES = HDR + NST * STAGE + DELTA + BARS;
  static constexpr int FIT = 227 * 1024 / (4 * WARP_BYTES + 1024), CAP = VPL == 2 ? 4 : D == 3 && R == 3 ? 5 : 8, BLOCKS = FIT < CAP ? FIT : CAP;
  static_assert(S::M % MC == 0 && ROW % 16 == 0 && HDR % 16 == 0 && (S::M * 4) % 16 == 0 && (REC * 4) % 16 == 0,
                "16-byte spans");
};

template <int D, int R, int SCHEME, int VPL>
__global__ void __launch_bounds__(128, TileDims<D, R, VPL>::BLOCKS) recon_tile_kernel(const KArgs a) {
  using Q = TileDims<D, R, VPL>;
  using S = Shape<D, R>;
  using L = Lay<D>;
  constexpr int NV = L::NV, NF = L::NF, NQ = L::NQ, ND = L::ND, PDS = L::PDS, NK = S::NK, M = S::M;
  constexpr int LPC = Q::LPC, CPW = Q::CPW, MC = Q::MC, NCH = Q::NCH, NST = Q::NST, SLOTS = Q::SLOTS, REC = Q::REC;
  extern __shared__ __align__(128) unsigned char smem[];
  unsigned char *const wmem = smem + (threadIdx.x >> 5) * Q::WARP_BYTES;
  unsigned char *const dmem = wmem + Q::HDR + NST * Q::STAGE;
  uint64_t *const bar = reinterpret_cast<uint64_t *>(dmem + Q::DELTA);  // header, stages, test hook
  const int lane = threadIdx.x & 31, grp = lane / LPC, s = lane - grp * LPC, base = grp * LPC, v0 = VPL * s;
  const int64_t N = a.N;
  const int64_t tile = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), c0 = tile * CPW;
  const int n = (int)max((int64_t)0, min((int64_t)CPW, N - c0));  // the warp's cells
  // chunk c of the warp's tile: announced by lane 0, copied whole by it or per cell by the first n lanes
  auto issue = [&](int c) {
    uint64_t *b = &bar[1 + c % NST];
    unsigned char *to = wmem + Q::HDR + (c % NST) * Q::STAGE;
    if (lane == 0) {
      mbar_arrive_expect_tx(b, (uint32_t)(n * Q::ROW));
      if (NCH == 1) bulk_copy_g2s(to, (const float *)a.Pc + c0 * (M * NK), (uint32_t)(n * Q::ROW), b);
    }
    if (NCH > 1) {
      __syncwarp();
      if (lane < n)
        bulk_copy_g2s(to + lane * Q::ROW, (const float *)a.Pc + (c0 + lane) * (M * NK) + c * (MC * NK), Q::ROW, b);
    }
  };
  if (n > 0) {
    if (lane == 0) {
      for (int b = 0; b < 2 + NST; ++b) mbar_init(&bar[b], 1);
      fence_barrier_init();
      mbar_arrive_expect_tx(&bar[0], (uint32_t)(n * (M * 4 + NF * PDS * 4)));
      bulk_copy_g2s(wmem + Q::HPD, a.st + c0 * M, (uint32_t)(n * M * 4), &bar[0]);
      bulk_copy_g2s(wmem, (const float *)a.Pd + c0 * (NF * PDS), (uint32_t)(n * NF * PDS * 4), &bar[0]);
    }
    __syncwarp();
#pragma unroll
    for (int c = 0; c < NST; ++c) issue(c);
  }
  __syncwarp();
  const bool active = grp < n;
  const int slot = active ? grp : max(n, 1) - 1;  // spare lanes shadow a valid cell and store nothing
  const int64_t i = min(c0 + slot, N - 1);
  const uint32_t info = __ldg(a.cinfo + i);
  pdl_wait(a);  // the state written by the previous stage's update
  if (a.dt_swap && blockIdx.x == 0)  // the CFL step: dt[next] -> dt[cur]
    for (int t = threadIdx.x; t < a.nmesh; t += blockDim.x) {
      a.dt[t] = a.dt[a.nmesh + t];
      a.dt[a.nmesh + t] = 1e300;
    }
  if (n == 0) return;  // a warp past the last cell
  // a bounded wait of the whole warp for its copies; on a timeout the warp reports it, gives the
  // copies in flight (the header before the first chunk, chunks c up to `last`) a second bounded wait and stops
  auto arrived = [&](uint64_t *b, uint32_t parity, int c, int last, uint64_t limit_ns = kStageWaitNs) {
    const bool ok = mbar_wait(b, parity, limit_ns);
    if (!__any_sync(0xffffffffu, !ok)) return true;
    if (lane == 0) {
      atomicOr(a.err, kErrTimeout);
      if (!c) mbar_wait(&bar[0], 0, kStageWaitNs);
      for (; c < last; ++c) mbar_wait(&bar[1 + c % NST], (uint32_t)((c / NST) & 1), kStageWaitNs);
    }
    __syncwarp();
    return false;
  };
  // test hook: a bounded wait on a barrier that nothing completes runs out
  if (a.test_wait_ns && !arrived(&bar[1 + NST], 0, 0, NST, a.test_wait_ns)) return;
  using Pairs = typename std::conditional<VPL == 2, float4, float2>::type;      // (hi, lo) of a lane's variables
  constexpr int NU = L::NVP / VPL;
  const Pairs *__restrict__ Uq = reinterpret_cast<const Pairs *>(after_wait(a.U32)) + s;
  const int32_t *__restrict__ sti = reinterpret_cast<const int32_t *>(wmem + Q::HPD) + slot * M;
  float *const sdel = reinterpret_cast<float *>(dmem) + VPL * lane;
  const Pairs own = __ldg(Uq + i * NU);
  float U0[VPL], L0[VPL];
  U0[0] = own.x, L0[0] = own.y;
  if constexpr (VPL == 2) U0[1] = own.z, L0[1] = own.w;
  if (!arrived(&bar[0], 0, 0, NST)) return;

  // central coefficients of both variables; the member states of the next chunk are gathered while a
  // chunk is multiplied
  float ao[VPL][NK];
#pragma unroll
  for (int t = 0; t < VPL; ++t)
#pragma unroll
    for (int k = 0; k < NK; ++k) ao[t][k] = 0.0f;
  Pairs nx[MC];
  auto fetch = [&](int c) {
#pragma unroll
    for (int g = 0; g < MC; g += 4) {
      const int4 j = *reinterpret_cast<const int4 *>(sti + c * MC + g);
      nx[g] = __ldg(Uq + (int64_t)j.x * NU);
      nx[g + 1] = __ldg(Uq + (int64_t)j.y * NU);
      nx[g + 2] = __ldg(Uq + (int64_t)j.z * NU);
      nx[g + 3] = __ldg(Uq + (int64_t)j.w * NU);
    }
  };
  fetch(0);
#pragma unroll 1
  for (int c = 0; c < NCH; ++c) {
    float du[MC][VPL];
#pragma unroll
    for (int g = 0; g < MC; ++g) {
      du[g][0] = (nx[g].x - U0[0]) + (nx[g].y - L0[0]);
      if constexpr (VPL == 2) du[g][1] = (nx[g].z - U0[1]) + (nx[g].w - L0[1]);
      if (c * MC + g < SLOTS) {
        float *to = sdel + (c * MC + g) * (32 * VPL);
        if constexpr (VPL == 2) *reinterpret_cast<float2 *>(to) = make_float2(du[g][0], du[g][1]);
        else *to = du[g][0];
      }
    }
    if (c + 1 < NCH) fetch(c + 1);
    if (!arrived(&bar[1 + c % NST], (uint32_t)((c / NST) & 1), c, min(c + NST, NCH))) return;
    const float *__restrict__ P =
        reinterpret_cast<const float *>(wmem + Q::HDR + (c % NST) * Q::STAGE) + slot * (MC * NK);
    float pb[4];
#pragma unroll
    for (int e = 0; e < MC * NK; ++e) {
      if (e % 4 == 0) load16<float, 4, true>(P + e, pb);
#pragma unroll
      for (int t = 0; t < VPL; ++t) ao[t][e % NK] += pb[e % 4] * du[e / NK][t];
    }
    if (NST < NCH && c + NST < NCH) {
      fence_proxy_async_shared();  // this lane's reads of the stage precede the copies that refill it
      __syncwarp();
      issue(c + NST);
    }
  }
  // directional coefficients (degree 1): the members of face f are the next slots of the list
  const uint32_t adm = (info >> kInfoAdmShift) & 0xFu;
  const float *__restrict__ Pdi = reinterpret_cast<const float *>(wmem) + slot * (NF * PDS);
  float ad[VPL][NF][D];
  {
    int off = 0;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const int nm = (info >> (4 * f)) & 15u;
#pragma unroll
      for (int k = 0; k < D; ++k)
#pragma unroll
        for (int t = 0; t < VPL; ++t) ad[t][f][k] = 0.0f;
      if ((adm >> f) & 1u) {
        float pf[PDS];
        load16<float, PDS, true>(Pdi + f * PDS, pf);
#pragma unroll
        for (int jj = 0; jj < ND; ++jj)
          if (jj < nm) {
            float du[VPL];
            const float *from = sdel + (off + jj) * (32 * VPL);
            if constexpr (VPL == 2) {
              const float2 x = *reinterpret_cast<const float2 *>(from);
              du[0] = x.x, du[1] = x.y;
            } else {
              du[0] = *from;
            }
#pragma unroll
            for (int k = 0; k < D; ++k)
#pragma unroll
              for (int t = 0; t < VPL; ++t) ad[t][f][k] += pf[jj * D + k] * du[t];
          }
      }
      off += nm;
    }
  }
  // selection and face values, into the tile's output records in shared memory
  constexpr float INV_FACT = (D == 2) ? 0.5f : (float)(1.0 / 6.0);
  auto oc = [](int idx) { return cO<float, R>(idx); };
  auto sid = [&](const float (&adf)[D]) {  // the linear block of O is |V0'| I
    float q = 0.0f;
#pragma unroll
    for (int k = 0; k < D; ++k) q += adf[k] * adf[k];
    return q * INV_FACT;
  };
  const uint32_t perm = info >> kInfoPermShift;
  float *const sout = reinterpret_cast<float *>(dmem);
  __syncwarp();  // the differences are no longer needed
  float low[VPL];    // bounds of the face values: the smallest
  uint32_t top[VPL];  // and the bits of the largest magnitude (not finite: above those of any number)
  float off[VPL] = {};
#pragma unroll
  for (int t = 0; t < VPL; ++t) {
    const uint32_t bits = lane_select<D, NK, D, float, SCHEME>(a, adm, ao[t], ad[t], oc, sid);
    if (a.flags && active && v0 + t < NV) a.flags[(v0 + t) * N + i] = (uint8_t)bits;
    low[t] = INFINITY;
    top[t] = 0u;
    if constexpr (D == 3) off[t] = PhiMono3<R>{perm}.offset(ao[t]);
  }
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const int p = (perm >> (3 * f)) & 7u;
    constexpr int UQ = D == 3 ? 1 : NQ;  // 3D: a rolled loop, straight-line code would overflow the instruction cache
#pragma unroll UQ
    for (int q = 0; q < NQ; ++q) {
      const int qq = (D == 2 && p) ? (NQ - 1 - q) : q;  // 2D: edge points in sorted-vertex order
#pragma unroll
      for (int t = 0; t < VPL; ++t) {
        float val = L0[t] - off[t];
        if constexpr (D == 3) {
          val = PhiMono3<R>{perm}.value(f, q, ao[t], val);
        } else {
#pragma unroll
          for (int k = 0; k < NK; ++k) val += cPhi2<float, R>((f * 2 + q) * NK + k) * ao[t][k];
        }
        val += U0[t];
        low[t] = fminf(low[t], val);
        top[t] = max(top[t], __float_as_uint(val) & 0x7FFFFFFFu);
        if (active && v0 + t < NV) sout[slot * REC + (f * NQ + qq) * NV + v0 + t] = val;
      }
    }
  }
  if (a.guard_on) {
    const float rho = __shfl_sync(0xffffffffu, low[0], base);
    const float E = __shfl_sync(0xffffffffu, low[(NV - 1) % VPL], base + (NV - 1) / VPL);
    float ke = 0.0f;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const float m = __uint_as_float(__shfl_sync(0xffffffffu, top[(1 + j) % VPL], base + (1 + j) / VPL));
      ke += m * m;
    }
    const float rE = rho * E;
    bool finite = true;
#pragma unroll
    for (int t = 0; t < VPL; ++t) finite = finite && top[t] < 0x7F800000u;
    const bool sure = finite && rho > 0.0f && E > 0.0f && rE - 0.5f * ke > 1e-5f * rE;
    if (__any_sync(0xffffffffu, active && !sure)) {
      __syncwarp();
      bool bad = false;
      for (int p = s; p < NF * NQ; p += LPC) {  // the points of the cell, shared by its lanes
        const float *u = sout + slot * REC + p * NV;
        float kp = 0.0f;
#pragma unroll
        for (int j = 0; j < D; ++j) kp += u[1 + j] * u[1 + j];
        bad = bad || !(u[0] > 0.0f) || !(u[0] * u[NV - 1] - 0.5f * kp > 0.0f);
      }
      const uint32_t who = __ballot_sync(0xffffffffu, bad && active);
      __syncwarp();
      if (active && ((who >> base) & ((1u << LPC) - 1u))) {
#pragma unroll
        for (int t = 0; t < VPL; ++t)
          if (v0 + t < NV)
            for (int p = 0; p < NF * NQ; ++p) sout[slot * REC + p * NV + v0 + t] = U0[t] + L0[t];
        if (s == 0) atomicAdd(a.guard, 1ull);
      }
    }
  }
  __syncwarp();
  float4 *__restrict__ Uf = reinterpret_cast<float4 *>((float *)a.Uf + c0 * REC);
  for (int t = lane; t < n * (REC / 4); t += 32) Uf[t] = reinterpret_cast<const float4 *>(sout)[t];
}

template <int D, int R, int SCHEME, int VPL>
cudaError_t launch_recon_tile(const KArgs &a, int threads, cudaStream_t s) {
  using Q = TileDims<D, R, VPL>;
  const int64_t cells = (int64_t)(threads / 32) * Q::CPW;
  const size_t smem = (size_t)(threads / 32) * Q::WARP_BYTES;
  auto kern = recon_tile_kernel<D, R, SCHEME, VPL>;
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  launch_stage_kernel(kern, (unsigned)((a.N + cells - 1) / cells), threads, smem, s, a);
  return cudaSuccess;
}

}  // namespace cteno
