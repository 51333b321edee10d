// tiles.h -- layout of the least-squares operators that a warp streams through shared memory (written by
// setup.cu; read by recon_fixed.cuh, the FP64 path, and recon_high.cuh, the mixed path's degrees 4 to 6).
//
// The cells are taken in tiles of CPW, the cells of one warp of the reconstruction, and a tile's
// central rows in chunks of MC members, so that the chunk a warp copies is one contiguous span:
//   Pc  [tile][M / MC][CPW][MC][NK]   (the last tile is allocated whole)
//   Pd  [cell][face][PDS]             (Dir<D, R>; FP64 path: member-major j * KD + k at every degree)
// Entries (E bytes): float, or on the FP64 path Pd double and Pc int2 (h, l), the integer h 2^29 + l of 57 bits
// and a sign in units of 2^(e - 57), e the exponent of its row (KArgs::Pe).
#pragma once

#include <cstdint>

#include "device.h"

namespace cteno {

template <int D, int R, int E>
struct TileShape {
  static constexpr int NV = D + 2, NVP = Lay<D>::NVP, NF = D + 1;
  static constexpr int NK = (D == 2 ? (R + 1) * (R + 2) / 2 : (R + 1) * (R + 2) * (R + 3) / 6) - 1;
  static constexpr int M = 2 * (NK + 1);
  static constexpr int NQ = D == 3 ? 4 : (R + 2) / 2 > 2 ? (R + 2) / 2 : 2;
  static constexpr int KD = Dir<D, R>::KD, ND = Dir<D, R>::ND, PDS = Dir<D, R>::PDS;
  static constexpr int CPW = 32 / NV;
  // Chunks of the central record, NST of them in flight, and the members whose differences are formed
  // together. FP64: all of it at 12 members (2D degree 2), else chunks of 4 or 6. Mixed: chunks of 2.7,
  // 3.8 and 3.5 kB a warp at degrees 4, 5 and 6; 5 to 12 kB in flight in each of 9 to 13 warps cover the
  // memory latency of an SM (about 45 kB at the full rate) through the arithmetic. Measured, us a
  // launch (MC x NST): degree 4, 215 000 cells 10 x 3 123.7, 10 x 2 115.1, 6 x 3 117.7, 6 x 2 112.4; degree 6,
  // 180 000 cells 8 x 2 223.3, 8 x 3 230.2, 4 x 3 219.7, 4 x 4 237.4.
  static constexpr int MC = E == 4 ? (R == 6 ? 4 : 6) : M == 12 ? 12 : M % 4 == 0 ? 4 : 6;
  static constexpr int NCH = M / MC, NMAX = E == 4 ? (R == 4 ? 2 : 3) : 2;
  static constexpr int NST = NCH < NMAX ? NCH : NMAX;
  static constexpr int G = E == 4 ? MC : M % 4 == 0 ? 4 : 6;
  static constexpr int SLOTS = M < NF * ND ? M : NF * ND;
  // FP64: face table (2D in shared memory; in 3D, where its 15 kB a block cost a third of the warps, read through
  // L1) [f][p][q][NKP], phi'_k as int2, rows of an even number of entries; 2D: the reversed edge
  // swaps the stored points, one order (NP = 1)
  static constexpr int NP = D == 3 ? 6 : 1, NKP = (NK + 1) / 2 * 2;
  static constexpr int PHI_BYTES = E == 8 && D == 2 ? NF * NP * NQ * NKP * 8 : 0;
  static constexpr int STAGE = CPW * MC * NK * E;
  // a warp's header: directional operators, then stencil ids
  static constexpr int HPD = CPW * NF * PDS * E, HDR = HPD + CPW * M * 4, DELTA = SLOTS * 32 * E;
  static constexpr int BARS = (2 + NST + 1) / 2 * 16;  // header, stages, test hook
  static constexpr int WARP_BYTES = HDR + NST * STAGE + DELTA + BARS;
  __host__ __device__ static constexpr int64_t index(int64_t cell, int m, int k) {  // of entry (m, k) of a cell in Pc
    const int64_t t = cell / CPW;
    return (((t * NCH + m / MC) * CPW + (cell - t * CPW)) * MC + m % MC) * NK + k;
  }
  static_assert(M % MC == 0 && MC % G == 0 && ND * KD <= PDS, "chunks of whole groups");
  // blocks of 4 warps that shared memory lets an SM hold, and the register cap that goes with them
  static constexpr int BLOCK_BYTES = PHI_BYTES + 16 + 4 * WARP_BYTES;
  static constexpr int FIT = 227 * 1024 / (BLOCK_BYTES + 1024), BLOCKS = FIT < 4 ? FIT : 4;
  static_assert((MC * NK * E) % 16 == 0 && (G * NK * E) % 16 == 0 && (PDS * E) % 16 == 0 && (M * 4) % 8 == 0 &&
                    HDR % 16 == 0, "16-byte spans");
};
// Cells of Pc's allocation: whole tiles of 32 / (d + 2).
inline int64_t tiled_cells(int d, int64_t n) {
  const int64_t cpw = 32 / (d + 2);
  return (n + cpw - 1) / cpw * cpw;
}

}  // namespace cteno
