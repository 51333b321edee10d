// fixed.h -- layout of the FP64 path's least-squares operators as block fixed-point integers
// (written by setup.cu, read by recon_fixed.cuh).
//
// Entries are int2 (h, l), the integer h 2^29 + l of 57 bits and a sign in units of 2^(e - 57), e the
// exponent of its block (KArgs::Pe). The cells are taken in tiles of CPW, the cells of one warp of the
// reconstruction, and a tile's central rows in chunks of MC members, so that the chunk a warp
// streams through shared memory is one contiguous span:
//   Pc  [tile][M / MC][CPW][MC][NK]   (the last tile is allocated whole)
//   Pd  [cell][face][member][KD], PDS entries a face
#pragma once

#include <cstdint>

#include "device.h"

namespace cteno {

template <int D, int R>
struct FixShape {
  static constexpr int NV = D + 2, NVP = Lay<D>::NVP, NF = D + 1;
  static constexpr int NK = (D == 2 ? (R + 1) * (R + 2) / 2 : (R + 1) * (R + 2) * (R + 3) / 6) - 1;
  static constexpr int M = 2 * (NK + 1);
  static constexpr int NQ = D == 3 ? 4 : (R + 2) / 2 > 2 ? (R + 2) / 2 : 2;
  static constexpr int KD = Dir<D, R>::KD, ND = Dir<D, R>::ND, PDS = Dir<D, R>::PDS;
  static constexpr int CPW = 32 / NV;
  // chunks of the central record: all of it up to 20 members (2D degrees 2, 3; 3D degree 2)
  static constexpr int MC = M <= 20 ? M : M % 4 == 0 ? 4 : 6;
  static constexpr int NCH = M / MC, NST = NCH < 3 ? NCH : 3;  // chunks; of them in flight
  static constexpr int G = M % 4 == 0 ? 4 : 6;    // members whose differences are formed together
  static constexpr int SLOTS = M < NF * ND ? M : NF * ND;
  // face table [f][p][q][NKP]: phi'_k as int2, rows of an even number of entries; 2D: the reversed edge
  // swaps the stored points, one order (NP = 1)
  static constexpr int NP = D == 3 ? 6 : 1, NKP = (NK + 1) / 2 * 2;
  static constexpr int PHI_BYTES = NF * NP * NQ * NKP * 8;
  static constexpr int STAGE = CPW * MC * NK * 8;
  static constexpr int HDR = CPW * NF * PDS * 8, DELTA = SLOTS * 32 * 8;
  static constexpr int BARS = (1 + NST + 1) / 2 * 16;
  static constexpr int WARP_BYTES = HDR + NST * STAGE + DELTA + BARS;
  __host__ __device__ static constexpr int64_t index(int64_t cell, int m, int k) {  // of entry (m, k) of a cell in Pc
    const int64_t t = cell / CPW;
    return (((t * NCH + m / MC) * CPW + (cell - t * CPW)) * MC + m % MC) * NK + k;
  }
  static_assert(M % MC == 0 && MC % G == 0 && ND * KD <= PDS, "chunks of whole groups");
  static_assert((MC * NK * 8) % 16 == 0 && (PDS * 8) % 16 == 0, "bulk copies need 16-byte spans");
};
// Cells of Pc's allocation: whole tiles of 32 / (d + 2).
inline int64_t fixed_cells(int d, int64_t n) {
  const int64_t cpw = 32 / (d + 2);
  return (n + cpw - 1) / cpw * cpw;
}

}  // namespace cteno
