// Adjoint form of the tiled TTMc (ttmc_tile.cuh): launches.  Tiles of at most 49 entries (40 with three
// and more remaining modes), since a lane holds two of them; chunks of eight are taken as 8 x 4 or smaller.
#include <algorithm>

#include "ttmc_tile.cuh"

namespace tk {

bool tile_adj_covers(int TA, int TB, int nother) { return TA * TB <= (nother <= 2 ? 49 : 40); }

#define TK_ADJ(NO, TA_, TB_) \
  if (TA == TA_ && TB == TB_) return run_tile<NO, TA_, TB_, true>(p, num_sms, s);

cudaError_t tile_dispatch_adj(int TA, int TB, TileParams &p, int num_sms, cudaStream_t s) {
  switch (p.nother) {
    case 1:
      TK_ADJ(1, 1, 4) TK_ADJ(1, 1, 5) TK_ADJ(1, 1, 6) TK_ADJ(1, 1, 7) TK_ADJ(1, 1, 8)
      break;
    case 2:
      TK_ADJ(2, 4, 4) TK_ADJ(2, 4, 5) TK_ADJ(2, 4, 6) TK_ADJ(2, 4, 7) TK_ADJ(2, 4, 8)
      TK_ADJ(2, 5, 4) TK_ADJ(2, 5, 5) TK_ADJ(2, 5, 6) TK_ADJ(2, 5, 7) TK_ADJ(2, 5, 8)
      TK_ADJ(2, 6, 4) TK_ADJ(2, 6, 5) TK_ADJ(2, 6, 6) TK_ADJ(2, 6, 7) TK_ADJ(2, 6, 8)
      TK_ADJ(2, 7, 4) TK_ADJ(2, 7, 5) TK_ADJ(2, 7, 6) TK_ADJ(2, 7, 7)
      TK_ADJ(2, 8, 4) TK_ADJ(2, 8, 5) TK_ADJ(2, 8, 6)
      break;
    case 3:
      TK_ADJ(3, 4, 4) TK_ADJ(3, 4, 5) TK_ADJ(3, 4, 6) TK_ADJ(3, 4, 8)
      TK_ADJ(3, 5, 4) TK_ADJ(3, 5, 5) TK_ADJ(3, 5, 6) TK_ADJ(3, 5, 8)
      TK_ADJ(3, 6, 4) TK_ADJ(3, 6, 5) TK_ADJ(3, 6, 6)
      TK_ADJ(3, 8, 4) TK_ADJ(3, 8, 5)
      break;
    default:
      TK_ADJ(7, 4, 4) TK_ADJ(7, 4, 5) TK_ADJ(7, 4, 8)
      TK_ADJ(7, 5, 4) TK_ADJ(7, 5, 5) TK_ADJ(7, 5, 8)
      TK_ADJ(7, 8, 4) TK_ADJ(7, 8, 5)
  }
  return cudaErrorInvalidConfiguration;
}

}  // namespace tk
