// Tiled form of the TTMc (ttmc_tile.cuh): launches for three and more remaining modes.
#include <algorithm>

#include "ttmc_tile.cuh"

namespace tk {

#define TK_TILE_N(NO, TA_, TB_) \
  if (TA == TA_ && TB == TB_) return run_tile<NO, TA_, TB_>(p, num_sms, s);
#define TK_TILE_ROW3(TA_) TK_TILE_N(3, TA_, 4) TK_TILE_N(3, TA_, 5) TK_TILE_N(3, TA_, 6) TK_TILE_N(3, TA_, 8)
#define TK_TILE_ROW7(TA_) TK_TILE_N(7, TA_, 4) TK_TILE_N(7, TA_, 5) TK_TILE_N(7, TA_, 8)

cudaError_t tile_dispatch_n(int TA, int TB, TileParams &p, int num_sms, cudaStream_t s) {
  if (p.nother == 3) {
    TK_TILE_ROW3(4)
    TK_TILE_ROW3(5)
    TK_TILE_ROW3(6)
    TK_TILE_ROW3(8)
  } else {
    TK_TILE_ROW7(4)
    TK_TILE_ROW7(5)
    TK_TILE_ROW7(8)
  }
  return cudaErrorInvalidConfiguration;
}

}  // namespace tk
