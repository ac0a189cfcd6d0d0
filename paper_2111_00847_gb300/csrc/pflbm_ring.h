// How a tile's halo ring is dealt to the warps of its block (k_tile for
// Cahn-Hilliard, k_adj_tile).  Host and device.
#pragma once

#ifdef __CUDACC__
#define PFLBM_HD __host__ __device__ __forceinline__
#else
#define PFLBM_HD inline
#endif

namespace pflbm {

// The ring R nodes wide of a bw x bh tile (bw <= 32) whose block has nth
// threads, in shares: first the 2R rows below and above (columns [0, bw)), a row
// a share, then the R columns on either side of all bh + 2R rows, `lanes` cells
// a share.  Shares go round the block's full warps, so every lane of a share is
// there: a tile of fewer than 32 columns need not be a multiple of 32 threads,
// and its last, partial warp takes none.  A block under a warp takes shares of
// its own size.  Cahn-Hilliard 4096^2, us a step: 597; every cell to thread
// e mod nth 603; the loop bounded by a count of shares 603.
template <int R>
struct RingDeal {
  int bw, bh, lanes, warps;
  PFLBM_HD RingDeal(int bw_, int bh_, int nth)
      : bw(bw_), bh(bh_), lanes(nth < 32 ? nth : 32), warps(nth < 32 ? 1 : nth >> 5) {}
  // first share of thread tid's warp (the next ones follow at a distance of
  // warps), and whether there is a share k
  PFLBM_HD int first(int tid) const { return (tid >> 5) < warps ? tid >> 5 : 1 << 20; }
  PFLBM_HD bool is_share(int k) const { return k < 2 * R || (k - 2 * R) * lanes < 2 * R * (bh + 2 * R); }
  // thread tid's cell of share k, relative to the tile; false: none
  PFLBM_HD bool place(int k, int tid, int& cx, int& cy) const {
    cx = tid & 31;
    if (k < 2 * R) {
      cy = k < R ? k - R : bh + k - R;
      return cx < bw;
    }
    const int q = (k - 2 * R) * lanes + cx;
    cy = q / (2 * R) - R;
    cx = q % (2 * R);
    cx = cx < R ? cx - R : bw + cx - R;
    return cy < bh + R;
  }
};

}  // namespace pflbm
