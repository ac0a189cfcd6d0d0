"""The dealing of a tile's halo ring to the threads of its block (pflbm_ring.h, used by the Cahn-Hilliard k_tile and by
k_adj_tile), compiled for the host: every ring cell is stored, and nothing outside the ring, for every tile a block of
up to 256 threads can have.  The kernels' blocks are bw x bh threads with bw <= 32; widths such as 3, 7 or 11 columns
give blocks that are no multiple of a warp, and blocks of fewer than 32 threads."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2111_00847_gb300", "csrc")

SOURCE = r"""
#include <vector>
#include "pflbm_ring.h"

// ring cells never stored, plus 1000 for each store that is no ring cell
template <int R>
static int faults(int bw, int bh) {
  const int nth = bw * bh, pw = bw + 2 * R, ph = bh + 2 * R;
  std::vector<char> seen((size_t)pw * ph, 0);
  int bad = 0;
  const pflbm::RingDeal<R> ring(bw, bh, nth);
  for (int tid = 0; tid < nth; ++tid)
    for (int k = ring.first(tid); ring.is_share(k); k += ring.warps) {
      int cx, cy;
      if (!ring.place(k, tid, cx, cy)) continue;
      const bool in = cx >= -R && cx < bw + R && cy >= -R && cy < bh + R;
      const bool tile = cx >= 0 && cx < bw && cy >= 0 && cy < bh;
      if (!in || tile) bad += 1000;
      else seen[(size_t)(cy + R) * pw + cx + R] = 1;
    }
  for (int y = -R; y < bh + R; ++y)
    for (int x = -R; x < bw + R; ++x)
      if (!(x >= 0 && x < bw && y >= 0 && y < bh) && !seen[(size_t)(y + R) * pw + x + R]) ++bad;
  return bad;
}
extern "C" int ring_faults(int r, int bw, int bh) { return r == 1 ? faults<1>(bw, bh) : faults<2>(bw, bh); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    src, so = d / "ring.cpp", d / "ring.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-I", CSRC, str(src), "-o", str(so)], check=True)
    return C.CDLL(str(so))


@pytest.mark.parametrize("radius", [1, 2])
def test_every_ring_cell_is_stored(lib, radius):
    bad = [(bw, bh) for bw in range(1, 33) for bh in range(1, 256 // bw + 1) if lib.ring_faults(radius, bw, bh)]
    assert not bad, f"{len(bad)} tiles, e.g. {bad[:8]}"


def test_no_shuffle_mask_depends_on_convergence():
    """A warp's lanes need not have met again after a loop of differing trip counts: shuffle masks come from sizes."""
    for name in os.listdir(CSRC):
        with open(os.path.join(CSRC, name)) as fh:
            assert "__activemask" not in fh.read(), name
