// The chunk length along s of the tiled stage kernel (s_chunk of
// paper_2011_02600_gb300/csrc/tile_map.cuh) compiled as host C++.  Built by
// tests/test_host_chunks.py.
#include <algorithm>

using std::max;
using std::min;

#define __ldg(p) (*(p))
#include "tile_map.cuh"

extern "C" int host_s_chunk(long long tiles, int nk, int nb, long long slots, double warm, int b, int extra) {
  return sbp::s_chunk(tiles, nk, nb, slots, warm, b, extra);
}
