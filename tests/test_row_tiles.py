"""The tail of a cluster's FP32 rows in global scratch (HybridRows): every
float of it lies inside the cluster's float4 [N] region of the scratch, up to
the largest frame the library takes.  Index arithmetic only, on the host."""
import subprocess

from paper_2012_12618_gb300 import build

SRC = r"""
#include <cstdio>
#include "rvh_scoring.cuh"
using namespace rvh;

template <int NC>
int check() {
  using Tail = decltype(HybridRows<NC>::g);
  int bad = 0;
  const long long sizes[] = {1537, 2080, 40000, (1ll << 29) - 1, 1ll << 29, (1ll << 31) / 3 + 5, 2147483392ll};
  for (long long N : sizes) {
    const int cap = (NC == 3 ? 2048 : 1536);
    const long long start = -(long long)cap * NC;  // of g.f, in floats from the cluster's region
    const int js[] = {cap, cap + 31, (int)(N / 2) | cap, (int)(N - 1)};
    for (int j : js) {
      if (j < cap || j >= N) continue;
      const long long want = (j / 32) * (32ll * NC) + j % 32;  // of the point's first component
      const long long got = 4 * (long long)Tail::tile(j >> 5) + (j & 31);
      const int q = j >> 2, k = NC - 1;
      const long long quad = 4 * (long long)(Tail::tile(q >> 3) + (k << 3) + (q & 7));  // of its last one's quad
      if (got != want || quad != want - j % 4 + 32 * k || start + got < 0 || start + quad + 3 >= 4 * N) {
        std::printf("NC %d N %lld point %d: float %lld, not %lld\n", NC, N, j, got, want);
        ++bad;
      }
    }
  }
  return bad;
}

int main() { return check<3>() + check<4>() ? 1 : 0; }
"""


def test_tail_offsets(tmp_path):
    src, exe = tmp_path / "tiles.cu", str(tmp_path / "tiles")
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, str(src), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
