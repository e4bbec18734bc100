"""How the ring lookups deal a batch to their warps (host code only): every key
once, blocks of 64 neighbours, and a long stretch of the batch to all warps."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1702_03154_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include <algorithm>
#include "keyring.cuh"
using namespace bbh;
static int check(u64 n, u64 warps, unsigned per_cta) {
  const RingShape sh = ring_shape(n, warps);
  const unsigned grid = ring_grid(sh, per_cta, warps / per_cta);
  std::vector<unsigned char> seen(n, 0);
  std::vector<u64> share(warps, 0);  // of the batch's first tenth
  const u64 tenth = n / 10;
  for (u64 w = 0; w < warps; w++) {
    const RingPart p(sh, (unsigned)w);
    if (p.len && w >= (u64)grid * per_cta) return 1;  // a warp that is not launched
    for (unsigned i = 0; i < p.len; i++) {
      const u64 at = p.place(sh, i);
      if (at >= n || seen[at]) return 2;
      seen[at] = 1;
      if (i % kBlock && at != p.place(sh, i - 1) + 1) return 3;
      share[w] += at < tenth;
    }
  }
  for (u64 i = 0; i < n; i++)
    if (!seen[i]) return 4;
  // a tenth of many turns of chunks: no warp has more than a chunk over another
  if (sh.cut && tenth >= sh.turn)
    if (*std::max_element(share.begin(), share.end()) >
        *std::min_element(share.begin(), share.end()) + kChunk) return 5;
  // no warp has much more than an even share
  const RingPart first(sh, 0);
  if (sh.cut && (u64)first.len * warps > n + 16 * warps) return 6;
  return 0;
}
int main() {
  for (u64 warps : {8ull, 40ull}) {
    const u64 turn = warps * kChunk;
    for (u64 n : {1ull, 15ull, 16ull, 17ull, 63ull, 64ull, 65ull, 127ull * warps, 128 * warps + 1,
                  turn - 1, turn, turn + 1, 2 * turn - 17, 2 * turn, 2 * turn + 1, 2 * turn + 64,
                  3 * turn - 1, 3 * turn, 3 * turn + 15, 11 * turn + turn / 2 + 7, 30 * turn + 5})
      if (int e = check(n, warps, 8)) {
        printf("n %llu warps %llu: %d\n", n, warps, e);
        return e;
      }
  }
  return 0;
}
"""


def test_dealing(tmp_path):
    from paper_1702_03154_gb300 import build_ext
    src, exe = tmp_path / "deal.cu", tmp_path / "deal"
    src.write_text(PROGRAM)
    subprocess.run([build_ext.nvcc()] + build_ext.ARCH + build_ext.NVCC_FLAGS +
                   ["-I" + CSRC, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
