"""The row ring of the activation quantisers (csrc/ring_geometry.h) over row
lengths, row counts and outputs, on the host: a warp's rows come back to its own
places of the ring (anything else could wait on a phase that reads as complete),
the ring fits, and every row length that fits 192 KB four times is taken."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2412_04787_gb300", "csrc")

SRC = r"""
#include "ring_geometry.h"
#include <cstdio>
#include <initializer_list>
using namespace dqt;
int main() {
  const int64_t Ts[] = {1, 64, 152, 1000, 4096, 8192, 16384, 200000, 2147483647};
  long n = 0;
  for (int kind = RING_CODES; kind <= RING_XDQ; ++kind)
    for (int64_t K = 8; K <= 60000; K += K < 9000 ? 8 : 104) {
      if (kind == RING_XDQ && K % 16) continue;
      const int64_t row = kind == RING_XDQ ? K : 2 * K;
      const int64_t chunk = row >= 8192 ? row : 8192 / row * row;
      for (int64_t T : Ts)
        for (int sms : {148, 152}) {
          int rpc = 0, W = 0, S = 0;
          const int64_t ring = ring_bytes(static_cast<RingKind>(kind), T, K, sms);
          const bool ok = ring_geometry(row, ring, rpc, W, S);
          if (ok != (kAqbRing / chunk >= 4)) { std::printf("taken %d %ld\n", kind, (long)K); return 1; }
          if (!ok) continue;
          ++n;
          if (ring > kAqbRing || rpc < 1 || W < 1 || W > kRingWarps || S < 1 || S > 48 ||
              S * rpc % W != 0 || S * rpc * row > ring || rpc * row != chunk) {
            std::printf("%d K=%ld T=%ld: rpc %d W %d S %d\n", kind, (long)K, (long)T, rpc, W, S);
            return 1;
          }
        }
    }
  std::printf("%ld\n", n);
}
"""


def test_ring_geometry(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 50000
