// Geometry of the row ring that the activation quantisers stage their rows in
// (act_quant_bulk_kernel, codes_to_xdq_bulk_kernel in quant.cu): host
// arithmetic alone, so that it can be checked without a GPU.
#ifndef DQT_RING_GEOMETRY_H_
#define DQT_RING_GEOMETRY_H_

#include <cstdint>
#include <numeric>

namespace dqt {

constexpr int kAqbRing = 192 * 1024;  // shared-memory bytes of the row ring at most
constexpr int kRingWarps = 24;        // consumer warps at most

// Chunks of about 8 KB (rows of up to 8 KB are copied one per chunk; rpc rows
// each), then as many slots S as fit in `ring` bytes (48 at most) and up to
// kRingWarps consumer warps W; false when fewer than four chunks fit.  One
// producer thread issues a bulk copy about every 0.2 us whatever its size, so
// copies below ~8 KB leave the ring short of bytes in flight.
//
// S rpc is a multiple of W: the row that a warp waits for and the one that used
// the same place of the ring before, S rpc rows earlier, are then the same
// warp's.  A warp that could reach a slot before the slot's previous chunk had
// landed would wait on a phase parity that reads as complete.
inline bool ring_geometry(int64_t row_bytes, int64_t ring, int& rpc, int& W, int& S) {
  rpc = row_bytes >= 8192 ? 1 : static_cast<int>(8192 / row_bytes);
  const int64_t fit = ring / (rpc * row_bytes);
  if (fit < 4) return false;
  const int smax = static_cast<int>(fit < 48 ? fit : 48);
  S = W = 0;
  for (int w = kRingWarps < smax * rpc ? kRingWarps : smax * rpc; w > 0; --w) {
    const int unit = w / std::gcd(w, rpc);  // S is a multiple of it
    const int s = smax / unit * unit;
    if (w * s > W * S) {
      W = w;
      S = s;
    }
  }
  return true;
}

// Bytes of the ring for T rows on `sms` CTAs.  With more rows in flight than
// the outputs keep up with, reads and writes disturb each other: the more bytes
// are written per byte read, the smaller the ring.  It holds 128 KB of rows that
// become codes, 96 KB of rows that become bf16 images and 64 KB of codes that
// become X_tilde; all 192 KB where the CTA's rows are few enough to be asked for
// at once, and of rows beyond 8 KB, whose chunks are larger.  Against 192 KB
// throughout (replayed, us): codes of 8192 x 2048 11.7 -> 10.3, the code image
// there 12.5 -> 11.1, X_tilde from 16384 x 4096 codes 38.9 -> 35.6.  E4M3 rows
// with X_tilde want more in flight (4096 x 3584: 12.1, with 128 KB 12.6), until
// the launch moves more than one and a half times the L2 (16384 x 3584: 53.7 ->
// 51.3).
enum RingKind { RING_CODES, RING_IMAGES, RING_E4M3, RING_E4M3_XDQ, RING_XDQ };

inline int64_t ring_bytes(RingKind kind, int64_t T, int64_t K, int sms) {
  const int64_t row_bytes = kind == RING_XDQ ? K : 2 * K;
  if ((T + sms - 1) / sms * row_bytes <= 128 * 1024) return kAqbRing;
  const int64_t l2_most = 192000000;  // bytes moved
  switch (kind) {
    case RING_CODES: return row_bytes <= 8192 ? 128 * 1024 : kAqbRing;
    case RING_IMAGES: return row_bytes <= 8192 ? 96 * 1024 : kAqbRing;
    case RING_XDQ: return row_bytes <= 8192 ? 64 * 1024 : kAqbRing;
    case RING_E4M3:
      return row_bytes <= 8192 || (row_bytes <= 16384 && 3 * T * K > l2_most) ? 128 * 1024 : kAqbRing;
    case RING_E4M3_XDQ:
      return K > 2048 && row_bytes <= 16384 && 5 * T * K > l2_most ? 128 * 1024 : kAqbRing;
  }
  return kAqbRing;
}

}  // namespace dqt

#endif  // DQT_RING_GEOMETRY_H_
