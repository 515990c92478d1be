// Choice between the streaming and the tile form of the fused Chebyshev chunks.
#include <algorithm>

#include "internal.h"
#include "kernels_stream.cuh"

// Strips of ST_TX columns; the rows are cut so that the warps that registers and the ring
// allow on an SM (8 / 10 / 14 for 8 / 6 / 4 layers) just fill the chip once, at least 8 rows
// each (a strip starts with 2 S rows).
StreamCut cheb_stream_cut(int nx, int ny, int L) {
  StreamCut c;
  c.strips = (nx + ST_TX - 1) / ST_TX;
  const int per_sm = L <= 4 ? 14 : (L <= 6 ? 10 : 8);
  const int nseg = std::max(1, std::min(device_sms() * per_sm / c.strips, (ny + 7) / 8));
  c.rows = (ny + nseg - 1) / nseg;
  c.warps = c.strips * ((ny + c.rows - 1) / c.rows);
  return c;
}

// The form with the shorter estimate for four steps.  Measured on one chip over 320^2 to
// 2048^2 columns: a strip's row takes 0.75 + 0.4 n us at 8 layers (n warps on a scheduler;
// 6 layers 0.75 + 0.38 n, 4 layers 0.5 + 0.25 n), a round of tiles 4.2 (4.05, 3.8) us, and a
// launch about 2 us besides.  At 8 layers the line lies near 700^2 columns (640^2: 23.3
// against 23.5 us; 768^2: 25.4 against 32.6), at 4 near 420^2 (320^2: 12.1 against 10.6;
// 448^2: 12.3 against 14.3).
bool cheb_stream_pays(int nx, int ny, int L) {
  if (L > 8 || nx % 4 != 0 || (long long)nx * ny >= (1LL << 30)) return false;
  const StreamCut c = cheb_stream_cut(nx, ny, L);
  const int sms = device_sms(), n = (c.warps + 4 * sms - 1) / (4 * sms);
  const double row = L <= 4 ? 0.5 + 0.25 * n : (L <= 6 ? 0.75 + 0.38 * n : 0.75 + 0.4 * n);
  const double round = L <= 4 ? 3.8 : (L <= 6 ? 4.05 : 4.2);
  const long long tiles = (long long)((nx + 23) / 24) * ((ny + 23) / 24);
  return (c.rows + 2 * TB_H) * row < 2.0 + round * (double)((tiles + sms - 1) / sms);
}
