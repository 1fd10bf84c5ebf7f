// Tiles of the marching level kernels (k_march.cu): host arithmetic only.
#pragma once

#include <algorithm>
#include <vector>

namespace smr {

// Tile of a launch: a CTA takes nbx parent boxes, one chunk of ncol columns x
// HN parts and one range of theta rows with T threads; the staged input
// columns number cc.  mcc, mper: multiply-high reciprocals of cc and ncol
// (exact for the small counts divided here).
struct MarchTile {
  int nbx, ncol, cc, T;
  int nbg, nck, nhk;                           // box groups, column chunks, part chunks
  unsigned mcc, mper;
};

inline unsigned magic_of(unsigned d) { return d > 1 ? (unsigned)(((1ull << 32) + d - 1) / d) : 0u; }

// Columns and boxes of a CTA.  lanes: threads per column; start[j]: first
// staged input column of output column j; width: input columns one output
// column reads; per input column, `boxcopies` 16-byte copies per box and part
// and `extra` more.  Whole rows where a row is short (of several boxes if
// `pack`), chunks of columns where it is long; at most `most` threads and
// nk copies per thread (threads without a column only copy).  The chunks are
// divided until that holds; T stays above `most` where a single column's
// copies are more than that.
inline MarchTile march_tile(int most, int nk, int lanes, int hn, bool pack, int nbox, int nph, int NT,
                            const std::vector<int>& start, int width, int boxcopies, int extra) {
  MarchTile m;
  m.nhk = NT / hn;
  const int cols = most / lanes;
  m.ncol = nph + 1;
  // n counts up to nph, where chunks are single columns: the normalised nck, the
  // fewest chunks of ncol columns, may be below n
  for (int n = (nph + cols - 1) / cols; m.ncol > 1; ++n) {
    const int ncol = (nph + n - 1) / n;
    if (ncol == m.ncol) continue;
    m.ncol = ncol;
    m.nck = (nph + ncol - 1) / ncol;
    m.cc = 0;
    for (int p = 0; p < nph; p += ncol)
      m.cc = std::max(m.cc, start[std::min(nph, p + ncol) - 1] + width - start[p]);
    m.nbx = !pack || m.nck > 1 ? 1 : std::max(1, std::min(nbox, most / (ncol * lanes)));
    auto threads = [&]() {
      const int E = m.cc * (m.nbx * boxcopies * hn + extra);
      return std::max(m.nbx * ncol * lanes, (E + nk - 1) / nk);
    };
    while (m.nbx > 1 && threads() > most) --m.nbx;
    m.T = (threads() + 31) / 32 * 32;
    if (m.T <= most) break;
  }
  m.nbg = (nbox + m.nbx - 1) / m.nbx;
  m.mcc = magic_of(m.cc);
  m.mper = magic_of(m.ncol);
  return m;
}

// Tile of an anterpolation whose child columns read `taps` consecutive parent
// columns: as many taps a launch as fit a CTA (*per_launch), all of them but for
// stencils of many hundred columns.
inline MarchTile anterp_tile(int most, int nk, int lanes, int hn, bool pack, int nbox, int nph, int NT,
                             const std::vector<int>& start, int taps, int extra, int* per_launch) {
  for (int n = 1;; ++n) {
    *per_launch = (taps + n - 1) / n;
    const MarchTile m = march_tile(most, nk, lanes, hn, pack, nbox, nph, NT, start, *per_launch, 1, extra);
    if (m.T <= most || *per_launch == 1) return m;
  }
}

// Theta rows of a CTA: the split of `rows` that finishes first when `per_sm`
// CTAs of an SM run at full speed at a time.  A CTA costs its rows plus about
// seven: the three stencil rows a range shares with its neighbour, and the
// ring's start.
inline int march_rows(const MarchTile& m, int rows, int per_sm, int most) {
  const long long ctas = (long long)m.nbg * m.nck * m.nhk, slots = 152LL * std::max(1, per_sm);
  int best = std::min(rows, most);
  long long cost = -1;
  for (int parts = 1; parts <= std::max(1, rows / 2); ++parts) {
    const int t = (rows + parts - 1) / parts;
    if (t > most) continue;
    const long long k = (ctas * ((rows + t - 1) / t) + slots - 1) / slots * (t + 7);
    if (cost < 0 || k < cost) {
      cost = k;
      best = t;
    }
  }
  return best;
}

}  // namespace smr
