// How many fine bins a layer of scalar weights may use (host side of the interval form).
//
// An iteration looks at all weights of the fine bins the centroids lie in, so a large layer gains from more bins; what they cost
// is in the build, which writes two bytes per weight to places that lie the farther apart.  The number of bins per coarse bin
// is a power of two, so 40960 instead of 32768 doubles it for the third of all ratios of range to tau where the product falls
// between the two.  There (40960 over 32768, forward and Jacobian-free backward, six such ratios, k = 2, 4, 8 and 16), one layer:
//   M weights      10           12 .. 16     24 .. 44     48           56           64
//   10 iterations   .99 - 1.07   .99 - 1.10  1.01 - 1.10   .98 - 1.05   .91 -  .99   .86 -  .94
//   30             1.01 - 1.16  1.01 - 1.19  1.03 - 1.22  1.03 - 1.15   .95 - 1.08   .90 - 1.04
//   100            1.06 - 1.29  1.05 - 1.34  1.09 - 1.46  1.13 - 1.39  1.07 - 1.32  1.00 - 1.26
// Smaller layers gain or lose by the ratio (30 iterations: 4 M .95 to 1.12, 8 M .97 to 1.15).  Beyond 48 M the places of the call's
// weights and the weights that stream by no longer fit in the 126 MB of L2, and every bin's part of a sector goes to memory by
// itself; so it is in calls of several large layers (30 iterations: 2 x 8 M .96 to 1.08, 3 x 16 M .93 to 1.02, 8 x 8 M .80 to .86).
#pragma once

namespace idkm {

constexpr int SC_FINE_MOST = 40960;    // a layer of at least SC_FINE_ROWS weights that has most of at most SC_FINE_CALL
constexpr int SC_FINE_BIG = 32768;     // the other ones of the SC_BIG_LAYERS largest
constexpr int SC_FINE_SMALL = 16384;   // the rest
constexpr long long SC_FINE_ROWS = 10LL << 20, SC_FINE_CALL = 44LL << 20;
constexpr int SC_BIG_LAYERS = 8;

// A layer of `rows` weights that `larger` others of the call's m_total come before in size.
inline int scalar_fine_bins(long long rows, int larger, long long m_total) {
  if (larger >= SC_BIG_LAYERS) return SC_FINE_SMALL;
  return rows >= SC_FINE_ROWS && 2 * rows > m_total && m_total <= SC_FINE_CALL ? SC_FINE_MOST : SC_FINE_BIG;
}
// Room for n_layers layers of m_total weights, however these are dealt to them; never less than for a smaller call.
inline int scalar_fine_total(long long m_total, int n_layers) {
  const int big = n_layers < SC_BIG_LAYERS ? n_layers : SC_BIG_LAYERS;
  return big * SC_FINE_BIG + (n_layers - big) * SC_FINE_SMALL + (m_total >= SC_FINE_ROWS ? SC_FINE_MOST - SC_FINE_BIG : 0);
}

}  // namespace idkm
