// Sizes of dda_scatter's far-field sums (farfield.cu): tiles of the digit
// products and the workspace of a call.  Host arithmetic only.
#pragma once

#include <algorithm>
#include <cstddef>

namespace dda {

constexpr int kFfSl = 7;              // digits per number
constexpr int kFfRows = 8;            // lattice rows per block
constexpr int kFfDirs = 32;           // directions per tile
constexpr int kFfJMax = 72;           // folded cells per chunk: 2 * 72 = 144 inner columns
constexpr int kFfBBlk = kFfSl * 1024; // bytes of one 16-column step of a direction tile

// inner dimension: H = ceil(nx / 2) folded cells in nchunk chunks of J, each
// ks steps of 16 columns (2 J padded with zeros)
struct FfShape { int H, J, nchunk, ks; };
inline FfShape ff_shape(int nx) {
  FfShape s;
  s.H = (nx + 1) / 2;
  s.nchunk = (s.H + kFfJMax - 1) / kFfJMax;
  s.J = (s.H + s.nchunk - 1) / s.nchunk;
  s.ks = (2 * s.J + 15) / 16;
  return s;
}
// row blocks x chunks of a lattice with nr rows
inline int ff_units(const FfShape& s, int nr) { return ((nr + kFfRows - 1) / kFfRows) * s.nchunk; }
inline int ff_tiles(int n_dir) { return (n_dir + kFfDirs - 1) / kFfDirs; }

// Workspace of the sums in up to `cap` directions at a time on a lattice of nx x
// ny x nz cells with nr rows: phase tables, their digits, the partial sums of
// `groups` row blocks in flight.  A call with more directions takes them in
// blocks, all of them with this one plan (the number of groups does not depend
// on the block, so a shorter last block needs no more than a full one).
struct FarfieldPlan {
  int cap, groups;
  size_t tab, pack, part;
  size_t bytes() const { return tab + pack + part; }
};
// bytes that the launches for nd directions write of each
inline size_t ff_tab_bytes(int nd, int nx, int ny, int nz) { return (size_t)nd * (nx + ny + nz) * 16; }
inline size_t ff_pack_bytes(int nd, int nx) {
  const FfShape s = ff_shape(nx);
  return (size_t)s.nchunk * ff_tiles(nd) * s.ks * kFfBBlk;
}
inline size_t ff_part_bytes(int nd, int groups) { return (size_t)groups * nd * 6 * sizeof(double); }

// groups: two row blocks per SM, no more than there are units, and partial
// sums of at most 64 MB
inline FarfieldPlan farfield_plan(int cap, int nx, int ny, int nz, int nr, int sms) {
  auto up256 = [](size_t b) { return (b + 255) / 256 * 256; };
  const long long fit = std::max(1LL, (64LL << 20) / (long long)ff_part_bytes(cap, 1));
  FarfieldPlan p;
  p.cap = cap;
  p.groups = (int)std::min<long long>(std::min(ff_units(ff_shape(nx), nr), 2 * sms), fit);
  p.tab = up256(ff_tab_bytes(cap, nx, ny, nz));
  p.pack = up256(ff_pack_bytes(cap, nx));
  p.part = up256(ff_part_bytes(cap, p.groups));
  return p;
}

}  // namespace dda
