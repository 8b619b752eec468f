// Geometry of the scored blocks of the selection (Eq. 8), shared by the selection kernels and the
// short-history kernels.
#pragma once
#include "common.cuh"

namespace blossom {

struct SelGeom {
  int n;       // scored blocks per (batch, key/value head): Mc, or M in the plain mode
  int l, s;    // their length and stride in positions
  int rs, rl;  // Bk / s and l / s, the two sums of Eq. 11 (1, 1 in the plain mode)
  int plain;
};

inline SelGeom sel_geom(const Shape &sh) {
  SelGeom g;
  if (sh.cmp_l > 0) {
    g.n = sh.Mc; g.l = sh.cmp_l; g.s = sh.cmp_s; g.rs = sh.Bk / sh.cmp_s; g.rl = sh.cmp_l / sh.cmp_s;
    g.plain = 0;
  } else {
    g.n = sh.M; g.l = sh.Bk; g.s = sh.Bk; g.rs = 1; g.rl = 1; g.plain = 1;
  }
  return g;
}

// scored blocks 0 .. nc - 1 end before query block b starts
__device__ __forceinline__ int n_candidates(const Shape &sh, const SelGeom &g, int b) {
  if (g.plain) return b;
  const int start = b * sh.Bk;
  return start >= g.l ? min(g.n, (start - g.l) / g.s + 1) : 0;
}
// the first scored block that holds a valid key (pad0 = number of padded positions)
__device__ __forceinline__ int first_live_scored(const SelGeom &g, int pad0) {
  return pad0 < g.l ? 0 : (pad0 - g.l) / g.s + 1;
}
// A score as the rankings take it: sums of probabilities are not negative, and what is no number ranks
// below all of them (but above the own block's -infinity), so that a ranking is an order whatever the inputs
// and a row never gets more blocks than it has room for.
template <typename F>
__device__ __forceinline__ F rankable(F x) { return x == x ? x : (F)-1; }

}  // namespace blossom
