// Closed-form footprints: unique sectors, unique lines and overlaps of the representative
// block, the wave and the y / z sets of a field, counted row by row without a bitmap: the
// geometry and the counting of a row, used by rows_kernel (ws_kernels.cu).  Which fields take
// it is decided by closed_form_ok (ws_plan.cpp).
//
// The points a level updates, whatever the folding, are the valid points of its blocks; the
// level's load (store) footprint is those points plus the raw offsets.  A level is a
// contiguous block range, so its points in one grid row (y, z) are one run of x.  With
// P = elem_bytes * stride_y, stride_x >= 0 and stride_z = Q * stride_y the rows are numbered
// r = (y - y0) + Q * (z - z0), their addresses step by P, and an offset splits into a
// whole number of rows d and a rest c of at most P / 2 bytes: the run of row r lands at
// row r + d, moved by c.  For one target row everything that lands there is
//   class P: runs that start at x = 0 (or every run of a level inside one block row),
//   class S: runs that start at the level's first block of its first block row,
// and within a class the ranges overlap or touch whenever a run is at least as long as the
// offsets are spread (checked by the host, closed_form_ok): the class is one byte range.
// Addresses matter modulo a line only, so the level's position is not limited; its size is only
// by the 32-bit counts of FootCounts (fewer than 2^32 sectors, checked by the host likewise).
// Two neighbouring target rows may still share sectors (row ends off the sector grid, offsets
// reaching over the row's end), so sectors and lines are counted in cells: the cell of target
// row t holds the lines from floor((A(t) + hmin) / 128) up to the next row's, A(t) being the
// address of its x = 0 and hmin the lowest byte any range starts at.  Ranges span less than
// two rows, so a cell receives ranges of its own row and of the row before it only.
#pragma once
#include <stdint.h>

#include "ws_internal.h"

#define WS_FOOT __device__ __forceinline__

namespace ws {

WS_FOOT uint32_t foot_div(uint32_t n, uint32_t m, uint32_t s) { return (__umulhi(n, m) + n) >> s; }
WS_FOOT uint32_t foot_div(uint32_t n, const FastDiv &f) { return foot_div(n, f.m, f.s); }
WS_FOOT int32_t foot_min(int32_t a, int32_t b) { return a < b ? a : b; }
WS_FOOT int32_t foot_max(int32_t a, int32_t b) { return a > b ? a : b; }
WS_FOOT uint32_t foot_umin(uint32_t a, uint32_t b) { return a < b ? a : b; }

constexpr int32_t kRowInf = 0x7fffffff;   // no further state change
constexpr int32_t kHullLo = 0x3fffffff, kHullHi = -0x3fffffff;   // an empty byte range
constexpr int32_t kSecLo = 0x40000000, kSecHi = 0x3fffffff;      // an empty sector range (length 0, 0 lines)

// A level in block rows: the rows R with R - first < count hold its points, as the run [lo, hi]
// (bytes from x = 0) except that the first row starts and the last one ends with the level.
struct alignas(16) FootLevel {
  int32_t first, count, lo, hi;
};

// Levels of one task: the wave (or the representative block) and, for loads, the y and z sets.
// The y set and, in the block rows before the last of their slab, the z set end early: the y
// set has no blocks in a slab's last block row, and the z set gives up to the y set what both
// hold (see the row walk).
struct alignas(16) FootGeo {
  FootLevel lev[3];
  // what a row's look-up reads, in 16-byte pieces
  int32_t z_count, z_hi;   // the z set's count and hi outside a slab's last block row
  int32_t full_hi;         // last byte of a whole row's run
  int32_t second;          // bit L: the runs of level L's first block row are class S
  uint32_t fq_m, fq_s;     // by q
  int32_t q;               // rows from plane to plane
  int32_t y0;              // grid row and plane of r = 0
  int32_t z0;
  int32_t z_end;           // first plane behind all levels
  int32_t n1;              // domain
  int32_t gy;              // block rows of a slab
  uint32_t fb1_m, fb1_s;   // by b1f
  uint32_t fb2_m, fb2_s;   // by b2f
  int32_t bp[12];          // block rows at which some level's state changes
  int32_t b1f, b2f;        // grid rows and planes of one block (B1, B2 * fold)
  int32_t rf[3], re[3];    // rows of each level, [rf, re)
  int32_t y_act;           // rows of one plane [0, y_act) hold all levels' points
};

// Fills level l of g, in two steps so that lanes can share them: foot_level for each of the
// three levels, then foot_finish.  Candidate c, rows q from plane to plane, esx >= 0 bytes from
// point to point; the wave and its y and z sets, or the representative block alone.
WS_FOOT void foot_level(FootGeo &g, const DCfg &c, int32_t q, int32_t esx, bool block, int l) {
  const int32_t gx = c.g[0], B0 = c.B[0], N0 = c.N[0];
  const int32_t lo = block ? (l == 0 ? (int32_t)c.rep : 0) : (int32_t)(l == 0 ? c.s : l == 1 ? c.y_lo : c.z_lo);
  const int32_t hi = block ? (l == 0 ? lo + 1 : 0) : (int32_t)(l == 0 ? c.s + c.weff : l == 1 ? c.y_hi : c.z_hi);
  const int32_t Ra = (int32_t)foot_div((uint32_t)lo, c.fd_gx), Rb = (int32_t)foot_div((uint32_t)hi, c.fd_gx);
  FootLevel L;
  L.first = Ra;
  L.count = L.lo = L.hi = 0;
  g.bp[4 * l] = Ra;
  g.bp[4 * l + 1] = Ra + 1;
  g.bp[4 * l + 2] = Rb;
  g.bp[4 * l + 3] = Rb + 1;
  auto last = [&](int32_t b, int32_t &count, int32_t &end) {   // of blocks [lo, b), b > lo
    const int32_t Rl = (int32_t)foot_div((uint32_t)(b - 1), c.fd_gx);
    count = Rl - Ra + 1;
    end = esx * (foot_min((b - Rl * gx) * B0, N0) - 1);
  };
  if (hi > lo) {
    last(hi, L.count, L.hi);
    L.lo = esx * ((lo - Ra * gx) * B0);
  }
  if (l == 2) {
    g.z_count = L.count;
    g.z_hi = L.hi;
    if (L.count > 0 && c.y_hi > c.y_lo && c.y_lo < hi) {
      g.z_count = 0;
      if (c.y_lo > lo) last((int32_t)c.y_lo, g.z_count, g.z_hi);
    }
  }
  g.rf[l] = lo - Ra * gx > 0 && L.count > 1;   // (until foot_finish) class S in its first block row
  g.lev[l] = L;
}

WS_FOOT void foot_finish(FootGeo &g, const DCfg &c, int32_t q, int32_t esx) {
  const int32_t fy = c.fold_axis == 1 ? c.fold : 1, fz = c.fold_axis == 2 ? c.fold : 1;
  const int32_t gy = c.g[1], n2 = c.N[2], b1f = c.B[1] * fy, b2f = c.B[2] * fz;
  g.gy = gy;
  g.b1f = b1f;
  g.b2f = b2f;
  g.n1 = c.N[1];
  g.q = q;
  g.fb1_m = c.fd_b1f.m;
  g.fb1_s = c.fd_b1f.s;
  g.fb2_m = c.fd_b2f.m;
  g.fb2_s = c.fd_b2f.s;
  g.full_hi = esx * (c.N[0] - 1);
  g.y0 = g.z0 = kRowInf;
  g.z_end = 0;
  g.second = 0;
  int32_t za[3], zb[3], ya[3], ye[3];
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    const FootLevel L = g.lev[l];
    za[l] = zb[l] = ya[l] = ye[l] = 0;
    if (L.count == 0) continue;
    const int32_t Rl = L.first + L.count - 1;
    za[l] = (int32_t)foot_div((uint32_t)L.first, c.fd_gy);
    zb[l] = (int32_t)foot_div((uint32_t)Rl, c.fd_gy);
    ya[l] = (L.first - za[l] * gy) * b1f;
    ye[l] = foot_min((Rl - zb[l] * gy + 1) * b1f, g.n1);
    g.y0 = foot_min(g.y0, za[l] == zb[l] ? ya[l] : 0);
    g.z0 = foot_min(g.z0, za[l] * b2f);
    g.z_end = foot_max(g.z_end, foot_min((zb[l] + 1) * b2f, n2));
    if (g.rf[l]) g.second |= 1 << l;
  }
  g.y_act = 0;
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    g.rf[l] = g.re[l] = 0;
    if (g.lev[l].count == 0) continue;
    g.rf[l] = ya[l] - g.y0 + q * (za[l] * b2f - g.z0);
    g.re[l] = ye[l] - g.y0 + q * (foot_min((zb[l] + 1) * b2f, n2) - 1 - g.z0);
    g.y_act = foot_max(g.y_act, (za[l] == zb[l] ? ye[l] : g.n1) - g.y0);
  }
}

// Byte ranges of one row, per level: [0] class P, [1] class S (empty: lo > hi).
struct FootHull {
  int32_t lo[3][2], hi[3][2];
  WS_FOOT void clear() {
#pragma unroll
    for (int l = 0; l < 3; ++l)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        lo[l][c] = kHullLo;
        hi[l][c] = kHullHi;
      }
  }
};

// Runs of the first nl levels (1 or 3) in one row: [lo, hi], and bit L of `second` where level L's
// is class S.
struct FootRow {
  int32_t lo[3], hi[3];
  uint32_t present, second;
};

// Looks up row r (without branches: the lanes' rows differ).  Returns the next row at which the
// state of a level may change (want_next; else anything).
WS_FOOT int32_t foot_row(const FootGeo &g, int nl, int32_t r, bool want_next, FootRow &o) {
  const int32_t zr = (int32_t)foot_div((uint32_t)r, g.fq_m, g.fq_s), row0 = zr * g.q;   // row0: the plane's first row
  const int32_t y = g.y0 + (r - row0), z = g.z0 + zr;
  const bool in = r >= 0 && z < g.z_end && y < g.n1;
  const int32_t by = (int32_t)foot_div((uint32_t)y, g.fb1_m, g.fb1_s), bz = (int32_t)foot_div((uint32_t)z, g.fb2_m, g.fb2_s);
  const int32_t R = by + g.gy * bz;
  const bool last = by == g.gy - 1;
  o.present = o.second = 0;
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    if (l > 0 && nl == 1) break;
    const FootLevel L = g.lev[l];
    const int32_t count = l == 0 || (l == 1) != last ? L.count : l == 1 ? 0 : g.z_count;
    const int32_t hi = l < 2 || last ? L.hi : g.z_hi;
    const uint32_t k = (uint32_t)(R - L.first);
    const bool on = in && k < (uint32_t)count, first = k == 0;
    o.lo[l] = first ? L.lo : 0;
    o.hi[l] = (int32_t)k + 1 == count ? hi : g.full_hi;
    o.present |= on ? 1u << l : 0u;
    o.second |= on && first ? (uint32_t)g.second & (1u << l) : 0u;
  }
  if (!want_next) return 0;
  // the states hold up to the next block row of bp, the slab's last block row or the plane's end
  uint32_t step = (uint32_t)(g.gy - by - 1);
#pragma unroll
  for (int k = 0; k < 12; ++k) step = foot_umin(step, (uint32_t)(g.bp[k] - R - 1));
  int32_t byn = by + 1 + (int32_t)step;
  if (!last) byn = foot_min(byn, g.gy - 1);
  const int32_t next = foot_min(row0 + (foot_min(byn * g.b1f, g.n1) - g.y0), row0 + g.q);
  return r < 0 ? 0 : z >= g.z_end ? kRowInf : y >= g.n1 ? row0 + g.q : next;
}

// Adds a row's runs, moved by [clo, chi], to h.
WS_FOOT void foot_add(const FootRow &o, int nl, int32_t clo, int32_t chi, FootHull &h) {
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    if (l > 0 && nl == 1) break;
    const bool p = ((o.present & ~o.second) >> l) & 1u;
    h.lo[l][0] = p ? foot_min(h.lo[l][0], o.lo[l] + clo) : h.lo[l][0];
    h.hi[l][0] = p ? foot_max(h.hi[l][0], o.hi[l] + chi) : h.hi[l][0];
  }
  if (o.second) {   // (few rows)
#pragma unroll
    for (int l = 0; l < 3; ++l)
      if ((o.second >> l) & 1u) {
        h.lo[l][1] = foot_min(h.lo[l][1], o.lo[l] + clo);
        h.hi[l][1] = foot_max(h.hi[l][1], o.hi[l] + chi);
      }
  }
}

// The two ranges of every level as one, [lo, hi].  Returns the levels present (bit l), and bit 3
// where two ranges leave a gap between them (a start at most one sector behind an end leaves no
// sector out): then one range will not do.
WS_FOOT uint32_t foot_join(const FootHull &h, int nl, int32_t lo[3], int32_t hi[3]) {
  uint32_t r = 0;
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    lo[l] = kHullLo;
    hi[l] = kHullHi;
    if (l > 0 && nl == 1) continue;
    lo[l] = foot_min(h.lo[l][0], h.lo[l][1]);
    hi[l] = foot_max(h.hi[l][0], h.hi[l][1]);
    if (lo[l] <= hi[l]) r |= 1u << l;
    if (foot_max(h.lo[l][0], h.lo[l][1]) > foot_min(h.hi[l][0], h.hi[l][1]) + 32 && h.lo[l][0] <= h.hi[l][0] &&
        h.lo[l][1] <= h.hi[l][1])
      r |= 8u;
  }
  return r;
}

// Planes from row r's target plane on (rows [r, r + q) move together) over which the states
// repeat from plane to plane: up to the end of the blocks' slab, or of the levels.
WS_FOOT int32_t foot_repeat(const FootGeo &g, int32_t r) {
  int32_t z = r >= 0 ? (int32_t)foot_div((uint32_t)r, g.fq_m, g.fq_s)
                     : -(int32_t)foot_div((uint32_t)(g.q - 1 - r), g.fq_m, g.fq_s);
  const int32_t yr = r - z * g.q;
  int32_t n = kRowInf;
#pragma unroll
  for (int k = 0; k < 2; ++k, ++z) {
    if (k == 0 ? yr >= g.y_act : yr == 0) continue;   // no rows of that plane with points
    int32_t m = kRowInf;
    const int32_t zz = z + g.z0;
    if (z < 0) m = -z;
    else if (zz < g.z_end) m = foot_min(((int32_t)foot_div((uint32_t)zz, g.fb2_m, g.fb2_s) + 1) * g.b2f, g.z_end) - zz;
    n = foot_min(n, m);
  }
  return n;
}

// Slab of plane z (from row 0's), -1 where no level has rows.
WS_FOOT int32_t foot_slab(const FootGeo &g, int32_t z) {
  const int32_t zz = z + g.z0;
  return z < 0 || zz >= g.z_end ? -1 : (int32_t)foot_div((uint32_t)zz, g.fb2_m, g.fb2_s);
}

// What rows r .. r + n - 1 (n <= q + 2) depend on: the row's place in its plane and the slabs of
// the planes they touch with rows that hold points (-2: none touched).  Two displacements that
// agree on these look up the same states throughout.  Returns whether any state can be present.
WS_FOOT bool foot_key(const FootGeo &g, int32_t r, int32_t n, int32_t key[4]) {
  const int32_t z = r >= 0 ? (int32_t)foot_div((uint32_t)r, g.fq_m, g.fq_s)
                           : -(int32_t)foot_div((uint32_t)(g.q - 1 - r), g.fq_m, g.fq_s);
  const int32_t yr = r - z * g.q;
  key[0] = yr;
  key[1] = yr < g.y_act ? foot_slab(g, z) : -2;
  key[2] = yr + n > g.q ? foot_slab(g, z + 1) : -2;
  key[3] = yr + n > 2 * g.q ? foot_slab(g, z + 2) : -2;
  return key[1] >= 0 || key[2] >= 0 || key[3] >= 0;
}

// What a task counts: sectors and lines of the first level, lines of the y and z sets, the
// first level's sectors shared with the y set, and with the z set outside the y set.  A level has
// fewer than 2^32 sectors (closed_form_ok), so no lane's and no warp's sum overflows; ovz is
// added to and taken from modulo 2^32.
struct FootCounts {
  uint32_t sec, lin, ylin, zlin, ovy, ovz;
};

struct SecRange {
  int32_t a, b;
};
WS_FOOT int32_t foot_len(const SecRange &r) { return r.b - r.a + 1; }
WS_FOOT int32_t foot_lines(const SecRange &r) { return (r.b >> 2) - (r.a >> 2) + 1; }
WS_FOOT int32_t foot_ov(const SecRange &p, const SecRange &q) {
  return foot_max(foot_min(p.b, q.b) - foot_max(p.a, q.a) + 1, 0);
}
WS_FOOT SecRange foot_cut(const SecRange &p, const SecRange &q) {
  SecRange r{foot_max(p.a, q.a), foot_min(p.b, q.b)};
  if (r.a > r.b) r = {kSecLo, kSecHi};
  return r;
}
// Sectors of the byte range [lo, hi] relative to address A, cut to [c0, c1).
WS_FOOT SecRange foot_clip(int32_t A, int32_t lo, int32_t hi, int32_t c0, int32_t c1) {
  SecRange r{kSecLo, kSecHi};
  if (lo <= hi) {
    const int32_t a = foot_max((A + lo) >> 5, c0), b = foot_min((A + hi) >> 5, c1 - 1);
    if (a <= b) r = {a, b};
  }
  return r;
}
// Two ranges as two disjoint ones that do not touch (the second empty when they did).
WS_FOOT void foot_merge(SecRange &p, SecRange &q) {
  if (foot_max(p.a, q.a) <= foot_min(p.b, q.b) + 1) {
    p = {foot_min(p.a, q.a), foot_max(p.b, q.b)};
    q = {kSecLo, kSecHi};
  }
}
// Lines of two disjoint ranges that do not touch (they can still meet in one line).
WS_FOOT int32_t foot_lines2(const SecRange &p, const SecRange &q) {
  return foot_lines(p) + foot_lines(q) - foot_max(foot_min(p.b >> 2, q.b >> 2) - foot_max(p.a >> 2, q.a >> 2) + 1, 0);
}

// Cell of the target row at address A (pitch P): sectors [c0, c1).
WS_FOOT void foot_cell(int32_t A, int32_t P, int32_t hmin, int32_t &c0, int32_t &c1) {
  c0 = ((A + hmin) >> 7) << 2;
  c1 = ((A + P + hmin) >> 7) << 2;
}

// Counts one cell `mult` times when every level has at most one range per row: lo / hi are those
// of the row (cur) and of the row before it (prv); bit l of `levels`: level l may be present, bit 4:
// the z set's lines are wanted.
WS_FOOT void foot_count(const int32_t clo[3], const int32_t chi[3], const int32_t plo[3], const int32_t phi[3],
                      int32_t A, int32_t P, int32_t hmin, uint32_t mult, uint32_t levels, FootCounts &out) {
  int32_t c0, c1;
  foot_cell(A, P, hmin, c0, c1);
  if (c1 <= c0) return;
  SecRange p[3], q[3];
  auto part = [&](int l) {
    p[l] = foot_clip(A - P, plo[l], phi[l], c0, c1);
    q[l] = foot_clip(A, clo[l], chi[l], c0, c1);
    foot_merge(p[l], q[l]);
  };
  if (levels & 1u) {
    part(0);
    out.sec += mult * (uint32_t)(foot_len(p[0]) + foot_len(q[0]));
    out.lin += mult * (uint32_t)foot_lines2(p[0], q[0]);
  }
  if (levels & 4u) {
    part(2);
    if (levels & 16u) out.zlin += mult * (uint32_t)foot_lines2(p[2], q[2]);
    if (levels & 1u)
      out.ovz += mult * (uint32_t)(foot_ov(p[0], p[2]) + foot_ov(p[0], q[2]) + foot_ov(q[0], p[2]) + foot_ov(q[0], q[2]));
  }
  if (levels & 2u) {
    part(1);
    out.ylin += mult * (uint32_t)foot_lines2(p[1], q[1]);
    if (levels & 1u) {
      int32_t y = 0, yz = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const SecRange wy = foot_cut(k & 1 ? p[0] : q[0], k & 2 ? p[1] : q[1]);
        y += foot_len(wy);
        if (levels & 4u) yz += foot_ov(wy, p[2]) + foot_ov(wy, q[2]);
      }
      out.ovy += mult * (uint32_t)y;
      out.ovz -= mult * (uint32_t)yz;
    }
  }
}

// Lines of the first level's cell alone.
WS_FOOT uint32_t foot_count_lines(int32_t clo, int32_t chi, int32_t plo, int32_t phi, int32_t A, int32_t P, int32_t hmin) {
  int32_t c0, c1;
  foot_cell(A, P, hmin, c0, c1);
  SecRange p = foot_clip(A - P, plo, phi, c0, c1), q = foot_clip(A, clo, chi, c0, c1);
  foot_merge(p, q);
  return (uint32_t)foot_lines2(p, q);
}

// foot_count for up to two ranges a level and row: walks the elementary pieces of the cell from
// left to right.
WS_FOOT void foot_count_pieces(const FootHull &cur, const FootHull &prv, int32_t A, int32_t P, int32_t hmin,
                             uint32_t mult, FootCounts &out) {
  int32_t c0, c1;
  foot_cell(A, P, hmin, c0, c1);
  SecRange s[3][4];
  int32_t last[3];   // last line counted of each level
  for (int l = 0; l < 3; ++l) {
    last[l] = -0x7fffffff;
    for (int c = 0; c < 2; ++c) {
      s[l][2 * c] = foot_clip(A - P, prv.lo[l][c], prv.hi[l][c], c0, c1);
      s[l][2 * c + 1] = foot_clip(A, cur.lo[l][c], cur.hi[l][c], c0, c1);
    }
  }
  for (int32_t pos = c0; pos < c1;) {
    int32_t nx = c1;
    bool in[3];
    for (int l = 0; l < 3; ++l) {
      in[l] = false;
      for (int k = 0; k < 4; ++k) {
        if (s[l][k].a > pos) nx = foot_min(nx, s[l][k].a);
        else if (s[l][k].b >= pos) {
          in[l] = true;
          nx = foot_min(nx, s[l][k].b + 1);
        }
      }
    }
    uint32_t ln[3];
    for (int l = 0; l < 3; ++l) {
      ln[l] = 0;
      if (in[l]) {
        ln[l] = mult * (uint32_t)(((nx - 1) >> 2) - (pos >> 2) + ((pos >> 2) != last[l] ? 1 : 0));
        last[l] = (nx - 1) >> 2;
      }
    }
    const uint32_t n = mult * (uint32_t)(nx - pos);
    out.lin += ln[0];
    out.ylin += ln[1];
    out.zlin += ln[2];
    if (in[0]) {
      out.sec += n;
      if (in[1]) out.ovy += n;
      else if (in[2]) out.ovz += n;
    }
    pos = nx;
  }
}

// The target rows of a load or store task, [t[2], t[3]) behind [t[0], t[1]): the second range
// covers the first level and the y set, the first one what only the z set reaches (empty when
// its lines are counted on the wave, moved).  dmin / dmax: smallest and largest displacement.  Ranges of a
// level's last row may reach into the cell after it.
WS_FOOT void foot_targets(const FootGeo &g, int nl, int32_t dmin, int32_t dmax, bool z_alone, int32_t t[4]) {
  t[2] = g.rf[0] + dmin;
  t[3] = g.re[0] + dmax + 1;
  if (nl == 3 && g.lev[1].count > 0) {
    t[2] = foot_min(t[2], g.rf[1] + dmin);
    t[3] = foot_max(t[3], g.re[1] + dmax + 1);
  }
  t[0] = t[1] = t[2];
  if (nl == 3 && z_alone && g.lev[2].count > 0) {
    t[0] = foot_min(t[2], g.rf[2] + dmin);
    t[3] = foot_max(t[3], g.re[2] + dmax + 1);
    t[1] = foot_min(t[2], foot_max(t[0], g.re[2] + dmax + 1));
    if (t[1] == t[2]) {
      t[2] = t[0];
      t[1] = t[0];
    }
  }
}

// Threads of blocks [0, n) of a candidate in launch order: `last` counts only those of the
// last block row of each slab, `part` only those with fewer valid folded points than the fold.
static __device__ __noinline__ int64_t foot_threads(const DCfg &c, int64_t n, bool last, bool part) {
  const uint32_t R = (uint32_t)n / (uint32_t)c.g[0];   // block ids stay below 2^31
  const int64_t gy = c.g[1], bz = R / (uint32_t)c.g[1];
  const int64_t bx = (uint32_t)n - R * (uint32_t)c.g[0], by = R - (uint32_t)bz * (uint32_t)c.g[1];
  const int32_t fy = c.fold_axis == 1 ? c.fold : 1, fz = c.fold_axis == 2 ? c.fold : 1;
  const int64_t m1 = (c.N[1] + fy - 1) / fy, m2 = (c.N[2] + fz - 1) / fz;   // thread rows in y and z
  const bool py = part && fy > 1, pz = part && fz > 1;
  if (part && !(py && c.N[1] % fy) && !(pz && c.N[2] % fz)) return 0;
  auto ysum = [&](int64_t b) -> int64_t {   // thread rows of block rows [0, b)
    if (py) return b == gy ? 1 : 0;
    const int64_t all = b * c.B[1] < m1 ? b * c.B[1] : m1;
    return !last ? all : b == gy ? m1 - (gy - 1) * c.B[1] : 0;
  };
  auto zsum = [&](int64_t b) -> int64_t {
    if (pz) return b == c.g[2] ? 1 : 0;
    return b * c.B[2] < m2 ? b * c.B[2] : m2;
  };
  const int64_t x = bx * c.B[0] < c.N[0] ? bx * c.B[0] : c.N[0];
  const int64_t z1 = bz < c.g[2] ? zsum(bz + 1) - zsum(bz) : 0;
  return c.N[0] * ysum(gy) * zsum(bz) + (c.N[0] * ysum(by) + x * (ysum(by + 1) - ysum(by))) * z1;
}

// Threads of the levels as sums of twelve such counts, term j of level j < 2 ? 0 : j < 6 ? 1 : 2
// (wave, y set, z set): the wave's range; the y set's less its blocks in last block rows; the
// z set's less what it shares with the y set.
WS_FOOT int64_t foot_thread_term(const DCfg &c, int j, bool part) {
  const bool has_y = c.y_hi > c.y_lo, has_z = c.z_hi > c.z_lo;
  const int64_t a = c.z_lo > c.y_lo ? c.z_lo : c.y_lo, b = c.z_hi < c.y_hi ? c.z_hi : c.y_hi;
  if ((j >= 2 && j < 6 && !has_y) || (j >= 6 && !has_z) || (j >= 8 && !(has_y && b > a))) return 0;
  const int64_t n = j == 0   ? c.s + c.weff
                    : j == 1 ? c.s
                    : j < 6  ? (j & 1 ? c.y_lo : c.y_hi)
                    : j == 6 ? c.z_hi
                    : j == 7 ? c.z_lo
                    : j & 1  ? a
                             : b;
  const bool last = j == 4 || j == 5 || j >= 10, minus = j == 1 || j == 3 || j == 4 || j == 7 || j == 8 || j == 11;
  const int64_t t = foot_threads(c, n, last, part);
  return minus ? -t : t;
}

}  // namespace ws
