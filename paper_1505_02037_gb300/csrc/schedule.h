// The work list of the SYNC step that runs the moment pass and the collide pass
// in one launch (k_step in kernels.cuh). Plain arithmetic, for host and device.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define LBNR_HD __host__ __device__ __forceinline__
#else
#define LBNR_HD inline
#endif

namespace lbnr {

// n / d for n < 2^31 by a multiply-high with a precomputed round-up
// multiplier (Granlund-Montgomery); d = 1 is passed through.
struct FastDiv {
  uint32_t d, mul, shift;
  LBNR_HD uint32_t div(uint32_t n) const {
#ifdef __CUDA_ARCH__
    return d == 1 ? n : (__umulhi(n, mul) >> shift);
#else
    return d == 1 ? n : (uint32_t)(((uint64_t)n * mul) >> 32) >> shift;
#endif
  }
};
inline FastDiv make_fastdiv(uint32_t d) {
  FastDiv f{d, 0, 0};
  if (d > 1) {
    uint32_t l = 0;
    while ((1ull << l) < d) ++l;  // ceil(log2 d)
    const uint32_t p = 31 + l;
    f.mul = (uint32_t)(((1ull << p) + d - 1) / d);
    f.shift = p - 32;
  }
  return f;
}

// The lattice as planes across its slowest axis (3D: nx ny cells, 2D: a row,
// 1D: a cell). A unit is a run of whole planes or, where one plane alone is
// larger than a unit should be, one strip of rows of one plane. Both passes go
// through the units of a strip plane by plane, strip after strip. Boundaries
// are rounded up to whole 32-cell tiles.
struct Schedule {
  uint32_t* cnt;       // [0] next item, [1 + p] finished moment items at list position p
  uint32_t* cnt_next;  // the counters of the next step, zeroed by this one
  uint32_t plane, row; // cells of a plane, and of a row within it
  uint32_t strips;     // strips along y (1: whole planes)
  uint32_t upu;        // units per strip
  uint32_t pq, pr;     // planes per unit: pq, and one more in the first pr units
  uint32_t rq, rr;     // rows per strip, likewise
  uint32_t slots;      // items per list position
  uint32_t units;      // strips * upu
  uint32_t wrap;       // the moment pass starts with this many of a strip's last units
  uint32_t ahead;      // list distance from a unit to that of its last upper neighbour
  uint32_t lead;       // list distance between the two passes
  FastDiv fslots, fupu;
  uint32_t items;
  uint32_t quota;      // finished moment items that complete a unit (slots)
  uint64_t wait_ns;    // bound of a collide tile's wait
};
constexpr uint64_t kWaitNs = 2000000000ull;

// A range of tiles, and a second one.
struct TileRange {
  uint32_t lo, n, lo2, n2;
};
// First tile that starts at cell c or after it.
LBNR_HD uint32_t tile_from(uint32_t c) { return (c + 31u) >> 5; }
LBNR_HD uint32_t plane_of(const Schedule& s, uint32_t v) { return v * s.pq + (v < s.pr ? v : s.pr); }
LBNR_HD uint32_t row_of(const Schedule& s, uint32_t t) { return t * s.rq + (t < s.rr ? t : s.rr); }

// Tiles of the collide pass of unit v of a strip.
LBNR_HD TileRange collide_tiles(const Schedule& s, uint32_t strip, uint32_t v) {
  const uint32_t base = plane_of(s, v) * s.plane;
  uint32_t lo, hi;
  if (s.strips == 1) {
    lo = tile_from(base);
    hi = tile_from(plane_of(s, v + 1) * s.plane);
  } else {
    lo = tile_from(base + row_of(s, strip) * s.row);
    hi = tile_from(base + row_of(s, strip + 1) * s.row);
  }
  return TileRange{lo, hi - lo, 0, 0};
}

// Tiles of the moment pass of unit v of a strip. With strips every boundary
// lies a row and a tile further on, so that the last row of a strip finds its
// upper neighbours done; the last row and tile of the plane go with the first
// strip, whose lower neighbours they are.
LBNR_HD TileRange moment_tiles(const Schedule& s, uint32_t strip, uint32_t v) {
  if (s.strips == 1) return collide_tiles(s, 0, v);
  const uint32_t base = plane_of(s, v) * s.plane, sh = s.row + 32u;
  const uint32_t last = base + s.plane - sh;
  TileRange r;
  r.lo = tile_from(strip == 0 ? base : base + row_of(s, strip) * s.row + sh);
  r.n = tile_from(strip + 1 == s.strips ? last : base + row_of(s, strip + 1) * s.row + sh) - r.lo;
  r.lo2 = r.n2 = 0;
  if (strip == 0) {
    r.lo2 = tile_from(last);
    r.n2 = tile_from(base + s.plane) - r.lo2;
  }
  return r;
}

// One item of the list: a tile of the moment pass at list position `pos` and
// the tile of the same slot of the collide pass `lead` positions behind it.
// Positions from `units` on have no moment tile, the first `lead` no collide
// tile, and a unit's last slots may be empty.
struct Item {
  uint32_t pos, slot;
};
LBNR_HD Item item_at(const Schedule& s, uint32_t i) {
  const uint32_t p = s.fslots.div(i);
  return Item{p, i - p * s.slots};
}
// The moment pass goes through a strip's units from its last `wrap` on.
LBNR_HD bool moment_tile(const Schedule& s, const Item& t, uint32_t& tile) {
  if (t.pos >= s.units) return false;
  const uint32_t strip = s.fupu.div(t.pos), w = t.pos - strip * s.upu;
  const TileRange r = moment_tiles(s, strip, w >= s.wrap ? w - s.wrap : w + s.upu - s.wrap);
  tile = t.slot < r.n ? r.lo + t.slot : r.lo2 + (t.slot - r.n);
  return t.slot < r.n + r.n2;
}
// need: the last position of the moment pass that the collide tile waits for
// (with every one before it).
LBNR_HD bool collide_tile(const Schedule& s, const Item& t, uint32_t& tile, uint32_t& need) {
  if (t.pos < s.lead) return false;
  const uint32_t p = t.pos - s.lead, strip = s.fupu.div(p), v = p - strip * s.upu;
  const TileRange r = collide_tiles(s, strip, v);
  tile = r.lo + t.slot;
  need = strip * s.upu + (v + s.ahead < s.upu ? v + s.ahead : s.upu - 1u);
  return t.slot < r.n;
}

// Cells of a unit. The two passes are about four units apart: shorter, and
// collide items wait for moment items still under way; longer, and the words
// leave the L2 in between. 256^3 D3Q19 FP32, us a step: 7015 at 2048 cells, 6885
// at 4096, 6900 at 8192, 7340 at 16384 (one unit further apart 7036, 6954, 7115,
// 7515); two launches 7690.
constexpr uint32_t kUnitCells = 4096;

// vset: the set's dimension.
inline Schedule make_schedule(uint32_t nx, uint32_t ny, uint32_t nz, int vset,
                              uint32_t unit_cells = kUnitCells) {
  Schedule s = {};
  const uint32_t planes = vset == 3 ? nz : vset == 2 ? ny : nx;
  s.plane = vset == 3 ? nx * ny : vset == 2 ? nx : 1u;
  s.row = vset == 3 ? nx : s.plane;
  s.strips = 1;
  if (vset == 3 && s.plane > unit_cells) {
    // strips of at least four rows, and long enough for the shifted bounds
    const uint32_t want = (s.plane + unit_cells - 1) / unit_cells;
    const uint32_t rows = (4u * s.row + 128u + s.row - 1) / s.row;
    const uint32_t most = ny / rows;
    s.strips = want < most ? want : (most > 1 ? most : 1u);
  }
  uint32_t per = 1;  // planes per unit
  if (s.strips == 1) per = (unit_cells + s.plane - 1) / s.plane;
  s.upu = planes / per > 1 ? planes / per : 1u;
  s.pq = planes / s.upu;
  s.pr = planes % s.upu;
  s.rq = ny / s.strips;
  s.rr = ny % s.strips;
  s.units = s.strips * s.upu;
  // a neighbour across the slowest axis is one plane away; where a unit is a
  // single plane that does not end on a tile, rounding reaches one more
  const bool exact = s.plane % 32u == 0 || (uint64_t)(s.pq - 1) * s.plane >= 32u;
  s.wrap = exact ? 1u : 2u;
  s.ahead = 2u * s.wrap;
  if (s.upu <= s.ahead + 1u) {
    s.wrap = 0;
    s.ahead = s.upu;
  }
  s.lead = s.ahead + 1u;
  if (s.lead > s.units) s.lead = s.units;
  uint64_t cells = (uint64_t)(s.pq + (s.pr ? 1 : 0)) * s.plane;
  if (s.strips > 1) cells = (uint64_t)(s.rq + (s.rr ? 1 : 0)) * s.row + 2u * (s.row + 32u);
  s.slots = (uint32_t)(cells / 32u) + 3u;
  s.fslots = make_fastdiv(s.slots);
  s.fupu = make_fastdiv(s.upu);
  s.items = s.slots * (s.units + s.lead);
  s.quota = s.slots;
  s.wait_ns = kWaitNs;
  return s;
}

}  // namespace lbnr
