// Work units of the dataflow sweeps: shared by the host, which cuts the fronts into units that
// fit the shared memory of a CTA, and by the kernel, which stages them.
#pragma once
#include <cuda_runtime.h>

#include "plan.h"

namespace fdfd {

// What a sweep needs of a front, one 96-byte record.  The records lie in sweep order (plan.h); those
// of the packed fronts lie a second time in the index store, each followed by the front's n grid
// cells and n children's slots (16 bits per child, 0xffff = none), so that the index data of
// neighbouring fronts are one contiguous copy as well.
struct __align__(16) SweepFront {
  int k, m, ld, ldk;
  long long st_off, iv_off, pk_off, v_off;
  long long u0, u1;        // where its children's update vectors start in a system's front vectors
  int inv0, inv1;          // its children's extend-add maps, -1 without that child
  int dep0, dep1;          // its children, -1 without that child
  int parent, f;
  int idx_off, piv_off;
};
static_assert(sizeof(SweepFront) == 96, "the index store's layout");
inline int meta_bytes(int n) { return (96 + 8 * n + 15) / 16 * 16; }

// One unit of work of a sweep, 48 bytes.
enum UnitKind {
  kUnitSmall = 0,          // packed fronts, neighbours in sweep order, one per working warp
  kUnitPacked = 1,         // one packed front, whole CTA
  kUnitFront = 2,          // one other front, whole CTA
  kUnitTri = 3,            // rows (L, U) or columns (U^T, L^T) of a large front's inverse block
  kUnitRect = 4,           // ... of its off-diagonal block
  kUnitEnd = 5             // (inside the kernel) no more units
};
constexpr int kUnitLast = 1 << 16;     // (inside the kernel) the unit's last part: it is done once this is
struct __align__(16) SweepUnit {
  int rec;                 // packed kinds: offset of the index data / 16; others: record
  int kind;                // kind | fronts << 8
  int r0, cnt;             // tri, rect: first row / column and their number; packed kinds: bytes of index data, of factor data
  long long fac;           // packed kinds: element offset of the factor data in its half of the packed store
  int vslice;              // small: bytes of one warp's vectors; tri, rect: contraction length of one part
  int part;                // (inside the kernel) tri, rect: the part in the buffer
  unsigned short off[8];   // small: offset / 16 of each front's record in the index data
};
static_assert(sizeof(SweepUnit) == 48, "three 16-byte words");

// Lanes per row of a product of r rows by th threads.
FDFD_HD inline int row_lanes(int r, int th) {
  int g = 2;
  while (g < 32 && 2 * g * r <= th) g *= 2;
  return g;
}

// Shared-memory row stride (elements) of rows of len elements read by g lanes each: with
// stride = g (mod 2 g) the rows of one access fall into distinct banks.  Rows start on 16 bytes.
FDFD_HD inline int row_stride(int len, int g, int es) {
  if (es == 16) {
    if (g >= 8) return len | 1;
    while (len % (2 * g) != g) ++len;
    return len;
  }
  len = (len + 1) & ~1;
  if (g >= 16) return len;
  while (len % (2 * g) != g) len += 2;
  return len;
}

// A tri or rect unit works through its contraction (the columns its rows, or the rows its columns,
// reach) in parts of a fixed length that fit a buffer, staged one after the other.
struct UnitRange {
  int lo, hi;
};
// sweep 0 L, 1 U, 2 U^T, 3 L^T; rows (0, 1) or columns (2, 3) [r0, r0 + cnt)
FDFD_HD inline UnitRange unit_range(int sweep, bool rect, int k, int m, int r0, int cnt) {
  const bool up = sweep == 0 || sweep == 2;
  if (rect) return UnitRange{0, up ? k : m};
  return up ? UnitRange{0, r0 + cnt} : UnitRange{r0, k};
}

// A block staged row by row: rows [row0, row0 + rows) and columns [col0, col0 + cols) of the
// inverse block (tri) or of the front (rect), in shared memory at a row stride of `stride`
// elements; the first wanted column is `shift` elements in (rows start on 16 bytes).  An empty block
// (the off-diagonal block of a front without boundary rows) has no rows: nothing is copied.
struct StageGeom {
  int row0, rows, col0, cols, stride, shift;
};

// es: bytes per entry; the lines [r0, r0 + cnt) of a unit and the part [a, b) of its contraction;
// th: working threads of the CTA.
FDFD_HD inline StageGeom stage_geom(int es, int sweep, bool rect, int k, int ld, int ldk, int r0, int cnt, int a, int b,
                                    int th) {
  StageGeom s{};
  if (cnt <= 0 || b <= a) return s;
  const int odd = es == 8 ? 1 : 0;             // alignment of a row's start and length: 2 entries of 8 bytes
  const int lim = rect ? ld : ldk;             // entries a row holds, a multiple of 4
  int c0, c1;                                  // wanted columns [c0, c1)
  if (sweep < 2) {
    s.row0 = (rect && sweep == 0 ? k : 0) + r0;
    s.rows = cnt;
    c0 = (rect && sweep == 1 ? k : 0) + a;
    c1 = c0 + b - a;
  } else {
    s.row0 = (rect && sweep == 3 ? k : 0) + a;
    s.rows = b - a;
    c0 = (rect && sweep == 2 ? k : 0) + r0;
    c1 = c0 + cnt;
  }
  s.col0 = c0 & ~odd;
  s.shift = c0 - s.col0;
  int e = (c1 + odd) & ~odd;
  if (e > lim) e = lim;
  s.cols = e - s.col0;
  s.stride = sweep < 2 ? row_stride(s.cols, row_lanes(cnt, th), es) : s.cols;
  return s;
}
// entries of a tri / rect unit's vectors in front of its staged block (16-byte multiples)
template <int NR> FDFD_HD inline int unit_vec(int nvec, int nsub) { return ((nvec + nsub) * NR + 1) & ~1; }
inline long long stage_bytes(const StageGeom& s, int es) { return (long long)s.rows * s.stride * es; }

}  // namespace fdfd
