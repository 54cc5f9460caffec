// Symbolic phase (paper Sec. II, "symbolic factorization"; Fig. 1): the
// sparsity pattern of A depends only on the grid, never on eps or omega, so
// the elimination order, the elimination tree, the front structure and every
// index map are computed once on the host and reused for all wavelengths and
// all design iterations.
//
// Ordering: geometric nested dissection of the nx x ny grid.  A rectangle is
// split by a full grid line (the separator) into two rectangles.  Rectangles
// that straddle the edge of the design box are split on the line just outside
// the box, so that every leaf subtree lies wholly inside or wholly outside the
// design box; this is what lets a design update refactor only the fronts on the
// paths from design pixels to the root.
#pragma once
#include <cstdint>
#include <string>
#include <vector>

namespace fdfd {

// Direction codes of one stencil entry A[row][col]: col = row + offset.
enum StencilDir { DIR_DIAG = 0, DIR_XM = 1, DIR_XP = 2, DIR_YM = 3, DIR_YP = 4 };

struct FrontDesc {           // plain-old-data, uploaded to the device as is
  int k;                     // pivots (fully summed variables) of this front
  int m;                     // boundary variables (eliminated in ancestors)
  int n;                     // k + m
  int ld;                    // row stride of the dense front (elements)
  long long st_off;          // element offset of the dense front in front storage
  long long v_off;           // element offset of the front vector (n entries) per RHS
  int idx_off;               // offset into idx: n grid cells (k pivots, then m boundary)
  int inv_off;               // offset into inv: n_parent entries (parent local -> my boundary t, or -1)
  int orig_off;              // offset into orig_ptr: n + 1 row pointers into orig entries
  int piv_off;               // offset into perm: k entries
  int parent;                // -1 for a root
  int child0;                // offset into children
  int nchild;
  int level;                 // 0 for leaves; parent level > child level
  int design;                // 1 if the subtree holds a design pixel (refactored on design change)
  int ldk;                   // row stride of the k x k inverse block (k rounded up to 4)
  long long iv_off;          // element offset of the inverse block (L11^-1 strictly lower, U11^-1 upper)
  long long pk_off;          // element offset of the packed block in each half (n <= kPackMaxN), see below
};

// Small fronts (n <= kPackMaxN) keep what the sweeps read in a packed store of two equal halves,
// one for the L side and one for the U side, a block of pack_block(m, k) entries per front in
// each, in sweep order, so that the blocks of neighbouring fronts are one contiguous copy:
//   - the triangle by diagonals, pack_diag(t, k) + i the entry at distance t:
//       L side: L11^-1[i + t][i] (t = 0: 1 / d in the symmetric form, unused in LU),
//       U side: U11^-1[i][i + t];
//   - L21, or U12 transposed: m rows of pack_stride(k) entries;
//   - L side: the pivot permutation (k ints).
// Diagonals and the odd row stride let the lanes of a warp walk rows or columns of a
// shared-memory copy without bank conflicts.
// Fronts of up to kTrimMaxN unknowns store nothing but their update matrix in the front store:
// row stride ld = m rounded up to 4, st_off set back so that entry (i, j) of the front, both
// >= k, is at st_off + i * ld + j as for the other fronts.
constexpr int kPackMaxN = 96;
constexpr int kTrimMaxN = 64;
#ifdef __CUDACC__
#define FDFD_HD __host__ __device__
#else
#define FDFD_HD
#endif
FDFD_HD inline int pack_stride(int k) { return k | 1; }
FDFD_HD inline int pack_diag(int t, int k) { return t * k - t * (t - 1) / 2; }
FDFD_HD inline int pack_rect(int k) { return k * (k + 1) / 2; }                       // where the rows start
FDFD_HD inline int pack_perm(int m, int k) { return pack_rect(k) + m * (k | 1); }     // where the permutation is
FDFD_HD inline int pack_block(int m, int k) { return (pack_perm(m, k) + (k + 1) / 2 + 1) / 2 * 2; }

struct Plan {
  int nx = 0, ny = 0;
  int bx0 = 0, by0 = 0, bw = 0, bh = 0;
  int leaf_area = 0;
  std::vector<FrontDesc> fronts;      // postorder: children precede parents
  std::vector<int> children;
  std::vector<int> idx;               // grid cells of each front
  std::vector<int> inv;               // extend-add inverse maps
  std::vector<int> orig_ptr;          // per front: n+1 offsets (absolute) into orig_entries
  std::vector<int> orig_col;          // local column of each original entry (n <= kPackMaxN: | local row << 16)
  std::vector<int> orig_code;         // cell * 5 + direction of each original entry (| kInterior, flag_interior)
  std::vector<int> pos;               // elimination position of each grid cell
  int n_levels = 0;
  std::vector<std::vector<int>> level_fronts;  // front ids per level
  long long store_total = 0;          // elements of front storage per omega
  std::vector<int> sweep_order;       // fronts by level, within a level n <= kTrimMaxN, n <= kPackMaxN, the others
  long long pack_total = 0;           // elements of one half of the packed store per omega
  long long inv_total = 0;            // elements of the triangular-inverse storage per omega
  long long vec_total = 0;            // elements of front vectors per RHS per omega
  int perm_total = 0;
  double flops_factor = 0;            // complex LU flops (8 real flops per complex FMA)
  double flops_design = 0;            // same, restricted to design-affected fronts
  long long factor_entries = 0;       // stored L and U entries (k*k + 2*k*m per front)
  int max_front = 0;
};

// Builds the plan.  Returns an empty string on success, otherwise an error message.
std::string build_plan(int nx, int ny, int bx0, int by0, int bw, int bh, int leaf_area, Plan* out);

// Marks the original entries of rows between the absorbing layers (px, py cells on each side), whose
// couplings are all -1, with kInterior: their values take no table.
constexpr int kInterior = (int)0x80000000u;
void flag_interior(Plan* p, int px, int py);

// Checks the plan's invariants (every original entry assembled once, injective
// extend-add maps, boundary eliminated after pivots).  Empty string when valid.
std::string validate_plan(const Plan& p);

}  // namespace fdfd
