// Panel steps of the large fronts' LU with pivoting inside each 32 x 32 diagonal block (paper Sec. II,
// the numeric factorisation), left-looking: no trailing updates.
//
// Step J (columns [j0, j0 + nb)), on a level whose row and column tiles fill the chip at most once, is
// one launch.  It finds its panel (the columns J of the rows from j0 on, and the rows J) updated by
// every pivot before the step before, p0 = j0 - 32, and applies those 32 itself:
//   D   the diagonal block B = F[J, J] - L[J, P] U[P, J], its LU with row pivoting inside the block,
//       perm, the block's triangular inverses (into the inverse store), growth;
//   L   rows r >= j0 + nb, 64 per CTA:  L[r, J] U_JJ = F[r, J] - L[r, P] U[P, J];
//   U   columns c >= j0 + nb:           L_JJ U[J, c] = P (F[J, c] - L[J, P] U[P, c]);
// L and U CTAs factor B too (the same bits), and beside them, for the next step's panel
// N = [j1, j1 + nb1), runs the update by all earlier pivots:
//   XL  rows r >= j1:          F[r, N] -= sum_{l < j0} L[r, l] U[l, N];
//   XU  columns c >= j1 + nb1: F[N, c] -= sum_{l < j0} L[N, l] U[l, c].
// X reads only what earlier steps finished and writes only the next panel, so the roles need no order.
// On other levels, and in complex128, the same parts are three launches: the panel's update by all
// pivots before it, the block's LU once per front, then its inverses, L and U.
// Rows of L left of the panel stay where they were (U's permutation is applied to U alone):
// lu_inv_fold_kernel reads them through perm, nothing else does.
//
// Why: the chain of steps bounds the levels with few fronts.  Right-looking, a step took two launches
// (32 us for the block LU and the substitutions, 17 us for a rank-32 update that reads and writes every
// remaining pivot row and column, at 21 TFLOP/s because two thirds of its traffic was that).
// Left-looking, an entry is updated once by a long contraction and once by 32 pivots.  What bounds the
// one-launch step now is the chain load - LU - substitution (2 800 + 11 000 + 5 000 cycles); the split
// steps issue 50 to 60% of the cycles.  All steps of one factorisation, before and now:
// 340 x 340, one wavelength 1.55 -> 0.82 ms; 540 x 540, 8: 6.4 -> 4.8 ms; 1760 x 1760, 2: 30.1 -> 24.2 ms;
// 200 x 200 in complex128: 7.7 -> 3.3 ms.
#include <algorithm>

#include "kernels.h"

namespace fdfd {

namespace {

constexpr int kNb = 32;        // pivots per step
constexpr int kKc = 16;        // contraction slice of the X products
constexpr int kPanelThreads = 256;

// Tile sizes.  complex64: 64 rows or columns a CTA, eight a warp; complex128, whose arithmetic bounds a CTA
// (two multiply-adds a clock and SM): eight, one a warp, so that a front's work spreads over the SMs.
template <typename T> struct Shape;
template <> struct Shape<float2> {
  static constexpr int kTile = 64;                  // rows (L) or columns (U) per CTA
  static constexpr int kXt = 64, kXp = kNb;         // product tiles: kXt along the panel, kXp across it
  static constexpr int kM = 4;                      // outputs per thread: kM x kM
};
template <> struct Shape<double2> {
  static constexpr int kTile = 8;
  static constexpr int kXt = 16, kXp = 16;
  static constexpr int kM = 1;
};

// LU of the nb x nb block in LU with row pivoting inside it, by warps 0-3 (lane = row, warp w the
// columns 8w .. 8w + 7 in registers); in place, rows in pivot order on return (after the caller's
// barrier).  No rows are swapped: pivot p is the unused lane with the largest |a_p| (one redux over
// keys: |a_p|^2 with its 5 low bits replaced by 31 - lane; ties to the lower lane, NaN wins).  Warp q
// factors its eight columns by itself, without barriers; then the warps right of it apply the eight
// updates.  The chain of one pivot to the next bounds it: the next column is updated and searched
// first, the others under that search's latency, and what else is known of a pivot leaves the loop.
// complex64: the loop over pivots stays rolled, the columns moving down one register per pivot: code
// that runs once is bound by instruction fetch.  complex128: unrolled, without the updates of columns
// already done.
// src[p]: the row that became row p, pos its inverse; dinv[p] = 1 / U[p][p].
template <typename T>
__device__ __forceinline__ void block_lu(T (*LU)[kNb + 1], int nb, int* src, int* pos, T* dinv) {
  using R = typename RealOf<T>::type;
  constexpr bool kRolled = sizeof(T) == 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T a[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int j = 8 * warp + c;
    a[c] = (lane < nb && j < nb) ? LU[lane][j] : (lane == j ? cmk(R(1), R(0)) : czero<T>());
  }
  if (warp == 0 && lane >= nb) {
    src[lane] = lane;
    pos[lane] = lane;
    dinv[lane] = cmk(R(1), R(0));
  }
  bool used = lane >= nb;
  // the pivot search of column ap and this lane's 1 / a
  auto search = [&](const T& ap, T& mine) -> unsigned {
    const unsigned v = __float_as_uint((float)cabs2(ap));
    const unsigned best = __reduce_max_sync(0xffffffffu, used ? 0u : ((v & ~31u) | (unsigned)(31 - lane)));
    mine = pivot_rcp(ap);
    return best;
  };
#pragma unroll 1
  for (int q = 0; q < 4; ++q) {
    if (8 * q >= nb) break;       // (uniform)
    const int np = min(8, nb - 8 * q);
    if (warp == q) {
      T mine, my = czero<T>();
      int myp = -1;
      unsigned best = search(a[0], mine);
      if constexpr (kRolled) {
#pragma unroll 1
        for (int c = 0; c < np; ++c) {
          const int r = 31 - (int)(best & 31u);
          const T inv = shfl_c(mine, r), ap = a[0];
          T l = cmul(ap, inv);
          if (lane == r) {
            myp = 8 * q + c;
            my = mine;
            used = true;
          }
          LU[lane][8 * q + c] = used ? ap : l;
          if (used) l = czero<T>();
          a[0] = cfms(l, shfl_c(a[1], r), a[1]);
          best = search(a[0], mine);
#pragma unroll
          for (int cc = 2; cc < 8; ++cc) a[cc - 1] = cfms(l, shfl_c(a[cc], r), a[cc]);
        }
      } else {
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (c < np) {
            const int r = 31 - (int)(best & 31u);
            const T inv = shfl_c(mine, r), ap = a[c];
            T l = cmul(ap, inv);
            if (lane == r) {
              myp = 8 * q + c;
              my = mine;
              used = true;
            }
            LU[lane][8 * q + c] = used ? ap : l;
            if (used) l = czero<T>();
#pragma unroll
            for (int cc = c + 1; cc < 8; ++cc) a[cc] = cfms(l, shfl_c(a[cc], r), a[cc]);
            if (c < 7) best = search(a[c + 1], mine);
          }
      }
      if (myp >= 0) {
        src[myp] = lane;
        pos[lane] = myp;
        dinv[myp] = my;
      }
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (warp > q) {
      T l[8];
      int r[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        r[c] = c < np ? src[8 * q + c] : lane;
        l[c] = c < np ? LU[lane][8 * q + c] : czero<T>();
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        used |= c < np && lane == r[c];
        if (used) l[c] = czero<T>();
#pragma unroll
        for (int cc = 0; cc < 8; ++cc) a[cc] = cfms(l[c], shfl_c(a[cc], r[c]), a[cc]);
      }
    }
  }
  // rows into pivot order: each warp its own columns
  const int to = pos[lane];
  T v[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) v[c] = LU[lane][8 * warp + c];
  __syncwarp();
#pragma unroll
  for (int c = 0; c < 8; ++c) LU[to][8 * warp + c] = v[c];
}

// C -= A B, C = F[r0 .. r0 + MR, c0 .. c0 + MC), A = F[rows, 0 .. K), B = F[0 .. K, columns), limited to rows < rlim
// and columns < clim; M x M outputs a thread.  Where the tile takes fewer threads than the CTA has,
// groups of threads share each slice of kKc pivots and their sums are added at the end: a CTA's latency
// stays that of all its warps, and four operand loads feed 64 multiply-adds.  The next slice's loads
// are in flight while one is multiplied.
template <typename T, int MR, int MC, int M>
__device__ __forceinline__ void panel_product(T* __restrict__ F, int ld, int r0, int rlim, int c0, int clim, int K,
                                              unsigned char* smem) {
  constexpr int TX = MC / M, NG = TX * (MR / M), G = kPanelThreads / NG;
  static_assert(G == 1 || G == 2, "one or two groups");
  constexpr int SA = MR + 2;                         // (even: two neighbouring rows in one load)
  T* As[2];
  T* Bs[2];
  As[0] = reinterpret_cast<T*>(smem);
  As[1] = As[0] + SA * kKc;
  Bs[0] = As[1] + SA * kKc;
  Bs[1] = Bs[0] + kKc * MC;
  const int tid = threadIdx.x, grp = tid / NG, t = tid % NG, tx = t % TX, ty = t / TX;
  constexpr int LA = MR * kKc / kPanelThreads, LB = MC * kKc / kPanelThreads;
  T ra[LA], rb[LB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < LA; ++q) {
      const int e = tid + q * kPanelThreads, i = e / kKc, l = k0 + e % kKc;
      ra[q] = (r0 + i < rlim && l < K) ? F[(size_t)(r0 + i) * ld + l] : czero<T>();
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) {
      const int e = tid + q * kPanelThreads, c = e % MC, l = k0 + e / MC;
      rb[q] = (c0 + c < clim && l < K) ? F[(size_t)l * ld + c0 + c] : czero<T>();
    }
  };
  auto stash = [&](int b) {
#pragma unroll
    for (int q = 0; q < LA; ++q) {
      const int e = tid + q * kPanelThreads;
      As[b][(e % kKc) * SA + e / kKc] = ra[q];
    }
#pragma unroll
    for (int q = 0; q < LB; ++q) Bs[b][tid + q * kPanelThreads] = rb[q];
  };
  T acc[M][M];
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int q = 0; q < M; ++q) acc[i][q] = czero<T>();
  fetch(0);
  stash(0);
  __syncthreads();
  for (int k0 = 0, b = 0; k0 < K; k0 += kKc, b ^= 1) {
    if (k0 + kKc < K) fetch(k0 + kKc);
    const T* Ab = As[b] + grp * (kKc / G) * SA + M * ty;
    const T* Bb = Bs[b] + grp * (kKc / G) * MC + M * tx;
#pragma unroll
    for (int kk = 0; kk < kKc / G; ++kk) {
      T av[M], bv[M];
      if constexpr (M % 2 == 0 && sizeof(T) == 8) {
#pragma unroll
        for (int i = 0; i < M; i += 2) {
          const float4 u = *reinterpret_cast<const float4*>(Ab + kk * SA + i);
          const float4 v = *reinterpret_cast<const float4*>(Bb + kk * MC + i);
          av[i] = make_float2(u.x, u.y);
          av[i + 1] = make_float2(u.z, u.w);
          bv[i] = make_float2(v.x, v.y);
          bv[i + 1] = make_float2(v.z, v.w);
        }
      } else {
#pragma unroll
        for (int i = 0; i < M; ++i) {
          av[i] = Ab[kk * SA + i];
          bv[i] = Bb[kk * MC + i];
        }
      }
#pragma unroll
      for (int i = 0; i < M; ++i)
#pragma unroll
        for (int q = 0; q < M; ++q) acc[i][q] = cfma(av[i], bv[q], acc[i][q]);
    }
    if (k0 + kKc < K) stash(b ^ 1);
    __syncthreads();
  }
  T cv[M / G][M];
  const int rw = r0 + M * ty + grp * (M / 2);        // this group's rows of the thread's
#pragma unroll
  for (int i = 0; i < M / G; ++i)
#pragma unroll
    for (int q = 0; q < M; ++q)
      cv[i][q] = (rw + i < rlim && c0 + M * tx + q < clim) ? F[(size_t)(rw + i) * ld + c0 + M * tx + q] : czero<T>();
  // each group finishes its half of the thread's rows: the other half through shared memory
  if constexpr (G == 2) {
    T* ex = reinterpret_cast<T*>(smem);
    static_assert(M * M / 2 * kPanelThreads <= 2 * kKc * (SA + MC), "the exchange fits the slices");
#pragma unroll
    for (int i = 0; i < M / 2; ++i)
#pragma unroll
      for (int q = 0; q < M; ++q) ex[(i * M + q) * kPanelThreads + tid] = grp ? acc[i][q] : acc[i + M / 2][q];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < M / 2; ++i)
#pragma unroll
      for (int q = 0; q < M; ++q) {
        const T o = ex[(i * M + q) * kPanelThreads + (tid ^ NG)];
        acc[i][q] = cadd(grp ? acc[i + M / 2][q] : acc[i][q], o);
      }
  }
#pragma unroll
  for (int i = 0; i < M / G; ++i)
#pragma unroll
    for (int q = 0; q < M; ++q)
      if (rw + i < rlim && c0 + M * tx + q < clim) F[(size_t)(rw + i) * ld + c0 + M * tx + q] = csub(cv[i][q], acc[i][q]);
}

// The update of panel [c0, c0 + nbp) by the pivots before K: its columns (rows c0 .. n, XL) or its rows
// (columns c0 + nbp .. n, XU), product tile t.
template <typename T>
__device__ __forceinline__ void panel_update(T* F, int ld, int n, int c0, int nbp, int K, bool cols, int t,
                                             unsigned char* smem) {
  using S = Shape<T>;
  constexpr int kParts = kNb / S::kXp;
  const int across = c0 + t % kParts * S::kXp, lim = c0 + nbp;
  const int along = c0 + (cols ? 0 : nbp) + t / kParts * S::kXt;
  if (along >= n || across >= lim) return;
  if (cols) panel_product<T, S::kXt, S::kXp, S::kM>(F, ld, along, n, across, lim, K, smem);
  else panel_product<T, S::kXp, S::kXt, S::kM>(F, ld, across, lim, along, n, K, smem);
}

// Threads and tile of a phase.  complex64, phase 2: a thread per row of 128, all of them in the substitution.
template <typename T, int PHASE> struct Cfg {
  static constexpr bool kC64 = sizeof(T) == 8;
  static constexpr int kThreads = PHASE == 1 || (PHASE == 2 && kC64) ? 128 : kPanelThreads;
  static constexpr int kTile = PHASE == 2 && kC64 ? 128 : Shape<T>::kTile;
  static constexpr int kCtas = PHASE == 0 || !kC64 ? 2 : PHASE == 3 ? 3 : 5;   // per SM, as shared memory allows
  // shared memory, elements of T.  Phase 0, 1: the block; L[J, P] and U[P, J], later the coefficients of the
  // substitutions; 1 / U_pp; the tile; its own operand, later its results.  Phase 2: the coefficients, the tile.
  static constexpr int kCf = kNb * (kNb + 2);
  static constexpr int kOffA = PHASE == 2 ? 0 : kNb * (kNb + 1), kOffB = kOffA + kCf;
  // (phase 2, role 0: both kinds of coefficients and up to 64 rows)
  static constexpr int kTile0 = 2 * kCf + (kTile < 2 * kNb ? kTile : 2 * kNb) * (kNb + 1), kTile12 = kCf + kTile * (kNb + 1);
  static constexpr int kDinv = PHASE != 2 ? kOffB + kCf : kTile0 > kTile12 ? kTile0 : kTile12, kWs = kDinv + kNb;
  static constexpr int kOp = kWs + kTile * (kNb + 1);
  static constexpr size_t kX = 2 * (size_t)kKc * (Shape<T>::kXt + Shape<T>::kXp + 2) * sizeof(T);
  static constexpr size_t kY = (size_t)(PHASE == 2 ? kWs : PHASE == 1 ? kWs : kOp + kTile * (kNb + 2)) * sizeof(T);
  static constexpr size_t kSmem = PHASE == 3 ? kX : PHASE == 0 && kX > kY ? kX : kY;
};

// PHASE 0: the whole step, every L and U CTA factoring the diagonal block itself (its update by P, and the
// next panel's by all before).  1: the block's LU, posted with its perm.  2: its inverses, L and U.
// 3: the update of panel J by all pivots before it.
template <typename T, int PHASE>
__global__ void __launch_bounds__(Cfg<T, PHASE>::kThreads, Cfg<T, PHASE>::kCtas)
panel_kernel(FactorLaunch a, const int* __restrict__ flist, int j0, int nt, int nx) {
  using R = typename RealOf<T>::type;
  using C = Cfg<T, PHASE>;
  constexpr int kTile = C::kTile, NT = C::kThreads, kRows = kTile * 32 / NT;   // rows a warp
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int src[kNb], pos[kNb];
  __shared__ R s_g[NT / 32];
  const int w = blockIdx.z + a.w0;
  const int f = flist[blockIdx.y];
  const FrontDesc d = a.P.fronts[f];
  const int k = d.k, ld = d.ld;
  if (j0 >= k) return;
  // L rows and U columns up to n; a front whose off-diagonal blocks come from the
  // tensor cores stops at its pivot block
  const int n = (a.pivonly && a.pivonly[f]) ? k : d.n;
  const int nb = min(kNb, k - j0), j1 = j0 + nb, p0 = j0 - kNb;
  T* F = reinterpret_cast<T*>(a.store) + (size_t)w * a.store_stride + d.st_off;
  const int bx = blockIdx.x;
  if constexpr (PHASE == 3) {
    panel_update<T>(F, ld, n, j0, nb, j0, bx < nx, bx % nx, smem_raw);
    return;
  } else {
  constexpr int kInvTiles = kTile >= 2 * kNb ? 1 : 2 * kNb / kTile;   // (role 0: 64 rows of inverses)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int role = 0, lo = bx * kTile;
  if (PHASE != 1 && bx >= kInvTiles) {
    const int t = bx - kInvTiles;
    if (PHASE == 0 && t >= 2 * nt) {
      if (j1 < k && j0 > 0)
        panel_update<T>(F, ld, n, j1, min(kNb, k - j1), j0, t - 2 * nt < nx, (t - 2 * nt) % nx, smem_raw);
      return;
    }
    role = 1 + t / nt;                               // 1 L, 2 U
    lo = j1 + t % nt * kTile;
    if (lo >= n) return;
  }
  T* sm = reinterpret_cast<T*>(smem_raw);
  T (*LU)[kNb + 1] = reinterpret_cast<T (*)[kNb + 1]>(sm);
  T (*Ljp)[kNb + 1] = reinterpret_cast<T (*)[kNb + 1]>(sm + C::kOffA);
  T (*Upj)[kNb + 2] = reinterpret_cast<T (*)[kNb + 2]>(sm + C::kOffB);
  T (*Cu)[kNb + 2] = reinterpret_cast<T (*)[kNb + 2]>(sm + C::kOffA);                   // U_jl at [j][l]
  T (*Cl)[kNb + 2] = reinterpret_cast<T (*)[kNb + 2]>(sm + (PHASE == 2 && role == 2 ? C::kOffA : C::kOffB));   // L_lj
  T* dinv = sm + C::kDinv;
  // row (L) or column (U) x J
  T (*Ws)[kNb + 1] = reinterpret_cast<T (*)[kNb + 1]>(sm + (PHASE != 2 ? C::kWs : role == 0 ? 2 * C::kCf : C::kCf));
  T* op = sm + C::kOp;                               // L: L[r, P] as [64][33]; U: U[P, c] as [32][66]
  T (*Wx)[kNb + 1] = PHASE == 2 ? Ws : reinterpret_cast<T (*)[kNb + 1]>(op);
  const size_t slot = (size_t)blockIdx.z * a.swp_stride + blockIdx.y;
  T* blk = reinterpret_cast<T*>(a.dblk) + slot * kDiagBlkElems;
  int* bsrc = a.swp + slot * kSwapScratchInts;       // src, pos
  const bool prev = PHASE == 0 && j0 > 0;
  // ---- operands into shared memory: many loads in flight before the first store ----
  constexpr int kB = kNb * kNb / NT, kW = kTile * kNb / NT, kChunk = kW < 8 ? kW : 8;
  {
    T vb[kB], vl[kB], vu[kB];
#pragma unroll
    for (int q = 0; q < kB; ++q) {
      const int e = tid + q * NT, i = e >> 5, j = e & 31;
      if (PHASE == 2) vb[q] = blk[e];
      else vb[q] = (i < nb && j < nb) ? F[(size_t)(j0 + i) * ld + j0 + j] : czero<T>();
      vl[q] = vu[q] = czero<T>();
      if (prev) {
        if (i < nb) vl[q] = F[(size_t)(j0 + i) * ld + p0 + j];
        if (j < nb) vu[q] = F[(size_t)(p0 + i) * ld + j0 + j];
      }
    }
    if (PHASE == 2 && tid < kNb) dinv[tid] = blk[kNb * kNb + tid];
    if (PHASE != 1 && role != 0) {
#pragma unroll 1
      for (int q0 = 0; q0 < kW; q0 += kChunk) {
        T vw[kChunk], vo[kChunk];
        int to[kChunk];
#pragma unroll
        for (int q = 0; q < kChunk; ++q) {
          vw[q] = vo[q] = czero<T>();
          if (role == 1) {
            constexpr int kStep = NT / 32;
            const int i = lo + warp + kStep * (q0 + q);
            const T* row = F + (size_t)(lo + warp) * ld + (size_t)(kStep * (q0 + q)) * ld + j0 + lane;
            if (i < n && lane < nb) vw[q] = row[0];
            if (prev && i < n) vo[q] = row[-kNb];
          } else {
            constexpr int kStep = NT / kTile;
            const int i = tid / kTile + kStep * (q0 + q), c = lo + tid % kTile;
            const T* row = F + (size_t)(j0 + tid / kTile) * ld + (size_t)(kStep * (q0 + q)) * ld + c;
            to[q] = PHASE == 2 ? bsrc[kNb + i] : i;
            if (c < n && i < nb) vw[q] = row[0];
            if (prev && c < n) vo[q] = row[-(ptrdiff_t)kNb * ld];
          }
        }
#pragma unroll
        for (int q = 0; q < kChunk; ++q) {
          const int e = tid + (q0 + q) * NT;
          if (role == 1) Ws[e >> 5][e & 31] = vw[q];
          else Ws[e % kTile][to[q]] = vw[q];
          if (prev) op[role == 1 ? (e >> 5) * (kNb + 1) + (e & 31) : e / kTile * (kTile + 2) + e % kTile] = vo[q];
        }
      }
    }
#pragma unroll
    for (int q = 0; q < kB; ++q) {
      const int e = tid + q * NT, i = e >> 5, j = e & 31;
      if (PHASE == 2) {
        if (role != 2) Cu[i][j] = vb[q];
        if (role != 1) Cl[j][i] = vb[q];
      } else {
        LU[i][j] = vb[q];
        if (prev) {
          Ljp[i][j] = vl[q];
          Upj[i][j] = vu[q];
        }
      }
    }
  }
  __syncthreads();
  R g = 0;
  if constexpr (PHASE == 0) {
    if (prev) {              // the block's update by P
      const int c = tid & 31, r = tid >> 5;
      T s[4] = {czero<T>(), czero<T>(), czero<T>(), czero<T>()};
#pragma unroll 4
      for (int l = 0; l < kNb; ++l) {
        const T u = Upj[l][c];
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] = cfma(Ljp[r + 8 * q][l], u, s[q]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) LU[r + 8 * q][c] = csub(LU[r + 8 * q][c], s[q]);
      __syncthreads();
    }
    if (warp >= 4 && prev && role != 0) {
      // the tile's update by P, beside the block's LU: 4 x 4 outputs a thread
      const int t = tid - 128, tx = role == 1 ? (t & 7) : (t & 15), ty = role == 1 ? t >> 3 : t >> 4;
      const T* ap = role == 1 ? op + 4 * ty * (kNb + 1) : &Ljp[4 * ty][0];
      const T* bp = role == 1 ? &Upj[0][4 * tx] : op + 4 * tx;
      const int sb = role == 1 ? kNb + 2 : kTile + 2;
      T acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][q] = czero<T>();
#pragma unroll 2
      for (int l = 0; l < kNb; ++l) {
        T av[4], bv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          av[i] = ap[i * (kNb + 1) + l];
          bv[i] = bp[l * sb + i];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[i][q] = cfma(av[i], bv[q], acc[i][q]);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          T& o = role == 1 ? Ws[4 * ty + i][4 * tx + q] : Ws[4 * tx + q][4 * ty + i];
          o = csub(o, acc[i][q]);
        }
    }
  }
  if (PHASE != 2) {
    if (warp < 4) block_lu<T>(LU, nb, src, pos, dinv);
    __syncthreads();
  }
  if (PHASE == 1) {
    for (int e = tid; e < kNb * kNb; e += NT) blk[e] = LU[e >> 5][e & 31];
    if (tid < kNb) {
      blk[kNb * kNb + tid] = dinv[tid];
      bsrc[tid] = src[tid];
      bsrc[kNb + tid] = pos[tid];
    }
  }
  if (PHASE != 2 && role == 0) {
    if (tid < nb) a.perm[(size_t)w * a.perm_stride + d.piv_off + j0 + tid] = j0 + src[tid];
#pragma unroll
    for (int q = 0; q < kB; ++q) {
      const int e = tid + q * NT, i = e >> 5, j = e & 31;
      if (i > j && i < nb) {
        const R a2 = cabs2(LU[i][j]);
        g = (a2 == a2) ? (a2 > g ? a2 : g) : R(INFINITY);
      }
    }
  }
  if constexpr (PHASE != 1) {
    if constexpr (PHASE == 0) {
      // coefficient (j, l) of the substitutions at [j][l]
#pragma unroll
      for (int q = 0; q < kB; ++q) {
        const int e = tid + q * NT, i = e >> 5, j = e & 31;
        const T v = LU[i][j];
        if (role != 2) Cu[i][j] = v;
        if (role != 1) Cl[j][i] = v;
      }
      __syncthreads();
    }
    // ---- substitutions: rows (L), columns (U) or, role 0, columns of L_JJ^-1 and rows of U_JJ^-1.
    // In rows, x_j = w_j / U_jj, then w_l -= x_j U_jl for l > j; in columns, w_l -= w_j L_lj.
    // complex64: a thread per row or column, eight entries in registers at a time, 4.6 instructions per
    // complex multiply-add (a lane per pivot: 6 200 cycles a tile in shuffles, and code unrolled over all
    // 32 entries is bound by its own fetch)
    const int nq = (nb + 7) >> 3;
    if constexpr (PHASE == 2 && sizeof(T) == 8) {
      // the earlier entries' products, then the 8 x 8 triangle
      if (role == 0 ? tid < 2 * kNb : lo + 32 * warp < n) {
        const bool rows = role == 1 || (role == 0 && tid >= kNb);
        T (*cf)[kNb + 2] = rows ? Cu : Cl;
        T* wr = Ws[tid];
#pragma unroll 1
        for (int q = 0; q < nq; ++q) {
          T x[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int l = 8 * q + i;
            if (role == 0) x[i] = cmk((tid & 31) == l ? R(1) : R(0), R(0));
            else x[i] = wr[l];
          }
#pragma unroll 2
          for (int j = 0; j < 8 * q; ++j) {
            const T xj = wr[j];
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
              const float4 c = *reinterpret_cast<const float4*>(&cf[j][8 * q + i]);
              x[i] = cfms(xj, make_float2(c.x, c.y), x[i]);
              x[i + 1] = cfms(xj, make_float2(c.z, c.w), x[i + 1]);
            }
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (rows) x[j] = cmul(x[j], dinv[8 * q + j]);
#pragma unroll
            for (int i = j + 1; i < 8; ++i) x[i] = cfms(x[j], cf[8 * q + j][8 * q + i], x[i]);
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) wr[8 * q + i] = x[i];
        }
      }
    } else if constexpr (PHASE == 0) {
      // the 8 x 8 triangle, then all warps' update of the later entries by the eight: the shorter chain
      const int row = tid & (kTile - 1), part = tid / kTile;
      const bool rows = role == 1 || (role == 0 && row >= kNb);
      T (*cf)[kNb + 2] = rows ? Cu : Cl;
      T* wr = Ws[row];
      if (role == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) wr[8 * part + i] = cmk((row & 31) == 8 * part + i ? R(1) : R(0), R(0));
        __syncthreads();
      }
#pragma unroll 1
      for (int q = 0; q < nq; ++q) {
        if (part == 0) {
          T x[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) x[i] = wr[role == 2 ? src[8 * q + i] : 8 * q + i];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (rows) x[j] = cmul(x[j], dinv[8 * q + j]);
#pragma unroll
            for (int i = j + 1; i < 8; ++i) x[i] = cfms(x[j], cf[8 * q + j][8 * q + i], x[i]);
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) Wx[row][8 * q + i] = x[i];
        }
        if (q + 1 == nq) break;
        __syncthreads();
        T x[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = Wx[row][8 * q + j];
#pragma unroll 1
        for (int c = 8 * (q + 1) + 2 * part; c < 8 * nq; c += 8) {
          T* w0 = wr + (role == 2 ? src[c] : c);
          T* w1 = wr + (role == 2 ? src[c + 1] : c + 1);
          T u = *w0, v = *w1;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float4 t = *reinterpret_cast<const float4*>(&cf[8 * q + j][c]);
            u = cfms(x[j], make_float2(t.x, t.y), u);
            v = cfms(x[j], make_float2(t.z, t.w), v);
          }
          *w0 = u;
          *w1 = v;
        }
        __syncthreads();
      }
    } else {
      // a warp per row or column, a lane per pivot: every lane of the few FP64 units busy
      const bool rows = role == 1 || (role == 0 && lo + warp >= kNb);
      T (*cf)[kNb + 2] = rows ? Cu : Cl;
      T x;
      if (role == 0) x = cmk(((lo + warp) & 31) == lane ? R(1) : R(0), R(0));
      else x = Ws[warp][lane];
#pragma unroll 4
      for (int j = 0; j < nb; ++j) {
        T xj = shfl_c(x, j);
        if (rows) xj = cmul(xj, dinv[j]);
        if (lane > j) x = cfms(xj, cf[j][lane], x);
        else if (lane == j) x = xj;
      }
      Wx[warp][lane] = x;
    }
    __syncthreads();
    // ---- the results: kRows rows or columns a warp ----
    const int r0 = warp * kRows;                     // in the tile
    T* X = reinterpret_cast<T*>(a.istore) + (size_t)w * a.istore_stride + d.iv_off;
    if (role == 0 && lo + r0 >= 2 * kNb) {
      // (no rows here)
    } else if (role == 1 || (role == 0 && lo + r0 >= kNb)) {
#pragma unroll 4
      for (int r = 0; r < kRows; ++r) {
        const int i = lo + r0 + r;
        const T v = Wx[r0 + r][lane];
        if (role == 1) {
          if (i < n && lane < nb) {
            F[(size_t)i * ld + j0 + lane] = v;
            const R a2 = cabs2(v);
            g = (a2 == a2) ? (a2 > g ? a2 : g) : R(INFINITY);
          }
        } else if (i - kNb < nb && lane >= i - kNb && lane < nb) {
          X[(size_t)(j0 + i - kNb) * d.ldk + j0 + lane] = v;       // U_JJ^-1: on and above the diagonal
        }
      }
    } else {
      // pieces of eight neighbouring columns: a warp's own, or (one column a warp) the tile's
#pragma unroll 4
      for (int q = 0; q < kRows; ++q) {
        const int cc = kRows >= 8 ? r0 + (lane & 7) + 8 * (q / 8) : tid & 7;
        const int i = kRows >= 8 ? (lane >> 3) + 4 * (q % 8) : tid >> 3;
        const int c = lo + cc;
        const T v = Wx[cc][i];
        if (role == 2) {
          if (c < n && i < nb) F[(size_t)(j0 + i) * ld + c] = v;
        } else if (i > c && i < nb) {
          X[(size_t)(j0 + i) * d.ldk + j0 + c] = v;                // L_JJ^-1: below it
        }
      }
    }
  }
  if (role == 2 || (PHASE == 2 && role == 0)) return;
  for (int o = 16; o > 0; o >>= 1) g = nanmax(g, __shfl_xor_sync(0xffffffffu, g, o));
  if (lane == 0) s_g[warp] = g;
  __syncthreads();
  if (tid == 0) {
    R gg = 0;
    for (int i = 0; i < NT / 32; ++i) gg = nanmax(gg, s_g[i]);
    float gv = (float)sqrt((double)gg);
    if (!(gv == gv)) gv = INFINITY;
    // max of non-negative floats is order independent as an int max
    atomicMax(reinterpret_cast<int*>(a.growth + (size_t)w * a.n_fronts + f), __float_as_int(gv));
  }
  }
}

// Update matrix of a complex128 front, S = F22 - L21 U12, in tiles of the panel's products: its arithmetic
// bounds a CTA, and 64 x 64 tiles left most SMs idle (480 us a launch at 200 x 200, one wavelength;
// all update matrices of that factorisation 2.57 -> 0.91 ms).
__global__ void __launch_bounds__(kPanelThreads) schur_fine_kernel(FactorLaunch a, const int* __restrict__ flist, int nt) {
  constexpr int kT = Shape<double2>::kXt;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int w = blockIdx.z + a.w0;
  const FrontDesc d = a.P.fronts[flist[blockIdx.y]];
  const int r0 = d.k + blockIdx.x / nt * kT, c0 = d.k + blockIdx.x % nt * kT;
  if (r0 >= d.n || c0 >= d.n) return;
  double2* F = reinterpret_cast<double2*>(a.store) + (size_t)w * a.store_stride + d.st_off;
  panel_product<double2, kT, kT, 1>(F, d.ld, r0, d.n, c0, d.n, d.k, smem_raw);
}

template <typename T, int PHASE>
cudaError_t panel_attribute() {
  return cudaFuncSetAttribute(panel_kernel<T, PHASE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)Cfg<T, PHASE>::kSmem);
}

}  // namespace

cudaError_t panel_init_attributes() {
  cudaError_t e = panel_attribute<float2, 0>();
  if (e == cudaSuccess) e = panel_attribute<float2, 1>();
  if (e == cudaSuccess) e = panel_attribute<float2, 2>();
  if (e == cudaSuccess) e = panel_attribute<float2, 3>();
  if (e == cudaSuccess) e = panel_attribute<double2, 1>();
  if (e == cudaSuccess) e = panel_attribute<double2, 2>();
  if (e == cudaSuccess) e = panel_attribute<double2, 3>();
  return e;
}

void launch_schur_fine(const FactorLaunch& a, const int* flist, int nf, int mmax, cudaStream_t s) {
  const int nt = (mmax + Shape<double2>::kXt - 1) / Shape<double2>::kXt;
  schur_fine_kernel<<<dim3(nt * nt, nf, a.n_omega), kPanelThreads, Cfg<double2, 3>::kSmem, s>>>(a, flist, nt);
}

template <typename T>
void launch_panel_step(const FactorLaunch& a, const int* flist, int nf, int j0, int nmax, cudaStream_t s) {
  using S = Shape<T>;
  if (nf <= 0 || nmax <= j0) return;
  auto ceil_div = [](int x, int y) { return (x + y - 1) / y; };
  constexpr int kParts = kNb / S::kXp;
  if constexpr (sizeof(T) == 8) {
    // CTAs resident at once on the current device
    int dev = 0, nsm = 0, per_sm = 0;
    const long long wave =
        (cudaGetDevice(&dev) == cudaSuccess &&
         cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
         cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, panel_kernel<T, 0>, Cfg<T, 0>::kThreads, Cfg<T, 0>::kSmem) ==
             cudaSuccess)
            ? (long long)std::max(1, per_sm) * nsm
            : (1LL << 40);
    // One launch while a level's L and U tiles fit the chip once (by the level's size alone: its steps are
    // all of one kind, as the look-ahead asks).  All steps of a factorisation with this rule / every level
    // split / every level in one launch: 340 x 340 0.82 / 1.49 / 0.83 ms, 540 x 540 with 8 wavelengths
    // 4.8 / 5.1 / 6.0 ms, 1760 x 1760 with 2 24.2 / 25.7 / 31.5 ms.
    if ((long long)(1 + 2 * ceil_div(nmax - 1, S::kTile)) * nf * a.n_omega <= wave) {
      const int nt = ceil_div(nmax - j0 - 1, S::kTile), nx = ceil_div(nmax - j0 - 1, S::kXt) * kParts;
      panel_kernel<T, 0><<<dim3(1 + 2 * nt + (j0 > 0 ? 2 * nx : 0), nf, a.n_omega), kPanelThreads, Cfg<T, 0>::kSmem, s>>>(
          a, flist, j0, std::max(1, nt), std::max(1, nx));
      return;
    }
  }
  if (j0 > 0) {
    const int nx = ceil_div(nmax - j0, S::kXt) * kParts;
    panel_kernel<T, 3><<<dim3(2 * nx, nf, a.n_omega), kPanelThreads, Cfg<T, 3>::kSmem, s>>>(a, flist, j0, 0, nx);
  }
  panel_kernel<T, 1><<<dim3(1, nf, a.n_omega), Cfg<T, 1>::kThreads, Cfg<T, 1>::kSmem, s>>>(a, flist, j0, 0, 0);
  constexpr int kTile2 = Cfg<T, 2>::kTile;
  const int nt2 = ceil_div(nmax - j0 - 1, kTile2);
  panel_kernel<T, 2><<<dim3(std::max(1, 2 * kNb / kTile2) + 2 * nt2, nf, a.n_omega), Cfg<T, 2>::kThreads, Cfg<T, 2>::kSmem,
                       s>>>(a, flist, j0, std::max(1, nt2), 0);
}
template void launch_panel_step<float2>(const FactorLaunch&, const int*, int, int, int, cudaStream_t);
template void launch_panel_step<double2>(const FactorLaunch&, const int*, int, int, int, cudaStream_t);

}  // namespace fdfd
