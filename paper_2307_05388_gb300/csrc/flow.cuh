// Triangular sweeps over the cached factors (paper Eq. 5 and Eq. 6; Sec. II,
// "back substitution").  Forward solve A x = b is L then U; the adjoint
// (transpose) solve A^T x = b reuses the same factors as U^T then L^T, so no
// second factorisation is needed (the first caching idea of Sec. II).
//
// Per front, with the factored front [L11\U11 U12; L21 S], its row permutation
// P and the triangular inverses X_L = L11^-1, X_U = U11^-1 stored at
// factorisation time:
//   L   : y = X_L (P v)_k,                 u = v_m - L21 y
//   U   : x_k = X_U (y - U12 x_m)
//   U^T : w = X_U^T v_k,                   u = v_m - U12^T w
//   L^T : x_k = P^T X_L^T (w - L21^T x_m)
// where v gathers the front's entries of the right-hand side (complex128, cast
// to the factor precision as it is gathered) plus the update
// vectors u of its children (through the same inverse extend-add maps as the
// factorisation) and x_m are the already final values of the boundary
// variables (the solution is stored in complex128 as it is produced).  Levels
// run bottom-up for L / U^T and top-down for U / L^T.
//
// With the inverses every step is a matrix-vector product.  One persistent
// launch per direction takes units of work in elimination-tree order (the
// dataflow sweep below): up to 8 small fronts, a warp each; one medium front by
// a CTA; rows or columns of a large front's inverse block (phase 1 bottom-up)
// or off-diagonal block (the other phase).
//
// What bounds a sweep is latency: 11 to 18 levels of the elimination tree, each
// a chain of dependent loads.  So everything of a unit that depends on no other
// front is in shared memory before the unit starts: a producer warp takes units
// from the queue one ahead of the eight that work and brings their factor
// blocks (and, for small fronts, their index data) in by bulk asynchronous
// copies into the other of two buffers (very large fronts leave room for one); the working warps only wait for the
// fronts they depend on and gather vector entries; and a third role publishes
// finished fronts, so that its fence delays nobody else.  Right-hand sides are
// taken two at a time from the staged copy, so each factor entry is read from
// memory once for all of a wavelength's right-hand sides.  Reductions run in a
// fixed order (deterministic).
//
// Measured per launch, before (fronts' factor rows loaded by the warps that use
// them, after the wait, one right-hand side after the other) and with this
// scheme: 1760 x 1760, two wavelengths x two sources: L 3.37 -> 2.03 ms, U 2.60
// -> 1.57, U^T 3.35 -> 2.16, L^T 2.82 -> 2.09 (a launch must read 3.4 GB of
// factors, 0.5 ms); 100 x 100: 83 -> 43, 65 -> 44, 77 -> 45, 66 -> 51 us.  The
// instructions of the small fronts' products and the gathers' latency bound it
// now.  Not kept: four CTAs of four working warps per SM (L 2.41 ms), three of
// eight (2.54 ms: 64 registers spill), units without a second buffer (2.6 ms).
#pragma once
#include "async.cuh"
#include "kernels.h"

namespace fdfd {

namespace {

// A CTA: TH working threads, the producer warp and the publishing warp.
// Limits of the waits, each longer than what it waits for may take: the producer's for a buffer (longer than
// every dependency wait), the publisher's for a finished unit, the working warps' for a staged one (the
// publisher ends that one first, staged_wait).
constexpr unsigned long long kFreeWaitNs = 6000000000ull;
constexpr unsigned long long kDoneWaitNs = 16000000000ull;
constexpr unsigned long long kStagedWaitNs = 32000000000ull;

// barrier of the working warps
template <int TH> __device__ __forceinline__ void work_sync() { asm volatile("bar.sync 1, %0;" ::"n"(TH) : "memory"); }

// mbar_wait with one answer for the whole warp: each lane's own limit may pass at another poll, and lanes
// that part here would meet different warp operations.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, unsigned long long limit_ns) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, limit_ns));
}

// Whether the CTA goes on: one word, written by the publisher alone.  The working warps share named barriers,
// so either all of them run a unit or none.  They do not time out on their own: when a unit is overdue the
// publisher asks, looks whether it is staged after all, and then says so once.  A warp that found the unit
// staged before the question is seen by that look; one that finds it staged later reads the question
// and waits for the answer.
enum StopWord { kGoOn = 0, kStopAsked = 1, kStopped = 2 };

// Working warps: the unit is staged and the CTA goes on.  (The limit alone ends it for a unit that no
// producer will stage any more; then every warp's does.)
__device__ __forceinline__ bool staged_wait(uint32_t bar, uint32_t parity, const volatile int* stop) {
  unsigned long long t0 = 0;
  for (uint32_t it = 0; it < (1u << 28); ++it) {
    const bool in = mbar_try(bar, parity);
    const int word = *stop;
    if (in && word == kGoOn) return true;
    if (word == kStopped) return false;
    if ((it & 63) == 63) {
      const unsigned long long now = gtimer();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kStagedWaitNs) return false;
    }
  }
  return false;
}

// The publisher (one lane): the unit behind `bar` is overdue.
__device__ __forceinline__ void stop_unless_staged(uint32_t bar, uint32_t parity, volatile int* stop) {
  *stop = kStopAsked;
  asm volatile("fence.sc.cta;" ::: "memory");
  *stop = mbar_try(bar, parity) ? kGoOn : kStopped;
}

// Vector entries written by other CTAs of the same launch (the dataflow sweep)
// are read through L2 only: the per-SM L1 is not coherent.
__device__ __forceinline__ float2 ldv(const float2* p) { return __ldcg(p); }
__device__ __forceinline__ double2 ldv(const double2* p) { return __ldcg(p); }

// The NR right-hand sides' values of one vector entry (adjacent in shared memory).
template <typename T, int NR> struct Vals { T v[NR]; };
template <typename T, int NR>
__device__ __forceinline__ Vals<T, NR> vget(const T* vec, int i) {
  Vals<T, NR> r;
  if constexpr (sizeof(T) == 8 && NR == 2) {
    const float4 q = *reinterpret_cast<const float4*>(vec + 2 * i);
    r.v[0] = make_float2(q.x, q.y);
    r.v[1] = make_float2(q.z, q.w);
  } else {
#pragma unroll
    for (int q = 0; q < NR; ++q) r.v[q] = vec[i * NR + q];
  }
  return r;
}
template <typename T, int NR>
__device__ __forceinline__ void vset(T* vec, int i, const Vals<T, NR>& x) {
  if constexpr (sizeof(T) == 8 && NR == 2) {
    *reinterpret_cast<float4*>(vec + 2 * i) = make_float4(x.v[0].x, x.v[0].y, x.v[1].x, x.v[1].y);
  } else {
#pragma unroll
    for (int q = 0; q < NR; ++q) vec[i * NR + q] = x.v[q];
  }
}
template <typename T, int NR> __device__ __forceinline__ Vals<T, NR> vzero() {
  Vals<T, NR> r;
#pragma unroll
  for (int q = 0; q < NR; ++q) r.v[q] = czero<T>();
  return r;
}
template <typename T, int NR>
__device__ __forceinline__ void vfma(T f, const Vals<T, NR>& x, Vals<T, NR>& acc) {
#pragma unroll
  for (int q = 0; q < NR; ++q) acc.v[q] = cfma(f, x.v[q], acc.v[q]);
}
template <typename T, int NR>
__device__ __forceinline__ Vals<T, NR> vadd(const Vals<T, NR>& a, const Vals<T, NR>& b) {
  Vals<T, NR> r;
#pragma unroll
  for (int q = 0; q < NR; ++q) r.v[q] = cadd(a.v[q], b.v[q]);
  return r;
}
template <typename T, int NR>
__device__ __forceinline__ Vals<T, NR> vsub(const Vals<T, NR>& a, const Vals<T, NR>& b) {
  Vals<T, NR> r;
#pragma unroll
  for (int q = 0; q < NR; ++q) r.v[q] = csub(a.v[q], b.v[q]);
  return r;
}
template <typename T, int NR>
__device__ __forceinline__ void vxor_add(Vals<T, NR>& a, int o) {
#pragma unroll
  for (int q = 0; q < NR; ++q) {
    a.v[q].x += __shfl_xor_sync(0xffffffffu, a.v[q].x, o);
    a.v[q].y += __shfl_xor_sync(0xffffffffu, a.v[q].y, o);
  }
}

// D[cell] of the symmetric form (stretch factors at the cell centre)
__device__ __forceinline__ double2 sym_d(const SolveLaunch& a, int w, int cell) {
  const int i = cell / a.P.ny, j = cell - i * a.P.ny;
  return cmul(a.sxc[(size_t)w * a.P.nx + i], a.syc[(size_t)w * a.P.ny + j]);
}

// The solution value written for cell: x, or D x for the transposed symmetric-form solve.
template <typename T>
__device__ __forceinline__ double2 out_val(const SolveLaunch& a, int w, int cell, T v) {
  const double2 x = cto64(v);
  return a.sym_out ? cmul(sym_d(a, w, cell), x) : x;
}

// x_m of a front below, read back from the output: D x was written there for the
// transposed symmetric-form solve
__device__ __forceinline__ double2 xm_val(const SolveLaunch& a, int w, int cell, double2 x) {
  if (!a.sym_out) return x;
  const double2 d = sym_d(a, w, cell);
  const double q = 1.0 / (d.x * d.x + d.y * d.y);
  return cmul(x, make_double2(d.x * q, -d.y * q));
}

// One chunk of NR right-hand sides of a wavelength (the last chunk of an odd count repeats
// its last one: the same values are computed and stored twice).
template <typename T, int NR> struct Chunk {
  T* vb[NR];
  const double2* rhs[NR];
  double2* xo[NR];
};
template <typename T, int NR>
__device__ __forceinline__ Chunk<T, NR> chunk_of(const SolveLaunch& a, int w, int rc, const double2* in, double2* out) {
  Chunk<T, NR> c;
#pragma unroll
  for (int q = 0; q < NR; ++q) {
    const int r = min(rc + q, a.r0 + a.nr - 1);
    const size_t sys = (size_t)w * a.nrhs + r;
    c.vb[q] = reinterpret_cast<T*>(a.vb) + sys * a.vec_stride;
    c.rhs[q] = in + sys * a.n;
    c.xo[q] = out + sys * a.n;
  }
  return c;
}

// Bottom-up gather of local slot src, in two halves: what no other front writes (map entries and
// right-hand side), then the children's update vectors.
template <typename T, int NR> struct Slot {
  int t0, t1;
  Vals<T, NR> b;
};
template <typename T, int NR>
__device__ __forceinline__ Slot<T, NR> slot_fetch(const SolveLaunch& a, const SweepFront& d, const Chunk<T, NR>& c,
                                                  int src, int w) {
  Slot<T, NR> s;
  s.t0 = d.inv0 >= 0 ? a.P.inv[d.inv0 + src] : -1;
  s.t1 = d.inv1 >= 0 ? a.P.inv[d.inv1 + src] : -1;
  s.b = vzero<T, NR>();
  if (src < d.k) {
    const int cell = a.P.idx[d.idx_off + src];
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      const double2 b = c.rhs[q][cell];
      s.b.v[q] = cfrom<T>(a.sym_in ? cmul(sym_d(a, w, cell), b) : b);
    }
  }
  return s;
}
// the same from a packed front's staged index data
template <typename T, int NR>
__device__ __forceinline__ Slot<T, NR> slot_staged(const SolveLaunch& a, int k, const int* cells, const unsigned* slots,
                                                   const Chunk<T, NR>& c, int src, int w) {
  Slot<T, NR> s;
  const unsigned t = slots[src];
  s.t0 = (t & 0xffffu) == 0xffffu ? -1 : (int)(t & 0xffffu);
  s.t1 = (t >> 16) == 0xffffu ? -1 : (int)(t >> 16);
  s.b = vzero<T, NR>();
  if (src < k) {
    const int cell = cells[src];
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      const double2 b = c.rhs[q][cell];
      s.b.v[q] = cfrom<T>(a.sym_in ? cmul(sym_d(a, w, cell), b) : b);
    }
  }
  return s;
}
// The slots of a thread, with every load issued before the first is used: N of them, those with on(p).
template <typename T, int NR, int N, typename On, typename Put>
__device__ __forceinline__ void slots_finish(const SweepFront& d, const Chunk<T, NR>& c, const Slot<T, NR> (&s)[N],
                                             On on, Put put) {
  Vals<T, NR> x0[N], x1[N];
#pragma unroll
  for (int p = 0; p < N; ++p) {
    const bool l0 = on(p) && s[p].t0 >= 0, l1 = on(p) && s[p].t1 >= 0;
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      x0[p].v[q] = czero<T>();
      x1[p].v[q] = czero<T>();
      if (l0) x0[p].v[q] = ldv(c.vb[q] + d.u0 + s[p].t0);
      if (l1) x1[p].v[q] = ldv(c.vb[q] + d.u1 + s[p].t1);
    }
  }
#pragma unroll
  for (int p = 0; p < N; ++p)
    if (on(p)) put(p, vadd(vadd(s[p].b, x0[p]), x1[p]));
}
template <typename T, int NR>
__device__ __forceinline__ Vals<T, NR> front_val(const SweepFront& d, const Chunk<T, NR>& c, int s) {
  Vals<T, NR> v;
#pragma unroll
  for (int q = 0; q < NR; ++q) v.v[q] = ldv(c.vb[q] + d.v_off + s);
  return v;
}
// y (U) or w = y / d (L^T of the symmetric form, 1 / d = *dinv) of pivot s
template <typename T, int SWEEP, int NR>
__device__ __forceinline__ Vals<T, NR> pivot_val(const SolveLaunch& a, const SweepFront& d, const Chunk<T, NR>& c,
                                                 const T* dinv, int s) {
  Vals<T, NR> v;
#pragma unroll
  for (int q = 0; q < NR; ++q) v.v[q] = ldv(c.vb[q] + d.v_off + s);
  if (SWEEP == 3 && a.sym_mid) {
    const T di = *dinv;
#pragma unroll
    for (int q = 0; q < NR; ++q) v.v[q] = cmul(v.v[q], di);
  }
  return v;
}
template <typename T, int SWEEP, int NR>
__device__ __forceinline__ Vals<T, NR> bound_val(const SolveLaunch& a, const Chunk<T, NR>& c, int cell, int w) {
  Vals<T, NR> v;
#pragma unroll
  for (int q = 0; q < NR; ++q) {
    const double2 x = ldv(c.xo[q] + cell);
    v.v[q] = cfrom<T>(SWEEP == 3 ? xm_val(a, w, cell, x) : x);
  }
  return v;
}
// a thread's boundary values (cells >= 0), loads first
template <typename T, int SWEEP, int NR, int N, typename Put>
__device__ __forceinline__ void bounds_put(const SolveLaunch& a, const Chunk<T, NR>& c, const int (&cell)[N], int w,
                                           Put put) {
  Vals<T, NR> x[N];
#pragma unroll
  for (int p = 0; p < N; ++p)
    if (cell[p] >= 0) x[p] = bound_val<T, SWEEP, NR>(a, c, cell[p], w);
#pragma unroll
  for (int p = 0; p < N; ++p)
    if (cell[p] >= 0) put(p, x[p]);
}
template <typename T, int SWEEP, int NR>
__device__ __forceinline__ void put_x(const SolveLaunch& a, const Chunk<T, NR>& c, int cell, int w,
                                      const Vals<T, NR>& v) {
#pragma unroll
  for (int q = 0; q < NR; ++q) c.xo[q][cell] = SWEEP == 3 ? out_val(a, w, cell, v.v[q]) : cto64(v.v[q]);
}
template <typename T, int NR>
__device__ __forceinline__ void put_v(const SweepFront& d, const Chunk<T, NR>& c, int s, const Vals<T, NR>& v) {
#pragma unroll
  for (int q = 0; q < NR; ++q) c.vb[q][d.v_off + s] = v.v[q];
}

// ---------------------------------------------------------------------------
// Products of a warp with a block in shared memory.  P = lanes over rows or columns (the power of
// two covering them, at most 32); the 32 / P lane groups split each sum and add up in a fixed
// butterfly.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int lanes_for(int n) { return n <= 4 ? 4 : n <= 8 ? 8 : n <= 16 ? 16 : 32; }


// The terms of one lane's sum: n entries from f on, step df apart (which itself changes by ddf per
// step: diagonals), with the vector entries from v on, dv apart.
template <typename T, int NR>
__device__ __forceinline__ Vals<T, NR> walk(const T* f, int df, int ddf, const T* v, int dv, int n) {
  Vals<T, NR> a0 = vzero<T, NR>(), a1 = vzero<T, NR>();
  for (; n >= 4; n -= 4) {
    T e[4];
    Vals<T, NR> x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      e[u] = *f;
      x[u] = vget<T, NR>(v, 0);
      f += df;
      df += ddf;
      v += dv;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) vfma(e[u], x[u], (u & 1) ? a1 : a0);
  }
  // the last terms, loads first
  T e[3];
  Vals<T, NR> x[3];
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    e[u] = czero<T>();
    x[u] = vzero<T, NR>();
    if (u < n) {
      e[u] = *f;
      x[u] = vget<T, NR>(v, 0);
    }
    f += df;
    df += ddf;
    v += dv;
  }
#pragma unroll
  for (int u = 0; u < 3; ++u) vfma(e[u], x[u], (u & 1) ? a1 : a0);
  return vadd(a0, a1);
}

// out(i, sum) over the lines i < n; one(i, g, G) gives the walk of lane group g of G
template <typename T, int NR, typename One, typename Out>
__device__ __forceinline__ void warp_lines(int n, One one, Out out) {
  const int lane = threadIdx.x & 31;
  const int P = lanes_for(n), lp = 31 - __clz(P), G = 32 >> lp;
  const int li = lane & (P - 1), g = lane >> lp;
  for (int i0 = 0; i0 < n; i0 += P) {
    const int i = i0 + li;
    Vals<T, NR> s = vzero<T, NR>();
    if (i < n) s = one(i, g, G);
    for (int o = P; o < 32; o <<= 1) vxor_add(s, o);
    if (g == 0 && i < n) out(i, s);
  }
}
// packed triangle, entries at distances t0, t0 + 1, .. from i: back (towards 0) or forward (towards k)
template <typename T, int NR, bool BACK>
__device__ __forceinline__ Vals<T, NR> tri_walk(const T* tri, int k, const T* vec, int t0, int i, int g, int G) {
  const int t = t0 + g, n = (BACK ? i + 1 : k - i) - t;
  // from distance t to t + G: pack_diag grows by G k - G t - G (G - 1) / 2, which falls by G^2 per step
  const int df = G * (k - t) - G * (G - 1) / 2 - (BACK ? G : 0);
  return walk<T, NR>(tri + pack_diag(t, k) + (BACK ? i - t : i), df, -G * G, vec + (BACK ? i - t : i + t) * NR,
                     BACK ? -G * NR : G * NR, n > 0 ? (n + G - 1) / G : 0);
}

// ---------------------------------------------------------------------------
// Products of a CTA with a block in shared or global memory.
// ---------------------------------------------------------------------------
// out(i, sum_{c in [lo(i), hi(i))} A[i][c] vec[c]) for rows i < nrows, G lanes per row
template <int TH, typename T, int NR, int UN, typename Lo, typename Hi, typename Out>
__device__ __forceinline__ void block_rows(const T* __restrict__ A, int stride, int nrows, int G, const T* vec, Lo lo,
                                           Hi hi, Out out) {
  const int lg = 31 - __clz(G), ng = TH >> lg;
  const int g = threadIdx.x & (G - 1), grp = threadIdx.x >> lg;
  for (int base = 0; base < nrows; base += ng) {     // same trip count for every lane of a warp
    const int i = base + grp;
    Vals<T, NR> a0 = vzero<T, NR>(), a1 = vzero<T, NR>();
    if (i < nrows) {
      const T* row = A + (size_t)i * stride;
      const int e = hi(i);
      int c = lo(i) + g;
      for (; c + (UN - 1) * G < e; c += UN * G) {
        T f[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) f[u] = row[c + u * G];
#pragma unroll
        for (int u = 0; u < UN; ++u) vfma(f[u], vget<T, NR>(vec, c + u * G), (u & 1) ? a1 : a0);
      }
      for (; c < e; c += G) vfma(row[c], vget<T, NR>(vec, c), a0);
    }
    a0 = vadd(a0, a1);
    for (int o = G >> 1; o > 0; o >>= 1) vxor_add(a0, o);
    if (i < nrows && g == 0) out(i, a0);
  }
}

// out(j, sum_{r in [lo(j), hi(j))} A[r][j] vec[r]) for columns j < ncols (rows < nrows): lanes over
// 16 or 32 columns, the rows split over the rest of the CTA; partial sums through red in a fixed
// order.  ORDERED: a thread adds its rows one to the next, else in two sums in turn.  Contains barriers of the
// working warps (none without columns).
template <int TH, typename T, int NR, int UN, bool ORDERED = false, typename Lo, typename Hi, typename Out>
__device__ __forceinline__ void block_cols(const T* __restrict__ A, int stride, int ncols, int nrows, const T* vec,
                                           Lo lo, Hi hi, Out out, T* red) {
  if (ncols <= 0) return;
  const int CW = ncols <= 16 ? 16 : 32;                // columns of a group
  const int tid = threadIdx.x;
  const int cl = tid & (CW - 1), part = tid / CW, parts = TH / CW;
  const int ncg = (ncols + CW - 1) / CW;
  const int ns = ncg >= parts ? 1 : parts / ncg;       // row slices per column group
  const int gpr = parts / ns;                          // column groups per round
  const int slen = (nrows + ns - 1) / ns;
  for (int g0 = 0; g0 < ncg; g0 += gpr) {
    const int gi = g0 + part / ns, si = part % ns;
    const int j = gi * CW + cl;
    Vals<T, NR> a0 = vzero<T, NR>(), a1 = vzero<T, NR>();
    if (part / ns < gpr && j < ncols) {
      const int re = min(hi(j), min(nrows, (si + 1) * slen));
      int r = max(lo(j), si * slen);
      for (; r + UN - 1 < re; r += UN) {
        T f[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) f[u] = A[(size_t)(r + u) * stride + j];
#pragma unroll
        for (int u = 0; u < UN; ++u) vfma(f[u], vget<T, NR>(vec, r + u), (u & 1) && !ORDERED ? a1 : a0);
      }
      for (; r < re; ++r) vfma(A[(size_t)r * stride + j], vget<T, NR>(vec, r), a0);
    }
    a0 = vadd(a0, a1);
    if (ns > 1) {
      vset<T, NR>(red, part * CW + cl, a0);
      work_sync<TH>();
      if (part % ns == 0 && part / ns < gpr && j < ncols) {
        for (int q = 1; q < ns; ++q) a0 = vadd(a0, vget<T, NR>(red, (part + q) * CW + cl));
        out(j, a0);
      }
      work_sync<TH>();
    } else if (part / ns < gpr && j < ncols) {
      out(j, a0);
    }
  }
}

// ---------------------------------------------------------------------------
// Dataflow sweep: one persistent launch runs every unit of one direction.
// CTAs take units from a queue in dependency order (bottom-up levels for
// L / U^T, top-down for U / L^T; inside a level, the phase-1 units of a large
// front before its phase-2 units); a unit waits for the per-front completion
// counters it depends on, runs, then bumps its front's counters.  A unit only
// ever waits for units earlier in the queue, which running CTAs hold, so the
// queue drains whatever the residency (a CTA takes its units in queue order and
// finishes them in that order, so the smallest unfinished unit of the queue is
// always some CTA's current one).
//   bottom-up: whole-front / inverse-block units wait for the children; the
//              off-diagonal units of a front wait for its inverse-block units;
//   top-down:  whole-front / off-diagonal units wait for the parent; the
//              inverse-block units of a front wait for its off-diagonal units.
// Every dependency wait gives up after kSpinLimit polls: it sets *err and the CTA's abort
// word; the CTA's producer then takes no more units, its working warps run the
// one or two staged units to the end (nothing of them is published) and the CTA
// leaves once its copies have landed.  The waits inside a CTA have limits of their own, and
// what follows one is decided for a whole warp, or for all working warps, at once
// (warp_wait, staged_wait).
// ---------------------------------------------------------------------------
constexpr int kSpinLimit = 1 << 21;

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ bool wait_ge(const int* p, int need, int* err) {
  for (int it = 0; it < kSpinLimit; ++it) {
    if (ld_acquire(p) >= need) return true;
    if ((it & 15) == 15 && ld_acquire(err) != 0) return false;
    __nanosleep(32);
  }
  atomicExch(err, 1);
  return false;
}

// A whole small front by one warp, from its staged record d (with its index data) and packed block;
// v: the warp's vectors [n + k][NR].  Returns false when a wait gave up.
template <typename T, int SWEEP, int NR>
__device__ __forceinline__ bool small_front(const SolveLaunch& a, const FlowQueue& q, const SweepFront& d,
                                            const T* __restrict__ pk, T* v, int w, const int* done,
                                            const double2* __restrict__ in, double2* __restrict__ out) {
  constexpr bool kUp = SWEEP == 0 || SWEEP == 2;
  constexpr int kPre = 3;                          // slots per lane (n <= 96)
  const int lane = threadIdx.x & 31;
  const int k = d.k, m = d.m, n = k + m, ks = k | 1;
  const int* cells = reinterpret_cast<const int*>(&d + 1);
  const unsigned* slots = reinterpret_cast<const unsigned*>(cells + n);
  const T* B = pk + pack_rect(k);
  const int* Pm = reinterpret_cast<const int*>(pk + pack_perm(m, k));
  T* ws = v + n * NR;
  bool ok = true;
  for (int rc = a.r0; rc < a.r0 + a.nr; rc += NR) {
    const Chunk<T, NR> c = chunk_of<T, NR>(a, w, rc, in, out);
    const bool first = rc == a.r0;
    if (kUp) {
      Slot<T, NR> s[kPre];
#pragma unroll
      for (int p = 0; p < kPre; ++p) {
        const int t = lane + 32 * p;
        if (t < n) s[p] = slot_staged<T, NR>(a, k, cells, slots, c, (SWEEP == 0 && t < k) ? Pm[t] : t, w);
      }
      if (first) {
        const int dep = lane == 0 ? d.dep0 : (lane == 1 ? d.dep1 : -1);
        const bool okl = dep < 0 || wait_ge(done + dep, q.need_all[dep], q.err);
        ok = __all_sync(0xffffffffu, okl);
        __syncwarp();
      }
      slots_finish<T, NR>(d, c, s, [&](int p) { return lane + 32 * p < n; },
                          [&](int p, const Vals<T, NR>& x) { vset<T, NR>(v, lane + 32 * p, x); });
    } else {
      Vals<T, NR> y[kPre];
#pragma unroll
      for (int p = 0; p < kPre; ++p) {
        const int t = lane + 32 * p;
        if (t < k) y[p] = pivot_val<T, SWEEP, NR>(a, d, c, pk + t, t);
      }
      if (first) {
        const bool okl = lane != 0 || d.parent < 0 || wait_ge(done + d.parent, q.need_all[d.parent], q.err);
        ok = __all_sync(0xffffffffu, okl);
        __syncwarp();
      }
#pragma unroll
      for (int p = 0; p < kPre; ++p) {
        const int t = lane + 32 * p;
        if (t >= k && t < n) y[p] = bound_val<T, SWEEP, NR>(a, c, cells[t], w);
      }
#pragma unroll
      for (int p = 0; p < kPre; ++p) {
        const int t = lane + 32 * p;
        if (t < n) vset<T, NR>(v, t, y[p]);
      }
    }
    __syncwarp();
    if (kUp) {                 // y = X_L (P v)_k;  w = X_U^T v_k
      warp_lines<T, NR>(k, [&](int i, int g, int G) { return tri_walk<T, NR, true>(pk, k, v, SWEEP == 0 ? 1 : 0, i, g, G); },
                        [&](int i, const Vals<T, NR>& s) {
                          const Vals<T, NR> y = SWEEP == 0 ? vadd(vget<T, NR>(v, i), s) : s;
                          vset<T, NR>(ws, i, y);
                          put_v<T, NR>(d, c, i, y);
                        });
    } else {                   // z = y - U12 x_m;  t = w - L21^T x_m
      warp_lines<T, NR>(k, [&](int i, int g, int G) {
                          return walk<T, NR>(B + g * ks + i, G * ks, 0, v + (k + g) * NR, G * NR, (m - g + G - 1) / G);
                        },
                        [&](int i, const Vals<T, NR>& s) { vset<T, NR>(ws, i, vsub(vget<T, NR>(v, i), s)); });
    }
    __syncwarp();
    if (kUp) {                 // u = v_m - (L21 or U12^T) (y or w)
      warp_lines<T, NR>(m, [&](int i, int g, int G) {
                          return walk<T, NR>(B + i * ks + g, G, 0, ws + g * NR, G * NR, (k - g + G - 1) / G);
                        },
                        [&](int i, const Vals<T, NR>& s) { put_v<T, NR>(d, c, k + i, vsub(vget<T, NR>(v, k + i), s)); });
    } else {                   // x_k = X_U z;  x_k = P^T X_L^T t
      warp_lines<T, NR>(k, [&](int i, int g, int G) { return tri_walk<T, NR, false>(pk, k, ws, SWEEP == 1 ? 0 : 1, i, g, G); },
                        [&](int i, const Vals<T, NR>& s) {
                          if (SWEEP == 1) put_x<T, SWEEP, NR>(a, c, cells[i], w, s);
                          else put_x<T, SWEEP, NR>(a, c, cells[Pm[i]], w, vadd(vget<T, NR>(ws, i), s));
                        });
    }
    __syncwarp();
  }
  return ok;
}

// rows of a block from global to shared memory, one bulk copy each, spread over a warp
template <typename T>
__device__ __forceinline__ void stage_rows(const T* src, int ld, const StageGeom& g, T* dst, uint32_t bar) {
  const uint32_t bytes = (uint32_t)(g.cols * (int)sizeof(T));
  for (int i = threadIdx.x & 31; i < g.rows; i += 32)
    bulk_g2s(smem_u32(dst + (size_t)i * g.stride), src + (size_t)(g.row0 + i) * ld + g.col0, bytes, bar);
}

// Row or column view of a staged triangle: entry (i, b) of X_L or X_U for the CTA's products.  A
// packed triangle is stored by diagonals, an inverse block by rows.
template <bool PACKED> __device__ __forceinline__ int tri_at(int hi, int lo, int k, int ld, bool lower) {
  return PACKED ? pack_diag(hi - lo, k) + lo : (lower ? hi * ld + lo : lo * ld + hi);
}

// The triangle products of a whole front by the CTA, G lanes per row or column:
//   SWEEP 0: y_i = v_i + sum_{b < i} X_L[i][b] v_b     SWEEP 2: w_i = sum_{b <= i} X_U[b][i] v_b
//   SWEEP 1: x_i = sum_{b >= i} X_U[i][b] z_b          SWEEP 3: q_i = t_i + sum_{b > i} X_L[b][i] t_b
template <int TH, typename T, int SWEEP, int NR, bool PACKED, typename Out>
__device__ __forceinline__ void block_tri(const T* __restrict__ X, int k, int ld, const T* vec, Out out) {
  constexpr bool kLow = SWEEP == 0 || SWEEP == 3;     // X_L, else X_U
  constexpr bool kBack = SWEEP == 0 || SWEEP == 2;    // entries b below i, else above
  constexpr int t0 = kLow ? 1 : 0;                    // distance of the nearest entry
  const int G = row_lanes(k, TH), lg = 31 - __clz(G), ng = TH >> lg;
  const int g = threadIdx.x & (G - 1), grp = threadIdx.x >> lg;
  for (int base = 0; base < k; base += ng) {          // same trip count for every lane of a warp
    const int i = base + grp;
    Vals<T, NR> a0 = vzero<T, NR>(), a1 = vzero<T, NR>();
    if (i < k) {
      const int e = kBack ? i + 1 : k - i;            // distances t0 .. e - 1
      auto at = [&](int t) { return kBack ? tri_at<PACKED>(i, i - t, k, ld, kLow) : tri_at<PACKED>(i + t, i, k, ld, kLow); };
      auto vi = [&](int t) { return kBack ? i - t : i + t; };
      int t = t0 + g;
      for (; t + 3 * G < e; t += 4 * G) {
        T f[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) f[u] = X[at(t + u * G)];
#pragma unroll
        for (int u = 0; u < 4; ++u) vfma(f[u], vget<T, NR>(vec, vi(t + u * G)), (u & 1) ? a1 : a0);
      }
      for (; t < e; t += G) vfma(X[at(t)], vget<T, NR>(vec, vi(t)), a0);
    }
    a0 = vadd(a0, a1);
    for (int o = G >> 1; o > 0; o >>= 1) vxor_add(a0, o);
    if (i < k && g == 0) out(i, a0);
  }
}

// A whole front by the CTA.  buf: its buffer, v: vectors [n + k][NR] in it behind the staged data.
//   PACKED: [record and index data | packed block]; else [record | X | off-diagonal block].
template <int TH, typename T, int SWEEP, int NR, bool PACKED>
__device__ __forceinline__ bool whole_front(const SolveLaunch& a, const FlowQueue& q, const SweepUnit& un, int w,
                                            const int* done, const double2* __restrict__ in,
                                            double2* __restrict__ out, unsigned char* buf, T* red, volatile int* s_ok) {
  constexpr bool kUp = SWEEP == 0 || SWEEP == 2;
  constexpr int es = (int)sizeof(T);
  constexpr int kPre = 2;
  const int tid = threadIdx.x;
  const SweepFront& d = *reinterpret_cast<const SweepFront*>(buf);
  const int k = d.k, m = d.m, n = k + m, ldk = d.ldk;
  StageGeom g{};
  const T* X;
  const T* B;
  T* v;
  int bs;
  if (PACKED) {
    X = reinterpret_cast<const T*>(buf + un.r0);
    B = X + pack_rect(k);
    bs = k | 1;
    v = reinterpret_cast<T*>(buf + un.r0 + un.cnt);
  } else {
    g = stage_geom(es, SWEEP, true, k, d.ld, ldk, 0, kUp ? m : k, 0, kUp ? k : m, TH);
    X = reinterpret_cast<const T*>(buf + sizeof(SweepFront));
    const T* Bs = X + k * ldk;
    B = Bs + g.shift;
    bs = g.stride;
    v = const_cast<T*>(Bs) + g.rows * g.stride;
  }
  T* ws = v + n * NR;
  const int* cells = PACKED ? reinterpret_cast<const int*>(&d + 1) : a.P.idx + d.idx_off;
  const unsigned* slots = reinterpret_cast<const unsigned*>(cells + n);
  const int* Pm = PACKED ? reinterpret_cast<const int*>(X + pack_perm(m, k))
                         : a.perm + (size_t)w * a.perm_stride + d.piv_off;
  auto fetch = [&](const Chunk<T, NR>& c, int t) {
    const int src = (SWEEP == 0 && t < k) ? Pm[t] : t;
    if constexpr (PACKED) return slot_staged<T, NR>(a, k, cells, slots, c, src, w);
    else return slot_fetch<T, NR>(a, d, c, src, w);
  };
  auto dinv = [&](int t) { return X + (PACKED ? t : t * ldk + t); };
  const int gm = row_lanes(m, TH), gk = row_lanes(k, TH);
  bool ok = true;
  for (int rc = a.r0; rc < a.r0 + a.nr; rc += NR) {
    const Chunk<T, NR> c = chunk_of<T, NR>(a, w, rc, in, out);
    const bool first = rc == a.r0;
    if (kUp) {
      Slot<T, NR> s[kPre];
#pragma unroll
      for (int p = 0; p < kPre; ++p) {
        const int t = tid + TH * p;
        if (t < n) s[p] = fetch(c, t);
      }
      if (first) {
        if (tid < 2) {
          const int dep = tid == 0 ? d.dep0 : d.dep1;
          if (dep >= 0 && !wait_ge(done + dep, q.need_all[dep], q.err)) *s_ok = 0;
        }
        work_sync<TH>();
      }
      slots_finish<T, NR>(d, c, s, [&](int p) { return tid + TH * p < n; },
                          [&](int p, const Vals<T, NR>& x) { vset<T, NR>(v, tid + TH * p, x); });
      for (int t = tid + TH * kPre; t < n; t += TH) {
        const Slot<T, NR> one[1] = {fetch(c, t)};
        slots_finish<T, NR>(d, c, one, [](int) { return true; }, [&](int, const Vals<T, NR>& x) { vset<T, NR>(v, t, x); });
      }
    } else {
      int cell[kPre];
#pragma unroll
      for (int p = 0; p < kPre; ++p) {
        const int t = tid + TH * p;
        cell[p] = t < m ? cells[k + t] : -1;
      }
      for (int t = tid; t < k; t += TH) vset<T, NR>(v, t, pivot_val<T, SWEEP, NR>(a, d, c, dinv(t), t));
      if (first) {
        if (tid == 0 && d.parent >= 0 && !wait_ge(done + d.parent, q.need_all[d.parent], q.err)) *s_ok = 0;
        work_sync<TH>();
      }
      bounds_put<T, SWEEP, NR>(a, c, cell, w, [&](int p, const Vals<T, NR>& x) { vset<T, NR>(v, k + tid + TH * p, x); });
      for (int t = tid + TH * kPre; t < m; t += TH)
        vset<T, NR>(v, k + t, bound_val<T, SWEEP, NR>(a, c, cells[k + t], w));
    }
    work_sync<TH>();
    if (first) ok = *s_ok != 0;
    if (kUp) {
      block_tri<TH, T, SWEEP, NR, PACKED>(X, k, ldk, v, [&](int i, const Vals<T, NR>& s) {
        vset<T, NR>(ws, i, SWEEP == 0 ? vadd(vget<T, NR>(v, i), s) : s);
      });
      work_sync<TH>();
      auto put = [&](int i, const Vals<T, NR>& s) { put_v<T, NR>(d, c, k + i, vsub(vget<T, NR>(v, k + i), s)); };
      if (SWEEP == 0 || PACKED)
        block_rows<TH, T, NR, 4>(B, bs, m, gm, ws, [](int) { return 0; }, [&](int) { return k; }, put);
      else
        block_cols<TH, T, NR, 4>(B, bs, m, k, ws, [](int) { return 0; }, [&](int) { return k; }, put, red);
      for (int i = tid; i < k; i += TH) put_v<T, NR>(d, c, i, vget<T, NR>(ws, i));
    } else {
      auto put = [&](int i, const Vals<T, NR>& s) { vset<T, NR>(ws, i, vsub(vget<T, NR>(v, i), s)); };
      if (SWEEP == 1 && !PACKED)
        block_rows<TH, T, NR, 4>(B, bs, k, gk, v + k * NR, [](int) { return 0; }, [&](int) { return m; }, put);
      else
        block_cols<TH, T, NR, 4>(B, bs, k, m, v + k * NR, [](int) { return 0; }, [&](int) { return m; }, put, red);
      work_sync<TH>();
      auto put_k = [&](int i, const Vals<T, NR>& s) {
        if (SWEEP == 1) put_x<T, SWEEP, NR>(a, c, cells[i], w, s);
        else put_x<T, SWEEP, NR>(a, c, cells[Pm[i]], w, vadd(vget<T, NR>(ws, i), s));
      };
      // L^T of a dense front: neighbouring rows one after the other in one thread's sum.  Where the symmetric form
      // meets a small pivot its row and the next have large entries that cancel; in sums that take rows in turn
      // every term between is rounded at that size (540 x 540, growth 2e4: 2 to 3 times the residual in
      // nine directions, and FGMRES took 12 to 14 vectors instead of 9).  complex128 factors always have pivots.
      if constexpr (SWEEP == 3 && !PACKED && es == 8)
        block_cols<TH, T, NR, 4, true>(X, ldk, k, k, ws, [](int j) { return j + 1; }, [&](int) { return k; }, put_k, red);
      else block_tri<TH, T, SWEEP, NR, PACKED>(X, k, ldk, ws, put_k);
    }
    if (rc + NR < a.r0 + a.nr) work_sync<TH>();
  }
  return ok;
}

// Rows or columns [r0, r0 + cnt) of a large front's inverse block (tri) or off-diagonal block (rect),
// one part [lo, hi) of their contraction; buf: [record | vector | addends | staged block].  The sums
// over the parts are kept in acc (64 lines per right-hand side), which the last part turns into the results.
template <int TH, typename T, int SWEEP, int NR>
__device__ __forceinline__ bool large_unit(const SolveLaunch& a, const FlowQueue& q, const SweepUnit& un, int w,
                                           const int* done, const int* ph1, const double2* __restrict__ in,
                                           double2* __restrict__ out, unsigned char* buf, T* red, T* acc,
                                           volatile int* s_ok) {
  constexpr bool kUp = SWEEP == 0 || SWEEP == 2;
  constexpr bool kRows = SWEEP < 2;
  constexpr int es = (int)sizeof(T);
  constexpr int kPre = 2;
  const int tid = threadIdx.x;
  const SweepFront& d = *reinterpret_cast<const SweepFront*>(buf);
  const bool rect = (un.kind & 0xff) == kUnitRect;
  const int r0 = un.r0, cnt = un.cnt;
  const int k = d.k, m = d.m, ldk = d.ldk;
  const T* Xg = reinterpret_cast<const T*>(a.istore) + (size_t)w * a.istore_stride + d.iv_off;
  const UnitRange ur = unit_range(SWEEP, rect, k, m, r0, cnt);
  const int lo = ur.lo + un.part * un.vslice, hi = min(lo + un.vslice, ur.hi), len = hi - lo;
  const bool first = un.part == 0, last = hi == ur.hi;
  const StageGeom g = stage_geom(es, SWEEP, rect, k, d.ld, ldk, r0, cnt, lo, hi, TH);
  T* v = reinterpret_cast<T*>(buf + sizeof(SweepFront));
  T* gt = v + un.vslice * NR;                         // what the sums are added to or subtracted from
  const T* B = v + unit_vec<NR>(un.vslice, cnt) + g.shift;
  const int* Pm = a.perm + (size_t)w * a.perm_stride + d.piv_off;
  const int* idx = a.P.idx + d.idx_off;
  Chunk<T, NR> c = chunk_of<T, NR>(a, w, a.r0, in, out);
  // before the wait: map entries, right-hand sides, boundary cells
  Slot<T, NR> sl[kPre];
  int cell[kPre] = {-1, -1};
  auto fetch = [&](int t) { return slot_fetch<T, NR>(a, d, c, SWEEP == 0 ? Pm[t] : t, w); };
  if (kUp && !rect) {
#pragma unroll
    for (int p = 0; p < kPre; ++p)
      if (tid + TH * p < len) sl[p] = fetch(lo + tid + TH * p);
  } else if (!kUp && rect) {
#pragma unroll
    for (int p = 0; p < kPre; ++p)
      if (tid + TH * p < len) cell[p] = idx[k + lo + tid + TH * p];
  }
  if (first) {
    if (tid < 2) {
      bool okl = true;
      if (kUp && !rect) {
        const int dep = tid == 0 ? d.dep0 : d.dep1;
        okl = dep < 0 || wait_ge(done + dep, q.need_all[dep], q.err);
      } else if (tid == 0) {
        if (kUp || !rect) okl = wait_ge(ph1 + d.f, q.need_ph1[d.f], q.err);
        else okl = d.parent < 0 || wait_ge(done + d.parent, q.need_all[d.parent], q.err);
      }
      if (!okl) *s_ok = 0;
    }
    work_sync<TH>();
  }
  const bool ok = *s_ok != 0;
  for (int rc = a.r0; rc < a.r0 + a.nr; rc += NR) {
    if (rc != a.r0) c = chunk_of<T, NR>(a, w, rc, in, out);
    T* sum = acc + (size_t)(rc - a.r0) * 64;          // NR values per line, 64 lines per chunk
    if (kUp && !rect) {
      if (rc != a.r0) {
#pragma unroll
        for (int p = 0; p < kPre; ++p)
          if (tid + TH * p < len) sl[p] = fetch(lo + tid + TH * p);
      }
      slots_finish<T, NR>(d, c, sl, [&](int p) { return tid + TH * p < len; },
                          [&](int p, const Vals<T, NR>& x) { vset<T, NR>(v, tid + TH * p, x); });
      for (int t = tid + TH * kPre; t < len; t += TH) {
        const Slot<T, NR> one[1] = {fetch(lo + t)};
        slots_finish<T, NR>(d, c, one, [](int) { return true; }, [&](int, const Vals<T, NR>& x) { vset<T, NR>(v, t, x); });
      }
      if (SWEEP == 0 && last && tid < cnt) {
        const Slot<T, NR> one[1] = {fetch(r0 + tid)};
        slots_finish<T, NR>(d, c, one, [](int) { return true; }, [&](int, const Vals<T, NR>& x) { vset<T, NR>(gt, tid, x); });
      }
    } else if (kUp) {
      for (int t = tid; t < len; t += TH) vset<T, NR>(v, t, front_val<T, NR>(d, c, lo + t));
      if (last && tid < cnt) {
        Slot<T, NR> one[1];
        one[0].t0 = d.inv0 >= 0 ? a.P.inv[d.inv0 + k + r0 + tid] : -1;
        one[0].t1 = d.inv1 >= 0 ? a.P.inv[d.inv1 + k + r0 + tid] : -1;
        one[0].b = vzero<T, NR>();
        slots_finish<T, NR>(d, c, one, [](int) { return true; }, [&](int, const Vals<T, NR>& x) { vset<T, NR>(gt, tid, x); });
      }
    } else if (!rect) {
      // z / t of this front's off-diagonal phase; m = 0: y itself
      auto val = [&](int t) {
        return m == 0 ? pivot_val<T, SWEEP, NR>(a, d, c, Xg + (size_t)t * ldk + t, t) : front_val<T, NR>(d, c, t);
      };
      for (int t = tid; t < len; t += TH) vset<T, NR>(v, t, val(lo + t));
      if (SWEEP == 3 && last && tid < cnt) vset<T, NR>(gt, tid, val(r0 + tid));
    } else {
      if (rc != a.r0) {
#pragma unroll
        for (int p = 0; p < kPre; ++p)
          if (tid + TH * p < len) cell[p] = idx[k + lo + tid + TH * p];
      }
      if (last && tid < cnt)
        vset<T, NR>(gt, tid, pivot_val<T, SWEEP, NR>(a, d, c, Xg + (size_t)(r0 + tid) * ldk + r0 + tid, r0 + tid));
      bounds_put<T, SWEEP, NR>(a, c, cell, w, [&](int p, const Vals<T, NR>& x) { vset<T, NR>(v, tid + TH * p, x); });
      for (int t = tid + TH * kPre; t < len; t += TH)
        vset<T, NR>(v, t, bound_val<T, SWEEP, NR>(a, c, idx[k + lo + t], w));
    }
    work_sync<TH>();
    // line i and the part's contraction index in local coordinates
    auto from = [&](int i) { return rect || kUp ? 0 : max(0, r0 + i + (SWEEP == 3 ? 1 : 0) - lo); };
    auto to = [&](int i) { return rect || !kUp ? len : min(len, r0 + i + (SWEEP == 2 ? 1 : 0) - lo); };
    auto put = [&](int i, const Vals<T, NR>& part) {
      Vals<T, NR> s = part;
      if (!first) s = vadd(vget<T, NR>(sum, i), s);
      if (!last) {
        vset<T, NR>(sum, i, s);
        return;
      }
      const int p = r0 + i;
      if (rect) put_v<T, NR>(d, c, kUp ? k + p : p, vsub(vget<T, NR>(gt, i), s));
      else if (SWEEP == 0) put_v<T, NR>(d, c, p, vadd(vget<T, NR>(gt, i), s));
      else if (SWEEP == 2) put_v<T, NR>(d, c, p, s);
      else if (SWEEP == 1) put_x<T, SWEEP, NR>(a, c, idx[p], w, s);
      else put_x<T, SWEEP, NR>(a, c, idx[Pm[p]], w, vadd(vget<T, NR>(gt, i), s));
    };
    if (kRows) block_rows<TH, T, NR, 4>(B, g.stride, cnt, row_lanes(cnt, TH), v, from, to, put);
    else block_cols<TH, T, NR, 4>(B, g.stride, cnt, len, v, from, to, put, red);
    if (rc + NR < a.r0 + a.nr) work_sync<TH>();
  }
  return ok;
}

// The producer, once a packed unit's index data has landed: brings what the unit will gather from
// global memory and no other front of this sweep writes (bottom-up the right-hand side, top-down the
// values the bottom-up sweep left) into L2.
template <typename T, int SWEEP>
__device__ __forceinline__ void prefetch_vectors(const SolveLaunch& a, const FlowQueue& q, const SweepUnit& un, int w,
                                                 const unsigned char* buf, uint32_t full, uint32_t parity,
                                                 const double2* __restrict__ in) {
  constexpr bool kUp = SWEEP == 0 || SWEEP == 2;
  const int lane = threadIdx.x & 31;
  if (!warp_wait(full, parity, kFreeWaitNs)) return;
  const int cnt = (un.kind >> 8) & 0xff;
  for (int j = 0; j < cnt; ++j) {
    const SweepFront& d = *reinterpret_cast<const SweepFront*>(buf + 16 * (size_t)un.off[j]);
    const int* cells = reinterpret_cast<const int*>(&d + 1);
    const int k = d.k;
    for (int r = a.r0; r < a.r0 + a.nr; ++r) {
      const size_t sys = (size_t)w * a.nrhs + r;
      if (kUp) {
        for (int t = lane; t < k; t += 32)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(in + sys * a.n + cells[t]));
      } else {
        const char* y = reinterpret_cast<const char*>(reinterpret_cast<const T*>(a.vb) + sys * a.vec_stride + d.v_off);
        if (32 * lane < k * (int)sizeof(T)) asm volatile("prefetch.global.L2 [%0];" ::"l"(y + 32 * lane));
      }
    }
  }
  __syncwarp();
}

// MINB: CTAs per SM the register allocation aims for
template <int TH, int MINB, typename T, int SWEEP, int NR>
__global__ void __launch_bounds__(TH + 64, MINB)
flow_kernel(SolveLaunch a, FlowQueue q, const double2* __restrict__ in, double2* __restrict__ out, int bufsz,
            int two) {
  constexpr bool kUp = SWEEP == 0 || SWEEP == 2;
  constexpr int es = (int)sizeof(T);
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(16) T red[TH * NR];
  __shared__ __align__(16) T acc[64 * kFlowMaxRhs];    // sums of a tri / rect unit over its parts
  // per buffer: full (staged), done (the working warps have finished it), free (its unit may be overwritten)
  __shared__ __align__(8) uint64_t bars[6];
  __shared__ __align__(16) SweepUnit s_unit[2];
  __shared__ int s_wl[2], s_ok[2];
  __shared__ int s_abort, s_stop;
  const int nf = q.n_fronts;
  int* head = q.ctr;
  int* done0 = q.ctr + 1;                       // [n_omega launched][nf]
  int* ph10 = done0 + (size_t)a.n_omega * nf;   // [n_omega launched][nf]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t full0 = smem_u32(&bars[0]), done_b0 = smem_u32(&bars[2]), free0 = smem_u32(&bars[4]);
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(full0 + 8 * i, 1);
      mbar_init(done_b0 + 8 * i, TH / 32);
      mbar_init(free0 + 8 * i, 1);
    }
    mbar_init_fence();
    s_abort = 0;
    s_stop = kGoOn;
  }
  __syncthreads();
  if (warp == TH / 32) {
    // ---- producer: takes units in queue order and stages them ----
    const int total = q.nunits * a.n_omega;
    int it = 0;
    bool gave_up = false, prev_packed = false;
    // units are taken, and their records read, one ahead of the buffer they will go to
    auto take = [&]() {
      int v = total;
      if (lane == 0 && *(volatile int*)&s_abort == 0) v = atomicAdd(head, 1);
      return __shfl_sync(0xffffffffu, v, 0);
    };
    // the working warps may set it at any time: one lane reads it for all
    auto aborted = [&]() { return __shfl_sync(0xffffffffu, *(volatile int*)&s_abort, 0) != 0; };
    int u = take();
    SweepUnit un{};
    if (u < total) un = q.units[u / a.n_omega];
    for (;; ++it) {
      const int b = it & two;
      unsigned char* buf = smem + (size_t)b * bufsz;
      if (prev_packed && two)
        prefetch_vectors<T, SWEEP>(a, q, s_unit[b ^ 1], s_wl[b ^ 1] + a.w0, smem + (size_t)(b ^ 1) * bufsz,
                                   full0 + 8 * (b ^ 1), ((it - 1) >> 1) & 1, in);
      prev_packed = false;
      if (it > two && !warp_wait(free0 + 8 * b, ((it >> two) - 1) & 1, kFreeWaitNs)) {
        if (lane == 0) { s_abort = 1; atomicExch(q.err, 1); }
        gave_up = true;
        break;
      }
      if (u >= total || (un.part == 0 && aborted())) {
        if (lane == 0) {
          s_unit[b].kind = kUnitEnd;
          mbar_arrive(full0 + 8 * b);
        }
        break;
      }
      const int wl = u - u / a.n_omega * a.n_omega, w = wl + a.w0;
      const int kind = un.kind & 0xff;
      bool last = true;
      SweepFront d;
      StageGeom g;
      if (kind > kUnitPacked) {
        d = q.fronts[un.rec];
        if (kind == kUnitFront) {
          g = stage_geom(es, SWEEP, true, d.k, d.ld, d.ldk, 0, kUp ? d.m : d.k, 0, kUp ? d.k : d.m, TH);
        } else {
          const bool rect = kind == kUnitRect;
          const UnitRange ur = unit_range(SWEEP, rect, d.k, d.m, un.r0, un.cnt);
          const int lo = ur.lo + un.part * un.vslice, hi = min(lo + un.vslice, ur.hi);
          last = hi == ur.hi;
          g = stage_geom(es, SWEEP, rect, d.k, d.ld, d.ldk, un.r0, un.cnt, lo, hi, TH);
        }
      }
      if (lane == 0) {
        s_unit[b] = un;
        if (last) s_unit[b].kind = un.kind | kUnitLast;
        s_wl[b] = wl;
        s_ok[b] = 1;
      }
      async_fence();
      if (kind <= kUnitPacked) {
        prev_packed = true;
        if (lane == 0) {
          const T* src = reinterpret_cast<const T*>(a.pack) + (size_t)w * a.pack_stride +
                         ((SWEEP == 1 || SWEEP == 2) ? a.pack_stride / 2 : 0) + un.fac;
          mbar_expect_tx(full0 + 8 * b, (uint32_t)(un.r0 + un.cnt));
          bulk_g2s(smem_u32(buf), q.meta + 16 * (size_t)un.rec, (uint32_t)un.r0, full0 + 8 * b);
          bulk_g2s(smem_u32(buf + un.r0), src, (uint32_t)un.cnt, full0 + 8 * b);
        }
      } else {
        const T* Xg = reinterpret_cast<const T*>(a.istore) + (size_t)w * a.istore_stride + d.iv_off;
        const T* Fg = reinterpret_cast<const T*>(a.store) + (size_t)w * a.store_stride + d.st_off;
        T* x0 = reinterpret_cast<T*>(buf + sizeof(SweepFront));
        const uint32_t xb = kind == kUnitFront ? (uint32_t)(d.k * d.ldk * es) : 0u;
        if (lane == 0) {
          mbar_expect_tx(full0 + 8 * b, (uint32_t)sizeof(SweepFront) + xb + (uint32_t)(g.rows * g.cols * es));
          bulk_g2s(smem_u32(buf), q.fronts + un.rec, (uint32_t)sizeof(SweepFront), full0 + 8 * b);
          if (xb) bulk_g2s(smem_u32(x0), Xg, xb, full0 + 8 * b);
        }
        __syncwarp();
        T* dst = kind == kUnitFront ? x0 + d.k * d.ldk : x0 + unit_vec<NR>(un.vslice, un.cnt);
        stage_rows<T>(kind == kUnitTri ? Xg : Fg, kind == kUnitTri ? d.ldk : d.ld, g, dst, full0 + 8 * b);
      }
      if (!last) {
        ++un.part;
      } else {
        u = take();
        if (u < total) un = q.units[u / a.n_omega];
      }
    }
    // The copies issued last have landed before the CTA leaves: the last unit's (the one before it
    // had landed when its buffer became free; after a give-up its landing is waited for here too).
    __syncwarp();
    for (int i = gave_up ? it - 1 - two : it - two; i < it; ++i)
      if (i >= 0) mbar_wait(full0 + 8 * (i & two), (i >> two) & 1, kFreeWaitNs);
  } else if (warp == TH / 32 + 1) {
    // ---- publisher: once the working warps have finished a unit, its buffer is free and its
    // fronts' counters go up, after a fence that orders the CTA's stores before them ----
    for (int it = 0;; ++it) {
      const int b = it & two;
      if (!warp_wait(done_b0 + 8 * b, (it >> two) & 1, kDoneWaitNs)) {
        if (lane == 0) {
          s_abort = 1;
          atomicExch(q.err, 1);
          stop_unless_staged(full0 + 8 * b, (it >> two) & 1, &s_stop);
        }
        break;
      }
      const int kc = s_unit[b].kind, kind = kc & 0xff;
      if (kind == kUnitEnd) break;
      const unsigned char* buf = smem + (size_t)b * bufsz;
      const int cnt = kind == kUnitSmall ? (kc >> 8) & 0xff : 1;
      const size_t base = (size_t)s_wl[b] * nf;
      int f = 0;
      if (lane < cnt)
        f = reinterpret_cast<const SweepFront*>(buf + (kind == kUnitSmall ? 16 * (size_t)s_unit[b].off[lane] : 0))->f;
      const bool ok = s_ok[b] != 0 && *(volatile int*)&s_abort == 0 && (kc & kUnitLast) != 0;
      __syncwarp();
      if (lane == 0) mbar_arrive(free0 + 8 * b);
      if (lane < cnt && ok) {
        __threadfence();
        // phase 1: inverse-block units bottom-up, off-diagonal units top-down
        if (kind == (kUp ? kUnitTri : kUnitRect)) atomicAdd(ph10 + base + f, 1);
        atomicAdd(done0 + base + f, 1);
      }
    }
  } else {
    // ---- working warps ----
    for (int it = 0;; ++it) {
      const int b = it & two;
      unsigned char* buf = smem + (size_t)b * bufsz;
      const bool staged = staged_wait(full0 + 8 * b, (it >> two) & 1, &s_stop);
      __syncwarp();
      if (!staged) {
        if (lane == 0) { s_abort = 1; atomicExch(q.err, 1); }
        break;
      }
      const SweepUnit& un = s_unit[b];
      const int kind = un.kind & 0xff;
      if (kind != kUnitEnd) {
        const int w = s_wl[b] + a.w0;
        const int* done = done0 + (size_t)s_wl[b] * nf;
        bool ok = true;
        if (kind == kUnitSmall) {
          if (warp < ((un.kind >> 8) & 0xff)) {
            const SweepFront& d = *reinterpret_cast<const SweepFront*>(buf + 16 * (size_t)un.off[warp]);
            const T* pk = reinterpret_cast<const T*>(buf + un.r0) + (d.pk_off - un.fac);
            T* v = reinterpret_cast<T*>(buf + un.r0 + un.cnt + (size_t)warp * un.vslice);
            ok = small_front<T, SWEEP, NR>(a, q, d, pk, v, w, done, in, out);
          }
        } else if (kind == kUnitPacked) {
          ok = whole_front<TH, T, SWEEP, NR, true>(a, q, un, w, done, in, out, buf, red, &s_ok[b]);
        } else if (kind == kUnitFront) {
          ok = whole_front<TH, T, SWEEP, NR, false>(a, q, un, w, done, in, out, buf, red, &s_ok[b]);
        } else {
          ok = large_unit<TH, T, SWEEP, NR>(a, q, un, w, done, ph10 + (size_t)s_wl[b] * nf, in, out, buf, red,
                                            acc, &s_ok[b]);
        }
        if (!ok) {
          s_ok[b] = 0;
          s_abort = 1;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(done_b0 + 8 * b);
      if (kind == kUnitEnd) break;
    }
  }
}


// The launches of one shape: instantiated once per translation unit.
template <int TH, int MINB, typename T, int NR>
void launch_flow(const SolveLaunch& a, int sweep, const FlowQueue& q, const FlowShape& sh, int grid, const double2* i,
                 double2* o, cudaStream_t s) {
  switch (sweep) {
    case 0: flow_kernel<TH, MINB, T, 0, NR><<<grid, TH + 64, sh.buffers * sh.smem, s>>>(a, q, i, o, sh.smem, sh.buffers - 1); break;
    case 1: flow_kernel<TH, MINB, T, 1, NR><<<grid, TH + 64, sh.buffers * sh.smem, s>>>(a, q, i, o, sh.smem, sh.buffers - 1); break;
    case 2: flow_kernel<TH, MINB, T, 2, NR><<<grid, TH + 64, sh.buffers * sh.smem, s>>>(a, q, i, o, sh.smem, sh.buffers - 1); break;
    default: flow_kernel<TH, MINB, T, 3, NR><<<grid, TH + 64, sh.buffers * sh.smem, s>>>(a, q, i, o, sh.smem, sh.buffers - 1); break;
  }
}

template <int TH, int MINB, typename T, int NR>
int blocks_per_sm(int smem) {
  int best = 1 << 20, nb = 0;
#define FDFD_OCC(S)                                                                                                  \
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, flow_kernel<TH, MINB, T, S, NR>, TH + 64, smem) != cudaSuccess) \
    nb = 1;                                                                                                          \
  best = nb < best ? nb : best;
  FDFD_OCC(0) FDFD_OCC(1) FDFD_OCC(2) FDFD_OCC(3)
#undef FDFD_OCC
  return best > 0 ? best : 1;
}

template <int TH, int MINB, typename T, int NR>
cudaError_t flow_attributes() {
  cudaError_t e = cudaSuccess;
#define FDFD_ATTR(S)     \
  if (e == cudaSuccess)  \
    e = cudaFuncSetAttribute(flow_kernel<TH, MINB, T, S, NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFlowMaxSmem);
  FDFD_ATTR(0) FDFD_ATTR(1) FDFD_ATTR(2) FDFD_ATTR(3)
#undef FDFD_ATTR
  return e;
}

}  // namespace

// One shape's launches, for the dispatch in solve.cu.
#define FDFD_FLOW_SHAPE(NAME, TH, MINB, T, NR)                                                                 \
  void flow_launch_##NAME(const SolveLaunch& a, int sweep, const FlowQueue& q, const FlowShape& sh, int grid,   \
                          const double2* in, double2* out, cudaStream_t s) {                                    \
    launch_flow<TH, MINB, T, NR>(a, sweep, q, sh, grid, in, out, s);                                                  \
  }                                                                                                             \
  int flow_blocks_##NAME(int smem) { return blocks_per_sm<TH, MINB, T, NR>(smem); }                                   \
  cudaError_t flow_init_##NAME() { return flow_attributes<TH, MINB, T, NR>(); }

}  // namespace fdfd
