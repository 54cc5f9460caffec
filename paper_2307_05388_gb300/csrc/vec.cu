// Operator assembly tables (Eq. 1-2 with stretched-coordinate PML), the FP64
// matrix-free stencil used by the refinement, FGMRES vector kernels, the
// mode-overlap objective with its adjoint source (Eq. 4) and the pixel
// gradient (Eq. 3).
//
// Operator (dimensionless: Eq. 1 multiplied by mu0 dx^2), row (i, j):
//   A[(i,j),(i-1,j)] = cxm[i] = -1 / (sx(i+1/2) sx(i)),   A[(i,j),(i+1,j)] = cxp[i] = -1 / (sx(i+1/2) sx(i+1))
//   A[(i,j),(i,j-1)] = cym[j],                            A[(i,j),(i,j+1)] = cyp[j]
//   A[(i,j),(i,j)]   = -(cxm + cxp + cym + cyp) - (k0 dx)^2 eps[i,j]
// with positions in cell units (cell i centred at i + 1/2) and the stretch
//   s(u) = 1 - i * [-(order+1) ln R / (2 k0dx npml)] * d(u)^order,
//   d(u) = max(npml - u, u - (n - npml), 0) / npml,
// i.e. e^{+i w t} convention: s = 1 - i sigma / (omega eps0).  Neighbours
// beyond the grid are zero (PEC behind the PML).
#include "kernels.h"

namespace fdfd {

namespace {

__device__ double2 stretch(double u, int n, int npml, double k0dx, double ln_R, double order) {
  if (npml <= 0) return make_double2(1.0, 0.0);
  double d = fmax(fmax((double)npml - u, u - (double)(n - npml)), 0.0) / (double)npml;
  double smax = -(order + 1.0) * ln_R / (2.0 * k0dx * (double)npml);
  double p = (order == 3.0) ? d * d * d : pow(d, order);
  return make_double2(1.0, -smax * p);
}

__device__ double2 neg_inv_prod(double2 a, double2 b) {
  double2 p = cmul(a, b);
  double2 r = crcp(p);
  return make_double2(-r.x, -r.y);
}

__global__ void coef_kernel(double2* cxm, double2* cxp, double2* cym, double2* cyp, double* k0dx2,
                            double2* sxc, double2* syc, const double* k0dx, int n_omega, int nx, int ny, int px,
                            int py, double ln_R, double order) {
  const int w = blockIdx.y;
  const double kd = k0dx[w];
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t == 0) k0dx2[w] = kd * kd;
  if (t < nx) {
    const double2 sc = stretch(t + 0.5, nx, px, kd, ln_R, order);
    cxm[(size_t)w * nx + t] = neg_inv_prod(sc, stretch(t, nx, px, kd, ln_R, order));
    cxp[(size_t)w * nx + t] = neg_inv_prod(sc, stretch(t + 1.0, nx, px, kd, ln_R, order));
    sxc[(size_t)w * nx + t] = sc;
  }
  if (t < ny) {
    const double2 sc = stretch(t + 0.5, ny, py, kd, ln_R, order);
    cym[(size_t)w * ny + t] = neg_inv_prod(sc, stretch(t, ny, py, kd, ln_R, order));
    cyp[(size_t)w * ny + t] = neg_inv_prod(sc, stretch(t + 1.0, ny, py, kd, ln_R, order));
    syc[(size_t)w * ny + t] = sc;
  }
}

__global__ void scatter_design_kernel(double* eps, const double* ed, int ny, int x0, int y0, int w, int h) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)w * h) return;
  const int i = (int)(t / h), j = (int)(t - (long long)i * h);
  eps[(size_t)(x0 + i) * ny + y0 + j] = ed[t];
}

// (A X)[cell] (transpose: A^T) for wavelength w, X one system's vector
__device__ __forceinline__ double2 stencil_at(const DevCoef& c, int w, int transpose, const double2* __restrict__ X,
                                              long long cell) {
  const int ci = (int)cell;                    // grids stay below 2^31 cells
  const int i = ci / c.ny, j = ci - i * c.ny;
  if (i > c.px && i < c.nx - 1 - c.px && j > c.py && j < c.ny - 1 - c.py) {
    // between the absorbing layers every coupling is exactly -1 (and A = A^T there): 9 FP64
    // operations per cell instead of 27
    const double2 xw = X[cell - c.ny], xe = X[cell + c.ny], xs = X[cell - 1], xn = X[cell + 1], x0 = X[cell];
    const double dg = fma(-c.k0dx2[w], c.eps[cell], 4.0);
    const double sx = (xw.x + xe.x) + (xs.x + xn.x), sy = (xw.y + xe.y) + (xs.y + xn.y);
    return make_double2(fma(dg, x0.x, -sx), fma(dg, x0.y, -sy));
  }
  const double2* cxm = c.cxm + (size_t)w * c.nx;
  const double2* cxp = c.cxp + (size_t)w * c.nx;
  const double2* cym = c.cym + (size_t)w * c.ny;
  const double2* cyp = c.cyp + (size_t)w * c.ny;
  double2 dg;
  dg.x = -(cxm[i].x + cxp[i].x + cym[j].x + cyp[j].x) - c.k0dx2[w] * c.eps[cell];
  dg.y = -(cxm[i].y + cxp[i].y + cym[j].y + cyp[j].y);
  double2 acc = cmul(dg, X[cell]);
  if (!transpose) {
    if (i > 0) acc = cfma(cxm[i], X[cell - c.ny], acc);
    if (i + 1 < c.nx) acc = cfma(cxp[i], X[cell + c.ny], acc);
    if (j > 0) acc = cfma(cym[j], X[cell - 1], acc);
    if (j + 1 < c.ny) acc = cfma(cyp[j], X[cell + 1], acc);
  } else {
    if (i > 0) acc = cfma(cxp[i - 1], X[cell - c.ny], acc);
    if (i + 1 < c.nx) acc = cfma(cxm[i + 1], X[cell + c.ny], acc);
    if (j > 0) acc = cfma(cyp[j - 1], X[cell - 1], acc);
    if (j + 1 < c.ny) acc = cfma(cym[j + 1], X[cell + 1], acc);
  }
  return acc;
}

// y = A x; transpose selects A^T.
__global__ void stencil_kernel(DevCoef c, int nrhs, int transpose, const double2* __restrict__ x,
                               double2* __restrict__ y) {
  const int sys = blockIdx.y;
  const long long N = (long long)c.nx * c.ny;
  const long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (cell >= N) return;
  y[(size_t)sys * N + cell] = stencil_at(c, sys / nrhs, transpose, x + (size_t)sys * N, cell);
}

constexpr int kDotThreads = 256;
constexpr int kMaxDot = 17;

// w[s] -= sum_i h[s][i] V_i[s] (set: from w = 0); the coefficients sit in shared memory.
__global__ void multiaxpy_kernel(const double2* __restrict__ V, long long vstride, int nv,
                                 const double2* __restrict__ h, int h_ld, double2* w, long long n, int set) {
  __shared__ double2 hh[kMaxDot];
  const int sys = blockIdx.y;
  if (threadIdx.x < nv) hh[threadIdx.x] = h[(size_t)sys * h_ld + threadIdx.x];
  __syncthreads();
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    double2 acc = set ? make_double2(0, 0) : w[(size_t)sys * n + t];
    for (int i = 0; i < nv; ++i) acc = cfms(hh[i], V[(size_t)i * vstride + (size_t)sys * n + t], acc);
    w[(size_t)sys * n + t] = acc;
  }
}

int grid_for(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b < 4096 ? b : 4096);
}

}  // namespace

void launch_coef(double2* cxm, double2* cxp, double2* cym, double2* cyp, double* k0dx2, double2* sxc,
                 double2* syc, const double* k0dx_dev, int n_omega, int nx, int ny, int npml_x, int npml_y,
                 double ln_R, double order, cudaStream_t s) {
  const int nmax = nx > ny ? nx : ny;
  coef_kernel<<<dim3((nmax + 127) / 128, n_omega), 128, 0, s>>>(cxm, cxp, cym, cyp, k0dx2, sxc, syc, k0dx_dev,
                                                               n_omega, nx, ny, npml_x, npml_y, ln_R, order);
}

void launch_scatter_design(double* eps, const double* eps_design, int ny, int x0, int y0, int w, int h,
                           cudaStream_t s) {
  const long long n = (long long)w * h;
  if (n <= 0) return;
  scatter_design_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(eps, eps_design, ny, x0, y0, w, h);
}

void launch_stencil(const DevCoef& c, int n_omega, int nrhs, int transpose, const double2* x, double2* y,
                    cudaStream_t s) {
  const long long N = (long long)c.nx * c.ny;
  stencil_kernel<<<dim3((unsigned)((N + 255) / 256), n_omega * nrhs), 256, 0, s>>>(c, nrhs, transpose, x, y);
}


int multidot_max_vectors() { return kMaxDot; }

void launch_multiaxpy(const double2* V, long long vstride, int nv, const double2* h, int h_ld, double2* w,
                      long long n, int nsys, int set, cudaStream_t s) {
  multiaxpy_kernel<<<dim3(grid_for(n), nsys), 256, 0, s>>>(V, vstride, nv, h, h_ld, w, n, set);
}

// ---------------------------------------------------------------------------
// FGMRES bookkeeping per system (one thread per system).
// ---------------------------------------------------------------------------
namespace {

// Start of a cycle for system s from |r|^2 (first: x = 0, r = b, and |b| is taken from it).
__device__ void start_system(const ArnoldiStep& g, int s, double rr2, int first) {
  // norms from sums of squares; a NaN stays NaN (fmax would turn it into 0, and a
  // poisoned solve would then look converged)
  const double beta = rr2 > 0.0 ? sqrt(rr2) : (rr2 == rr2 ? 0.0 : rr2);
  if (first) g.bnorm[s] = beta;
  const double bn = first ? beta : g.bnorm[s];
  for (int i = 0; i <= g.m; ++i) g.g[(size_t)s * (g.m + 1) + i] = make_double2(0, 0);
  g.g[(size_t)s * (g.m + 1)] = make_double2(beta, 0);
  g.resid[s] = bn > 0 ? beta / bn : 0.0;
  const int act = (bn > 0) && (beta > g.tol * bn) && (beta == beta);
  g.active[s] = act;
  g.vscale[s] = act ? 1.0 / beta : 0.0;
  g.nj_out[s] = first ? 0 : g.nj[s];   // Krylov vectors of the cycle that ended
  g.nj[s] = 0;
  if (first) g.reorth[s] = 0;
  g.loss[s] = 0.0;
}

// Column j of the Hessenberg matrix of system s from its projections h[0..j]
// and hn2 = |w|^2: earlier rotations applied, a new one formed, the residual
// estimate updated; a system whose estimate meets tol (or breaks down: exact
// solution) becomes inactive.
__device__ void givens_step(int s, const double2* hs, double hn2, int j, int m, double tol, double2* H, double2* cs,
                            double2* sn, double2* g, double* vscale, int* active, double* resid,
                            const double* bnorm) {
  double2* Hc = H + ((size_t)s * m + j) * (m + 1);   // column j of H
  for (int i = 0; i <= j; ++i) Hc[i] = hs[i];
  const double hnorm = hn2 > 0.0 ? sqrt(hn2) : (hn2 == hn2 ? 0.0 : hn2);
  Hc[j + 1] = make_double2(hnorm, 0);
  double2* C = cs + (size_t)s * m;
  double2* S = sn + (size_t)s * m;
  for (int i = 0; i < j; ++i) {   // apply earlier rotations
    const double2 x = Hc[i], y = Hc[i + 1];
    const double c = C[i].x;
    Hc[i] = cadd(make_double2(c * x.x, c * x.y), cmul(S[i], y));
    Hc[i + 1] = csub(make_double2(c * y.x, c * y.y), cmul(cconj(S[i]), x));
  }
  const double2 a = Hc[j];
  const double b = hnorm;
  const double aa = sqrt(a.x * a.x + a.y * a.y);
  double c;
  double2 sv, r;
  if (aa == 0.0) {
    c = 0.0; sv = make_double2(1, 0); r = make_double2(b, 0);
  } else {
    const double t = sqrt(aa * aa + b * b);
    const double2 ph = make_double2(a.x / aa, a.y / aa);
    c = aa / t;
    sv = make_double2(ph.x * b / t, ph.y * b / t);
    r = make_double2(ph.x * t, ph.y * t);
  }
  C[j] = make_double2(c, 0);
  S[j] = sv;
  Hc[j] = r;
  Hc[j + 1] = make_double2(0, 0);
  double2* G = g + (size_t)s * (m + 1);
  const double2 gj = G[j];
  G[j + 1] = make_double2(-(sv.x * gj.x + sv.y * gj.y), -(sv.x * gj.y - sv.y * gj.x));  // -conj(s) g_j
  G[j] = make_double2(c * gj.x, c * gj.y);
  const double rn = sqrt(G[j + 1].x * G[j + 1].x + G[j + 1].y * G[j + 1].y);
  const double bn = bnorm[s];
  resid[s] = rn / bn;
  vscale[s] = hnorm > 0 ? 1.0 / hnorm : 0.0;
  if (!(rn > tol * bn) || !(hnorm > 0)) active[s] = 0;   // converged (or breakdown: solution exact)
}

// y = R^-1 g over the first nj columns, then x += sum_i y_i Z_i is done by multiaxpy with -y.
__global__ void gm_solve_kernel(const double2* H, const double2* g, int nsys, int m, const int* njs,
                                double2* ny_out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nsys) return;
  const int nj = njs[s];
  const double2* Hs = H + (size_t)s * m * (m + 1);
  const double2* G = g + (size_t)s * (m + 1);
  double2 y[kMaxDot];
  for (int i = nj - 1; i >= 0; --i) {
    double2 acc = G[i];
    for (int q = i + 1; q < nj; ++q) acc = cfms(Hs[(size_t)q * (m + 1) + i], y[q], acc);
    y[i] = cmul(acc, crcp(Hs[(size_t)i * (m + 1) + i]));
  }
  for (int i = 0; i < kMaxDot; ++i)
    ny_out[(size_t)s * kMaxDot + i] = i < nj ? make_double2(-y[i].x, -y[i].y) : make_double2(0, 0);
}

__global__ void scale_vec_kernel(double2* dst, const double2* src, const double* scale, long long n) {
  const int sys = blockIdx.y;
  const double sc = scale[sys];
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const double2 v = src[(size_t)sys * n + t];
    dst[(size_t)sys * n + t] = make_double2(v.x * sc, v.y * sc);
  }
}


// ---------------------------------------------------------------------------
// FGMRES over the vectors of every system: one launch per pass, CTA (chunk of PER * 256 entries,
// system).  Each CTA writes its partial sums and the last CTA of a system (a counter it resets
// afterwards) adds them in chunk order, so results do not depend on timing, and runs the
// system's bookkeeping.
//
//   kPassStart  |b|^2, start of the first cycle (x = 0)
//   kPassResid  r = b - A x, |r|^2, start of a later cycle
//   kPassApply  e = A z_j - v_j,             h_i = V_i^H e,  |e|^2
//   kPassProj   e -= sum_i h_i V_i,          |e|^2, then the Givens update of column j
//   kPassDots2  h2_i = V_i^H e               (systems marked by kPassProj)
//   kPassProj2  e -= sum_i h2_i V_i,         |e|^2, then their Givens update
//
// The preconditioner is close to A^-1, so A z_j lies almost along v_j and projecting it once leaves a
// vector that is orthogonal only to the rounding of the large component: Gram-Schmidt used to run
// twice for that.  Taking v_j off first (h_jj = 1 + V_j^H e) removes the large component exactly, and
// one projection of the small rest is enough unless it cancels again.  What one projection loses is
// followed per system: loss_{j+1} = (loss_j |e| + 2^-52) / |e'|.  Where it would pass 1e-3 the second
// projection (kPassDots2, kPassProj2) runs, after which loss_{j+1} = (loss_j + 2^-52) |e'| / |e''|.  Its two
// launches are left out until a system has asked for it: the first time, the cycle of that system ends there
// (the next one starts from the true residual) and the host launches them from then on, in this solve and
// in the following ones of that direction on these factors as long as they run for some system.
//
// FP64 is 2 multiply-adds per clock and SM on this part and bounds these passes.  Eight entries per thread and
// a butterfly that halves the values with the lanes (6 additions for two complex sums where a plain
// shuffle tree takes 20) keep the reductions' share small, and the stencil takes 9 operations between the
// absorbing layers.
// ---------------------------------------------------------------------------
constexpr double kMaxLoss = 1e-3;

// Sums of two complex values over the warp: lanes 0, 8, 16, 24 end up with a.x, a.y, b.x, b.y.
__device__ __forceinline__ double warp_sum2(double2 a, double2 b, int lane) {
  const bool up16 = lane & 16, up8 = lane & 8;
  const double k0 = up16 ? b.x : a.x, k1 = up16 ? b.y : a.y, s0 = up16 ? a.x : b.x, s1 = up16 ? a.y : b.y;
  const double r0 = k0 + __shfl_xor_sync(0xffffffffu, s0, 16), r1 = k1 + __shfl_xor_sync(0xffffffffu, s1, 16);
  double v = (up8 ? r1 : r0) + __shfl_xor_sync(0xffffffffu, up8 ? r0 : r1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Column nv - 1 of system s from the projections h (and h2) and |e'|^2.
__device__ void finish_column(const ArnoldiStep& g, int s, const double2* h, const double2* h2, double hn2) {
  double2 hs[kMaxDot];
  for (int i = 0; i < g.nv; ++i) hs[i] = h2 ? cadd(h[i], h2[i]) : h[i];
  hs[g.nv - 1].x += 1.0;
  g.nj[s] += 1;
  givens_step(s, hs, hn2, g.nv - 1, g.m, g.tol, g.H, g.cs, g.sn, g.g, g.vscale, g.active, g.resid, g.bnorm);
}

template <int PER>
__global__ void __launch_bounds__(kDotThreads, PER >= 8 ? 2 : 3)
arnoldi_kernel(ArnoldiStep g, int pass) {
  __shared__ double red[kDotThreads / 32][2 * (kMaxDot + 1)];
  __shared__ double2 hc[kMaxDot];
  __shared__ int s_last;
  const int sys = blockIdx.y;
  const bool begin = pass == kPassStart || pass == kPassResid;
  if (!begin && !g.active[sys]) return;
  if ((pass == kPassDots2 || pass == kPassProj2) && !g.again[sys]) return;
  const int nv = g.nv, nblk = gridDim.x;
  const long long n = (long long)g.C.nx * g.C.ny;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool project = pass == kPassProj || pass == kPassProj2;
  if (project && tid < nv) hc[tid] = (pass == kPassProj ? g.h1 : g.h2)[(size_t)sys * kMaxDot + tid];
  __syncthreads();
  double2* W = g.w + (size_t)sys * n;
  const double2* Vs = g.V + (size_t)sys * n;
  const long long t0 = (long long)blockIdx.x * (kDotThreads * PER) + tid;
  double2 wv[PER];
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const long long t = t0 + (long long)u * kDotThreads;
    double2 x = make_double2(0, 0);
    if (t < n) {
      if (pass == kPassStart) {
        x = g.b[(size_t)sys * n + t];
      } else if (pass == kPassResid) {
        x = csub(g.b[(size_t)sys * n + t], stencil_at(g.C, sys / g.nrhs, g.transpose, g.z + (size_t)sys * n, t));
        W[t] = x;
      } else if (pass == kPassApply) {
        x = csub(stencil_at(g.C, sys / g.nrhs, g.transpose, g.z + (size_t)sys * n, t),
                 Vs[(size_t)(nv - 1) * g.vstride + t]);
        W[t] = x;
      } else {
        x = W[t];
      }
    }
    wv[u] = x;
  }
  if (project) {
    for (int i = 0; i < nv; ++i) {
      const double2 h = hc[i];
      const double2* Vi = Vs + (size_t)i * g.vstride;
      double2 vv[PER];
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        const long long t = t0 + (long long)u * kDotThreads;
        vv[u] = t < n ? Vi[t] : make_double2(0, 0);
      }
#pragma unroll
      for (int u = 0; u < PER; ++u) wv[u] = cfms(h, vv[u], wv[u]);
    }
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const long long t = t0 + (long long)u * kDotThreads;
      if (t < n) W[t] = wv[u];
    }
  }
  // outputs 0 .. nd - 1: V_i^H w; output nd: |w|^2 (but in kPassDots2)
  const int nd = (pass == kPassApply || pass == kPassDots2) ? nv : 0;
  const int nout = pass == kPassDots2 ? nd : nd + 1;
  for (int i = 0; i < nout; i += 2) {
    double2 acc[2] = {make_double2(0, 0), make_double2(0, 0)};
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      if (i + p < nd) {
        const double2* Vi = Vs + (size_t)(i + p) * g.vstride;
        double2 vv[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
          const long long t = t0 + (long long)u * kDotThreads;
          vv[u] = t < n ? Vi[t] : make_double2(0, 0);
        }
#pragma unroll
        for (int u = 0; u < PER; ++u) acc[p] = cfma(cconj(vv[u]), wv[u], acc[p]);
      } else if (i + p == nd) {
#pragma unroll
        for (int u = 0; u < PER; ++u) acc[p].x = fma(wv[u].x, wv[u].x, fma(wv[u].y, wv[u].y, acc[p].x));
      }
    }
    const double v = warp_sum2(acc[0], acc[1], lane);
    if ((lane & 7) == 0) red[warp][2 * i + (lane >> 3)] = v;
  }
  __syncthreads();
  if (tid < 2 * nout) {
    double sum = red[0][tid];
    for (int q = 1; q < kDotThreads / 32; ++q) sum += red[q][tid];
    reinterpret_cast<double*>(g.partial)[(((size_t)sys * (kMaxDot + 1) + (tid >> 1)) * nblk + blockIdx.x) * 2 + (tid & 1)] = sum;
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&g.cnt[sys], 1) == nblk - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double2* out = pass == kPassDots2 ? g.h2 : pass == kPassApply ? g.h1 : nullptr;
  double2* norm = (pass == kPassApply ? g.e2 : g.hn) + sys;
  for (int o = warp; o < nout; o += kDotThreads / 32) {   // warp adds outputs o, o + 8, ...: lane-strided, then a shuffle tree
    const double2* p = g.partial + ((size_t)sys * (kMaxDot + 1) + o) * nblk;
    double2 sum = make_double2(0, 0);
    for (int b = lane; b < nblk; b += 32) sum = cadd(sum, __ldcg(p + b));
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) {
      sum.x += __shfl_xor_sync(0xffffffffu, sum.x, q);
      sum.y += __shfl_xor_sync(0xffffffffu, sum.y, q);
    }
    if (lane == 0) {
      if (o < nd) out[(size_t)sys * kMaxDot + o] = sum;
      else *norm = sum;
    }
  }
  if (tid == 0) g.cnt[sys] = 0;
  __syncthreads();
  if (tid != 0) return;
  if (begin) {
    start_system(g, sys, norm->x, pass == kPassStart);
    if (sys == 0) *g.err_out = *g.err;
  } else if (project) {
    const double2* h = g.h1 + (size_t)sys * kMaxDot;
    const double hn2 = norm->x, en2 = g.e2[sys].x;         // after and before this projection
    const double hn = hn2 > 0.0 ? sqrt(hn2) : 0.0, en = en2 > 0.0 ? sqrt(en2) : 0.0;
    // the rounding that the vector carries into its normalised form: of v_j's size in the first projection,
    // of the vector's own in the second
    const double u = 2.220446049250313e-16 * (pass == kPassProj ? 1.0 : en);
    const double loss = hn > 0.0 ? (g.loss[sys] * en + u) / hn : 0.0;
    if (pass == kPassProj && loss > kMaxLoss && g.second) {
      g.again[sys] = 1;                   // the Givens update waits for the second projection
      g.reorth[sys] = 1;
      g.e2[sys] = make_double2(hn2, 0.0);
      return;
    }
    g.again[sys] = 0;
    finish_column(g, sys, h, pass == kPassProj ? nullptr : g.h2 + (size_t)sys * kMaxDot, hn2);
    g.loss[sys] = loss;
    if (loss > kMaxLoss) {
      g.active[sys] = 0;
      g.reorth[sys] = 1;
    }
  }
}

}  // namespace

void gm_solve(const double2* H, const double2* g, int nsys, int m, const int* njs, double2* ny_out,
              cudaStream_t s) {
  gm_solve_kernel<<<(nsys + 63) / 64, 64, 0, s>>>(H, g, nsys, m, njs, ny_out);
}
void gm_scale(double2* dst, const double2* src, const double* scale, long long n, int nsys, cudaStream_t s) {
  scale_vec_kernel<<<dim3(grid_for(n), nsys), 256, 0, s>>>(dst, src, scale, n);
}
// Entries per thread: eight, but few enough that the CTAs still cover the SMs three times over.
static int arnoldi_per(long long n, int nsys, int nsm) {
  int per = 8;
  while (per > 1 && (n + kDotThreads * per - 1) / (kDotThreads * per) * nsys < 3LL * nsm) per /= 2;
  return per;
}
long long arnoldi_partials(long long n, int nsys, int nsm) {
  const int per = arnoldi_per(n, nsys, nsm);
  return (long long)nsys * (kMaxDot + 1) * ((n + kDotThreads * per - 1) / (kDotThreads * per));
}
void launch_arnoldi(const ArnoldiStep& g, int nsys, int pass, cudaStream_t s) {
  const long long n = (long long)g.C.nx * g.C.ny;
  const int per = arnoldi_per(n, nsys, g.nsm);
  const dim3 grid((unsigned)((n + kDotThreads * per - 1) / (kDotThreads * per)), nsys);
  switch (per) {
    case 8: arnoldi_kernel<8><<<grid, kDotThreads, 0, s>>>(g, pass); break;
    case 4: arnoldi_kernel<4><<<grid, kDotThreads, 0, s>>>(g, pass); break;
    case 2: arnoldi_kernel<2><<<grid, kDotThreads, 0, s>>>(g, pass); break;
    default: arnoldi_kernel<1><<<grid, kDotThreads, 0, s>>>(g, pass); break;
  }
}

// ---------------------------------------------------------------------------
// Objective (mode overlap), adjoint source and pixel gradient.
// ---------------------------------------------------------------------------
namespace {

__global__ void overlap_kernel(const double2* __restrict__ x, long long N, int ny, const int* cols,
                               const double2* __restrict__ gline, double2* o) {
  __shared__ double2 red[8];
  const int sys = blockIdx.x;
  const int col = cols[sys];
  if (col < 0 || (long long)(col + 1) * ny > N) {   // monitor column outside the grid
    if (threadIdx.x == 0) o[sys] = make_double2(NAN, NAN);
    return;
  }
  const double2* X = x + (size_t)sys * N + (size_t)col * ny;
  const double2* G = gline + (size_t)sys * ny;
  double2 acc = make_double2(0, 0);
  for (int j = threadIdx.x; j < ny; j += blockDim.x) acc = cfma(G[j], X[j], acc);
  for (int off = 16; off > 0; off >>= 1) {
    acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
    acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double2 s = make_double2(0, 0);
    for (int q = 0; q < 8; ++q) s = cadd(s, red[q]);
    o[sys] = s;
  }
}

// F = sum_q w_q |o_q|^2, or with targets t_q the squared transmission error
// F = sum_q w_q (|o_q|^2 - t_q)^2 (summed in system order by one thread)
__global__ void objective_kernel(const double2* o, const double* weight, const double* target, int nsys, double* F) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double s = 0;
  for (int q = 0; q < nsys; ++q) {
    const double p = o[q].x * o[q].x + o[q].y * o[q].y;
    const double wt = weight ? weight[q] : 1.0;
    if (target) {
      const double d = p - target[q];
      s += wt * d * d;
    } else {
      s += wt * p;
    }
  }
  *F = s;
}

// (dF/dE)^T on the monitor column (Wirtinger derivative, E* held fixed):
// w conj(o) g for F = w |o|^2, and 2 w (|o|^2 - t) conj(o) g for F = w (|o|^2 - t)^2
__global__ void adjoint_source_kernel(const double2* o, const double* weight, const double* target, long long N,
                                      int ny, const int* cols, const double2* __restrict__ gline, double2* badj) {
  const int sys = blockIdx.y;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= ny || cols[sys] < 0 || (long long)(cols[sys] + 1) * ny > N) return;
  double wt = weight ? weight[sys] : 1.0;
  if (target) wt *= 2.0 * (o[sys].x * o[sys].x + o[sys].y * o[sys].y - target[sys]);
  const double2 oc = make_double2(wt * o[sys].x, -wt * o[sys].y);
  badj[(size_t)sys * N + (size_t)cols[sys] * ny + j] = cmul(oc, gline[(size_t)sys * ny + j]);
}

__global__ void grad_kernel(const double2* __restrict__ xf, const double2* __restrict__ xa, long long N, int ny,
                            int x0, int y0, int w, int h, int n_omega, int nrhs, const double* k0dx2,
                            const double* weight, double* grad, int accumulate) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)w * h) return;
  const int i = (int)(t / h), j = (int)(t - (long long)i * h);
  const size_t cell = (size_t)(x0 + i) * ny + y0 + j;
  double acc = 0;
  for (int om = 0; om < n_omega; ++om)
    for (int r = 0; r < nrhs; ++r) {
      const size_t sys = (size_t)om * nrhs + r;
      const double2 p = cmul(xa[sys * N + cell], xf[sys * N + cell]);
      acc += (weight ? weight[sys] : 1.0) * 2.0 * k0dx2[om] * p.x;
    }
  grad[t] = accumulate ? grad[t] + acc : acc;
}

}  // namespace

void launch_objective(const double2* x, long long N, int ny, const int* cols, const double2* gline,
                      const double* weight, const double* target, int nsys, double2* o, double* F, double2* badj,
                      cudaStream_t s) {
  overlap_kernel<<<nsys, 256, 0, s>>>(x, N, ny, cols, gline, o);
  objective_kernel<<<1, 32, 0, s>>>(o, weight, target, nsys, F);
  if (badj) {
    cudaMemsetAsync(badj, 0, sizeof(double2) * (size_t)nsys * N, s);
    adjoint_source_kernel<<<dim3((ny + 255) / 256, nsys), 256, 0, s>>>(o, weight, target, N, ny, cols, gline,
                                                                        badj);
  }
}

void launch_grad(const double2* xf, const double2* xa, long long N, int ny, int x0, int y0, int w, int h,
                 int n_omega, int nrhs, const double* k0dx2, const double* weight, double* grad, int accumulate,
                 cudaStream_t s) {
  const long long n = (long long)w * h;
  if (n <= 0) return;
  grad_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(xf, xa, N, ny, x0, y0, w, h, n_omega, nrhs, k0dx2,
                                                          weight, grad, accumulate);
}

}  // namespace fdfd
