// Launches of the dataflow sweeps (flow.cuh): this file holds the dispatch and the complex64 kernels of
// small problems; sweep_wide.cu those of large ones, sweep_f64.cu the complex128 kernels.
#include "flow.cuh"

namespace fdfd {

FDFD_FLOW_SHAPE(narrow1, kFlowThreads, 1, float2, 1)
FDFD_FLOW_SHAPE(narrow2, kFlowThreads, 1, float2, 2)
#define FDFD_FLOW_DECL(NAME)                                                                                  \
  void flow_launch_##NAME(const SolveLaunch& a, int sweep, const FlowQueue& q, const FlowShape& sh, int grid, \
                          const double2* in, double2* out, cudaStream_t s);                                   \
  int flow_blocks_##NAME(int smem);                                                                           \
  cudaError_t flow_init_##NAME();
FDFD_FLOW_DECL(wide1) FDFD_FLOW_DECL(wide2) FDFD_FLOW_DECL(f64)

// One wait on *flag >= 1 (nothing sets it) by one thread: exercises the
// bounded wait of the dataflow sweep, which must give up, set *err and return.
__global__ void wait_probe_kernel(const int* flag, int* err) {
  if (threadIdx.x == 0) (void)wait_ge(flag, 1, err);
}

cudaError_t launch_wait_probe(const int* flag, int* err, cudaStream_t s) {
  wait_probe_kernel<<<1, 32, 0, s>>>(flag, err);
  return cudaGetLastError();
}

// A warp per record: the record, its n grid cells, its n children's slots, zeros up to 16 bytes.  Written here from
// the plan's arrays, which are on the device anyway: as a host loop and an upload it took a twelfth of the
// symbolic phase (1200 x 1200: 76 of 915 ms, and 40 MB).
__global__ void meta_kernel(const SweepFront* __restrict__ fronts, int n, const size_t* __restrict__ moff,
                            const int* __restrict__ idx, const int* __restrict__ inv, unsigned char* meta) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= n || moff[i + 1] == moff[i]) return;        // (not packed)
  const SweepFront& d = fronts[i];
  const int nn = d.k + d.m, words = (int)(moff[i + 1] - moff[i]) / 4, head = (int)sizeof(SweepFront) / 4;
  unsigned* out = reinterpret_cast<unsigned*>(meta + moff[i]);
  const unsigned* rec = reinterpret_cast<const unsigned*>(&d);
  for (int j = lane; j < words; j += 32) {
    const int t = j - head, u = t - nn;
    unsigned v = 0;
    if (t < 0) v = rec[j];
    else if (u < 0) v = (unsigned)idx[d.idx_off + t];
    else if (u < nn)
      v = (d.inv0 >= 0 ? (unsigned)inv[d.inv0 + u] & 0xffffu : 0xffffu) |
          (d.inv1 >= 0 ? (unsigned)inv[d.inv1 + u] & 0xffffu : 0xffffu) << 16;
    out[j] = v;
  }
}

cudaError_t launch_meta(const SweepFront* fronts, int n, const size_t* moff, const int* idx, const int* inv,
                        unsigned char* meta, cudaStream_t s) {
  constexpr int kWarps = 8;
  if (n > 0) meta_kernel<<<(n + kWarps - 1) / kWarps, 32 * kWarps, 0, s>>>(fronts, n, moff, idx, inv, meta);
  return cudaGetLastError();
}

// Right-hand sides are taken two at a time when there are two (complex64).
template <typename T>
void launch_sweep_flow(const SolveLaunch& a, int sweep, const FlowQueue& q, const FlowShape& sh, int grid,
                       const void* in, void* out, cudaStream_t s) {
  if (q.nunits <= 0) return;
  const double2* i = reinterpret_cast<const double2*>(in);
  double2* o = reinterpret_cast<double2*>(out);
  if (sizeof(T) == 16) flow_launch_f64(a, sweep, q, sh, grid, i, o, s);
  else if (sh.wide) (a.nr >= 2 ? flow_launch_wide2 : flow_launch_wide1)(a, sweep, q, sh, grid, i, o, s);
  else (a.nr >= 2 ? flow_launch_narrow2 : flow_launch_narrow1)(a, sweep, q, sh, grid, i, o, s);
}

// Persistent CTAs per SM for the given shape: the fewest over the sweeps.
int flow_blocks_per_sm(int elem_bytes, const FlowShape& sh) {
  const int smem = sh.buffers * sh.smem;
  if (elem_bytes == 16) return flow_blocks_f64(smem);
  const bool wide = sh.wide;
  const int n1 = wide ? flow_blocks_wide1(smem) : flow_blocks_narrow1(smem);
  const int n2 = wide ? flow_blocks_wide2(smem) : flow_blocks_narrow2(smem);
  return n1 < n2 ? n1 : n2;
}

cudaError_t solve_init_attributes() {
  cudaError_t e = flow_init_narrow1();
  if (e == cudaSuccess) e = flow_init_narrow2();
  if (e == cudaSuccess) e = flow_init_wide1();
  if (e == cudaSuccess) e = flow_init_wide2();
  if (e == cudaSuccess) e = flow_init_f64();
  return e;
}

template void launch_sweep_flow<float2>(const SolveLaunch&, int, const FlowQueue&, const FlowShape&, int, const void*,
                                        void*, cudaStream_t);
template void launch_sweep_flow<double2>(const SolveLaunch&, int, const FlowQueue&, const FlowShape&, int, const void*,
                                         void*, cudaStream_t);

}  // namespace fdfd
