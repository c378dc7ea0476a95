// FDTD kinetic step (Eq. HK0) fused with the imaginary-time update: launchers of the
// kernels in qf_stencil_flat.cuh (one step) and qf_stencil_tb.cuh (two steps).
//
// (H_K^(0) psi)(r) = -1/(2 m a^2) sum over the six neighbours of (psi(nbr) - psi(r)), with
// psi pinned to 0 on the Dirichlet planes (any index 0; a neighbour index N wraps onto
// the plane 0).  One pass: read psi and V, write psi' = s (coef_A psi - coef_B dtau H psi)
// into the other buffer, plus the FP64 partial sums of <psi|psi>, <psi|H_K psi>,
// <psi|V psi> on check steps.  A lone lattice is a group of one, so it runs the same
// code alone and inside a batch.
#include "qf_stencil_tb.cuh"

namespace qf {

// Partial-sum rows of one lattice's launch.
int stencil_blocks(int n) { return stencil_member_blocks(n); }

template <typename R>
cudaError_t launch_stencil(const StencilGroup<R>& g, cudaStream_t st) {
  if (g.count < 1 || g.count > kGroupMax) return cudaErrorInvalidValue;
  // the block table: member i's blocks follow member i-1's
  StencilGroup<R> gl = g;
  long long total = 0;
  for (int i = 0; i < g.count; ++i) {
    if (g.nm[i] < 2) return cudaErrorInvalidValue;
    gl.start[i] = (int)total;
    total += stencil_member_blocks(g.nm[i]);
  }
  if (total > (1LL << 30)) return cudaErrorInvalidValue;
  gl.start[g.count] = (int)total;
  stencil_flat_kernel<R><<<(unsigned)total, kFlatThreads, 0, st>>>(gl);
  return cudaGetLastError();
}

// Two steps for every member of g (any sizes, one kind of potential) in one launch.
cudaError_t launch_stencil_tb(const StencilTbGroup& g, cudaStream_t st) {
  if (g.count < 1 || g.count > kGroupMax) return cudaErrorInvalidValue;
  StencilTbGroup gl = g;
  long long total = 0;
  for (int i = 0; i < g.count; ++i) {
    const StencilTbArgs& m = g.m[i];
    if (m.n < 2 || m.nzb < 1 || m.nzb > m.n || m.v_real != g.m[0].v_real) return cudaErrorInvalidValue;
    gl.start[i] = (int)total;
    total += stencil_tb_member_blocks(m.n, m.nzb);
  }
  if (total > (1LL << 30)) return cudaErrorInvalidValue;
  gl.start[g.count] = (int)total;
  // the L2 prefetch pays for its instructions only where psi and V do not stay in L2 (N = 192:
  // 44.5 / 43.3 us without / with it, N = 250: 89.0 / 86.8, N = 384: 291 / 274, N = 128: 16.9 / 17.0)
  bool pre = true;
  for (int i = 0; i < g.count; ++i) pre = pre && g.m[i].n >= 192;
  const unsigned nb = (unsigned)total;
  if (g.m[0].v_real) {
    if (pre) stencil_tb_kernel<true, true><<<nb, 32, 0, st>>>(gl);
    else stencil_tb_kernel<true, false><<<nb, 32, 0, st>>>(gl);
  } else {
    if (pre) stencil_tb_kernel<false, true><<<nb, 32, 0, st>>>(gl);
    else stencil_tb_kernel<false, false><<<nb, 32, 0, st>>>(gl);
  }
  return cudaGetLastError();
}

template cudaError_t launch_stencil<float>(const StencilGroup<float>&, cudaStream_t);
template cudaError_t launch_stencil<double>(const StencilGroup<double>&, cudaStream_t);

}  // namespace qf
