// Launchers of the plane form of the FFT step (kernels in qf_fft_plane.cuh), with the pass
// numbers of the two-pass form: 0 A, 1 Z, 2 P; energy of a field that is not stepped: 3 A with
// sums, 4 Z forward with sums.
#include "qf_fft_plane.cuh"

namespace qf {

template <typename... KArgs, typename... Args>
static cudaError_t plane_launch(void (*kern)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t st, bool pdl,
                                Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = pdl ? 1 : 0;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <int N>
static bool plane_setup() {
  using G = PlaneG<N>;
  const void* p[] = {(const void*)plane_a_kernel<N, false>, (const void*)plane_a_kernel<N, true>,
                     (const void*)plane_p_kernel<N, true, false>, (const void*)plane_p_kernel<N, true, true>,
                     (const void*)plane_p_kernel<N, false, false>, (const void*)plane_p_kernel<N, false, true>};
  for (const void* f : p) cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM_P);
  for (const void* f : {(const void*)plane_z_kernel<N, false>, (const void*)plane_z_kernel<N, true>})
    cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM_Z);
  return true;
}

template <int N>
static cudaError_t plane_pass(int pass, const FftGroup<float>& g, cudaStream_t st) {
  using G = PlaneG<N>;
  static PerDevice done;
  done.ready(current_device(), plane_setup<N>);
  if (g.count < 1 || g.count > kGroupMax) return cudaErrorInvalidValue;
  const dim3 gp(N, g.count), gz(G::Z_BLOCKS, g.count);
  constexpr int tp = G::P_THREADS, tz = 32 * G::Z_WARPS;
  const bool vreal = g.a[0].v_real != 0, sums = g.a[0].reduce != 0;
  switch (pass) {
    case 0: return plane_launch(plane_a_kernel<N, false>, gp, tp, G::SMEM_P, st, false, g);
    case 3: return plane_launch(plane_a_kernel<N, true>, gp, tp, G::SMEM_P, st, false, g);
    case 1: return plane_launch(plane_z_kernel<N, false>, gz, tz, G::SMEM_Z, st, true, g, 0);
    case 4: return plane_launch(plane_z_kernel<N, true>, gz, tz, G::SMEM_Z, st, false, g, N);
    case 2:
      if (!g.a[0].write_psi || !g.a[0].emit_next) return cudaErrorInvalidValue;
      if (vreal) return plane_launch(sums ? plane_p_kernel<N, true, true> : plane_p_kernel<N, true, false>, gp, tp,
                                     G::SMEM_P, st, true, g);
      return plane_launch(sums ? plane_p_kernel<N, false, true> : plane_p_kernel<N, false, false>, gp, tp, G::SMEM_P, st,
                          true, g);
    default: return cudaErrorInvalidValue;
  }
}

bool plane_supported(int n) { return n == 48 || n == 64 || n == 96; }
int plane_final_blocks(int n) { return n; }
int plane_measure_blocks(int n) {
  return n + (n == 48 ? PlaneG<48>::Z_BLOCKS : n == 64 ? PlaneG<64>::Z_BLOCKS : PlaneG<96>::Z_BLOCKS);
}

cudaError_t launch_plane_pass(int n, int pass, const FftGroup<float>& g, cudaStream_t st) {
  switch (n) {
    case 48: return plane_pass<48>(pass, g, st);
    case 64: return plane_pass<64>(pass, g, st);
    case 96: return plane_pass<96>(pass, g, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace qf
