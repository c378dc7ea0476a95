// Launchers of the line form's passes (kernels in qf_fft_line.cuh): pass 4 (x inverse and update) and,
// at N = 192, pass 2 (z) of the four-pass step.
#include "qf_fft_line.cuh"

namespace qf {

template <int N>
static bool line_setup() {
  using L = LineG<N>;
  const void* x[] = {(const void*)line_x_kernel<N, true, false, true>, (const void*)line_x_kernel<N, true, true, true>,
                     (const void*)line_x_kernel<N, false, false, true>, (const void*)line_x_kernel<N, false, true, true>};
  for (const void* f : x) cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::SMEM_X);
  if constexpr (N == 192)
    cudaFuncSetAttribute((const void*)line_z_kernel<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::SMEM_Z);
  return true;
}

template <int N>
static cudaError_t line_pass(int pass, const FftGroup<float>& g, cudaStream_t st) {
  using L = LineG<N>;
  static PerDevice done;
  done.ready(current_device(), line_setup<N>);
  const dim3 gz(L::Z_BLOCKS, g.count), gx(L::X_BLOCKS, g.count);
  constexpr int tx = 32 * L::X_WARPS;
  if (pass == 2) {
    if constexpr (N == 192) line_z_kernel<N><<<gz, L::Z_THREADS, L::SMEM_Z, st>>>(g);
    else return cudaErrorInvalidValue;
  } else {
    const bool sums = g.a[0].reduce != 0;
    if (g.a[0].v_real) {
      if (sums) line_x_kernel<N, true, true, true><<<gx, tx, L::SMEM_X, st>>>(g);
      else line_x_kernel<N, true, false, true><<<gx, tx, L::SMEM_X, st>>>(g);
    } else {
      if (sums) line_x_kernel<N, false, true, true><<<gx, tx, L::SMEM_X, st>>>(g);
      else line_x_kernel<N, false, false, true><<<gx, tx, L::SMEM_X, st>>>(g);
    }
  }
  return cudaGetLastError();
}

bool line_supported(int n) { return n == 192 || n == 512; }
bool line_has_pass(int n, int pass) { return pass == 4 || (pass == 2 && n == 192); }
int line_final_blocks(int n) { return n == 192 ? LineG<192>::X_BLOCKS : n == 512 ? LineG<512>::X_BLOCKS : 0; }

cudaError_t launch_line_pass(int n, int pass, const FftGroup<float>& g, cudaStream_t st) {
  if (g.count < 1 || g.count > kGroupMax || (pass != 2 && pass != 4)) return cudaErrorInvalidValue;
  if (n == 192) return line_pass<192>(pass, g, st);
  if (n == 512) return line_pass<512>(pass, g, st);
  return cudaErrorInvalidValue;
}

}  // namespace qf
