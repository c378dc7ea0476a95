// Launchers of the resident FFT steps (kernels in qf_fft_res.cuh).
#include "qf_fft_res.cuh"

namespace qf {

template <int N, typename K>
static cudaError_t res_launch(K kern, int members, cudaStream_t st, const void* arg) {
  using G = ResG<N>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(G::C, members);
  cfg.blockDim = dim3(G::THREADS);
  cfg.dynamicSmemBytes = G::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = G::C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  void* args[] = {const_cast<void*>(arg)};
  return cudaLaunchKernelExC(&cfg, (const void*)kern, args);
}

// Shared-memory and cluster limits of every variant of size N; whether the device can hold a
// cluster at all (16 blocks exceed the portable 8).
template <int N>
static bool res_setup() {
  using G = ResG<N>;
  const void* k[] = {(const void*)fft_res_kernel<N, true, true>, (const void*)fft_res_kernel<N, true, false>,
                     (const void*)fft_res_kernel<N, false, true>, (const void*)fft_res_kernel<N, false, false>,
                     (const void*)fft_res_static_kernel<N, true, true>, (const void*)fft_res_static_kernel<N, true, false>,
                     (const void*)fft_res_static_kernel<N, false, true>, (const void*)fft_res_static_kernel<N, false, false>};
  bool ok = true;
  for (const void* f : k) {
    ok = ok && cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::SMEM) == cudaSuccess;
    ok = ok && cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(G::C);
    cfg.blockDim = dim3(G::THREADS);
    cfg.dynamicSmemBytes = G::SMEM;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = G::C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    ok = ok && cudaOccupancyMaxActiveClusters(&clusters, f, &cfg) == cudaSuccess && clusters > 0;
  }
  if (!ok) cudaGetLastError();  // (a refusal above is an answer, not an error)
  return ok;
}
template <int N>
static bool res_ready() {
  static PerDevice done;
  return done.ready(current_device(), res_setup<N>);
}

#define QF_RES_CASES QF_CASE(8) QF_CASE(12) QF_CASE(16) QF_CASE(24) QF_CASE(32)

int fft_res_blocks(int n) {
  switch (n) {
#define QF_CASE(NN) \
  case NN:          \
    return res_ready<NN>() ? ResG<NN>::C : 0;
    QF_RES_CASES
#undef QF_CASE
    default:
      return 0;
  }
}

cudaError_t launch_fft_res(int n, const ResGroup& g, bool v_real, bool reduce, cudaStream_t st) {
  if (g.count < 1 || g.count > kGroupMax || fft_res_blocks(n) == 0) return cudaErrorInvalidValue;
  switch (n) {
#define QF_CASE(NN)                                                                                          \
  case NN:                                                                                                   \
    return res_launch<NN>(v_real ? (reduce ? fft_res_kernel<NN, true, true> : fft_res_kernel<NN, true, false>) \
                                 : (reduce ? fft_res_kernel<NN, false, true> : fft_res_kernel<NN, false, false>), \
                          g.count, st, &g);
    QF_RES_CASES
#undef QF_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_fft_res_static(int n, const ResStatic& g, bool v_real, bool reduce, cudaStream_t st) {
  if (fft_res_blocks(n) == 0) return cudaErrorInvalidValue;
  switch (n) {
#define QF_CASE(NN)                                                                                                  \
  case NN:                                                                                                           \
    return res_launch<NN>(v_real ? (reduce ? fft_res_static_kernel<NN, true, true> : fft_res_static_kernel<NN, true, false>) \
                                 : (reduce ? fft_res_static_kernel<NN, false, true> : fft_res_static_kernel<NN, false, false>), \
                          1, st, &g);
    QF_RES_CASES
#undef QF_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

__global__ void bounded_wait_probe(int* err, unsigned spin) {
  __shared__ alignas(8) unsigned long long bar;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"((unsigned)__cvta_generic_to_shared(&bar)) : "memory");
    res_expect(&bar, 16);  // no copy follows
  }
  __syncthreads();
  const bool done = res_wait(&bar, 0, true, spin);
  if (__syncthreads_or(done) == 0 && threadIdx.x == 0) atomicExch(err, 1);
}
cudaError_t launch_bounded_wait_probe(int* err, unsigned spin, cudaStream_t st) {
  bounded_wait_probe<<<1, 32, 0, st>>>(err, spin);
  return cudaGetLastError();
}

}  // namespace qf
