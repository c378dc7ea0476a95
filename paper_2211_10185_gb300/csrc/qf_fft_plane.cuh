// Two-pass imaginary-time FFT step for complex-FP32 lattices whose z-plane fits one block's
// shared memory (Eqs. HK1-HK3 and the update of Sec. 2), sm_103a.
//
// A steady-state step is two launches over the scratch field S (natural order, transformed
// along y and x):
//   Z  z forward, T(k), z inverse, on columns;
//   P  one block per z-plane: y inverse, x inverse -> H_K psi, the update of psi (and the FP64
//      check sums), then x forward and y forward of psi_{t+1} for the next step.
// A (first step of a run) is P's forward half on psi.
//
// A transform of N = 4 E points runs on 4 lanes of a warp, lane g holding the elements i = g + 4 m:
// an E-point transform over m in registers, the twiddle wN^{g k}, one exchange among the four
// lanes through the line's own place in shared memory (warp synchronisation only), and a
// 4-point transform over g.  The outputs g + 4 m land on the lane that holds those inputs, in
// either direction, so T(k) and the update happen in registers and nothing is reordered
// between a transform and the next along the same axis.
//
// Shared memory holds the plane as [y][x] at idx = NP y + 4 ((y >> 1) & 1) + x, NP = 8 (mod 16): a
// half-warp of 8 columns x 2 rows or of 4 rows x 4 neighbouring x covers all banks once, also
// in the exchange, whose element (g, k) lies at 16 (k >> 2) + 4 g + (g ^ (k & 3)).
//
// What bounds it: the latency of a block's four transforms with 6-12 warps per SM, on N of the 152
// SMs in P (the four-pass form: that of four launches, 11.6-25 us a step).  One step with
// Eq. HK2 (of 64 with a check), before and now: N = 48: 12.8 / 5.8 us, 64: 11.6-13 / 8.7 (Eq. HK3
// 9.5), 96: 25.1 / 17.9 (not the default there).  N = 128 took 40 us so (32 elements a thread, one block of 16
// warps per SM, spills) against 25.7 in the split form.
#pragma once
#include "qf_fft_reg.cuh"

namespace qf {

template <int N>
struct PlaneG {
  static_assert(N % 16 == 0, "lines of 4 lanes x E elements, E a multiple of 4");
  static constexpr int E = N / 4;
  static constexpr int TWP = E + 2;  // pitch of the twiddle rows [g][k]: the four lanes' reads spread over banks
  static constexpr int NP = (N % 16 == 8 ? N : N + 8);
  static constexpr int PLANE = N * NP;
  static constexpr int P_THREADS = 4 * N;
  static constexpr size_t SMEM_P = (size_t)(4 * TWP + PLANE) * 8 + 32 * kNumSums * 8;
  // Z: warps of 8 columns
  static constexpr int Z_WARPS = N % 32 == 0 ? 4 : 2;
  static constexpr int Z_BLOCKS = N * N / (8 * Z_WARPS);
  static constexpr size_t SMEM_Z = (size_t)(4 * TWP + Z_WARPS * 8 * N) * 8 + N * 4 + 32 * kNumSums * 8;
};

// wN^{g k} (forward), g < 4, k < E
template <int N>
struct PlaneTable {
  cpx<float> w[N];
  constexpr PlaneTable() : w() {
    for (int g = 0; g < 4; ++g)
      for (int k = 0; k < N / 4; ++k) {
        const RcTwiddle t = rc_twiddle(g * k % N, N);
        w[g * (N / 4) + k].x = t.c;
        w[g * (N / 4) + k].y = -t.s;
      }
  }
};
template <int N>
__device__ const PlaneTable<N> plane_table = PlaneTable<N>();

template <int N>
__device__ __forceinline__ void plane_twiddles(cpx<float>* tw_s, int threads) {
  constexpr int E = PlaneG<N>::E;
  for (int i = threadIdx.x; i < N; i += threads) tw_s[(i / E) * PlaneG<N>::TWP + i % E] = plane_table<N>.w[i];
}

// One line on its four lanes: v[m] = element g + 4 m, before and after; at(i) is the place of
// element i, used by these lanes only.
template <int N, bool INV, typename F>
__device__ __forceinline__ void plane_line(cpx<float> (&v)[N / 4], int g, const cpx<float>* tw_s, F at) {
  constexpr int E = N / 4;
  rc_dft<E, INV, 1>(v);
  const float4* tw = reinterpret_cast<const float4*>(tw_s + g * PlaneG<N>::TWP);
#pragma unroll
  for (int k = 0; k < E; k += 2) {
    const float4 w = tw[k / 2];
    const cpx<float> w0 = mk<float>(w.x, w.y), w1 = mk<float>(w.z, w.w);
    v[k] = INV ? cmulc<float>(v[k], w0) : cmul<float>(v[k], w0);
    v[k + 1] = INV ? cmulc<float>(v[k + 1], w1) : cmul<float>(v[k + 1], w1);
  }
  __syncwarp();  // the line's earlier reads are done
#pragma unroll
  for (int k = 0; k < E; ++k) *at(16 * (k >> 2) + 4 * g + (g ^ (k & 3))) = v[k];
  __syncwarp();
#pragma unroll
  for (int m = 0; m < E / 4; ++m) {  // k = g + 4 m: outputs k + E q
    cpx<float> u[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) u[h] = *at(16 * m + 4 * h + (h ^ g));
    rc_dft4<INV>(u[0], u[1], u[2], u[3]);
#pragma unroll
    for (int q = 0; q < 4; ++q) v[m + (E / 4) * q] = u[q];
  }
}

template <int N>
__device__ __forceinline__ int plane_idx(int y, int x) {
  return y * PlaneG<N>::NP + 4 * ((y >> 1) & 1) + x;
}

// Programmatic dependent launch (as in the two-pass step of N = 128 and 256): wait for the
// kernel before, then let the next one start.
__device__ __forceinline__ void plane_dependency() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

__device__ __forceinline__ cpx<float> plane_ld_early(const cpx<float>* p) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  cpx<float> c;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(c.x), "=f"(c.y) : "l"(w));
  return c;
}

// Forward half: x lines in v -> plane, y forward, S.
template <int N>
__device__ __forceinline__ void plane_forward(cpx<float> (&v)[N / 4], int xg, int line, int cg, int col, int z,
                                              const cpx<float>* tw_s, cpx<float>* plane, cpx<float>* S) {
  constexpr int E = N / 4;
  auto x_at = [&](int i) { return plane + plane_idx<N>(line, i); };
  auto y_at = [&](int i) { return plane + plane_idx<N>(i, col); };
  plane_line<N, false>(v, xg, tw_s, x_at);
  __syncwarp();
#pragma unroll
  for (int m = 0; m < E; ++m) *x_at(xg + 4 * m) = v[m];
  __syncthreads();
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = *y_at(cg + 4 * m);
  plane_line<N, false>(v, cg, tw_s, y_at);
#pragma unroll
  for (int m = 0; m < E; ++m) S[((long long)z * N + cg + 4 * m) * N + col] = v[m];
}

// A: psi (or src) -> S; with SUMS also <src|src> and <src|V src> into partial row blockIdx.x.
template <int N, bool SUMS>
__global__ void __launch_bounds__(PlaneG<N>::P_THREADS) plane_a_kernel(const __grid_constant__ FftGroup<float> gr) {
  using G = PlaneG<N>;
  constexpr int E = G::E;
  const FftPassArgs<float>& a = gr.a[blockIdx.y];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<float>* tw_s = reinterpret_cast<cpx<float>*>(smem_raw);
  cpx<float>* plane = tw_s + 4 * G::TWP;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, z = blockIdx.x;
  const int xg = lane & 3, line = warp * 8 + (lane >> 2), cg = lane >> 3, col = warp * 8 + (lane & 7);
  const cpx<float>* __restrict__ src = a.src ? a.src : a.psi;
  const long long row = ((long long)z * N + line) * N + xg;
  plane_twiddles<N>(tw_s, G::P_THREADS);
  cpx<float> v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = src[row + 4 * m];
  if constexpr (SUMS) {
    CheckSums<float> cs;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      const cpx<float> w = a.v_real ? mk<float>(reinterpret_cast<const float*>(a.v)[row + 4 * m], 0.f)
                                    : reinterpret_cast<const cpx<float>*>(a.v)[row + 4 * m];
      cs.add(v[m], mk<float>(0.f, 0.f), w);
    }
    double acc[kNumSums];
    cs.to(acc);
    block_sum_store<kNumSums>(acc, reinterpret_cast<double*>(plane + G::PLANE), a.partials + (long long)z * kPartialStride);
  }
  __syncthreads();
  plane_forward<N>(v, xg, line, cg, col, z, tw_s, plane, a.data);
}

// Z: columns of S in place.  With SUMS (energy of a field that is not stepped): after the
// forward transform <v|H_K v> = sum_k T(k)/N^3 |v^(k)|^2 (Parseval) into partial row row0 +
// blockIdx.x, and nothing is written back.
template <int N, bool SUMS>
__global__ void __launch_bounds__(32 * PlaneG<N>::Z_WARPS) plane_z_kernel(const __grid_constant__ FftGroup<float> gr,
                                                                          int row0) {
  using G = PlaneG<N>;
  constexpr int E = G::E;
  const FftPassArgs<float>& a = gr.a[blockIdx.y];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<float>* tw_s = reinterpret_cast<cpx<float>*>(smem_raw);
  cpx<float>* buf = tw_s + 4 * G::TWP;  // per warp: [z][8 columns]
  float* sym = reinterpret_cast<float*>(buf + G::Z_WARPS * 8 * N);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 3, c = ((int)blockIdx.x * G::Z_WARPS + warp) * 8 + (lane & 7);
  const int kx = c % N, ky = c / N;
  plane_twiddles<N>(tw_s, 32 * G::Z_WARPS);
  for (int i = tid; i < N; i += 32 * G::Z_WARPS) sym[i] = a.symbol[i];
  plane_dependency();
  cpx<float>* __restrict__ S = a.data + c;
  cpx<float> v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = S[(long long)(g + 4 * m) * N * N];
  __syncthreads();
  cpx<float>* col = buf + warp * 8 * N + (lane & 7);
  auto at = [&](int i) { return col + 8 * i; };
  plane_line<N, false>(v, g, tw_s, at);
  const float sxy = sym[kx] + sym[ky];
  if constexpr (SUMS) {
    CheckSums<float> cs;
#pragma unroll
    for (int m = 0; m < E; ++m)
      cs.add(v[m], cscale<float>(v[m], kin_mult_acc(a.kinetic, sxy, sym[g + 4 * m], a.tcoef, a.am2)),
             mk<float>(0.f, 0.f));
    double acc[kNumSums];
    cs.to(acc);
    acc[0] = acc[3] = acc[4] = 0.0;  // norm and potential terms come from A
    block_sum_store<kNumSums>(acc, reinterpret_cast<double*>(sym + N),
                              a.partials + (long long)(row0 + blockIdx.x) * kPartialStride);
    return;
  }
  const float am = sqrtf(a.am2);
#pragma unroll
  for (int m = 0; m < E; ++m)
    v[m] = cscale<float>(v[m], kin_mult_rest(a.kinetic, sxy, sym[g + 4 * m], a.tcoef, a.am2, am));
  plane_line<N, true>(v, g, tw_s, at);
#pragma unroll
  for (int m = 0; m < E; ++m) S[(long long)(g + 4 * m) * N * N] = v[m];
}

// P: S -> update of psi (and sums) -> S of psi_{t+1}.
template <int N, bool VREAL, bool SUMS>
__global__ void __launch_bounds__(PlaneG<N>::P_THREADS) plane_p_kernel(const __grid_constant__ FftGroup<float> gr) {
  using G = PlaneG<N>;
  constexpr int E = G::E;
  const FftPassArgs<float>& a = gr.a[blockIdx.y];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<float>* tw_s = reinterpret_cast<cpx<float>*>(smem_raw);
  cpx<float>* plane = tw_s + 4 * G::TWP;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, z = blockIdx.x;
  const int xg = lane & 3, line = warp * 8 + (lane >> 2), cg = lane >> 3, col = warp * 8 + (lane & 7);
  const long long row = ((long long)z * N + line) * N + xg;
  plane_twiddles<N>(tw_s, G::P_THREADS);
  // psi and V of the thread's sites x = xg + 4 m of its line, and the scale, are read ahead of the
  // dependency (behind it a step takes 6.3 us instead of 5.8 at N = 48, 9.3 instead of 8.5 at 64).  The
  // Z pass that this block may overlap writes none of them.  V is constant.  What wrote psi and
  // the scale (P of the step before, the check's finishing sums) came before that Z pass, whose
  // blocks let this launch start only behind their own griddepcontrol.wait, that is with those
  // kernels complete and their writes performed in global memory.  This grid has not waited for
  // them itself, so nothing promises that a first-level cache holds no older copy: these
  // loads are relaxed at GPU scope, which L2 serves.
  cpx<float> psi[E], vv[VREAL ? 1 : E];
  float vr[VREAL ? E : 1];
#pragma unroll
  for (int m = 0; m < E; ++m) {
    psi[m] = plane_ld_early(a.psi + row + 4 * m);
    if constexpr (VREAL) vr[m] = reinterpret_cast<const float*>(a.v)[row + 4 * m];
    else vv[m] = reinterpret_cast<const cpx<float>*>(a.v)[row + 4 * m];
  }
  double scale;
  asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];" : "=d"(scale) : "l"(a.scale) : "memory");
  const float sc = float(scale);
  plane_dependency();
  cpx<float>* __restrict__ S = a.data;
  cpx<float> v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = S[((long long)z * N + cg + 4 * m) * N + col];
  __syncthreads();
  {
    auto y_at = [&](int i) { return plane + plane_idx<N>(i, col); };
    plane_line<N, true>(v, cg, tw_s, y_at);
    __syncwarp();
#pragma unroll
    for (int m = 0; m < E; ++m) *y_at(cg + 4 * m) = v[m];
  }
  __syncthreads();
  auto x_at = [&](int i) { return plane + plane_idx<N>(line, i); };
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = *x_at(xg + 4 * m);
  plane_line<N, true>(v, xg, tw_s, x_at);
  // v = H_K psi (1/N^3 inside T)
  if (a.kinetic == KIN_FFT_REL) {
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = rest_mass(psi[m], v[m], a.t0, a.t0_lo);
  }
  if constexpr (SUMS) {
    CheckSums<float> cs;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      if constexpr (VREAL) cs.add(psi[m], v[m], mk<float>(vr[m], 0.f));
      else cs.add(psi[m], v[m], vv[m]);
    }
    double acc[kNumSums];
    cs.to(acc);
    block_sum_store<kNumSums>(acc, reinterpret_cast<double*>(plane + G::PLANE), a.partials + (long long)z * kPartialStride);
  }
#pragma unroll
  for (int m = 0; m < E; ++m) {
    if constexpr (VREAL) v[m] = reg_update(psi[m], v[m], vr[m], a.half_dtau, a.dtau, a.dtau_lo, sc);
    else v[m] = reg_update(psi[m], v[m], vv[m], a.half_dtau, a.dtau, a.dtau_lo, sc);
    a.psi[row + 4 * m] = v[m];
  }
  plane_forward<N>(v, xg, line, cg, col, z, tw_s, plane, S);
}

}  // namespace qf
