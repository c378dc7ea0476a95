// Line form of the heaviest passes of the four-pass FFT step for complex-FP32 lattices (Eqs.
// HK1-HK3 and the update of Sec. 2), sm_103a: the x pass (x inverse, update of psi, FP64 check
// sums, x forward of psi_{t+1}) of N = 192 and 512 and the z pass (z forward, T(k), z inverse)
// of N = 192.  The others are those of qf_fft_impl.cuh; the field between passes is in natural
// order.
//
// A transform of N = E G points runs on G lanes, lane g holding the elements i = g + G m: an
// E-point transform over m in registers, the twiddle wN^{g k}, one exchange through shared
// memory, E / G transforms of G points.  The outputs g + G m land on the lane that holds those
// inputs, in either direction, so T(k) and the update happen in registers.  Element (g, k) of
// an exchange lies at (k / G) G^2 + g G + (g ^ (k mod G)): no bank conflicts.
//
// x pass: the G lanes belong to one warp, so a warp goes through load, both transforms and store
// of its 32 / G lines with warp synchronisation only, and the warps of an SM overlap one
// another's loads and arithmetic (the four-pass kernel: three stages each way, a block barrier
// or two for each).  z pass: a block takes 8 neighbouring columns (64-byte segments).
//
// What bounds it: the x pass HBM and L2 (N = 512: 6.4 TB/s of its 40 bytes a site, complex V; N = 192:
// 6.1 TB/s, partly from L2).  Before and now (event-bracketed): x pass N = 192 64.4 / 41.5 us, N
// = 512 1222 / 801 us; z pass N = 192 30.8 / 28.2 us.  At N = 512 the z pass so takes 700 us
// against 580 with 8 columns x 512 threads, so it stays there.
#pragma once
#include "qf_fft_reg.cuh"

namespace qf {

template <int N>
struct LineG {
  static_assert(N == 192 || N == 512, "line form");
  static constexpr int E = N == 192 ? 24 : 32, G = N / E;
  static constexpr int TWP = E + 2;  // pitch of the twiddle rows [g][k]
  // x pass: X_WARPS warps of 32 / G lines; line pitch 8 (mod 16) elements where two lines share
  // a half-warp
  static constexpr int X_WARPS = 4, LPW = 32 / G;
  static constexpr int LP = G == 8 ? N + 8 : N;
  static constexpr int X_BLOCKS = N * N / (X_WARPS * LPW);
  static constexpr int X_PER_SM = N == 192 ? 3 : 2;
  static constexpr size_t SMEM_X = (size_t)(G * TWP + X_WARPS * LPW * LP) * 8 + 32 * kNumSums * 8;
  // z pass: 8 columns x G lanes
  static constexpr int Z_THREADS = 8 * G;
  static constexpr int Z_BLOCKS = N * N / 8;
  static constexpr size_t SMEM_Z = (size_t)(G * TWP + 8 * N) * 8 + N * 4;
};

// wN^{g k} (forward), g < G, k < E
template <int N>
struct LineTable {
  cpx<float> w[N];
  constexpr LineTable() : w() {
    for (int g = 0; g < LineG<N>::G; ++g)
      for (int k = 0; k < LineG<N>::E; ++k) {
        const RcTwiddle t = rc_twiddle(g * k % N, N);
        w[g * LineG<N>::E + k].x = t.c;
        w[g * LineG<N>::E + k].y = -t.s;
      }
  }
};
template <int N>
__device__ const LineTable<N> line_table = LineTable<N>();

template <int N>
__device__ __forceinline__ void line_twiddles(cpx<float>* tw_s, int threads) {
  constexpr int E = LineG<N>::E;
  for (int i = threadIdx.x; i < N; i += threads) tw_s[(i / E) * LineG<N>::TWP + i % E] = line_table<N>.w[i];
}

// One line: v[m] = element g + G m, before and after; at(i) is the place of element i; sync()
// separates the line's lanes.
template <int N, bool INV, typename F, typename Sync>
__device__ __forceinline__ void line_fft(cpx<float> (&v)[LineG<N>::E], int g, const cpx<float>* tw_s, F at, Sync sync) {
  constexpr int E = LineG<N>::E, G = LineG<N>::G;
  rc_dft<E, INV, 1>(v);
  const float4* tw = reinterpret_cast<const float4*>(tw_s + g * LineG<N>::TWP);
#pragma unroll
  for (int k = 0; k < E; k += 2) {
    const float4 w = tw[k / 2];
    const cpx<float> w0 = mk<float>(w.x, w.y), w1 = mk<float>(w.z, w.w);
    v[k] = INV ? cmulc<float>(v[k], w0) : cmul<float>(v[k], w0);
    v[k + 1] = INV ? cmulc<float>(v[k + 1], w1) : cmul<float>(v[k + 1], w1);
  }
  sync();  // earlier reads of the places are done
#pragma unroll
  for (int k = 0; k < E; ++k) *at((k / G) * G * G + g * G + (g ^ (k % G))) = v[k];
  sync();
#pragma unroll
  for (int m = 0; m < E / G; ++m) {  // k = g + G m: outputs k + E q
    cpx<float> u[G];
#pragma unroll
    for (int h = 0; h < G; ++h) u[h] = *at(m * G * G + h * G + (h ^ g));
    rc_dft<G, INV, 1>(u);
#pragma unroll
    for (int q = 0; q < G; ++q) v[m + (E / G) * q] = u[q];
  }
}

// z pass (in place on a.data)
template <int N>
__global__ void __launch_bounds__(LineG<N>::Z_THREADS) line_z_kernel(const __grid_constant__ FftGroup<float> gr) {
  using L = LineG<N>;
  constexpr int E = L::E, G = L::G;
  const FftPassArgs<float>& a = gr.a[blockIdx.y];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<float>* tw_s = reinterpret_cast<cpx<float>*>(smem_raw);
  cpx<float>* buf = tw_s + G * L::TWP;  // [place][8 columns]
  float* sym = reinterpret_cast<float*>(buf + 8 * N);
  const int tid = threadIdx.x, c = tid & 7, g = tid >> 3;
  const int col = (int)blockIdx.x * 8 + c, kx = col % N, ky = col / N;
  cpx<float>* __restrict__ S = a.data + col;
  cpx<float> v[E];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = S[(long long)(g + G * m) * N * N];
  line_twiddles<N>(tw_s, L::Z_THREADS);
  for (int i = tid; i < N; i += L::Z_THREADS) sym[i] = a.symbol[i];
  __syncthreads();
  auto at = [&](int i) { return buf + 8 * i + c; };
  auto sync = [] { __syncthreads(); };
  line_fft<N, false>(v, g, tw_s, at, sync);
  const float sxy = sym[kx] + sym[ky], am = sqrtf(a.am2);
#pragma unroll
  for (int m = 0; m < E; ++m)
    v[m] = cscale<float>(v[m], kin_mult_rest(a.kinetic, sxy, sym[g + G * m], a.tcoef, a.am2, am));
  line_fft<N, true>(v, g, tw_s, at, sync);
#pragma unroll
  for (int m = 0; m < E; ++m) S[(long long)(g + G * m) * N * N] = v[m];
}

// x pass: a.data -> update of psi (and sums) -> x transform of psi_{t+1} into a.data (with NEXT).
// Blocks walk the lines from the last to the first, as the four-pass kernel does: the y pass
// wrote those last.
template <int N, bool VREAL, bool SUMS, bool NEXT>
__global__ void __launch_bounds__(32 * LineG<N>::X_WARPS, LineG<N>::X_PER_SM)
    line_x_kernel(const __grid_constant__ FftGroup<float> gr) {
  using L = LineG<N>;
  constexpr int E = L::E, G = L::G;
  const FftPassArgs<float>& a = gr.a[blockIdx.y];
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<float>* tw_s = reinterpret_cast<cpx<float>*>(smem_raw);
  cpx<float>* lines = tw_s + G * L::TWP;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane % G, l = warp * L::LPW + lane / G;
  const int bid = (int)gridDim.x - 1 - (int)blockIdx.x;
  const long long row = ((long long)bid * L::X_WARPS * L::LPW + l) * N + g;
  cpx<float>* __restrict__ S = a.data;
  cpx<float> v[E], psi[E], vv[VREAL ? 1 : E];
  float vr[VREAL ? E : 1];
#pragma unroll
  for (int m = 0; m < E; ++m) v[m] = S[row + G * m];
#pragma unroll
  for (int m = 0; m < E; ++m) {
    psi[m] = a.psi[row + G * m];
    if constexpr (VREAL) vr[m] = reinterpret_cast<const float*>(a.v)[row + G * m];
    else vv[m] = reinterpret_cast<const cpx<float>*>(a.v)[row + G * m];
  }
  line_twiddles<N>(tw_s, 32 * L::X_WARPS);
  const float sc = float(*a.scale);
  __syncthreads();
  auto at = [&](int i) { return lines + l * L::LP + i; };
  auto sync = [] { __syncwarp(); };
  line_fft<N, true>(v, g, tw_s, at, sync);
  // v = H_K psi (1/N^3 inside T)
  if (N == 192 && a.kinetic == KIN_FFT_REL) {  // (the z pass of 512 is the four-pass kernel's, with all of T)
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
    block_sum_store<kNumSums>(acc, reinterpret_cast<double*>(lines + L::X_WARPS * L::LPW * L::LP),
                              a.partials + (long long)bid * kPartialStride);
  }
#pragma unroll
  for (int m = 0; m < E; ++m) {
    if constexpr (VREAL) v[m] = reg_update(psi[m], v[m], vr[m], a.half_dtau, a.dtau, a.dtau_lo, sc);
    else v[m] = reg_update(psi[m], v[m], vv[m], a.half_dtau, a.dtau, a.dtau_lo, sc);
    a.psi[row + G * m] = v[m];
  }
  if constexpr (NEXT) {
    line_fft<N, false>(v, g, tw_s, at, sync);
#pragma unroll
    for (int m = 0; m < E; ++m) S[row + G * m] = v[m];
  }
}

}  // namespace qf
