// Resident imaginary-time FFT steps for small complex-FP32 lattices (N <= 32; Eqs. HK1-HK3
// and the update of Sec. 2), sm_103a.
//
// One thread-block cluster holds a whole lattice and takes any number of steps per launch:
// psi and V stay in registers, the transformed field in shared memory, and the two
// redistributions of a step go through distributed shared memory.  Each of the cluster's C
// blocks owns P = N / C z-planes; a thread (N = 32: four lanes) transforms a whole line:
//   x forward, y forward on its planes  ->  column (kx, ky) to the block that owns ky
//   z forward, T(k), z inverse          ->  column element z to the block that owns z
//   y inverse, x inverse, update of psi in registers, and round again.
// A step has two block barriers and no cluster barrier: an element is stored into the block
// that needs it (st.async), whose barrier counts the bytes, and a block goes on when all of
// its P N^2 elements are in.  Nothing is overwritten early: a block stores into the buffer
// that a peer read last only after it has received everything that the peer sends once it
// has read it.
//
// A wait is bounded.  A thread whose wait runs out sends nothing more and re-arms no barrier, but
// keeps to the block barriers; without its share no later redistribution completes, so every
// other thread's next wait runs out too and a launch ends after two limits.  Such a thread
// stores NaN for its sites (the allocation-free step has no other way to say so), sets the
// error flag, and holds its block until no thread of the cluster can store into it any more.
//
// What bounds it: instruction issue and latency of few warps (N = 32: eight per SM on 16 SMs; with a
// line per thread, two per SM, 5.4 us a step, 6.3 with complex V and 6.0 with Eq. HK3).
// The four-pass form needs four launches a step, each bound by the 2-3 us that any kernel
// takes.  One step, before and now: N = 8: 7.0 / 1.6 us, 12: 11.2 / 2.1, 16: 13.0 / 2.2, 24:
// 14.8 / 4.2, 32: 11.6 / 5.0.  At N = 48 (13.3 against 12.8 us) the 16 SMs of a cluster are too few.
#pragma once
#include "qf_fft_plane.cuh"

namespace qf {

// Lattices per launch and their arguments.  Members run on clusters of their own and need
// not be stepped alike (nsteps, reduce).
struct ResArgs {
  cpx<float>* psi;           // psi_t in, psi_{t + nsteps} out
  const void* v;             // potential: cpx<float> or float
  const float* symbol;       // per-axis kinetic symbol
  const double* scale;       // output scale of the first step
  const double* scale2;      // and of the others
  double* partials;          // kNumSums per block of the cluster when reducing
  float tcoef, am2, half_dtau, dtau, dtau_lo, t0, t0_lo;
  int* err;                  // set to 1 when a bounded wait ran out
  int kinetic, nsteps;
  unsigned spin;             // tries of a wait (kResSpin)
};
struct ResGroup {
  int count;
  ResArgs a[kGroupMax];
};
// One step of a caller that keeps no tables: they travel in the kernel's parameters.
struct ResStatic {
  ResArgs a;
  float sym[32];
  double out_scale;
};

// Tries before a wait runs out, and for what may still be under way after that (a store between
// the blocks of a cluster takes microseconds, a try tens of nanoseconds at least).
constexpr unsigned kResSpin = 1u << 24, kResDrain = 1u << 16;

constexpr bool res_supported(int n) { return n == 8 || n == 12 || n == 16 || n == 24 || n == 32; }

template <int N>
struct ResG {
  static constexpr int C = N == 8 ? 2 : N == 12 ? 4 : N <= 24 ? 8 : 16;  // blocks per cluster
  static constexpr int P = N / C;
  static constexpr int LANES = N == 32 ? 4 : 1;  // per line
  static constexpr int THREADS = P * N * LANES;
  // row pitch in elements: odd where a thread has a line, so that lanes along a column and
  // along a row both spread over all banks; else the plane form's layout
  static constexpr int NP = LANES == 1 ? N + 1 : N + 8;
  static constexpr int SLAB = N * NP;  // a plane [y][x], or a ky [z][kx]
  static constexpr size_t TW = LANES == 1 ? 0 : 4 * (N / 4 + 2);
  static constexpr unsigned BYTES = P * N * N * 8;  // a block's share of a redistribution
  static constexpr size_t SMEM = (TW + 2 * P * SLAB) * 8 + N * 8 + 32 * kNumSums * 8;
  static_assert(N % C == 0 && THREADS <= 1024, "resident geometry");
};

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// Stores into the shared memory of block `rank` of the cluster, at the place `p` has in this
// one's, and counts the bytes on that block's barrier at the place of `bar`.
__device__ __forceinline__ unsigned res_map(const void* p, int rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(cpx<float>* p, int rank, cpx<float> v, const unsigned long long* bar) {
  unsigned long long w;
  asm("mov.b64 %0, {%1, %2};" : "=l"(w) : "f"(v.x), "f"(v.y));
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];\n" ::"r"(res_map(p, rank)),
               "l"(w), "r"(res_map(bar, rank))
               : "memory");
}
// Bounded wait for phase `parity` of the block's own barrier (acquires what the cluster's
// blocks stored); after a time-out it returns false at once for the rest of the launch.
__device__ __forceinline__ bool res_wait(unsigned long long* bar, unsigned parity, bool ok, unsigned spin) {
  const unsigned b = (unsigned)__cvta_generic_to_shared(bar);
  for (unsigned it = 0; ok && it < spin; ++it) {
    unsigned done;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(done)
                 : "r"(b), "r"(parity)
                 : "memory");
    if (done) return true;
  }
  return false;
}
__device__ __forceinline__ void res_expect(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"((unsigned)__cvta_generic_to_shared(bar)), "r"(bytes)
               : "memory");
}

// End of a thread whose wait ran out (see above).  Every thread that has not exited has sent all it
// will once it has arrived here (and one that has exited counts as arrived: its block had
// received everything).  What is still under way counts on the phases that the block's barriers
// are in: of the two waits on each, one is for the phase before and returns at once.
__device__ __forceinline__ void res_close(bool ok, int* err, unsigned long long* bars) {
  if (ok) return;
  if (err) atomicExch(err, 1);
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
  for (int i = 0; i < 4; ++i) res_wait(&bars[i >> 1], i & 1, true, kResDrain);
}

// The block's sums (THREADS need not fill its last warp) to out[0 .. kNumSums).
template <int THREADS>
__device__ __forceinline__ void res_block_sum(double (&s)[kNumSums], double* scratch, double* out) {
  constexpr int WARPS = (THREADS + 31) / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lanes = warp + 1 < WARPS ? 32 : THREADS - 32 * (WARPS - 1);
  const unsigned mask = lanes == 32 ? 0xffffffffu : (1u << lanes) - 1u;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int i = 0; i < kNumSums; ++i) {
      const double t = __shfl_down_sync(mask, s[i], off);
      if (lane + off < lanes) s[i] += t;
    }
  if (lane == 0)
#pragma unroll
    for (int i = 0; i < kNumSums; ++i) scratch[warp * kNumSums + i] = s[i];
  __syncthreads();
  if (threadIdx.x < kNumSums) {
    double t = 0.0;
    for (int w = 0; w < WARPS; ++w) t += scratch[w * kNumSums + threadIdx.x];
    out[threadIdx.x] = t;
  }
}

// N = 32: four lanes a line, as in the plane form (lane g holds the elements g + 4 m), so that a
// block has 8 warps instead of 2.
template <int N, bool VREAL, bool SUMS>
__device__ __forceinline__ void res_body4(const ResArgs& a, const float* sym_g, float sc1, float sc2) {
  using G = ResG<N>;
  constexpr int P = G::P, E = N / 4, ST = N * 4;  // ST threads a slab
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* red_s = reinterpret_cast<double*>(smem_raw);
  cpx<float>* tw_s = reinterpret_cast<cpx<float>*>(red_s + 32 * kNumSums);
  cpx<float>* plane = tw_s + G::TW;
  cpx<float>* cols = plane + P * G::SLAB;
  float* sym = reinterpret_cast<float*>(cols + P * G::SLAB);
  __shared__ alignas(8) unsigned long long bars[2];
  const int tid = threadIdx.x, rank = blockIdx.x;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"((unsigned)__cvta_generic_to_shared(&bars[i])) : "memory");
      res_expect(&bars[i], G::BYTES);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  bool ok = true;
  unsigned parity = 0;
  const float am = sqrtf(a.am2);
  plane_twiddles<N>(tw_s, G::THREADS);
  for (int i = tid; i < N; i += G::THREADS) sym[i] = sym_g[i];
  const int s = tid / ST, warp = (tid % ST) >> 5, lane = tid & 31;
  const int xg = lane & 3, line = warp * 8 + (lane >> 2), cg = lane >> 3, col = warp * 8 + (lane & 7);
  auto x_at = [&](int i) { return plane + s * G::SLAB + plane_idx<N>(line, i); };
  auto y_at = [&](int i) { return plane + s * G::SLAB + plane_idx<N>(i, col); };
  auto z_at = [&](int i) { return cols + s * G::SLAB + plane_idx<N>(i, col); };
  auto slab_sync = [&] { asm volatile("bar.sync %0, %1;\n" ::"r"(1 + s), "n"(ST) : "memory"); };
  const long long row = (((long long)rank * P + s) * N + line) * N + xg;
  cpx<float> v[E], psi[E];
  float vr[E], vi[VREAL ? 1 : E];
#pragma unroll
  for (int m = 0; m < E; ++m) {
    psi[m] = a.psi[row + 4 * m];
    if constexpr (VREAL) {
      vr[m] = reinterpret_cast<const float*>(a.v)[row + 4 * m];
    } else {
      const cpx<float> w = reinterpret_cast<const cpx<float>*>(a.v)[row + 4 * m];
      vr[m] = w.x;
      vi[m] = w.y;
    }
  }
  cluster_sync();  // the tables are in place, and every block of the cluster is running
  for (int t = 0; t < (SUMS ? 1 : a.nsteps); ++t) {
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = psi[m];
    plane_line<N, false>(v, xg, tw_s, x_at);
    __syncwarp();
#pragma unroll
    for (int m = 0; m < E; ++m) *x_at(xg + 4 * m) = v[m];
    slab_sync();
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = *y_at(cg + 4 * m);
    plane_line<N, false>(v, cg, tw_s, y_at);
    // a block of the cluster receives from two of the four lanes of a line only, and may store into
    // this buffer once it has: no lane sends before all have read
    __syncwarp();
    if (ok) {
#pragma unroll
      for (int m = 0; m < E; ++m) {
        const int ky = cg + 4 * m;
        st_cluster(cols + (ky % P) * G::SLAB + plane_idx<N>(rank * P + s, col), ky / P, v[m], &bars[0]);
      }
    }
    ok = res_wait(&bars[0], parity, ok, a.spin);
    if (ok && tid == 0) res_expect(&bars[0], G::BYTES);
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = *z_at(cg + 4 * m);
    plane_line<N, false>(v, cg, tw_s, z_at);
    const float sxy = sym[col] + sym[rank * P + s];
#pragma unroll
    for (int m = 0; m < E; ++m)
      v[m] = cscale<float>(v[m], kin_mult_rest(a.kinetic, sxy, sym[cg + 4 * m], a.tcoef, a.am2, am));
    plane_line<N, true>(v, cg, tw_s, z_at);
    __syncwarp();  // (as above)
    if (ok) {
#pragma unroll
      for (int m = 0; m < E; ++m) {
        const int z = cg + 4 * m;
        st_cluster(plane + (z % P) * G::SLAB + plane_idx<N>(rank * P + s, col), z / P, v[m], &bars[1]);
      }
    }
    ok = res_wait(&bars[1], parity, ok, a.spin);
    if (ok && tid == 0) res_expect(&bars[1], G::BYTES);
    parity ^= 1;
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = *y_at(cg + 4 * m);
    plane_line<N, true>(v, cg, tw_s, y_at);
    __syncwarp();
#pragma unroll
    for (int m = 0; m < E; ++m) *y_at(cg + 4 * m) = v[m];
    slab_sync();
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = *x_at(xg + 4 * m);
    plane_line<N, true>(v, xg, tw_s, x_at);
    if (a.kinetic == KIN_FFT_REL) {
#pragma unroll
      for (int m = 0; m < E; ++m) v[m] = rest_mass(psi[m], v[m], a.t0, a.t0_lo);
    }
    if constexpr (SUMS) {
      CheckSums<float> sum;
#pragma unroll
      for (int m = 0; m < E; ++m) sum.add(psi[m], v[m], mk<float>(vr[m], VREAL ? 0.f : vi[VREAL ? 0 : m]));
      double acc[kNumSums];
      sum.to(acc);
      if (!ok) acc[0] = __longlong_as_double(-1LL);
      res_block_sum<G::THREADS>(acc, red_s, a.partials + (long long)rank * kPartialStride);
    }
    const float sc = t == 0 ? sc1 : sc2;
#pragma unroll
    for (int m = 0; m < E; ++m) {
      if constexpr (VREAL) psi[m] = reg_update(psi[m], v[m], vr[m], a.half_dtau, a.dtau, a.dtau_lo, sc);
      else psi[m] = reg_update(psi[m], v[m], mk<float>(vr[m], vi[m]), a.half_dtau, a.dtau, a.dtau_lo, sc);
    }
  }
  const float nan = __int_as_float(-1);
#pragma unroll
  for (int m = 0; m < E; ++m) a.psi[row + 4 * m] = ok ? psi[m] : mk<float>(nan, nan);
  res_close(ok, a.err, bars);
}

template <int N, bool VREAL, bool SUMS>
__device__ __forceinline__ void res_body(const ResArgs& a, const float* sym_g, float sc1, float sc2) {
  using G = ResG<N>;
  constexpr int P = G::P, NP = G::NP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* red_s = reinterpret_cast<double*>(smem_raw);
  cpx<float>* plane = reinterpret_cast<cpx<float>*>(red_s + 32 * kNumSums);  // [z_l][y][x]
  cpx<float>* cols = plane + P * G::SLAB;                                    // [ky_l][z][kx]
  float* sym = reinterpret_cast<float*>(cols + P * G::SLAB);
  __shared__ alignas(8) unsigned long long bars[2];  // data in cols, in plane
  const int tid = threadIdx.x, rank = blockIdx.x;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"((unsigned)__cvta_generic_to_shared(&bars[i])) : "memory");
      res_expect(&bars[i], G::BYTES);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  bool ok = true;
  unsigned parity = 0;
  const float am = sqrtf(a.am2);
  for (int i = tid; i < N; i += G::THREADS) sym[i] = sym_g[i];
  // the thread's line: row `l` of slab `s` as an x line, column `l` of slab s as a y or z line
  const int s = tid / N, l = tid % N;
  cpx<float>* xline = plane + s * G::SLAB + l * NP;
  cpx<float>* ycol = plane + s * G::SLAB + l;
  cpx<float>* zcol = cols + s * G::SLAB + l;
  const long long row = (((long long)rank * P + s) * N + l) * N;
  // psi and V of the line
  cpx<float> v[N], psi[N];
  float vr[N], vi[VREAL ? 1 : N];
#pragma unroll
  for (int x = 0; x < N; ++x) {
    psi[x] = a.psi[row + x];
    if constexpr (VREAL) {
      vr[x] = reinterpret_cast<const float*>(a.v)[row + x];
    } else {
      const cpx<float> w = reinterpret_cast<const cpx<float>*>(a.v)[row + x];
      vr[x] = w.x;
      vi[x] = w.y;
    }
  }
  cluster_sync();  // the symbol is in place, and every block of the cluster is running
  for (int t = 0; t < (SUMS ? 1 : a.nsteps); ++t) {
    // One copy of the transform's code a direction for the longer lines: with 2-3 warps per SM
    // straight code of all six ran at the pace of the instruction cache (N = 24: 4.4 us a step,
    // 4.2 so; N = 16: 2.2 straight, 2.4 so).
    constexpr int kUnroll = N <= 16 ? 3 : 1;
#pragma unroll
    for (int x = 0; x < N; ++x) v[x] = psi[x];
#pragma unroll kUnroll
    for (int ph = 0; ph < 3; ++ph) {  // x, y, z forward
      rc_dft<N, false, 1>(v);
      if (ph == 0) {
#pragma unroll
        for (int x = 0; x < N; ++x) xline[x] = v[x];
        __syncthreads();
#pragma unroll
        for (int y = 0; y < N; ++y) v[y] = ycol[y * NP];
      } else if (ph == 1) {
        if (ok) {
#pragma unroll
          for (int ky = 0; ky < N; ++ky)
            st_cluster(cols + (ky % P) * G::SLAB + (rank * P + s) * NP + l, ky / P, v[ky], &bars[0]);
        }
        ok = res_wait(&bars[0], parity, ok, a.spin);
        if (ok && tid == 0) res_expect(&bars[0], G::BYTES);
#pragma unroll
        for (int z = 0; z < N; ++z) v[z] = zcol[z * NP];
      }
    }
    const float sxy = sym[l] + sym[rank * P + s];
#pragma unroll
    for (int z = 0; z < N; ++z) v[z] = cscale<float>(v[z], kin_mult_rest(a.kinetic, sxy, sym[z], a.tcoef, a.am2, am));
#pragma unroll kUnroll
    for (int ph = 0; ph < 3; ++ph) {  // z, y, x inverse
      rc_dft<N, true, 1>(v);
      if (ph == 0) {
        if (ok) {
#pragma unroll
          for (int z = 0; z < N; ++z)
            st_cluster(plane + (z % P) * G::SLAB + (rank * P + s) * NP + l, z / P, v[z], &bars[1]);
        }
        ok = res_wait(&bars[1], parity, ok, a.spin);
        if (ok && tid == 0) res_expect(&bars[1], G::BYTES);
        parity ^= 1;
#pragma unroll
        for (int y = 0; y < N; ++y) v[y] = ycol[y * NP];
      } else if (ph == 1) {
#pragma unroll
        for (int y = 0; y < N; ++y) ycol[y * NP] = v[y];
        __syncthreads();
#pragma unroll
        for (int x = 0; x < N; ++x) v[x] = xline[x];
      }
    }
    // v = H_K psi at the sites of psi; update
    if (a.kinetic == KIN_FFT_REL) {
#pragma unroll
      for (int x = 0; x < N; ++x) v[x] = rest_mass(psi[x], v[x], a.t0, a.t0_lo);
    }
    if constexpr (SUMS) {
      CheckSums<float> sum;
#pragma unroll
      for (int x = 0; x < N; ++x) sum.add(psi[x], v[x], mk<float>(vr[x], VREAL ? 0.f : vi[VREAL ? 0 : x]));
      double acc[kNumSums];
      sum.to(acc);
      if (!ok) acc[0] = __longlong_as_double(-1LL);
      res_block_sum<G::THREADS>(acc, red_s, a.partials + (long long)rank * kPartialStride);
    }
    const float sc = t == 0 ? sc1 : sc2;
#pragma unroll
    for (int x = 0; x < N; ++x) {
      if constexpr (VREAL) psi[x] = reg_update(psi[x], v[x], vr[x], a.half_dtau, a.dtau, a.dtau_lo, sc);
      else psi[x] = reg_update(psi[x], v[x], mk<float>(vr[x], vi[x]), a.half_dtau, a.dtau, a.dtau_lo, sc);
    }
  }
  const float nan = __int_as_float(-1);
#pragma unroll
  for (int x = 0; x < N; ++x) a.psi[row + x] = ok ? psi[x] : mk<float>(nan, nan);
  res_close(ok, a.err, bars);
}

template <int N, bool VREAL, bool SUMS>
__global__ void __launch_bounds__(ResG<N>::THREADS) fft_res_kernel(const __grid_constant__ ResGroup g) {
  const ResArgs& a = g.a[blockIdx.y];
  if constexpr (ResG<N>::LANES == 4) res_body4<N, VREAL, SUMS>(a, a.symbol, (float)*a.scale, (float)*a.scale2);
  else res_body<N, VREAL, SUMS>(a, a.symbol, (float)*a.scale, (float)*a.scale2);
}
template <int N, bool VREAL, bool SUMS>
__global__ void __launch_bounds__(ResG<N>::THREADS) fft_res_static_kernel(const __grid_constant__ ResStatic g) {
  if constexpr (ResG<N>::LANES == 4) res_body4<N, VREAL, SUMS>(g.a, g.sym, (float)g.out_scale, (float)g.out_scale);
  else res_body<N, VREAL, SUMS>(g.a, g.sym, (float)g.out_scale, (float)g.out_scale);
}

// nsteps steps of every member of g (one lattice size, one kind of potential) in one launch;
// with `reduce` one step and its check sums.
cudaError_t launch_fft_res(int n, const ResGroup& g, bool v_real, bool reduce, cudaStream_t st);
cudaError_t launch_fft_res_static(int n, const ResStatic& g, bool v_real, bool reduce, cudaStream_t st);
// Self-test of res_wait: one block waits, `spin` tries, for bytes that nobody sends; *err is set when
// every thread's wait ran out.
cudaError_t launch_bounded_wait_probe(int* err, unsigned spin, cudaStream_t st);
// Partial-sum rows of a member; 0 where the size has no resident form or the device cannot
// run its cluster.
int fft_res_blocks(int n);

}  // namespace qf
