// Single FDTD step (Eq. HK0), sm_103a: the per-site update shared by every stencil kernel
// and the kernel of one step.
#pragma once
#include "qf_common.cuh"

namespace qf {

// ---- the per-site FDTD update, shared by every kernel that computes a site ------------
// Each operation is rounded explicitly (no contraction left to the compiler), so the
// single-step kernel and the temporally blocked kernel produce the same bits for a site.
template <typename R> __device__ __forceinline__ R add_rn(R a, R b);
template <typename R> __device__ __forceinline__ R mul_rn(R a, R b);
template <typename R> __device__ __forceinline__ R fma_rn(R a, R b, R c);
template <typename R> __device__ __forceinline__ R scaled_inverse(R s, R d);
template <> __device__ __forceinline__ float add_rn<float>(float a, float b) { return __fadd_rn(a, b); }
template <> __device__ __forceinline__ double add_rn<double>(double a, double b) { return __dadd_rn(a, b); }
template <> __device__ __forceinline__ float mul_rn<float>(float a, float b) { return __fmul_rn(a, b); }
template <> __device__ __forceinline__ double mul_rn<double>(double a, double b) { return __dmul_rn(a, b); }
template <> __device__ __forceinline__ float fma_rn<float>(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <> __device__ __forceinline__ double fma_rn<double>(double a, double b, double c) { return __fma_rn(a, b, c); }
// s / d: FP32 as s times the hardware reciprocal (about 2 ulp, two instructions; 0 for
// |d| > 2^126, as the fast division has it); FP64 through the correctly rounded reciprocal
__device__ __forceinline__ float rcp_fast(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return r;
}
template <> __device__ __forceinline__ float scaled_inverse<float>(float s, float d) { return __fmul_rn(s, rcp_fast(d)); }
template <> __device__ __forceinline__ double scaled_inverse<double>(double s, double d) {
  return __dmul_rn(s, __drcp_rn(d));
}

// sum of the six neighbours in the fixed order ((x- + x+) + (y- + y+)) + (z- + z+)
template <typename R>
__device__ __forceinline__ cpx<R> six_sum(cpx<R> xm, cpx<R> xp, cpx<R> ym, cpx<R> yp, cpx<R> zm, cpx<R> zp) {
  return mk<R>(add_rn<R>(add_rn<R>(add_rn<R>(xm.x, xp.x), add_rn<R>(ym.x, yp.x)), add_rn<R>(zm.x, zp.x)),
               add_rn<R>(add_rn<R>(add_rn<R>(xm.y, xp.y), add_rn<R>(ym.y, yp.y)), add_rn<R>(zm.y, zp.y)));
}

// lap = sum of neighbours - 6 psi, so that H_K^(0) psi = -kcoef * lap (Eq. HK0)
template <typename R>
__device__ __forceinline__ cpx<R> lap_of(cpx<R> c, cpx<R> nbs) {
  return mk<R>(fma_rn<R>(R(-6), c.x, nbs.x), fma_rn<R>(R(-6), c.y, nbs.y));
}

// psi' = s (coef_A psi - coef_B dtau H_K psi) with d = 1 + dtau V / 2:
// psi' = s ((2 - d) psi + kd lap) conj(d) / |d|^2, kd = dtau * kcoef.  For real V,
// conj(d)/|d|^2 = 1/d.
template <typename R>
__device__ __forceinline__ cpx<R> fdtd_update(cpx<R> c, cpx<R> lap, cpx<R> v, bool v_real, R half_dtau, R kd, R sc) {
  const R dx = fma_rn<R>(half_dtau, v.x, R(1));
  const R tx = add_rn<R>(R(2), -dx);
  if (v_real) {
    const R inv = scaled_inverse<R>(sc, dx);
    return mk<R>(mul_rn<R>(fma_rn<R>(kd, lap.x, mul_rn<R>(tx, c.x)), inv),
                 mul_rn<R>(fma_rn<R>(kd, lap.y, mul_rn<R>(tx, c.y)), inv));
  }
  const R dy = mul_rn<R>(half_dtau, v.y);
  // (2 - d) psi = (tx - i dy) psi
  const R ax = fma_rn<R>(tx, c.x, mul_rn<R>(dy, c.y));
  const R ay = fma_rn<R>(tx, c.y, -mul_rn<R>(dy, c.x));
  const R nx = fma_rn<R>(kd, lap.x, ax), ny = fma_rn<R>(kd, lap.y, ay);
  const R inv = scaled_inverse<R>(sc, fma_rn<R>(dx, dx, mul_rn<R>(dy, dy)));
  return mk<R>(mul_rn<R>(fma_rn<R>(nx, dx, mul_rn<R>(ny, dy)), inv),
               mul_rn<R>(fma_rn<R>(ny, dx, -mul_rn<R>(nx, dy)), inv));
}


// ---- one step -----------------------------------------------------------------------------
// A thread owns one in-plane position p = y n + x (128 consecutive positions per block, so no
// lane is lost on sizes that 32 does not divide) and marches through zc planes with the
// z-neighbours in registers; the four in-plane neighbours come through L1 and L2.  Nothing is
// staged in shared memory.  What bounds it: the FP64 pipe in complex FP64 (2 fused
// multiply-adds per clock and SM: 20 per site with the table of a real V, 29
// without), HBM and L2 in complex FP32, latency on small lattices, which need as many blocks as
// they have rows: the 32 x 32 tiles of 8 planes used before left all but 4 SMs idle at N = 32.
// One step, tiles / now (mean of a run of steps): complex FP64 with real V N = 32: 69 / 4.3 us,
// 64: 71 / 15, 128: 133 / 97, 160: 260 / 196; with complex V 64: 97 / 26, 128: 175 / 156, 160: 339 /
// 295; complex FP32 N = 32: 23 / 4.2 us, 250: 112 / 76, 512: 783 / 559.
constexpr int kFlatThreads = 128;

// Members of one launch may have different lattice sizes: member i runs
// ceil(n_i^2 / 128) x ceil(n_i / zc_i) blocks, numbered from start[i] in a one-dimensional
// grid (in-plane block fastest, then z-chunk), exactly the blocks it runs alone.
template <typename R>
struct StencilGroup {
  StencilArgs<R> a[kGroupMax];
  int nm[kGroupMax];        // lattice size of member i
  int start[kGroupMax + 1]; // first block of member i; start[count] = blocks in all
  int count;
};

__host__ __device__ __forceinline__ int stencil_plane_blocks(int n) { return (n * n + kFlatThreads - 1) / kFlatThreads; }

// Planes per block: as many as leave about 8 blocks per SM (a block's first plane reads two
// planes that its neighbour chunk reads too), at most 16.
__host__ __device__ __forceinline__ int stencil_zchunk(int n) {
  const int zc = (int)((long long)n * stencil_plane_blocks(n) / (152 * 8));
  return zc < 1 ? 1 : zc > 16 ? 16 : zc;
}

// Blocks (partial-sum rows) member i of a stencil group runs.
__host__ __device__ __forceinline__ int stencil_member_blocks(int n) {
  const int zc = stencil_zchunk(n);
  return stencil_plane_blocks(n) * ((n + zc - 1) / zc);
}

template <typename R>
__global__ void __launch_bounds__(kFlatThreads) stencil_flat_kernel(const __grid_constant__ StencilGroup<R> g) {
  // member of this block (last i with start[i] <= block), then its positions and z-chunk
  int member = 0;
  {
    int hi = g.count - 1;
    while (member < hi) {
      const int mid = (member + hi + 1) >> 1;
      if (g.start[mid] <= (int)blockIdx.x) member = mid;
      else hi = mid - 1;
    }
  }
  const StencilArgs<R>& a = g.a[member];
  const int n = g.nm[member], n2 = n * n, nbp = stencil_plane_blocks(n), zc = stencil_zchunk(n);
  const int local = (int)blockIdx.x - g.start[member];
  const int pb = local % nbp, zb = local / nbp;
  const int p = pb * kFlatThreads + (int)threadIdx.x;
  const int y = p / n, x = p - y * n;
  const int z0 = zb * zc, z1 = min(n, z0 + zc);
  const bool in_plane = p < n2;
  // sites with an index 0 (the Dirichlet planes) are zero, whatever the input holds there, and
  // so are neighbours on those planes or outside the lattice
  const bool live = in_plane && x >= 1 && y >= 1;
  const bool hxm = live && x > 1, hxp = live && x + 1 < n, hym = live && y > 1, hyp = live && y + 1 < n;
  const cpx<R> zero = mk<R>(R(0), R(0));
  const cpx<R>* __restrict__ in = a.in;
  const R sc = R(*a.scale), ks = a.kd * sc, khs = R(0.5) * ks;
  CheckSums<R> cs;
  long long site = (long long)z0 * n2 + p;
  cpx<R> zm = zero, c = zero;
  if (live && z0 >= 2) zm = in[site - n2];
  if (live && z0 >= 1) c = in[site];
  for (int z = z0; z < z1; ++z, site += n2) {
    const bool up = z >= 1;
    cpx<R> zp = zero, xm = zero, xp = zero, ym = zero, yp = zero, vv = zero;
    if (live && z + 1 < n) zp = in[site + n2];
    if (up) {
      if (hxm) xm = in[site - 1];
      if (hxp) xp = in[site + 1];
      if (hym) ym = in[site - n];
      if (hyp) yp = in[site + n];
      if (live && (sizeof(R) == 4 || !a.coef_u || a.reduce)) vv = a.v_real ? mk<R>(reinterpret_cast<const R*>(a.v)[site], R(0)) : reinterpret_cast<const cpx<R>*>(a.v)[site];
    }
    if (live && up) {
      const cpx<R> nbs = six_sum<R>(xm, xp, ym, yp, zm, zp);
      if constexpr (sizeof(R) == 8) {
        if (a.coef_u && a.write_psi && !a.reduce) {
          // psi' = sc (psi - u psi + kd (1 - u/2) lap), u = 1 - coef_A from the lattice's table: 20
          // FP64 operations a site, where lap, the update and the division take 29
          const R u = a.coef_u[site], us = u * sc, cb = fma(-khs, u, ks);
          const cpx<R> lap = lap_of<R>(c, nbs);
          a.out[site] = mk<R>(fma(sc, c.x, -fma(us, c.x, -(cb * lap.x))), fma(sc, c.y, -fma(us, c.y, -(cb * lap.y))));
          zm = c;
          c = zp;
          continue;
        }
      }
      const cpx<R> lap = lap_of<R>(c, nbs);
      if (a.reduce) cs.add(c, mk<R>(mul_rn<R>(-a.kcoef, lap.x), mul_rn<R>(-a.kcoef, lap.y)), vv);
      if (a.write_psi) a.out[site] = fdtd_update<R>(c, lap, vv, a.v_real != 0, a.half_dtau, a.kd, sc);
    } else if (in_plane && a.write_psi) {
      a.out[site] = zero;
    }
    zm = c;
    c = zp;
  }
  if (a.reduce) {
    __shared__ double red_s[32 * kNumSums];
    double acc[kNumSums];
    cs.to(acc);
    block_sum_store<kNumSums>(acc, red_s, a.partials + (long long)local * kPartialStride);
  }
}

}  // namespace qf
