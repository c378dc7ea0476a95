// Two FDTD steps per pass over HBM (kinetic term of Eq. HK0, complex FP32 fields), sm_103a.
//
// Two consecutive steps read psi_t and V and write psi_{t+2}; the intermediate psi_{t+1}
// never leaves the registers of a warp.  A warp owns 4 rows of 28 output columns and marches
// through a chunk of z, lane = x (32 columns: the outputs and a halo of 2 on either side).
// Three levels are in flight at once:
//   level 0  psi_t on 8 rows (halo 2), three planes of it in registers;
//   level 1  psi_{t+1} on 6 rows (halo 1) of the middle plane: y- and z-neighbours are the
//            lane's own registers, x-neighbours come by shuffle;
//   level 2  psi_{t+2} on the 4 rows, one plane behind level 1, stored by lanes 2 .. 29.
// Loads of the plane after next are issued once level 1 has freed the oldest plane's
// registers.  No shared memory and no barrier, one warp per block (so that everything but
// the column is the same in all lanes for the compiler; blocks of 4 or 8 warps, whose halo
// rows meet in L1, came out 15-35 % slower).  The arithmetic is on packed pairs (re, im), one
// instruction where two were needed, and the lane's address of a row is one instruction.
//
// What bounds it: instruction issue and load latency about equally (N = 256: 68 M warp
// instructions, 62 % of issue slots, 16 warps per SM at 128 registers), not yet HBM (20
// bytes per site and two steps).  The form before kept both levels in shared memory
// (TMA-filled 36 x 36 planes, seven reads a site, a block barrier per plane, about 190
// instructions a site).  Two steps, before and now: N = 64: 31 / 8.4 us, 128: 25 / 17 us,
// 250: 131 / 86 us (3.6 TB/s of the 20 bytes), 256: 134 / 97 us, 384: 402 / 274 us.
//
// Sites with an index 0 (the Dirichlet planes) and sites outside the lattice are zero at
// every level; the input field must already be zero on the Dirichlet planes (true after
// any FDTD step), so a load from outside is redirected to one of them.  Each site is computed
// with the same rounded operations as the single-step kernel, so two single steps and one
// pass give the same bits.
//
// A group launch steps several lattices of any sizes at once: a one-dimensional grid whose
// blocks are numbered member by member from a block table; a lone lattice is a group of one.
#pragma once
#include <type_traits>
#include <utility>

#include "qf_stencil_flat.cuh"

namespace qf {

constexpr int TB_XOUT = 28, TB_ROWS = 4;
constexpr int TB_R0 = TB_ROWS + 4, TB_R1 = TB_ROWS + 2;

struct StencilTbArgs {
  const cpx<float>* in;   // psi_t
  cpx<float>* out;        // psi_{t+2}
  const void* v;          // V: float (v_real) or complex float
  int v_real;
  float half_dtau;        // dtau / 2
  float kd;               // dtau / (2 m a^2)
  const double* scale;    // output scale of the first of the two steps
  const double* scale2;   // output scale of the second
  int n;
  int nzb;                // z-chunks: chunk b holds planes [b n/nzb, (b+1) n/nzb)
};

// Members of a group launch: blocks of member i are start[i] .. start[i+1] - 1 (the
// launcher fills start).  All members have the same kind of potential (v_real).
struct StencilTbGroup {
  StencilTbArgs m[kGroupMax];
  int start[kGroupMax + 1];
  int count;
};

__host__ __device__ inline int stencil_tb_xtiles(int n) { return (n + TB_XOUT - 1) / TB_XOUT; }
__host__ __device__ inline int stencil_tb_ytiles(int n) { return (n + TB_ROWS - 1) / TB_ROWS; }
__host__ __device__ inline int stencil_tb_member_blocks(int n, int nzb) {
  return stencil_tb_xtiles(n) * stencil_tb_ytiles(n) * nzb;
}

// z-chunks for lattice size n.  Two planes a chunk while all warps fit the GPU at once (16
// resident warps per SM at 128 registers): a small lattice is bound by the latency of a
// warp's march.  Beyond that as many chunks as make whole waves of resident warps, with at
// least 16 planes each (a chunk repeats two planes of level 1 and four loads); one wave if
// its chunks are shorter than that.  Measured, us per pass: N = 64: 8.6 in chunks of 2 planes, 9.3 of
// 4, 17 of 16; N = 192: 43.9 in one wave, 47.7 in 1.7; N = 250: 85.7 / 86.5 / 87.6 / 89.2 in
// 1 / 2 / 3 / 4 waves, 96 in 7; N = 384: 315 in 1.7 waves, 281 in 2.8, 268 in 8, 275 in 13 (taken),
// 297 in 26.
inline int stencil_tb_chunks(int n) {
  const long long cap = 152 * 16, tiles = stencil_tb_member_blocks(n, 1);
  if (tiles * ((n + 1) / 2) <= cap) return (n + 1) / 2;
  long long best = cap / tiles > 1 ? cap / tiles : 1;
  for (long long w = 2; w * cap / tiles * 16 <= n; ++w) best = w * cap / tiles > 1 ? w * cap / tiles : 1;
  return (int)best;
}

// ---- packed complex FP32 (re in the low half): each half rounded as the scalar operation ---
using pk = unsigned long long;
__device__ __forceinline__ pk pk_make(float lo, float hi) {
  pk r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ cpx<float> pk_get(pk a) {
  cpx<float> c;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(c.x), "=f"(c.y) : "l"(a));
  return c;
}
__device__ __forceinline__ pk pk_add(pk a, pk b) {
  pk r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ pk pk_mul(pk a, pk b) {
  pk r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ pk pk_fma(pk a, pk b, pk c) {
  pk r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// base + k * stride bytes in one instruction (k a constant, stride the same in all lanes)
template <int K>
__device__ __forceinline__ unsigned long long tb_addr(unsigned long long base, unsigned stride) {
  unsigned long long r;
  if constexpr (K == 0) r = base;
  else asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(stride), "n"(K), "l"(base));
  return r;
}
template <typename F, int... I>
__device__ __forceinline__ void tb_rows(F&& f, std::integer_sequence<int, I...>) {
  (f(std::integral_constant<int, I>{}), ...);
}

// One site: c and its neighbours, potential (vx, vy), output scale sc; live: whether the site
// may be nonzero (else the result is zero, whatever V holds there: a dead site reads V at an
// index 0, where a caller may have put an infinite wall).  The same operations, in the same order,
// as fdtd_update after lap_of(six_sum).
template <bool VREAL>
__device__ __forceinline__ pk tb_site(pk c, pk xm, pk xp, pk ym, pk yp, pk zm, pk zp, float vx, float vy, float hd,
                                      pk kd2, pk m6, float sc, bool live) {
  const pk nbs = pk_add(pk_add(pk_add(xm, xp), pk_add(ym, yp)), pk_add(zm, zp));
  const pk lap = pk_fma(m6, c, nbs);
  const float dx = fma_rn<float>(hd, vx, 1.f), tx = add_rn<float>(2.f, -dx);
  if constexpr (VREAL) {
    const float inv = scaled_inverse<float>(sc, dx);
    const pk u = pk_mul(pk_fma(kd2, lap, pk_mul(pk_make(tx, tx), c)), pk_make(inv, inv));
    return live ? u : 0ull;
  } else {
    // (2 - d) psi = (tx - i dy) psi, d = dx + i dy
    const float dy = mul_rn<float>(hd, vy);
    const cpx<float> cc = pk_get(c);
    const float ax = fma_rn<float>(tx, cc.x, mul_rn<float>(dy, cc.y));
    const float ay = fma_rn<float>(tx, cc.y, -mul_rn<float>(dy, cc.x));
    const cpx<float> nn = pk_get(pk_fma(kd2, lap, pk_make(ax, ay)));
    const float inv = scaled_inverse<float>(sc, fma_rn<float>(dx, dx, mul_rn<float>(dy, dy)));
    const pk u = pk_make(mul_rn<float>(fma_rn<float>(nn.x, dx, mul_rn<float>(nn.y, dy)), inv),
                         mul_rn<float>(fma_rn<float>(nn.y, dx, -mul_rn<float>(nn.x, dy)), inv));
    return live ? u : 0ull;
  }
}

// The two steps for output columns [28 bx, 28 bx + 28), rows [y0, y0 + 4) and planes [z0, z1)
// of the lattice in g.  EDGE: some row of the warp's levels is row 0 or lies outside the
// lattice.  Positions that must read as zero are redirected to plane 0 or column 0 (zero); dead
// positions are zero at both levels by selection, whatever V or a neighbour holds.
template <bool VREAL, bool EDGE, bool PRE>
__device__ __forceinline__ void stencil_tb_march(const StencilTbArgs& g, int bx, int y0, int z0, int z1) {
  using u64 = unsigned long long;
  const int n = g.n, lane = threadIdx.x;
  const long long n2 = (long long)n * n;
  const int x = bx * TB_XOUT - 2 + lane;
  const bool xlive = x >= 1 && x < n;
  const bool xout = lane >= 2 && lane < 2 + TB_XOUT && x < n;
  const unsigned xo = xlive ? x : 0;  // column 0 is zero
  const float sc1 = (float)*g.scale, sc2 = (float)*g.scale2, hd = g.half_dtau;
  const pk kd2 = pk_make(g.kd, g.kd), m6 = pk_make(-6.f, -6.f);
  const unsigned s8 = n * 8, sv = n * (VREAL ? 4 : 8);
  const u64 in0 = (u64)(reinterpret_cast<const pk*>(g.in) + xo), out0 = (u64)(reinterpret_cast<pk*>(g.out) + x);
  const u64 v0 = VREAL ? (u64)(reinterpret_cast<const float*>(g.v) + xo) : (u64)(reinterpret_cast<const pk*>(g.v) + xo);
  auto ylive = [&](int y) { return !EDGE || (y >= 1 && y < n); };
  // row i of level 0 is y0 - 2 + i
  auto zlo = [&](int z) { return (EDGE ? 0LL : (long long)(y0 - 2) * n) + (z >= 1 && z < n ? z * n2 : 0LL); };
  auto erow = [&](int i) { return ylive(y0 - 2 + i) ? (unsigned)(y0 - 2 + i) : 0u; };
  using R0 = std::make_integer_sequence<int, TB_R0>;
  using R1 = std::make_integer_sequence<int, TB_R1>;
  pk A[3][TB_R0], B[3][TB_R1];
  float vx[3][TB_R1], vy[VREAL ? 1 : 3][VREAL ? 1 : TB_R1];
  auto load0 = [&](pk(&a)[TB_R0], int z) {
    const u64 q = in0 + 8 * zlo(z);
    tb_rows([&](auto i) {
      const u64 p = EDGE ? q + (u64)erow(i) * s8 : tb_addr<i()>(q, s8);
      asm volatile("ld.global.nc.b64 %0, [%1];" : "=l"(a[i()]) : "l"(p));
    }, R0{});
  };
  auto loadv = [&](auto kc, int z) {
    constexpr int K = decltype(kc)::value;
    const u64 q = v0 + (VREAL ? 4 : 8) * zlo(z);
    tb_rows([&](auto i) {
      const u64 p = EDGE ? q + (u64)erow(i + 1) * sv : tb_addr<i() + 1>(q, sv);
      if constexpr (VREAL) asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(vx[K][i()]) : "l"(p));
      else asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(vx[K][i()]), "=f"(vy[VREAL ? 0 : K][VREAL ? 0 : i()]) : "l"(p));
    }, R1{});
  };
  // PRE: prefetch into L2 of the warp's own rows, TB_AHEAD planes on, one line a lane: lanes
  // 0-11 take psi (3 lines of 128 bytes cover 32 sites of a row), lanes 12-19 V
  constexpr int TB_AHEAD = 4;
  const int pl = lane < 12 ? lane : lane - 12, prow = min(y0 + (lane < 12 ? pl / 3 : pl >> 1), n - 1);
  const int pcol = min(max(bx * TB_XOUT - 2, 0) + (lane < 12 ? (pl % 3) * 16 : (pl & 1) * (VREAL ? 32 : 16)), n - 1);
  const u64 pre0 = lane < 12 ? (u64)(reinterpret_cast<const pk*>(g.in) + (long long)prow * n + pcol)
                             : (u64)g.v + (VREAL ? 4 : 8) * ((long long)prow * n + pcol);
  const u64 pst = (u64)n2 * (lane < 12 || !VREAL ? 8 : 4);
  // psi_{t+1} of plane p into B[K]: level-0 planes p-1, p, p+1 in A[K], A[K+1], A[K+2] (mod 3)
  // and V of planes p-1, p in v[K+2], v[K]; then psi_{t+2} of plane p-1 from B[K+1], B[K+2], B[K]
  auto plane = [&](auto kc, int p) {
    constexpr int K = decltype(kc)::value, K1 = (K + 1) % 3, K2 = (K + 2) % 3;
    if (p < z1) loadv(std::integral_constant<int, K1>{}, p + 1);
    if constexpr (PRE)
      if (lane < 20 && p + TB_AHEAD < n)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(pre0 + (u64)(p + TB_AHEAD) * pst));
    const bool live1 = xlive && p >= 1 && p < n;
#pragma unroll
    for (int i = 0; i < TB_R1; ++i) {
      const pk c = A[K1][i + 1];
      const pk xm = __shfl_up_sync(0xffffffffu, c, 1), xp = __shfl_down_sync(0xffffffffu, c, 1);
      B[K][i] = tb_site<VREAL>(c, xm, xp, A[K1][i], A[K1][i + 2], A[K][i + 1], A[K2][i + 1], vx[K][i],
                               VREAL ? 0.f : vy[VREAL ? 0 : K][VREAL ? 0 : i], hd, kd2, m6, sc1,
                               live1 && ylive(y0 - 1 + i));
    }
    if (p < z1) load0(A[K], p + 2);
    if (p > z0) {
      const int q = p - 1;
      const u64 dst = out0 + 8 * (q * n2 + (long long)y0 * n);
      tb_rows([&](auto ic) {
        constexpr int i = decltype(ic)::value;
        const pk c = B[K2][i + 1];
        const pk xm = __shfl_up_sync(0xffffffffu, c, 1), xp = __shfl_down_sync(0xffffffffu, c, 1);
        const pk u = tb_site<VREAL>(c, xm, xp, B[K2][i], B[K2][i + 2], B[K1][i + 1], B[K][i + 1], vx[K2][i + 1],
                                    VREAL ? 0.f : vy[VREAL ? 0 : K2][VREAL ? 0 : i + 1], hd, kd2, m6, sc2,
                                    xlive && q >= 1 && ylive(y0 + i));
        const int st = xout && (!EDGE || y0 + i < n);
        asm volatile("{\n .reg .pred p;\n setp.ne.s32 p, %2, 0;\n @p st.global.b64 [%0], %1;\n}\n" ::"l"(
                         tb_addr<i>(dst, s8)), "l"(u), "r"(st) : "memory");
      }, std::make_integer_sequence<int, TB_ROWS>{});
    }
  };
  load0(A[0], z0 - 2);
  load0(A[1], z0 - 1);
  load0(A[2], z0);
  loadv(std::integral_constant<int, 0>{}, z0 - 1);
  for (int p = z0 - 1; p <= z1; p += 3) {
    plane(std::integral_constant<int, 0>{}, p);
    if (p + 1 > z1) break;
    plane(std::integral_constant<int, 1>{}, p + 1);
    if (p + 2 > z1) break;
    plane(std::integral_constant<int, 2>{}, p + 2);
  }
}

template <bool VREAL, bool PRE>
__global__ void __launch_bounds__(32, VREAL ? 16 : 12) stencil_tb_kernel(const __grid_constant__ StencilTbGroup gr) {
  // member of this block: the last i with start[i] <= block
  int member = 0;
  {
    int hi = gr.count - 1;
    while (member < hi) {
      const int mid = (member + hi + 1) >> 1;
      if (gr.start[mid] <= (int)blockIdx.x) member = mid;
      else hi = mid - 1;
    }
  }
  const StencilTbArgs& g = gr.m[member];
  const int nbx = stencil_tb_xtiles(g.n), nby = stencil_tb_ytiles(g.n);
  const int local = (int)blockIdx.x - gr.start[member];
  const int bx = local % nbx, by = (local / nbx) % nby, bz = local / (nbx * nby);
  const int y0 = by * TB_ROWS;
  const int z0 = (int)((long long)bz * g.n / g.nzb), z1 = (int)((long long)(bz + 1) * g.n / g.nzb);
  const bool inner = y0 >= 2 && y0 + TB_ROWS + 2 <= g.n;
  if (inner) stencil_tb_march<VREAL, false, PRE>(g, bx, y0, z0, z1);
  else stencil_tb_march<VREAL, true, PRE>(g, bx, y0, z0, z1);
}

}  // namespace qf
