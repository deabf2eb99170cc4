// FP64 path: spread and gather, one block per particle (the block-per-particle scheme of Appendix C).
//
// GB300 executes two FP64 FMAs per SM and clock, 1/64 of FP32, so both kernels are bound by the FP64
// instructions they issue per window point and are written to issue few of them with full warps; integer
// and shared-memory work beside them is free. The kernel's polynomial P = A + B (dx^2 + dy^2 + dz^2) and
// the torque's cross products are split into one-dimensional tables and per-row coefficients.
//
// * spread: f_c(x) += G alpha_c g(x) + G w_c(x), two FMAs per point and component (Sigma_D = Sigma; two widths take
//   five more per point, from the torque's own row factors);
//   threads take window points in x-fastest order, so the FP64 reductions of a row are contiguous;
// * gather: a thread per window row, eight FMAs per point (the x moments of u), then the row's factors;
//   the six sums are reduced across lanes by halving the values with the lanes (nine additions, not 30).
// Measured at N = 8,192, M_G = 14, torques, Sigma_D = Sigma (64^3), against a thread per row with the full kernel
// at every point and serial reductions: spread 0.76 -> 0.33 ms, gather 1.09 -> 0.47 ms. Six and eight FMAs per
// point at the FP64 rate are 0.21 and 0.29 ms; the rest is the tables, the rows' factors and the last, part-full
// warp of the 196 rows.
// Formulas as in spread_f32.cu and gather_f32.cu; the pair correction is in pair_f64.cu.
#include "fcm_internal.cuh"

namespace fcm {

namespace {

constexpr int kSpread64Threads = 128;
constexpr int kMaxRows = kMaxMG * kMaxMG;

struct Axes64 {
  double d[3][kMaxMG];    // x_g - Y
  double g[3][kMaxMG];    // exp(-d^2/(2 Sigma^2))
  double gd[3][kMaxMG];   // exp(-d^2/(2 Sigma_D^2))
};

// Displacements and Gaussians along the three axes; at[d][j] = wrapped grid index. One pass of the block.
template <bool SAMEW>
__device__ inline void fill_axes(const Geometry<double>& g, const KernelConsts<double>& kc, const Vec4<double>& y,
                                 Axes64& t, int (*at)[kMaxMG]) {
  for (int k = threadIdx.x; k < 3 * g.MG; k += blockDim.x) {
    const int d = k / g.MG, j = k - d * g.MG;
    const double yd = d == 0 ? y.x : (d == 1 ? y.y : y.z);
    const int i0 = window_start_d(g, d, yd);
    const double dd = (double)(i0 + j) * sel3(g.h, d) - yd;
    const double q = -dd * dd;
    const double gs = exp(q * kc.inv2S2);
    t.d[d][j] = dd;
    t.g[d][j] = gs;
    t.gd[d][j] = SAMEW ? gs : exp(q * kc.inv2SD2);
    at[d][j] = pmod(i0 + j, sel3(g.M, d));
  }
}

}  // namespace

template <bool TORQUE, bool SAMEW>
__global__ void __launch_bounds__(kSpread64Threads) spread_bpp_f64(Geometry<double> g, KernelConsts<double> kc,
                                                                   const Vec4<double>* __restrict__ pos,
                                                                   const Vec4<double>* __restrict__ Fv,
                                                                   const Vec4<double>* __restrict__ Tv,
                                                                   double* __restrict__ grid) {
  __shared__ Axes64 t;
  __shared__ int at[3][kMaxMG];
  __shared__ double wx[3][kMaxMG];     // B F'_c d^2 g (+ the torque's d g) along x
  __shared__ double ay[3][kMaxMG], az[3][kMaxMG];   // alpha_c split into its y and z parts
  __shared__ Vec4<double> row[kMaxRows];   // {G alpha_x, G alpha_y, G alpha_z, G}
  constexpr bool TWO = TORQUE && !SAMEW;   // the torque has a Gaussian of its own, H = g_D(dy) g_D(dz)
  __shared__ Vec4<double> trow[TWO ? kMaxRows : 1];   // H {U'y dz - U'z dy, -U'x dz, U'x dy, 1}
  __shared__ double tx[2][TWO ? kMaxMG : 1];          // U'z d g_D and -U'y d g_D along x
  __shared__ long long off[kMaxRows];
  const int p = blockIdx.x;
  const Vec4<double> y = pos[p];
  const Vec4<double> f = Fv[p];
  Vec4<double> u = {0.0, 0.0, 0.0, 0.0};
  if (TORQUE) u = Tv[p];
  fill_axes<SAMEW || !TORQUE>(g, kc, y, t, at);
  __syncthreads();
  const int MG = g.MG;
  const double Fx = kc.nrm * f.x, Fy = kc.nrm * f.y, Fz = kc.nrm * f.z;
  const double Ux = kc.tq * u.x, Uy = kc.tq * u.y, Uz = kc.tq * u.z;
  constexpr bool FOLD = TORQUE && SAMEW;   // the torque shares the force's Gaussian
  for (int k = threadIdx.x; k < 3 * MG; k += blockDim.x) {
    const int d = k / MG, j = k - d * MG;
    const double dd = t.d[d][j], bq = kc.B * dd * dd;
    if (d == 0) {
      if (TWO) {
        tx[0][j] = Uz * dd * t.gd[0][j];
        tx[1][j] = -Uy * dd * t.gd[0][j];
      }
      const double q = bq * t.g[0][j], dg = dd * t.g[0][j];
      wx[0][j] = Fx * q;
      wx[1][j] = FOLD ? fma(Uz, dg, Fy * q) : Fy * q;
      wx[2][j] = FOLD ? fma(-Uy, dg, Fz * q) : Fz * q;
    } else if (d == 1) {
      const double P = kc.A + bq;
      ay[0][j] = FOLD ? fma(-Uz, dd, Fx * P) : Fx * P;
      ay[1][j] = Fy * P;
      ay[2][j] = FOLD ? fma(Ux, dd, Fz * P) : Fz * P;
    } else {
      az[0][j] = FOLD ? fma(Uy, dd, Fx * bq) : Fx * bq;
      az[1][j] = FOLD ? fma(-Ux, dd, Fy * bq) : Fy * bq;
      az[2][j] = Fz * bq;
    }
  }
  __syncthreads();
  for (int r = threadIdx.x; r < MG * MG; r += blockDim.x) {
    const int jz = r / MG, jy = r - jz * MG;
    const double G = t.g[1][jy] * t.g[2][jz];
    row[r] = {G * (ay[0][jy] + az[0][jz]), G * (ay[1][jy] + az[1][jz]), G * (ay[2][jy] + az[2][jz]), G};
    if (TWO) {
      const double H = t.gd[1][jy] * t.gd[2][jz], dy = t.d[1][jy], dz = t.d[2][jz];
      trow[r] = {H * fma(Uy, dz, -Uz * dy), -H * Ux * dz, H * Ux * dy, H};
    }
    off[r] = ((long long)at[2][jz] * g.M[1] + at[1][jy]) * g.M[0];
  }
  __syncthreads();
  const size_t Mtot = (size_t)g.M[0] * g.M[1] * g.M[2];
  // window points e = r M_G + j in x-fastest order
  const int dr = kSpread64Threads / MG, dj = kSpread64Threads - dr * MG;
  int r = threadIdx.x / MG, j = threadIdx.x - r * MG;
  while (r < MG * MG) {
    const Vec4<double> a = row[r];
    const double gx = t.g[0][j];
    double fx = fma(a.w, wx[0][j], a.x * gx);
    double fy = fma(a.w, wx[1][j], a.y * gx);
    double fz = fma(a.w, wx[2][j], a.z * gx);
    if (TWO) {
      const Vec4<double> c = trow[r];
      const double gd = t.gd[0][j];
      fx = fma(c.x, gd, fx);
      fy = fma(c.y, gd, fma(c.w, tx[0][j], fy));
      fz = fma(c.z, gd, fma(c.w, tx[1][j], fz));
    }
    double* q = grid + off[r] + at[0][j];
    atomicAdd(q, fx);
    atomicAdd(q + Mtot, fy);
    atomicAdd(q + 2 * Mtot, fz);
    r += dr;
    j += dj;
    if (j >= MG) { j -= MG; ++r; }
  }
}

namespace {

// Sums v[0 .. 7] over the warp: lane l ends with the total of v[l & 7] (lanes 0 .. 7 hold them all). Each step
// halves the values a lane carries, so 4 + 2 + 1 + 1 + 1 additions replace eight five-step trees.
__device__ inline double warp_sum8(double (&v)[8]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int half = 4; half >= 1; half >>= 1) {
    const bool up = lane & half;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k < half) {
        const double keep = up ? v[k + half] : v[k], give = up ? v[k] : v[k + half];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, give, half);
      }
    }
  }
  double s = v[0];
  s += __shfl_xor_sync(0xffffffffu, s, 8);
  s += __shfl_xor_sync(0xffffffffu, s, 16);
  return s;
}

}  // namespace

template <bool TORQUE, bool SAMEW>
__global__ void __launch_bounds__(256) gather_bpp_f64(Geometry<double> g, KernelConsts<double> kc,
                                                      const Vec4<double>* __restrict__ pos,
                                                      const double* __restrict__ grid,
                                                      const double* __restrict__ upair,
                                                      const double* __restrict__ wpair,
                                                      double* __restrict__ U, double* __restrict__ W) {
  __shared__ Axes64 t;
  __shared__ int at[3][kMaxMG];
  __shared__ double mx[2][kMaxMG];   // d^2 g and d g_D along x
  __shared__ double red[8][8];
  const int p = blockIdx.x;
  const Vec4<double> y = pos[p];
  fill_axes<SAMEW || !TORQUE>(g, kc, y, t, at);
  __syncthreads();
  const int MG = g.MG;
  if (threadIdx.x < MG) {
    const double d = t.d[0][threadIdx.x];
    mx[0][threadIdx.x] = d * d * t.g[0][threadIdx.x];
    if (TORQUE) mx[1][threadIdx.x] = d * t.gd[0][threadIdx.x];
  }
  __syncthreads();
  const size_t Mtot = (size_t)g.M[0] * g.M[1] * g.M[2];
  double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int r = threadIdx.x; r < MG * MG; r += blockDim.x) {
    const int jz = r / MG, jy = r - jz * MG;
    const double* row = grid + ((size_t)at[2][jz] * g.M[1] + at[1][jy]) * g.M[0];
    double s0[3] = {0, 0, 0}, s2[3] = {0, 0, 0}, e0[3] = {0, 0, 0}, e1y = 0, e1z = 0;
#pragma unroll 2
    for (int j = 0; j < MG; ++j) {
      const int gx = at[0][j];
      const double ux = row[gx], uy = row[Mtot + gx], uz = row[2 * Mtot + gx];
      const double g0 = t.g[0][j], g2 = mx[0][j];
      s0[0] = fma(g0, ux, s0[0]); s0[1] = fma(g0, uy, s0[1]); s0[2] = fma(g0, uz, s0[2]);
      s2[0] = fma(g2, ux, s2[0]); s2[1] = fma(g2, uy, s2[1]); s2[2] = fma(g2, uz, s2[2]);
      if (TORQUE) {
        const double g1 = mx[1][j];
        e1y = fma(g1, uy, e1y);
        e1z = fma(g1, uz, e1z);
        if (!SAMEW) {
          const double gd = t.gd[0][j];
          e0[0] = fma(gd, ux, e0[0]); e0[1] = fma(gd, uy, e0[1]); e0[2] = fma(gd, uz, e0[2]);
        }
      }
    }
    const double dy = t.d[1][jy], dz = t.d[2][jz];
    const double G = t.g[1][jy] * t.g[2][jz];
    const double GB = G * kc.B, GQ = fma(GB, fma(dy, dy, dz * dz), G * kc.A);
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[c] = fma(GQ, s0[c], fma(GB, s2[c], acc[c]));
    if (TORQUE) {
      const double H = SAMEW ? G : t.gd[1][jy] * t.gd[2][jz];
      const double* e = SAMEW ? s0 : e0;
      acc[3] = fma(H, fma(dy, e[2], -dz * e[1]), acc[3]);
      acc[4] = fma(H, fma(dz, e[0], -e1z), acc[4]);
      acc[5] = fma(H, fma(-dy, e[0], e1y), acc[5]);
    }
  }
  const double s = warp_sum8(acc);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane < 8) red[wid][lane] = s;
  __syncthreads();
  if (threadIdx.x < (TORQUE ? 6 : 3)) {
    double v = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) v += red[k][threadIdx.x];
    const size_t o = 3 * (size_t)index_from_w(y.w);
    const int c = threadIdx.x;
    if (c < 3) U[o + c] = kc.h3 * kc.nrm * v + (upair ? upair[o + c] : 0.0);
    else if (W) W[o + c - 3] = kc.h3 * kc.tq * v + (wpair ? wpair[o + c - 3] : 0.0);
  }
}

void launch_spread_f64(const Geometry<double>& g, const KernelConsts<double>& kc, bool torque,
                       const BinBuffers& b, int n, double* grid, cudaStream_t s, long long* launches) {
  if (n <= 0) return;
  auto k = !torque ? spread_bpp_f64<false, true> : (kc.same_width ? spread_bpp_f64<true, true> : spread_bpp_f64<true, false>);
  k<<<n, kSpread64Threads, 0, s>>>(g, kc, (const Vec4<double>*)b.t_pos, (const Vec4<double>*)b.t_F,
                                   (const Vec4<double>*)b.t_T, grid);
  *launches += 1;
}

void launch_gather_f64(const Geometry<double>& g, const KernelConsts<double>& kc, bool torque,
                       const BinBuffers& b, int n, const double* grid, const double* up, const double* wp,
                       double* U, double* W, cudaStream_t s, long long* launches) {
  if (n <= 0) return;
  // a thread per window row in as few rounds of at most 256 threads as there are, whole warps
  const int rows = g.MG * g.MG, rounds = (rows + 255) / 256;
  const int threads = ((rows + rounds - 1) / rounds + 31) / 32 * 32;
  auto k = !torque ? gather_bpp_f64<false, true> : (kc.same_width ? gather_bpp_f64<true, true> : gather_bpp_f64<true, false>);
  k<<<n, threads, 0, s>>>(g, kc, (const Vec4<double>*)b.t_pos, grid, up, wp, U, W);
  *launches += 1;
}

}  // namespace fcm
