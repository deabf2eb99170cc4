// FP64 pairwise correction (Section 4 step 6, eq. correction_VF / WF / WT, Appendix B).
//
// GB300 executes two FP64 FMAs per SM and clock (1/64 of FP32), so the pair stage is bound by the number
// of FP64 instructions per pair and by how many of a warp's lanes they serve. The closed form takes six
// erfc and six exp per ordered pair, several hundred FP64 instructions. Here:
// * the five radial coefficients are polynomials of degree 5 in s = r^2 on intervals that split each
//   octave of s into 128 (even functions of r: no square root), interpolated at Chebyshev points of the
//   closed form in FP64 when the handle is made: 25 FMAs. On an interval |ds| / s <= 2^-8, so for a
//   Gaussian exp(-s / 4 w^2) at s = 10 w^2 the sixth-order remainder is below 1e-16 of the value;
// * each unordered pair is evaluated once for both particles (half shell of cells);
// * candidates are tested in FP32 (with a margin that covers the rounding of positions and of the test),
//   and the pairs that pass are queued by (i, j) across particles, so the FP64 instructions run with
//   32 pairs per warp whatever the number of neighbours; the queue evaluates the FP64 cutoff again;
// * sums go to the output with FP64 reductions in L2 (the order of the additions is not fixed).
// Measured against a thread per particle with the closed form over 27 cells: N = 8,192 at phi = 5% (146
// neighbours, torques) 18.7 -> 0.25 ms; N = 1,000 with 20 neighbours, forces only, 1.89 -> 0.029 ms. About 113
// FP64 instructions per pair of 32 lanes at 64 clocks each bound the first: 0.11 ms at full lanes and balance.
#include <cstring>

#include "pair_common.cuh"

namespace fcm {

namespace {

constexpr unsigned kAll = 0xffffffffu;
constexpr int kWarps64 = 4;
constexpr int kChunk64 = 512;      // staged candidates per pass
constexpr int kQueue64 = 64;

constexpr int kDeg = kPair64Degree;
constexpr int kShiftBits = 20 - kPair64Bits;   // high-word bits below an interval's index

__device__ inline int interval_of(double s) { return __double2hiint(s) >> kShiftBits; }
__device__ inline double interval_mid(int idx) {
  return __hiloint2double((idx << kShiftBits) | (1 << (kShiftBits - 1)), 0);
}

// Coefficients of interval base + k: Chebyshev interpolation of the closed form at kDeg + 1 points,
// expanded in powers of (s - mid).
__global__ void __launch_bounds__(64) build_table64(PairConsts<double> pc, int base, int n, double* __restrict__ coef) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const double mid = interval_mid(base + k);
  const double lo = __hiloint2double((base + k) << kShiftBits, 0);
  const double w = mid - lo;   // a power of two
  PairConsts<double> c = pc;
  double f[5][kDeg + 1], ch[5][kDeg + 1];
  for (int j = 0; j <= kDeg; ++j) {
    const double x = cospi((j + 0.5) / (kDeg + 1));
    pair_coeffs<double>(mid + w * x, c, f[0][j], f[1][j], f[2][j], f[3][j], f[4][j]);
  }
  for (int q = 0; q < 5; ++q)
    for (int m = 0; m <= kDeg; ++m) {
      double s = 0.0;
      for (int j = 0; j <= kDeg; ++j) s += f[q][j] * cospi(m * (j + 0.5) / (kDeg + 1));
      ch[q][m] = s * (m == 0 ? 1.0 : 2.0) / (kDeg + 1);
    }
  // T_0 .. T_5 in powers of x
  static_assert(kDeg == 5, "power form of T_0 .. T_5");
  for (int q = 0; q < 5; ++q) {
    const double* a = ch[q];
    const double p[6] = {a[0] - a[2] + a[4], a[1] - 3.0 * a[3] + 5.0 * a[5], 2.0 * a[2] - 8.0 * a[4],
                         4.0 * a[3] - 20.0 * a[5], 8.0 * a[4], 16.0 * a[5]};
    double iw = 1.0;
    double* out = coef + ((size_t)k * 5 + q) * (kDeg + 1);
    for (int m = 0; m <= kDeg; ++m) {
      out[m] = p[m] * iw;
      iw /= w;
    }
  }
}

__device__ inline double poly64(const double* __restrict__ c, double t) {
  double s = __ldg(c + kDeg);
#pragma unroll
  for (int m = kDeg - 1; m >= 0; --m) s = fma(s, t, __ldg(c + m));
  return s;
}

// d minus the box edge nearest to it, as d > L/2 ? d - L : (d < -L/2 ? d + L : d); the comparison is made on
// the high words (integer pipe), and in FP64 only where they are equal.
__device__ inline double nearest_image(double d, double L) {
  const double half = 0.5 * L;
  const int hd = __double2hiint(d), ha = hd & 0x7fffffff, hh = __double2hiint(half);
  bool out = ha > hh;
  if (ha == hh) out = fabs(d) > half;
  return out ? (hd < 0 ? d + L : d - L) : d;
}

template <bool TORQUE>
__device__ __forceinline__ void eval_pair64(const Geometry<double>& g, const PairConsts<double>& pc,
                                            const PairTable64& tab, const Vec4<double>* __restrict__ cpos,
                                            const Vec4<double>* __restrict__ cF, const Vec4<double>* __restrict__ cT,
                                            int i, int j, double* __restrict__ Uo, double* __restrict__ Wo) {
  const Vec4<double> yi = cpos[i], yj = cpos[j];
  const double dx = nearest_image(yi.x - yj.x, g.L[0]);
  const double dy = nearest_image(yi.y - yj.y, g.L[1]);
  const double dz = nearest_image(yi.z - yj.z, g.L[2]);
  const double s = fma(dx, dx, fma(dy, dy, dz * dz));
  // both sides are positive, so the order of the values is the order of the bit patterns
  if (!(__double_as_longlong(s) < __double_as_longlong(pc.rc2))) return;
  double al, bt, cr = 0.0, gm = 0.0, dl = 0.0;
  if (s < pc.rs2) {
    pair_coeffs<double>(s, pc, al, bt, cr, gm, dl);   // the Taylor branch
  } else {
    const int idx = min(max(interval_of(s) - tab.base, 0), tab.n - 1);
    const double* c = tab.coef + (size_t)idx * 5 * (kDeg + 1);
    const double t = s - interval_mid(idx + tab.base);
    al = poly64(c, t);
    bt = poly64(c + (kDeg + 1), t);
    if (TORQUE) {
      cr = poly64(c + 2 * (kDeg + 1), t);
      gm = poly64(c + 3 * (kDeg + 1), t);
      dl = poly64(c + 4 * (kDeg + 1), t);
    }
  }
  const Vec4<double> Fi = cF[i], Fj = cF[j];
  const double bj = bt * fma(dx, Fj.x, fma(dy, Fj.y, dz * Fj.z));
  const double bi = bt * fma(dx, Fi.x, fma(dy, Fi.y, dz * Fi.z));
  double u[3] = {fma(bj, dx, al * Fj.x), fma(bj, dy, al * Fj.y), fma(bj, dz, al * Fj.z)};
  double v[3] = {fma(bi, dx, al * Fi.x), fma(bi, dy, al * Fi.y), fma(bi, dz, al * Fi.z)};
  const size_t oi = 3 * (size_t)index_from_w(yi.w), oj = 3 * (size_t)index_from_w(yj.w);
  if (TORQUE) {
    const Vec4<double> Ti = cT[i], Tj = cT[j];
    const double cx = cr * dx, cy = cr * dy, cz = cr * dz;
    // U_i += cr (T_j x x), U_j -= cr (T_i x x)
    u[0] = fma(Tj.y, cz, fma(-Tj.z, cy, u[0]));
    u[1] = fma(Tj.z, cx, fma(-Tj.x, cz, u[1]));
    u[2] = fma(Tj.x, cy, fma(-Tj.y, cx, u[2]));
    v[0] = fma(-Ti.y, cz, fma(Ti.z, cy, v[0]));
    v[1] = fma(-Ti.z, cx, fma(Ti.x, cz, v[1]));
    v[2] = fma(-Ti.x, cy, fma(Ti.y, cx, v[2]));
    if (Wo) {
      const double ej = dl * fma(dx, Tj.x, fma(dy, Tj.y, dz * Tj.z));
      const double ei = dl * fma(dx, Ti.x, fma(dy, Ti.y, dz * Ti.z));
      // W_i += cr (F_j x x) + gm T_j + dl x (x.T_j), W_j the same with x -> -x
      atomicAdd(Wo + oi + 0, fma(Fj.y, cz, fma(-Fj.z, cy, fma(ej, dx, gm * Tj.x))));
      atomicAdd(Wo + oi + 1, fma(Fj.z, cx, fma(-Fj.x, cz, fma(ej, dy, gm * Tj.y))));
      atomicAdd(Wo + oi + 2, fma(Fj.x, cy, fma(-Fj.y, cx, fma(ej, dz, gm * Tj.z))));
      atomicAdd(Wo + oj + 0, fma(-Fi.y, cz, fma(Fi.z, cy, fma(ei, dx, gm * Ti.x))));
      atomicAdd(Wo + oj + 1, fma(-Fi.z, cx, fma(Fi.x, cz, fma(ei, dy, gm * Ti.y))));
      atomicAdd(Wo + oj + 2, fma(-Fi.x, cy, fma(Fi.y, cx, fma(ei, dz, gm * Ti.z))));
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    atomicAdd(Uo + oi + c, u[c]);
    atomicAdd(Uo + oj + c, v[c]);
  }
}

// The particles i of the cell with (i - first) mod parts == part, against the half shell.
template <bool TORQUE>
__device__ __forceinline__ void half_cell64(const Geometry<double>& g, const PairConsts<double>& pc,
                                            const PairTable64& tab, double inv, float rc2f,
                                            const Vec4<double>* __restrict__ cpos, const Vec4<double>* __restrict__ cF,
                                            const Vec4<double>* __restrict__ cT, const int* __restrict__ cstart,
                                            double* __restrict__ Uo, double* __restrict__ Wo, int cell, int part,
                                            int parts) {
  __shared__ float4 spos[kChunk64];       // x, y, z over the longest box edge in FP32, cell-sorted index
  __shared__ int2 queue[kWarps64][kQueue64];
  __shared__ int meta[2 * kPieces + 2];
  __shared__ float4 shift[kPieces];
  const int i_begin = cstart[cell], i_end = cstart[cell + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp == 0) half_shell_pieces(g, cell, cstart, meta, shift);
  __syncthreads();
  const int total = meta[2 * kPieces + 1];
  const float Lx = (float)(g.L[0] * inv), Ly = (float)(g.L[1] * inv), Lz = (float)(g.L[2] * inv);
  const unsigned lt = (1u << lane) - 1u;
  int2* q = queue[warp];
  int qn = 0;   // queued pairs (the same in every lane)
  for (int cb = 0; cb < total; cb += kChunk64) {
    const int nc = min(kChunk64, total - cb);
    __syncthreads();
    for (int p = 0; p < kPieces; ++p) {
      const int lo = max(meta[2 * p + 1], cb), hi = min(meta[2 * p + 3], cb + nc);
      const int src = meta[2 * p] + (lo - meta[2 * p + 1]);
      for (int k = threadIdx.x; k < hi - lo; k += blockDim.x) {
        const Vec4<double> y = cpos[src + k];
        spos[lo - cb + k] = make_float4((float)(y.x * inv), (float)(y.y * inv), (float)(y.z * inv), __int_as_float(src + k));
      }
    }
    __syncthreads();
    for (int i = i_begin + part + parts * warp; i < i_end; i += parts * kWarps64) {
      const Vec4<double> yd = cpos[i];
      const float yx = (float)(yd.x * inv), yy = (float)(yd.y * inv), yz = (float)(yd.z * inv);
      if (cb == 0 && lane < 3) {   // the self terms of Appendix B
        const size_t o = 3 * (size_t)index_from_w(yd.w);
        const Vec4<double> F = cF[i];
        atomicAdd(Uo + o + lane, pc.selfVF * (lane == 0 ? F.x : (lane == 1 ? F.y : F.z)));
        if (TORQUE && Wo) {
          const Vec4<double> T = cT[i];
          atomicAdd(Wo + o + lane, pc.selfWT * (lane == 0 ? T.x : (lane == 1 ? T.y : T.z)));
        }
      }
      const int start = max(i - i_begin + 1 - cb, 0);   // the own cell is staged first: later slots only
      for (int base = start; base < nc; base += 32) {
        const int k = base + lane;
        bool hit = false;
        int j = 0;
        if (k < nc) {
          const float4 y = spos[k];
          float dx = fabsf(yx - y.x), dy = fabsf(yy - y.y), dz = fabsf(yz - y.z);
          dx = fminf(dx, fabsf(Lx - dx));
          dy = fminf(dy, fabsf(Ly - dy));
          dz = fminf(dz, fabsf(Lz - dz));
          hit = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < rc2f;
          j = __float_as_int(y.w);
        }
        const unsigned m = __ballot_sync(kAll, hit);
        if (m == 0u) continue;
        if (hit) q[qn + __popc(m & lt)] = make_int2(i, j);   // qn < 32 here, so the slot is < 64
        qn += __popc(m);
        if (qn >= 32) {
          __syncwarp();
          const int2 e = q[lane];
          eval_pair64<TORQUE>(g, pc, tab, cpos, cF, cT, e.x, e.y, Uo, Wo);
          __syncwarp();
          if (lane < qn - 32) q[lane] = q[32 + lane];   // the overflow moves to the front
          qn -= 32;
          __syncwarp();
        }
      }
    }
  }
  __syncwarp();
  if (lane < qn) {
    const int2 e = q[lane];
    eval_pair64<TORQUE>(g, pc, tab, cpos, cF, cT, e.x, e.y, Uo, Wo);
  }
}

// CTA b takes part b mod `parts` of cell b / parts, unless the cell is crowded. The last `sharers` CTAs then share the
// crowded cells' parts, which the binning's scan lists (kSplit64 CTAs to a listed part): 20,000 particles in one cell of
// many would otherwise run in one CTA (1,329 ms; a thread per particle over 27 cells, the kernel before this one, 942 ms;
// so 8.2 ms).
constexpr int kSplit64 = 4;

template <bool TORQUE>
__global__ void __launch_bounds__(kWarps64 * 32) pair_half_f64(Geometry<double> g, PairConsts<double> pc,
                                                               PairTable64 tab, double inv, float rc2f,
                                                               const Vec4<double>* __restrict__ cpos,
                                                               const Vec4<double>* __restrict__ cF,
                                                               const Vec4<double>* __restrict__ cT,
                                                               const int* __restrict__ cstart,
                                                               double* __restrict__ Uo, double* __restrict__ Wo,
                                                               const int* __restrict__ crowd, int ncells, int nparts,
                                                               int sharers) {
  int cell = blockIdx.x / nparts, part = blockIdx.x - cell * nparts, parts = nparts;
  const int place = (int)blockIdx.x - ((int)gridDim.x - sharers);   // among the sharers
  bool own = cell < ncells;   // first the CTA's own cell, then every sharers-th item
  for (int k = own ? place - sharers : place;; k += sharers) {
    if (!own) {
      if (k < 0 || k >= kSplit64 * crowd[1]) return;
      cell = crowd[2 + 2 * (k / kSplit64)];
      part = kSplit64 * crowd[3 + 2 * (k / kSplit64)] + k % kSplit64;
    }
    const int n = cstart[cell + 1] - cstart[cell];
    if (!own) parts = kSplit64 * crowd_parts(n);
    if (part < n && (!own || n <= kCrowdCell))
      half_cell64<TORQUE>(g, pc, tab, inv, rc2f, cpos, cF, cT, cstart, Uo, Wo, cell, part, parts);
    own = false;
    __syncthreads();   // the next part reuses the shared memory
  }
}

}  // namespace

void pair_table64_range(double rs2, double rc2, int* base, int* n) {
  auto idx = [](double s) {
    uint64_t b;
    memcpy(&b, &s, sizeof(b));
    return (int)((b >> 32) >> kShiftBits);
  };
  *base = idx(rs2);
  *n = idx(std::max(rc2, rs2)) - *base + 1;
}

void launch_pair_table64(const PairConsts<double>& pc, const PairTable64& tab, double* coef, cudaStream_t s) {
  PairConsts<double> c = pc;
  c.rs2 = 0.0;   // the closed form throughout the tabulated range
  build_table64<<<(tab.n + 63) / 64, 64, 0, s>>>(c, tab.base, tab.n, coef);
}

void launch_pair_f64(const Geometry<double>& g, const PairConsts<double>& pc, const PairTable64& tab, bool torque,
                     const BinBuffers& b, int n, double* upair, double* wpair, cudaStream_t s, long long* launches) {
  if (n <= 0) return;
  launch_zero(upair, sizeof(double) * 3 * (size_t)n, s, launches);
  if (torque && wpair) launch_zero(wpair, sizeof(double) * 3 * (size_t)n, s, launches);
  // FP32 candidate test over the longest edge: positions and differences carry at most 2^-22, the square 2^-22 of itself
  const double Lmax = std::max(g.L[0], std::max(g.L[1], g.L[2]));
  const double reach = std::sqrt(pc.rc2) / Lmax + 2e-6;
  const float rc2f = (float)(reach * reach * (1.0 + 1e-5));
  // parts of a cell: enough CTAs for four per SM when the cells are few
  const int parts = std::min(16, std::max(1, (4 * device_sm_count() + b.ncells - 1) / b.ncells));
  const int sharers = std::min(4 * device_sm_count(), kSplit64 * crowd_items(n)), grid = std::max(b.ncells * parts, sharers);
  const Vec4<double>* pos = (const Vec4<double>*)b.c_pos;
  const Vec4<double>* F = (const Vec4<double>*)b.c_F;
  const Vec4<double>* T = (const Vec4<double>*)b.c_T;
  if (torque)
    pair_half_f64<true><<<grid, kWarps64 * 32, 0, s>>>(g, pc, tab, 1.0 / Lmax, rc2f, pos, F, T, b.cell_start,
                                                            upair, wpair, b.crowd, b.ncells, parts, sharers);
  else
    pair_half_f64<false><<<grid, kWarps64 * 32, 0, s>>>(g, pc, tab, 1.0 / Lmax, rc2f, pos, F, T, b.cell_start,
                                                            upair, wpair, b.crowd, b.ncells, parts, sharers);
  *launches += 1;
}

}  // namespace fcm
