// FP32 pairwise correction (Section 4 step 6, eq. correction_VF / WF / WT, Appendix B).
//
// For particle n and every m with minimum-image r = |Y_n - Y_m| < r_c:
//   U_n += al F_m + bt x (x.F_m) + cr (T_m x x)
//   W_n += cr (F_m x x) + gm T_m + dl x (x.T_m)
// with x = Y_n - Y_m and radial coefficients al .. dl, plus the self correction. Each unordered pair is
// evaluated once: the coefficients depend on r only and the partner's terms follow from x -> -x. One CTA
// per pair cell stages its own cell and a half shell of 13 neighbour cells (pair_common.cuh).
//
// What bounds it: a candidate within r_c costs about 120 FP32 instructions, but a kernel that takes one
// particle at a time and reads everything else per pair (partner, five table entries at random r, six
// shared-memory atomics, which are compare-and-swap loops) is bound by shared-memory and L1 wavefronts,
// about 170 of them per 32 pairs. So:
// * a warp takes four particles at once (a cluster, consecutive in the octant order of their cell, hence
//   close together). Lanes test 32 candidates against all four; candidates within r_c of any are queued, and a
//   pass of 32 queued partners evaluates 4 x 32 pairs from registers. At 5% (146 neighbours) 61% of those are
//   within r_c; one load of the partner and one addition of its sums serve four pairs;
// * beyond a radius r_near the coefficients are exp(-r^2 / 4 Sigma^2) times polynomials in 1/r (degree 11 for al, 9 for
//   the others), fitted to the closed form in FP64 when the handle is made (weighted minimax, error below 1e-9 of
//   the self mobility and FP32 rounding; r_near is the smallest radius at which the fit reaches that, 2.1 to 3.0
//   Sigma): 47 FMAs with constant operands instead of 20 random 16-byte reads per quarter warp;
// * closer pairs (5%) go to a second queue, evaluated with the piecewise-cubic table (Taylor series below
//   sigma/2, which covers coincident points). Where no such fit exists (r_near above 0.6 r_c, Sigma_D far from
//   Sigma) and in cells that see a load that is not finite (or above 1e18), whose product with a masked pair's zero is NaN,
//   every pair goes that way;
// * partners' sums are added to per-particle accumulators in cell order with 16-byte reductions in L2 (one for
//   U, one for W: a reduction costs the same for one float or four), the cluster's sums after a halving
//   reduction across lanes; a small kernel brings them to input order. The order of the additions is not fixed;
// * a cell of more than kCrowdCell particles is crowded: it is listed in parts by the binning's scan, which the last CTAs
//   of the launch share out when they have done their own cells, and its sums are reduced in FP64, six reductions instead
//   of two. A particle receives one addition per cluster that meets it. The 30 of a suspension (5%, 146 neighbours) cost
//   less than the coefficients' rounding; hundreds of them do not, and FP64 throughout costs all others 10%. Error of U's
//   pair part against 64 bits (rms, of 1e-9) with one FP32 sum per chunk of candidates and cell, compensated for a
//   particle's own pairs / FP32 reductions alone / FP64 in crowded cells: 65,536 at 5% 190 / 188 / 185, 20,000 with 640
//   neighbours 245 / 282 / 216, 4,000 in one cell 149 / 203 / 146. Sharing out keeps a suspension that fills a corner
//   of its box from running in a few CTAs: 65,536 in 125 cells 2.76 / 3.58 / 0.69 ms, 4,000 in one cell 11.9 / 9.3 / 0.21 ms.
// Measured against one particle at a time, tables and shared-memory atomics: 32 systems of 65,536 at 5%, torques,
// 4.04 -> 2.82 ms; 1,048,576 at 10% 2.64 -> 1.77 ms; 122,231 at 0.8%, forces only, 153 -> 100 us; without a fit (Sigma_D =
// 1.27 Sigma, every pair by the table) 65,536 at 5% 122 -> 117 us. Now 1,023 instructions per particle, the schedulers
// issue 59% of the time and the FMA pipe is busy 46%.
#include "pair_common.cuh"

namespace fcm {

namespace {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kHalfChunk = 640;   // staged candidates; above the half-shell count of the 5% suspension (about 530)
static_assert(kHalfChunk % 32 == 0, "candidate chunks are padded to whole 32-candidate passes");
constexpr int kCluster = 4;
constexpr int kQueue = 64;                      // fewer than 32 left over, 32 of a pass
constexpr int kNearQueue = 32 + 32 * kCluster;  // fewer than 32 left over, all pairs of a pass

// CTAs per SM that the register file is split for, by warps of a CTA and by the sums a thread keeps (128 registers, 80 for
// four warps without torques); the shared memory leaves six of two warps with torques.
__host__ __device__ constexpr int cell_blocks(int warps, bool torque) { return warps == 2 ? 8 : (torque ? 4 : 6); }

template <bool TORQUE, int WARPS>
constexpr size_t cluster_smem() {
  return sizeof(float4) * (size_t)kHalfChunk * (TORQUE ? 3 : 2) + sizeof(float4) * 3 * kCluster * WARPS +
         sizeof(int) * (kHalfChunk + WARPS * (kQueue + kNearQueue + 4)) + sizeof(int) * (2 * kPieces + 4) +
         sizeof(float4) * kPieces;
}

__device__ inline float nearest(float d, float L) {
  if (d > 0.5f * L) d -= L;
  else if (d < -0.5f * L) d += L;
  return d;
}

// Loads whose products with a masked pair's separation (at most 2e18) and zero coefficient are zero.
__device__ inline bool bounded3(float4 v) { return fabsf(v.x) < 1e18f && fabsf(v.y) < 1e18f && fabsf(v.z) < 1e18f; }

__device__ __forceinline__ void red4(float4* p, float a, float b, float c) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(0.f) : "memory");
}

// Three sums to the accumulators of particle k, U's (w = 0) or W's (w = 1).
template <bool CROWDED>
__device__ __forceinline__ void add_sums(float4* psum, double* psum64, int k, int w, float a, float b, float c) {
  if (CROWDED) {
    double* q = psum64 + 6 * (size_t)k + 3 * w;
    atomicAdd(q, (double)a);
    atomicAdd(q + 1, (double)b);
    atomicAdd(q + 2, (double)c);
  } else {
    red4(psum + 2 * (size_t)k + w, a, b, c);
  }
}

template <int F>
__device__ __forceinline__ float poly_eval(const PairPoly& p, float t) {
  constexpr int D = pair_poly_degree(F);
  float s = p.c[F][D];
#pragma unroll
  for (int m = D - 1; m >= 0; --m) s = fmaf(s, t, p.c[F][m]);
  return s;
}

__device__ __forceinline__ float exp2_approx(float v) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}
// 1 / sqrt(v) of both halves: the approximation (2^-22.9) and one Newton step, r + r (1 - v r^2) / 2.
__device__ __forceinline__ float2 rsqrt2(float2 v) {
  float2 r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(v.x));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(v.y));
  const float2 e = __ffma2_rn(make_float2(-v.x, -v.y), __fmul2_rn(r, r), make_float2(1.f, 1.f));
  return __ffma2_rn(__fmul2_rn(r, make_float2(0.5f, 0.5f)), e, r);
}

// Halves the N values a lane carries with the lanes at distance `o`: a lane keeps the upper half where its bit is set.
template <int N>
__device__ __forceinline__ void halve(float* v, int o) {
  const bool up = threadIdx.x & o;
#pragma unroll
  for (int k = 0; k < N / 2; ++k) {
    const float keep = up ? v[k + N / 2] : v[k], give = up ? v[k] : v[k + N / 2];
    v[k] = keep + __shfl_xor_sync(kFullMask, give, o);
  }
}

__device__ __forceinline__ float2 two(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 dot2(float2 ax, float2 ay, float2 az, float2 bx, float2 by, float2 bz) {
  return fma2(ax, bx, fma2(ay, by, mul2(az, bz)));
}

}  // namespace

// The pairs of a cell's particles with themselves and with the half shell: of all of them, or of a crowded cell's clusters
// of one part (every crowd_parts-th WARPS of them).
template <bool TORQUE, bool SHIFT, int WARPS, bool CROWDED>
__device__ __forceinline__ void cell_pairs(const Geometry<float>& g, const PairConsts<float>& pc, const PairTable& tab,
                                           const PairPoly& poly, const float4* __restrict__ cpos,
                                           const float4* __restrict__ cF, const float4* __restrict__ cT,
                                           const int* __restrict__ cstart, float4* __restrict__ psum,
                                           double* __restrict__ psum64, int cell, int part) {
  constexpr int V = TORQUE ? 6 : 3;   // sums per particle
  constexpr int W2 = TORQUE ? 9 : 6;  // values per particle of a cluster: position, force, torque
  extern __shared__ float4 sm4[];
  float4* spos = sm4;                 // position from the cell's corner; w: r_c^2 (with margin) - |position|^2
  float4* sF = spos + kHalfChunk;
  float4* sT = sF + kHalfChunk;
  const int i_begin = cstart[cell], i_end = cstart[cell + 1];
  if (i_begin >= i_end || (!CROWDED && i_end - i_begin > kCrowdCell)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float4* si_all = TORQUE ? sT + kHalfChunk : sT;                     // [warps][2 pairs][value] float2, padded
  float4* pshift = si_all + 3 * kCluster * WARPS;
  int* sidx = reinterpret_cast<int*>(pshift + kPieces);               // where a staged particle's sums go
  int* q_all = sidx + kHalfChunk;
  int* meta = q_all + WARPS * (kQueue + kNearQueue + 4);         // pieces: source start, prefix
  int* odd_load = meta + 2 * kPieces + 2;                             // a staged load is not finite
  float2* si = reinterpret_cast<float2*>(si_all + 3 * kCluster * warp);   // [pair h][W2]: particles 2 h and 2 h + 1
  int* qj = q_all + (kQueue + kNearQueue + 4) * warp;   // queued candidate slots
  int* qn = qj + kQueue;                                // queued near pairs: slot * 4 + particle of the cluster
  int* qn_len = qn + kNearQueue;
  if (warp == 0) half_shell_pieces(g, cell, cstart, meta, pshift);
  if (threadIdx.x == 0) *odd_load = poly.ok ? 0 : 1;
  __syncthreads();
  const int total = meta[2 * kPieces + 1];
  const unsigned lt = (1u << lane) - 1u;
  const int ni = i_end - i_begin, parts = CROWDED ? crowd_parts(ni) : 1;
  // Positions are staged from a point beside the cell's first particle: small numbers, so the test can use
  // |x_i|^2 + |x_j|^2 - 2 x_i.x_j (three FMAs per particle) with a margin for its cancellation (at most 20
  // roundings of 2^-24 of the squared extent of two cells). The point is a multiple of the box edge's last place, so
  // the differences are exact but for coordinates of a smaller binade than themselves.
  float4 org = make_float4(0.f, 0.f, 0.f, 0.f);
  float rc2t = 0.f;
  if (SHIFT) {
    const float4 y = cpos[i_begin];
    org = make_float4(__fsub_rn(__fadd_rn(y.x, g.L[0]), g.L[0]), __fsub_rn(__fadd_rn(y.y, g.L[1]), g.L[1]),
                      __fsub_rn(__fadd_rn(y.z, g.L[2]), g.L[2]), 0.f);
    const float ex = 2.f / g.cellw_inv[0], ey = 2.f / g.cellw_inv[1], ez = 2.f / g.cellw_inv[2];
    rc2t = pc.rc2 * (1.f + 1e-6f) + 2e-6f * (ex * ex + ey * ey + ez * ez);
  }

  for (int cb = 0; cb < total; cb += kHalfChunk) {
    const int nc = min(kHalfChunk, total - cb);
    __syncthreads();
    bool fin = true;
    for (int q = 0; q < kPieces; ++q) {
      const int lo = max(meta[2 * q + 1], cb), hi = min(meta[2 * q + 3], cb + nc);
      const int src = meta[2 * q] + (lo - meta[2 * q + 1]);
      const float4 sh = pshift[q];
      for (int k = threadIdx.x; k < hi - lo; k += blockDim.x) {
        float4 y = cpos[src + k];
        if (SHIFT) {
          y.x = (y.x + sh.x) - org.x;
          y.y = (y.y + sh.y) - org.y;
          y.z = (y.z + sh.z) - org.z;
          y.w = rc2t - fmaf(y.x, y.x, fmaf(y.y, y.y, y.z * y.z));
        }
        spos[lo - cb + k] = y;
        sidx[lo - cb + k] = src + k;
        const float4 f = cF[src + k];
        sF[lo - cb + k] = f;
        fin = fin && bounded3(f);
        if (TORQUE) {
          const float4 t = cT[src + k];
          sT[lo - cb + k] = t;
          fin = fin && bounded3(t);
        }
      }
    }
    // pad to whole 32-candidate passes with dummies out of every particle's reach: no bounds test in the loop
    const int ncp = (nc + 31) & ~31;
    for (int k = nc + threadIdx.x; k < ncp; k += blockDim.x) spos[k] = make_float4(1e18f, 1e18f, 1e18f, -3e38f);
    // the cell's own loads are staged in the first chunk, so later chunks know about them too
    if (!fin) *odd_load = 1;
    __syncthreads();
    const bool all_near = *odd_load != 0;

    for (int cl = warp + WARPS * part; kCluster * cl < ni; cl += WARPS * parts) {
      const int a = kCluster * cl;              // first particle of the cluster (slot of the own cell)
      const int ci = min(kCluster, ni - a);
      const int first = max(a + 1 - cb, 0);     // candidates after the first particle's own slot
      if (first >= nc) continue;
      if (lane < 3 * kCluster) {
        const int m = lane / 3, w = lane - 3 * m;
        if (w < W2 / 3) {
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (m < ci) {
            v = (w == 0 ? cpos : (w == 1 ? cF : cT))[i_begin + a + m];
            if (SHIFT && w == 0) { v.x -= org.x; v.y -= org.y; v.z -= org.z; }
          } else if (w == 0) {
            v = make_float4(-1e18f, -1e18f, -1e18f, 0.f);
          }
          float* o = reinterpret_cast<float*>(si + (m >> 1) * W2 + 3 * w) + (m & 1);
          o[0] = v.x; o[2] = v.y; o[4] = v.z;
        }
      }
      if (lane == 0) *qn_len = 0;
      __syncwarp();
      float2 X[2], Y[2], Z[2];   // positions of the four particles in pairs
      float2 X2[2], Y2[2], Z2[2], S2[2];   // -2 x_i and |x_i|^2 (SHIFT)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        X[h] = si[h * W2];
        Y[h] = si[h * W2 + 1];
        Z[h] = si[h * W2 + 2];
        if (SHIFT) {
          X2[h] = mul2(X[h], two(-2.f));
          Y2[h] = mul2(Y[h], two(-2.f));
          Z2[h] = mul2(Z[h], two(-2.f));
          S2[h] = dot2(X[h], Y[h], Z[h], X[h], Y[h], Z[h]);
        }
      }
      float2 u[2][V];   // sums of the cluster: U then W of particles 2 h and 2 h + 1
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < V; ++c) u[h][c] = two(0.f);
      int nq = 0, nn = 0;   // queued candidates and near pairs (the same in every lane)

      for (int base = first & ~31;; base += 32) {
        const bool last = base >= ncp;
        if (!last) {   // 32 candidates against the four particles
          const int k = base + lane;
          const float4 p = spos[k];
          bool hit;
          if (SHIFT) {
            float2 s[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) s[h] = fma2(X2[h], two(p.x), fma2(Y2[h], two(p.y), fma2(Z2[h], two(p.z), S2[h])));
            hit = fminf(fminf(s[0].x, s[0].y), fminf(s[1].x, s[1].y)) < p.w;
          } else {   // the smaller of |d| and L - |d|
            float r2 = 3e38f;
#pragma unroll
            for (int m = 0; m < kCluster; ++m) {
              const float px = m & 1 ? X[m >> 1].y : X[m >> 1].x, py = m & 1 ? Y[m >> 1].y : Y[m >> 1].x;
              const float pz = m & 1 ? Z[m >> 1].y : Z[m >> 1].x;
              float dx = fabsf(px - p.x), dy = fabsf(py - p.y), dz = fabsf(pz - p.z);
              dx = fminf(dx, g.L[0] - dx);
              dy = fminf(dy, g.L[1] - dy);
              dz = fminf(dz, g.L[2] - dz);
              r2 = fminf(r2, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
            }
            hit = r2 < pc.rc2;
          }
          hit = hit && k >= first;
          const unsigned b = __ballot_sync(kFullMask, hit);
          if (hit) qj[nq + __popc(b & lt)] = k;   // nq < 32 here, so the slot is < 64
          nq += __popc(b);
        }
        if (nq >= 32 || (last && nq > 0)) {   // a pass of up to 32 queued candidates against the four particles
          __syncwarp();
          const int cnt = min(nq, 32);
          nq -= cnt;
          const bool on = lane < cnt;
          const int k = on ? qj[nq + lane] : 0;
          float4 pj = spos[k];
          if (!on) pj.x = 1e18f;
          const int own = k + cb - a;   // partner slots up to the particle's own are other pairs or itself
          unsigned near = 0;
          if (all_near) {
#pragma unroll
            for (int m = 0; m < kCluster; ++m) {
              const float px = m & 1 ? X[m >> 1].y : X[m >> 1].x, py = m & 1 ? Y[m >> 1].y : Y[m >> 1].x;
              const float pz = m & 1 ? Z[m >> 1].y : Z[m >> 1].x;
              const float dx = SHIFT ? px - pj.x : nearest(px - pj.x, g.L[0]);
              const float dy = SHIFT ? py - pj.y : nearest(py - pj.y, g.L[1]);
              const float dz = SHIFT ? pz - pj.z : nearest(pz - pj.z, g.L[2]);
              if (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < pc.rc2 && own > m) near |= 1u << m;
            }
          } else {
            const float4 Fj = sF[k];
            const float4 Tj = TORQUE ? sT[k] : make_float4(0.f, 0.f, 0.f, 0.f);
            float2 v[V];   // the partner's sums from even and odd particles
#pragma unroll
            for (int c = 0; c < V; ++c) v[c] = two(0.f);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              float2 dx = __fadd2_rn(X[h], two(-pj.x)), dy = __fadd2_rn(Y[h], two(-pj.y)), dz = __fadd2_rn(Z[h], two(-pj.z));
              if (!SHIFT) {
                dx = make_float2(nearest(dx.x, g.L[0]), nearest(dx.y, g.L[0]));
                dy = make_float2(nearest(dy.x, g.L[1]), nearest(dy.y, g.L[1]));
                dz = make_float2(nearest(dz.x, g.L[2]), nearest(dz.y, g.L[2]));
              }
              const float2 r2 = dot2(dx, dy, dz, dx, dy, dz);
              const bool hit0 = r2.x < pc.rc2 && own > 2 * h, hit1 = r2.y < pc.rc2 && own > 2 * h + 1;
              const bool close0 = r2.x < poly.near2, close1 = r2.y < poly.near2;
              if (hit0 && close0) near |= 1u << (2 * h);
              if (hit1 && close1) near |= 2u << (2 * h);
              // a masked pair gets exp = 0; its polynomials are finite (r is kept at r_near or above)
              const float2 ir = rsqrt2(make_float2(fmaxf(r2.x, poly.near2), fmaxf(r2.y, poly.near2)));
              const float t0 = fmaf(ir.x, poly.scale, poly.offset), t1 = fmaf(ir.y, poly.scale, poly.offset);
              const float2 e = make_float2(hit0 && !close0 ? exp2_approx(r2.x * poly.expo) : 0.f,
                                           hit1 && !close1 ? exp2_approx(r2.y * poly.expo) : 0.f);
              const float2 al = mul2(e, make_float2(poly_eval<0>(poly, t0), poly_eval<0>(poly, t1)));
              const float2 bt = mul2(e, make_float2(poly_eval<1>(poly, t0), poly_eval<1>(poly, t1)));
              const float2 Fx = si[h * W2 + 3], Fy = si[h * W2 + 4], Fz = si[h * W2 + 5];
              const float2 bj = mul2(bt, dot2(dx, dy, dz, two(Fj.x), two(Fj.y), two(Fj.z)));
              const float2 bi = mul2(bt, dot2(dx, dy, dz, Fx, Fy, Fz));
              u[h][0] = fma2(al, two(Fj.x), fma2(bj, dx, u[h][0]));
              u[h][1] = fma2(al, two(Fj.y), fma2(bj, dy, u[h][1]));
              u[h][2] = fma2(al, two(Fj.z), fma2(bj, dz, u[h][2]));
              v[0] = fma2(al, Fx, fma2(bi, dx, v[0]));
              v[1] = fma2(al, Fy, fma2(bi, dy, v[1]));
              v[2] = fma2(al, Fz, fma2(bi, dz, v[2]));
              if constexpr (TORQUE) {
                const float2 cr = mul2(e, make_float2(poly_eval<2>(poly, t0), poly_eval<2>(poly, t1)));
                const float2 gm = mul2(e, make_float2(poly_eval<3>(poly, t0), poly_eval<3>(poly, t1)));
                const float2 dl = mul2(e, make_float2(poly_eval<4>(poly, t0), poly_eval<4>(poly, t1)));
                const float2 nr = make_float2(-cr.x, -cr.y);
                const float2 cx = mul2(cr, dx), cy = mul2(cr, dy), cz = mul2(cr, dz);
                const float2 nx = mul2(nr, dx), ny = mul2(nr, dy), nz = mul2(nr, dz);
                const float2 Tx = si[h * W2 + 6], Ty = si[h * W2 + 7], Tz = si[h * W2 + 8];
                // U_i += cr (T_j x x), U_j -= cr (T_i x x)
                u[h][0] = fma2(two(Tj.y), cz, fma2(two(Tj.z), ny, u[h][0]));
                u[h][1] = fma2(two(Tj.z), cx, fma2(two(Tj.x), nz, u[h][1]));
                u[h][2] = fma2(two(Tj.x), cy, fma2(two(Tj.y), nx, u[h][2]));
                v[0] = fma2(Ty, nz, fma2(Tz, cy, v[0]));
                v[1] = fma2(Tz, nx, fma2(Tx, cz, v[1]));
                v[2] = fma2(Tx, ny, fma2(Ty, cx, v[2]));
                // W_i += cr (F_j x x) + gm T_j + dl x (x.T_j), W_j += -cr (F_i x x) + gm T_i + dl x (x.T_i)
                const float2 ej = mul2(dl, dot2(dx, dy, dz, two(Tj.x), two(Tj.y), two(Tj.z)));
                const float2 ei = mul2(dl, dot2(dx, dy, dz, Tx, Ty, Tz));
                u[h][3] = fma2(two(Fj.y), cz, fma2(two(Fj.z), ny, fma2(gm, two(Tj.x), fma2(ej, dx, u[h][3]))));
                u[h][4] = fma2(two(Fj.z), cx, fma2(two(Fj.x), nz, fma2(gm, two(Tj.y), fma2(ej, dy, u[h][4]))));
                u[h][5] = fma2(two(Fj.x), cy, fma2(two(Fj.y), nx, fma2(gm, two(Tj.z), fma2(ej, dz, u[h][5]))));
                v[3] = fma2(Fy, nz, fma2(Fz, cy, fma2(gm, Tx, fma2(ei, dx, v[3]))));
                v[4] = fma2(Fz, nx, fma2(Fx, cz, fma2(gm, Ty, fma2(ei, dy, v[4]))));
                v[5] = fma2(Fx, ny, fma2(Fy, cx, fma2(gm, Tz, fma2(ei, dz, v[5]))));
              }
            }
            if (on) {
              const int o = sidx[k];
              add_sums<CROWDED>(psum, psum64, o, 0, v[0].x + v[0].y, v[1].x + v[1].y, v[2].x + v[2].y);
              if constexpr (TORQUE)
                add_sums<CROWDED>(psum, psum64, o, 1, v[3].x + v[3].y, v[4].x + v[4].y, v[5].x + v[5].y);
            }
          }
          while (near) {   // few lanes have any
            const int m = __ffs(near) - 1;
            near &= near - 1;
            qn[atomicAdd(qn_len, 1)] = 4 * k + m;
          }
          __syncwarp();
          nn = *qn_len;
        }
        while (nn >= 32 || (last && nn > 0)) {   // up to 32 near pairs with the table, one per lane
          const int cnt = min(nn, 32);
          nn -= cnt;
          if (lane < cnt) {
            const int e = qn[nn + lane];
            const int k = e >> 2, m = e & 3;
            const float* pi = reinterpret_cast<const float*>(si + (m >> 1) * W2) + (m & 1);
            const float4 pj = spos[k];
            const float dx = SHIFT ? pi[0] - pj.x : nearest(pi[0] - pj.x, g.L[0]);
            const float dy = SHIFT ? pi[2] - pj.y : nearest(pi[2] - pj.y, g.L[1]);
            const float dz = SHIFT ? pi[4] - pj.z : nearest(pi[4] - pj.z, g.L[2]);
            float al, bt, cr, gm, dl;
            pair_coeffs_table(fmaf(dx, dx, fmaf(dy, dy, dz * dz)), pc, tab, al, bt, cr, gm, dl);
            const float3 Fi = make_float3(pi[6], pi[8], pi[10]);
            const float4 Fj = sF[k];
            const float bj = bt * (dx * Fj.x + dy * Fj.y + dz * Fj.z), bi = bt * (dx * Fi.x + dy * Fi.y + dz * Fi.z);
            float w[V], v[V];
            w[0] = fmaf(bj, dx, al * Fj.x); w[1] = fmaf(bj, dy, al * Fj.y); w[2] = fmaf(bj, dz, al * Fj.z);
            v[0] = fmaf(bi, dx, al * Fi.x); v[1] = fmaf(bi, dy, al * Fi.y); v[2] = fmaf(bi, dz, al * Fi.z);
            if constexpr (TORQUE) {
              const float3 Ti = make_float3(pi[12], pi[14], pi[16]);
              const float4 Tj = sT[k];
              const float cx = cr * dx, cy = cr * dy, cz = cr * dz;
              const float ej = dl * (dx * Tj.x + dy * Tj.y + dz * Tj.z), ei = dl * (dx * Ti.x + dy * Ti.y + dz * Ti.z);
              w[0] += Tj.y * cz - Tj.z * cy; w[1] += Tj.z * cx - Tj.x * cz; w[2] += Tj.x * cy - Tj.y * cx;
              v[0] -= Ti.y * cz - Ti.z * cy; v[1] -= Ti.z * cx - Ti.x * cz; v[2] -= Ti.x * cy - Ti.y * cx;
              w[3] = Fj.y * cz - Fj.z * cy + fmaf(ej, dx, gm * Tj.x);
              w[4] = Fj.z * cx - Fj.x * cz + fmaf(ej, dy, gm * Tj.y);
              w[5] = Fj.x * cy - Fj.y * cx + fmaf(ej, dz, gm * Tj.z);
              v[3] = fmaf(ei, dx, gm * Ti.x) - (Fi.y * cz - Fi.z * cy);
              v[4] = fmaf(ei, dy, gm * Ti.y) - (Fi.z * cx - Fi.x * cz);
              v[5] = fmaf(ei, dz, gm * Ti.z) - (Fi.x * cy - Fi.y * cx);
            }
            const int o = sidx[k];
            add_sums<CROWDED>(psum, psum64, o, 0, v[0], v[1], v[2]);
            if constexpr (TORQUE) add_sums<CROWDED>(psum, psum64, o, 1, v[3], v[4], v[5]);
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
              for (int c = 0; c < V; ++c) {
                u[h][c].x += m == 2 * h ? w[c] : 0.f;
                u[h][c].y += m == 2 * h + 1 ? w[c] : 0.f;
              }
          }
          __syncwarp();
          if (lane == 0) *qn_len = nn;
          __syncwarp();
        }
        if (last) break;
      }
      // sums of the four particles over the warp: lanes 0, 4, 8, .. (0, 8, .. without torques) hold (particle, U or W)
      float sum[kCluster * V];   // [particle][component]
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < V; ++c) {
          sum[2 * h * V + c] = u[h][c].x;
          sum[(2 * h + 1) * V + c] = u[h][c].y;
        }
      halve<kCluster * V>(sum, 16);      // particles 0, 1 | 2, 3
      halve<kCluster * V / 2>(sum, 8);   // the particle
      if constexpr (TORQUE) {
        halve<V>(sum, 4);                // U | W
      } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) sum[c] += __shfl_xor_sync(kFullMask, sum[c], 4);
      }
#pragma unroll
      for (int o = 2; o > 0; o >>= 1)
#pragma unroll
        for (int c = 0; c < 3; ++c) sum[c] += __shfl_xor_sync(kFullMask, sum[c], o);
      const int m = 2 * (lane >> 4) + ((lane >> 3) & 1), w = TORQUE ? (lane >> 2) & 1 : 0;
      if ((lane & (TORQUE ? 3 : 7)) == 0 && m < ci)
        add_sums<CROWDED>(psum, psum64, i_begin + a + m, w, sum[0], sum[1], sum[2]);
      __syncwarp();
    }
  }
}

// CTA c takes cell c unless it is crowded. The last `sharers` CTAs (as many as run at once, at most one per possible part;
// more of them than cells where cells are few) then share the crowded cells' parts.
template <bool TORQUE, bool SHIFT, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, cell_blocks(WARPS, TORQUE))
    pair_cluster_kernel(Geometry<float> g, PairConsts<float> pc, PairTable tab, PairPoly poly,
                        const float4* __restrict__ cpos, const float4* __restrict__ cF, const float4* __restrict__ cT,
                        const int* __restrict__ cstart, float4* __restrict__ psum, double* __restrict__ psum64,
                        const int* __restrict__ crowd, int ncells, int sharers) {
  if ((int)blockIdx.x < ncells)
    cell_pairs<TORQUE, SHIFT, WARPS, false>(g, pc, tab, poly, cpos, cF, cT, cstart, psum, psum64, blockIdx.x, 0);
  int k = (int)blockIdx.x - ((int)gridDim.x - sharers);
  if (k < 0) return;
  for (const int items = crowd[1]; k < items; k += sharers) {
    __syncthreads();   // the next part reuses the shared memory
    cell_pairs<TORQUE, SHIFT, WARPS, true>(g, pc, tab, poly, cpos, cF, cT, cstart, psum, psum64, crowd[2 + 2 * k],
                                           crowd[3 + 2 * k]);
  }
}

// Pair sums in cell order, plus the self terms, to input order: U = or U += (ADD), W likewise.
template <bool ADD>
__global__ void __launch_bounds__(256) pair_merge_kernel(PairConsts<float> pc, const float4* __restrict__ psum,
                                                         const double* __restrict__ psum64,
                                                         const int* __restrict__ crowd,
                                                         const float4* __restrict__ cF, const float4* __restrict__ cT,
                                                         const unsigned* __restrict__ slot, int n,
                                                         const int* __restrict__ n_dev, float* __restrict__ U,
                                                         float* __restrict__ W) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (n_dev) n = min(n, *n_dev);
  if (i >= n) return;
  const size_t s = slot[i], o = 3 * (size_t)i;
  const float4 F = cF[s];
  float4 a = psum[2 * s], b = W ? psum[2 * s + 1] : a;   // all loads before the branch
  if (crowd[1] > 0) {   // some sums are in FP64
    const double* q = psum64 + 6 * s;
    a = make_float4((float)(a.x + q[0]), (float)(a.y + q[1]), (float)(a.z + q[2]), 0.f);
    b = make_float4((float)(b.x + q[3]), (float)(b.y + q[4]), (float)(b.z + q[5]), 0.f);
  }
  const float u[3] = {fmaf(pc.selfVF, F.x, a.x), fmaf(pc.selfVF, F.y, a.y), fmaf(pc.selfVF, F.z, a.z)};
#pragma unroll
  for (int c = 0; c < 3; ++c) U[o + c] = ADD ? U[o + c] + u[c] : u[c];
  if (W) {
    const float4 T = cT[s];
    const float w[3] = {fmaf(pc.selfWT, T.x, b.x), fmaf(pc.selfWT, T.y, b.y), fmaf(pc.selfWT, T.z, b.z)};
#pragma unroll
    for (int c = 0; c < 3; ++c) W[o + c] = ADD ? W[o + c] + w[c] : w[c];
  }
}

template <bool TORQUE, bool SHIFT, int WARPS>
static void cluster_variant(const Geometry<float>& g, const PairConsts<float>& pc, const PairTable& tab,
                            const PairPoly& poly, const BinBuffers& b, int n, cudaStream_t s) {
  const size_t smem = cluster_smem<TORQUE, WARPS>();
  auto k = pair_cluster_kernel<TORQUE, SHIFT, WARPS>;
  allow_dynamic_smem(k, smem);
  const int sharers = std::min(cell_blocks(WARPS, TORQUE) * device_sm_count(), crowd_items(n));
  k<<<std::max(b.ncells, sharers), WARPS * 32, smem, s>>>(g, pc, tab, poly, (const float4*)b.c_pos, (const float4*)b.c_F,
                                       (const float4*)b.c_T, b.cell_start, (float4*)b.c_sum, b.c_sum64,
                                     b.crowd, b.ncells, sharers);
}

// Warps of a CTA: a cell's clusters are dealt out to them, so cells of about eight particles (two clusters; the cell
// size rule aims at eight) take two and fuller ones four; crowded cells are shared out in either. Measured with 2 / 4 / 8 warps: 122,231 particles in cells
// of 8.8, forces only, 95 / 141 / 268 us; rods at 8.2 per cell, torques, 0.69 / 0.77 / 1.38 ms; 32 systems at 38 per
// cell 3.14 / 2.87 / 3.47 ms; rigid rods, 12 per cell on average but all in one layer of three, 73 / 55 / 63 us.
constexpr double kTwoWarpCell = 10.0;

template <bool TORQUE, bool SHIFT>
static void cluster_launch(const Geometry<float>& g, const PairConsts<float>& pc, const PairTable& tab,
                           const PairPoly& poly, const BinBuffers& b, int n, cudaStream_t s) {
  if ((double)n < kTwoWarpCell * b.ncells) cluster_variant<TORQUE, SHIFT, 2>(g, pc, tab, poly, b, n, s);
  else cluster_variant<TORQUE, SHIFT, 4>(g, pc, tab, poly, b, n, s);
}

void launch_pair_f32(const Geometry<float>& g, const PairConsts<float>& pc, const PairTable& tab, const PairPoly& poly,
                     bool torque, const BinBuffers& b, int n, cudaStream_t s, long long* launches) {
  if (n <= 0) return;
  if (torque) {
    if (g.shift) cluster_launch<true, true>(g, pc, tab, poly, b, n, s);
    else cluster_launch<true, false>(g, pc, tab, poly, b, n, s);
  } else {
    if (g.shift) cluster_launch<false, true>(g, pc, tab, poly, b, n, s);
    else cluster_launch<false, false>(g, pc, tab, poly, b, n, s);
  }
  *launches += 1;
}

void launch_pair_merge(const PairConsts<float>& pc, bool torque, const BinBuffers& b, int n, bool add, float* U, float* W,
                       cudaStream_t s, long long* launches) {
  if (n <= 0) return;
  auto k = add ? pair_merge_kernel<true> : pair_merge_kernel<false>;
  k<<<(n + 255) / 256, 256, 0, s>>>(pc, (const float4*)b.c_sum, b.c_sum64, b.crowd, (const float4*)b.c_F,
                                    (const float4*)b.c_T, b.cell_rank, n, b.n_dev, U, torque ? W : nullptr);
  *launches += 1;
}

}  // namespace fcm
