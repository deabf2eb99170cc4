// FP32 interpolation J~ + N~ on tiles (trapezoidal rule of Section 2.1 step 3,
// eq. avg_particle_vel_mod and eq. avg_particle_rot_mod):
//   U = h^3 sum_g u(x_g) Delta~(x_g - Y; Sigma)
//   W = h^3 sum_g Delta(x_g - Y; Sigma_D) (d_g x u(x_g)) / (2 Sigma_D^2),  d_g = x_g - Y
// (the second line is (1/2) int (curl u) Delta after one integration by parts,
// the exact adjoint of the torque spread).
//
// One CTA per z-pencil of tiles, taking the tiles in turn: the extended region of u is held in
// shared memory as a ring of its z planes, and each step copies only the tile's new planes
// (tile_z of the E_Z, with asynchronous 4-byte copies, no register round trip); a warp owns a
// particle and its lanes own window rows; the M_G x-profiles are computed by
// M_G lanes and broadcast into registers with warp shuffles. Per point: a 4-byte
// load (x) and an 8-byte load (y, z interleaved) from shared memory, and 6 FMAs with
// torques (gather_particle; 8 with two widths or supports without a compiled variant)
// or 5 for forces only.
// What bounds it: shared-memory reads (12 bytes per point) and, about a quarter of the
// time, the copy of a tile's new planes, which the other CTA of the SM covers in part.
// 32 x 65,536 spheres on 128^3, M_G = 14, torques: 4.62 ms with 8 FMAs per point, a row
// copied per warp and butterfly sums, 4.36 with packed sums, 4.31 with
// full-lane copies; 8 x 65,536 rods, M_G = 12: 978, 938, 878 us; 122,231 on
// 216^3, M_G = 10, forces only: 271 -> 245 us.
// The pair-correction sums, when present, are added when U and W are written
// in input order.
#include "grid_common.cuh"

namespace fcm {

__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }

// One halving step of a warp sum over two values: lanes with bit `s` clear keep the sum of a, the
// others that of b (one shuffle for both; each value's additions are those of the butterfly).
__device__ __forceinline__ float fold2(float a, float b, int s, bool hi) {
  return (hi ? b : a) + __shfl_xor_sync(kFullMask32, hi ? a : b, s);
}

__device__ __forceinline__ float fold1(float a, int s) { return a + __shfl_xor_sync(kFullMask32, a, s); }

// Sums over the warp's lanes, times h^3, to row `i` of U and W (plus the pair sums, where given). The sum
// halves its values as it goes: 8 shuffles for six values, 6 for three, instead of 30 and 15.
template <bool TORQUE>
__device__ __forceinline__ void gather_store(int lane, int i, float h3, float u0, float u1, float u2, float w0,
                                             float w1, float w2, const float* __restrict__ upair,
                                             const float* __restrict__ wpair, float* __restrict__ U,
                                             float* __restrict__ W) {
  const bool b16 = lane & 16, b8 = lane & 8, b4 = lane & 4;
  const size_t oi = 3 * (size_t)i;
  if (TORQUE) {
    const float v0 = fold2(u0, w0, 16, b16), v1 = fold2(u1, w1, 16, b16), v2 = fold2(u2, w2, 16, b16);
    const float v = fold1(fold1(fold2(fold2(v0, v1, 8, b8), fold1(v2, 8), 4, b4), 2), 1);
    const int c = b4 ? 2 : (b8 ? 1 : 0);   // lanes 0, 8, 4 hold U, lanes 16, 24, 20 W
    float* out = b16 ? W : U;
    const float* add = b16 ? wpair : upair;
    if ((lane & 3) == 0 && !(b4 && b8) && out) out[oi + c] = h3 * v + (add ? add[oi + c] : 0.f);
  } else {
    const float v = fold1(fold1(fold1(fold2(fold2(u0, u1, 16, b16), fold1(u2, 16), 8, b8), 4), 2), 1);
    const int c = b8 ? 2 : (b16 ? 1 : 0);   // lanes 0, 16, 8
    if ((lane & 7) == 0 && !(b8 && b16)) U[oi + c] = h3 * v + (upair ? upair[oi + c] : 0.f);
  }
}

// One particle's sums (each lane's part) with torques, one width and a compiled support, in packed FMAs: with
// S = sum_x g u along a row and T(x) = sum_rows G u down a column (G = g(dy) g(dz)), six FMAs per window point,
//   U = nrm (sum_rows G P S + B sum_x d^2 g T),  P = A + B (dy^2 + dz^2),
//   W = tq  (sum_rows G (dy S_z - dz S_y, dz S_x, -dy S_x) + sum_x d g (0, -T_z, T_y)).
// The general form's eight FMAs per point were 43% of the kernel's instructions, at 65% of the issue slots
// (M_G = 14): 363 M -> 268 M warp instructions for 3 x 65,536 particles.
template <int MGT>
__device__ __forceinline__ void gather_particle(const Geometry<float>& g, const KernelConsts<float>& kc,
                                                const ExtLayout& l, const float* acc, int zs,
                                                const TileOrigin& o, int lane, float4 y, float& u0, float& u1,
                                                float& u2, float& w0, float& w1, float& w2) {
  const int ring = l.EZ;
  const int3 i0 = window_starts(g, y);
  const int4 off = window_offset(g, o, i0);
  const float dxl = (float)(i0.x + lane) * g.h[0] - y.x;
  const float dyl = (float)(i0.y + lane) * g.h[1] - y.y;
  const float dzl = (float)(i0.z + lane) * g.h[2] - y.z;
  const float gxl = expf(-dxl * dxl * kc.inv2S2);
  const float gyl = expf(-dyl * dyl * kc.inv2S2);
  const float gzl = expf(-dzl * dzl * kc.inv2S2);
  u0 = u1 = u2 = w0 = w1 = w2 = 0.f;
  float2 gg[MGT], gp[MGT / 2];       // g(x) twice; of two points
  float2 tyz[MGT], tx[MGT / 2];      // column sums of (u_y, u_z); of u_x at two points
#pragma unroll
  for (int j = 0; j < MGT; ++j) {
    gg[j] = dup2(__shfl_sync(kFullMask32, gxl, j));
    tyz[j] = make_float2(0.f, 0.f);
  }
#pragma unroll
  for (int j = 0; j < MGT / 2; ++j) {
    gp[j] = make_float2(gg[2 * j].x, gg[2 * j + 1].x);
    tx[j] = make_float2(0.f, 0.f);
  }
  int zb = zs + off.z;   // ring slot of the window's first plane
  if (zb >= ring) zb -= ring;
  const float* pbase = acc + off.y * l.P + off.x;
  const float2* yzbase = reinterpret_cast<const float2*>(acc + yz_plane_offset(l)) + off.y * l.P + off.x;
  constexpr int NFULL = MGT * MGT / 32, TAIL = MGT * MGT % 32;
  constexpr bool SPLIT_TAIL = TAIL > 0 && TAIL * MGT <= 64;   // a short last pass: split it by points
#pragma unroll
  for (int it = 0; it < (SPLIT_TAIL ? NFULL : (MGT * MGT + 31) / 32); ++it) {
    // window row r = jy + M_G jz of lane and pass it: fixed per lane
    const int r = 32 * it + lane;
    const bool active = r < MGT * MGT;
    const int jz = active ? r / MGT : 0, jy = active ? r - (r / MGT) * MGT : 0;
    int sl = zb + jz;
    if (sl >= ring) sl -= ring;
    const int ro = sl * l.Q + jy * l.P;
    const float dy = __shfl_sync(kFullMask32, dyl, jy);
    const float gy = __shfl_sync(kFullMask32, gyl, jy);
    const float dz = __shfl_sync(kFullMask32, dzl, jz);
    const float gz = __shfl_sync(kFullMask32, gzl, jz);
    const float G = active ? gy * gz : 0.f;
    const float2 G2 = dup2(G);
    float2 sx = make_float2(0.f, 0.f), syz = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < MGT; j += 2) {
      const float2 ux = make_float2(pbase[ro + j], pbase[ro + j + 1]);
      const float2 ua = yzbase[ro + j], ub = yzbase[ro + j + 1];
      sx = __ffma2_rn(gp[j / 2], ux, sx);
      tx[j / 2] = __ffma2_rn(G2, ux, tx[j / 2]);
      syz = __ffma2_rn(gg[j], ua, syz);
      tyz[j] = __ffma2_rn(G2, ua, tyz[j]);
      syz = __ffma2_rn(gg[j + 1], ub, syz);
      tyz[j + 1] = __ffma2_rn(G2, ub, tyz[j + 1]);
    }
    const float s0 = sx.x + sx.y;
    const float GP = G * fmaf(kc.B, fmaf(dy, dy, dz * dz), kc.A);
    u0 = fmaf(GP, s0, u0);
    u1 = fmaf(GP, syz.x, u1);
    u2 = fmaf(GP, syz.y, u2);
    const float Gs0 = G * s0;
    w0 = fmaf(G, dy * syz.y - dz * syz.x, w0);
    w1 = fmaf(dz, Gs0, w1);
    w2 = fmaf(-dy, Gs0, w2);
  }
  if (SPLIT_TAIL) {
    // the last TAIL rows have TAIL * M_G (row, point) items: each lane takes up to two and applies
    // the row's y, z factors to each item itself
#pragma unroll
    for (int pass = 0; pass < 2; ++pass) {
      const int e = lane + 32 * pass;
      const bool valid = e < TAIL * MGT;
      const int t = valid ? e / MGT : 0, j = valid ? e - (e / MGT) * MGT : 0;
      const int r = 32 * NFULL + t;
      const int jz = r / MGT, jy = r - jz * MGT;
      const float gj = __shfl_sync(kFullMask32, gxl, j);
      const float dj = __shfl_sync(kFullMask32, dxl, j);
      const float dy = __shfl_sync(kFullMask32, dyl, jy);
      const float gy = __shfl_sync(kFullMask32, gyl, jy);
      const float dz = __shfl_sync(kFullMask32, dzl, jz);
      const float gz = __shfl_sync(kFullMask32, gzl, jz);
      if (valid) {
        int sl = zb + jz;
        if (sl >= ring) sl -= ring;
        const int ro = sl * l.Q + jy * l.P + j;
        const float ux = pbase[ro];
        const float2 uyz = yzbase[ro];
        const float g3 = gy * gz * gj;
        const float wgt = g3 * fmaf(kc.B, fmaf(dj, dj, fmaf(dy, dy, dz * dz)), kc.A);
        u0 = fmaf(wgt, ux, u0);
        u1 = fmaf(wgt, uyz.x, u1);
        u2 = fmaf(wgt, uyz.y, u2);
        w0 = fmaf(g3, dy * uyz.y - dz * uyz.x, w0);
        w1 = fmaf(g3, dz * ux - dj * uyz.y, w1);
        w2 = fmaf(g3, dj * uyz.x - dy * ux, w2);
      }
    }
  }
  // the terms in d and d^2 along x, from the column sums
  float2 qx = make_float2(0.f, 0.f), qyz = qx, kyz = qx;
#pragma unroll
  for (int j = 0; j < MGT; j += 2) {
    const float2 da = dup2(__shfl_sync(kFullMask32, dxl, j)), db = dup2(__shfl_sync(kFullMask32, dxl, j + 1));
    const float2 ka = __fmul2_rn(da, gg[j]), kb = __fmul2_rn(db, gg[j + 1]);
    const float2 qa = __fmul2_rn(da, ka), qb = __fmul2_rn(db, kb);
    qx = __ffma2_rn(make_float2(qa.x, qb.x), tx[j / 2], qx);
    qyz = __ffma2_rn(qa, tyz[j], qyz);
    qyz = __ffma2_rn(qb, tyz[j + 1], qyz);
    kyz = __ffma2_rn(ka, tyz[j], kyz);
    kyz = __ffma2_rn(kb, tyz[j + 1], kyz);
  }
  u0 = kc.nrm * fmaf(kc.B, qx.x + qx.y, u0);
  u1 = kc.nrm * fmaf(kc.B, qyz.x, u1);
  u2 = kc.nrm * fmaf(kc.B, qyz.y, u2);
  w0 *= kc.tq;
  w1 = kc.tq * (w1 - kyz.y);
  w2 = kc.tq * (w2 + kyz.x);
}

// CTAs per SM asked of the compiler: what the region's shared memory allows. Forces only with M_G = 10, three
// (122,231 spheres on 216^3: 271 us, with two 312 us), with smaller supports more; from M_G = 12 on, and with
// torques, two of 128 registers a thread (one of more registers: 32 x 65,536 spheres, M_G = 14, 5.76 against
// 4.36 ms). Supports up to 8 with torques and one width fit three (40,000 spheres on 72^3, M_G = 8: 51 us, with two
// 62 us); of the two largest, whose regions are made to leave two, M_G up to 20 with one width takes them (M_G = 18 /
// 20: 372 / 1,198 us, with one 521 / 2,010 us), the others are no faster so (M_G = 24: 1,472 us, with two 1,529 us).
constexpr int gather_ctas(int MGT, bool guard, bool torque, bool samew) {
  if (MGT > 16) return MGT <= 20 && samew ? 2 : 1;
  if (MGT <= 8) return !torque ? 4 : (samew ? 3 : 2);
  return torque || (!guard && MGT >= 12) ? 2 : 3;
}

template <int MGT, bool GUARD, bool TORQUE, bool SAMEW>
__global__ void __launch_bounds__(256, gather_ctas(MGT, GUARD, TORQUE, SAMEW)) gather_tile_kernel(Geometry<float> g, KernelConsts<float> kc,
                                                          const float4* __restrict__ pos,
                                                          const int* __restrict__ tstart,
                                                          const float* __restrict__ grid,
                                                          const float* __restrict__ upair,
                                                          const float* __restrict__ wpair,
                                                          float* __restrict__ U, float* __restrict__ W,
                                                          int segl) {
  extern __shared__ float4 sm4[];
  float* acc = reinterpret_cast<float*>(sm4);
  // the CTA's segment (segl tiles) of a z-pencil of tiles (tx, ty, 0 .. ntile_z - 1) of one system, walked in z
  const int ntx = g.ntile[0], nty = g.ntile[1], ntz = g.ntile[2];
  const int per = ntx * nty;
  const int nseg = (ntz + segl - 1) / segl;
  const int sys = blockIdx.x / (per * nseg);
  const int rem = blockIdx.x - sys * per * nseg;
  const int pcl = rem / nseg;
  const int z0 = (rem - pcl * nseg) * segl, z1 = min(ntz, z0 + segl);
  const int tx = pcl % ntx, ty = pcl / ntx;
  const int tbase = sys * g.tiles_per + pcl;   // tile (tx, ty, 0): tiles are numbered x fastest
  if (g.nsys > 1) grid += (size_t)sys * (size_t)g.grid_stride;
  const int MG = GUARD ? g.MG : MGT;
  const ExtLayout l = ext_layout(g.tile, MG);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  TileOrigin pen;   // the pencil's origin: region plane ez of tile tz is pencil plane tz tile_z + ez
  pen.ox0 = tx * g.tile[0];
  pen.oy0 = ty * g.tile[1];
  pen.oz0 = 0;
  int staged = 0;   // pencil planes below this are in the ring (plane P in slot P mod E_Z)
  for (int tz = z0; tz < z1; ++tz) {
    const int t = tbase + per * tz;
    const int p0 = tstart[t], p1 = tstart[t + 1];
    if (p0 >= p1) continue;
    const int zlo = tz * g.tile[2];
    __syncthreads();   // every warp is done with the planes this step replaces
    stage_region_async(g, pen, l, grid, acc, max(staged, zlo), zlo + l.EZ);
    staged = zlo + l.EZ;
    __syncthreads();
    TileOrigin o = pen;
    o.oz0 = zlo;
    const int zs = zlo % l.EZ;   // ring slot of the tile's region plane 0

    for (int p = p0 + warp; p < p1; p += nwarp) {
      const float4 y = pos[p];
      float u0 = 0.f, u1 = 0.f, u2 = 0.f, w0 = 0.f, w1 = 0.f, w2 = 0.f;
      if constexpr (!GUARD && TORQUE && SAMEW) {
        gather_particle<MGT>(g, kc, l, acc, zs, o, lane, y, u0, u1, u2, w0, w1, w2);
        gather_store<TORQUE>(lane, index_from_w(y.w), kc.h3, u0, u1, u2, w0, w1, w2, upair, wpair, U, W);
        continue;
      }
      const int3 i0 = window_starts(g, y);
      const int4 off = window_offset(g, o, i0);
      const float dxl = (float)(i0.x + lane) * g.h[0] - y.x;
      const float dyl = (float)(i0.y + lane) * g.h[1] - y.y;
      const float dzl = (float)(i0.z + lane) * g.h[2] - y.z;
      const float gxl = expf(-dxl * dxl * kc.inv2S2);
      const float gyl = expf(-dyl * dyl * kc.inv2S2);
      const float gzl = expf(-dzl * dzl * kc.inv2S2);
      const float gdxl = SAMEW ? gxl : expf(-dxl * dxl * kc.inv2SD2);
      const float gdyl = SAMEW ? gyl : expf(-dyl * dyl * kc.inv2SD2);
      const float gdzl = SAMEW ? gzl : expf(-dzl * dzl * kc.inv2SD2);
      float gx[MGT], gx2[MGT], gx1[MGT], gdx[MGT];
#pragma unroll
      for (int j = 0; j < MGT; ++j) {
        const float gj = __shfl_sync(kFullMask32, gxl, j);
        const float dj = __shfl_sync(kFullMask32, dxl, j);
        const float gdj = SAMEW ? gj : __shfl_sync(kFullMask32, gdxl, j);
        gx[j] = gj;
        gx2[j] = dj * dj * gj;
        gdx[j] = gdj;
        gx1[j] = dj * gdj;
      }
      // one window row (jy, jz) of this particle: x sums over the row, times the row's y, z factors
      auto row_update = [&](const float* row, int sy, int sz, bool active) {
        const float dy = __shfl_sync(kFullMask32, dyl, sy);
        const float gy = __shfl_sync(kFullMask32, gyl, sy);
        const float dz = __shfl_sync(kFullMask32, dzl, sz);
        const float gz = __shfl_sync(kFullMask32, gzl, sz);
        const float gdy = SAMEW ? gy : __shfl_sync(kFullMask32, gdyl, sy);
        const float gdz = SAMEW ? gz : __shfl_sync(kFullMask32, gdzl, sz);
        if (!active) return;
        if (!TORQUE) {   // forces only: one weight per point, w = GQ g + GB d^2 g, for the three components
          const float G = kc.nrm * gy * gz;
          const float GQ = G * fmaf(kc.B, fmaf(dy, dy, dz * dz), kc.A);
          const float GB = G * kc.B;
          float a0 = 0.f, a1 = 0.f, a2 = 0.f;
#pragma unroll
          for (int j = 0; j < MGT; ++j) {
            if (!GUARD || j < MG) {
              const float w = fmaf(GB, gx2[j], GQ * gx[j]);
              const float ux = row[j];
              const float2 uyz = reinterpret_cast<const float2*>(acc + yz_plane_offset(l))[(row - acc) + j];
              a0 = fmaf(w, ux, a0);
              a1 = fmaf(w, uyz.x, a1);
              a2 = fmaf(w, uyz.y, a2);
            }
          }
          u0 += a0;
          u1 += a1;
          u2 += a2;
          return;
        }
        float sx0 = 0.f, sy0 = 0.f, sz0 = 0.f, sx2 = 0.f, sy2 = 0.f, sz2 = 0.f;
        float dx0 = 0.f, dy0 = 0.f, dz0 = 0.f, dy1 = 0.f, dz1 = 0.f;
#pragma unroll
        for (int j = 0; j < MGT; ++j) {
          if (!GUARD || j < MG) {
            const float ux = row[j];
            const float2 uyz = reinterpret_cast<const float2*>(acc + yz_plane_offset(l))[(row - acc) + j];
            const float uy = uyz.x, uz = uyz.y;
            sx0 = fmaf(gx[j], ux, sx0); sy0 = fmaf(gx[j], uy, sy0); sz0 = fmaf(gx[j], uz, sz0);
            sx2 = fmaf(gx2[j], ux, sx2); sy2 = fmaf(gx2[j], uy, sy2); sz2 = fmaf(gx2[j], uz, sz2);
            if (TORQUE) {
              if (!SAMEW) { dx0 = fmaf(gdx[j], ux, dx0); dy0 = fmaf(gdx[j], uy, dy0); dz0 = fmaf(gdx[j], uz, dz0); }
              dy1 = fmaf(gx1[j], uy, dy1);
              dz1 = fmaf(gx1[j], uz, dz1);
            }
          }
        }
        const float G = kc.nrm * gy * gz;
        const float GQ = G * fmaf(kc.B, fmaf(dy, dy, dz * dz), kc.A);
        const float GB = G * kc.B;
        u0 = fmaf(GQ, sx0, fmaf(GB, sx2, u0));
        u1 = fmaf(GQ, sy0, fmaf(GB, sy2, u1));
        u2 = fmaf(GQ, sz0, fmaf(GB, sz2, u2));
        if (TORQUE) {
          if (SAMEW) { dx0 = sx0; dy0 = sy0; dz0 = sz0; }
          const float H = kc.tq * gdy * gdz;
          w0 = fmaf(H, dy * dz0 - dz * dy0, w0);
          w1 = fmaf(H, dz * dx0 - dz1, w1);
          w2 = fmaf(H, dy1 - dy * dx0, w2);
        }
      };
      if (!GUARD) {
        // window row r = jy + M_G jz of lane and pass it: fixed per lane, so the row offsets inside the
        // staged region (jz Q + jy P) are loop invariants of the particle loop
        int zb = zs + off.z;   // ring slot of the window's first plane
        if (zb >= l.EZ) zb -= l.EZ;
        const float* pbase = acc + off.y * l.P + off.x;
        constexpr int NFULL = MGT * MGT / 32, TAIL = MGT * MGT % 32;
        constexpr bool SPLIT_TAIL = TAIL > 0 && TAIL * MGT <= 64;   // a short last pass: split it by points
#pragma unroll
        for (int it = 0; it < (SPLIT_TAIL ? NFULL : (MGT * MGT + 31) / 32); ++it) {
          const int r = 32 * it + lane;
          const bool active = r < MGT * MGT;
          const int jz = active ? r / MGT : 0, jy = active ? r - (r / MGT) * MGT : 0;
          int sl = zb + jz;
          if (sl >= l.EZ) sl -= l.EZ;
          row_update(pbase + sl * l.Q + jy * l.P, jy, jz, active);
        }
        if (SPLIT_TAIL) {
          // the last TAIL rows have TAIL * M_G (row, point) items: each lane takes up to two and applies
          // the row's y, z factors to each item itself
#pragma unroll
          for (int pass = 0; pass < 2; ++pass) {
            const int e = lane + 32 * pass;
            const bool valid = e < TAIL * MGT;
            const int t = valid ? e / MGT : 0, j = valid ? e - (e / MGT) * MGT : 0;
            const int r = 32 * NFULL + t;
            const int jz = r / MGT, jy = r - jz * MGT;
            const float gj = __shfl_sync(kFullMask32, gxl, j);
            const float dj = __shfl_sync(kFullMask32, dxl, j);
            const float gdj = SAMEW ? gj : __shfl_sync(kFullMask32, gdxl, j);
            const float dy = __shfl_sync(kFullMask32, dyl, jy);
            const float gy = __shfl_sync(kFullMask32, gyl, jy);
            const float dz = __shfl_sync(kFullMask32, dzl, jz);
            const float gz = __shfl_sync(kFullMask32, gzl, jz);
            const float gdy = SAMEW ? gy : __shfl_sync(kFullMask32, gdyl, jy);
            const float gdz = SAMEW ? gz : __shfl_sync(kFullMask32, gdzl, jz);
            if (valid) {
              int sl = zb + jz;
              if (sl >= l.EZ) sl -= l.EZ;
              const float* row = pbase + sl * l.Q + jy * l.P;
              const float ux = row[j];
            const float2 uyz = reinterpret_cast<const float2*>(acc + yz_plane_offset(l))[(row - acc) + j];
            const float uy = uyz.x, uz = uyz.y;
              const float G = kc.nrm * gy * gz;
              const float GQ = G * fmaf(kc.B, fmaf(dy, dy, dz * dz), kc.A);
              const float GB = G * kc.B;
              const float wgt = fmaf(GB, dj * dj * gj, GQ * gj);
              u0 = fmaf(wgt, ux, u0);
              u1 = fmaf(wgt, uy, u1);
              u2 = fmaf(wgt, uz, u2);
              if (TORQUE) {
                const float H = kc.tq * gdy * gdz;
                const float g1 = dj * gdj;
                w0 = fmaf(H, gdj * (dy * uz - dz * uy), w0);
                w1 = fmaf(H, dz * gdj * ux - g1 * uz, w1);
                w2 = fmaf(H, g1 * uy - dy * gdj * ux, w2);
              }
            }
          }
        }
      } else {
        int jy = lane, jz = 0;
        while (jy >= MG) { jy -= MG; ++jz; }
        for (int r0 = 0; r0 < MG * MG; r0 += 32) {
          const bool active = r0 + lane < MG * MG;
          const int sy = active ? jy : 0, sz = active ? jz : 0;
          int sl = zs + off.z + sz;
          while (sl >= l.EZ) sl -= l.EZ;
          row_update(acc + sl * l.Q + (off.y + sy) * l.P + off.x, sy, sz, active);
          jy += 32;
          while (jy >= MG) { jy -= MG; ++jz; }
        }
      }
      gather_store<TORQUE>(lane, index_from_w(y.w), kc.h3, u0, u1, u2, w0, w1, w2, upair, wpair, U, W);
    }
  }
}

template <int MGT, bool GUARD, bool TORQUE, bool SAMEW>
static void gather_variant(const Geometry<float>& g, const KernelConsts<float>& kc, const BinBuffers& b,
                           const float* grid, const float* up, const float* wp, float* U, float* W,
                           cudaStream_t s) {
  const size_t smem = tile_smem_bytes(g.tile, g.MG);
  auto k = gather_tile_kernel<MGT, GUARD, TORQUE, SAMEW>;
  allow_dynamic_smem(k, kTileSmemLimit);   // any tile and support
  const int nsys = g.nsys > 1 ? g.nsys : 1;
  const int pencils = nsys * g.ntile[0] * g.ntile[1];
  // one CTA per z-pencil of tiles; pencils are split into segments when there are too few of them for
  // two waves of two CTAs per SM
  const int nseg = std::min(g.ntile[2], std::max(1, (4 * device_sm_count() + pencils - 1) / pencils));
  const int segl = (g.ntile[2] + nseg - 1) / nseg;
  const int blocks = pencils * ((g.ntile[2] + segl - 1) / segl);
  k<<<blocks, 256, smem, s>>>(g, kc, (const float4*)b.t_pos, b.tile_start, grid, up, wp, U, W, segl);
}

void launch_gather_f32(const Geometry<float>& g, const KernelConsts<float>& kc, bool torque,
                       const BinBuffers& b, const float* grid, const float* up, const float* wp,
                       float* U, float* W, cudaStream_t s, long long* launches) {
#define GATHER_CALL(MGT, GUARD)                                                                     \
  if (!torque) gather_variant<MGT, GUARD, false, true>(g, kc, b, grid, up, wp, U, W, s);           \
  else if (kc.same_width) gather_variant<MGT, GUARD, true, true>(g, kc, b, grid, up, wp, U, W, s); \
  else gather_variant<MGT, GUARD, true, false>(g, kc, b, grid, up, wp, U, W, s);
  FCM_DISPATCH_MG(g.MG, GATHER_CALL)
#undef GATHER_CALL
  *launches += 1;
}

}  // namespace fcm
