// The Stokes solve along z in one pass over the spectrum: transform along z, inverse Stokes operator
// (Section 2.1, step 2 (b), as in spectral.cu), transform back. cuFFT transforms the (x, y) planes before
// and after.
//
// A three-dimensional transform each way with the operator between them reads and writes the spectrum seven
// times; the two z transforms and the operator are three of them and need nothing but columns in z. A block
// takes neighbouring columns (contiguous in memory) of all three components, keeps them in
// shared memory from the first read to the last write, and transforms them there: Stockham steps of radix 2
// to 16 between two copies of the columns, the first reading and the last writing global memory.
// Twiddle factors come from a table rounded from FP64. What bounds it in FP32 is issue: about 150 instructions per
// value, addresses and factors among them; the schedulers issue 57% of the time and next wait for instructions (the
// unrolled butterflies of both directions) and for the first loads, while shared memory is busy 47% and HBM moves
// its 16 bytes per value at 0.40 of the copy rate. Measured against transforms and operator in three kernels: 32
// systems of 128^3 841 -> 591 us (615 with complex values declared at the alignment of one real, two accesses for
// one), 256^3 261 -> 210 us, 240 x 240 x 16 13.5 -> 9.2 us, 13 systems of 90 x 72 x 54 65 -> 49 us, FP64 64^3 80 -> 43 us.
// Lengths of threes alone gain nothing (243^3: the whole chain 585 -> 611 us, 8 x 81^3 146 -> 147 us).
#include <cmath>
#include <vector>

#include "fcm_internal.cuh"

namespace fcm {

namespace {

constexpr int kZThreads = 192;   // a multiple of three components times the columns of a block
// Columns per block, a power of two: at least 64 bytes of them (8 in FP32, 4 in FP64), and as many as keep a block's
// two copies within 50 KB (25 KB in FP64), so that short columns still give every thread a butterfly (16 points: 19 -> 9
// us on a 240 x 240 x 16 grid); fewer again where that leaves less than two blocks per SM.
constexpr size_t kBlockSmem = 50 * 1024;
constexpr size_t kPlanSmem = kTileSmemLimit / 2 - 1024;   // the most a plan may take: two blocks per SM

template <typename R> struct Pair2;
template <> struct Pair2<float> { typedef float2 T; };
template <> struct Pair2<double> { typedef double2 T; };

__device__ inline int quot(int n, unsigned magic) { return magic ? (int)__umulhi((unsigned)n, magic) : n; }

template <typename R>
struct alignas(2 * sizeof(R)) C {   // as the float2 or double2 it is read as
  R x, y;
};
template <typename R> __device__ inline C<R> operator+(C<R> a, C<R> b) { return {a.x + b.x, a.y + b.y}; }
template <typename R> __device__ inline C<R> operator-(C<R> a, C<R> b) { return {a.x - b.x, a.y - b.y}; }
template <typename R> __device__ inline C<R> operator*(R s, C<R> a) { return {s * a.x, s * a.y}; }
template <typename R> __device__ inline C<R> mul(C<R> a, C<R> b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
// i a for the backward transform, -i a for the forward one
template <int SIGN, typename R> __device__ inline C<R> turn(C<R> a) { return SIGN < 0 ? C<R>{a.y, -a.x} : C<R>{-a.y, a.x}; }

// v <- DFT of length 2, 3, 4, 5, 8 with kernel exp(SIGN 2 pi i j k / r).
template <int SIGN, typename R>
__device__ inline void dft2(C<R>& a, C<R>& b) {
  const C<R> t = a - b;
  a = a + b;
  b = t;
}
template <int SIGN, typename R>
__device__ inline void dft4(C<R>& a, C<R>& b, C<R>& c, C<R>& d) {
  const C<R> s0 = a + c, d0 = a - c, s1 = b + d, d1 = turn<SIGN>(b - d);
  a = s0 + s1;
  b = d0 + d1;
  c = s0 - s1;
  d = d0 - d1;
}
template <int SIGN, typename R>
__device__ inline void dft(C<R> (&v)[2]) { dft2<SIGN>(v[0], v[1]); }
template <int SIGN, typename R>
__device__ inline void dft(C<R> (&v)[3]) {
  const R h = R(0.86602540378443864676);   // sin(2 pi / 3)
  const C<R> s = v[1] + v[2], d = turn<SIGN>(h * (v[1] - v[2])), m = v[0] - R(0.5) * s;
  v[0] = v[0] + s;
  v[1] = m + d;
  v[2] = m - d;
}
template <int SIGN, typename R>
__device__ inline void dft(C<R> (&v)[4]) { dft4<SIGN>(v[0], v[1], v[2], v[3]); }
template <int SIGN, typename R>
__device__ inline void dft(C<R> (&v)[5]) {
  const R c1 = R(0.30901699437494742410), c2 = R(-0.80901699437494742410);   // cos(2 pi / 5), cos(4 pi / 5)
  const R s1 = R(0.95105651629515357212), s2 = R(0.58778525229247312917);    // sin(2 pi / 5), sin(4 pi / 5)
  const C<R> a1 = v[1] + v[4], b1 = v[1] - v[4], a2 = v[2] + v[3], b2 = v[2] - v[3];
  const C<R> m1 = v[0] + c1 * a1 + c2 * a2, m2 = v[0] + c2 * a1 + c1 * a2;
  const C<R> n1 = turn<SIGN>(s1 * b1 + s2 * b2), n2 = turn<SIGN>(s2 * b1 - s1 * b2);
  v[0] = v[0] + a1 + a2;
  v[1] = m1 + n1;
  v[4] = m1 - n1;
  v[2] = m2 + n2;
  v[3] = m2 - n2;
}
template <int SIGN, typename R>
__device__ inline void dft(C<R> (&v)[8]) {
  const R h = R(0.70710678118654752440);
  // even and odd halves, then the odd ones times exp(SIGN 2 pi i k / 8)
  C<R> e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4<SIGN>(e0, e1, e2, e3);
  dft4<SIGN>(o0, o1, o2, o3);
  const C<R> w1 = h * (o1 + turn<SIGN>(o1)), w2 = turn<SIGN>(o2), w3 = h * (turn<SIGN>(o3) - o3);
  v[0] = e0 + o0; v[4] = e0 - o0;
  v[1] = e1 + w1; v[5] = e1 - w1;
  v[2] = e2 + w2; v[6] = e2 - w2;
  v[3] = e3 + w3; v[7] = e3 - w3;
}

// Coprime lengths A, B: input n = B n1 + A n2 (mod A B), output k with k = k1 (mod A), k = k2 (mod B): no factors
// between the two transforms.
template <int SIGN, int A, int B, typename R>
__device__ inline void dft_coprime(C<R> (&v)[A * B]) {
  C<R> t[A][B];
#pragma unroll
  for (int n2 = 0; n2 < B; ++n2) {
    C<R> a[A];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) a[n1] = v[(B * n1 + A * n2) % (A * B)];
    dft<SIGN>(a);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) t[k1][n2] = a[k1];
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    dft<SIGN>(t[k1]);
#pragma unroll
    for (int k = 0; k < A * B; ++k)
      if (k % A == k1) v[k] = t[k1][k % B];
  }
}

// Length A B with input n = B n1 + n2, output k = k1 + A k2, and factors exp(SIGN 2 pi i n2 k1 / A B) between, where
// cs[m] = (cos, sin)(2 pi m / A B).
template <int SIGN, int A, int B, typename R>
__device__ inline void dft_factors(C<R> (&v)[A * B], const double (&cs)[(A - 1) * (B - 1) + 1][2]) {
  C<R> t[A][B];
#pragma unroll
  for (int n2 = 0; n2 < B; ++n2) {
    C<R> a[A];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) a[n1] = v[B * n1 + n2];
    dft<SIGN>(a);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1)
      t[k1][n2] = n2 * k1 == 0 ? a[k1] : mul(a[k1], C<R>{R(cs[n2 * k1][0]), R(SIGN * cs[n2 * k1][1])});
  }
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    dft<SIGN>(t[k1]);
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = t[k1][k2];
  }
}

template <int SIGN, typename R> __device__ inline void dft(C<R> (&v)[6]) { dft_coprime<SIGN, 2, 3>(v); }
template <int SIGN, typename R> __device__ inline void dft(C<R> (&v)[10]) { dft_coprime<SIGN, 2, 5>(v); }
template <int SIGN, typename R> __device__ inline void dft(C<R> (&v)[12]) { dft_coprime<SIGN, 4, 3>(v); }
template <int SIGN, typename R>
__device__ inline void dft(C<R> (&v)[9]) {
  constexpr double cs[5][2] = {{1.0, 0.0},
                               {0.76604444311897803520, 0.64278760968653932632},    // 40 degrees
                               {0.17364817766693034885, 0.98480775301220805937},    // 80
                               {-0.5, 0.86602540378443864676},
                               {-0.93969262078590838405, 0.34202014332566873304}};  // 160
  dft_factors<SIGN, 3, 3>(v, cs);
}
template <int SIGN, typename R>
__device__ inline void dft(C<R> (&v)[16]) {
  constexpr double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173, h = 0.70710678118654752440;   // pi / 8
  constexpr double cs[10][2] = {{1.0, 0.0}, {c1, s1}, {h, h}, {s1, c1}, {0.0, 1.0},
                                {-s1, c1}, {-h, h}, {-c1, s1}, {-1.0, 0.0}, {-c1, -s1}};
  dft_factors<SIGN, 4, 4>(v, cs);
}

// One Stockham step: butterfly j reads points j + q N / r, multiplies them by exp(SIGN 2 pi i q k / (n r)) with
// k = j mod n (n = product of the earlier radices) and writes points (j / n) n r + k + q n. `in` and `out` are the
// columns in shared memory ([component][z][line]) or, where the flag says so, the spectrum itself.
template <int SIGN, int RADIX, bool GIN, bool GOUT, typename R>
__device__ inline void z_step(const ZPlan& p, int step, const C<R>* __restrict__ in, C<R>* __restrict__ out,
                              const C<R>* __restrict__ tw, int lines, size_t plane, size_t comp) {
  const int sh = p.lines_log2, LN = 1 << sh;
  const int nr = p.N / RADIX, n = p.n[step], tstep = p.tstep[step];
  for (int e = threadIdx.x; e < 3 * nr * LN; e += kZThreads) {
    const int line = e & (LN - 1), b = e >> sh;
    const int c = b >= 2 * nr ? 2 : (b >= nr ? 1 : 0), j = b - c * nr;
    const int g = quot(j, p.magic[step]), k = j - g * n;
    if ((GIN || GOUT) && line >= lines) continue;
    C<R> v[RADIX];
#pragma unroll
    for (int q = 0; q < RADIX; ++q) {
      const int z = j + q * nr;
      v[q] = GIN ? in[c * comp + (size_t)z * plane + line] : in[((c * p.N + z) << sh) + line];
    }
    if (step > 0) {
#pragma unroll
      for (int q = 1; q < RADIX; ++q) {
        C<R> w = tw[q * k * tstep];
        if (SIGN > 0) w.y = -w.y;
        v[q] = mul(v[q], w);
      }
    }
    dft<SIGN>(v);
#pragma unroll
    for (int q = 0; q < RADIX; ++q) {
      const int z = g * n * RADIX + k + q * n;
      if (GOUT) out[c * comp + (size_t)z * plane + line] = v[q];
      else out[((c * p.N + z) << sh) + line] = v[q];
    }
  }
}

template <int SIGN, bool GIN, bool GOUT, typename R>
__device__ inline void z_any_step(const ZPlan& p, int step, const C<R>* in, C<R>* out, const C<R>* tw, int lines,
                                  size_t plane, size_t comp) {
  switch (p.radix[step]) {
    case 2: z_step<SIGN, 2, GIN, GOUT>(p, step, in, out, tw, lines, plane, comp); break;
    case 3: z_step<SIGN, 3, GIN, GOUT>(p, step, in, out, tw, lines, plane, comp); break;
    case 4: z_step<SIGN, 4, GIN, GOUT>(p, step, in, out, tw, lines, plane, comp); break;
    case 5: z_step<SIGN, 5, GIN, GOUT>(p, step, in, out, tw, lines, plane, comp); break;
    case 6: z_step<SIGN, 6, GIN, GOUT>(p, step, in, out, tw, lines, plane, comp); break;
    case 8: z_step<SIGN, 8, GIN, GOUT>(p, step, in, out, tw, lines, plane, comp); break;
    case 9: z_step<SIGN, 9, GIN, GOUT>(p, step, in, out, tw, lines, plane, comp); break;
    case 10: z_step<SIGN, 10, GIN, GOUT>(p, step, in, out, tw, lines, plane, comp); break;
    case 12: z_step<SIGN, 12, GIN, GOUT>(p, step, in, out, tw, lines, plane, comp); break;
    default: z_step<SIGN, 16, GIN, GOUT>(p, step, in, out, tw, lines, plane, comp); break;
  }
}

// kx0, ky0, kz0 = 2 pi / L. SQRT: the square root of the operator (Brownian noise).
template <typename R, bool SQRT>
__global__ void __launch_bounds__(kZThreads, sizeof(R) == 4 ? 4 : 2) zsolve_kernel(ZPlan p, int Mx, int My, R kx0, R ky0, R kz0, R scale,
                                                           const typename Pair2<R>::T* __restrict__ table,
                                                           typename Pair2<R>::T* __restrict__ spectrum) {
  const int LN = 1 << p.lines_log2;
  extern __shared__ float4 zsm[];
  C<R>* tw = reinterpret_cast<C<R>*>(zsm);
  C<R>* now = tw + (p.N + 1) / 2 * 2;   // the columns, and room for the next step's
  C<R>* next = now + 3 * p.N * LN;
  const int Mh = Mx / 2 + 1;
  const size_t plane = (size_t)Mh * My, comp = plane * p.N;
  const size_t first = (size_t)blockIdx.x * LN;
  const int lines = (int)min((size_t)LN, plane - first);
  C<R>* g = reinterpret_cast<C<R>*>(spectrum) + (size_t)blockIdx.y * 3 * comp + first;
  for (int k = threadIdx.x; k < p.N; k += kZThreads) tw[k] = reinterpret_cast<const C<R>*>(table)[k];
  z_any_step<-1, true, false, R>(p, 0, g, now, tw, lines, plane, comp);
  for (int s = 1; s < p.steps; ++s) {
    __syncthreads();
    z_any_step<-1, false, false, R>(p, s, now, next, tw, lines, plane, comp);
    C<R>* t = now;
    now = next;
    next = t;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < p.N * LN; e += kZThreads) {
    const int line = e & (LN - 1), iz = e >> p.lines_log2;
    if (line >= lines) continue;
    const int l = (int)(first + line), iy = l / Mh, ix = l - iy * Mh;
    C<R>* f = now + iz * LN + line;
    C<R> a = f[0], b = f[p.N * LN], c = f[2 * p.N * LN];
    const bool nyq = ((Mx & 1) == 0 && ix == Mx / 2) || ((My & 1) == 0 && iy == My / 2) || ((p.N & 1) == 0 && iz == p.N / 2);
    const R kx = R(ix) * kx0, ky = R(iy <= My / 2 ? iy : iy - My) * ky0, kz = R(iz <= p.N / 2 ? iz : iz - p.N) * kz0;
    const R k2 = kx * kx + ky * ky + kz * kz;
    if (nyq || k2 == R(0)) {
      a = b = c = {R(0), R(0)};
    } else {
      const R ik2 = R(1) / k2;
      const C<R> d = ik2 * (kx * a + ky * b + kz * c);
      const R sc = SQRT ? scale / sqrt(k2) : scale * ik2;
      a = sc * (a - kx * d);
      b = sc * (b - ky * d);
      c = sc * (c - kz * d);
    }
    f[0] = a;
    f[p.N * LN] = b;
    f[2 * p.N * LN] = c;
  }
  for (int s = 0; s + 1 < p.steps; ++s) {
    __syncthreads();
    z_any_step<1, false, false, R>(p, s, now, next, tw, lines, plane, comp);
    C<R>* t = now;
    now = next;
    next = t;
  }
  __syncthreads();
  z_any_step<1, false, true, R>(p, p.steps - 1, now, g, tw, lines, plane, comp);
}

size_t z_smem(int N, int lines_log2, bool fp64) {
  return (fp64 ? 16 : 8) * ((size_t)(N + 1) / 2 * 2 + 6 * (size_t)N * (1 << lines_log2));
}

}  // namespace

bool make_zplan(int N, bool fp64, ZPlan* p) {
  p->N = N;
  p->steps = 0;
  // two blocks per SM at least: one reads or writes global memory while the other works in shared memory
  p->lines_log2 = fp64 ? 2 : 3;
  if (N < 2 || z_smem(N, p->lines_log2, fp64) > kPlanSmem) return false;
  while (p->lines_log2 < 6 && z_smem(N, p->lines_log2 + 1, fp64) <= (fp64 ? kBlockSmem / 2 : kBlockSmem)) p->lines_log2 += 1;
  // the fewest steps, then the smallest largest radix (every step is a pass over shared memory; a radix is registers)
  static const int kRadix[] = {2, 3, 4, 5, 6, 8, 9, 10, 12, 16};
  std::vector<int> steps(N + 1, kZMaxSteps + 1), worst(N + 1, 0), last(N + 1, 0);
  steps[1] = 0;
  for (int m = 2; m <= N; ++m) {
    if (N % m) continue;
    for (int r : kRadix) {
      if (m % r || steps[m / r] > kZMaxSteps) continue;
      const int st = steps[m / r] + 1, w = std::max(worst[m / r], r);
      if (st < steps[m] || (st == steps[m] && w < worst[m])) {
        steps[m] = st;
        worst[m] = w;
        last[m] = r;
      }
    }
  }
  if (steps[N] > kZMaxSteps) return false;
  int n = 1;
  for (int m = N; m > 1; m /= last[m]) {
    const int r = last[m], k = p->steps++;
    p->radix[k] = r;
    p->n[k] = n;
    p->tstep[k] = N / (n * r);
    p->magic[k] = n == 1 ? 0u : (unsigned)((1ull << 32) / (unsigned)n + 1);   // exact for j < 2^16
    n *= r;
  }
  return true;
}

void z_twiddles(int N, bool fp64, void* host) {
  for (int k = 0; k < N; ++k) {
    const double t = -2.0 * kPi * k / N;
    if (fp64) ((double2*)host)[k] = make_double2(std::cos(t), std::sin(t));
    else ((float2*)host)[k] = make_float2((float)std::cos(t), (float)std::sin(t));
  }
}

// factor: 0 for the operator itself, otherwise the amplitude of its square root.
template <typename R>
void launch_zsolve(const Geometry<R>& g, const ZPlan& plan, R eta, R factor, const void* table, void* spectrum,
                   cudaStream_t s, long long* launches) {
  ZPlan p = plan;
  const double mtot = (double)g.M[0] * g.M[1] * g.M[2];
  const size_t plane = (size_t)(g.M[0] / 2 + 1) * g.M[1];
  const R twopi = R(2.0 * kPi);
  const R kx0 = twopi / g.L[0], ky0 = twopi / g.L[1], kz0 = twopi / g.L[2];
  const R scale = factor == R(0) ? R(1.0 / ((double)eta * mtot)) : R((double)factor / (std::sqrt((double)eta) * mtot));
  const unsigned nsys = g.nsys > 1 ? (unsigned)g.nsys : 1u;
  auto blocks = [&]() { return (unsigned)((plane + (1u << p.lines_log2) - 1) >> p.lines_log2); };
  while (p.lines_log2 > (sizeof(R) == 8 ? 2 : 3) && blocks() * nsys < 2u * (unsigned)device_sm_count()) p.lines_log2 -= 1;
  const dim3 grid(blocks(), nsys);
  const size_t smem = z_smem(p.N, p.lines_log2, sizeof(R) == 8);
  typedef typename Pair2<R>::T T2;
  auto k = factor == R(0) ? zsolve_kernel<R, false> : zsolve_kernel<R, true>;
  allow_dynamic_smem(k, kPlanSmem);
  k<<<grid, kZThreads, smem, s>>>(p, g.M[0], g.M[1], kx0, ky0, kz0, scale, (const T2*)table, (T2*)spectrum);
  *launches += 1;
}

template void launch_zsolve<float>(const Geometry<float>&, const ZPlan&, float, float, const void*, void*, cudaStream_t,
                                   long long*);
template void launch_zsolve<double>(const Geometry<double>&, const ZPlan&, double, double, const void*, void*,
                                    cudaStream_t, long long*);

}  // namespace fcm
