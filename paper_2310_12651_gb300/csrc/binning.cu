// Spatial hashing, counting sort and cell lists (Section 4, steps 1-2).
//
// Two keys per particle: the spread/gather tile that holds the first point of
// its M_G^3 window, and the pair cell of Section 4 step 1 (m_i = max(int(L_i/r_c), 3)
// cells, index x_c + (y_c + z_c m_y) m_x). Counting sort by each key gives the
// tile-sorted arrays used by spread/gather and the cell-sorted arrays with
// start offsets used by the pair correction. The rank of a particle inside its
// bin is the value its atomic increment returned, so three kernels suffice:
// key+count, scan, scatter (and a fourth that adds up chunks of counters, where the
// scan has many). The scatter leaves the counters at zero for the next call.
// Inside an 8-point tile particles are ordered by the half of the tile's x range their
// window starts in (two counters per tile, one scan over them all): the pencil spread
// steps along x by half a tile.
#include "fcm_internal.cuh"

namespace fcm {

// System of stacked row i: the s with sys_off[s] <= i < sys_off[s + 1] (binary search).
__device__ inline int system_of(const BinBuffers& b, int i) {
  if (b.nsys <= 1 || !b.sys_off) return 0;
  int lo = 0, hi = b.nsys - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(b.sys_off + mid) <= i) lo = mid; else hi = mid - 1;
  }
  return lo;
}

template <typename R>
__global__ void __launch_bounds__(256) key_count_kernel(Geometry<R> g, int n, const R* __restrict__ pos,
                                                        BinBuffers b, int need) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0 && (need & kBinCells)) b.crowd[1] = 0;   // for the scan to fill
  if (b.n_dev) n = min(n, *b.n_dev);
  if (i >= n) return;
  const int sys = system_of(b, i);
  int bad = 0;
  R y[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) y[d] = wrap_coord(pos[3 * (size_t)i + d], g.L[d], &bad);
  if (bad) atomicOr(b.status, kStatusNonFinite);
  if (need & kBinTiles) {
    int t[3], xoff = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int i0 = pmod(window_start_d(g, d, y[d]), g.M[d]);
      t[d] = i0 / g.tile[d];
      if (d == 0) xoff = i0 - t[0] * g.tile[0];
    }
    unsigned tk = (unsigned)(t[0] + g.ntile[0] * (t[1] + g.ntile[1] * t[2]));
    if (sys) tk += (unsigned)sys * (unsigned)g.tiles_per;
    tk = kTileParts * tk + (g.tile[0] == 8 ? (unsigned)(xoff / (8 / kTileParts)) : 0u);
    b.tile_key[i] = tk;
    b.tile_rank[i] = (unsigned)atomicAdd(&b.tile_count[tk], 1);
  }
  if (need & kBinCells) {
    int c[3];
    unsigned oct = 0;   // bit d: the upper half of the cell along d
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      c[d] = cell_coord(y[d], g.cellw_inv[d], g.mcell[d]);
      if (y[d] * g.cellw_inv[d] - R(c[d]) >= R(0.5)) oct |= 1u << d;
    }
    unsigned ck = (unsigned)(c[0] + g.mcell[0] * (c[1] + g.mcell[1] * c[2]));
    if (sys) ck += (unsigned)sys * (unsigned)g.cells_per;
    // octants in Gray-code order: consecutive ones share a face (0, 1, 3, 2, 6, 7, 5, 4 are steps 0 .. 7)
    if (b.cell_parts == 8) ck = 8u * ck + ((oct >> 2) * 7u ^ ((oct >> 1 & 1u) * 3u) ^ (oct & 1u));
    b.cell_key[i] = ck;
    b.cell_rank[i] = (unsigned)atomicAdd(&b.cell_count[ck], 1);
  }
}

// Counters of one system's bins: [first, first + nb) of count, split into chunks of kScanChunk.
struct ScanPart {
  const int* count;
  int nb, chunk;
  bool tiles, last;   // tile counters (kTileParts per tile); the launch's last system
};

__device__ inline ScanPart scan_part(const BinBuffers& b, int tile_chunks) {
  const int sys = blockIdx.y, nsys = max(b.nsys, 1);
  ScanPart p;
  p.tiles = (int)blockIdx.x < tile_chunks;
  p.nb = (p.tiles ? kTileParts * b.ntiles : b.cell_parts * b.ncells) / nsys;
  p.chunk = p.tiles ? blockIdx.x : blockIdx.x - tile_chunks;
  p.count = (p.tiles ? b.tile_count : b.cell_count) + (size_t)sys * p.nb;
  p.last = sys == nsys - 1;
  return p;
}

__device__ inline int warp_total(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum of every chunk of counters (only launched for many chunks).
__global__ void __launch_bounds__(kScanThreads) chunk_sum_kernel(BinBuffers b, int tile_chunks) {
  __shared__ int part[kScanThreads / 32];
  const ScanPart p = scan_part(b, tile_chunks);
  const int lo = p.chunk * kScanChunk, hi = min(p.nb, lo + kScanChunk);
  int v = 0;
  for (int k = lo + threadIdx.x; k < hi; k += kScanThreads) v += p.count[k];
  v = warp_total(v);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = warp_total(threadIdx.x < kScanThreads / 32 ? part[threadIdx.x] : 0);
    if (threadIdx.x == 0) b.chunk_sum[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = v;
  }
}

// Lists a pair cell's parts if it is crowded.
__device__ inline void note_cell(const BinBuffers& b, int cell, int count) {
  if (count <= kCrowdCell) return;
  const int parts = crowd_parts(count);
  int* item = b.crowd + 2 + 2 * atomicAdd(&b.crowd[1], parts);
  for (int p = 0; p < parts; ++p, item += 2) {
    item[0] = cell;
    item[1] = p;
  }
}

// Exclusive scan: block (c, s) writes the starts of chunk c of system s's bins. It adds up the counters
// before its chunk by itself (from the chunk sums when they were made), so the blocks need no order. A system's
// bins are contiguous and its particles are the stacked rows from sys_off[s]: segments start there.
__global__ void __launch_bounds__(kScanThreads) scan_kernel(BinBuffers b, int tile_chunks, int use_sums) {
  __shared__ int before_w[kScanThreads / 32], own_w[kScanThreads / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const ScanPart p = scan_part(b, tile_chunks);
  const int lo = p.chunk * kScanChunk;
  int before = 0;
  if (use_sums) {
    const int* cs = b.chunk_sum + (size_t)blockIdx.y * gridDim.x + (p.tiles ? 0 : tile_chunks);
    for (int k = threadIdx.x; k < p.chunk; k += kScanThreads) before += cs[k];
  } else {
#pragma unroll 8
    for (int k = threadIdx.x; k < lo; k += kScanThreads) before += p.count[k];
  }
  constexpr int kPer = kScanChunk / kScanThreads;
  const int first = lo + kPer * threadIdx.x;
  int v[kPer], own = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    v[k] = first + k < p.nb ? p.count[first + k] : 0;
    own += v[k];
  }
  if (!p.tiles) {
    const int at = (int)blockIdx.y * p.nb + first;   // the thread's first counter
    static_assert(kPer == 4, "two neighbouring threads per cell of eight counters");
    if (b.cell_parts == 8) {
      const int cell = own + __shfl_xor_sync(0xffffffffu, own, 1);
      if (!(lane & 1)) note_cell(b, at / 8, cell);
    } else {
#pragma unroll
      for (int k = 0; k < kPer; ++k) note_cell(b, at + k, v[k]);
    }
  }
  before = warp_total(before);
  int incl = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) {
    before_w[wid] = before;
    own_w[wid] = incl;
  }
  __syncthreads();
  int excl = incl - own;
  for (int w = 0; w < kScanThreads / 32; ++w) excl += before_w[w] + (w < wid ? own_w[w] : 0);
  if (b.nsys > 1 && b.sys_off) excl += b.sys_off[blockIdx.y];
  const size_t at = (size_t)blockIdx.y * p.nb + first;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    if (first + k < p.nb) {
      if (p.tiles) {
        b.part_start[at + k] = excl;
        if ((first + k) % kTileParts == 0) b.tile_start[(at + k) / kTileParts] = excl;
      } else {
        b.cell_part_start[at + k] = excl;
        if ((first + k) % b.cell_parts == 0) b.cell_start[(at + k) / b.cell_parts] = excl;
      }
      excl += v[k];
      if (p.last && first + k == p.nb - 1) {   // the end of the last bin
        if (p.tiles) {
          b.part_start[at + k + 1] = excl;
          b.tile_start[b.ntiles] = excl;
        } else {
          b.cell_part_start[at + k + 1] = excl;
          b.cell_start[b.ncells] = excl;
        }
      }
    }
  }
}

template <typename R>
__global__ void __launch_bounds__(256) scatter_kernel(Geometry<R> g, int n, const R* __restrict__ pos,
                                                      const R* __restrict__ F, const R* __restrict__ T,
                                                      BinBuffers b, int need) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool crowded = (need & kBinCells) && b.crowd[1] > 0;
  // the counters back to zero for the next call (16 bytes per store; the arrays are padded to 256 bytes)
  const int nz_t = (need & kBinTiles) ? (kTileParts * b.ntiles + 3) / 4 : 0, nz_c = (need & kBinCells) ? (b.cell_parts * b.ncells + 3) / 4 : 0;
  for (int k = i; k < nz_t + nz_c; k += gridDim.x * blockDim.x)
    (k < nz_t ? reinterpret_cast<int4*>(b.tile_count)[k] : reinterpret_cast<int4*>(b.cell_count)[k - nz_t]) =
        make_int4(0, 0, 0, 0);
  if (b.n_dev) n = min(n, *b.n_dev);
  if (i >= n) return;
  int bad = 0;
  Vec4<R> p, f, t;
  p.x = wrap_coord(pos[3 * (size_t)i + 0], g.L[0], &bad);
  p.y = wrap_coord(pos[3 * (size_t)i + 1], g.L[1], &bad);
  p.z = wrap_coord(pos[3 * (size_t)i + 2], g.L[2], &bad);
  p.w = as_real_bits(i, R(0));
  f.x = F[3 * (size_t)i + 0]; f.y = F[3 * (size_t)i + 1]; f.z = F[3 * (size_t)i + 2]; f.w = R(0);
  if (T) { t.x = T[3 * (size_t)i + 0]; t.y = T[3 * (size_t)i + 1]; t.z = T[3 * (size_t)i + 2]; }
  else   { t.x = R(0); t.y = R(0); t.z = R(0); }
  t.w = R(0);
  // keys and ranks come from key_count_kernel; both bins are in range by construction
  if (need & kBinTiles) {
    int dt = b.part_start[b.tile_key[i]] + (int)b.tile_rank[i];
    dt = min(max(dt, 0), n - 1);
    ((Vec4<R>*)b.t_pos)[dt] = p;
    ((Vec4<R>*)b.t_F)[dt] = f;
    ((Vec4<R>*)b.t_T)[dt] = t;
  }
  if (need & kBinCells) {
    int dc = b.cell_part_start[b.cell_key[i]] + (int)b.cell_rank[i];
    dc = min(max(dc, 0), n - 1);
    b.cell_rank[i] = (unsigned)dc;   // from here on the particle's place in cell order
    if (b.c_sum) {
      const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
      ((float4*)b.c_sum)[2 * (size_t)dc] = zero;
      ((float4*)b.c_sum)[2 * (size_t)dc + 1] = zero;
      if (crowded)
        for (int k = 0; k < 3; ++k) reinterpret_cast<float4*>(b.c_sum64 + 6 * (size_t)dc)[k] = zero;
    }
    ((Vec4<R>*)b.c_pos)[dc] = p;
    ((Vec4<R>*)b.c_F)[dc] = f;
    ((Vec4<R>*)b.c_T)[dc] = t;
  }
}

template <typename R>
void launch_binning(const Geometry<R>& g, int n, const R* pos, const R* F, const R* T,
                    const BinBuffers& b, int need, cudaStream_t s, long long* launches) {
  if (n <= 0) return;
  const int nsys = b.nsys > 1 ? b.nsys : 1;
  const int tiles = (need & kBinTiles) ? b.ntiles : 0, cells = (need & kBinCells) ? b.cell_parts * b.ncells : 0;
  const int tile_chunks = scan_chunks(kTileParts * (tiles / nsys)), cell_chunks = scan_chunks(cells / nsys);
  const int blocks = (n + 255) / 256;
  key_count_kernel<R><<<blocks, 256, 0, s>>>(g, n, pos, b, need);
  *launches += 1;
  if (need == 0) return;   // no order needed (a correction that is identically zero): the position check alone
  // Every block reading all counters before its chunk costs chunks^2 / 2 chunk reads from L2: below a microsecond
  // at 16 chunks, 8 at 64 (each block's own reads are a chain of loads); past that the chunk sums pay their launch.
  const bool sums = std::max(tile_chunks, cell_chunks) > kScanSumsAbove && b.chunk_sum != nullptr;
  const dim3 grid(tile_chunks + cell_chunks, nsys);
  if (sums) {
    chunk_sum_kernel<<<grid, kScanThreads, 0, s>>>(b, tile_chunks);
    *launches += 1;
  }
  scan_kernel<<<grid, kScanThreads, 0, s>>>(b, tile_chunks, sums ? 1 : 0);
  // enough blocks for the particles and for at most eight counter stores per thread
  const int zero_blocks = (int)((((long long)kTileParts * tiles + cells) / 4 + 2 + 2047) / 2048);
  scatter_kernel<R><<<std::max(blocks, zero_blocks), 256, 0, s>>>(g, n, pos, F, T, b, need);
  *launches += 2;
}

template void launch_binning<float>(const Geometry<float>&, int, const float*, const float*, const float*,
                                    const BinBuffers&, int, cudaStream_t, long long*);
template void launch_binning<double>(const Geometry<double>&, int, const double*, const double*, const double*,
                                     const BinBuffers&, int, cudaStream_t, long long*);

__global__ void write_offsets_kernel(SysOffsets o, int n, int* dst) {
  for (int k = threadIdx.x; k <= n; k += blockDim.x) dst[k] = o.off[k];
}

void launch_write_offsets(const SysOffsets& o, int n, int* dst, cudaStream_t s, long long* launches) {
  write_offsets_kernel<<<1, 256, 0, s>>>(o, n, dst);
  *launches += 1;
}

template <typename R>
__global__ void __launch_bounds__(256) add_kernel(R* __restrict__ U, const R* __restrict__ up, R* __restrict__ W,
                                                  const R* __restrict__ wp, size_t count, const int* n_dev) {
  if (n_dev) count = min(count, 3 * (size_t)max(*n_dev, 0));
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < count; k += stride) {
    U[k] += up[k];
    if (W) W[k] += wp[k];
  }
}

template <typename R>
void launch_add(R* U, const R* up, R* W, const R* wp, size_t count, cudaStream_t s, long long* launches,
                const int* n_dev) {
  if (count == 0) return;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t want = (count + 255) / 256;
  const int blocks = (int)(want < (size_t)sms * 8 ? want : (size_t)sms * 8);
  add_kernel<R><<<blocks, 256, 0, s>>>(U, up, W, wp, count, n_dev);
  *launches += 1;
}

template void launch_add<double>(double*, const double*, double*, const double*, size_t, cudaStream_t, long long*,
                                 const int*);

__global__ void zero_kernel(uint4* p, size_t n16, unsigned char* tail, size_t ntail) {
  size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t k = i; k < n16; k += stride) p[k] = make_uint4(0, 0, 0, 0);
  if (i < ntail) tail[i] = 0;
}

void launch_zero(void* p, size_t bytes, cudaStream_t s, long long* launches) {
  if (bytes == 0) return;
  size_t n16 = bytes / 16, ntail = bytes - n16 * 16;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  size_t want = (n16 + 255) / 256;
  int blocks = (int)(want < (size_t)sms * 8 ? (want > 0 ? want : 1) : (size_t)sms * 8);
  zero_kernel<<<blocks, 256, 0, s>>>((uint4*)p, n16, (unsigned char*)p + n16 * 16, ntail);
  *launches += 1;
}

}  // namespace fcm
