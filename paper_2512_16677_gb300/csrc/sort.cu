// sort.cu -- spatial order of the points for the block-sparse tensor-core
// path.
//
// Tiles of 25 consecutive points decide which (tile, AO chunk) blocks the
// contraction multiplies (Sec. 3.2's sparse AO matrix at tile granularity).
// Points that are close in space share their nonzero AOs, so tiles cut from
// a spatial order carry fewer live blocks than tiles cut from the caller's
// order.  The order here: cells of a 32 x 32 x 32 grid over the nuclear
// bounding box (points outside are clamped to the border cells) visited in
// Morton (Z-curve) order, points of one cell by ascending index: a stable
// radix sort of the cell keys, so the permutation depends on the
// coordinates only.  The permutation changes which points share a tile, never a point's
// own values: each AO value and each output row is computed from that point
// alone.
#include "internal.h"

namespace qk {
namespace {

constexpr int kCellBits = 5;  // per axis

__device__ __forceinline__ uint32_t spread3(uint32_t v) {
  // bit i of v -> bit 3 i
  uint32_t r = 0;
#pragma unroll
  for (int i = 0; i < kCellBits; ++i) r |= ((v >> i) & 1u) << (3 * i);
  return r;
}

__device__ __forceinline__ uint32_t cell_of(float x, float lo, float inv) {
  const float f = (x - lo) * inv;
  const int c = f <= 0.0f ? 0 : (f >= (float)((1 << kCellBits) - 1) ? (1 << kCellBits) - 1 : (int)f);
  return (uint32_t)c;
}

__device__ __forceinline__ uint32_t cell_key(const PointsDev& p, int64_t i, float3 lo, float3 inv) {
  const uint32_t cx = cell_of(p.hi[i], lo.x, inv.x);
  const uint32_t cy = cell_of(p.hi[p.ld + i], lo.y, inv.y);
  const uint32_t cz = cell_of(p.hi[2 * p.ld + i], lo.z, inv.z);
  return spread3(cx) | (spread3(cy) << 1) | (spread3(cz) << 2);
}

// Stable LSD radix sort of the cell keys, 8-bit digits.  Block b owns keys
// [b * size, (b + 1) * size), size = rounds * kSortThreads with as few rounds
// as keep the blocks at kMaxBlocks.  A pass: per-block digit counts, an
// exclusive scan of each digit's counts over the blocks (a warp per digit),
// then a scatter: a key's place is the number of keys of smaller digits (each
// block scans the 256 totals), of its digit in earlier blocks and of its digit
// before it in the block (round, warp and lane order).  Equal keys therefore
// keep their index order and the result is unique.  Bound: the latency of a
// chain of short kernels, so many small blocks; with blocks of 4096 keys and
// the counts scanned by one block, a scatter took 15 us and a scan 4 us at
// 25 000 points, 16 and 51 us at 10^6; now 6 and 3 us, 13 and 4 us.
constexpr int kSortThreads = 1024;
constexpr int kMaxBlocks = 256;
constexpr int kDigitBits = 8;
constexpr int kBins = 1 << kDigitBits;
constexpr int kWarps = kSortThreads / 32;

__global__ void cell_key_kernel(PointsDev p, float3 lo, float3 inv, uint32_t* key) {
  griddep_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < p.n;
       i += (int64_t)gridDim.x * blockDim.x)
    key[i] = cell_key(p, i, lo, inv);
}

__global__ void __launch_bounds__(kSortThreads)
    digit_count_kernel(const uint32_t* key, int64_t n, int shift, int rounds, uint32_t* hist) {
  griddep_wait();
  __shared__ uint32_t cnt[kBins];
  const int t = threadIdx.x;
  if (t < kBins) cnt[t] = 0;
  __syncthreads();
  for (int r = 0; r < rounds; ++r) {
    const int64_t i = ((int64_t)blockIdx.x * rounds + r) * kSortThreads + t;
    if (i < n) atomicAdd(&cnt[(key[i] >> shift) & (kBins - 1)], 1u);
  }
  __syncthreads();
  if (t < kBins) hist[(int64_t)t * gridDim.x + blockIdx.x] = cnt[t];
}

// Exclusive scan of each digit's counts over the nb blocks in place; the
// digit's total goes behind the table.
constexpr int kScanThreads = 256;
__global__ void __launch_bounds__(kScanThreads) digit_scan_kernel(uint32_t* hist, int nb) {
  griddep_wait();
  const int lane = threadIdx.x & 31;
  const int d = blockIdx.x * (kScanThreads / 32) + (threadIdx.x >> 5);
  uint32_t* row = hist + (int64_t)d * nb;
  uint32_t run = 0;
  for (int k0 = 0; k0 < nb; k0 += 32) {
    const uint32_t c = k0 + lane < nb ? row[k0 + lane] : 0u;
    uint32_t inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (k0 + lane < nb) row[k0 + lane] = run + inc - c;
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
  if (lane == 0) hist[(int64_t)kBins * nb + d] = run;
}

// Shared memory of one block's placement step.
struct PlaceSmem {
  uint32_t wcnt[kWarps][kBins];  // per warp: keys of each digit, then their first place
  uint32_t place[kBins];         // where the next key of each digit goes
  uint32_t wsum[kBins / 32];
};

// place[d] = first[d] + the number of keys of smaller digits, total[d] keys
// each (threads below kBins bring their digit's).
__device__ __forceinline__ void digit_bases(PlaceSmem& sh, uint32_t total, uint32_t first) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (t < kBins) {
    uint32_t inc = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) sh.wsum[warp] = inc;
    sh.place[t] = inc - total + first;
  }
  __syncthreads();
  if (t < kBins) {
    uint32_t add = 0;
    for (int w = 0; w < warp; ++w) add += sh.wsum[w];
    sh.place[t] += add;
  }
}

// The place of this thread's key (digit d < kBins; kBins: no key) in round,
// warp and lane order; the whole block calls this.
__device__ __forceinline__ uint32_t place_of(PlaceSmem& sh, int d) {
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
#pragma unroll
  for (int k = t; k < kWarps * kBins; k += kSortThreads) (&sh.wcnt[0][0])[k] = 0;
  __syncthreads();
  const unsigned peers = __match_any_sync(0xffffffffu, d);
  const int wrank = __popc(peers & ((1u << lane) - 1u));
  if (d < kBins && wrank == 0) sh.wcnt[warp][d] = __popc(peers);
  __syncthreads();
  if (t < kBins) {
    uint32_t at = sh.place[t];
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const uint32_t c = sh.wcnt[w][t];
      sh.wcnt[w][t] = at;
      at += c;
    }
    sh.place[t] = at;
  }
  __syncthreads();
  const uint32_t pos = d < kBins ? sh.wcnt[warp][d] + wrank : 0u;
  __syncthreads();  // before the next round clears wcnt
  return pos;
}

__global__ void __launch_bounds__(kSortThreads)
    digit_scatter_kernel(const uint32_t* key_in, const int32_t* val_in, uint32_t* key_out,
                         int32_t* val_out, int64_t n, int shift, int rounds,
                         const uint32_t* hist) {
  griddep_wait();
  __shared__ PlaceSmem sh;
  const int t = threadIdx.x;
  const int nb = (int)gridDim.x;
  uint32_t total = 0, first = 0;
  if (t < kBins) {
    total = hist[(int64_t)kBins * nb + t];
    first = hist[(int64_t)t * nb + blockIdx.x];
  }
  digit_bases(sh, total, first);
  for (int r = 0; r < rounds; ++r) {
    const int64_t i = ((int64_t)blockIdx.x * rounds + r) * kSortThreads + t;
    const bool live = i < n;
    const uint32_t k = live ? key_in[i] : 0u;
    const uint32_t pos = place_of(sh, live ? (int)((k >> shift) & (kBins - 1)) : kBins);
    if (live) {
      key_out[pos] = k;
      val_out[pos] = val_in ? val_in[i] : (int32_t)i;
    }
  }
}

// Point i into slot s of sorted arrays of leading dimension ld.  The float
// parts are formed again (as points_soa_kernel forms them): three scattered
// reads per point instead of nine.
__device__ __forceinline__ void store_point(const PointsDev& p, int64_t i, int64_t s, int64_t ld,
                                            double* x, double* y, double* z, float* hi, float* lo) {
  const double c[3] = {p.x[i], p.y[i], p.z[i]};
  x[s] = c[0];
  y[s] = c[1];
  z[s] = c[2];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float h = __double2float_rn(c[k]);
    hi[k * ld + s] = h;
    lo[k * ld + s] = __double2float_rn(c[k] - (double)h);
  }
}

// Sorted copy of the point arrays: slot s holds point perm[s].
__global__ void gather_points_kernel(PointsDev p, const int32_t* perm, double* x, double* y,
                                     double* z, float* hi, float* lo) {
  griddep_wait();
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < p.n;
       s += (int64_t)gridDim.x * blockDim.x) {
    store_point(p, perm[s], s, p.n, x, y, z, hi, lo);
  }
}

// The whole order of at most kSmallPoints points in one block: keys, both
// passes in shared memory, the sorted arrays.  Bound: latency; eight launches
// otherwise, of which a small call consists mostly.
constexpr int kSmallRounds = 4;
constexpr int kSmallPoints = kSmallRounds * kSortThreads;
struct SmallSmem {
  PlaceSmem place;
  uint32_t cnt[kBins];
  uint32_t key[2][kSmallPoints];
  uint16_t val[2][kSmallPoints];
};
__global__ void __launch_bounds__(kSortThreads)
    small_order_kernel(PointsDev p, float3 lo, float3 inv, int32_t* perm, double* x, double* y,
                       double* z, float* hi, float* lo_out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmallSmem& sh = *reinterpret_cast<SmallSmem*>(smem_raw);
  const int t = threadIdx.x, n = (int)p.n;
  griddep_wait();
  for (int i = t; i < n; i += kSortThreads) {
    sh.key[0][i] = cell_key(p, i, lo, inv);
    sh.val[0][i] = (uint16_t)i;
  }
  for (int pass = 0; pass < 2; ++pass) {
    const int shift = pass * kDigitBits;
    if (t < kBins) sh.cnt[t] = 0;
    __syncthreads();
    for (int i = t; i < n; i += kSortThreads)
      atomicAdd(&sh.cnt[(sh.key[pass][i] >> shift) & (kBins - 1)], 1u);
    __syncthreads();
    digit_bases(sh.place, t < kBins ? sh.cnt[t] : 0u, 0u);
    for (int r = 0; r * kSortThreads < n; ++r) {
      const int i = r * kSortThreads + t;
      const bool live = i < n;
      const uint32_t k = live ? sh.key[pass][i] : 0u;
      const uint32_t pos = place_of(sh.place, live ? (int)((k >> shift) & (kBins - 1)) : kBins);
      if (live) {
        sh.key[pass ^ 1][pos] = k;
        sh.val[pass ^ 1][pos] = sh.val[pass][i];
      }
    }
    __syncthreads();
  }
  for (int s = t; s < n; s += kSortThreads) {
    const int i = sh.val[0][s];
    perm[s] = i;
    store_point(p, i, s, n, x, y, z, hi, lo_out);
  }
}

// ---- several problems in one order

// The problem that global index g falls in: the largest j with off[j] <= g
// (empty problems share their offset with the next one and are passed over).
__device__ __forceinline__ int problem_of(const int64_t* off, int nprob, int64_t g) {
  int lo = 0, hi = nprob - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= g)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

__global__ void batch_cell_key_kernel(const SortProblem* probs, const int64_t* off, int nprob,
                                      int64_t total, uint32_t* key) {
  griddep_wait();
  for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < total;
       g += (int64_t)gridDim.x * blockDim.x) {
    const int j = problem_of(off, nprob, g);
    const SortProblem& P = probs[j];
    const uint32_t cell = P.spatial ? cell_key(P.p, g - off[j], P.lo, P.inv) : 0u;
    key[g] = ((uint32_t)j << (3 * kCellBits)) | cell;
  }
}

// Sorted copy of every problem's points (slot s holds global point perm[s],
// of the problem that owns slot s) and the problem-local permutation.
__global__ void batch_gather_kernel(const SortProblem* probs, const int64_t* off, int nprob,
                                   int64_t total, const int32_t* perm, double* x, double* y,
                                   double* z, float* hi, float* lo, int32_t* perm_local) {
  griddep_wait();
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < total;
       s += (int64_t)gridDim.x * blockDim.x) {
    const int j = problem_of(off, nprob, s);
    const PointsDev& p = probs[j].p;
    const int64_t i = (int64_t)perm[s] - off[j];
    store_point(p, i, s, total, x, y, z, hi, lo);
    perm_local[s] = (int32_t)i;
  }
}

unsigned grid_for(int64_t n) {
  const int64_t b = (n + 255) / 256;
  return (unsigned)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

// Keys per thread and blocks of the sort kernels.
int sort_rounds(int64_t n) {
  const int64_t per = (int64_t)kSortThreads * kMaxBlocks;
  return n > per ? (int)((n + per - 1) / per) : 1;
}
int sort_blocks(int64_t n) {
  const int64_t size = (int64_t)sort_rounds(n) * kSortThreads;
  return (int)((n + size - 1) / size);
}
size_t al256(size_t x) { return (x + 255) / 256 * 256; }
size_t hist_bytes(int64_t n) {  // counts [kBins][blocks], then totals
  return al256(sizeof(uint32_t) * (size_t)kBins * (sort_blocks(n) + 1));
}

// The radix passes over key[0].
cudaError_t launch_passes(int passes, int64_t n, uint32_t* const key[2], int32_t* const val[2],
                          uint32_t* hist, cudaStream_t s) {
  const int nb = sort_blocks(n), rounds = sort_rounds(n);
  cudaError_t e = cudaSuccess;
  for (int pass = 0; pass < passes && e == cudaSuccess; ++pass) {
    const int in = pass & 1, out = in ^ 1, shift = kDigitBits * pass;
    e = launch_pdl(digit_count_kernel, nb, kSortThreads, 0, s, (const uint32_t*)key[in], n, shift,
                   rounds, hist);
    if (e == cudaSuccess)
      e = launch_pdl(digit_scan_kernel, kBins / (kScanThreads / 32), kScanThreads, 0, s, hist, nb);
    if (e == cudaSuccess)
      e = launch_pdl(digit_scatter_kernel, nb, kSortThreads, 0, s, (const uint32_t*)key[in],
                     (const int32_t*)(pass == 0 ? nullptr : val[in]), key[out], val[out], n, shift,
                     rounds, (const uint32_t*)hist);
  }
  return e;
}

}  // namespace

void cell_grid(const float box_lo[3], const float box_hi[3], float3* lo, float3* inv) {
  const float span = (float)(1 << kCellBits);
  lo->x = box_lo[0];
  lo->y = box_lo[1];
  lo->z = box_lo[2];
  inv->x = span / fmaxf(box_hi[0] - box_lo[0], 1e-3f);
  inv->y = span / fmaxf(box_hi[1] - box_lo[1], 1e-3f);
  inv->z = span / fmaxf(box_hi[2] - box_lo[2], 1e-3f);
}

size_t spatial_order_bytes(int64_t n) {
  return hist_bytes(n) + 2 * al256(sizeof(uint32_t) * n) + 2 * al256(sizeof(int32_t) * n) +
         al256(3 * sizeof(double) * n) + al256(6 * sizeof(float) * n);
}

int spatial_order_kernels(int64_t n) {
  constexpr int kPasses = (3 * kCellBits + kDigitBits - 1) / kDigitBits;
  if (n <= kSmallPoints) return n > 0 ? 1 : 0;
  return 2 + 3 * kPasses;
}

cudaError_t launch_spatial_order(const PointsDev& p, const float box_lo[3],
                                 const float box_hi[3], void* scratch, int32_t** perm_out,
                                 PointsDev* sorted, cudaStream_t s) {
  const int64_t n = p.n;
  unsigned char* w = (unsigned char*)scratch;
  uint32_t* hist = (uint32_t*)w;
  w += hist_bytes(n);
  uint32_t* key[2] = {(uint32_t*)w, nullptr};
  w += al256(sizeof(uint32_t) * n);
  key[1] = (uint32_t*)w;
  w += al256(sizeof(uint32_t) * n);
  int32_t* val[2] = {(int32_t*)w, nullptr};
  w += al256(sizeof(int32_t) * n);
  val[1] = (int32_t*)w;
  w += al256(sizeof(int32_t) * n);
  double* x = (double*)w;
  w += al256(3 * sizeof(double) * n);
  float* hi = (float*)w;
  sorted->n = n;
  sorted->x = x;
  sorted->y = x + n;
  sorted->z = x + 2 * n;
  sorted->hi = hi;
  sorted->lo = hi + 3 * n;
  sorted->ld = n;
  constexpr int kKeyBits = 3 * kCellBits;
  constexpr int kPasses = (kKeyBits + kDigitBits - 1) / kDigitBits;
  *perm_out = val[kPasses & 1];  // where the last pass leaves the values
  if (n == 0) return cudaSuccess;
  float3 lo, inv;
  cell_grid(box_lo, box_hi, &lo, &inv);
  // each kernel waits for its predecessor's results first thing
  // (programmatic dependent launches: only the launch latency overlaps)
  if (n <= kSmallPoints) {
    static_assert(kPasses == 2, "the one-block order makes two passes");
    KernelFacts f;
    cudaError_t e = kernel_facts<small_order_kernel>(sizeof(SmallSmem), kSortThreads, &f);
    if (e != cudaSuccess) return e;
    return launch_pdl(small_order_kernel, 1, kSortThreads, sizeof(SmallSmem), s, p, lo, inv,
                      *perm_out, x, x + n, x + 2 * n, hi, hi + 3 * n);
  }
  cudaError_t e = launch_pdl(cell_key_kernel, grid_for(n), 256, 0, s, p, lo, inv, key[0]);
  if (e == cudaSuccess) e = launch_passes(kPasses, n, key, val, hist, s);
  if (e == cudaSuccess)
    e = launch_pdl(gather_points_kernel, grid_for(n), 256, 0, s, p, (const int32_t*)*perm_out, x,
                   x + n, x + 2 * n, hi, hi + 3 * n);
  return e;
}

namespace {
int problem_bits(int nprob) {
  int b = 0;
  while (b < 31 && ((int64_t)1 << b) < nprob) ++b;
  return b;
}
}  // namespace

size_t spatial_order_batch_bytes(int64_t total, int nprob) {
  (void)nprob;
  return hist_bytes(total) + 2 * al256(sizeof(uint32_t) * total) + 3 * al256(sizeof(int32_t) * total) +
         al256(3 * sizeof(double) * total) + al256(6 * sizeof(float) * total);
}

BatchOrder spatial_order_batch_layout(void* scratch, int64_t total, int nprob) {
  BatchOrder o{};
  unsigned char* w = (unsigned char*)scratch;
  o.hist = (uint32_t*)w;
  w += hist_bytes(total);
  for (int k = 0; k < 2; ++k) {
    o.key[k] = (uint32_t*)w;
    w += al256(sizeof(uint32_t) * total);
  }
  for (int k = 0; k < 2; ++k) {
    o.val[k] = (int32_t*)w;
    w += al256(sizeof(int32_t) * total);
  }
  o.perm = (int32_t*)w;
  w += al256(sizeof(int32_t) * total);
  double* x = (double*)w;
  w += al256(3 * sizeof(double) * total);
  float* hi = (float*)w;
  o.sorted.n = total;
  o.sorted.x = x;
  o.sorted.y = x + total;
  o.sorted.z = x + 2 * total;
  o.sorted.hi = hi;
  o.sorted.lo = hi + 3 * total;
  o.sorted.ld = total;
  o.total = total;
  o.nprob = nprob;
  const int bits = 3 * kCellBits + problem_bits(nprob);
  o.passes = (bits + kDigitBits - 1) / kDigitBits;
  return o;
}

cudaError_t launch_spatial_order_batch(const BatchOrder& o, const SortProblem* d_probs,
                                       const int64_t* d_off, cudaStream_t s) {
  const int64_t n = o.total;
  if (n == 0) return cudaSuccess;
  if (3 * kCellBits + problem_bits(o.nprob) > 32) return cudaErrorInvalidValue;
  cudaError_t e = launch_pdl(batch_cell_key_kernel, grid_for(n), 256, 0, s, d_probs, d_off,
                             o.nprob, n, o.key[0]);
  if (e == cudaSuccess) e = launch_passes(o.passes, n, o.key, o.val, o.hist, s);
  if (e == cudaSuccess) {
    double* x = const_cast<double*>(o.sorted.x);
    float* hi = const_cast<float*>(o.sorted.hi);
    e = launch_pdl(batch_gather_kernel, grid_for(n), 256, 0, s, d_probs, d_off, o.nprob, n,
                   (const int32_t*)o.val[o.passes & 1], x, x + n, x + 2 * n, hi, hi + 3 * n,
                   o.perm);
  }
  return e;
}

}  // namespace qk
