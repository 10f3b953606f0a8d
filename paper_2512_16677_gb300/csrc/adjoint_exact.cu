// adjoint_exact.cu -- the FP64 backward's products as exact digit products
// (exact.cuh), over the forward's tiled block-sparse AO tensor.
//
// For L = sum W . mo_vgl (Sec. 3.6): Abar = W C, rows (point, component) by
// AOs, and dL/dC = W^T AO, MOs by AOs, a sum over all rows.
//
//  - Abar: A = rows of W (an exponent per row), B = C^T (digits kept per
//    upload of C), k = MOs.
//  - dL/dC^T: A = columns of the AO tensor, B = columns of W, k = the points
//    (in the tiles' order) of one slab and one component, each with exponents
//    of its own: the components of AOs and weights differ by orders of
//    magnitude.  A partial result per (slab, component), added in FP64 in a
//    fixed order.  Dead blocks of the AO tensor count as zeros, and k-steps
//    whose blocks are all dead are skipped.
//
// Both keep their outputs' accuracy for any operands (exact.cuh: outputs that
// lost their terms' digits are formed with multiply-adds).  W is known on the
// device only.  So that such outputs stay few, the slicers check it as
// c_rows_kernel checks C: half of each row's (column's) entries within
// 2^-9 of the largest, all finite.  Where that fails (weights on few points
// or MOs), or the list of small outputs overflows, *unfit is set: the digit
// kernels still to come return at once (the columns of W come before those of
// the AO tensor, so that little has run by then), and the SIMT kernels that
// follow in the stream, which return at once otherwise, form the results.
//
// Bound: the slicers HBM and L2 (every AO column and W entry is read twice
// and written as 16 bytes of digits), the products the tensor pipe.  On the
// C/H chain (25 600 points, 500 AOs, 100 MOs) the backward went from 29.1 ms
// with FP64 SIMT products to 4.6 (2.7 of it dL/dR).  In FP32 the SIMT
// products are the faster ones (1.64 against 1.67 ms; 0.28 against 0.33 at
// 1600 points), so this is FP64 only.
#include "exact.cuh"

namespace qk {
namespace {

using T = double;

constexpr int kSlabGroups = 48;                 // k-steps of 16 points of a slab
constexpr size_t kAdjBudget = (size_t)1 << 30;  // digits of one range of A
constexpr int kBlock = 1024;
constexpr uint32_t kSmallCap = 1u << 20;        // small outputs listed by one product

struct AdjShape {
  int64_t P, rows;       // points, 5 P
  int N, K, nchunk;      // MOs, AOs, chunks
  int groups;            // k-steps of a row of W
  int64_t row_tiles, row_range;  // 128-row tiles of W, and those of one range
  int kg, n_mt;          // k-steps of a slab, 128-column tiles of the AO tensor
  int64_t slabs, slab_range;
  int c_parts, c_pw;     // parts of W's columns
  size_t set_bytes;      // W digits of a (slab, component)
  size_t o_unfit, o_small, o_a, o_key, o_ng, o_gl, o_b, o_ec, o_part, total;
};

AdjShape adj_shape(int64_t P, int nchunk, int64_t N, int64_t K) {
  AdjShape s{};
  s.P = P;
  s.rows = 5 * P;
  s.N = (int)N;
  s.K = (int)K;
  s.nchunk = nchunk;
  s.groups = (int)((N + kGroup - 1) / kGroup);
  s.row_tiles = (s.rows + kTileRows - 1) / kTileRows;
  auto fit = [](int64_t want, size_t each) {
    const int64_t most = std::max<int64_t>((int64_t)(kAdjBudget / each), 1);
    const int64_t ranges = (want + most - 1) / most;
    return (want + ranges - 1) / ranges;
  };
  constexpr size_t A = Shape<T>::A_BYTES;
  s.row_range = fit(s.row_tiles, (size_t)s.groups * A);
  s.kg = (int)std::min<int64_t>(kSlabGroups, (P + kGroup - 1) / kGroup);
  s.n_mt = (nchunk + 1) / 2;
  const int64_t per = (int64_t)s.kg * kGroup;
  s.slabs = (P + per - 1) / per;
  s.slab_range = fit(s.slabs, (size_t)5 * s.n_mt * s.kg * A);
  s.c_pw = part_cols<T>(N, &s.c_parts);
  s.set_bytes = digit_bytes<T>(s.c_parts, s.c_pw, (int64_t)s.kg * kGroup);
  const int64_t sets = 5 * s.slab_range, tiles = sets * s.n_mt;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t o = at;
    at += align256(bytes);
    return o;
  };
  s.o_unfit = take(3 * sizeof(int));  // and the number of listed outputs, the item counter
  s.o_small = take(kSmallCap * sizeof(uint2));
  s.o_a = take(std::max((size_t)s.row_range * s.groups, (size_t)tiles * s.kg) * A);
  s.o_key = take((size_t)std::max(s.row_range, tiles) * kTileRows * sizeof(int32_t));
  s.o_ng = take((size_t)std::max(s.row_range, tiles) * sizeof(int32_t));
  s.o_gl = take(std::max((size_t)s.row_range * s.groups, (size_t)tiles * s.kg) * sizeof(uint32_t));
  s.o_b = take((size_t)sets * s.set_bytes);
  s.o_ec = take((size_t)sets * N * sizeof(int32_t));
  s.o_part = take((size_t)tiles * kTileRows * N * sizeof(T));
  s.total = at;
  return s;
}

// An entry within 2^-9 (or so) of a largest with biased exponent `most`.
__device__ __forceinline__ int large_entry(unsigned be, unsigned most) {
  return be + 9u >= most && be > 0u ? 1 : 0;
}

// Whether W was refused already (the same answer for the whole block).
__device__ __forceinline__ bool refused(const int* unfit) {
  return __syncthreads_or(*(const volatile int*)unfit != 0) != 0;
}

// Rows of W [rows][N] from row0 on: 128-row tile t of the range, one CTA; four
// sets of 256 threads take a k-step each (two threads per row, 8 MOs each).
__global__ void __launch_bounds__(kBlock, 1)
    slice_w_rows_kernel(const T* w, int64_t rows, int N, int groups, int64_t row0, int64_t tiles,
                        unsigned char* dig, uint32_t* keys, int32_t* ng, uint32_t* gl, int* unfit,
                        uint32_t* small_num) {
  constexpr int kSets = kBlock / 256;
  __shared__ unsigned s_key[kSets][kTileRows];
  __shared__ int s_large[kTileRows];
  const int tid = threadIdx.x, set = tid >> 8, r = (tid & 255) >> 1, h = tid & 1;
  griddep_wait();
  if (refused(unfit)) return;
  if (blockIdx.x == 0 && tid == 0) *small_num = 0u;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int64_t row = row0 + t * kTileRows + r;
    const T* src = w + row * N;
    auto load = [&](int g, T(&x)[8]) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int k = g * kGroup + 8 * h + j;
        x[j] = row < rows && k < N ? src[k] : T(0);
      }
    };
    if (tid < kTileRows) s_large[tid] = 0;
    unsigned key = 0;
    for (int g = set; g < groups; g += kSets) {
      T x[8];
      load(g, x);
      key = max(key, piece_key(x, (unsigned)(2 * g + h)));
    }
    key = max(key, __shfl_xor_sync(0xffffffffu, key, 1));
    if (h == 0) s_key[set][r] = key;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSets; ++k) key = max(key, s_key[k][r]);
    const int E = key_exponent<T>(key);
    const unsigned be = key >> kPieceBits;
    if (h == 0 && set == 0) keys[t * kTileRows + r] = key;
    int large = 0;
    unsigned char* out = dig + t * groups * (int64_t)Shape<T>::A_BYTES + h * 2048 + r * 16;
    for (int g = set; g < groups; g += kSets) {
      T x[8];
      load(g, x);
#pragma unroll
      for (int j = 0; j < 8; ++j) large += large_entry(biased_exp(x[j]), be);
      store_slices(x, E, out + (int64_t)g * Shape<T>::A_BYTES, Shape<T>::A_SLICE);
      if (r == 0 && h == 0) gl[t * groups + g] = (uint32_t)g;
    }
    if (large) atomicAdd(&s_large[r], large);
    if (tid == 0) ng[t] = groups;
    __syncthreads();
    if (tid < kTileRows && row0 + t * kTileRows + tid < rows) {
      unsigned most = 0;
#pragma unroll
      for (int k = 0; k < kSets; ++k) most = max(most, s_key[k][tid] >> kPieceBits);
      if (most == kExpMax<T> || (most > 0u && 2 * s_large[tid] < N)) atomicOr(unfit, 1);
    }
    __syncthreads();
  }
}

// AO columns of slabs slab0 .. of the range: tile (set, mt), set = 5 slab +
// component, mt a pair of chunks, one CTA; 8 sets of 128 threads (a column
// each) take 8 points at a time.
__global__ void __launch_bounds__(kBlock, 1)
    slice_ao_cols_kernel(const T* a, const uint8_t* mask, int nchunk, int64_t P, int kg, int n_mt,
                         int64_t slab0, int64_t tiles, unsigned char* dig, uint32_t* keys,
                         int32_t* ng, uint32_t* gl, int* unfit) {
  constexpr int kSets = kBlock / kTileRows;
  __shared__ unsigned s_key[kSets][kTileRows];
  __shared__ int s_n;
  __shared__ uint32_t s_list[kSlabGroups];
  const int tid = threadIdx.x, col = tid & (kTileRows - 1), set = tid / kTileRows;
  const int mld = mask_ld(nchunk);
  griddep_wait();
  if (refused(unfit)) return;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int mt = (int)(t % n_mt);
    const int64_t sc = t / n_mt;
    const int c = (int)(sc % 5);
    const int64_t p0 = (slab0 + sc / 5) * kg * kGroup;
    const int q = 2 * mt + (col >> 6), loc = col & 63;
    const T* base = a + blocked_offset(0, q, nchunk, 1, 0, c, loc, (int)sizeof(T));
    constexpr int W = 128 / (int)sizeof(T);  // columns of a slice: its row pitch
    // 8 points from p of this column (zeros past the points, in dead blocks
    // and dead column groups).  They lie in one tile or two: two mask bytes,
    // then eight loads that wait on nothing else (a mask byte before each
    // load: 389 us for 25 600 points x 500 AOs, now 326).
    auto load = [&](int64_t p, T(&x)[8]) {
      const int64_t tile = p / kTilePoints;
      const int j = (int)(p - tile * kTilePoints);
      const int first = kTilePoints - j;  // points in the first tile
      const int valid = P - p < 8 ? (int)(P - p) : 8;
      auto live = [&](int64_t t) { return q < nchunk && ((mask[t * mld + q] >> (loc >> 4)) & 1u); };
      const bool live0 = valid > 0 && live(tile);
      const bool live1 = valid > first && live(tile + 1);
      const T* s0 = base + tile * nchunk * kBlockElems + 5 * j * W;
      const T* s1 = s0 + nchunk * kBlockElems - 5 * kTilePoints * W;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        x[k] = T(0);
        if (k < valid && (k < first ? live0 : live1)) x[k] = (k < first ? s0 : s1)[5 * k * W];
      }
    };
    if (tid < 64) {  // the k-steps whose points have a live block in either chunk
      const int g = tid;
      bool live = false;
      if (g < kg) {
        const int64_t pa = p0 + (int64_t)g * kGroup;
        const int64_t pb = (pa + kGroup < P ? pa + kGroup : P) - 1;
        for (int64_t tile = pa / kTilePoints; pa < P && tile <= pb / kTilePoints; ++tile) {
          live |= mask[tile * mld + 2 * mt] != 0;
          if (2 * mt + 1 < nchunk) live |= mask[tile * mld + 2 * mt + 1] != 0;
        }
      }
      const unsigned m = __ballot_sync(0xffffffffu, live);
      const int lane = tid & 31;
      if (tid < 32) {
        if (live) s_list[__popc(m & ((1u << lane) - 1u))] = (uint32_t)g;
        if (lane == 0) s_n = __popc(m);
      }
      asm volatile("bar.sync 1, 64;" ::: "memory");  // the first warp's count
      if (tid >= 32) {
        const int n0 = s_n;
        asm volatile("bar.sync 1, 64;" ::: "memory");
        if (live) s_list[n0 + __popc(m & ((1u << lane) - 1u))] = (uint32_t)g;
        if (lane == 0) s_n = n0 + __popc(m);
      } else {
        asm volatile("bar.sync 1, 64;" ::: "memory");
      }
    }
    __syncthreads();
    const int n = s_n;
    if (tid < n) gl[t * kg + tid] = s_list[tid];
    if (tid == 0) ng[t] = n;
    unsigned key = 0;
    for (int i = set; i < 2 * n; i += kSets) {
      T x[8];
      const unsigned piece = 2u * s_list[i >> 1] + (unsigned)(i & 1);
      load(p0 + 8 * (int64_t)piece, x);
      key = max(key, piece_key(x, piece));
    }
    s_key[set][col] = key;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSets; ++k) key = max(key, s_key[k][col]);
    const int E = key_exponent<T>(key);
    if (set == 0) {
      keys[t * kTileRows + col] = key;
      if (key >> kPieceBits == kExpMax<T>) atomicOr(unfit, 1);
    }
    unsigned char* out = dig + t * kg * (int64_t)Shape<T>::A_BYTES + col * 16;
    for (int i = set; i < 2 * n; i += kSets) {
      T x[8];
      load(p0 + (int64_t)s_list[i >> 1] * kGroup + 8 * (i & 1), x);
      store_slices(x, E, out + (int64_t)(i >> 1) * Shape<T>::A_BYTES + (i & 1) * 2048,
                   Shape<T>::A_SLICE);
    }
    __syncthreads();
  }
}

// Columns of W [P][5][N] at the points of slabs slab0 .. (slot s is point
// perm[s]): set (slab, component), one CTA; 8 sets of 128 threads (an MO each)
// take 8 points at a time.
__global__ void __launch_bounds__(kBlock, 1)
    slice_w_cols_kernel(const T* w, const int32_t* perm, int64_t P, int N, int kg, int pw,
                        int64_t slab0, int64_t sets, unsigned char* dig, int64_t set_bytes,
                        int32_t* ec, int* unfit, uint32_t* small_num) {
  constexpr int kSets = kBlock / 128;
  constexpr int S = Split<T>::S;
  __shared__ unsigned s_be[kSets][128];
  __shared__ int s_large[128];
  const int tid = threadIdx.x, col = tid & 127, set = tid >> 7;
  griddep_wait();
  if (refused(unfit)) return;
  if (blockIdx.x == 0 && tid == 0) *small_num = 0u;
  for (int64_t sc = blockIdx.x; sc < sets; sc += gridDim.x) {
    const int c = (int)(sc % 5);
    const int64_t p0 = (slab0 + sc / 5) * kg * kGroup;
    const int pts = (int)(P - p0 < (int64_t)kg * kGroup ? P - p0 : (int64_t)kg * kGroup);
    const int parts = (N + pw - 1) / pw;
    for (int i0 = 0; i0 < parts * pw; i0 += 128) {
      const int i = i0 + col;
      auto load = [&](int k0, T(&x)[8]) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int64_t s = p0 + k0 + k;
          x[k] = k0 + k < pts && i < N
                     ? w[((perm ? (int64_t)perm[s] : s) * 5 + c) * N + i]
                     : T(0);
        }
      };
      if (tid < 128) s_large[tid] = 0;
      unsigned be = 0;
      for (int k = set; k < 2 * kg; k += kSets) {
        T x[8];
        load(8 * k, x);
#pragma unroll
        for (int j = 0; j < 8; ++j) be = max(be, biased_exp(x[j]));
      }
      s_be[set][col] = be;
      __syncthreads();
#pragma unroll
      for (int k = 0; k < kSets; ++k) be = max(be, s_be[k][col]);
      const int E = row_exponent<T>(be);
      if (set == 0 && i < N) ec[sc * N + i] = E;
      const int part = i / pw, n = i % pw;
      int large = 0;
      for (int k = set; k < 2 * kg; k += kSets) {
        T x[8];
        load(8 * k, x);
#pragma unroll
        for (int j = 0; j < 8; ++j) large += large_entry(biased_exp(x[j]), be);
        if (part < parts)
          store_slices(x, E,
                       dig + sc * set_bytes +
                           (((int64_t)(part >> 1) * kg + (k >> 1)) * 2 + (part & 1)) *
                               (int64_t)(S * pw * 32) +
                           (k & 1) * (S * pw * 16) + n * 16,
                       pw * 16);
      }
      if (large) atomicAdd(&s_large[col], large);
      __syncthreads();
      if (set == 0 && i < N &&
          (be == kExpMax<T> || (be > 0u && 2 * s_large[col] < pts)))
        atomicOr(unfit, 1);
      __syncthreads();
    }
  }
}

// dL/dC [N][K] (the caller's AO order) from the partials [set][mt][128][N]:
// added over the sets in order, onto the earlier ranges' sum when add.
__global__ void reduce_sets_kernel(const T* part, int64_t sets, int n_mt, int N, int K,
                                   const int4* chunk, int nchunk, const int32_t* ao_caller,
                                   int add, const int* unfit, double* dC) {
  griddep_wait();
  if (*unfit != 0) return;
  const int64_t rows = (int64_t)n_mt * kTileRows;
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < rows * N;
       x += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = x / N;
    const int i = (int)(x - r * N);
    const int q = (int)(r >> 6), loc = (int)(r & 63);
    if (q >= nchunk) continue;
    const int4 ch = chunk[q];
    if (loc >= ch.w - ch.z) continue;
    double sum = 0.0;
#pragma unroll 4
    for (int64_t s = 0; s < sets; ++s) sum += (double)part[(s * rows + r) * N + i];
    const int ao = ch.z + loc;
    double* d = dC + (int64_t)i * K + (ao_caller ? ao_caller[ao] : ao);
    *d = add ? *d + sum : sum;
  }
}

// C^T [ao][ld] (padding zero) from C [mo][ldc].
__global__ void transpose_c_kernel(const T* c, int64_t ldc, int64_t mo, int64_t ao, int64_t ld,
                                   T* ct) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < ao * ld;
       x += (int64_t)gridDim.x * blockDim.x) {
    const int64_t k = x / ld, i = x - k * ld;
    ct[x] = i < mo ? c[i * ldc + k] : T(0);
  }
}

cudaError_t adjoint_products(const BasisDev& b, int64_t P, const AOTensor& ao, const T* W,
                             int64_t N, const T* ct, const void* ctdig, double* d_dC, T* abar, int64_t ld,
                             void* scratch, int* err_flag, cudaStream_t s) {
  if (!ao.tiled || !ao.blocked || ao.comps == 1) return cudaErrorInvalidValue;
  const AdjShape sh = adj_shape(P, b.nchunk, N, b.ao_num);
  unsigned char* w = (unsigned char*)scratch;
  int* unfit = (int*)(w + sh.o_unfit);
  uint32_t* small_num = (uint32_t*)unfit + 1;
  uint32_t* counter = (uint32_t*)unfit + 2;
  unsigned char* dig = w + sh.o_a;
  uint32_t* keys = (uint32_t*)(w + sh.o_key);
  int32_t* ng = (int32_t*)(w + sh.o_ng);
  uint32_t* gl = (uint32_t*)(w + sh.o_gl);
  const int sms = device_sms();
  cudaError_t e = cudaMemsetAsync(unfit, 0, sizeof(int), s);
  ExactArgs<T> x{};
  x.a = dig;
  x.key = keys;
  x.ngroups = ng;
  x.glist = gl;
  x.tile_rows = kTileRows;
  x.small = 1ull << (Split<T>::kSmallSum - 32);
  x.small_list = (uint2*)(w + sh.o_small);
  x.small_num = small_num;
  x.small_cap = kSmallCap;
  x.unfit = unfit;
  if (abar) {
    x.av = W;
    x.ldw = N;
    x.cv = ct;
    x.ldc = (int64_t)sh.groups * kGroup;
    x.kvalid = N;
    x.pw = part_cols<T>(sh.K, &x.n_parts);
    x.b = (const unsigned char*)ctdig;
    x.ec = (const int32_t*)(x.b + digit_bytes<T>(x.n_parts, x.pw, (int64_t)sh.groups * kGroup));
    x.cap = sh.groups;
    x.b_div = INT32_MAX;
    x.D = abar;
    x.ldd = ld;
    x.N = sh.K;
    x.M = sh.rows;
    for (int64_t t0 = 0; t0 < sh.row_tiles && e == cudaSuccess; t0 += sh.row_range) {
      x.tile0 = t0;
      x.tiles = std::min(sh.row_range, sh.row_tiles - t0);
      e = launch_pdl(slice_w_rows_kernel, (unsigned)std::min<int64_t>(x.tiles, sms), kBlock, 0,
                     s, W, sh.rows, sh.N, sh.groups, t0 * kTileRows, x.tiles, dig, keys, ng, gl,
                     unfit, small_num);
      if (e == cudaSuccess) e = launch_product(x, counter, err_flag, s);
      if (e == cudaSuccess)
        e = launch_pdl(mend_kernel<T, kWCt>, (unsigned)(4 * sms), kMendThreads, 0, s, x);
    }
  }
  if (d_dC) {
    unsigned char* db = w + sh.o_b;
    int32_t* ec = (int32_t*)(w + sh.o_ec);
    T* part = (T*)(w + sh.o_part);
    x.av = (const T*)ao.a;
    x.cv = W;
    x.kvalid = P;
    x.mask = ao.mask;
    x.slot = ao.perm;
    x.slab_points = sh.kg * kGroup;
    x.n_mt = sh.n_mt;
    x.nchunk = sh.nchunk;
    x.n_parts = sh.c_parts;
    x.pw = sh.c_pw;
    x.b = db;
    x.ec = ec;
    x.cap = sh.kg;
    x.b_div = sh.n_mt;
    x.b_stride = (int64_t)sh.set_bytes;
    x.D = part;
    x.ldd = N;
    x.N = N;
    x.tile0 = 0;
    for (int64_t s0 = 0; s0 < sh.slabs && e == cudaSuccess; s0 += sh.slab_range) {
      const int64_t sets = 5 * std::min(sh.slab_range, sh.slabs - s0);
      x.slab0 = s0;
      x.tiles = sets * sh.n_mt;
      x.M = x.tiles * kTileRows;
      e = launch_pdl(slice_w_cols_kernel, (unsigned)std::min<int64_t>(sets, sms), kBlock, 0, s, W,
                     ao.perm, P, sh.N, sh.kg, sh.c_pw, s0, sets, db, (int64_t)sh.set_bytes, ec,
                     unfit, small_num);
      if (e == cudaSuccess)
        e = launch_pdl(slice_ao_cols_kernel, (unsigned)std::min<int64_t>(x.tiles, sms), kBlock, 0,
                       s, (const T*)ao.a, (const uint8_t*)ao.mask, sh.nchunk, P, sh.kg, sh.n_mt,
                       s0, x.tiles, dig, keys, ng, gl, unfit);
      if (e == cudaSuccess) e = launch_product(x, counter, err_flag, s);
      if (e == cudaSuccess)
        e = launch_pdl(mend_kernel<T, kAoW>, (unsigned)(4 * sms), kMendThreads, 0, s, x);
      const int64_t n = (int64_t)sh.n_mt * kTileRows * N;
      if (e == cudaSuccess)
        e = launch_pdl(reduce_sets_kernel, (unsigned)std::min<int64_t>((n + 255) / 256, 4096),
                       256, 0, s, (const T*)part, sets, sh.n_mt, sh.N, sh.K, b.chunk, sh.nchunk,
                       (const int32_t*)b.ao_caller, s0 > 0 ? 1 : 0, (const int*)unfit, d_dC);
    }
  }
  return e;
}

// C^T padded to whole k-steps, then its digits.
size_t ct_bytes(int64_t N, int64_t K) {
  return align256((size_t)K * ((N + kGroup - 1) / kGroup * kGroup) * sizeof(T));
}

}  // namespace

size_t adjoint_exact_scratch_bytes(int64_t P, int nchunk, int64_t N, int64_t K) {
  return adj_shape(P, nchunk, N, K).total;
}

size_t adjoint_exact_ct_bytes(int64_t N, int64_t K) {
  return ct_bytes(N, K) + c_bytes<T>(K, (N + kGroup - 1) / kGroup * kGroup);
}

cudaError_t launch_adjoint_exact_ct(const double* C, int64_t N, int64_t K, void* dst, int* bad,
                                    int* bad_host, cudaStream_t s) {
  const int64_t ld = (N + kGroup - 1) / kGroup * kGroup;
  transpose_c_kernel<<<(unsigned)std::min<int64_t>((K * ld + 255) / 256, 8192), 256, 0, s>>>(
      C, K, N, K, ld, (T*)dst);
  return prepare_c((const T*)dst, (const double*)dst, N, ld, K, ld,
                   (unsigned char*)dst + ct_bytes(N, K), bad, bad_host, s);
}

cudaError_t launch_adjoint_exact(const BasisDev& b, int64_t P, const AOTensor& ao, const double* W,
                                 int64_t N, const void* ct, double* d_dC, double* abar, int64_t ld,
                                 void* scratch, const int** unfit, int* err_flag, cudaStream_t s) {
  *unfit = (const int*)scratch;  // o_unfit is the first piece
  return adjoint_products(b, P, ao, W, N, (const T*)ct,
                          (const unsigned char*)ct + ct_bytes(N, b.ao_num), d_dC, abar, ld, scratch,
                          err_flag, s);
}

}  // namespace qk
