// mo_exact.cu -- the FP64 and FP32 MO contraction (Eqs. 5-7) over the tiled
// block-sparse AO tensor as exact digit products (exact.cuh): the digits of
// the live 16-AO column groups, one pass per range of tiles, then the product.
#include "cluster.cuh"
#include "exact.cuh"

namespace qk {
namespace {

// AO digits of a range of tiles.  One CTA per tile: the tile's list of live
// groups, each row's key over them, then the digits.  Four sets of 256
// threads take a group each (two threads per row, 8 of its 16 columns each).
// One CTA of 1024 threads per SM keeps the tiles in flight within L2 (about
// 400 KB each in FP64), so that the second read of a tile does not go to HBM.
// Bound: HBM, 8 bytes in and 16 out per live entry in FP64, 4 and 10 in FP32.
// Calls of few tiles run a cluster of 2, 4 or 8 CTAs per tile, each taking its
// share of the groups and the row keys from all of them: a tile of many
// groups on one SM took 29 us (11 tiles, 27 chunks, FP64), on eight 11.6 us.
template <typename T>
__global__ void __launch_bounds__(kSliceThreads, 1)
    slice_ao_kernel(const T* a, const uint8_t* mask, int nchunk, int64_t tiles, unsigned char* dig,
                    uint32_t* keys, int32_t* ngroups, uint32_t* glist) {
  constexpr int kSets = kSliceThreads / 256;
  __shared__ int s_n;
  __shared__ unsigned s_key[kSets][kTileRows];
  const int tid = threadIdx.x, lane = tid & 31;
  const int set = tid >> 8, r = (tid & 255) >> 1, h = tid & 1;
  const unsigned ctas = cluster_ctas(), rank = cluster_cta();
  const int first = (int)rank * kSets + set, stride = (int)ctas * kSets;
  griddep_wait();
  for (int64_t t = blockIdx.x / ctas; t < tiles; t += gridDim.x / ctas) {
    // (each CTA of a cluster writes the same list and count)
    uint32_t* list = glist + t * (4 * (int64_t)nchunk);
    if (tid < 32) {
      int n = 0;
      for (int q0 = 0; q0 < nchunk; q0 += 32) {
        const int q = q0 + lane;
        const unsigned m = q < nchunk ? mask[t * mask_ld(nchunk) + q] & 0xFu : 0u;
        int pos = __popc(m);
        const int own = pos;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, pos, o);
          if (lane >= o) pos += v;
        }
        const int total = __shfl_sync(0xffffffffu, pos, 31);
        int at = n + pos - own;
        for (unsigned left = m; left; left &= left - 1u)
          list[at++] = 4u * (unsigned)q + (unsigned)(__ffs(left) - 1);
        n += total;
      }
      if (lane == 0) {
        s_n = n;
        ngroups[t] = n;
      }
    }
    __syncthreads();
    const int n = s_n;
    const T* base = a + t * nchunk * kBlockElems;
    auto src = [&](int i) {
      const uint32_t id = list[i];
      return base + blocked_offset(0, (int)(id >> 2), nchunk, 1, 0, r, 16 * (int)(id & 3u) + 8 * h,
                                   (int)sizeof(T));
    };
    unsigned key = 0;
#pragma unroll 2
    for (int i = first; i < n; i += stride) {
      T x[8];
      load8(src(i), x);
      key = max(key, piece_key(x, 2u * list[i] + (unsigned)h));
    }
    key = max(key, __shfl_xor_sync(0xffffffffu, key, 1));
    if (h == 0) s_key[set][r] = key;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSets; ++k) key = max(key, s_key[k][r]);
    if (ctas > 1) {
      __syncthreads();  // s_key is read
      if (h == 0 && set == 0) s_key[0][r] = key;
      cluster_barrier();
      for (unsigned k = 0; k < ctas; ++k) key = max(key, cluster_load(&s_key[0][r], k));
      cluster_barrier();  // before another tile's keys, and before any CTA leaves
    }
    const int E = key_exponent<T>(key);
    if (h == 0 && set == 0 && rank == 0) keys[t * kTileRows + r] = key;
    unsigned char* out = dig + (t * 4 * nchunk) * (int64_t)Shape<T>::A_BYTES + h * 2048 + r * 16;
#pragma unroll 2
    for (int i = first; i < n; i += stride) {
      T x[8];
      load8(src(i), x);
      store_slices(x, E, out + (int64_t)i * Shape<T>::A_BYTES, Shape<T>::A_SLICE);
    }
    __syncthreads();  // the list, s_n and s_key are read by every thread
  }
}

// Scratch of `tiles` tiles: digits, row keys, group counts and lists, and the
// product's item counter.
template <typename T>
size_t tile_scratch(int64_t tiles, int nchunk) {
  return align256((size_t)tiles * 4 * nchunk * Shape<T>::A_BYTES) +
         align256((size_t)tiles * kTileRows * sizeof(uint32_t)) +
         align256((size_t)tiles * sizeof(int32_t)) +
         align256((size_t)tiles * 4 * nchunk * sizeof(uint32_t)) + 256;
}

// The most tiles of one launch range that the budget asks room for.
template <typename T>
int64_t most_tiles(int64_t tiles, int nchunk) {
  const int64_t most = (int64_t)(kDigitBudget / ((size_t)4 * nchunk * Shape<T>::A_BYTES));
  return std::min(tiles, std::max<int64_t>(most, 1));
}
// The tiles whose digits `bytes` of scratch hold, and the equal ranges that `tiles`
// tiles are cut into.
template <typename T>
int64_t fitting_tiles(size_t bytes, int64_t tiles, int nchunk) {
  int64_t t = std::min(tiles, (int64_t)(bytes / ((size_t)4 * nchunk * Shape<T>::A_BYTES)));
  while (t > 0 && tile_scratch<T>(t, nchunk) > bytes) --t;
  return t;
}
template <typename T>
int64_t range_tiles(size_t bytes, int64_t tiles, int nchunk) {
  const int64_t most = fitting_tiles<T>(bytes, tiles, nchunk);
  if (most < 1) return 0;
  const int64_t ranges = (tiles + most - 1) / most;
  return (tiles + ranges - 1) / ranges;
}

template <typename T>
cudaError_t contract_exact(const AOTensor& ao, const T* C, const void* cdig, int64_t kpad,
                           int64_t N, T* D, int64_t out_rows, int* err_flag, cudaStream_t s) {
  if (!ao.tiled || !ao.blocked || ao.comps == 1 || !ao.scratch) return cudaErrorInvalidValue;
  if (kpad != (int64_t)ao.nchunk * kChunkAO || out_rows > INT32_MAX ||
      kpad / 8 > (int64_t)kPieceMask)
    return cudaErrorInvalidValue;
  const int64_t tiles = ao.rows / kTileRows;
  if (tiles == 0 || N == 0) return cudaSuccess;
  KernelFacts fs;
  cudaError_t e = kernel_facts<slice_ao_kernel<T>>(0, kSliceThreads, &fs);
  if (e != cudaSuccess) return e;
  if (fs.occ < 1) return cudaErrorInvalidConfiguration;
  const int64_t per = range_tiles<T>(ao.scratch_bytes, tiles, ao.nchunk);
  if (per < 1) return cudaErrorInvalidValue;
  unsigned char* dig = (unsigned char*)ao.scratch;
  uint32_t* keys = (uint32_t*)(dig + align256((size_t)per * 4 * ao.nchunk * Shape<T>::A_BYTES));
  int32_t* ng = (int32_t*)((unsigned char*)keys + align256((size_t)per * kTileRows * 4));
  uint32_t* gl = (uint32_t*)((unsigned char*)ng + align256((size_t)per * 4));
  uint32_t* counter =
      (uint32_t*)((unsigned char*)gl + align256((size_t)per * 4 * ao.nchunk * sizeof(uint32_t)));
  ExactArgs<T> x{};
  x.pw = part_cols<T>(N, &x.n_parts);
  x.a = dig;
  x.b = (const unsigned char*)cdig;
  x.key = keys;
  x.ec = (const int32_t*)(x.b + digit_bytes<T>(x.n_parts, x.pw, kpad));
  x.ngroups = ng;
  x.glist = gl;
  x.cap = 4 * ao.nchunk;
  x.small = 1ull << (sizeof(T) == 8 ? Split<T>::kSmall - 32 : Split<T>::kSmall);
  x.b_div = INT32_MAX;  // one B
  x.b_stride = 0;
  x.av = (const T*)ao.a;
  x.cv = C;
  x.ldc = kpad;
  x.D = D;
  x.ldd = N;
  x.tile_rows = 5 * kTilePoints;
  x.M = out_rows;
  x.N = N;
  x.perm = ao.perm;
  x.nchunk = ao.nchunk;
  for (int64_t t0 = 0; t0 < tiles; t0 += per) {
    x.tile0 = t0;
    x.tiles = tiles - t0 < per ? tiles - t0 : per;
    // CTAs per tile: as many as leave each a chunk and an SM
    int ctas = 1;
    while (ctas < 8 && 2 * ctas <= ao.nchunk && 2 * ctas * x.tiles <= fs.sms) ctas *= 2;
    const int64_t slots = (int64_t)fs.occ * fs.sms;
    e = launch_pdl_cluster(slice_ao_kernel<T>,
                           (unsigned)(std::min<int64_t>(x.tiles, slots) * ctas), kSliceThreads, 0,
                           ctas, s, x.av + t0 * ao.nchunk * kBlockElems,
                           ao.mask + t0 * mask_ld(ao.nchunk), ao.nchunk, x.tiles, dig, keys, ng, gl);
    if (e != cudaSuccess) return e;
    e = launch_product(x, counter, err_flag, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

size_t exact_scratch_bytes(int mode, int64_t tiles, int nchunk) {
  if (tiles == 0 || nchunk == 0) return 0;
  // room for the largest range that any part of the tiles may take
  return mode == QK_FP64 ? tile_scratch<double>(most_tiles<double>(tiles, nchunk), nchunk)
                         : tile_scratch<float>(most_tiles<float>(tiles, nchunk), nchunk);
}

int exact_kernels(int mode, const AOTensor& ao) {
  const int64_t tiles = ao.rows / kTileRows;
  if (tiles == 0 || ao.nchunk == 0 || !ao.scratch) return 0;
  const int64_t per = mode == QK_FP64 ? range_tiles<double>(ao.scratch_bytes, tiles, ao.nchunk)
                                      : range_tiles<float>(ao.scratch_bytes, tiles, ao.nchunk);
  return per < 1 ? 0 : 2 * (int)((tiles + per - 1) / per);
}

size_t exact_c_bytes(int mode, int64_t N, int64_t kpad) {
  return mode == QK_FP64 ? c_bytes<double>(N, kpad) : c_bytes<float>(N, kpad);
}

cudaError_t launch_exact_c(int mode, const void* C, const double* c64, int64_t cols, int64_t N,
                           int64_t kpad, void* dst, int* bad, int* bad_host, cudaStream_t s) {
  return mode == QK_FP64
             ? prepare_c((const double*)C, c64, cols, cols, N, kpad, dst, bad, bad_host, s)
             : prepare_c((const float*)C, c64, cols, cols, N, kpad, dst, bad, bad_host, s);
}

cudaError_t launch_mo_exact(int mode, const AOTensor& ao, const void* C, const void* cdig,
                            int64_t kpad, int64_t N, void* D, int64_t out_rows, int* err_flag,
                            cudaStream_t s) {
  return mode == QK_FP64 ? contract_exact(ao, (const double*)C, cdig, kpad, N, (double*)D,
                                          out_rows, err_flag, s)
                         : contract_exact(ao, (const float*)C, cdig, kpad, N, (float*)D, out_rows,
                                          err_flag, s);
}

}  // namespace qk
