// mo_sparse.cu -- the FP64 / FP32 MO contraction over the block-sparse AO
// tensor with fused multiply-adds.  It serves the C that mo_exact.cu's
// fixed-point split does not suit (steeply graded rows), workspaces without
// room for digits, and calls captured into a graph before C's digits exist.
//
// Eqs. 5-7, D[5P x N_mo] = AO[5P x N_ao] . C^T, restricted to what
// screening (Eq. 3) leaves: the AO tensor is in the tiled layout (25 points
// = 125 rows of a 128-row tile, 64-AO column chunks) and only the live 16-AO
// column groups of its live (tile, chunk) blocks are multiplied, as the
// sparse-AO MO product of Sec. 3.2 does; skipped terms are exact zeros.
//
// A CTA computes a 128-row x 64-column tile of D.  Per live column group it
// stages the 128 x 16 AO block (16 columns of a 128-byte-wide slice of the
// blocked layout; k-major in shared memory) and the 64 x 16 block of C in shared
// memory, double buffered so that the next group loads while this one is
// multiplied; each thread accumulates an 8-row x 4-column block in
// registers.  The output rows go to the caller's points through the tile
// permutation.  Every product and sum is a fused multiply-add, in a
// fixed order (groups ascending, k ascending within a group).
#include "internal.h"

namespace qk {
namespace {

constexpr int kThreads = 256;
constexpr int kBN = 64;    // output columns per CTA
constexpr int kBK = 16;    // one column group

template <typename T>
struct SparseArgs {
  const T* A;             // tiled AO tensor, blocked
  const uint8_t* mask;    // [tiles][mask_ld(nchunk)] live column groups
  int nchunk;
  const T* C;             // [N][ldc] chunked columns (padding zero)
  int64_t ldc;
  int64_t N;
  T* D;                   // [M][N]
  int64_t M;              // output rows (5 x points)
  const int32_t* perm;    // slot -> point (NULL: identity)
  int64_t m_tiles;
};

template <typename T>
__global__ void __launch_bounds__(kThreads)
    mo_sparse_kernel(const SparseArgs<T> a) {
  // staged blocks, double buffered: AO [2][16][128] and C [2][16][64]
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T(*As)[kBK][kTileRows] = reinterpret_cast<T(*)[kBK][kTileRows]>(smem_raw);
  T(*Cs)[kBK][kBN] =
      reinterpret_cast<T(*)[kBK][kBN]>(smem_raw + sizeof(T) * 2 * kBK * kTileRows);
  constexpr int V = 16 / (int)sizeof(T);  // values of a 16-byte piece
  struct alignas(16) Piece {
    T v[V];
  };
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;  // 16 x 16 threads
  const int n0 = blockIdx.x * kBN;
  griddep_wait();
  for (int64_t mt = blockIdx.y; mt < a.m_tiles; mt += gridDim.y) {
    const uint8_t* gm = a.mask + mt * mask_ld(a.nchunk);  // this tile's mask byte per chunk
    T acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
    // walk the live groups: (q, g) pairs in ascending order
    int q = 0, g = -1;
    auto next_group = [&](int& qq, int& gg) -> bool {
      for (;;) {
        ++gg;
        if (gg == 4) {
          gg = 0;
          ++qq;
        }
        if (qq >= a.nchunk) return false;
        if ((gm[qq] >> gg) & 1u) return true;
      }
    };
    // staging of one group into buffer b (k-major): AO rows r of the tile,
    // columns 64 q + 16 g + k; C rows n0 + n, same columns
    auto stage = [&](int b, int qq, int gg) {
      const int64_t col = (int64_t)qq * kChunkAO + 16 * gg;
      {
        // 128 rows x 16 columns: thread -> row tid / 2, columns 8 (tid & 1) .. + 7
        const int r = tid >> 1, k0 = (tid & 1) * 8;
        const Piece* src = reinterpret_cast<const Piece*>(
            a.A + blocked_offset(mt, qq, a.nchunk, 1, 0, r, 16 * gg + k0, (int)sizeof(T)));
#pragma unroll
        for (int k = 0; k < 8 / V; ++k) {
          const Piece p = src[k];
#pragma unroll
          for (int j = 0; j < V; ++j) As[b][k0 + V * k + j][r] = p.v[j];
        }
      }
      {
        // 64 rows x 16 columns: thread -> row tid / 4, columns 4 (tid & 3) .. + 3
        const int n = tid >> 2, k0 = (tid & 3) * 4;
        const int64_t row = n0 + n;
#pragma unroll
        for (int k = 0; k < 4 / V; ++k) {
          Piece p{};
          if (row < a.N) p = reinterpret_cast<const Piece*>(a.C + row * a.ldc + col + k0)[k];
#pragma unroll
          for (int j = 0; j < V; ++j) Cs[b][k0 + V * k + j][n] = p.v[j];
        }
      }
    };
    bool have = next_group(q, g);
    int buf = 0;
    if (have) stage(0, q, g);
    __syncthreads();
    while (have) {
      int q2 = q, g2 = g;
      const bool more = next_group(q2, g2);
      if (more) stage(buf ^ 1, q2, g2);  // the next group loads while this one multiplies
#pragma unroll
      for (int k = 0; k < kBK; ++k) {
        T av[8], cv[4];
#pragma unroll
        for (int i = 0; i < 8 / V; ++i)
          *reinterpret_cast<Piece*>(av + V * i) =
              reinterpret_cast<const Piece*>(&As[buf][k][ty * 8])[i];
#pragma unroll
        for (int i = 0; i < 4 / V; ++i)
          *reinterpret_cast<Piece*>(cv + V * i) =
              reinterpret_cast<const Piece*>(&Cs[buf][k][tx * 4])[i];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], cv[j], acc[i][j]);
      }
      __syncthreads();
      buf ^= 1;
      q = q2;
      g = g2;
      have = more;
    }
    // epilogue: rows 8 ty .. + 7 of the tile, columns n0 + 4 tx .. + 3
    const int64_t row0 = mt * (5 * kTilePoints);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int loc = ty * 8 + i;
      const int64_t lin = row0 + loc;
      if (loc >= 5 * kTilePoints || lin >= a.M) continue;
      const int64_t orow = a.perm ? 5 * (int64_t)a.perm[lin / 5] + lin % 5 : lin;
      T* dst = a.D + orow * a.N;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t col = n0 + 4 * tx + j;
        if (col < a.N) dst[col] = acc[i][j];
      }
    }
  }
}

template <typename T>
cudaError_t launch_sparse(const AOTensor& ao, const T* C, int64_t ldc, int64_t N, T* D,
                          int64_t out_rows, cudaStream_t s) {
  if (!ao.tiled || !ao.blocked || ao.comps == 1) return cudaErrorInvalidValue;
  const int64_t m_tiles = ao.rows / kTileRows;
  if (m_tiles == 0 || N == 0) return cudaSuccess;
  SparseArgs<T> a;
  a.A = static_cast<const T*>(ao.a);
  a.mask = ao.mask;
  a.nchunk = ao.nchunk;
  a.C = C;
  a.ldc = ldc;
  a.N = N;
  a.D = D;
  a.M = out_rows;
  a.perm = ao.perm;
  a.m_tiles = m_tiles;
  const int64_t nt = (N + kBN - 1) / kBN;
  if (nt > INT32_MAX) return cudaErrorInvalidValue;
  // enough CTAs for a few waves; each walks M tiles
  const int64_t want = 8 * (int64_t)device_sms();
  int64_t gy = (want + nt - 1) / nt;
  if (gy > m_tiles) gy = m_tiles;
  if (gy > 65535) gy = 65535;
  constexpr size_t smem = sizeof(T) * 2 * kBK * (kTileRows + kBN);
  KernelFacts f;
  cudaError_t e = kernel_facts<mo_sparse_kernel<T>>(smem, kThreads, &f);
  if (e != cudaSuccess) return e;
  return launch_pdl(mo_sparse_kernel<T>, dim3((unsigned)nt, (unsigned)gy), kThreads, smem, s, a);
}

}  // namespace

cudaError_t launch_mo_sparse(int mode, const AOTensor& ao, const void* C, int64_t ldc, int64_t N,
                             void* D, int64_t out_rows, cudaStream_t s) {
  return mode == QK_FP64
             ? launch_sparse(ao, (const double*)C, ldc, N, (double*)D, out_rows, s)
             : launch_sparse(ao, (const float*)C, ldc, N, (float*)D, out_rows, s);
}

}  // namespace qk
