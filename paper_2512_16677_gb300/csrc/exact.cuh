// exact.cuh -- FP64 and FP32 matrix products on the bf16 tensor cores through
// exact fixed-point sums: the digits of an operand and the kernel that
// multiplies them (the forward contraction, mo_exact.cu; the backward
// products, adjoint_exact.cu).
//
// Eqs. 5-7, D[5P x N_mo] = AO[5P x N_ao] . C^T, over the live 16-AO column
// groups of the tiled block-sparse AO tensor (and the backward's products W .
// C and W^T . AO), is what mo_sparse.cu computes with fused multiply-adds.
// Here each operand is split into S slices of
// 8-bit signed digits (the error-free transformation of Ozaki, Ogita, Oishi
// and Rump, Numer. Algorithms 59, 2012, with a power-of-two scale per row):
//
//   x = 2^E sum_s d_s 2^-(8 (s + 1) - 1),  |d_0| <= 64, -128 <= d_s <= 127,
//
// E from the largest magnitude of the row (AO: over the tile's live groups;
// C: over the MO's coefficients).  S = 8 keeps 63 bits below 2^E for FP64,
// S = 5 keeps 39 for FP32.  A digit is a whole number of at most 8 bits and
// so a bf16 value; the products of digits i and j add up, without rounding,
// in the FP32 accumulator of level i + j as long as the sum stays within
// 2^24, which kSeg k-steps of 16 AOs guarantee for any input (level S - 1
// takes S products per AO: two of at most 2^13 and S - 2 of at most 2^14).  After each such segment the
// epilogue adds the levels into a 64-bit (FP32) or 96-bit (FP64) integer per
// output, and rounds once at the end: the result is the exact product of the
// sliced operands, rounded, whatever the tiles, groups or point order were.
// Levels >= S are not formed; they are below the slices' own truncation.
//
// Against sequential fused multiply-adds the largest normwise error falls
// from 1.8e-15 to 9e-17 in FP64 and from 8.4e-7 to 5e-8 in FP32 (organic
// chain).
//
// What the cut at 2^(E - 63) or 2^(E - 39) costs is relative to 2^(EA + EC),
// not to the output's own terms: where one AO dominates a row (the Laplacian
// of a tight s function near its nucleus is 10^8 times its neighbours') and
// the MO's coefficient on it is zero or tiny, the output is the sum of terms
// that mostly fell off the end (C zero on the s shells, 10^-3 bohr from a
// nucleus: 4e-10 in FP64, 3e-3 in FP32, of the sum of the terms' sizes).  So
// each output below 2^(EA + EC - 14) (FP32: 15) is looked at again: unless a
// term of the 8 AOs that hold the row's largest value is within 2^-kGraded of
// the largest possible one, it is formed with multiply-adds over the live
// groups (mend_outputs, mend_kernel).  The same outputs are then off by at most 3e-15 and
// 6e-8.  The bound lies where the multiply-adds' own error is about reached;
// a factor of four less error means four times the outputs looked at.
// Of random normal C and sampled electrons one output in 1200 (2500) is looked
// at and fewer than one in 10^6 formed again; 153 600 points x 300 MOs take the
// same time within 0.5%, a call of few tiles 1 to 3 us more.  Where most are formed
// again (19 200 points within 0.1 bohr of nuclei x 300 MOs without s functions)
// FP64 takes 11.4 ms and FP32 3.6; multiply-adds throughout 18.0 and (dense) 4.7.
//
// Why: GB300 runs 2 FP64 fused multiply-adds per clock and SM, 128 FP32 ones
// and 4096 in bf16.  36 (FP64) or 15 (FP32) digit products per multiply-add
// leave the tensor cores 57 and 2 times ahead of the FP64 and FP32 units.
//
// The columns of D go in parts of pw (a multiple of 16, at most 32 in FP64 and
// 48 in FP32).  One CTA per SM computes 128 rows x two parts, each with 256
// TMEM columns of its own (one part per CTA when two would leave SMs idle).
// The S slices of a part of C lie one after another as rows of one B operand,
// so that AO slice i times C slices 0 .. S-1-i is one MMA of N = (S - i) pw,
// whose columns land on levels i .. S - 1: 8 MMAs per part and k-step in FP64
// (N = 256 .. 32, 622 clocks) and 5 in FP32 (N = 240 .. 48, 383 clocks).
// Stages are one k-step (16 AOs): S x 4 KB of AO digits and S pw x 32 B of C
// digits per part, each one contiguous bulk copy (no swizzle: 8 x 16-byte core
// matrices; they run at the same rate as the swizzled layouts).  Each part has
// its own issuing warp and epilogue warps, and the second part's segments end
// half a segment later, so that one part multiplies while the other is read
// out of TMEM.
//
// Roles (640 threads): warps 0-7 and 8-15 epilogue of part 0 and 1 (a TMEM
// lane quarter and half of the part's columns each: one warp per scheduler
// would leave the read-out latency-bound and longer than the ring can hide),
// lane 0 of warp 16 copies the AO digits and that of warp 17 the C digits
// (one copy for both parts: a thread's copies complete about 600 clocks apart
// whatever their size), warps 18 and 19 issue the MMAs of part 0 and 1
// (warp 18 allocates TMEM).
// Every wait is bounded (clock64); a wait that gives up records a code in the
// caller's error word and raises the CTA's abort flag.
#pragma once

#include <algorithm>

#include "tc_common.cuh"

namespace qk {
namespace {

using namespace tc;

constexpr int kEpiWarps = 16;
constexpr int kIssuer = kEpiWarps + 2;  // first MMA warp, after two producers
constexpr int kThreads = 32 * (kIssuer + 2);
constexpr int kSliceThreads = 1024;
constexpr int kPartCols = 256;         // TMEM columns of one part
constexpr int kItems = 4;              // items on their way between the roles
constexpr int kGroup = 16;             // AOs of one k-step
constexpr int kNonFinite = -(1 << 28); // row exponent of a row with an infinity or NaN
// Two factors whose magnitudes are 2^-kGraded of their rows' largest together
// count as large terms.
constexpr unsigned kGraded = 9;
// Row keys: the largest biased exponent of the row, above the number of the
// 8-element piece that holds it (the last such piece).
constexpr int kPieceBits = 21;
constexpr uint32_t kPieceMask = (1u << kPieceBits) - 1u;
constexpr size_t kSmemLimit = 232448;
// Digits of one launch range: enough tiles for many waves of CTAs, a bound
// on the scratch memory.
constexpr size_t kDigitBudget = (size_t)4 << 30;

template <typename T>
struct Split;
template <>
struct Split<double> {
  static constexpr int S = 8;        // slices
  static constexpr int kSeg = 9;     // k-steps whose level sums stay within 2^24
  static constexpr int kPart = 32;   // most columns of a part: S kPart <= 256
  static constexpr int kStages = 4;
  // D = 2^(EA + EC - kExp) V, V = sum_l V_l 2^(8 (S - 1 - l))
  static constexpr int kExp = 14 + 8 * (S - 1);
  // outputs with |V| below 2^kSmall are looked at (the backward's: below
  // 2^kSmallSum, parts of longer sums)
  static constexpr int kSmall = kExp - 14;
  static constexpr int kSmallSum = kExp - 17;
};
template <>
struct Split<float> {
  static constexpr int S = 5;
  static constexpr int kSeg = 16;
  static constexpr int kPart = 48;
  static constexpr int kStages = 5;
  static constexpr int kExp = 14 + 8 * (S - 1);
  static constexpr int kSmall = kExp - 15;
};
static_assert((Split<double>::S - 1) * Split<double>::kSeg * kGroup * 128 * 128 <= 1 << 24, "exact");
static_assert((Split<float>::S - 1) * Split<float>::kSeg * kGroup * 128 * 128 <= 1 << 24, "exact");

template <typename T>
struct Shape {
  using P = Split<T>;
  static constexpr uint32_t A_SLICE = kTileRows * kGroup * 2;  // 4 KB
  static constexpr uint32_t A_BYTES = P::S * A_SLICE;
  static constexpr uint32_t B_MAX = P::S * P::kPart * kGroup * 2;  // one part
  static constexpr uint32_t STAGE = A_BYTES + 2 * B_MAX;
  // output staging per warp: OUT columns x 32 rows of Sum (column pitch 33)
  static constexpr int OUT = 32 / (int)sizeof(T);
  static constexpr uint32_t EPI_WARP = (OUT * 33 * (sizeof(T) == 8 ? 12 : 8) + 15) / 16 * 16;
  static constexpr uint32_t EPI = kEpiWarps * EPI_WARP;
  static constexpr size_t SMEM = 128 + (size_t)P::kStages * STAGE + EPI;
  static_assert(SMEM + 512 + kEpiWarps * P::kPart * 2 <= kSmemLimit, "shared memory budget");
  static_assert(P::kPart % 16 == 0 && P::S * P::kPart <= kPartCols, "TMEM columns of a part");
  static_assert(A_BYTES % 128 == 0 && B_MAX % 128 == 0, "16-byte copies");
};

// ------------------------------------------------------------------ digits

__device__ __forceinline__ unsigned biased_exp(double x) {
  return ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
}
__device__ __forceinline__ unsigned biased_exp(float x) {
  return (__float_as_uint(x) >> 23) & 0xffu;
}
template <typename T>
constexpr unsigned kExpMax = sizeof(T) == 8 ? 0x7ffu : 0xffu;
// Row exponent E with |x| < 2^(E - 1) for every x of the row, from the
// largest biased exponent.
template <typename T>
__device__ __forceinline__ int row_exponent(unsigned be) {
  if (be == kExpMax<T>) return kNonFinite;
  return (int)(be > 0u ? be : 1u) - (sizeof(T) == 8 ? 1021 : 125);
}
// The key of 8 values.
template <typename T>
__device__ __forceinline__ uint32_t piece_key(const T (&x)[8], uint32_t piece) {
  unsigned be = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) be = max(be, biased_exp(x[j]));
  return (be << kPieceBits) | piece;
}
template <typename T>
__device__ __forceinline__ int key_exponent(uint32_t key) {
  return row_exponent<T>(key >> kPieceBits);
}

// x 2^-E in fixed point (63 or 39 fraction bits, round half up in
// magnitude), each byte offset by 128: the bytes are d_s + 128, d_{S-1} in the
// lowest.
__device__ __forceinline__ uint64_t digits_of(double x, int E) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ffu);
  const uint64_t man = (b & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull);
  const int sh = (e ? e : 1) - 1012 - E;  // <= 9
  uint64_t m;
  if (sh >= 0)
    m = man << sh;
  else
    m = sh > -54 ? (man + (1ull << (-sh - 1))) >> -sh : 0ull;
  if (b >> 63) m = 0ull - m;
  return m + 0x8080808080808080ull;
}
__device__ __forceinline__ uint64_t digits_of(float x, int E) {
  const uint32_t b = __float_as_uint(x);
  const int e = (int)((b >> 23) & 0xffu);
  const uint32_t man = (b & 0x7fffffu) | (e ? 1u << 23 : 0u);
  const int sh = (e ? e : 1) - 111 - E;  // <= 14
  uint64_t m;
  if (sh >= 0)
    m = (uint64_t)man << sh;
  else
    m = sh > -25 ? (man + (1u << (-sh - 1))) >> -sh : 0u;
  if (b >> 31) m = 0ull - m;
  return m + 0x8080808080ull;
}
// Digit s of two numbers as a bf16 pair (the byte becomes the low mantissa
// byte of 2^23, the offset leaves by an exact subtraction).
template <int kByte>
__device__ __forceinline__ uint32_t digit_pair(uint32_t w0, uint32_t w1) {
  const float f0 = __uint_as_float(__byte_perm(w0, 0x4B000000u, 0x7540 | kByte)) - 8388736.0f;
  const float f1 = __uint_as_float(__byte_perm(w1, 0x4B000000u, 0x7540 | kByte)) - 8388736.0f;
  return __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
}
// Slices of 8 consecutive elements of one row, 16 bytes each, `stride` bytes
// apart from `dst`.  Rows with an infinity or NaN get zeros (their outputs are
// small sums and so looked at).
template <typename T>
__device__ __forceinline__ void store_slices(const T (&x)[8], int E, unsigned char* dst,
                                             uint32_t stride) {
  uint32_t hi[8], lo[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint64_t u = digits_of(E == kNonFinite ? T(0) : x[j], E);
    hi[j] = (uint32_t)(u >> 32);
    lo[j] = (uint32_t)u;
  }
  constexpr int S = Split<T>::S;
#define QK_SLICE(s_, w_, b_)                                                 \
  *reinterpret_cast<uint4*>(dst + (s_) * stride) =                           \
      make_uint4(digit_pair<b_>(w_[0], w_[1]), digit_pair<b_>(w_[2], w_[3]), \
                 digit_pair<b_>(w_[4], w_[5]), digit_pair<b_>(w_[6], w_[7]));
  if constexpr (S == 8) {
    QK_SLICE(0, hi, 3) QK_SLICE(1, hi, 2) QK_SLICE(2, hi, 1)
  }
  QK_SLICE(S - 5, hi, 0)
  QK_SLICE(S - 4, lo, 3) QK_SLICE(S - 3, lo, 2) QK_SLICE(S - 2, lo, 1) QK_SLICE(S - 1, lo, 0)
#undef QK_SLICE
  static_assert(S == 5 || S == 8, "digit layout");
}

__device__ __forceinline__ void load8(const double* p, double (&x)[8]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const double2 v = reinterpret_cast<const double2*>(p)[j];
    x[2 * j] = v.x;
    x[2 * j + 1] = v.y;
  }
}
__device__ __forceinline__ void load8(const float* p, float (&x)[8]) {
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float4 v = reinterpret_cast<const float4*>(p)[j];
    x[4 * j] = v.x;
    x[4 * j + 1] = v.y;
    x[4 * j + 2] = v.z;
    x[4 * j + 3] = v.w;
  }
}

// Row exponents of C [rows][ld] (cols valid; one warp per row), and whether C
// suits the split: in every window of 64 consecutive AOs at least half of each
// MO's coefficients are within 2^-9 of its largest, so that few outputs are
// small beside 2^(EA + EC) and formed again with multiply-adds (any C is right,
// a steeply graded one would be slow); and every value is an ordinary one in FP32
// too.  bad (zero before): bit 0 not for FP64, bit 1 not for FP32.
template <typename T>
__global__ void c_rows_kernel(const double* c, int64_t rows, int64_t cols, int64_t ld, int32_t* ec,
                              int* bad) {
  const int64_t r = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (r >= rows) return;
  const double* x = c + r * ld;
  double top = 0.0;
  int flags = 0;
#pragma unroll 4
  for (int64_t k = lane; k < cols; k += 32) {
    const double v = fabs(x[k]);
    if (!(v <= 1.7976931348623157e308)) flags = 3;
    top = fmax(top, v);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
  const bool finite = __all_sync(0xffffffffu, flags == 0);
  if (top > 3.0e38 || (top > 0.0 && top < 1.0e-30)) flags |= 2;
  // an MO without any coefficient is exactly zero either way
  const double low = top * (1.0 / (1 << kGraded));
#pragma unroll 4
  for (int64_t w = 0; w < cols; w += 64) {
    const int64_t k0 = w + 64 <= cols ? w : (cols > 64 ? cols - 64 : 0);
    const int n = (int)(cols - k0 < 64 ? cols - k0 : 64);
    const bool a = lane < n && fabs(x[k0 + lane]) >= low;
    const bool b = lane + 32 < n && fabs(x[k0 + lane + 32]) >= low;
    if (2 * (__popc(__ballot_sync(0xffffffffu, a)) + __popc(__ballot_sync(0xffffffffu, b))) < n &&
        top > 0.0)
      flags |= 3;
  }
  flags = __reduce_or_sync(0xffffffffu, flags);
  if (lane == 0) {
    ec[r] = finite ? row_exponent<T>(biased_exp((T)top)) : kNonFinite;
    if (flags) atomicOr(bad, flags);
  }
}

// C digits: [pair of parts][group][part of the pair][k half][slice][pw / 8]
// [8 columns][8 AOs] bf16.  One thread per (column, group, half); columns past
// N are zeros.
template <typename T>
__global__ void slice_c_kernel(const T* c, int64_t N, int64_t ld, int pw, int n_parts,
                               const int32_t* ec, unsigned char* dig, int* bad) {
  constexpr int S = Split<T>::S;
  if (blockIdx.x == 0 && threadIdx.x == 0) *bad = 0;  // it has been copied
  const int64_t groups = ld / kGroup;
  const int64_t total = (int64_t)n_parts * pw * groups * 2;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int h = (int)(i & 1);
    const int64_t g = (i >> 1) % groups;
    const int64_t row = (i >> 1) / groups;
    const int64_t part = row / pw;
    const int n = (int)(row % pw);
    T x[8] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
    int E = 0;
    if (row < N) {
      load8(c + row * ld + g * kGroup + 8 * h, x);
      E = ec[row];
    }
    unsigned char* dst =
        dig + (((part >> 1) * groups + g) * 2 + (part & 1)) * (int64_t)(S * pw * 32) +
        h * (S * pw * 16) + n * 16;
    store_slices(x, E, dst, pw * 16);
  }
}

// ------------------------------------------------------------- contraction

// What a product multiplies, for outputs formed with multiply-adds: element k of
// row r of A and of column n of B.
enum Operands {
  kAoC,   // the tile's row r, AO k (chunked columns) times C [n][ldc] at k (mend_outputs)
  kWCt,   // W [row][ldw] at MO k times C^T [n][ldc] at k
  kAoW,   // AO column r at point k of the slab times W [point][5][N] at MO n
};

template <typename T>
struct ExactArgs {
  const unsigned char* a;    // A digits [tile][cap][S][2][128][8]
  const unsigned char* b;    // B digits [set][pair of parts][cap]...
  const uint32_t* key;       // [tile][128] row keys of A
  const int32_t* ec;         // [set][N]
  const int32_t* ngroups;    // [tile] k-steps
  const uint32_t* glist;     // [tile][cap] the group of B that each multiplies
  int cap;                   // groups a tile (and B) has room for
  int b_div;                 // tiles t of one B set: t / b_div
  int64_t b_stride;          // bytes of a B set
  const T* av;               // the AO tensor (kAoC, kAoW) or W
  const T* cv;               // C, C^T or W
  int64_t ldw, ldc;
  int64_t kvalid;            // kWCt: MOs; kAoW: points in all
  const uint8_t* mask;       // kAoW: live groups of the AO tensor's blocks
  const int32_t* slot;       // kAoW: slot -> point (NULL: identity)
  int64_t slab0;             // kAoW: first slab of the range
  int slab_points, n_mt;     // kAoW: points of a slab; 128-column tiles
  uint64_t small;            // 2^kSmall or 2^kSmallSum (FP64: 2^32 less)
  uint2* small_list;         // small outputs (128 tile + row, column), for mend_kernel
  uint32_t* small_num;       //   (NULL: mended by the product kernel itself), their
  uint32_t small_cap;        //   number, and the list's room; more of them set *unfit
  int* unfit;                // nonzero: nothing is done (NULL: always done)
  T* D;                      // [M][ldd]
  int64_t ldd;
  int tile_rows;             // rows of D per tile (125: vgl tiles, through perm; or 128)
  int64_t M, N;
  const int32_t* perm;       // slot -> point (NULL: identity)
  int64_t tile0, tiles;      // first tile of the range; tiles of the range
  int n_parts, pw;           // parts of D's columns, and the columns of each
  int ppt, n_tiles;          // parts per CTA (1 or 2), N tiles of ppt parts
  int nchunk;
  int block_m;               // tiles of one scheduling block
  uint32_t* counter;         // items handed out so far (zero at launch); NULL: fixed strides
};

// Item p: blocks of block_m tiles x every N tile, the tiles of a block
// fastest, so that the CTAs of a moment share both AO and C digits in L2.  The N
// tiles rotate from block to block: a CTA would else keep one N tile, and with
// an odd number of parts the last one is half the work of the others (FP32, 300
// MOs, 38 400 points: 995 -> 925 us).
template <typename T>
__device__ __forceinline__ void item_of(const ExactArgs<T>& x, uint32_t p, uint32_t& mt, int& nt) {
  // (fewer than 2^31 items: D would not fit the device otherwise)
  const uint32_t per = (uint32_t)x.block_m * (uint32_t)x.n_tiles;
  const uint32_t blk = p / per;
  const uint32_t r = p - blk * per;
  const uint32_t m0 = blk * (uint32_t)x.block_m;
  const uint32_t left = (uint32_t)x.tiles - m0;
  const uint32_t mb = left < (uint32_t)x.block_m ? left : (uint32_t)x.block_m;
  const uint32_t k = r / mb;
  nt = (int)((k + blk) % (uint32_t)x.n_tiles);
  mt = m0 + r - k * mb;
}
// The part of D's columns that a CTA's part q of N tile nt is (-1: none).
template <typename T>
__device__ __forceinline__ int part_of(const ExactArgs<T>& x, int nt, int q) {
  const int p = nt * x.ppt + q;
  return q < x.ppt && p < x.n_parts ? p : -1;
}

// No-swizzle K-major operand: 8 x 16-byte core matrices, `lbo` bytes between
// the two K halves, 128 bytes between 8-row groups; descriptor version 1.
__device__ __forceinline__ uint64_t core_desc(uint32_t addr, uint32_t lbo) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(lbo >> 4) << 16) |
         ((uint64_t)(128 >> 4) << 32) | ((uint64_t)1 << 46);
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

// Columns taddr .. + 7 of this warp's TMEM lanes (no wait).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr));
}

// A level sum v below 2^22 in magnitude is an integer offset by kBias in the
// bits of v + 1.5 2^23 (conversions run at an eighth of that addition's rate);
// a pair of levels a, b goes into 32 bits as 256 a + b + kPair without
// overflow.  The running sums keep these offsets, one per segment, and drop
// them at the end.
constexpr uint32_t kBias = 0x4B400000u;
constexpr uint32_t kPair = kBias * 257u;  // mod 2^32: 0x8B400000
__device__ __forceinline__ uint32_t biased(float v) { return __float_as_uint(v + 12582912.0f); }

// a m + c, 32 x 32 + 64 bits: one instruction where a shift and an addition of
// 64 bits take four.
__device__ __forceinline__ uint64_t mad_wide(uint32_t a, uint32_t m, uint64_t c) {
  uint64_t d;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(m), "l"(c));
  return d;
}

// The offset pair of two level sums: in 32 bits when both are small, else
// whole (sums up to 2^24 that operands with most digits at their limits reach).
__device__ __forceinline__ uint32_t level_pair_small(uint32_t a, uint32_t b) {
  return biased(__uint_as_float(a)) * 256u + biased(__uint_as_float(b));
}
__device__ __forceinline__ uint64_t level_pair(uint32_t a, uint32_t b) {
  return (uint64_t)((int64_t)__float2int_rn(__uint_as_float(a)) * 256 +
                    __float2int_rn(__uint_as_float(b)) + (int64_t)kPair);
}

// Running integer sums of one output over its segments.  add<I>: the offset
// pair of levels 2 I and 2 I + 1 of a segment.
template <typename T>
struct Sum;
template <>
struct Sum<float> {
  uint64_t t;
  __device__ __forceinline__ void clear() { t = 0; }
  template <int I>
  __device__ __forceinline__ void add(uint64_t pair) {
    t += pair << (I == 0 ? 24 : 8);
  }
  template <int I>
  __device__ __forceinline__ void add(uint32_t pair) {
    t = mad_wide(pair, 1u << (I == 0 ? 24 : 8), t);
  }
  __device__ __forceinline__ void add_last(uint32_t v) {  // level 4
    t += (uint64_t)((int64_t)__float2int_rn(__uint_as_float(v)) + (int64_t)kBias);
  }
  __device__ __forceinline__ void add_last_small(uint32_t v) { t += biased(__uint_as_float(v)); }
  // without the offsets of n segments
  __device__ __forceinline__ void settle(int n) {
    t -= (uint64_t)n * ((uint64_t)kPair * ((1u << 24) + 256u) + kBias);
  }
  // column c, row r of a staging area
  __device__ __forceinline__ void put(unsigned char* st, int c, int r) const {
    reinterpret_cast<uint64_t*>(st)[c * 33 + r] = t;
  }
  __device__ __forceinline__ void get(const unsigned char* st, int c, int r) {
    t = reinterpret_cast<const uint64_t*>(st)[c * 33 + r];
  }
  // 2^k t, rounded to nearest (the 64-bit integer by its leading 24 bits: the
  // conversion instruction would hold up the next segment); *small: |t| < limit
  __device__ __forceinline__ float value(int k, uint64_t limit, bool* small) const {
    k = k < -252 ? -252 : (k > 252 ? 252 : k);  // beyond: 0 or an infinity either way
    const int k1 = k >> 1, k2 = k - k1;
    const bool neg = (int64_t)t < 0;
    const uint64_t m = neg ? 0ull - t : t;
    *small = m < limit;
    if (m == 0ull) return 0.0f;
    const int z = __clzll((long long)m);
    const uint32_t top = (uint32_t)((m << z) >> 39);  // 25 bits
    const uint32_t man = (top >> 1) + (top & 1u);     // 2^23 .. 2^24
    const uint32_t b = ((uint32_t)(127 + 63 - z) << 23) + (man - (1u << 23)) + (neg ? 1u << 31 : 0u);
    return __uint_as_float(b) * __uint_as_float((uint32_t)(127 + k1) << 23) *
           __uint_as_float((uint32_t)(127 + k2) << 23);
  }
};
template <>
struct Sum<double> {
  int64_t hi;   // t = 2^32 hi + lo
  uint32_t lo;
  __device__ __forceinline__ void clear() {
    hi = 0;
    lo = 0u;
  }
  template <int I>
  __device__ __forceinline__ void add(uint64_t pair) {
    if constexpr (I < 2) {
      hi = (int64_t)((uint64_t)hi + (pair << (I == 0 ? 16 : 0)));
    } else {
      // a whole pair may be negative (level sums down to -2^24): its borrow is
      // the sign-extended upper half
      const uint64_t l = (pair << (I == 2 ? 16 : 0)) + lo;
      lo = (uint32_t)l;
      hi += (int64_t)l >> 32;
    }
  }
  template <int I>
  __device__ __forceinline__ void add(uint32_t pair) {
    if constexpr (I < 2) {
      hi = (int64_t)mad_wide(pair, I == 0 ? 1u << 16 : 1u, (uint64_t)hi);
    } else {
      const uint64_t l = mad_wide(pair, I == 2 ? 1u << 16 : 1u, lo);
      lo = (uint32_t)l;
      hi = (int64_t)((uint64_t)hi + (l >> 32));
    }
  }
  // without the offsets of n segments
  __device__ __forceinline__ void settle(int n) {
    const uint64_t off = (uint64_t)n * ((uint64_t)kPair * ((1u << 16) + 1u));
    const uint64_t l = (uint64_t)lo - off;  // borrows from hi
    hi -= (int64_t)off - ((int64_t)l >> 32);
    lo = (uint32_t)l;
  }
  __device__ __forceinline__ void put(unsigned char* st, int c, int r) const {
    reinterpret_cast<int64_t*>(st)[c * 33 + r] = hi;
    reinterpret_cast<uint32_t*>(st + Shape<double>::OUT * 33 * 8)[c * 33 + r] = lo;
  }
  __device__ __forceinline__ void get(const unsigned char* st, int c, int r) {
    hi = reinterpret_cast<const int64_t*>(st)[c * 33 + r];
    lo = reinterpret_cast<const uint32_t*>(st + Shape<double>::OUT * 33 * 8)[c * 33 + r];
  }
  // 2^k t, rounded to nearest.  Integer arithmetic: GB300 converts and adds
  // 2 FP64 values per clock and SM, which would hold up the next segment.
  // *small: |t| < 2^32 limit.
  __device__ __forceinline__ double value(int k, uint64_t limit, bool* small) const {
    const bool neg = hi < 0;
    uint64_t mh = (uint64_t)hi;
    uint32_t ml = lo;
    if (neg) {
      ml = 0u - ml;
      mh = ~mh + (ml == 0u ? 1ull : 0ull);
    }
    *small = mh < limit;
    uint32_t w2 = (uint32_t)(mh >> 32), w1 = (uint32_t)mh, w0 = ml;
    int e = 95;  // exponent of the leading bit
    if (w2 == 0u) {
      w2 = w1;
      w1 = w0;
      w0 = 0u;
      e = 63;
      if (w2 == 0u) {
        w2 = w1;
        w1 = 0u;
        e = 31;
      }
    }
    if (w2 == 0u) return 0.0;
    const int z = __clz((int)w2);
    e -= z;
    const uint32_t h = __funnelshift_l(w1, w2, z), l = __funnelshift_l(w0, w1, z);
    const uint64_t man = (((uint64_t)(h >> 11) << 32) | __funnelshift_r(l, h, 11)) +
                         ((l >> 10) & 1u);  // 2^52 .. 2^53
    const int be = e + k + 1023;
    if (be >= 1 && be <= 2045) {
      const uint64_t b = ((uint64_t)(uint32_t)((be - 1) << 20) << 32) + man + (neg ? 1ull << 63 : 0ull);
      return __longlong_as_double((long long)b);
    }
    const double v = scalbn((double)man, e - 52 + k);
    return neg ? -v : v;
  }
};

// Levels 2 I and 2 I + 1 of 8 columns from `taddr` into their sums.
template <typename T, int I>
__device__ __forceinline__ void drain_pair(Sum<T>* sum, uint32_t taddr, int pw) {
  uint32_t a[8], b[8];
  tmem_ld8(taddr + 2 * I * pw, a);
  tmem_ld8(taddr + (2 * I + 1) * pw, b);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  float most = 0.0f;
#pragma unroll
  for (int c = 0; c < 8; ++c)
    most = fmaxf(most, fmaxf(fabsf(__uint_as_float(a[c])), fabsf(__uint_as_float(b[c]))));
  if (__all_sync(0xffffffffu, most < 4194304.0f)) {
#pragma unroll
    for (int c = 0; c < 8; ++c) sum[c].template add<I>(level_pair_small(a[c], b[c]));
  } else {
#pragma unroll
    for (int c = 0; c < 8; ++c) sum[c].template add<I>(level_pair(a[c], b[c]));
  }
}

// Every level of 8 columns.
__device__ __forceinline__ void drain(Sum<double>* sum, uint32_t taddr, int pw) {
  drain_pair<double, 0>(sum, taddr, pw);
  drain_pair<double, 1>(sum, taddr, pw);
  drain_pair<double, 2>(sum, taddr, pw);
  drain_pair<double, 3>(sum, taddr, pw);
}
__device__ __forceinline__ void drain(Sum<float>* sum, uint32_t taddr, int pw) {
  drain_pair<float, 0>(sum, taddr, pw);
  drain_pair<float, 1>(sum, taddr, pw);
  uint32_t a[8];
  tmem_ld8(taddr + 4 * pw, a);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  float most = 0.0f;
#pragma unroll
  for (int c = 0; c < 8; ++c) most = fmaxf(most, fabsf(__uint_as_float(a[c])));
  if (__all_sync(0xffffffffu, most < 4194304.0f)) {
#pragma unroll
    for (int c = 0; c < 8; ++c) sum[c].add_last_small(a[c]);
  } else {
#pragma unroll
    for (int c = 0; c < 8; ++c) sum[c].add_last(a[c]);
  }
}

// Elements k[0 .. 7] of row `row` of A and column col of B in tile mt: zeros for
// k < 0, past the end and in dead blocks.  All loads of a step are independent,
// so that a batch waits for memory once (kAoW: twice).
template <typename T, int WHAT>
__device__ __forceinline__ void operand_pairs(const ExactArgs<T>& x, uint32_t mt, int row, int col,
                                              const int (&k)[8], T (&a)[8], T (&b)[8]) {
  static_assert(WHAT == kWCt || WHAT == kAoW, "listed outputs");
#pragma unroll
  for (int j = 0; j < 8; ++j) a[j] = b[j] = T(0);
  if constexpr (WHAT == kWCt) {
    const T* w = x.av + ((x.tile0 + mt) * kTileRows + row) * x.ldw;
    const T* c = x.cv + col * x.ldc;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (k[j] >= 0 && k[j] < x.kvalid) {
        a[j] = w[k[j]];
        b[j] = c[k[j]];
      }
  } else {
    const uint32_t set = mt / (uint32_t)x.n_mt;
    const int c = (int)(set % 5u), q = 2 * (int)(mt % (uint32_t)x.n_mt) + (row >> 6), loc = row & 63;
    const int64_t p0 = (x.slab0 + set / 5u) * x.slab_points;
    const int64_t left = x.kvalid - p0;
    unsigned live[8];
    int64_t pt[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      live[j] = 0u;
      pt[j] = p0 + k[j];
      if (k[j] >= 0 && k[j] < x.slab_points && k[j] < left && q < x.nchunk) {
        live[j] = x.mask[pt[j] / kTilePoints * mask_ld(x.nchunk) + q] >> (loc >> 4) & 1u;
        if (x.slot) pt[j] = x.slot[pt[j]];
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (live[j]) {
        const int64_t p = p0 + k[j], tile = p / kTilePoints;
        a[j] = x.av[tile * x.nchunk * kBlockElems +
                    blocked_offset(0, q, x.nchunk, 1, 0, 5 * (int)(p - tile * kTilePoints) + c, loc,
                                   (int)sizeof(T))];
        b[j] = x.cv[(pt[j] * 5 + c) * x.N + col];
      }
  }
}

// Whether a small output may have lost its terms' digits: none of the 8 terms
// a b at the row's largest element is large.  ec: the column's exponent.
template <typename T>
__device__ __forceinline__ bool lost_terms(const T (&a)[8], const T (&b)[8], uint32_t key, int ec) {
  const unsigned ba = key >> kPieceBits, bb = (unsigned)(ec - row_exponent<T>(0u) + 1);
  if (ba == kExpMax<T> || ec == kNonFinite) return true;
  if (ba == 0u || bb <= 1u) return false;  // zeros and subnormal numbers, which keep every bit
  unsigned best = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const unsigned ea = biased_exp(a[j]), eb = biased_exp(b[j]);
    if (ea > 0u && eb > 0u) best = max(best, ea + eb);
  }
  return best + kGraded < ba + bb;
}
template <typename T, int WHAT>
__device__ __forceinline__ bool lost_digits(const ExactArgs<T>& x, uint32_t mt, int row, int col,
                                            uint32_t key) {
  const int k0 = (int)(key & kPieceMask) * 8;
  int k[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) k[j] = k0 + j;
  T a[8], b[8];
  operand_pairs<T, WHAT>(x, mt, row, col, k, a, b);
  return lost_terms(a, b, key, x.ec[mt / (uint32_t)x.b_div * x.N + col]);
}
// An output with multiply-adds in FP64, by a warp, every 32nd element a lane.
template <typename T, int WHAT>
__device__ __forceinline__ T warp_dot(const ExactArgs<T>& x, uint32_t mt, int row, int col) {
  const int lane = threadIdx.x & 31;
  double sum = 0.0;
  const int n = WHAT == kWCt ? (int)(x.kvalid + 31) / 32 : (x.slab_points + 31) / 32;
#pragma unroll 1
  for (int i = 0; i < n; i += 8) {
    int k[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) k[j] = 32 * (i + j) + lane;
    T a[8], b[8];
    operand_pairs<T, WHAT>(x, mt, row, col, k, a, b);
#pragma unroll
    for (int j = 0; j < 8; ++j) sum = fma((double)a[j], (double)b[j], sum);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  return (T)sum;
}
// The read-out of an item walks its columns OUT at a time, rows r and r + 16 of
// them by lanes 2 r and 2 r + 1, kPer columns a lane: value `pos` of lane l.
template <typename T>
struct OutPos {
  static constexpr int OUT = Shape<T>::OUT, kPer = 16 / (int)sizeof(T);
  __device__ static int row(int pos, int lane) { return (lane >> 1) + 16 * (pos / kPer & 1); }
  __device__ static int col(int pos, int lane) {
    return pos / (2 * kPer) * OUT + (lane & 1) * kPer + pos % kPer;
  }
  // the bits of row r (the others are row r + 16's)
  static constexpr unsigned kFirst = kPer == 2 ? 0x33333333u : 0x0F0F0F0Fu;
  static_assert(Split<T>::kPart / 2 / OUT * 2 * kPer <= 32, "a bit each");
};
__device__ __forceinline__ void load4(const double* p, double (&x)[4]) {
  const double2 u = reinterpret_cast<const double2*>(p)[0], v = reinterpret_cast<const double2*>(p)[1];
  x[0] = u.x;
  x[1] = u.y;
  x[2] = v.x;
  x[3] = v.y;
}
__device__ __forceinline__ void load4(const float* p, float (&x)[4]) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  x[0] = v.x;
  x[1] = v.y;
  x[2] = v.z;
  x[3] = v.w;
}
// Rows with many lost outputs (kManyLost or more of the warp's columns), by the whole
// warp: lane 16 h + c takes column c (then 16 + c) and half h of each group's AOs, so
// that four rows (FP64: two) share the loads of C.  lost: the columns of row row0 +
// lane (bits).  Bound: the latency of its loads in FP32, the FP64 pipe in FP64.
// (Inlined, like mend_outputs: a call reads the arguments through generic addresses
// and costs the read-out registers.)
constexpr int kManyLost = 4;
template <typename T>
__device__ __forceinline__ void mend_rows(const ExactArgs<T>& x, uint32_t mt, int row0, int n0,
                                       int32_t out_row, unsigned lost) {
  constexpr int HC = Split<T>::kPart / 2, R = sizeof(T) == 8 ? 2 : 4;
  constexpr int kUnroll = sizeof(T) == 8 ? 1 : 2, kPitch = 128 / (int)sizeof(T);
  const int lane = threadIdx.x & 31, h = lane >> 4;
  const T* tile = x.av + (x.tile0 + mt) * x.nchunk * kBlockElems;
  const T* cv = x.cv;
  const int64_t ldc = x.ldc;
  const uint32_t* list = x.glist + mt * (int64_t)x.cap;
  const int n = x.ngroups[mt], N = (int)x.N;
  unsigned rows = __ballot_sync(0xffffffffu, lost != 0u);
  while (rows) {
    int r[R];
    unsigned cols[R];
    int count = 0;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      r[j] = rows ? __ffs(rows) - 1 : r[j > 0 ? j - 1 : 0];
      count += rows ? 1 : 0;
      rows &= rows - 1u;
      cols[j] = __shfl_sync(0xffffffffu, lost, r[j]);
    }
    for (int cb = 0; cb < HC; cb += 16) {
      unsigned any = 0;
#pragma unroll
      for (int j = 0; j < R; ++j) any |= cols[j];
      if ((any >> cb & 0xffffu) == 0u) continue;
      const int c = cb + (lane & 15), col = n0 + c < N ? n0 + c : N - 1;
      const T* cp = cv + col * ldc + 8 * h;
      T sum[R] = {};
#pragma unroll kUnroll
      for (int i = 0; i < n; ++i) {
        const uint32_t id = list[i];
        const T* ap = tile + blocked_offset(0, (int)(id >> 2), 1, 1, 0, row0,
                                            16 * (int)(id & 3u) + 8 * h, (int)sizeof(T));
#pragma unroll
        for (int k0 = 0; k0 < 8; k0 += 4) {
          T b[4];
          load4(cp + kGroup * (int64_t)id + k0, b);
#pragma unroll
          for (int j = 0; j < R; ++j) {
            T a[4];
            load4(ap + r[j] * kPitch + k0, a);
#pragma unroll
            for (int k = 0; k < 4; ++k) sum[j] = fma(a[k], b[k], sum[j]);
          }
        }
      }
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const T v = sum[j] + __shfl_xor_sync(0xffffffffu, sum[j], 16);
        const int32_t orow = __shfl_sync(0xffffffffu, out_row, r[j]);
        if (j < count && h == 0 && c < HC && (cols[j] >> c & 1u)) x.D[orow * x.ldd + n0 + c] = v;
      }
    }
  }
}
// The whole warp, after its columns n0 .. of rows row0 .. + 31 are stored: bit pos
// of `small` marks a small output of this lane; those that may have lost their
// digits are formed again with multiply-adds over the live groups.  key, out_row:
// those of row row0 + lane.  Lost outputs mostly share rows (a nucleus's points):
// many of a row go to mend_rows, few take a pass over its AOs together, lane 16 h +
// c AO c of the groups of parity h.  Which way a row goes and the order of its sums do
// not depend on its tile.  19 200 points within 0.1 bohr of nuclei x 300 MOs without s
// functions, FP32: 51 ms one output at a time, 7.8 with four of a row together, 3.7 with
// mend_rows.
template <typename T>
__device__ __forceinline__ void mend_outputs(const ExactArgs<T>& x, uint32_t mt, int row0, int n0,
                                             uint32_t key, int32_t out_row, unsigned small) {
  constexpr int kCols = kManyLost - 1, kStep = 4;
  const int lane = threadIdx.x & 31;
  const T* tile = x.av + (x.tile0 + mt) * x.nchunk * kBlockElems;
  const T* cv = x.cv + n0 * x.ldc;
  unsigned many = 0, few = 0;  // of row `lane`: lost columns
  while (__any_sync(0xffffffffu, small != 0u)) {
    // a bit of each lane: a lane looks at the output, the row's lane collects it
    const int pos = small ? __ffs(small) - 1 : 0;
    const int r = OutPos<T>::row(pos, lane), c = OutPos<T>::col(pos, lane);
    const uint32_t rkey = __shfl_sync(0xffffffffu, key, r);
    bool l = small != 0u;
    if (l) {
      const int k0 = (int)(rkey & kPieceMask) * 8;
      T a[8], b[8];
      load8(tile + blocked_offset(0, k0 / kChunkAO, 1, 1, 0, row0 + r, k0 % kChunkAO,
                                  (int)sizeof(T)),
            a);
      load8(cv + c * x.ldc + k0, b);
      l = lost_terms(a, b, rkey, x.ec[mt / (uint32_t)x.b_div * x.N + n0 + c]);
    }
    unsigned todo = __ballot_sync(0xffffffffu, l);
    while (todo) {
      const int s = __ffs(todo) - 1;
      todo &= todo - 1u;
      const int sr = __shfl_sync(0xffffffffu, r, s), sc = __shfl_sync(0xffffffffu, c, s);
      if (lane == sr) few |= 1u << sc;
    }
    small &= small - 1u;
  }
  if (__popc(few) >= kManyLost) {
    many = few;
    few = 0u;
  }
  unsigned todo = __ballot_sync(0xffffffffu, few != 0u);
  while (todo) {
    const int r = __ffs(todo) - 1;
    todo &= todo - 1u;
    unsigned cols = __shfl_sync(0xffffffffu, few, r);
    const int32_t orow = __shfl_sync(0xffffffffu, out_row, r);
    const int count = __popc(cols);
    int c[kCols];
#pragma unroll
    for (int j = 0; j < kCols; ++j) {
      c[j] = cols ? __ffs(cols) - 1 : c[j > 0 ? j - 1 : 0];
      cols &= cols - 1u;
    }
    const uint32_t* list = x.glist + mt * (int64_t)x.cap;
    const int n = x.ngroups[mt];
    T sum[kCols] = {};
#pragma unroll 1
    for (int i = 0; i < n; i += kStep) {
      T a[kStep], b[kStep][kCols];
#pragma unroll
      for (int s = 0; s < kStep; ++s) {
        const uint32_t id = i + s < n ? list[i + s] : ~(uint32_t)(lane >> 4);
        const int k = 16 * (int)(id & 3u) + (lane & 15), q = (int)(id >> 2);
        a[s] = T(0);
#pragma unroll
        for (int j = 0; j < kCols; ++j) b[s][j] = T(0);
        if ((id & 1u) == (uint32_t)lane >> 4) {
          a[s] = tile[blocked_offset(0, q, 1, 1, 0, row0 + r, k, (int)sizeof(T))];
#pragma unroll
          for (int j = 0; j < kCols; ++j) b[s][j] = cv[c[j] * x.ldc + (int64_t)q * kChunkAO + k];
        }
      }
#pragma unroll
      for (int s = 0; s < kStep; ++s)
#pragma unroll
        for (int j = 0; j < kCols; ++j) sum[j] = fma(a[s], b[s][j], sum[j]);
    }
#pragma unroll
    for (int j = 0; j < kCols; ++j) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], o);
      if (lane == j && j < count) x.D[orow * x.ldd + n0 + c[j]] = sum[j];
    }
  }
  if (__any_sync(0xffffffffu, many != 0u)) mend_rows(x, mt, row0, n0, out_row, many);
}
// The same outputs into the list instead.
template <typename T>
__device__ __forceinline__ void list_outputs(const ExactArgs<T>& x, uint32_t mt, int row0, int n0,
                                             unsigned small) {
  const int lane = threadIdx.x & 31;
  uint32_t at = (uint32_t)__popc(small);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, at, o);
    if (lane >= o) at += v;
  }
  const uint32_t total = __shfl_sync(0xffffffffu, at, 31);
  uint32_t base = 0;
  if (lane == 31) base = atomicAdd(x.small_num, total);
  base = __shfl_sync(0xffffffffu, base, 31);
  if (base + total > x.small_cap) {
    if (lane == 0) atomicOr(x.unfit, 1);
    return;
  }
  at += base - (uint32_t)__popc(small);
  for (; small; small &= small - 1u, ++at) {
    const int pos = __ffs(small) - 1;
    x.small_list[at] = make_uint2(mt * kTileRows + (uint32_t)(row0 + OutPos<T>::row(pos, lane)),
                                  (uint32_t)(n0 + OutPos<T>::col(pos, lane)));
  }
}
// The listed outputs, over all warps of the grid: a lane looks at each, the warp
// forms those again that may have lost their digits.  For products whose lost
// outputs may sit together (the weight of one MO tiny at the one point that
// dominates a slab: 77 columns of dL/dC in one block of the product kernel, which
// took it from 0.35 to 0.55 ms).
constexpr int kMendThreads = 256;
template <typename T, int WHAT>
__global__ void __launch_bounds__(kMendThreads)
    mend_kernel(const __grid_constant__ ExactArgs<T> x) {
  griddep_wait();
  const uint32_t num = *x.small_num;
  // (an overflowed list has gaps)
  if (num > x.small_cap || *x.unfit != 0) return;  // every result will be replaced
  const uint32_t warps = gridDim.x * (kMendThreads / 32);
  const uint32_t warp = blockIdx.x * (kMendThreads / 32) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  uint32_t per = (num + warps - 1) / warps;  // entries a warp looks at together
  if (per > 32) per = 32;
  for (uint32_t i0 = warp * per; i0 < num; i0 += warps * per) {
    const uint32_t i = i0 + (uint32_t)lane;
    const bool mine = (uint32_t)lane < per && i < num;
    const uint2 e = mine ? x.small_list[i] : make_uint2(0u, 0u);
    const uint32_t mt = e.x / kTileRows;
    const int row = (int)(e.x % kTileRows), col = (int)e.y;
    unsigned todo = __ballot_sync(
        0xffffffffu, mine && lost_digits<T, WHAT>(x, mt, row, col, x.key[e.x]));
    while (todo) {
      const int l = __ffs(todo) - 1;
      todo &= todo - 1u;
      const T v = warp_dot<T, WHAT>(x, __shfl_sync(0xffffffffu, mt, l),
                                    __shfl_sync(0xffffffffu, row, l),
                                    __shfl_sync(0xffffffffu, col, l));
      if (lane == l) x.D[((x.tile0 + mt) * kTileRows + row) * x.ldd + col] = v;
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 1)
    mo_exact_kernel(const __grid_constant__ ExactArgs<T> x, int* err_flag) {
  using P = Split<T>;
  using H = Shape<T>;
  constexpr int S = P::S, ST = P::kStages;
  extern __shared__ unsigned char smem_raw[];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag, skip_slot;
  __shared__ __align__(8) uint64_t bars[2 * ST + 4 + 2 * kItems];
  __shared__ uint32_t item_slot[kItems];
  __shared__ int ec_smem[kEpiWarps][P::kPart / 2];
  const uint32_t base = (smem_u32(smem_raw) + 127u) & ~127u;
  auto full_bar = [&](int s) { return smem_u32(&bars[s]); };
  auto empty_bar = [&](int s) { return smem_u32(&bars[ST + s]); };
  auto tfull_bar = [&](int part) { return smem_u32(&bars[2 * ST + part]); };
  auto tempty_bar = [&](int part) { return smem_u32(&bars[2 * ST + 2 + part]); };
  auto item_full = [&](int s) { return smem_u32(&bars[2 * ST + 4 + s]); };
  auto item_empty = [&](int s) { return smem_u32(&bars[2 * ST + 4 + kItems + s]); };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_v = &abort_flag;
  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; ++s) {
      mbar_init(full_bar(s), 2);  // the producers
      mbar_init(empty_bar(s), 2);  // the two issuers
    }
    for (int part = 0; part < 2; ++part) {
      mbar_init(tfull_bar(part), 1);
      mbar_init(tempty_bar(part), kEpiWarps / 2);
    }
    for (int s = 0; s < kItems; ++s) {
      mbar_init(item_full(s), 1);
      mbar_init(item_empty(s), kEpiWarps + 3);  // all roles but the AO producer
    }
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kIssuer) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                     smem_u32(&tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  griddep_wait();
  bool skip = false;
  if constexpr (sizeof(T) == 8)  // (the backward's products: FP32 has none)
    if (x.unfit) {  // (one thread reads it: a full list may set it meanwhile)
      if (threadIdx.x == 0) skip_slot = *x.unfit;
      __syncthreads();
      skip = skip_slot != 0;
    }
  const uint32_t total = skip ? 0u : (uint32_t)(x.tiles * x.n_tiles);
  const int pw = x.pw;
  const uint32_t b_bytes = (uint32_t)(S * pw * 32);
  // The k-th item of this CTA (total or more: none).  The first is the CTA's
  // own; with a counter the AO producer hands out the next ones, through a ring
  // of slots, else they lie gridDim.x apart.
  auto item_at = [&](uint32_t k, bool& ok) -> uint32_t {
    if (k == 0 || !x.counter) return blockIdx.x + k * gridDim.x;
    const int s = (int)((k - 1) % kItems);
    ok = mbar_wait(item_full(s), ((k - 1) / kItems) & 1u, abort_v);
    if (!ok) {
      flag_error(err_flag, abort_v, 4);
      return total;
    }
    return *(volatile uint32_t*)&item_slot[s];
  };
  // ... read by this role (one arrival per role's warp)
  auto item_read = [&](uint32_t k) {
    if (k && x.counter) mbar_arrive(item_empty((int)((k - 1) % kItems)));
  };

  if (warp >= kEpiWarps && warp < kIssuer) {
    // -------------------------------------------------- producers
    const bool a_side = warp == kEpiWarps;
    uint32_t it = 0, p = blockIdx.x;
    bool ok = true;
    for (uint32_t k = 0; ok; ++k) {
      if (!a_side) {
        p = item_at(k, ok);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        __syncwarp();
        if (lane == 0) item_read(k);
      }
      if (p >= total) break;
      // the item after this one, handed out when this one's copies are issued
      uint32_t next = p + gridDim.x;
      if (a_side && x.counter && lane == 0) next = gridDim.x + atomicAdd(x.counter, 1u);
      uint32_t mt;
      int nt;
      item_of(x, p, mt, nt);
      const int n = x.ngroups[mt];
      // the parts' digits of a group are neighbours (a CTA of one part takes its own)
      const int part = nt * x.ppt;
      const uint32_t bytes =
          a_side ? H::A_BYTES : (part_of(x, nt, 1) >= 0 ? 2u * b_bytes : b_bytes);
      const unsigned char* src =
          a_side ? x.a + (int64_t)mt * x.cap * H::A_BYTES
                 : x.b + mt / (uint32_t)x.b_div * x.b_stride +
                       ((int64_t)(part >> 1) * 2 * x.cap + (part & 1)) * b_bytes;
      const uint32_t* list = x.glist + mt * (int64_t)x.cap;
      for (int i0 = 0; i0 < n && ok; i0 += 32) {
        const uint32_t mine = !a_side && i0 + lane < n ? list[i0 + lane] : 0u;
        const int m = n - i0 < 32 ? n - i0 : 32;
        for (int j = 0; j < m && ok; ++j, ++it) {
          const uint32_t id = __shfl_sync(0xffffffffu, mine, j);
          if (lane == 0) {
            const int s = it % ST;
            ok = mbar_wait(empty_bar(s), ((it / ST) & 1u) ^ 1u, abort_v);
            if (!ok) {
              flag_error(err_flag, abort_v, 1);
            } else {
              mbar_expect_tx(full_bar(s), bytes);
              bulk_load(base + s * H::STAGE + (a_side ? 0u : H::A_BYTES),
                        src + (a_side ? (int64_t)(i0 + j) * H::A_BYTES : (int64_t)id * 2 * b_bytes),
                        bytes, full_bar(s));
            }
          }
          ok = __shfl_sync(0xffffffffu, ok, 0);
        }
      }
      if (a_side && x.counter && ok) {
        const int s = (int)(k % kItems);
        if (lane == 0) {
          ok = mbar_wait(item_empty(s), ((k / kItems) & 1u) ^ 1u, abort_v);
          if (!ok) {
            flag_error(err_flag, abort_v, 4);
          } else {
            *(volatile uint32_t*)&item_slot[s] = next;
            mbar_arrive(item_full(s));
          }
        }
        next = __shfl_sync(0xffffffffu, next, 0);
        ok = __shfl_sync(0xffffffffu, ok, 0);
      }
      p = next;
    }
    if (lane == 0 && *abort_v) {
      // wait (bounded) for the copies in flight: each stage this warp filled
      // last completes once every producer's bytes are in, or times out
      const uint32_t first = it > (uint32_t)ST ? it - ST : 0u;
      for (uint32_t k = first; k < it; ++k) {
        const long long t0 = clock64();
        while (!mbar_try_wait(full_bar(k % ST), (k / ST) & 1u) && clock64() - t0 < kWaitCycles) {
        }
      }
    }
  } else if (warp >= kIssuer) {
    // -------------------------------------------------- MMA issuers
    // The whole warp walks the stages and one elected lane issues: a single diverged
    // lane moved the descriptors into uniform registers for each MMA.  38 400 points
    // x 300 MOs with slicing FP64 1644 -> 1551 us, FP32 856 -> 791; 8000 points x 2000
    // MOs FP32 2958 -> 2602.
    const int q = warp - kIssuer;
    const uint32_t el = elect_one();
    {
      const uint32_t tfull = tfull_bar(q), tempty = tempty_bar(q);
      const int off = q ? P::kSeg / 2 : 0;  // segments end where (i + 1 + off) % kSeg == 0
      uint32_t it = 0, seg = 0;
      bool ok = true, open = false;
      const uint64_t da0 = core_desc(base, 2048);
      const uint64_t db0 = core_desc(base + H::A_BYTES + q * b_bytes, (uint32_t)(S * pw * 16));
      const uint32_t idesc0 = make_idesc(1, kBM, S * pw);
      const uint32_t istep = (uint32_t)(pw >> 3) << 17;
      const uint32_t d0 = tmem + (uint32_t)(q * kPartCols);
      for (uint32_t k = 0; ok; ++k) {
        const uint32_t p = __shfl_sync(0xffffffffu, item_at(k, ok), 0);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        if (el) item_read(k);
        if (p >= total) break;
        uint32_t mt;
        int nt;
        item_of(x, p, mt, nt);
        const int n = x.ngroups[mt];
        const bool idle = part_of(x, nt, q) < 0;
        for (int i = 0; i < n; ++i, ++it) {
          const int s = it % ST;
          const bool first = i == 0 || (i + off) % P::kSeg == 0;
          if (first && !idle) {
            ok = __all_sync(0xffffffffu, mbar_wait(tempty, (seg & 1u) ^ 1u, abort_v));
            if (!ok) break;
            open = true;
          }
          ok = __all_sync(0xffffffffu, mbar_wait(full_bar(s), (it / ST) & 1u, abort_v));
          if (!ok) break;
          if (idle) {
            if (el) mbar_arrive(empty_bar(s));
            continue;
          }
          tc_fence_after();
          const uint64_t so = (uint64_t)(s * H::STAGE) >> 4;
          const uint64_t da = da0 + so, db = db0 + so;
#pragma unroll
          for (int k = 0; k < S; ++k)  // AO slice k x C slices 0 .. S-1-k -> levels k .. S-1
            umma_el<QK_BF16X3>(d0 + (uint32_t)(k * pw), da + (uint64_t)(k * H::A_SLICE >> 4), db,
                               idesc0 - (uint32_t)k * istep, first && k == 0 ? 0u : 1u, el);
          umma_commit_el(empty_bar(s), el);
          if (i == n - 1 || (i + 1 + off) % P::kSeg == 0) {
            umma_commit_el(tfull, el);
            open = false;
            ++seg;
          }
        }
      }
      if (!ok) {
        flag_error(err_flag, abort_v, 2);
        // the MMAs issued so far must have finished before TMEM is given back
        if (open) {
          umma_commit_el(tfull, el);
          ++seg;
        }
        const long long t0 = clock64();
        while (seg > 0 && !mbar_try_wait(tfull, (seg - 1) & 1u) && clock64() - t0 < kWaitCycles) {
        }
      }
    }
  } else {
    // -------------------------------------------------- epilogue
    constexpr int HC = P::kPart / 2;  // most columns of a warp
    const int quarter = warp & 3, sub = (warp >> 2) & 1, q = warp >> 3;
    const int cols = pw / 2;          // columns of this warp (a multiple of 8)
    const uint32_t tfull = tfull_bar(q), tempty = tempty_bar(q);
    const int off = q ? P::kSeg / 2 : 0;
    const int row = quarter * 32 + lane;
    const uint32_t tbase =
        tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(q * kPartCols + sub * cols);
    unsigned char* stg = smem_raw + (base - smem_u32(smem_raw)) + (size_t)ST * H::STAGE +
                         (size_t)warp * H::EPI_WARP;
    constexpr int kPer = 16 / (int)sizeof(T);  // values of a 16-byte piece
    const bool vec = (x.ldd * (int64_t)sizeof(T)) % 16 == 0 &&
                     (reinterpret_cast<uintptr_t>(x.D) & 15) == 0;
    // An item's scalars, read one item ahead of its read-out.
    struct Item {
      uint32_t mt;
      int part, n, E;
      uint32_t key;
      int32_t out_row;  // the row of D that this lane's row goes to (-1: padding)
    };
    auto load_item = [&](uint32_t p) {
      Item y;
      int nt;
      item_of(x, p, y.mt, nt);
      y.part = part_of(x, nt, q);
      y.n = x.ngroups[y.mt];
      y.key = x.key[(int64_t)y.mt * kTileRows + row];
      y.E = key_exponent<T>(y.key);
      const int64_t lin = (x.tile0 + y.mt) * x.tile_rows + row;
      y.out_row = -1;
      if (row < x.tile_rows && lin < x.M) {
        const uint32_t l = (uint32_t)lin, pt = l / 5u;
        y.out_row = x.perm ? 5 * x.perm[pt] + (int32_t)(l - 5u * pt) : (int32_t)l;
      }
      return y;
    };
    // column exponents of this warp's part and B set
    int* ecs = ec_smem[warp];
    int ec_of = -1;
    uint32_t seg = 0;
    bool ok = true;
    for (uint32_t k = 0; ok; ++k) {
      const uint32_t p = item_at(k, ok);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      __syncwarp();
      if (lane == 0) item_read(k);
      if (p >= total) break;
      const Item y = load_item(p);
      if (y.part < 0) continue;
      const int nseg = y.n ? (y.n + off + P::kSeg - 1) / P::kSeg : 0;
      const int set = (int)(y.mt / (uint32_t)x.b_div);
      const int n0 = y.part * pw + sub * cols;
      if (set * x.n_parts + y.part != ec_of) {
        ec_of = set * x.n_parts + y.part;
        __syncwarp();
        if (lane < cols) ecs[lane] = n0 + lane < x.N ? x.ec[set * x.N + n0 + lane] - P::kExp : 0;
        __syncwarp();
      }
      Sum<T> sum[HC];
#pragma unroll
      for (int c = 0; c < HC; ++c) sum[c].clear();
      for (int sg = 0; sg < nseg && ok; ++sg, ++seg) {
        ok = mbar_wait(tfull, seg & 1u, abort_v);
        if (!ok) flag_error(err_flag, abort_v, 3);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < HC; c += 8)
          if (c < cols) drain(sum + c, tbase + c, pw);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty);
      }
      if (!ok) break;
      // OUT columns at a time through the staging area, then lanes over
      // (row, 16 bytes of columns): stores of 32 contiguous bytes per row
      unsigned small = 0;  // outputs to look at again (OutPos)
#pragma unroll
      for (int c0 = 0; c0 < HC; c0 += H::OUT) {
        if (c0 < cols) {
#pragma unroll
          for (int c = 0; c < H::OUT; ++c) sum[c0 + c].put(stg, c, lane);
          __syncwarp();
          const int c = (lane & 1) * kPer;
          const int col = n0 + c0 + c;
          int ec[kPer];
#pragma unroll
          for (int j = 0; j < kPer; ++j) ec[j] = ecs[c0 + c + j];
#pragma unroll 1
          for (int r = lane >> 1; r < 32; r += 16) {
            const int er = __shfl_sync(0xffffffffu, y.E, r);
            const int32_t orow = __shfl_sync(0xffffffffu, y.out_row, r);
            if (orow < 0 || col >= x.N) continue;
            T v[kPer];
            unsigned sm = 0;
#pragma unroll
            for (int j = 0; j < kPer; ++j) {
              Sum<T> t;
              t.get(stg, c + j, r);
              t.settle(nseg);
              bool one;
              v[j] = t.value(er + ec[j], x.small, &one);
              if (one) sm |= 1u << j;
            }
            T* dst = x.D + (int64_t)orow * x.ldd + col;
            if (vec && col + kPer <= x.N) {
              *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(v);
            } else {
#pragma unroll
              for (int j = 0; j < kPer; ++j) {
                if (col + j < x.N)
                  dst[j] = v[j];
                else
                  sm &= ~(1u << j);
              }
            }
            small |= sm << (c0 / H::OUT * 2 * kPer + (r >> 4) * kPer);
          }
          __syncwarp();
        }
      }
      // rows of zeros (dead columns of the AO tensor, screened points) lost nothing
      const unsigned zero = __ballot_sync(0xffffffffu, y.key >> kPieceBits == 0u) >> (lane >> 1);
      if (zero & 1u) small &= ~OutPos<T>::kFirst;
      if (zero & 0x10000u) small &= OutPos<T>::kFirst;
      if (__any_sync(0xffffffffu, small != 0u)) {
        bool listed = false;
        if constexpr (sizeof(T) == 8) listed = x.small_list != nullptr;
        if (listed)
          list_outputs(x, y.mt, quarter * 32, n0, small);
        else
          mend_outputs(x, y.mt, quarter * 32, n0, y.key, y.out_row, small);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kIssuer) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
}

// The product of prepared operands: one persistent launch.  counter: a word of the
// operands' own scratch (products on different streams may run at once).
template <typename T>
cudaError_t launch_product(ExactArgs<T>& x, uint32_t* counter, int* err_flag, cudaStream_t s) {
  if (x.tiles == 0 || x.N == 0) return cudaSuccess;
  if (x.M > INT32_MAX) return cudaErrorInvalidValue;
  KernelFacts f;
  cudaError_t e = kernel_facts<mo_exact_kernel<T>>(Shape<T>::SMEM, kThreads, &f);
  if (e != cudaSuccess) return e;
  if (f.occ < 1) return cudaErrorInvalidConfiguration;
  // two parts per CTA share its A digits; one where two would leave SMs idle
  x.ppt = x.tiles * ((x.n_parts + 1) / 2) < f.sms ? 1 : 2;
  x.n_tiles = (x.n_parts + x.ppt - 1) / x.ppt;
  // about one wave of CTAs per scheduling block, at most 12 N tiles wide
  const int wide = x.n_tiles < 12 ? x.n_tiles : 12;
  x.block_m = (f.sms + wide - 1) / wide;
  // Tiles differ in their live groups: from four items a CTA on, the next one goes
  // to the CTA that is free:
  // 38 400 points x 300 MOs FP64 1780 -> 1734 us, FP32 925 -> 910, 1600 points x
  // 2000 MOs FP32 3255 -> 3098 (AO slicing included).  Small calls keep fixed
  // strides: the memset would cost them 2 us.
  x.counter = nullptr;
  if (x.tiles * x.n_tiles >= 4 * (int64_t)f.sms) {
    x.counter = counter;
    e = cudaMemsetAsync(x.counter, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(mo_exact_kernel<T>,
                    (unsigned)std::min<int64_t>(x.tiles * x.n_tiles, f.sms), kThreads,
                    Shape<T>::SMEM, s, x, err_flag);
}

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

// Columns of a part: the fewest parts of at most kPart, then the narrowest
// multiple of 16 that covers N with them.
template <typename T>
int part_cols(int64_t N, int* n_parts) {
  const int64_t np = (N + Split<T>::kPart - 1) / Split<T>::kPart;
  *n_parts = (int)np;
  return (int)(((N + np - 1) / np + 15) / 16 * 16);
}

// The digits of C, by pairs of parts.
template <typename T>
size_t digit_bytes(int n_parts, int pw, int64_t kpad) {
  return align256((size_t)((n_parts + 1) / 2) * 2 * pw * kpad * 2 * Split<T>::S);
}

template <typename T>
size_t c_bytes(int64_t N, int64_t kpad) {
  int np;
  const int pw = part_cols<T>(N, &np);
  return digit_bytes<T>(np, pw, kpad) + align256(sizeof(int32_t) * N);
}

// Exponents and digits of C [N][kpad] into dst, and its verdict into *bad_host
// through the device word *bad (zero before and after).  c64: the same C in FP64
// [N][ld], cols valid.
template <typename T>
cudaError_t prepare_c(const T* C, const double* c64, int64_t cols, int64_t ld, int64_t N,
                      int64_t kpad, void* dst, int* bad, int* bad_host, cudaStream_t s) {
  *bad_host = 0;
  if (N == 0 || kpad == 0) return cudaSuccess;
  int np;
  const int pw = part_cols<T>(N, &np);
  const int64_t pieces = (int64_t)np * pw * (kpad / kGroup) * 2;
  unsigned char* dig = (unsigned char*)dst;
  int32_t* ec = (int32_t*)(dig + digit_bytes<T>(np, pw, kpad));
  c_rows_kernel<T><<<(unsigned)((N + 7) / 8), 256, 0, s>>>(c64, N, cols, ld, ec, bad);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(bad_host, bad, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return e;
  slice_c_kernel<T><<<(unsigned)std::min<int64_t>((pieces + 255) / 256, 16384), 256, 0, s>>>(
      C, N, kpad, pw, np, ec, dig, bad);
  return cudaGetLastError();
}

}  // namespace
}  // namespace qk
