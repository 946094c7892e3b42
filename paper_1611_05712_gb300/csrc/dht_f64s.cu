// DHT of the FP64 form on the 5th-generation tensor cores, with FP64 results.
//
// The discrete Hankel transform along r (section "Finite order pseudo-spectral solvers":
// Hankel transform along r) is, per (component, mode) pair, Y = A X with A the Nr x Nr
// FP64 matrix and X the Nr x 2Nz FP64 panel.  GB300 runs FP64 arithmetic at 1/64 of its
// FP32 rate and far below its tensor rate, so this path computes the product exactly in
// pieces on the BF16 tensor cores and combines them in integers (the splitting idea of Ozaki
// et al., "Error-free transformations of matrix multiplication by using fast routines of
// matrix multiplication and its applications", Numer. Algorithms 59, 2012, here with
// fixed-width integer digits):
//   * every row n of A and every column c of X is scaled by a power of two, 2^E_n and
//     2^E_c, so that its entries lie in (-1, 1); the scaled value v is rounded to B bits and
//     written in S balanced base-256 digits, v = sum_i d_i 2^(-(T + 8 i)) + r with |d_i| <= 128
//     for i >= 1 and |r| <= 2^-(B+1), B = T + 8 (S - 1): each digit is exactly a BF16 number
//     (8 significant bits hold the integers up to 256).  Digits with signs of their own carry a
//     bit more than a sign and a magnitude would, and what a kept product misses has mean 0;
//   * a digit product summed over K <= 256 terms is an integer of at most 2^22 (2^23, 2^24
//     with one, two first digits of S = 6), and the tensor cores' FP32 accumulators hold
//     sums up to 2^24 exactly.  Group g collects the products d_i d_j with i + j = g (weight
//     2^(-(2T + 8g))); products with i + j >= S are left out;
//   * the epilogue combines the group accumulators in 64-bit integer arithmetic, converts to
//     FP64 with one rounding and scales by 2^(E_c + E_n).
// Two forms (F64sForm below):
//   Nr <= 256: S = 6, T = 8, B = 48, 21 products.  The first digit reaches 256, so groups 2
//     and 3 are split over two accumulators each to stay exact; groups 4 and 5 add at most an
//     FP32 rounding at weight <= 2^-48.  At worst, with every digit left out of one sign, 2^-46 of
//     max|A_n| max|X_c| K is missing (a term's five products of group 6 are up to 5 2^14 2^-64 =
//     2^-47.7, its operands' rounding 2^-48); the signs average, and the error found is about
//     2^-50 of max|A_n| max|X_c| sqrt(K) (on the Hankel matrices with random, beam-like, decaying and
//     smooth panels 2 to 6 times smaller than the seven sign-magnitude 7-bit slices, 28 products,
//     that stood here before);
//   Nr > 256: S = 8, T = 6, B = 62, 36 products, the accumulators drained into integers every
//     256 K: groups 0..3 exact, the rest exact unless sums align adversarially (more than 2^24 units
//     of one sign: then FP32 roundings at weight <= 2^-44).  All 53 bits of entries down to 2^-9 of the
//     largest take part.  At worst 2^-59 of max|A_n| max|X_c| K is missing (a term's seven products of
//     group 8, up to 7 2^14 2^-76 = 2^-59.2, and its operands' rounding, 2^-62), and the rest is
//     rounded once: no further off than the float64 product's own accumulated roundings.
// Measured, one cycle's 20 DHTs with their panels' digits: 2048 x 256 x 2 modes 0.45 -> 0.32 ms
// against the seven-slice form; 1800 x 400 x 2 modes 21.1 ms on the FP64 SIMT GEMM -> 1.04 ms.
//
// Pieces: k_f64s_matrix writes the matrices' digit planes at set-up (S BF16 planes each,
// K-major); per DHT k_f64s_panel finds the column exponents and writes the panels' K-major
// planes; k_dht_f64s is a persistent warp-specialised tcgen05 kernel: one thread issues the
// tensor-memory-access copies of both operands (S planes each, 64-byte swizzle, 32 K elements
// per stage) into a ring of stages, three threads (one per warp, each owning whole
// accumulators) issue the digit products per 16 K elements into 8 TMEM accumulators of a 128 x
// 64 tile (all 512 columns), and 16 epilogue warps combine them and store Y.
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>
#include <cstring>
#include <mutex>

#include "pic_internal.cuh"
#include "tc_common.cuh"

namespace pic {
namespace {

constexpr int kF64sM = 128;         // panel columns c per tile (TMEM lanes)
constexpr int kF64sN = 64;          // matrix rows n per tile, at most (F64sParams::nw)
constexpr int kF64sAcc = 8;         // accumulators in TMEM (kF64sN columns each: all 512)
constexpr int kF64sKC = 32;         // K elements per stage (one 64-byte swizzle row of BF16)
constexpr int kF64sKBlock = 256;    // K elements between drains of the accumulators (exactness)
constexpr int kF64sThreads = 640;   // warp 0: copies, warps 1-3: MMA, warps 4..19: epilogue
constexpr uint32_t kF64sPlaneA = kF64sM * 64;   // bytes of one panel plane per stage
constexpr uint32_t kF64sPlaneB = kF64sN * 64;   // bytes of one matrix plane per stage

// The two forms: S digits, T bits above the point of the first digit, stages of shared
// memory (3 x 72 KB or 2 x 96 KB of the 227 KB).
template <int S> struct F64sForm;
template <> struct F64sForm<kF64sDigits> {
  static constexpr int top = 8, stages = 3;
  // accumulator of the product d_i d_j, g = i + j: 0, 1, 2 (with d_0), 3 (d_1 d_1), 4 (g = 3
  // with d_0), 5 (g = 3 without), 6 (g = 4), 7 (g = 5)
  __host__ __device__ static constexpr int acc(int i, int j) {
    const int g = i + j;
    const bool first = i == 0 || j == 0;
    return g <= 1 ? g : g == 2 ? (first ? 2 : 3) : g == 3 ? (first ? 4 : 5) : g + 2;
  }
  // issuing warp (1..3) of each accumulator: 7 products each (acc 7 has 6, acc 0 has 1)
  __host__ __device__ static constexpr int warp(int a) { return a == 0 || a == 7 ? 1 : a == 6 || a == 2 ? 2 : 3; }
};
template <> struct F64sForm<kF64sDigitsWide> {
  static constexpr int top = 6, stages = 2;
  __host__ __device__ static constexpr int acc(int i, int j) { return i + j; }
  // 12 products each: 7 + 3 (8 + 4), 6 + 4 (7 + 5), 5 + 2 + 1 + 0 (6 + 3 + 2 + 1)
  __host__ __device__ static constexpr int warp(int a) { return a == 7 || a == 3 ? 1 : a == 6 || a == 4 ? 2 : 3; }
};
template <int S> constexpr int f64s_bits() { return F64sForm<S>::top + 8 * (S - 1); }
template <int S> constexpr uint32_t f64s_stage_bytes() { return S * (kF64sPlaneA + kF64sPlaneB); }
template <int S> constexpr size_t f64s_smem() { return 1024 + (size_t)F64sForm<S>::stages * f64s_stage_bytes<S>() + 256; }
static_assert(kF64sAcc * kF64sN <= 512, "accumulators exceed tensor memory");
static_assert(f64s_smem<kF64sDigits>() <= 227 * 1024 && f64s_smem<kF64sDigitsWide>() <= 227 * 1024,
              "stages exceed shared memory");

// The S balanced base-256 digits of v = x 2^-E (|v| < 1) as floats (exact BF16 numbers), by
// integer operations on the bits of x: F = round(|x| 2^(B - E)) with its sign, then one
// addition of 128 to each byte below the first digit makes every digit a byte less 128.
template <int S>
__device__ __forceinline__ void digits_of(double x, int E, float out[S]) {
  constexpr int B = f64s_bits<S>();
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int ebits = (int)((bits >> 52) & 0x7ff);
  const unsigned long long mant = (bits & 0xfffffffffffffull) | (ebits ? (1ull << 52) : 0ull);
  const int sh = 1075 - B + E - (ebits ? ebits : 1);   // F = mant 2^-sh, sh >= 53 - B for |v| < 1
  unsigned long long F;
  if (B > 53 && sh <= 0) {
    F = mant << min(-sh, 63);
  } else {
    const int r = min(max(sh, 1), 63);
    F = (mant + (1ull << (r - 1))) >> r;
  }
  const unsigned long long neg = (unsigned long long)((long long)bits >> 63);   // 0 or all ones
  constexpr unsigned long long bias = (0x8080808080808080ull >> (8 * (8 - (S - 1))));
  const unsigned long long t = ((F ^ neg) - neg) + bias;
  const uint32_t lo = (uint32_t)t, hi = (uint32_t)(t >> 32);
  // 2^23 + byte as a float, less 2^23 + 128
#pragma unroll
  for (int i = 1; i < S; ++i) {
    const int byte = S - 1 - i;
    const uint32_t f = __byte_perm(byte < 4 ? lo : hi, 0x4B000000u, 0x7650u + (byte & 3));
    out[i] = __uint_as_float(f) - 8388736.f;
  }
  const int d0 = (int)((long long)t >> (8 * (S - 1)));   // |d0| <= 2^top
  out[0] = __uint_as_float(0x4B000000u + (uint32_t)(d0 + 512)) - 8389120.f;
}

// Exponent E with max|entries| < 2^E (0 for an all-zero vector), from the bits of the
// maximum (non-negative doubles order like their bits, so maxima are integer compares).  An
// infinity or a NaN gives 1025, more than any finite maximum: such a column's outputs are NaN.
constexpr int kExpNonFinite = 1025;
__device__ __forceinline__ int exp_above(unsigned long long mbits) {
  if (mbits == 0ull) return 0;
  const int e = (int)(mbits >> 52);
  return e ? e - 1022 : -1010 - __clzll((long long)mbits);   // subnormal: top bit p, 2^(p - 1074) <= m
}

__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

// Set-up: rows of every matrix (mats of Nr x Nr, row-major [n][j]) into S BF16 planes
// [mat * S + plane][n][pitch] and the row exponents rowexp[mat][n].  One warp per row.
template <int S>
__global__ void k_f64s_matrix(const double* __restrict__ A, int nmat, int Nr, int pitch, uint16_t* __restrict__ planes,
                              int32_t* __restrict__ rowexp) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= nmat * Nr) return;
  const int mat = warp / Nr, n = warp - mat * Nr;
  const double* row = A + ((size_t)mat * Nr + n) * Nr;
  unsigned long long m = 0ull;
  for (int j = lane; j < Nr; j += 32) m = max(m, abs_bits(row[j]));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int E = exp_above(m);
  if (lane == 0) rowexp[mat * Nr + n] = E;
  const size_t plane_elems = (size_t)Nr * pitch;
  for (int j = lane; j < pitch; j += 32) {
    float d[S];
    digits_of<S>(j < Nr ? row[j] : 0.0, E, d);
#pragma unroll
    for (int i = 0; i < S; ++i)
      planes[((size_t)mat * S + i) * plane_elems + (size_t)n * pitch + j] = (uint16_t)(__float_as_uint(d[i]) >> 16);
  }
}

// Per DHT: the panels' column exponents and their S K-major BF16 planes [b * S + plane][c][jpad].
// One CTA per 32 columns of an item: the first walk over the rows takes the column maxima, the
// second (from L2: the CTA's Nr x 256 bytes were just read) cuts the digits, in tiles of 64 rows
// through shared memory, read along c and written along j in 16-byte stores.  Bound by its
// memory traffic, 8 bytes in and 2 S out per value.  One kernel instead of a column-maximum
// kernel with atomics, its memset and a slicing kernel that read the panel from HBM again.
constexpr int kPanelC = 32, kPanelJ = 64, kPanelPitch = kPanelJ / 2 + 1;   // 32-bit words per row
template <int S>
__global__ void __launch_bounds__(256) k_f64s_panel(DhtBatch bt, int b0, int Nr, int Nc, int jpad,
                                                    int32_t* __restrict__ colexp, uint16_t* __restrict__ planes) {
  __shared__ uint32_t tile[S][kPanelC][kPanelPitch];   // two j per word; odd pitch: no bank conflicts
  __shared__ unsigned long long cmax[8][kPanelC];
  const int c0 = blockIdx.x * kPanelC;
  const double* X = static_cast<const double*>(bt.X[b0 + blockIdx.y]);
  const int tc = threadIdx.x & (kPanelC - 1), tj = threadIdx.x >> 5;   // 32 x 8
  const int c = c0 + tc;
  const bool in = c < Nc;
  unsigned long long m = 0ull;
  if (in) {
#pragma unroll 16
    for (int j = tj; j < Nr; j += 8) m = max(m, abs_bits(X[(size_t)j * Nc + c]));
  }
  cmax[tj][tc] = m;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q) m = max(m, cmax[q][tc]);
  const int E = exp_above(m);
  if (tj == 0 && in) colexp[(size_t)blockIdx.y * Nc + c] = E;   // for the epilogue
  const size_t plane_elems = (size_t)Nc * jpad;
  uint16_t* out = planes + (size_t)blockIdx.y * S * plane_elems;
  for (int j0 = 0; j0 < Nr; j0 += kPanelJ) {
    double xv[kPanelJ / 8];   // all loads first, then the digits; row pairs (2 jp, 2 jp + 1)
#pragma unroll
    for (int u = 0; u < kPanelJ / 8; ++u) {
      const int j = j0 + 2 * (tj + 8 * (u >> 1)) + (u & 1);
      xv[u] = (in && j < Nr) ? X[(size_t)j * Nc + c] : 0.0;
    }
    __syncthreads();   // the previous tile has been written out
#pragma unroll
    for (int u = 0; u < kPanelJ / 16; ++u) {
      float a[S], b[S];
      digits_of<S>(xv[2 * u], E, a);
      digits_of<S>(xv[2 * u + 1], E, b);
#pragma unroll
      for (int i = 0; i < S; ++i)   // the high halves: two BF16
        tile[i][tc][tj + 8 * u] = __byte_perm(__float_as_uint(a[i]), __float_as_uint(b[i]), 0x7632);
    }
    __syncthreads();
    // 8 consecutive j (16 bytes) per store; jpad and j0 are multiples of 8, so a group lies
    // inside the row or past it whole
    constexpr int kQ = kPanelJ / 8;
    for (int idx = threadIdx.x; idx < S * kPanelC * kQ; idx += 256) {
      const int jq = idx % kQ, cc = idx / kQ % kPanelC, i = idx / (kQ * kPanelC);
      const int cg = c0 + cc, jg = j0 + 8 * jq;
      if (cg < Nc && jg < jpad) {
        const uint32_t* w = &tile[i][cc][4 * jq];
        *reinterpret_cast<uint4*>(out + i * plane_elems + (size_t)cg * jpad + jg) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
  }
}

// SM100 shared-memory matrix descriptor: K-major, 64-byte swizzle (TMA's SWIZZLE_64B), 8-row
// groups 512 B apart.  The high word is constant; the low word holds the start address in
// 16-byte units, so that moving along the stage is one 32-bit addition.
constexpr uint32_t kDescHi = (512u >> 4) | (1u << 14) | (4u << 29);   // stride, SM100 version, SWIZZLE_64B
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return ((saddr >> 4) & 0x3FFFu) | (1u << 16); }
__device__ __forceinline__ uint64_t desc_of(uint32_t lo) { return ((uint64_t)kDescHi << 32) | lo; }

// 3-D tiled tensor copy global -> shared (inner coordinate x, then y, z), completing its
// bytes on `bar`.  x is a multiple of 32 BF16 elements: 64-byte aligned.
__device__ __forceinline__ void tma_load_3d(void* dst, const void* tmap, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

struct F64sMaps {
  Sim::TensorMapBytes panel;   // [b * S + plane][c][j], box 32 j x 128 c
  Sim::TensorMapBytes mats;    // [mat * S + plane][n][j], box 32 j x 64 n
};

struct F64sParams {
  int Nr, Nc, n_tiles, m_tiles, tiles_total;
  int nw;            // matrix rows n of a tile: 64, or 32 or 16 where 64 would leave SMs without a tile
  int b0;            // first batch item of this launch
  int16_t mat[24];   // compact matrix index of each batch item
};

struct F64sTile {
  int b, n0, c0;
};

// n fastest: the CTAs that run at the same time share a panel tile (it stays in L2).
__device__ __forceinline__ F64sTile f64s_tile(int t, const F64sParams& P) {
  const int nt = t % P.n_tiles;
  const int rest = t / P.n_tiles;
  return F64sTile{rest / P.m_tiles, nt * P.nw, (rest % P.m_tiles) * kF64sM};
}

// The issuing thread of warp W: the products of its accumulators over the digit pairs of one 16-K
// step.  fresh: the step opens a K block, so each accumulator's first product overwrites it.
template <int S, int W>
__device__ __forceinline__ void issue_products(uint32_t tmem, uint32_t la, uint32_t lb, uint32_t idesc, bool fresh) {
  using F = F64sForm<S>;
#pragma unroll
  for (int a = 0; a < kF64sAcc; ++a) {
    if (F::warp(a) != W) continue;
    bool first = true;
#pragma unroll
    for (int i = 0; i < S; ++i) {   // matrix digit i, panel digit j
#pragma unroll
      for (int j = 0; i + j < S; ++j) {
        if (F::acc(i, j) != a) continue;
        mma_f16(tmem + a * kF64sN, desc_of(la + j * (kF64sPlaneA >> 4)), desc_of(lb + i * (kF64sPlaneB >> 4)), idesc,
                first && fresh ? 0u : 1u);
        first = false;
      }
    }
  }
}

// 4 columns of one accumulator.
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}

__device__ __forceinline__ int acc_int(uint32_t r) { return __float2int_rn(__uint_as_float(r)); }

// (double)v by integer operations (round to nearest, ties to even): the conversion and the test for
// zero ran on the float64 unit, 4 us of a tile's epilogue where no other tile's products hide it.
__device__ __forceinline__ double to_double_rn(long long v) {
  const unsigned long long a = (unsigned long long)(v < 0 ? -v : v);
  if (a == 0ull) return 0.0;
  const int lz = __clzll((long long)a);
  const unsigned long long t = a << lz, rest = t & 0x7ffull;
  unsigned long long r = t >> 11;   // 53 bits; the leading one carries into the exponent
  r += rest > 0x400ull || (rest == 0x400ull && (r & 1ull)) ? 1ull : 0ull;
  return __longlong_as_double((long long)((((unsigned long long)(1085 - lz)) << 52) + r) |
                              (v < 0 ? (long long)0x8000000000000000ull : 0ll));
}

// y = t 2^k (t a float64 near an integer), the scaling as an addition to the exponent field
// while the result stays normal.
__device__ __forceinline__ double scale_pow2(double t, int k) {
  const long long bits = __double_as_longlong(t);
  const int ex = (int)((bits >> 52) & 0x7ff) + k;
  if ((bits << 1) != 0 && ex > 0 && ex < 2047) return __longlong_as_double(bits + (long long)k * (1LL << 52));
  return t * ldexp(1.0, k);   // zero, or a result outside the normal range
}

// A tile's accumulators are drained in two steps: the group sums of a thread's 16 outputs are
// combined into 64-bit integers and TMEM is released at once, so that the next tile's products
// run while these warps convert to float64 (on the integer units; S = 8 adds its two sums in one
// float64 operation an output) and store.  With the conversions before the release the products
// stood still for 14 k of a tile's 35 k cycles.
template <int S>
__global__ void __launch_bounds__(kF64sThreads, 1) k_dht_f64s(DhtBatch bt, F64sParams P,
                                                               const __grid_constant__ F64sMaps maps,
                                                               const int32_t* __restrict__ colexp,
                                                               const int32_t* __restrict__ rowexp, int32_t* err) {
  constexpr int kStages = F64sForm<S>::stages;
  constexpr uint32_t kStageBytes = f64s_stage_bytes<S>();
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(base + kStages * kStageBytes);
  uint64_t* empty = full + kStages;
  uint64_t* tfull = empty + kStages;
  uint64_t* tempty = tfull + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nK = (P.Nr + kF64sKC - 1) / kF64sKC;       // K chunks of a tile
  constexpr int kPerBlock = kF64sKBlock / kF64sKC;     // K chunks between drains
  constexpr uint32_t kTmemCols = 512;

  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&full[i], 1);    // the copy issuer's arrive.expect_tx
      mbar_init(&empty[i], 3);   // one MMA commit per issuing warp
    }
    mbar_init(tfull, 3);    // the issuing warps' commits after a K block's last chunk
    mbar_init(tempty, 16);  // one arrival per epilogue warp
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  // kind::f16: D f32, A and B bf16, both K-major; N = nw, M = 128
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(P.nw >> 3) << 17) |
                         ((uint32_t)(kF64sM >> 4) << 24);

  auto fail = [&]() {
    *abort_flag = 1;
    atomicOr(err, kErrTimeout);
  };

  if (warp == 0) {
    // ---------------------------------------------------------------- copy issuer
    if (lane == 0) {
      uint32_t g = 0;
      int last_armed = -1;
      for (int t = blockIdx.x; t < P.tiles_total && !*abort_flag; t += gridDim.x) {
        const F64sTile w = f64s_tile(t, P);
        const int zm = P.mat[P.b0 + w.b] * S, zp = w.b * S;
        bool ok = true;
        for (int kc = 0; kc < nK; ++kc, ++g) {
          const int st = (int)(g % (uint32_t)kStages);
          const uint32_t use = g / (uint32_t)kStages;
          if (use > 0 && !mbar_wait(&empty[st], (use - 1) & 1)) { fail(); ok = false; break; }
          if (*abort_flag) { ok = false; break; }
          unsigned char* sA = base + st * kStageBytes;
          unsigned char* sB = sA + S * kF64sPlaneA;
          mbar_arrive_expect_tx(&full[st], kStageBytes);
#pragma unroll
          for (int p = 0; p < S; ++p)
            tma_load_3d(sA + p * kF64sPlaneA, &maps.panel, kc * kF64sKC, w.c0, zp + p, &full[st]);
#pragma unroll
          for (int p = 0; p < S; ++p)
            tma_load_3d(sB + p * kF64sPlaneB, &maps.mats, kc * kF64sKC, w.n0, zm + p, &full[st]);
          last_armed = st;
        }
        if (!ok) break;
      }
      // before shared memory is released: the last armed stage's copies must have landed
      if (last_armed >= 0 && *abort_flag) {
        const uint32_t gl = g == 0 ? 0 : g - 1;
        mbar_wait(&full[last_armed], (gl / (uint32_t)kStages) & 1);
      }
    }
    __syncwarp();
  } else if (warp >= 1 && warp <= 3) {
    // ---------------------------------------------------------------- MMA issuers
    // Three warps issue the products, each into its own accumulators (so every accumulator's
    // first, overwriting product comes from one thread).  One thread issuing all of them left
    // the tensor pipe three quarters idle.
    if (lane == 0) {
      uint32_t g = 0, i = 0;   // chunks, K blocks
      uint64_t* last_bar = nullptr;
      uint32_t last_parity = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < P.tiles_total && !*abort_flag; t += gridDim.x) {
        for (int k0 = 0; ok && k0 < nK; k0 += kPerBlock, ++i) {
          if (i > 0 && !mbar_wait(tempty, (i - 1) & 1)) { fail(); ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const int k1 = min(k0 + kPerBlock, nK);
          for (int kc = k0; kc < k1; ++kc, ++g) {
            const int st = (int)(g % (uint32_t)kStages);
            if (!mbar_wait(&full[st], (g / (uint32_t)kStages) & 1)) { fail(); ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t la = desc_lo(smem_u32(base + st * kStageBytes)), lb = la + ((S * kF64sPlaneA) >> 4);
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {   // 16 K: 32 bytes along the swizzled row
              const bool fresh = kc == k0 && ks == 0;
              if (warp == 1) issue_products<S, 1>(tmem, la + 2 * ks, lb + 2 * ks, idesc, fresh);
              else if (warp == 2) issue_products<S, 2>(tmem, la + 2 * ks, lb + 2 * ks, idesc, fresh);
              else issue_products<S, 3>(tmem, la + 2 * ks, lb + 2 * ks, idesc, fresh);
            }
            mma_commit(&empty[st]);
            last_bar = &empty[st];
            last_parity = (g / (uint32_t)kStages) & 1;
          }
          if (!ok) break;
          mma_commit(tfull);
          last_bar = tfull;
          last_parity = i & 1;
        }
      }
      if (*abort_flag && last_bar) mbar_wait(last_bar, last_parity);
    }
    __syncwarp();
  } else if (warp >= 4) {
    // ---------------------------------------------------------------- epilogue (warps 4-19)
    // four warps per TMEM lane quarter (warp % 4 == q: lanes 32q .. 32q + 31), each taking
    // a quarter of the tile's columns
    constexpr int kCols = kF64sN / 4;
    const int cols = P.nw / 4, q = warp & 3, jh = ((warp - 4) >> 2) * cols;
    const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)jh;
    uint32_t i = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < P.tiles_total && !*abort_flag; t += gridDim.x) {
      const F64sTile w = f64s_tile(t, P);
      // S = 6: sum = hi 2^-54 (group 5 rounded to that unit); S = 8: sum = hi 2^-36 + lo 2^-68
      long long hi[kCols], lo[S == kF64sDigits ? 1 : kCols];
#pragma unroll
      for (int e = 0; e < kCols; ++e) {
        hi[e] = 0;
        if (S != kF64sDigits) lo[e] = 0;
      }
      for (int k0 = 0; k0 < nK; k0 += kPerBlock, ++i) {
        if (!mbar_wait(tfull, i & 1)) { fail(); ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int j = 0; j < kCols; j += 4) {
          if (j >= cols) break;
          uint32_t r[kF64sAcc][4];
#pragma unroll
          for (int a = 0; a < kF64sAcc; ++a) tmem_ld4(taddr + a * kF64sN + j, r[a]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if constexpr (S == kF64sDigits) {
              // one K block: the groups' weights are 2^-(16 + 8 g); |sum| <= 2^8
              const long long a0 = acc_int(r[0][e]), a1 = acc_int(r[1][e]);
              const long long a2 = acc_int(r[2][e]) + acc_int(r[3][e]), a3 = acc_int(r[4][e]) + acc_int(r[5][e]);
              const int a4 = acc_int(r[6][e]), a5 = __float2int_rn(__uint_as_float(r[7][e]) * 0.25f);
              hi[j + e] = a0 * (1LL << 38) + a1 * (1LL << 30) + a2 * (1LL << 22) + a3 * (1LL << 14) +
                          ((long long)a4 * 64 + a5);
            } else {
              // weights 2^-(12 + 8 g); |a_g| <= 2^25 a block and at most 4 blocks: both sums < 2^53
              hi[j + e] += (long long)acc_int(r[0][e]) * (1 << 24) + (long long)acc_int(r[1][e]) * (1 << 16) +
                           (long long)acc_int(r[2][e]) * (1 << 8) + acc_int(r[3][e]);
              lo[j + e] += (long long)acc_int(r[4][e]) * (1 << 24) + (long long)acc_int(r[5][e]) * (1 << 16) +
                           (long long)acc_int(r[6][e]) * (1 << 8) + acc_int(r[7][e]);
            }
            // combined before the next columns are loaded (else their raw sums pile up in registers)
            asm volatile("" : "+l"(hi[j + e]));
            if (S != kF64sDigits) asm volatile("" : "+l"(lo[S == kF64sDigits ? 0 : j + e]));
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty);
      }
      if (!ok) break;
      double* __restrict__ Y = static_cast<double*>(bt.Y[P.b0 + w.b]);
      const int c = w.c0 + q * 32 + lane, n0 = w.n0 + jh;
      if (c < P.Nc) {
        const int Ec = colexp[(size_t)w.b * P.Nc + c];
        const int32_t* rexp = rowexp + (size_t)P.mat[P.b0 + w.b] * P.Nr;
#pragma unroll
        for (int e = 0; e < kCols; ++e) {
          const int n = n0 + e;
          if (e < cols && n < P.Nr) {
            double v;
            int k = Ec + rexp[n];
            if constexpr (S == kF64sDigits) {
              v = to_double_rn(hi[e]);
              k -= 54;
            } else {
              v = fma(to_double_rn(lo[e]), 0x1p-32, to_double_rn(hi[e]));   // exact conversions, one rounding
              k -= 36;
            }
            Y[(size_t)n * P.Nc + c] =
                Ec == kExpNonFinite ? __longlong_as_double(0x7ff8000000000000ll) : scale_pow2(v, k);
          }
          asm volatile("" ::: "memory");   // one output at a time: no pile of addresses and exponents
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

int f64s_pitch(int Nr) { return split_pitch_b16(Nr); }   // BF16 row pitch, 16-byte rows

int blocks_for(size_t n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

bool f64s_supported(const pic_config& c) { return c.precision == PIC_FP64 && c.Nr <= kF64sMaxNr; }

int f64s_digits(const pic_config& c) { return c.Nr <= kF64sMaxNr ? kF64sDigits : kF64sDigitsWide; }

// Items whose panel planes are held at a time.  The wide form's planes are twice the panels' bytes: a
// launch takes as many items as fit 1 GB (all 12 of a 2-mode run up to 2048 x 1024).  The planes share
// their memory with the spare particle buffer, so only handles of few particles a cell grow with them (by up
// to a third, at 1800 x 400 x 2 without particles).  Fewer items a launch cost more than they save: field
// cycles at 1800 x 400 x 2 and 4096 x 512 x 3 take 1.98 and 7.59 ms at 1 GB, 2.03 and 7.89 at 256 MB, 2.30
// and 9.06 at 64 MB (last waves of tiles).
int f64s_items(const pic_config& c) {
  const size_t item = (size_t)f64s_digits(c) * 2 * c.Nz * f64s_pitch(c.Nr) * 2;
  const int all = 6 * c.Nm;
  if (c.Nr <= kF64sMaxNr) return all;
  return std::max(1, std::min<int>(all, (int)(((size_t)1 << 30) / item)));
}

bool f64s_active(const Sim* s) { return s->cfg.precision == PIC_FP64 && s->dht_path != PIC_DHT_F64_GEMM; }

pic_status f64s_configure_device() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  PIC_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  if (dev >= 0 && dev < 64 && done[dev]) return PIC_OK;
  PIC_CUDA(cudaFuncSetAttribute(k_dht_f64s<kF64sDigits>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)f64s_smem<kF64sDigits>()));
  PIC_CUDA(cudaFuncSetAttribute(k_dht_f64s<kF64sDigitsWide>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)f64s_smem<kF64sDigitsWide>()));
  if (dev >= 0 && dev < 64) done[dev] = true;
  return PIC_OK;
}

// Set-up (after the FP64 matrices are final): digits of the forward matrices (compact
// index 0 .. 3Nm-1) and of the inverse matrices (3Nm .. 6Nm-1).
pic_status launch_f64s_setup(Sim* s) {
  const int Nr = s->cfg.Nr, nm3 = 3 * s->cfg.Nm, pitch = f64s_pitch(Nr), S = f64s_digits(s->cfg);
  uint16_t* planes = s->at<uint16_t>(s->lay.f64s_mat);
  int32_t* rowexp = s->at<int32_t>(s->lay.f64s_rowexp);
  const size_t mat_elems = (size_t)S * Nr * pitch;
  const int blocks = blocks_for((size_t)nm3 * Nr * 32, 256);
  auto* k = S == kF64sDigits ? k_f64s_matrix<kF64sDigits> : k_f64s_matrix<kF64sDigitsWide>;
  k<<<blocks, 256, 0, s->stream>>>(s->at<double>(s->lay.mfwd), nm3, Nr, pitch, planes, rowexp);
  PIC_LAUNCHED(s);
  k<<<blocks, 256, 0, s->stream>>>(s->at<double>(s->lay.binv), nm3, Nr, pitch, planes + (size_t)nm3 * mat_elems,
                                   rowexp + (size_t)nm3 * Nr);
  PIC_LAUNCHED(s);
  return PIC_OK;
}

// Tensor maps of the panel planes and matrix planes (3-D: inner j, then c or n, then
// item or matrix x plane), 64-byte swizzle; coordinates past Nr (j, n) or Nc read zero.
pic_status f64s_make_maps(Sim* s) {
  std::memset(s->f64s_maps, 0, sizeof(s->f64s_maps));
  if (s->cfg.precision != PIC_FP64) return PIC_OK;
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  Encode encode = reinterpret_cast<Encode>(tensor_map_encoder());
  if (!encode) {
    set_error("cuTensorMapEncodeTiled is not available from the driver");
    return PIC_ERR_CUDA;
  }
  const int Nr = s->cfg.Nr, Nc = 2 * s->cfg.Nz, pitch = f64s_pitch(Nr), S = f64s_digits(s->cfg);
  auto make = [&](int id, size_t off, int rows, int planes, int box_rows, const char* what) -> pic_status {
    const cuuint32_t estr[3] = {1, 1, 1};
    const cuuint64_t dims[3] = {(cuuint64_t)Nr, (cuuint64_t)rows, (cuuint64_t)planes};
    const cuuint64_t strides[2] = {(cuuint64_t)pitch * 2, (cuuint64_t)rows * pitch * 2};
    const cuuint32_t box[3] = {(cuuint32_t)kF64sKC, (cuuint32_t)box_rows, 1};
    const CUresult r = encode(reinterpret_cast<CUtensorMap*>(s->f64s_maps[id].b), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
                              s->at<char>(off), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r == CUDA_SUCCESS) return PIC_OK;
    set_error("cuTensorMapEncodeTiled failed (%d) for the sliced %s", (int)r, what);
    return PIC_ERR_CUDA;
  };
  for (int b = 0; b < 2; ++b)
    if (const pic_status st = make(b, s->lay.f64s_panel[b], Nc, f64s_items(s->cfg) * S, kF64sM, "panels")) return st;
  return make(2, s->lay.f64s_mat, Nr, 6 * s->cfg.Nm * S, kF64sN, "matrices");
}

namespace {

template <int S>
pic_status launch_items(Sim* s, const DhtBatch& b, F64sParams P, int items) {
  const int Nr = P.Nr, Nc = P.Nc;
  int32_t* colexp = s->at<int32_t>(s->lay.f64s_colexp);
  k_f64s_panel<S><<<dim3(blocks_for(Nc, kPanelC), items), 256, 0, s->stream>>>(
      b, P.b0, Nr, Nc, f64s_pitch(Nr), colexp, s->at<uint16_t>(s->lay.f64s_panel[s->cur]));
  PIC_LAUNCHED(s);
  F64sMaps maps;
  maps.panel = s->f64s_maps[s->cur];
  maps.mats = s->f64s_maps[2];
  // narrower tiles while all of them still find an SM at once (256 x 64 x 2 modes, 32 and 48 tiles of
  // 64 rows: 17.3 -> 12.5 us a launch with 16 and 32 rows and the epilogue off the float64 unit)
  P.nw = kF64sN;
  const auto tiles = [&](int nw) { return (Nr + nw - 1) / nw * P.m_tiles * items; };
  while (P.nw > 16 && tiles(P.nw / 2) <= dht_tc_sm_count()) P.nw /= 2;
  P.n_tiles = (Nr + P.nw - 1) / P.nw;
  P.tiles_total = P.n_tiles * P.m_tiles * items;
  const int grid = std::min(P.tiles_total, dht_tc_sm_count());
  k_dht_f64s<S><<<grid, kF64sThreads, f64s_smem<S>(), s->stream>>>(b, P, maps, colexp,
                                                                   s->at<int32_t>(s->lay.f64s_rowexp),
                                                                   s->at<int32_t>(s->lay.err));
  PIC_LAUNCHED(s);
  return PIC_OK;
}

}  // namespace

// Y = A X of a batch in the FP64 form on the tensor cores: column exponents and panel digits,
// then the persistent product kernel.
pic_status launch_dht_f64s(Sim* s, const DhtBatch& b) {
  const int Nm = s->cfg.Nm;
  if (b.n < 1 || b.n > 6 * Nm) {
    set_error("sliced FP64 DHT: batch of %d items (1 .. %d)", b.n, 6 * Nm);
    return PIC_ERR_ARG;
  }
  F64sParams P{};
  P.Nr = s->cfg.Nr;
  P.Nc = 2 * s->cfg.Nz;
  P.m_tiles = (P.Nc + kF64sM - 1) / kF64sM;
  for (int i = 0; i < b.n; ++i) {
    const int id = b.mat[i], per = kMaxModes * 3;
    const int dir = id / per, mi = id % per;
    if (id < 0 || dir > 1 || mi >= 3 * Nm) {
      set_error("sliced FP64 DHT: batch entry %d has no matrix", i);
      return PIC_ERR_ARG;
    }
    P.mat[i] = (int16_t)(dir * 3 * Nm + mi);
  }
  const int most = f64s_items(s->cfg);
  for (; P.b0 < b.n; P.b0 += most) {
    const int items = std::min(most, b.n - P.b0);
    const pic_status st = f64s_digits(s->cfg) == kF64sDigits ? launch_items<kF64sDigits>(s, b, P, items)
                                                             : launch_items<kF64sDigitsWide>(s, b, P, items);
    if (st != PIC_OK) return st;
  }
  return PIC_OK;
}

}  // namespace pic
