// Row DFT along z of the FP64 form (a5, a9) in 64-bit block fixed point, for every 7-smooth
// length (Fourier transform along z of the quasi-cylindrical scheme, section "Finite order
// pseudo-spectral solvers"):
//   forward: Fhat(k) = sum_i F(z_i) e^{-2 pi i k i / Nz}
//   inverse: F(z_i) = (1/Nz) sum_k Fhat(k) e^{+2 pi i k i / Nz}
// GB300's float64 unit does 2 operations a clock and SM, its integer and float32 units 128, and
// an FFT's numbers share one scale: float64 rows are no more accurate than eps times the row's
// norm.  So a row is held as 64-bit integers with one exponent:
//   * the row's largest exponent scales its values to |re|, |im| < 2^59 (2^58 each for the two
//     rows of a combination);
//   * a pass multiplies by twiddles (61 fraction bits; the product keeps half, so that it has the
//     head room for the butterfly), adds, and collects the bits of its outputs' magnitudes; the
//     next pass shifts the row so that its largest value lies between 2^59 and 2^60, and the
//     row's exponent counts it.  Sums are exact; a product is off by at most 2 units;
//   * the last pass converts to float64 with one rounding.
// The error stays near 2^-57 of the row's largest value, below the rounding of the twiddles
// (float64 values) and of the results: against extended precision the tests hold it, at every length
// and shape of row, below 1.25 times that of the IEEE float64 passes or one rounding of the row's norm.
// A 64-bit addition is two instructions and a complex product about 22 (12 wide multiply-adds of
// 31-bit halves), against 11 and 54 for pairs of floats and, for float64, the time of 64 and 256.
// Rows with an infinity or a NaN become NaN.
// Bound by instruction issue (about half of the issue slots; the integer unit's 64 lanes a clock
// are its busiest part).  The power-of-two kernel spills 504 bytes of stores and 816 of loads a thread
// at its 64 registers forward (two sources' eight values and their sums), 108 and 500 inverse.
// Measured, forward + inverse rows of one cycle: 2048 points x 256 x 2 modes 126 + 204 us with float
// pairs -> 95 + 163 us; 1800 points x 400 x 2 modes 558 + 859 us in IEEE float64 -> 200 + 300 us.
//
// Radix-8 (4, 2, 3, 5, 7) self-sorting Stockham passes, butterflies in registers, the first
// pass from global memory with the component combination (J_+- = (J_r -+ i J_theta)/2 before
// the forward transform, E_r = E_+ + E_-, E_theta = i (E_+ - E_-) before the inverse one) and
// the last pass to global memory.  Power-of-two rows exchange values through one shared row
// buffer (8 values per thread, several short rows per CTA), other lengths between two.
#include <algorithm>
#include <mutex>

#include "dword.cuh"
#include "pic_internal.cuh"

namespace pic {
namespace {

struct fx2 {
  long long x, y;
};

__device__ __forceinline__ fx2 operator+(fx2 a, fx2 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ fx2 operator-(fx2 a, fx2 b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ fx2 shr(fx2 a, int s) { return {a.x >> s, a.y >> s}; }

__device__ __forceinline__ long long wide(int a, int b) { return (long long)a * b; }
__device__ __forceinline__ int hi31(long long a) { return (int)(a >> 31); }                // |a| < 2^62
__device__ __forceinline__ int lo31(long long a) { return (int)((unsigned)a & 0x7fffffffu); }

// v w / 2 for a twiddle w = (c + i s) 2^-61, c = w.x 2^31 + w.y, s = w.z 2^31 + w.w, and |re|,
// |im| of v below 2^60: the products of the low halves are left out (below one unit).
__device__ __forceinline__ fx2 cmul_half(fx2 v, int4 w) {
  const int xh = hi31(v.x), xl = lo31(v.x), yh = hi31(v.y), yl = lo31(v.y);
  const long long tr = wide(xh, w.y) + wide(xl, w.x) - wide(yh, w.w) - wide(yl, w.z);
  const long long ti = wide(xh, w.w) + wide(xl, w.z) + wide(yh, w.y) + wide(yl, w.x);
  return {wide(xh, w.x) - wide(yh, w.z) + (tr >> 31), wide(xh, w.z) + wide(yh, w.x) + (ti >> 31)};
}

// a c 2^-62 for a constant c = ch 2^31 + cl below 2^62 in magnitude and |a| < 2^62.
__device__ __forceinline__ long long mul_const(long long a, int ch, int cl) {
  const int ah = hi31(a), al = lo31(a);
  return wide(ah, ch) + ((wide(ah, cl) + wide(al, ch)) >> 31);
}
// a times the constant c in (-1, 1), its halves folded at compile time.
__host__ __device__ constexpr long long fix62(double c) { return (long long)(c * 4611686018427387904.0); }
__device__ __forceinline__ long long mul_c(long long a, double c) {
  const long long f = fix62(c);
  return mul_const(a, (int)(f >> 31), (int)(f & 0x7fffffff));
}

template <bool INV> __device__ __forceinline__ fx2 mul_mi(fx2 a) {   // times -i (forward) or +i
  return INV ? fx2{-a.y, a.x} : fx2{a.y, -a.x};
}

template <bool INV> __device__ __forceinline__ void dft4(fx2* v) {
  const fx2 s02 = v[0] + v[2], d02 = v[0] - v[2], s13 = v[1] + v[3], d13 = mul_mi<INV>(v[1] - v[3]);
  v[0] = s02 + s13;
  v[1] = d02 + d13;
  v[2] = s02 - s13;
  v[3] = d02 - d13;
}

// 8 points as two 4-point DFTs: even outputs of a_r = v_r + v_{r+4}, odd ones of
// b_r = (v_r - v_{r+4}) w_8^r.
template <bool INV> __device__ __forceinline__ void dft8(fx2* v) {
  constexpr double h = 0.70710678118654752440;
  fx2 a[4], b[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    a[r] = v[r] + v[r + 4];
    b[r] = v[r] - v[r + 4];
  }
  const fx2 p = b[1], q = b[3];
  b[1] = INV ? fx2{mul_c(p.x - p.y, h), mul_c(p.x + p.y, h)} : fx2{mul_c(p.x + p.y, h), mul_c(p.y - p.x, h)};
  b[2] = mul_mi<INV>(b[2]);
  b[3] = INV ? fx2{-mul_c(q.x + q.y, h), mul_c(q.x - q.y, h)} : fx2{mul_c(q.y - q.x, h), -mul_c(q.x + q.y, h)};
  dft4<INV>(a);
  dft4<INV>(b);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    v[2 * r] = a[r];
    v[2 * r + 1] = b[r];
  }
}

// cos and sin of 2 pi j / R, 1 <= j <= (R - 1) / 2, R = 3, 5, 7.
__host__ __device__ constexpr double root_cos(int R, int j) {
  return R == 3 ? -0.5
       : R == 5 ? (j == 1 ? 0.3090169943749474241023 : -0.8090169943749474241023)
       : (j == 1 ? 0.6234898018587335305250 : j == 2 ? -0.2225209339563144042889 : -0.9009688679024191262361);
}
__host__ __device__ constexpr double root_sin(int R, int j) {
  return R == 3 ? 0.8660254037844386467637
       : R == 5 ? (j == 1 ? 0.9510565162951535721164 : 0.5877852522924731291687)
       : (j == 1 ? 0.7818314824680298087084 : j == 2 ? 0.9749279121818236070181 : 0.4338837391175581204758);
}

// y_m, y_{R-m} = v_0 + sum_q (v_q + v_{R-q}) cos(2 pi q m / R) -+ i sum_q (v_q - v_{R-q})
// sin(2 pi q m / R), R odd.
template <bool INV, int R> __device__ __forceinline__ void dft_odd(fx2* v) {
  constexpr int H = (R - 1) / 2;
  fx2 sp[H + 1], sm[H + 1], y0 = v[0];
#pragma unroll
  for (int q = 1; q <= H; ++q) {
    sp[q] = v[q] + v[R - q];
    sm[q] = v[q] - v[R - q];
    y0 = y0 + sp[q];
  }
#pragma unroll
  for (int m = 1; m <= H; ++m) {
    fx2 a = v[0], b = {0, 0};
#pragma unroll
    for (int q = 1; q <= H; ++q) {
      const int j = (q * m) % R, jj = j <= H ? j : R - j;
      const double sn = j <= H ? root_sin(R, jj) : -root_sin(R, jj);
      a = a + fx2{mul_c(sp[q].x, root_cos(R, jj)), mul_c(sp[q].y, root_cos(R, jj))};
      b = b + fx2{mul_c(sm[q].x, sn), mul_c(sm[q].y, sn)};
    }
    const fx2 lo = {a.x + b.y, a.y - b.x}, hi = {a.x - b.y, a.y + b.x};   // a - i b, a + i b
    v[m] = INV ? hi : lo;
    v[R - m] = INV ? lo : hi;
  }
  v[0] = y0;
}

template <bool INV, int R> __device__ __forceinline__ void dft(fx2* v) {
  if constexpr (R == 2) {
    const fx2 a = v[0], b = v[1];
    v[0] = a + b;
    v[1] = a - b;
  } else if constexpr (R == 4) {
    dft4<INV>(v);
  } else if constexpr (R == 8) {
    dft8<INV>(v);
  } else {
    dft_odd<INV, R>(v);
  }
}

// Magnitude bits of v's components (their high words), for the row's common exponent.
__device__ __forceinline__ unsigned mag_bits(fx2 v) {
  const int a = (int)(v.x >> 32), b = (int)(v.y >> 32);
  return (unsigned)(a ^ (a >> 31)) | (unsigned)(b ^ (b >> 31));
}
// Right shift (left where negative) that brings components whose high words have these bits
// below 2^60, the largest to at least 2^59.
__device__ __forceinline__ int shift_for(unsigned bits) { return 4 - __clz((int)(bits | 1u)); }
// v 2^-s, s the same for a whole row.
template <int M> __device__ __forceinline__ void shift_all(fx2 (&v)[M], int s) {
  if (s > 0) {
#pragma unroll
    for (int e = 0; e < M; ++e) v[e] = shr(v[e], s);
  } else if (s < 0) {
#pragma unroll
    for (int e = 0; e < M; ++e) v[e] = {v[e].x << -s, v[e].y << -s};
  }
}

__device__ __forceinline__ unsigned abs_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// x 2^(Q - E) as an integer, |x| < 2^E: r0 = 1086 - Q + E (bits below one unit are cut off).
// Rows whose largest value is above 2^-900 need no care for subnormal x: they come out as 0 or 1.
__device__ __forceinline__ long long to_fixed(double x, int r0, bool tiny) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  int e = (int)((hi >> 20) & 0x7ffu);
  unsigned mh = (hi & 0xfffffu) | 0x100000u;
  if (tiny && e == 0) {
    mh = hi & 0xfffffu;
    e = 1;
  }
  // the mantissa, top aligned, shifted right by r >= 5: the shifts of 32 and more give 0
  const unsigned th = (mh << 11) | (lo >> 21), tl = lo << 11;
  const unsigned r = (unsigned)(r0 - e);
  const unsigned s = r > 32u ? r - 32u : 0u;
  const unsigned fl = s < 32u ? __funnelshift_rc(tl, th, r) >> s : 0u, fh = r < 32u ? th >> r : 0u;
  const long long F = (long long)(((unsigned long long)fh << 32) | fl);
  return (int)hi < 0 ? -F : F;
}

// Conversion of a row's integers v to v 2^k: the two halves of v become the low mantissa bits of
// 2^(84+k) (high half, offset by 2^31) and 2^(52+k), and two float64 additions (the first exact)
// take the offsets away and round once.  A conversion instruction would be a longer sequence on
// the float64 unit.
struct OutScale {
  int hi_word, lo_word;   // exponent words of 2^(84+k) and 2^(52+k)
  double off;             // 2^(84+k) + 2^(63+k) + 2^(52+k)
  int k;
  bool slow;              // k outside the range of these numbers, or a row to be NaN
};

__device__ __forceinline__ OutScale out_scale(int k, bool bad) {
  OutScale o;
  o.k = bad ? 100000 : k;
  o.slow = bad || k < -1000 || k > 900;
  const int e = o.slow ? 0 : k;
  o.hi_word = (1023 + 84 + e) << 20;
  o.lo_word = (1023 + 52 + e) << 20;
  o.off = __hiloint2double(o.hi_word, (int)0x80000000) + __hiloint2double(o.lo_word, 0);   // 2^84 + 2^63, + 2^52
  return o;
}

__device__ __forceinline__ double to_double(long long v, const OutScale& o) {
  if (o.slow) return o.k == 100000 ? __longlong_as_double(0x7ff8000000000000ll) : ldexp((double)v, o.k);
  const double h = __hiloint2double(o.hi_word, (int)(v >> 32) ^ (int)0x80000000);
  const double l = __hiloint2double(o.lo_word, (int)v);
  return (h - o.off) + l;
}

struct FixArgs {
  const double2* in;
  double2* out;
  float4* out_dw;      // double-word copy of out, or null
  const int4* tw;      // per-pass twiddles, entry L - 1 + (r - 1) L + k
  int N, rows, rows_per_comp;
  int srcA[6], srcB[6];   // srcB < 0: none
  int rotA[6], rotB[6];   // power of i each source is multiplied by
  int half[6];            // 1: the combination is halved
  int nc_hi, nc_lo, nc_exp;   // inverse of a length that is no power of two: 2^nc_exp / N at 62 bits
  int n_pass;
  unsigned long long radix;   // 4 bits each
};

// One row's sources, destination and exponent.
struct RowIO {
  const double2* a;
  const double2* b;
  double2* o;
  float4* odw;
  int ra, rb, r0, ex;
  bool bad, tiny;   // an infinity or a NaN among the inputs; all below 2^-900
};

__device__ __forceinline__ RowIO row_io(const FixArgs& A, int row) {
  RowIO io;
  const int comp = row / A.rows_per_comp, rr = row - comp * A.rows_per_comp;
  io.a = A.in + ((size_t)A.srcA[comp] * A.rows_per_comp + rr) * A.N;
  io.b = A.srcB[comp] >= 0 ? A.in + ((size_t)A.srcB[comp] * A.rows_per_comp + rr) * A.N : nullptr;
  io.ra = A.rotA[comp];
  io.rb = A.rotB[comp];
  io.o = A.out + (size_t)row * A.N;
  io.odw = A.out_dw ? A.out_dw + (size_t)row * A.N : nullptr;
  io.ex = -A.half[comp];
  return io;
}

// The row's scale from the largest high word of its inputs.
__device__ __forceinline__ void set_scale(RowIO& io, unsigned top) {
  const int e = (int)(top >> 20);
  io.bad = e == 0x7ff;
  io.tiny = e < 123;
  const int E = e - 1022, Q = io.b ? 58 : 59;
  io.r0 = 1086 - Q + E;
  io.ex += E - Q;
}

__device__ __forceinline__ fx2 rotate(fx2 v, int r) {   // times i^r (r the same for a whole row)
  if (r & 1) v = {-v.y, v.x};
  if (r & 2) v = {-v.x, -v.y};
  return v;
}

__device__ __forceinline__ fx2 load_in(const RowIO& io, int i) {
  const double2 u = io.a[i];
  fx2 v = rotate({to_fixed(u.x, io.r0, io.tiny), to_fixed(u.y, io.r0, io.tiny)}, io.ra);
  if (io.b) {
    const double2 w = io.b[i];
    v = v + rotate({to_fixed(w.x, io.r0, io.tiny), to_fixed(w.y, io.r0, io.tiny)}, io.rb);
  }
  return v;
}

template <bool INV>
__device__ __forceinline__ void store_out(const FixArgs& A, const RowIO& io, int i, fx2 v, const OutScale& os) {
  if (INV && A.nc_hi) {   // times 1 / N (powers of two: in the exponent)
    v = shr(v, 1);
    v = {mul_const(v.x, A.nc_hi, A.nc_lo), mul_const(v.y, A.nc_hi, A.nc_lo)};
  }
  const double2 y = make_double2(to_double(v.x, os), to_double(v.y, os));
  io.o[i] = y;
  if (io.odw) {
    const dw r = dw_from_double(y.x), m = dw_from_double(y.y);
    io.odw[i] = make_float4(r.hi, r.lo, m.hi, m.lo);
  }
}

// The output scale: the row's exponent, less log2 N (or the factor of store_out) for the inverse.
template <bool INV> __device__ __forceinline__ OutScale out_of(const FixArgs& A, const RowIO& io) {
  return out_scale(INV ? io.ex - A.nc_exp + (A.nc_hi ? 1 : 0) : io.ex, io.bad);
}

// One value of padding per 8 (128 bytes): strides of 8 values, those of the first pass's stores,
// would meet in the same banks.
__device__ __forceinline__ int padded(int i) { return i + (i >> 3); }

// Twiddles and the R-point DFT of one butterfly; v holds inputs below 2^60 (2^59 when FIRST).
template <bool INV, int R, bool FIRST>
__device__ __forceinline__ void butterfly(fx2 (&v)[R], const int4* __restrict__ tw, int L, int k) {
  if (!FIRST) {
    v[0] = shr(v[0], 1);
#pragma unroll
    for (int r = 1; r < R; ++r) {
      int4 w = __ldg(tw + L - 1 + (r - 1) * L + k);
      if (INV) { w.z = -w.z; w.w = -w.w; }
      v[r] = cmul_half(v[r], w);
    }
  }
  dft<INV, R>(v);
}

// ---- power-of-two rows: 8 values per thread, one shared row buffer ----
// A pass of radix R holds 8 / R butterflies per thread: t = tr + q N/8 (q < 8 / R), inputs
// x[t + r N/R], outputs out[j L R + s L + k], k = t mod L, j = t / L.
template <bool INV, int R, bool FIRST, bool LAST>
__device__ __forceinline__ unsigned pow2_pass(fx2 (&v)[8], const FixArgs& A, const RowIO& io, fx2* buf, int tr, int lgL,
                                              bool active, const OutScale& os) {
  const int TR = A.N >> 3, L = 1 << lgL;
  unsigned bits = 0;
#pragma unroll
  for (int q = 0; q < 8 / R; ++q) {
    const int t = tr + q * TR, k = t & (L - 1);
    fx2 u[R];
#pragma unroll
    for (int r = 0; r < R; ++r) u[r] = v[q * R + r];
    butterfly<INV, R, FIRST>(u, A.tw, L, k);
    const int base = ((t >> lgL) * R << lgL) + k;
#pragma unroll
    for (int s = 0; s < R; ++s) {
      const int i = base + (s << lgL);
      if (LAST) {
        if (active) store_out<INV>(A, io, i, u[s], os);
      } else {
        buf[padded(i)] = u[s];
        bits |= mag_bits(u[s]);
      }
    }
  }
  return bits;
}

template <int R> __device__ __forceinline__ void pow2_load(fx2 (&v)[8], const fx2* buf, int N, int tr, int s) {
  const int TR = N >> 3, NR = N / R;
#pragma unroll
  for (int q = 0; q < 8 / R; ++q)
#pragma unroll
    for (int r = 0; r < R; ++r) v[q * R + r] = buf[padded(tr + q * TR + r * NR)];
  shift_all(v, s);
}

// The row's maximum (or union of bits) into a shared word: per warp where a warp lies in one row,
// else (SHORT, rows of less than 256 points) per thread.
template <bool SHORT> __device__ __forceinline__ void row_max(unsigned* word, unsigned m) {
  if constexpr (SHORT) {
    atomicMax(word, m);
  } else {
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(word, m);
  }
}
template <bool SHORT> __device__ __forceinline__ void row_or(unsigned* word, unsigned m) {
  if constexpr (SHORT) {
    atomicOr(word, m);
  } else {
    m = __reduce_or_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicOr(word, m);
  }
}

// A CTA of up to T threads transforms 8 threads / N rows (at least one).
template <bool INV, int T, bool SHORT>
__global__ void __launch_bounds__(T, 1024 / T) k_fft_fix_pow2(const __grid_constant__ FixArgs A, int lgN) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int kMaxRows = SHORT ? T : T / 32;   // a row takes one thread at least (N >= 8), or a warp
  __shared__ unsigned top[kMaxRows], bits[5][kMaxRows];
  const int TR = A.N >> 3, lr = threadIdx.x / TR, tr = threadIdx.x - lr * TR;
  const int rpc = blockDim.x / TR, row = blockIdx.x * rpc + lr;
  const bool active = row < A.rows;
  fx2* buf = reinterpret_cast<fx2*>(smem_raw) + (size_t)lr * (A.N + (A.N >> 3));
  RowIO io = row_io(A, active ? row : 0);
  for (int i = threadIdx.x; i < rpc; i += blockDim.x) {
    top[i] = 0;
#pragma unroll
    for (int p = 0; p < 5; ++p) bits[p][i] = 0;
  }
  __syncthreads();
  {   // the row's scale
    unsigned m = 0;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const double2 u = io.a[tr + r * TR];
      m = max(m, max(abs_hi(u.x), abs_hi(u.y)));
      if (io.b) {
        const double2 w = io.b[tr + r * TR];
        m = max(m, max(abs_hi(w.x), abs_hi(w.y)));
      }
    }
    row_max<SHORT>(&top[lr], m);
  }
  __syncthreads();
  set_scale(io, top[lr]);
  fx2 v[8];
#pragma unroll
  for (int r = 0; r < 8; ++r) v[r] = load_in(io, tr + r * TR);
  const int n8 = lgN / 3, rem = lgN - 3 * n8;
  if (n8 == 1 && rem == 0) {   // 8 points
    pow2_pass<INV, 8, true, true>(v, A, io, buf, tr, 0, active, out_of<INV>(A, io));
    return;
  }
  int lgL = 0;
  for (int p = 0;; ++p) {
    const unsigned b = p == 0 ? pow2_pass<INV, 8, true, false>(v, A, io, buf, tr, lgL, active, OutScale{})
                              : pow2_pass<INV, 8, false, false>(v, A, io, buf, tr, lgL, active, OutScale{});
    row_or<SHORT>(&bits[p][lr], b);
    __syncthreads();   // the pass's outputs are in the buffer
    lgL += 3;
    const int s = shift_for(bits[p][lr]);
    io.ex += s + 1;    // the shift, and the next pass's halving products
    const int left = lgN - lgL;
    if (left >= 3) pow2_load<8>(v, buf, A.N, tr, s);
    else if (left == 2) pow2_load<4>(v, buf, A.N, tr, s);
    else pow2_load<2>(v, buf, A.N, tr, s);
    if (left <= 3) break;
    __syncthreads();   // the buffer is read in full before it is rewritten
  }
  const int left = lgN - lgL;
  const OutScale os = out_of<INV>(A, io);
  if (left == 3) pow2_pass<INV, 8, false, true>(v, A, io, buf, tr, lgL, active, os);
  else if (left == 2) pow2_pass<INV, 4, false, true>(v, A, io, buf, tr, lgL, active, os);
  else pow2_pass<INV, 2, false, true>(v, A, io, buf, tr, lgL, active, os);
}

// ---- other 7-smooth lengths: one row per CTA, passes between two shared row buffers ----
template <bool INV, int R, bool FIRST, bool LAST>
__device__ __forceinline__ unsigned mixed_pass(const FixArgs& A, const RowIO& io, const fx2* src, fx2* dst, int L, int s,
                                               const OutScale& os) {
  const int NR = A.N / R;
  const float invL = 1.0f / (float)L;
  unsigned bits = 0;
  for (int t = threadIdx.x; t < NR; t += blockDim.x) {
    // j = t / L, k = t mod L (t, L < 2^13: the float quotient is off by at most one)
    int j = (int)((float)t * invL);
    int k = t - j * L;
    if (k >= L) { ++j; k -= L; }
    if (k < 0) { --j; k += L; }
    fx2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = FIRST ? load_in(io, t + r * NR) : src[padded(t + r * NR)];
    if (!FIRST) shift_all(v, s);
    butterfly<INV, R, FIRST>(v, A.tw, L, k);
    const int base = j * L * R + k;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      if (LAST) {
        store_out<INV>(A, io, base + q * L, v[q], os);
      } else {
        dst[padded(base + q * L)] = v[q];
        bits |= mag_bits(v[q]);
      }
    }
  }
  return bits;
}

template <bool INV, bool FIRST, bool LAST>
__device__ __forceinline__ unsigned mixed_pass_r(int R, const FixArgs& A, const RowIO& io, const fx2* src, fx2* dst,
                                                 int L, int s, const OutScale& os) {
  switch (R) {
    case 2: return mixed_pass<INV, 2, FIRST, LAST>(A, io, src, dst, L, s, os);
    case 3: return mixed_pass<INV, 3, FIRST, LAST>(A, io, src, dst, L, s, os);
    case 4: return mixed_pass<INV, 4, FIRST, LAST>(A, io, src, dst, L, s, os);
    case 5: return mixed_pass<INV, 5, FIRST, LAST>(A, io, src, dst, L, s, os);
    case 7: return mixed_pass<INV, 7, FIRST, LAST>(A, io, src, dst, L, s, os);
    default: return mixed_pass<INV, 8, FIRST, LAST>(A, io, src, dst, L, s, os);
  }
}

template <bool INV, int T>
__global__ void __launch_bounds__(T, 1024 / T) k_fft_fix_rows(const __grid_constant__ FixArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ unsigned top, bits[kMaxRadixPasses];
  RowIO io = row_io(A, blockIdx.x);
  fx2* src = reinterpret_cast<fx2*>(smem_raw);
  fx2* dst = src + A.N + (A.N >> 3) + 1;
  if (threadIdx.x < kMaxRadixPasses) bits[threadIdx.x] = 0;
  if (threadIdx.x == 0) top = 0;
  __syncthreads();
  unsigned m = 0;
  for (int i = threadIdx.x; i < A.N; i += T) {
    const double2 u = io.a[i];
    m = max(m, max(abs_hi(u.x), abs_hi(u.y)));
    if (io.b) {
      const double2 w = io.b[i];
      m = max(m, max(abs_hi(w.x), abs_hi(w.y)));
    }
  }
  row_max<false>(&top, m);
  __syncthreads();
  set_scale(io, top);
  const int np = A.n_pass;   // two at least (the shortest length is 9 = 3 x 3)
  int R = (int)(A.radix & 15);
  unsigned b = mixed_pass_r<INV, true, false>(R, A, io, src, src, 1, 0, OutScale{});
  int L = R;
  for (int p = 1;; ++p) {
    row_or<false>(&bits[p - 1], b);
    __syncthreads();
    const int s = shift_for(bits[p - 1]);
    io.ex += s + 1;   // the shift, and this pass's halving products
    R = (int)((A.radix >> (4 * p)) & 15);
    if (p == np - 1) {
      mixed_pass_r<INV, false, true>(R, A, io, src, dst, L, s, out_of<INV>(A, io));
      return;
    }
    b = mixed_pass_r<INV, false, false>(R, A, io, src, dst, L, s, OutScale{});
    fx2* t = src;
    src = dst;
    dst = t;
    L *= R;
  }
}

// Twiddles (cos, sin) as 61-bit fractions in 31-bit halves.
__global__ void k_fix_twiddles(const double2* __restrict__ tw, int4* __restrict__ out, int N) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const long long c = llrint(tw[i].x * 0x1p61), s = llrint(tw[i].y * 0x1p61);
  out[i] = make_int4((int)(c >> 31), (int)(c & 0x7fffffff), (int)(s >> 31), (int)(s & 0x7fffffff));
}

size_t pow2_smem(int N, int T) { return (size_t)(T / (N >> 3)) * (N + (N >> 3)) * sizeof(fx2); }
size_t rows_smem(int N) { return 2 * ((size_t)N + (N >> 3) + 1) * sizeof(fx2); }

template <bool INV> pic_status configure() {
  PIC_CUDA(cudaFuncSetAttribute(k_fft_fix_pow2<INV, 256, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pow2_smem(2048, 256)));
  PIC_CUDA(cudaFuncSetAttribute(k_fft_fix_pow2<INV, 512, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pow2_smem(4096, 512)));
  PIC_CUDA(cudaFuncSetAttribute(k_fft_fix_pow2<INV, 1024, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pow2_smem(8192, 1024)));
  PIC_CUDA(cudaFuncSetAttribute(k_fft_fix_rows<INV, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rows_smem(4096)));
  PIC_CUDA(cudaFuncSetAttribute(k_fft_fix_rows<INV, 384>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rows_smem(4096)));
  return PIC_OK;
}

template <bool INV> void launch(Sim* s, const FixArgs& A) {
  const int N = A.N;
  if (fft_is_pow2(N)) {
    int lgN = 0;
    while ((1 << lgN) < N) ++lgN;
    const int T = N <= 2048 ? 256 : N >> 3;
    // few short rows: smaller CTAs, down to 64 threads, until there are two for each SM (512 and 768
    // rows of 256 points: 19.5 -> 18.2 and 25.7 -> 24.8 us; 32 threads give no more: a thread's own
    // chain of three passes over 8 points is what is left)
    int t = T;
    while (t > 64 && t > N >> 3 && (int64_t)A.rows * (N >> 3) < (int64_t)t * 2 * 152) t >>= 1;
    const int rpc = t / (N >> 3), grid = (A.rows + rpc - 1) / rpc;
    auto* k = N < 256    ? k_fft_fix_pow2<INV, 256, true>
              : T == 256 ? k_fft_fix_pow2<INV, 256, false>
              : T == 512 ? k_fft_fix_pow2<INV, 512, false>
                         : k_fft_fix_pow2<INV, 1024, false>;
    k<<<grid, t, pow2_smem(N, t), s->stream>>>(A, lgN);
  } else if (N <= 2048) {
    k_fft_fix_rows<INV, 256><<<A.rows, 256, rows_smem(N), s->stream>>>(A);
  } else {
    k_fft_fix_rows<INV, 384><<<A.rows, 384, rows_smem(N), s->stream>>>(A);
  }
}

// A combination coefficient as a power of i and an optional halving; false for any other value.
bool unit_coef(double re, double im, int* rot, int* half) {
  if ((re != 0.0) == (im != 0.0)) return false;
  const double v = re != 0.0 ? re : im, m = v < 0 ? -v : v;
  if (m != 1.0 && m != 0.5) return false;
  *rot = (re != 0.0 ? 0 : 1) + (v < 0 ? 2 : 0);
  *half = m == 0.5;
  return true;
}

}  // namespace

bool fft_fix_active(const Sim* s) {
  return s->cfg.precision == PIC_FP64 && s->blue_M == 0 && s->dht_path != PIC_DHT_F64_GEMM;
}

pic_status fft_fix_configure_device() {
  const pic_status st = configure<false>();
  return st != PIC_OK ? st : configure<true>();
}

pic_status launch_fft_fix_setup(Sim* s) {
  const int N = s->cfg.Nz;
  k_fix_twiddles<<<(N + 127) / 128, 128, 0, s->stream>>>(s->at<double2>(s->lay.twp), s->at<int4>(s->lay.twp_fx), N);
  PIC_LAUNCHED(s);
  return PIC_OK;
}

pic_status launch_fft_fix(Sim* s, const void* in, void* out, const RowCombine& rc, bool inverse) {
  FixArgs A{};
  A.in = static_cast<const double2*>(in);
  A.out = static_cast<double2*>(out);
  A.out_dw = static_cast<float4*>(rc.out_dw);
  A.tw = s->at<int4>(s->lay.twp_fx);
  A.N = s->cfg.Nz;
  A.rows_per_comp = s->cfg.Nm * s->cfg.Nr;
  A.rows = rc.n_out * A.rows_per_comp;
  for (int k = 0; k < rc.n_out; ++k) {
    int hb = 0;
    A.srcA[k] = rc.srcA[k];
    A.srcB[k] = rc.srcB[k];
    bool ok = unit_coef(rc.caRe[k], rc.caIm[k], &A.rotA[k], &A.half[k]);
    if (ok && rc.srcB[k] >= 0) ok = unit_coef(rc.cbRe[k], rc.cbIm[k], &A.rotB[k], &hb) && hb == A.half[k];
    if (!ok) {
      set_error("row FFT: combination %d is not of +-1, +-i or their halves", k);
      return PIC_ERR_ARG;
    }
  }
  A.n_pass = s->n_radix;
  for (int p = 0; p < s->n_radix; ++p) A.radix |= (unsigned long long)s->radix[p] << (4 * p);
  while ((1 << A.nc_exp) < A.N) ++A.nc_exp;
  if (inverse && !fft_is_pow2(A.N)) {   // 1/N = c 2^-nc_exp with c in (1, 2): keep c/2
    const __int128 c = (((__int128)1 << (62 + A.nc_exp - 1)) + A.N / 2) / A.N;
    A.nc_hi = (int)(c >> 31);
    A.nc_lo = (int)(c & 0x7fffffff);
    A.nc_exp -= 1;
  }
  if (inverse) launch<true>(s, A);
  else launch<false>(s, A);
  PIC_LAUNCHED(s);
  return PIC_OK;
}

}  // namespace pic
