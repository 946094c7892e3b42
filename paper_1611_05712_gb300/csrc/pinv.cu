// Pseudo-inverses of the Hankel matrices (a0; forward transforms M_p = pinv(B_p) with singular
// values <= 1e-3 sigma_max dropped), FP64, all 3 Nm matrices of a handle together.
//
// A Hankel matrix has at most a few singular values near or below the cut (B_{m-1} lacks the k = 0
// Dini function r^{m-1}; the others lie above about 3e-3), so its pseudo-inverse is the plain
// inverse with those directions taken out:
//   1. C = B^-1 by Gauss-Jordan elimination with row pivoting, one launch per column;
//   2. the four smallest singular values and right vectors V from subspace iteration with C C^T
//      (they are its largest), the largest singular value from subspace iteration with B B^T;
//   3. with V reduced to the dropped directions and U their left vectors (C^T V, orthonormal),
//      X = (I - V V^T) C (I - U U^T), after two refinements U <- U - B (X U), V <- V - X (B V): they
//      take the rounding of an inverse of condition up to 1e9 out of the directions;
//   4. one Newton-Schulz step X <- X (2I - B X).
// The result agrees with a singular value decomposition's to a few 1e-15 (a one-sided Jacobi
// SVD's, the fallback, to 6e-14).  The fallback is taken, for the whole handle, when a singular
// value lies within 5 % of the cut, when the four smallest may not hold all dropped ones, on a
// zero or non-finite pivot, and when step 4 still moves X by more than 1e-6.
// The SVD's rounds were bound by their latency (a launch per round of column pairs, each a dozen
// dependent float64 divisions and roots) and by the float64 unit (about 5.5 n^3 operations a
// sweep, 10 sweeps); here n launches carry n^3 operations in all.
#include <algorithm>

#include "pic_internal.cuh"

namespace pic {
namespace {

constexpr int kQ = 4;   // vectors of the subspace iterations

// ---- Gauss-Jordan ----
// Pivot candidates: |value| with its low 10 bits replaced by the row, so that atomicMax finds the
// row of the largest (to 2^-42); the order of ties does not depend on the order of the atomics.
__device__ __forceinline__ unsigned long long pivot_key(double v, int row) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  return (b & ~1023ull) | (unsigned)row;
}

__global__ void k_gj_init(const double* __restrict__ A, double* __restrict__ W, unsigned long long* piv, int n, int nmat) {
  const size_t total = (size_t)nmat * n * n;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const double v = A[i];
    W[i] = v;
    if (i % n == 0) {
      const size_t r = i / n;
      atomicMax(piv + r / n * n, pivot_key(v, (int)(r % n)));
    }
  }
}

// Step k: rows k and p (the pivot's) swapped, row k divided by the pivot, its multiples taken from
// the others, column k replaced by the inverse's (the swaps are undone on its columns at the
// end).  From src to dst, so that no element is read after it is written.  Tiles of 32 columns x
// 64 rows.
constexpr int kGjRows = 64;
__global__ void __launch_bounds__(256) k_gj_step(const double* __restrict__ src_all, double* __restrict__ dst_all,
                                                 unsigned long long* __restrict__ piv_all, int n, int k, int32_t* bad) {
  const double* src = src_all + (size_t)blockIdx.z * n * n;
  double* dst = dst_all + (size_t)blockIdx.z * n * n;
  unsigned long long* piv = piv_all + (size_t)blockIdx.z * n;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int j = blockIdx.x * 32 + tx, p = (int)(piv[k] & 1023ull);
  double pv = src[(size_t)p * n + k];
  if (!(fabs(pv) > 0.0) || !(fabs(pv) < 1e300)) {
    *bad = 1;
    pv = 1.0;
  }
  const double inv = 1.0 / pv;
  if (j >= n) return;
  const double r = (j == k ? 1.0 : src[(size_t)p * n + j]) * inv;
  unsigned long long best = 0;
#pragma unroll
  for (int u = 0; u < kGjRows / 8; ++u) {
    const int i = blockIdx.y * kGjRows + ty + 8 * u;
    if (i >= n) break;
    double v = r;
    if (i != k) {
      const size_t s = (size_t)(i == p ? k : i) * n;
      v = fma(-src[s + k], r, j == k ? 0.0 : src[s + j]);
    }
    dst[(size_t)i * n + j] = v;
    if (j == k + 1 && i > k) best = max(best, pivot_key(v, i));
  }
  if (best) atomicMax(piv + k + 1, best);
}

// X[i][perm] = W[i][j]: the row swaps undone, last first, on the inverse's columns.
__global__ void k_gj_columns(const double* __restrict__ W_all, double* __restrict__ X_all,
                             const unsigned long long* __restrict__ piv_all, int n) {
  extern __shared__ int col[];   // column of W that column j of X takes
  const double* W = W_all + (size_t)blockIdx.x * n * n;
  double* X = X_all + (size_t)blockIdx.x * n * n;
  for (int j = threadIdx.x; j < n; j += blockDim.x) col[j] = j;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = n - 1; k >= 0; --k) {
      const int p = (int)(piv_all[(size_t)blockIdx.x * n + k] & 1023ull);
      const int t = col[k];
      col[k] = col[p];
      col[p] = t;
    }
  __syncthreads();
  for (int i = blockIdx.y; i < n; i += gridDim.y)
    for (int j = threadIdx.x; j < n; j += blockDim.x) X[(size_t)i * n + j] = W[(size_t)i * n + col[j]];
}

// ---- products with kQ vectors ([matrix][kQ][n]) ----
__device__ __forceinline__ double warp_total(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// out = M in, one warp per row.
__global__ void __launch_bounds__(256) k_mv(const double* __restrict__ M, const double* __restrict__ in,
                                            double* __restrict__ out, int n) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= n) return;
  const double* row = M + ((size_t)blockIdx.y * n + i) * n;
  const double* x = in + (size_t)blockIdx.y * kQ * n;
  double a[kQ] = {0, 0, 0, 0};
  for (int j = lane; j < n; j += 32) {
    const double m = row[j];
#pragma unroll
    for (int q = 0; q < kQ; ++q) a[q] = fma(m, x[q * n + j], a[q]);
  }
#pragma unroll
  for (int q = 0; q < kQ; ++q) {
    const double t = warp_total(a[q]);
    if (lane == 0) out[((size_t)blockIdx.y * kQ + q) * n + i] = t;
  }
}

// out = M^T in: 32 columns per CTA, the rows split over its 8 warps.
__global__ void __launch_bounds__(256) k_mvt(const double* __restrict__ M_all, const double* __restrict__ in,
                                             double* __restrict__ out, int n) {
  __shared__ double part[8][kQ][32];
  const double* M = M_all + (size_t)blockIdx.y * n * n;
  const double* x = in + (size_t)blockIdx.y * kQ * n;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, j = blockIdx.x * 32 + lane;
  double a[kQ] = {0, 0, 0, 0};
  if (j < n)
    for (int i = w; i < n; i += 8) {
      const double m = M[(size_t)i * n + j];
#pragma unroll
      for (int q = 0; q < kQ; ++q) a[q] = fma(m, x[q * n + i], a[q]);
    }
#pragma unroll
  for (int q = 0; q < kQ; ++q) part[w][q][lane] = a[q];
  __syncthreads();
  if (w < kQ && j < n) {
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += part[k][w][lane];
    out[((size_t)blockIdx.y * kQ + w) * n + j] = t;
  }
}

// X -= sum_q l_q r_q^T.
__global__ void k_rank(double* __restrict__ X, const double* __restrict__ l, const double* __restrict__ r, int n) {
  const size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (e >= (size_t)n * n) return;
  const int i = (int)(e / n), j = (int)(e - (size_t)i * n);
  const double *L = l + (size_t)blockIdx.y * kQ * n, *R = r + (size_t)blockIdx.y * kQ * n;
  double v = X[(size_t)blockIdx.y * n * n + e];
#pragma unroll
  for (int q = 0; q < kQ; ++q) v = fma(-L[q * n + i], R[q * n + j], v);
  X[(size_t)blockIdx.y * n * n + e] = v;
}

__device__ __forceinline__ double warp_dot(const double* a, const double* b, int n) {
  double t = 0.0;
  for (int i = threadIdx.x; i < n; i += 32) t = fma(a[i], b[i], t);
  return warp_total(t);
}

// V <- orthonormal basis of V - S (S null: of V) by Gram-Schmidt, twice; a zero vector stays zero.
// One warp per matrix.
__global__ void __launch_bounds__(32) k_orth(double* __restrict__ V_all, const double* __restrict__ S, int n) {
  double* V = V_all + (size_t)blockIdx.x * kQ * n;
  if (S)
    for (int i = threadIdx.x; i < kQ * n; i += 32) V[i] -= S[(size_t)blockIdx.x * kQ * n + i];
  __syncwarp();
  for (int q = 0; q < kQ; ++q) {
    double* v = V + q * n;
    for (int pass = 0; pass < 2; ++pass) {
      for (int p = 0; p < q; ++p) {
        const double g = warp_dot(V + p * n, v, n);
        for (int i = threadIdx.x; i < n; i += 32) v[i] = fma(-g, V[p * n + i], v[i]);
        __syncwarp();
      }
      const double s = warp_dot(v, v, n);
      const double f = s > 0.0 ? 1.0 / sqrt(s) : 0.0;
      for (int i = threadIdx.x; i < n; i += 32) v[i] *= f;
      __syncwarp();
    }
  }
}

// Deterministic starting vectors without structure.
__global__ void k_start(double* V, int n, int total) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  unsigned h = (unsigned)(i % (kQ * n)) * 2654435761u + 12345u;
  h ^= h >> 15; h *= 2246822519u; h ^= h >> 13; h *= 3266489917u; h ^= h >> 16;
  V[i] = (double)h * 0x1p-31 - 1.0;
}

// One-sided Jacobi rotations of W = B V (columns) and V until W's columns are orthogonal: their
// norms are the singular values on the subspace, sig[matrix][kQ].  One warp per matrix.
__global__ void __launch_bounds__(32) k_ritz(double* W_all, double* V_all, double* sig, int n) {
  double *W = W_all + (size_t)blockIdx.x * kQ * n, *V = V_all + (size_t)blockIdx.x * kQ * n;
  for (int sweep = 0; sweep < 10; ++sweep) {
    bool rotated = false;
    for (int p = 0; p < kQ - 1; ++p)
      for (int q = p + 1; q < kQ; ++q) {
        const double a = warp_dot(W + p * n, W + p * n, n), b = warp_dot(W + q * n, W + q * n, n);
        const double g = warp_dot(W + p * n, W + q * n, n);
        if (!(fabs(g) > 1e-14 * sqrt(a * b))) continue;
        rotated = true;
        const double zeta = (b - a) / (2.0 * g);
        const double t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
        const double c = 1.0 / sqrt(1.0 + t * t), s = c * t;
        for (int i = threadIdx.x; i < n; i += 32) {
          const double x = W[p * n + i], y = W[q * n + i], u = V[p * n + i], v = V[q * n + i];
          W[p * n + i] = c * x - s * y;
          W[q * n + i] = s * x + c * y;
          V[p * n + i] = c * u - s * v;
          V[q * n + i] = s * u + c * v;
        }
        __syncwarp();
      }
    if (!rotated) break;
  }
  for (int q = 0; q < kQ; ++q) {
    const double s = sqrt(warp_dot(W + q * n, W + q * n, n));
    if (threadIdx.x == 0) sig[blockIdx.x * kQ + q] = s;
  }
}

// Vectors of kept singular values become zero.  The decision needs sigma_max (its estimate from
// below, large: within 2 %) times 1e-3 clear of every value, and the largest of the four above it.
__global__ void k_drop(double* V_all, const double* small, const double* large, int n, int32_t* bad) {
  double top = 0.0, most = 0.0;
  for (int q = 0; q < kQ; ++q) {
    top = fmax(top, large[blockIdx.x * kQ + q]);
    most = fmax(most, small[blockIdx.x * kQ + q]);
  }
  const double cut = kPinvRcond * top;
  for (int q = 0; q < kQ; ++q) {
    const double s = small[blockIdx.x * kQ + q];
    if (!(s < 0.95 * cut || s > 1.05 * cut) && threadIdx.x == 0) *bad = 1;
    if (s < cut) continue;
    for (int i = threadIdx.x; i < n; i += blockDim.x) V_all[((size_t)blockIdx.x * kQ + q) * n + i] = 0.0;
  }
  if (!(most > 1.05 * cut) && threadIdx.x == 0) *bad = 1;
}

// Newton-Schulz moved X by more than 1e-6 of its largest entry (or X is not finite): bad.
__global__ void __launch_bounds__(1024) k_moved(const double* __restrict__ X, const double* __restrict__ Y, int n, int32_t* bad) {
  __shared__ unsigned long long mx, md;
  if (threadIdx.x == 0) mx = md = 0;
  __syncthreads();
  const size_t off = (size_t)blockIdx.x * n * n;
  double x = 0.0, d = 0.0;
  bool nan = false;
  for (size_t e = threadIdx.x; e < (size_t)n * n; e += blockDim.x) {
    const double a = X[off + e], b = Y[off + e];
    nan = nan || !(fabs(b) < 1e300) || !(fabs(a) < 1e300);
    x = fmax(x, fabs(b));
    d = fmax(d, fabs(b - a));
  }
  atomicMax(&mx, (unsigned long long)__double_as_longlong(x));
  atomicMax(&md, (unsigned long long)__double_as_longlong(d));
  if (nan) *bad = 1;
  __syncthreads();
  if (threadIdx.x == 0 && !(__longlong_as_double((long long)md) <= 1e-6 * __longlong_as_double((long long)mx))) *bad = 1;
}

int blocks_for(size_t n, int t) { return (int)((n + t - 1) / t); }

}  // namespace

size_t pinv_scratch_bytes(const pic_config& c) {
  const size_t vec = (size_t)3 * c.Nm * kQ * c.Nr;
  return (4 * vec + 2 * 3 * c.Nm * kQ) * sizeof(double);
}

// mfwd <- X before the Newton-Schulz step; svd_w, svd_v and svd_d are scratch, *bad is raised as
// described above.
pic_status launch_pinv(Sim* s, int32_t* bad) {
  const int n = s->cfg.Nr, nmat = 3 * s->cfg.Nm;
  const double* B = s->at<double>(s->lay.binv);
  double* X = s->at<double>(s->lay.mfwd);
  double *w0 = s->at<double>(s->lay.svd_w), *w1 = s->at<double>(s->lay.svd_v);
  unsigned long long* piv = s->at<unsigned long long>(s->lay.svd_d);
  const size_t vec = (size_t)nmat * kQ * n;
  double *V = s->at<double>(s->lay.pinv), *U = V + vec, *T = U + vec, *Y = T + vec;
  double *sig_small = Y + vec, *sig_large = sig_small + nmat * kQ;
  cudaStream_t st = s->stream;
  PIC_CUDA(cudaMemsetAsync(piv, 0, (size_t)nmat * n * sizeof(unsigned long long), st));
  k_gj_init<<<std::min(blocks_for((size_t)nmat * n * n, 256), 152 * 16), 256, 0, st>>>(B, w0, piv, n, nmat);
  PIC_LAUNCHED(s);
  const dim3 ggj(blocks_for(n, 32), blocks_for(n, kGjRows), nmat);
  for (int k = 0; k < n; ++k) {
    k_gj_step<<<ggj, 256, 0, st>>>(w0, w1, piv, n, k, bad);
    PIC_LAUNCHED(s);
    std::swap(w0, w1);
  }
  k_gj_columns<<<dim3(nmat, 16), 256, n * sizeof(int), st>>>(w0, X, piv, n);
  PIC_LAUNCHED(s);
  const dim3 gmv(blocks_for((size_t)n * 32, 256), nmat), gmt(blocks_for(n, 32), nmat), grk(blocks_for((size_t)n * n, 256), nmat);
  auto mv = [&](const double* M, const double* in, double* out) -> pic_status {
    k_mv<<<gmv, 256, 0, st>>>(M, in, out, n);
    PIC_LAUNCHED(s);
    return PIC_OK;
  };
  auto mvt = [&](const double* M, const double* in, double* out) -> pic_status {
    k_mvt<<<gmt, 256, 0, st>>>(M, in, out, n);
    PIC_LAUNCHED(s);
    return PIC_OK;
  };
  auto orth = [&](double* v, const double* minus) -> pic_status {
    k_orth<<<nmat, 32, 0, st>>>(v, minus, n);
    PIC_LAUNCHED(s);
    return PIC_OK;
  };
  auto rank = [&](const double* l, const double* r) -> pic_status {   // X -= l r^T
    k_rank<<<grk, 256, 0, st>>>(X, l, r, n);
    PIC_LAUNCHED(s);
    return PIC_OK;
  };
  auto start = [&](double* v) -> pic_status {
    k_start<<<blocks_for(vec, 256), 256, 0, st>>>(v, n, (int)vec);
    PIC_LAUNCHED(s);
    return orth(v, nullptr);
  };
#define PIC_TRY(call) do { if (const pic_status e__ = (call)) return e__; } while (0)
  // the largest singular value (Y: left vectors of B, T = B^T Y)
  PIC_TRY(start(Y));
  for (int it = 0; it < 10; ++it) {
    PIC_TRY(mvt(B, Y, T));
    PIC_TRY(mv(B, T, Y));
    PIC_TRY(orth(Y, nullptr));
  }
  PIC_TRY(mvt(B, Y, T));
  k_ritz<<<nmat, 32, 0, st>>>(T, Y, sig_large, n);
  PIC_LAUNCHED(s);
  // the smallest ones (V: right vectors of B)
  PIC_TRY(start(V));
  for (int it = 0; it < 5; ++it) {
    PIC_TRY(mvt(X, V, T));
    PIC_TRY(mv(X, T, V));
    PIC_TRY(orth(V, nullptr));
  }
  PIC_TRY(mv(B, V, T));
  k_ritz<<<nmat, 32, 0, st>>>(T, V, sig_small, n);
  PIC_LAUNCHED(s);
  k_drop<<<nmat, 256, 0, st>>>(V, sig_small, sig_large, n, bad);
  PIC_LAUNCHED(s);
  // X = (I - V V^T) C (I - U U^T), U = orth(C^T V)
  PIC_TRY(mvt(X, V, U));
  PIC_TRY(rank(V, U));
  PIC_TRY(orth(U, nullptr));
  PIC_TRY(mv(X, U, T));
  PIC_TRY(rank(T, U));
  for (int it = 0; it < 2; ++it) {
    PIC_TRY(mv(X, U, T));
    PIC_TRY(mv(B, T, Y));
    PIC_TRY(orth(U, Y));
    PIC_TRY(mv(X, U, T));
    PIC_TRY(rank(T, U));
    PIC_TRY(mv(B, V, T));
    PIC_TRY(mv(X, T, Y));
    PIC_TRY(orth(V, Y));
    PIC_TRY(mvt(X, V, T));
    PIC_TRY(rank(V, T));
  }
#undef PIC_TRY
  return PIC_OK;
}

pic_status launch_pinv_check(Sim* s, const double* before, const double* after, int32_t* bad) {
  k_moved<<<3 * s->cfg.Nm, 1024, 0, s->stream>>>(before, after, s->cfg.Nr, bad);
  PIC_LAUNCHED(s);
  return PIC_OK;
}

}  // namespace pic
