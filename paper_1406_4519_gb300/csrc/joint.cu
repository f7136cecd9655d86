// joint.cu -- joint matrix completion and tensor factorization (Appendix F).
//
// A ratings matrix Y (users x items, observed entries Omega^Y) and the user x
// item x word tensor X share the user factor A and the item factor B:
//   f = 1/2 sum_{(i,j) in Omega^Y} (y_ij - a_i . b_j)^2 + mu 1/2 ||X - [[A,B,C]]||^2
//       + lambda 1/2 (||A||^2 + ||B||^2 + ||C||^2)                (Eq. joint-obj-fn)
// with lambda the handle's lambda_reg.  Every row of A has the system of
// Eq. grad-joint-A:
//   rhs_i = sum_{j in Omega_i} y_ij b_j + mu N_A[i],   N_A = X^1 (C kr B) (MTTKRP)
//   H_i   = sum_{j in Omega_i} b_j^T b_j + mu (C^T C * B^T B) + lambda I
// (B the same with the roles of A and B swapped; C with no ratings).  ALS sets
// a_i = rhs_i H_i^-1 row by row; GD takes grad_i = -rhs_i + a_i H_i for every
// row at the current point and searches along the ray.  The X^1 (C kr B) term
// is the library's MTTKRP (Algorithm 1), as the appendix says.
//
// The ratings are kept as two CSR copies (by user and by item), sorted with
// the library's radix sort: both kernels walk a row's ratings in ascending
// column order, so every sum has a fixed order.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <new>

#include "../../include/dfacto.h"
#include "device.cuh"
#include "internal.h"

namespace dfacto {

struct JointState {
  double mu = 0.0;
  int64_t nnzY = 0;
  int64_t* ptr[2] = {nullptr, nullptr};  // [dims[side] + 1]
  int32_t* col[2] = {nullptr, nullptr};  // [nnzY]: item (side 0) or user (side 1)
  float* val[2] = {nullptr, nullptr};    // [nnzY]
  double* base = nullptr;                // [R x R] mu Gamma + lambda I
  float* gam32 = nullptr;                // [R x R] Gamma
  double* ycoef = nullptr;               // [5] ratings quartic along the ray
  bool heavy[2] = {false, false};        // a row has more than kHeavyRatings ratings
  unsigned char* slots = nullptr;        // heavy rows' pieces, two per chunk of ratings (lazy)
  double* part = nullptr;                // block partials
  int64_t part_cap = 0;                  // doubles
};

namespace {

constexpr int kJT = 256;       // threads of the gradient and quartic kernels
constexpr int kJMaxBlocks = 152 * 8;

unsigned jgrid(int64_t rows, int warps) {
  const int64_t b = (rows + warps - 1) / warps;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, kJMaxBlocks));
}

__global__ void ratings_in_range(const int32_t* __restrict__ yidx, int64_t n, int32_t I, int32_t J,
                                 int32_t* __restrict__ flag) {
  bool bad = false;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride) {
    const int32_t i = yidx[t], j = yidx[n + t];
    bad |= (i < 0) | (i >= I) | (j < 0) | (j >= J);
  }
  if (__any_sync(kFull, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, 1);
}

// key = (row << bits_col) | col for the CSR of `side` (row = user for side 0).
__global__ void rating_keys(const int32_t* __restrict__ yidx, int64_t n, int side, int bits_col,
                            uint64_t* __restrict__ key, uint32_t* __restrict__ perm) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride) {
    const uint64_t row = (uint32_t)yidx[(int64_t)side * n + t];
    const uint64_t col = (uint32_t)yidx[(int64_t)(1 - side) * n + t];
    key[t] = (row << bits_col) | col;
    perm[t] = (uint32_t)t;
  }
}

__global__ void rating_scatter(const uint64_t* __restrict__ key, const uint32_t* __restrict__ perm,
                               const float* __restrict__ yval, int64_t n, int bits_col,
                               int32_t* __restrict__ col, float* __restrict__ val,
                               int32_t* __restrict__ dup) {
  const uint64_t mask = (uint64_t(1) << bits_col) - 1;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  bool d = false;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += stride) {
    col[t] = (int32_t)(key[t] & mask);
    val[t] = yval[perm[t]];
    d |= t > 0 && key[t] == key[t - 1];
  }
  if (__any_sync(kFull, d) && (threadIdx.x & 31) == 0) atomicOr(dup, 1);
}

// ptr[r] = first position whose row is >= r.
__global__ void rating_ptr(const uint64_t* __restrict__ key, int64_t n, int64_t rows, int bits_col,
                           int64_t* __restrict__ ptr) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r <= rows; r += stride) {
    const uint64_t k = (uint64_t)r << bits_col;
    int64_t lo = 0, hi = n;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (key[mid] < k) lo = mid + 1; else hi = mid;
    }
    ptr[r] = lo;
  }
}

__global__ void fill_ones(double* p, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) p[i] = 1.0;
}

// base = mu (Gf * Gi) + lambda I (FP64) and Gamma = Gf * Gi (FP32).
__global__ void joint_base(const double* __restrict__ Gf, const double* __restrict__ Gi, int R,
                           double mu, double lambda, double* __restrict__ base,
                           float* __restrict__ gam32) {
  for (int e = threadIdx.x; e < R * R; e += blockDim.x) {
    const double g = Gf[e] * Gi[e];
    base[e] = mu * g + (e / R == e % R ? lambda : 0.0);
    gam32[e] = (float)g;
  }
}

__device__ __forceinline__ float ld_f(const float* p) { return *p; }
__device__ __forceinline__ float ld_f(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// ---------------------------------------------------------------------------
// ALS row update: F[row] = rhs H^-1 with H = base + sum over the row's ratings
// of v^T v and rhs = mu N[row] + sum of y v (H is positive definite for
// lambda > 0).  A block takes 32 rows: its warps form the 32 systems (ratings
// Grams in FP32 registers over at most kHeavyRatings ratings, everything above
// in FP64), then one warp solves them, a thread per system, so that every FP64
// instruction serves 32 rows (this GPU retires two FP64 lanes per clock and SM:
// the FP64 pipe bounds the solves, about R^3 / 6 + R^2 lane operations a row; a
// warp per row left most lanes of them idle).
//
// A row with more ratings (one user of a power-law rating matrix holds tens of
// thousands) would be one warp's serial chain, so such rows are cut: the ratings
// are chunks of kHeavyRatings positions, and joint_heavy leaves, per chunk, the
// Gram and right side of the piece of a heavy row that begins before the chunk
// or at its start (slot 0) and of one that begins inside it and runs past its
// end (slot 1); the row's block adds its pieces in order.
//
// 100,000 users x 50,000 items x 20,000 words, 2M ratings, R = 16: 63.4 ms per
// sweep with a warp per row (most of it one user's ratings), 2.2 ms now (3.0 with
// pieces of 1,024: the rows just below that length share a few blocks).
// ---------------------------------------------------------------------------
constexpr int kHeavyRatings = 256;
constexpr int kJTileLd = 33;  // rows of a block, padded

// RP: R padded to 8, 16 or 32 columns.  Lane (i, h), i = lane % RP, h = lane /
// RP, holds H[i][h CPL .. + CPL).
template <int RP>
struct JShape {
  static constexpr int CG = 32 / RP;   // lane groups
  static constexpr int CPL = RP / CG;  // columns per lane
  static constexpr int LD = RP + 4;    // floats of a staged row
};
constexpr int kJSolveWarps = 8;

__host__ __device__ constexpr int jtri(int R) { return R * (R + 1) / 2; }
// Bytes of a chunk slot: the lower triangle in FP32, the right side in FP64.
__host__ __device__ constexpr size_t jslot_bytes(int R) {
  return (sizeof(float) * jtri(R) + 7) / 8 * 8 + sizeof(double) * R;
}

// Gram and right side of ratings [p0, p1) over the rows of `other`, by one
// warp; the ratings are staged 32 at a time in `tile` ([32][LD] floats, the
// warp's own).  rhs is complete in every lane of column i.
template <typename T, int RP>
__device__ __forceinline__ void joint_accumulate(const int32_t* __restrict__ ycol,
                                                 const float* __restrict__ yval,
                                                 const T* __restrict__ other, int64_t p0, int64_t p1,
                                                 int R, float* tile, float (&hrow)[JShape<RP>::CPL],
                                                 double& rhs) {
  using S = JShape<RP>;
  const int lane = threadIdx.x & 31, i = lane % RP, h = lane / RP;
#pragma unroll
  for (int c = 0; c < S::CPL; ++c) hrow[c] = 0.f;
  rhs = 0.0;
  int o_n = p0 + lane < p1 ? ycol[p0 + lane] : 0;
  float y_n = p0 + lane < p1 ? yval[p0 + lane] : 0.f;
  for (int64_t p = p0; p < p1; p += 32) {
    const int n = (int)min((int64_t)32, p1 - p);
    const int o = o_n;
    const float y = y_n;
    if (p + 32 + lane < p1) {  // the next 32 ratings
      o_n = ycol[p + 32 + lane];
      y_n = yval[p + 32 + lane];
    }
    __syncwarp();  // the tile's last use is over
#pragma unroll 8
    for (int k = 0; k < 32 / S::CG; ++k) {
      const int t = k * S::CG + h;
      const int ot = __shfl_sync(kFull, o, t);
      tile[t * S::LD + i] = (t < n && i < R) ? ld_f(other + (int64_t)ot * R + i) : 0.f;
    }
    __syncwarp();
    for (int t = 0; t < n; ++t) {
      const float vi = tile[t * S::LD + i];
      float w[S::CPL];
      const float* q = tile + t * S::LD + h * S::CPL;
      if constexpr (S::CPL % 4 == 0) {
#pragma unroll
        for (int c = 0; c < S::CPL; c += 4) {
          const float4 f = *reinterpret_cast<const float4*>(q + c);
          w[c] = f.x; w[c + 1] = f.y; w[c + 2] = f.z; w[c + 3] = f.w;
        }
      } else {
#pragma unroll
        for (int c = 0; c < S::CPL; ++c) w[c] = q[c];
      }
#pragma unroll
      for (int c = 0; c < S::CPL; ++c) hrow[c] = fmaf(vi, w[c], hrow[c]);
    }
    // the groups take every CG-th rating of the right side (conversions run on
    // the FP64 pipe too: y is converted once, a rating per lane)
    const double yd = y;
    for (int t0 = 0; t0 < n; t0 += S::CG) {
      const int t = t0 + h;  // < 32
      const double yt = __shfl_sync(kFull, yd, t);
      if (t < n) rhs += yt * (double)tile[t * S::LD + i];
    }
  }
#pragma unroll
  for (int d = RP; d < 32; d <<= 1) rhs += __shfl_xor_sync(kFull, rhs, d);
}

// Row of rating position p: the largest r with ptr[r] <= p (and a rating).
__device__ __forceinline__ int64_t rating_row(const int64_t* __restrict__ ptr, int64_t rows, int64_t p) {
  int64_t lo = 0, hi = rows - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (ptr[mid] <= p) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__global__ void any_heavy(const int64_t* __restrict__ ptr, int64_t rows, int32_t* __restrict__ flag) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  bool any = false;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += stride)
    any |= ptr[r + 1] - ptr[r] > kHeavyRatings;
  if (__any_sync(kFull, any) && (threadIdx.x & 31) == 0) atomicOr(flag, 1);
}

// Pieces of heavy rows, one warp per chunk of kHeavyRatings ratings.
template <typename T, int RP>
__global__ void __launch_bounds__(kJSolveWarps * 32) joint_heavy(
    const int64_t* __restrict__ yptr, const int32_t* __restrict__ ycol,
    const float* __restrict__ yval, const T* __restrict__ other, int64_t rows, int64_t nnzY, int R,
    unsigned char* __restrict__ slots) {
  using S = JShape<RP>;
  __shared__ __align__(16) float tiles[kJSolveWarps][32 * S::LD];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = lane % RP, h = lane / RP;
  const int64_t chunk = (int64_t)blockIdx.x * kJSolveWarps + warp;
  const int64_t c0 = chunk * kHeavyRatings, c1 = min(c0 + kHeavyRatings, nnzY);
  if (c0 >= nnzY) return;
  const int64_t r0 = rating_row(yptr, rows, c0), r1 = rating_row(yptr, rows, c1 - 1);
  for (int slot = 0; slot < 2; ++slot) {
    const int64_t r = slot == 0 ? r0 : r1;
    const int64_t b = yptr[r], e = yptr[r + 1];
    if ((slot == 1 && r1 == r0) || e - b <= kHeavyRatings) continue;
    float hrow[S::CPL];
    double rhs;
    joint_accumulate<T, RP>(ycol, yval, other, max(b, c0), min(e, c1), R, tiles[warp], hrow, rhs);
    unsigned char* out = slots + (2 * chunk + slot) * jslot_bytes(R);
    float* tri = reinterpret_cast<float*>(out);
    double* rs = reinterpret_cast<double*>(out + jslot_bytes(R) - sizeof(double) * R);
#pragma unroll
    for (int c = 0; c < S::CPL; ++c) {
      const int j = h * S::CPL + c;
      if (i < R && j <= i) tri[jtri(i) + j] = hrow[c];
    }
    if (h == 0 && i < R) rs[i] = rhs;
  }
}

// The pieces of the heavy row with ratings [b, e), added in order: entry (ti, tj)
// of the lower triangle to tri(ti, tj, sum) and entry ti of the right side to
// rhs(ti, sum), a thread per entry (thread t of n).
template <class Tri, class Rhs>
__device__ __forceinline__ void add_pieces(const unsigned char* __restrict__ slots, int64_t b, int64_t e, int R,
                                           int t0, int n, Tri&& tri, Rhs&& rhs) {
  const int64_t k0 = b / kHeavyRatings, np = (e - 1) / kHeavyRatings - k0;
  const unsigned char* p0 = slots + (2 * k0 + (b % kHeavyRatings ? 1 : 0)) * jslot_bytes(R);
  const unsigned char* pk = slots + 2 * (k0 + 1) * jslot_bytes(R);  // the pieces after the first
  const size_t step = 2 * jslot_bytes(R);
  for (int t = t0; t < jtri(R) + R; t += n) {
    if (t < jtri(R)) {
      int ti = 0;
      while (jtri(ti + 1) <= t) ++ti;
      double a = (double)reinterpret_cast<const float*>(p0)[t];
#pragma unroll 8
      for (int64_t k = 0; k < np; ++k) a += (double)reinterpret_cast<const float*>(pk + k * step)[t];
      tri(ti, t - jtri(ti), a);
    } else {
      const int ti = t - jtri(R);
      const size_t at = jslot_bytes(R) - sizeof(double) * (R - ti);
      double a = *reinterpret_cast<const double*>(p0 + at);
#pragma unroll 8
      for (int64_t k = 0; k < np; ++k) a += *reinterpret_cast<const double*>(pk + k * step + at);
      rhs(ti, a);
    }
  }
}

// The systems of 32 rows and their solutions.  Shared memory: the lower
// triangles [entry][row] and right sides [column][row] in FP64 (rows padded to
// kJTileLd: conflict-free by entry and by row), and a staging tile per warp.
template <typename T, int RP>
__global__ void __launch_bounds__(kJSolveWarps * 32) joint_solve(
    const int64_t* __restrict__ yptr, const int32_t* __restrict__ ycol,
    const float* __restrict__ yval, const T* __restrict__ other, const float* __restrict__ N,
    const double* __restrict__ base, double mu, int64_t rows, int R,
    const unsigned char* __restrict__ slots, T* __restrict__ F, int32_t* __restrict__ bad_flag) {
  using S = JShape<RP>;
  extern __shared__ __align__(16) double jsm[];
  double* Hs = jsm;                              // [jtri(R)][kJTileLd]
  double* xs = Hs + (size_t)jtri(R) * kJTileLd;  // [R][kJTileLd]
  float* tiles = reinterpret_cast<float*>(jsm + (((size_t)(jtri(R) + R) * kJTileLd + 1) & ~(size_t)1));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = lane % RP, h = lane / RP;
  const int64_t ntiles = (rows + 31) / 32;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    // rows tile, tile + ntiles, ...: neighbouring rows, which rate alike where
    // labels are ordered by use, go to different blocks
    const int nr = (int)((rows - tile + ntiles - 1) / ntiles);  // <= 32
    for (int rr = warp; rr < nr; rr += kJSolveWarps) {
      const int64_t row = tile + rr * ntiles;
      const int64_t b = yptr ? yptr[row] : 0, e = yptr ? yptr[row + 1] : 0;
      if (e - b > kHeavyRatings) continue;  // below, by the whole block
      float hrow[S::CPL];
      double rhs;
      joint_accumulate<T, RP>(ycol, yval, other, b, e, R, tiles + (size_t)warp * 32 * S::LD, hrow, rhs);
#pragma unroll
      for (int c = 0; c < S::CPL; ++c) {
        const int j = h * S::CPL + c;
        if (i < R && j <= i) Hs[(jtri(i) + j) * kJTileLd + rr] = base[i * R + j] + (double)hrow[c];
      }
      if (h == 0 && i < R) xs[i * kJTileLd + rr] = mu * (double)N[row * R + i] + rhs;
    }
    if (slots && yptr) {
      const int64_t own = tile + lane * ntiles;
      unsigned heavy = __ballot_sync(kFull, lane < nr && yptr[own + 1] - yptr[own] > kHeavyRatings);
      for (; heavy; heavy &= heavy - 1u) {
        const int rr = __ffs(heavy) - 1;
        const int64_t row = tile + rr * ntiles;
        const int64_t b = yptr[row], e = yptr[row + 1];
        add_pieces(slots, b, e, R, threadIdx.x, kJSolveWarps * 32,
                   [&](int ti, int tj, double a) { Hs[(jtri(ti) + tj) * kJTileLd + rr] = base[ti * R + tj] + a; },
                   [&](int ti, double a) { xs[ti * kJTileLd + rr] = mu * (double)N[row * R + ti] + a; });
      }
    }
    __syncthreads();
    if (warp == 0 && lane < nr) {
      // Cholesky H = L L^T row by row below the diagonal, then L L^T x = rhs;
      // the diagonal holds 1 / L[j][j].
      double* H = Hs + lane;
      double* x = xs + lane;
      bool bad = false;
      for (int j = 0; j < R; ++j) {
        const int rj = jtri(j);
        double d = H[(rj + j) * kJTileLd];
        for (int k = 0; k < j; ++k) {
          const double l = H[(rj + k) * kJTileLd];
          d -= l * l;
        }
        bad |= !(d > 0.0);
        const double inv = rsqrt(fmax(d, 1e-300));
        H[(rj + j) * kJTileLd] = inv;
        int m = j + 1;
        for (; m + 4 <= R; m += 4) {  // four rows at a time (independent chains)
          const int a0 = jtri(m), a1 = jtri(m + 1), a2 = jtri(m + 2), a3 = jtri(m + 3);
          double s0 = H[(a0 + j) * kJTileLd], s1 = H[(a1 + j) * kJTileLd], s2 = H[(a2 + j) * kJTileLd],
                 s3 = H[(a3 + j) * kJTileLd];
#pragma unroll 2
          for (int k = 0; k < j; ++k) {
            const double l = H[(rj + k) * kJTileLd];
            s0 -= l * H[(a0 + k) * kJTileLd];
            s1 -= l * H[(a1 + k) * kJTileLd];
            s2 -= l * H[(a2 + k) * kJTileLd];
            s3 -= l * H[(a3 + k) * kJTileLd];
          }
          H[(a0 + j) * kJTileLd] = s0 * inv;
          H[(a1 + j) * kJTileLd] = s1 * inv;
          H[(a2 + j) * kJTileLd] = s2 * inv;
          H[(a3 + j) * kJTileLd] = s3 * inv;
        }
        for (; m < R; ++m) {
          const int a0 = jtri(m);
          double s0 = H[(a0 + j) * kJTileLd];
          for (int k = 0; k < j; ++k) s0 -= H[(rj + k) * kJTileLd] * H[(a0 + k) * kJTileLd];
          H[(a0 + j) * kJTileLd] = s0 * inv;
        }
      }
      for (int r = 0; r < R; ++r) {
        double s0 = x[r * kJTileLd];
        for (int k = 0; k < r; ++k) s0 -= H[(jtri(r) + k) * kJTileLd] * x[k * kJTileLd];
        x[r * kJTileLd] = s0 * H[(jtri(r) + r) * kJTileLd];
      }
      for (int r = R - 1; r >= 0; --r) {
        double s0 = x[r * kJTileLd];
        for (int k = r + 1; k < R; ++k) s0 -= H[(jtri(k) + r) * kJTileLd] * x[k * kJTileLd];
        x[r * kJTileLd] = s0 * H[(jtri(r) + r) * kJTileLd];
      }
      if (bad) atomicOr(bad_flag, 1);
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nr * R; t += kJSolveWarps * 32)
      st_elem(F + (tile + (t / R) * ntiles) * R + t % R, (float)xs[(t % R) * kJTileLd + t / R]);
    __syncthreads();  // before the next 32 rows
  }
}

// The same for a side of few rows: a warp per row, lane m on row m of its system
// (R <= 32).  An FP64 instruction serves one row here, but the chain of a row is
// R^2 / 2 of them, not R^3 / 6, which is what counts where the SMs have a block or
// less each.
template <typename T, int RP>
__global__ void __launch_bounds__(kJSolveWarps * 32) joint_solve_few(
    const int64_t* __restrict__ yptr, const int32_t* __restrict__ ycol,
    const float* __restrict__ yval, const T* __restrict__ other, const float* __restrict__ N,
    const double* __restrict__ base, double mu, int64_t rows, int R,
    const unsigned char* __restrict__ slots, T* __restrict__ F, int32_t* __restrict__ bad_flag) {
  using S = JShape<RP>;
  extern __shared__ __align__(16) double jsm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = lane % RP, h = lane / RP;
  const int LD = R + 1, own = R * LD + R;
  // per warp: the lower triangle [R][LD] and the right side [R]; then the tiles
  double* H = jsm + (size_t)warp * own;
  double* x = H + (size_t)R * LD;
  float* tile = reinterpret_cast<float*>(jsm + ((size_t)kJSolveWarps * own + 1) / 2 * 2) + (size_t)warp * 32 * S::LD;
  const int64_t row0 = (int64_t)blockIdx.x * kJSolveWarps, row = row0 + warp;
  if (row < rows) {
    const int64_t b = yptr ? yptr[row] : 0, e = yptr ? yptr[row + 1] : 0;
    if (e - b <= kHeavyRatings) {
      float hrow[S::CPL];
      double rhs;
      joint_accumulate<T, RP>(ycol, yval, other, b, e, R, tile, hrow, rhs);
#pragma unroll
      for (int c = 0; c < S::CPL; ++c) {
        const int j = h * S::CPL + c;
        if (i < R && j <= i) H[i * LD + j] = base[i * R + j] + (double)hrow[c];
      }
      if (h == 0 && i < R) x[i] = mu * (double)N[row * R + i] + rhs;
    }
  }
  if (slots && yptr) {  // heavy rows, by the whole block
    for (int w = 0; w < kJSolveWarps && row0 + w < rows; ++w) {
      const int64_t r = row0 + w, b = yptr[r], e = yptr[r + 1];
      if (e - b <= kHeavyRatings) continue;
      double* Hw = jsm + (size_t)w * own;
      add_pieces(slots, b, e, R, threadIdx.x, kJSolveWarps * 32,
                 [&](int ti, int tj, double a) { Hw[ti * LD + tj] = base[ti * R + tj] + a; },
                 [&](int ti, double a) { Hw[R * LD + ti] = mu * (double)N[r * R + ti] + a; });
    }
    __syncthreads();
  }
  __syncwarp();
  if (row >= rows) return;
  bool bad = false;
  double xl = lane < R ? x[lane] : 0.0, inv_own = 0.0;
  for (int k = 0; k < R; ++k) {  // column k of L below the diagonal, then L y = rhs as it goes
    const double d = H[k * LD + k];
    bad |= !(d > 0.0);
    const double inv = rsqrt(fmax(d, 1e-300));
    double lk = 0.0;
    if (lane > k && lane < R) {
      lk = H[lane * LD + k] * inv;
      H[lane * LD + k] = lk;
    }
    if (lane == k) inv_own = inv;
    const double yk = __shfl_sync(kFull, xl, k) * inv;
    if (lane == k) xl = yk;
    else if (lane > k) xl -= lk * yk;
    __syncwarp();
    if (lane > k && lane < R)
      for (int m = k + 1; m <= lane; ++m) H[lane * LD + m] -= lk * H[m * LD + k];
    __syncwarp();
  }
  for (int k = R - 1; k >= 0; --k) {  // L^T x = y
    const double xk = __shfl_sync(kFull, xl * inv_own, k);
    if (lane == k) xl = xk;
    else if (lane < k) xl -= H[k * LD + lane] * xk;
  }
  if (lane < R) st_elem(F + row * R + lane, (float)xl);
  if (bad && lane == 0) atomicOr(bad_flag, 1);
}

template <int RP>
size_t joint_few_smem(int R) {
  return sizeof(double) * (((size_t)kJSolveWarps * (R * (R + 1) + R) + 1) / 2 * 2) +
         sizeof(float) * kJSolveWarps * 32 * JShape<RP>::LD;
}

// Which row solver: a warp per row while that is at most a block per SM, and above
// R = 28, where joint_solve's systems leave room for one block per SM.  A sweep
// with 8 ratings per row, warp per row against 32 rows per block: 1,000 rows per
// side 304 and 413 us at R = 16, 397 and 750 at R = 24 (a warp per row without
// these kernels 577 and 717); 2,500 rows 461 and 420, 763 and 752; 50,000 rows
// 3.54 and 1.17 ms at R = 16, 8.35 and 8.36 at R = 28, 9.86 and 11.46 at R = 32.
bool few_rows(int64_t rows, int R) { return rows <= 152 * kJSolveWarps || R > 28; }

template <int RP>
size_t joint_solve_smem(int R) {
  return sizeof(double) * (((size_t)(jtri(R) + R) * kJTileLd + 1) & ~(size_t)1) +
         sizeof(float) * kJSolveWarps * 32 * JShape<RP>::LD;
}

__device__ __forceinline__ float wsum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Block sum of per-thread doubles in a fixed order (into thread 0).
__device__ __forceinline__ double jblock_sum(double v, double* s) {
  s[threadIdx.x] = v;
  __syncthreads();
  for (int w = kJT / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
    __syncthreads();
  }
  const double t = s[0];
  __syncthreads();
  return t;
}

// GD gradient rows (Eq. grad-joint-A), one warp per row, lane l on column l:
//   g = mu (-N[row] + F[row] Gamma) + lambda F[row]
//       + sum over the row's ratings of (F[row] . v - y) v
// with per-block partials of ||g||^2, <g, N>, <F, N> (part[block][3]).
template <typename T>
__global__ void __launch_bounds__(kJT) joint_grad(
    const int64_t* __restrict__ yptr, const int32_t* __restrict__ ycol,
    const float* __restrict__ yval, const T* __restrict__ other, const float* __restrict__ N,
    const float* __restrict__ gam32, double mu, double lambda, int64_t rows, int R,
    const T* __restrict__ F, float* __restrict__ grad, double* __restrict__ part) {
  __shared__ float sg[32 * 32];
  __shared__ double red[kJT];
  for (int e = threadIdx.x; e < R * R; e += blockDim.x) sg[e] = gam32[e];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int W = kJT / 32;
  const int64_t nw = (int64_t)gridDim.x * W;
  double a_g2 = 0.0, a_gn = 0.0, a_fn = 0.0;
  for (int64_t row = (int64_t)blockIdx.x * W + warp; row < rows; row += nw) {
    const float f = lane < R ? ld_f(F + row * R + lane) : 0.f;
    const float n = lane < R ? N[row * R + lane] : 0.f;
    float fg = 0.f;
    for (int m = 0; m < R; ++m) {
      const float fm = __shfl_sync(kFull, f, m);
      if (lane < R) fg = fmaf(fm, sg[m * R + lane], fg);
    }
    float g = (float)(mu * (double)(fg - n) + lambda * (double)f);
    if (yptr) {
      const int64_t p1 = yptr[row + 1];
      for (int64_t p = yptr[row]; p < p1; ++p) {
        const int64_t o = ycol[p];
        const float v = lane < R ? ld_f(other + o * R + lane) : 0.f;
        const float e = wsum(f * v) - yval[p];
        g = fmaf(e, v, g);
      }
    }
    if (lane < R) {
      grad[row * R + lane] = g;
      a_g2 += (double)g * g;
      a_gn += (double)g * n;
      a_fn += (double)f * n;
    }
  }
  const double v0 = jblock_sum(a_g2, red);
  const double v1 = jblock_sum(a_gn, red);
  const double v2 = jblock_sum(a_fn, red);
  if (threadIdx.x == 0) {
    part[(size_t)blockIdx.x * 3] = v0;
    part[(size_t)blockIdx.x * 3 + 1] = v1;
    part[(size_t)blockIdx.x * 3 + 2] = v2;
  }
}

// scal[kG2] += sum ||g||^2; scal[dst1] = <g, N> (T100, T010 or T001);
// scal[dst2] = <F, N> (T000, mode 0 only).
__global__ void __launch_bounds__(kJT) joint_grad_scalars(const double* __restrict__ part, int nb,
                                                         double* __restrict__ scal, int dst1, int dst2) {
  __shared__ double red[kJT];
  double v[3];
  for (int t = 0; t < 3; ++t) {
    double a = 0.0;
    for (int b = threadIdx.x; b < nb; b += kJT) a += part[(size_t)b * 3 + t];
    v[t] = jblock_sum(a, red);
  }
  if (threadIdx.x == 0) {
    scal[kG2] += v[0];
    scal[dst1] = v[1];
    if (dst2 >= 0) scal[dst2] = v[2];
  }
}

// The ratings term along the ray theta - alpha grad, a thread per rating (rows
// of any length spread over the GPU; a warp per user row left the longest row,
// tens of thousands of ratings on power-law data, as one serial chain):
// r(alpha) = y - (a - alpha ga) . (b - alpha gb) = e0 + e1 alpha + e2 alpha^2
// and 1/2 r^2 has coefficients 1/2 e0^2, e0 e1, 1/2 e1^2 + e0 e2, e1 e2, 1/2 e2^2;
// per-block partials part[block][5].  Without RAY only the first (the ratings
// loss at the current point) is formed.
//
// The dot products are trees over the RP columns (zeros past R), the order of a
// warp's shuffle reduction.  A chain over the columns rounds more often: objective
// of 11,220 ratings, R = 16, 1.7e-10 from 64 bits with it and 1.1e-10 with the
// tree; a sweep over 2M ratings takes 2.19 and 2.17 ms.
template <int RP>
__device__ __forceinline__ float tree_sum(float (&v)[RP]) {
#pragma unroll
  for (int h = RP / 2; h > 0; h >>= 1)
#pragma unroll
    for (int m = 0; m < h; ++m) v[m] += v[m + h];
  return v[0];
}

template <typename T, int RP, bool RAY>
__global__ void __launch_bounds__(kJT) ratings_quartic(
    const int64_t* __restrict__ yptr, const int32_t* __restrict__ ycol,
    const float* __restrict__ yval, const T* __restrict__ A, const T* __restrict__ B,
    const float* __restrict__ GA, const float* __restrict__ GB, int64_t rows, int64_t nnzY, int R,
    double* __restrict__ part) {
  __shared__ double red[kJT];
  double c[5] = {0, 0, 0, 0, 0};
  const int64_t stride = (int64_t)gridDim.x * kJT;
  for (int64_t p = (int64_t)blockIdx.x * kJT + threadIdx.x; p < nnzY; p += stride) {
    const int64_t row = rating_row(yptr, rows, p), o = ycol[p];
    float u[RP], s1[RAY ? RP : 1], s2[RAY ? RP : 1];
#pragma unroll
    for (int m = 0; m < RP; ++m) {
      const float a = m < R ? ld_f(A + row * R + m) : 0.f, b = m < R ? ld_f(B + o * R + m) : 0.f;
      u[m] = __fmul_rn(a, b);  // no contraction into the tree
      if constexpr (RAY) {
        const float ga = m < R ? GA[row * R + m] : 0.f, gb = m < R ? GB[o * R + m] : 0.f;
        s1[m] = fmaf(a, gb, ga * b);
        s2[m] = __fmul_rn(ga, gb);
      }
    }
    const double e0 = (double)yval[p] - (double)tree_sum<RP>(u);
    c[0] += 0.5 * e0 * e0;
    if constexpr (RAY) {
      const double e1 = (double)tree_sum<RP>(s1), e2 = -(double)tree_sum<RP>(s2);
      c[1] += e0 * e1;
      c[2] += 0.5 * e1 * e1 + e0 * e2;
      c[3] += e1 * e2;
      c[4] += 0.5 * e2 * e2;
    }
  }
  for (int k = 0; k < 5; ++k) {
    const double v = jblock_sum(c[k], red);
    if (threadIdx.x == 0) part[(size_t)blockIdx.x * 5 + k] = v;
  }
}

__global__ void __launch_bounds__(kJT) sum5(const double* __restrict__ part, int nb,
                                           double* __restrict__ out) {
  __shared__ double red[kJT];
  for (int k = 0; k < 5; ++k) {
    double a = 0.0;
    for (int b = threadIdx.x; b < nb; b += kJT) a += part[(size_t)b * 5 + k];
    const double v = jblock_sum(a, red);
    if (threadIdx.x == 0) out[k] = v;
  }
}

// The joint objective at the current point: ratings loss ycoef[0], the tensor
// loss from the fit's pieces (lambda weights are 1), the ridge from the Grams.
__global__ void joint_objective_k(const double* __restrict__ ycoef, const double* __restrict__ GA,
                                  const double* __restrict__ GB, const double* __restrict__ GC, int R,
                                  double mu, double lambda, double* __restrict__ scal) {
  if (threadIdx.x != 0) return;
  double tr = 0.0;
  for (int r = 0; r < R; ++r) tr += GA[r * R + r] + GB[r * R + r] + GC[r * R + r];
  const double ft = 0.5 * (scal[kNormX2] - 2.0 * scal[kInner] + scal[kModelNorm2]);
  scal[kLoss] = ycoef[0] + mu * ft + 0.5 * lambda * tr;
}

dfacto_status grow_part(dfacto_t* h, int64_t doubles) {
  JointState* J = h->joint;
  if (doubles <= J->part_cap) return DFACTO_OK;
  if (J->part) dfree(h, J->part, sizeof(double) * (size_t)J->part_cap);
  J->part = nullptr;
  J->part_cap = 0;
  dfacto_status st = dalloc(h, reinterpret_cast<void**>(&J->part), sizeof(double) * (size_t)doubles);
  if (st == DFACTO_OK) J->part_cap = doubles;
  return st;
}

int bits_for(int64_t dim) {
  int b = 1;
  while (b < 40 && (int64_t(1) << b) < dim) ++b;
  return b;
}

template <typename T, int RP>
dfacto_status joint_solve_side(dfacto_t* h, int side) {
  JointState* J = h->joint;
  const int R = h->R;
  cudaStream_t s = h->stream;
  const int64_t rows = h->dims[side];
  const bool rated = side < 2;
  const T* other = static_cast<const T*>(h->F[side == 0 ? 1 : 0]);
  if (rated && J->heavy[side]) {
    const int64_t chunks = (J->nnzY + kHeavyRatings - 1) / kHeavyRatings;
    if (!J->slots) {
      const dfacto_status st = dalloc(h, reinterpret_cast<void**>(&J->slots), 2 * (size_t)chunks * jslot_bytes(R));
      if (st != DFACTO_OK) return st;
    }
    joint_heavy<T, RP><<<(unsigned)((chunks + kJSolveWarps - 1) / kJSolveWarps), kJSolveWarps * 32, 0, s>>>(
        J->ptr[side], J->col[side], J->val[side], other, rows, J->nnzY, R, J->slots);
    DF_COUNT();
  }
  const bool few = few_rows(rows, R);
  const size_t smem = few ? joint_few_smem<RP>(R) : joint_solve_smem<RP>(R);
  const unsigned grid = few ? (unsigned)((rows + kJSolveWarps - 1) / kJSolveWarps) : jgrid(rows, 32);
  auto kernel = few ? joint_solve_few<T, RP> : joint_solve<T, RP>;
  DF_CUDA(h, ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), smem));
  kernel<<<grid, kJSolveWarps * 32, smem, s>>>(
      rated ? J->ptr[side] : nullptr, rated ? J->col[side] : nullptr, rated ? J->val[side] : nullptr,
      other, h->N, J->base, J->mu, rows, R, J->slots, static_cast<T*>(h->F[side]),
      h->flags + kFlagInternal);
  DF_COUNT();
  DF_CUDA(h, cudaGetLastError());
  return DFACTO_OK;
}

template <typename T>
dfacto_status joint_rows_side(dfacto_t* h, int side) {
  JointState* J = h->joint;
  const int R = h->R;
  cudaStream_t s = h->stream;
  dfacto_status st;
  const int f = (side + 2) % 3, in = (side + 1) % 3;
  for (int m : {f, in})
    if (!h->gram_valid[m] && (st = gram_of_factor(h, m)) != DFACTO_OK) return st;
  joint_base<<<1, 256, 0, s>>>(h->gram[f], h->gram[in], R, J->mu, h->lambda_reg, J->base, J->gam32);
  DF_COUNT();
  if ((st = mttkrp_launch(h, side, h->N)) != DFACTO_OK) return st;
  st = R <= 8 ? joint_solve_side<T, 8>(h, side) : R <= 16 ? joint_solve_side<T, 16>(h, side)
                                                          : joint_solve_side<T, 32>(h, side);
  if (st != DFACTO_OK) return st;
  h->gram_valid[side] = h->pad_valid[side] = false;
  return DFACTO_OK;
}

// The ratings term's coefficients J->ycoef at the current point (RAY: along the
// ray, the gradients are h->grad).
template <typename T, bool RAY>
dfacto_status ratings_term(dfacto_t* h) {
  JointState* J = h->joint;
  const unsigned nb = jgrid(J->nnzY, kJT);
  const dfacto_status st = grow_part(h, (int64_t)nb * 5);
  if (st != DFACTO_OK) return st;
  auto go = [&](auto kernel) {
    kernel<<<nb, kJT, 0, h->stream>>>(J->ptr[0], J->col[0], J->val[0], static_cast<const T*>(h->F[0]),
                                      static_cast<const T*>(h->F[1]), RAY ? h->grad[0] : nullptr,
                                      RAY ? h->grad[1] : nullptr, h->dims[0], J->nnzY, h->R, J->part);
  };
  if (h->R <= 8) go(ratings_quartic<T, 8, RAY>);
  else if (h->R <= 16) go(ratings_quartic<T, 16, RAY>);
  else go(ratings_quartic<T, 32, RAY>);
  DF_COUNT();
  sum5<<<1, kJT, 0, h->stream>>>(J->part, (int)nb, J->ycoef);
  DF_COUNT();
  DF_CUDA(h, cudaGetLastError());
  return DFACTO_OK;
}

template <typename T>
dfacto_status joint_objective_T(dfacto_t* h) {
  JointState* J = h->joint;
  cudaStream_t s = h->stream;
  dfacto_status st;
  fill_ones<<<1, 128, 0, s>>>(h->lambda, h->R);
  DF_COUNT();
  if ((st = fit_direct(h)) != DFACTO_OK) return st;  // <X, Xhat>, ||Xhat||^2 (and the Grams)
  if ((st = ratings_term<T, false>(h)) != DFACTO_OK) return st;
  joint_objective_k<<<1, 32, 0, s>>>(J->ycoef, h->gram[0], h->gram[1], h->gram[2], h->R, J->mu,
                                     h->lambda_reg, h->scal);
  DF_COUNT();
  DF_CUDA(h, cudaGetLastError());
  return DFACTO_OK;
}

template <typename T>
dfacto_status joint_gd_T(dfacto_t* h) {
  JointState* J = h->joint;
  const int R = h->R;
  cudaStream_t s = h->stream;
  dfacto_status st;
  DF_CUDA(h, cudaMemsetAsync(h->scal + kG2, 0, sizeof(double), s));
  for (int side = 0; side < 3; ++side) {
    const int f = (side + 2) % 3, in = (side + 1) % 3;
    for (int m : {f, in})
      if (!h->gram_valid[m] && (st = gram_of_factor(h, m)) != DFACTO_OK) return st;
    joint_base<<<1, 256, 0, s>>>(h->gram[f], h->gram[in], R, J->mu, h->lambda_reg, J->base,
                                 J->gam32);
    DF_COUNT();
    if ((st = mttkrp_launch(h, side, h->N)) != DFACTO_OK) return st;
    const int64_t rows = h->dims[side];
    const unsigned nb = jgrid(rows, kJT / 32);
    if ((st = grow_part(h, (int64_t)nb * 5)) != DFACTO_OK) return st;
    const bool rated = side < 2;
    joint_grad<T><<<nb, kJT, 0, s>>>(rated ? J->ptr[side] : nullptr, rated ? J->col[side] : nullptr,
                                     rated ? J->val[side] : nullptr,
                                     static_cast<const T*>(h->F[side == 0 ? 1 : 0]), h->N, J->gam32,
                                     J->mu, h->lambda_reg, rows, R, static_cast<const T*>(h->F[side]),
                                     h->grad[side], J->part);
    DF_COUNT();
    const int tlin = side == 0 ? kT100 : (side == 1 ? kT010 : kT001);
    joint_grad_scalars<<<1, kJT, 0, s>>>(J->part, (int)nb, h->scal, tlin, side == 0 ? kT000 : -1);
    DF_COUNT();
    DF_CUDA(h, cudaGetLastError());
  }
  if ((st = ratings_term<T, true>(h)) != DFACTO_OK) return st;  // along the ray
  if ((st = ray_matrices(h)) != DFACTO_OK) return st;
  if ((st = dual_pass(h)) != DFACTO_OK) return st;
  if ((st = line_search(h, J->mu, J->ycoef)) != DFACTO_OK) return st;
  return apply_step(h);
}

dfacto_status read_flags(dfacto_t* h) {
  DF_CUDA(h, cudaMemcpyAsync(h->host_scal, h->scal, sizeof(double) * kNumScalars,
                             cudaMemcpyDeviceToHost, h->stream));
  DF_CUDA(h, cudaMemcpyAsync(h->host_flags, h->flags, sizeof(int32_t) * kNumFlags,
                             cudaMemcpyDeviceToHost, h->stream));
  DF_CUDA(h, cudaStreamSynchronize(h->stream));
  if (h->host_flags[kFlagInternal]) return fail(h, DFACTO_EINTERNAL, "joint row solve failed");
  return DFACTO_OK;
}

}  // namespace

void joint_free(dfacto_t* h) {
  JointState* J = h->joint;
  if (!J) return;
  for (int side = 0; side < 2; ++side)
    for (void* q : {(void*)J->ptr[side], (void*)J->col[side], (void*)J->val[side]})
      if (q) cudaFreeAsync(q, h->stream);
  for (void* q : {(void*)J->base, (void*)J->gam32, (void*)J->ycoef, (void*)J->part, (void*)J->slots})
    if (q) cudaFreeAsync(q, h->stream);
  delete J;
  h->joint = nullptr;
}

}  // namespace dfacto

using namespace dfacto;

extern "C" {

dfacto_status dfacto_joint_set_ratings(dfacto_t* h, const int32_t* yidx, const float* yval,
                                       int64_t nnzY, double mu) {
  if (!h || nnzY < 0 || nnzY > kMaxNnz || (nnzY > 0 && (!yidx || !yval)) || !(mu >= 0.0))
    return DFACTO_EINVAL;
  if (h->R > 32) return fail(h, DFACTO_EINVAL, "the joint model takes R <= 32");
  if (h->batch) return fail(h, DFACTO_EINVAL, "handle is in a batch");
  cudaStream_t s = h->stream;
  joint_free(h);
  JointState* J = new (std::nothrow) JointState();
  if (!J) return DFACTO_ENOMEM;
  h->joint = J;
  J->mu = mu;
  J->nnzY = nnzY;
  const int R = h->R;
  dfacto_status st = DFACTO_OK;
  auto bail = [&](dfacto_status e) {
    joint_free(h);
    return e;
  };
  if ((st = dalloc(h, (void**)&J->base, sizeof(double) * R * R)) != DFACTO_OK) return bail(st);
  if ((st = dalloc(h, (void**)&J->gam32, sizeof(float) * R * R)) != DFACTO_OK) return bail(st);
  if ((st = dalloc(h, (void**)&J->ycoef, sizeof(double) * 8)) != DFACTO_OK) return bail(st);
  for (int side = 0; side < 2; ++side) {
    if ((st = dalloc(h, (void**)&J->ptr[side], sizeof(int64_t) * ((size_t)h->dims[side] + 1))) != DFACTO_OK)
      return bail(st);
    if ((st = dalloc(h, (void**)&J->col[side], sizeof(int32_t) * (size_t)nnzY)) != DFACTO_OK)
      return bail(st);
    if ((st = dalloc(h, (void**)&J->val[side], sizeof(float) * (size_t)nnzY)) != DFACTO_OK)
      return bail(st);
  }
  // the ratings on the device
  const int32_t* d_idx = yidx;
  const float* d_val = yval;
  int32_t* tmp_idx = nullptr;
  float* tmp_val = nullptr;
  uint64_t* k0 = nullptr;
  uint64_t* k1 = nullptr;
  uint32_t* v0 = nullptr;
  uint32_t* v1 = nullptr;
  auto cleanup = [&]() {
    for (void* q : {(void*)tmp_idx, (void*)tmp_val, (void*)k0, (void*)k1, (void*)v0, (void*)v1})
      if (q) cudaFreeAsync(q, s);
  };
  auto cuda_bail = [&](cudaError_t e, const char* what) {
    cleanup();
    st = cuda_fail(h, e, what);
    joint_free(h);
    return st;
  };
  cudaError_t e = cudaSuccess;
  if (nnzY > 0 && !is_device_ptr(yidx)) {
    if ((e = cudaMallocAsync((void**)&tmp_idx, sizeof(int32_t) * 2 * nnzY, s)) != cudaSuccess)
      return cuda_bail(e, "ratings copy");
    if ((e = cudaMemcpyAsync(tmp_idx, yidx, sizeof(int32_t) * 2 * nnzY, cudaMemcpyHostToDevice, s)) != cudaSuccess)
      return cuda_bail(e, "ratings copy");
    d_idx = tmp_idx;
  }
  if (nnzY > 0 && !is_device_ptr(yval)) {
    if ((e = cudaMallocAsync((void**)&tmp_val, sizeof(float) * nnzY, s)) != cudaSuccess)
      return cuda_bail(e, "ratings copy");
    if ((e = cudaMemcpyAsync(tmp_val, yval, sizeof(float) * nnzY, cudaMemcpyHostToDevice, s)) != cudaSuccess)
      return cuda_bail(e, "ratings copy");
    d_val = tmp_val;
  }
  if ((e = cudaMemsetAsync(h->flags, 0, sizeof(int32_t) * kNumFlags, s)) != cudaSuccess ||
      (e = cudaMemsetAsync(J->ycoef, 0, sizeof(double) * 8, s)) != cudaSuccess)  // heavy-row flags below
    return cuda_bail(e, "flags");
  if (nnzY > 0) {
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((nnzY + 255) / 256, 152 * 32));
    ratings_in_range<<<g, 256, 0, s>>>(d_idx, nnzY, h->dims[0], h->dims[1], h->flags + kFlagRange);
    DF_COUNT();
    if ((e = cudaMallocAsync((void**)&k0, sizeof(uint64_t) * nnzY, s)) != cudaSuccess ||
        (e = cudaMallocAsync((void**)&k1, sizeof(uint64_t) * nnzY, s)) != cudaSuccess ||
        (e = cudaMallocAsync((void**)&v0, sizeof(uint32_t) * nnzY, s)) != cudaSuccess ||
        (e = cudaMallocAsync((void**)&v1, sizeof(uint32_t) * nnzY, s)) != cudaSuccess)
      return cuda_bail(e, "ratings sort buffers");
  }
  for (int side = 0; side < 2; ++side) {
    const int64_t rows = h->dims[side];
    const int bc = bits_for(h->dims[1 - side]), br = bits_for(rows);
    bool alt = false;
    if (nnzY > 0) {
      const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((nnzY + 255) / 256, 152 * 32));
      rating_keys<<<g, 256, 0, s>>>(d_idx, nnzY, side, bc, k0, v0);
      DF_COUNT();
      if ((e = sort_pairs64(k0, v0, k1, v1, nnzY, 0, bc + br, s, &alt)) != cudaSuccess)
        return cuda_bail(e, "ratings sort");
      const uint64_t* ks = alt ? k1 : k0;
      const uint32_t* vs = alt ? v1 : v0;
      rating_scatter<<<g, 256, 0, s>>>(ks, vs, d_val, nnzY, bc, J->col[side], J->val[side],
                                       h->flags + kFlagDup);
      DF_COUNT();
      rating_ptr<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>((rows + 256) / 256, 152 * 32)), 256, 0, s>>>(
          ks, nnzY, rows, bc, J->ptr[side]);
      DF_COUNT();
      any_heavy<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>((rows + 255) / 256, 152 * 8)), 256, 0, s>>>(
          J->ptr[side], rows, reinterpret_cast<int32_t*>(J->ycoef) + side);
      DF_COUNT();
    } else {
      if ((e = cudaMemsetAsync(J->ptr[side], 0, sizeof(int64_t) * (rows + 1), s)) != cudaSuccess)
        return cuda_bail(e, "ratings pointers");
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_bail(e, "ratings build");
  }
  cleanup();
  int32_t flags[kNumFlags], heavy[2];
  if ((e = cudaMemcpyAsync(flags, h->flags, sizeof(flags), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
      (e = cudaMemcpyAsync(heavy, J->ycoef, sizeof(heavy), cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
      (e = cudaStreamSynchronize(s)) != cudaSuccess)
    return cuda_bail(e, "ratings check");
  if (flags[kFlagRange]) {
    joint_free(h);
    return fail(h, DFACTO_ERANGE, "a rating lies outside dims[0] x dims[1]");
  }
  if (flags[kFlagDup]) {
    joint_free(h);
    return fail(h, DFACTO_EDUP, "two ratings share (user, item)");
  }
  J->heavy[0] = heavy[0] != 0;
  J->heavy[1] = heavy[1] != 0;
  return DFACTO_OK;
}

dfacto_status dfacto_get_ratings_csr(dfacto_t* h, int side, dfacto_ratings_view* v) {
  if (!h || !v || side < 0 || side > 1) return DFACTO_EINVAL;
  if (!h->joint) return fail(h, DFACTO_EINVAL, "no ratings set");
  v->rows = h->dims[side];
  v->nnz = h->joint->nnzY;
  v->ptr = h->joint->ptr[side];
  v->col = h->joint->col[side];
  v->val = h->joint->val[side];
  return DFACTO_OK;
}

dfacto_status dfacto_joint_als_iter(dfacto_t* h, double* obj_out) {
  if (!h) return DFACTO_EINVAL;
  if (!h->joint) return fail(h, DFACTO_EINVAL, "no ratings set");
  if (!(h->lambda_reg > 0.0)) return fail(h, DFACTO_EINVAL, "the joint ALS needs lambda_reg > 0");
  DF_CUDA(h, cudaMemsetAsync(h->flags, 0, sizeof(int32_t) * kNumFlags, h->stream));
  dfacto_status st;
  for (int side = 0; side < 3; ++side) {
    st = h->dtype == DFACTO_BF16 ? joint_rows_side<__nv_bfloat16>(h, side) : joint_rows_side<float>(h, side);
    if (st != DFACTO_OK) return st;
  }
  if (!obj_out) return DFACTO_OK;
  st = h->dtype == DFACTO_BF16 ? joint_objective_T<__nv_bfloat16>(h) : joint_objective_T<float>(h);
  if (st != DFACTO_OK) return st;
  if ((st = read_flags(h)) != DFACTO_OK) return st;
  *obj_out = h->host_scal[kLoss];
  return DFACTO_OK;
}

dfacto_status dfacto_joint_gd_iter(dfacto_t* h, double* obj_out, double* alpha_out) {
  if (!h) return DFACTO_EINVAL;
  if (!h->joint) return fail(h, DFACTO_EINVAL, "no ratings set");
  dfacto_status st;
  for (int m = 0; m < 3; ++m)
    if (!h->grad[m] &&
        (st = dalloc(h, (void**)&h->grad[m], sizeof(float) * (size_t)h->dims[m] * h->R)) != DFACTO_OK)
      return st;
  DF_CUDA(h, cudaMemsetAsync(h->flags, 0, sizeof(int32_t) * kNumFlags, h->stream));
  st = h->dtype == DFACTO_BF16 ? joint_gd_T<__nv_bfloat16>(h) : joint_gd_T<float>(h);
  if (st != DFACTO_OK) return st;
  if (!obj_out && !alpha_out) return DFACTO_OK;
  if ((st = read_flags(h)) != DFACTO_OK) return st;
  if (obj_out) *obj_out = h->host_scal[kLoss];
  if (alpha_out) *alpha_out = h->host_scal[kStep];
  return h->host_flags[kFlagLsFail] ? DFACTO_ELSFAIL : DFACTO_OK;
}

dfacto_status dfacto_joint_objective(dfacto_t* h, double* obj_out) {
  if (!h || !obj_out) return DFACTO_EINVAL;
  if (!h->joint) return fail(h, DFACTO_EINVAL, "no ratings set");
  DF_CUDA(h, cudaMemsetAsync(h->flags, 0, sizeof(int32_t) * kNumFlags, h->stream));
  dfacto_status st =
      h->dtype == DFACTO_BF16 ? joint_objective_T<__nv_bfloat16>(h) : joint_objective_T<float>(h);
  if (st != DFACTO_OK) return st;
  if ((st = read_flags(h)) != DFACTO_OK) return st;
  *obj_out = h->host_scal[kLoss];
  return DFACTO_OK;
}

}  // extern "C"
