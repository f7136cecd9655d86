// mttkrp.cuh -- the fused two-SpMV MTTKRP of DFacTo (Algorithm 1), batched
// over all R columns.
//
// For mode n and every output row o:
//   N[o, :] = sum over fibers q = (o, f) of  F_f[f, :] (*) v_q,
//   v_q     = sum over nonzeros (in, x) of fiber q of  x * F_in[in, :],
// where v_q is row q of value(M^r) for all r at once (first SpMV, (Xhat)^T b_r)
// and the outer sum is the second SpMV, M^r c_r.  v_q never leaves registers.
//
// Work split (GB300): the nonzero stream is cut into segments of `seg`
// nonzeros, independent of row and fiber boundaries, so heavy (power-law)
// rows and fibers are spread over many lanes.  A group of G lanes walks one
// segment; each lane owns VEC consecutive columns and gathers them with one
// vector load per factor row.  The group's lanes fetch G upcoming (in, x)
// pairs with one coalesced load and pass them around by shuffles.  Splitting
// inside a fiber is exact because the second SpMV is linear in v.
//
// A row finished inside a segment is stored directly.  A segment's first and
// last rows may continue into neighbouring segments: their partial sums go to
// shared memory and are merged in segment order, first inside each warp, then
// across the CTA's warps.  Rows that continue beyond the CTA's range are left
// as per-CTA carries that mttkrp_fixup adds up in CTA order.  Every sum
// therefore has a fixed order: results are bitwise reproducible.
#pragma once

#include <type_traits>

#include "device.cuh"
#include "internal.h"

namespace dfacto {

struct MttkrpParams {
  const int64_t* fiber_ptr;
  const int32_t* fiber_idx;
  const int32_t* fiber_row;
  const int64_t* nz_ptr;
  const int32_t* nz_idx;
  const float* nz_val;
  const int32_t* seg_fib;
  const uint32_t* end_bits;  // bit p set iff nonzero p ends its fiber (walk2)
  const uint32_t* row_bits;  // bit p set iff nonzero p starts its row (walk2)
  const void* Fin;
  const void* Ff;
  float* out;
  float* carry;       // [ncta][2][R]
  int32_t* carry_row; // [ncta][2]
  int64_t nnz;
  int64_t nfib;
  int64_t dim_o;
  int R;
  int seg;
};

constexpr int kMaxColsPerLane = 4;  // R <= 128 in the CTA merge (lane-strided columns)

// Merge a sequence of (row, partial) entries into runs of equal rows, in order.
// flush(row, vals, is_first, is_last) is called once per run; is_first/is_last
// say whether the run contains the first/last valid entry.  Executed by one
// full warp; lane handles columns lane, lane+32, ...
template <typename Flush>
__device__ __forceinline__ void merge_runs(const int32_t* rows, const float* vals, int count, int R,
                                           int lane, Flush&& flush) {
  int run_row = -1;
  bool run_first = true;
  float run[kMaxColsPerLane];
#pragma unroll
  for (int k = 0; k < kMaxColsPerLane; ++k) run[k] = 0.f;
  for (int e = 0; e < count; ++e) {
    const int row = rows[e];
    if (row < 0) continue;
    if (row != run_row) {
      if (run_row >= 0) {
        flush(run_row, run, run_first, false);
        run_first = false;
      }
      run_row = row;
#pragma unroll
      for (int k = 0; k < kMaxColsPerLane; ++k) run[k] = 0.f;
    }
#pragma unroll
    for (int k = 0; k < kMaxColsPerLane; ++k) {
      const int col = lane + 32 * k;
      if (col < R) run[k] += vals[(size_t)e * R + col];
    }
  }
  if (run_row >= 0) flush(run_row, run, run_first, true);
}

// Merge the segment slots of one CTA (s_row/s_val: [SEGS * 2] entries), first
// inside each warp, then across warps; store complete rows and leave the CTA's
// partial first/last rows as carries.  Called by all threads after the walk.
template <int SEGS, int NG>
__device__ __forceinline__ void mttkrp_merge_cta(const MttkrpParams& a, int cta, int32_t* s_row,
                                                 float* s_val, int32_t* w_row, float* w_val, int lane,
                                                 int warp, int64_t cta_p0, int64_t cta_p1) {
  const int R = a.R;
  // Level 1: each warp merges its NG segments.  Runs strictly inside the
  // warp's range are complete rows.
  {
    if (lane == 0) { w_row[warp * 2] = -1; w_row[warp * 2 + 1] = -1; }
    __syncwarp();
    merge_runs(s_row + warp * NG * 2, s_val + (size_t)warp * NG * 2 * R, NG * 2, R, lane,
               [&](int row, const float (&run)[kMaxColsPerLane], bool first, bool last) {
                 const int k = first ? 0 : (last ? 1 : -1);
                 if (k < 0) {
#pragma unroll
                   for (int q = 0; q < kMaxColsPerLane; ++q) {
                     const int col = lane + 32 * q;
                     if (col < R) a.out[(int64_t)row * R + col] = run[q];
                   }
                 } else {
                   if (lane == 0) w_row[warp * 2 + k] = row;
#pragma unroll
                   for (int q = 0; q < kMaxColsPerLane; ++q) {
                     const int col = lane + 32 * q;
                     if (col < R) w_val[(size_t)(warp * 2 + k) * R + col] = run[q];
                   }
                 }
               });
  }
  __syncthreads();

  // Level 2: warp 0 merges the warps.  The CTA's first run may have started in
  // an earlier CTA, its last run may continue in a later one.
  if (warp == 0) {
    int first_row = -1, last_row = -1;
    for (int e = 0; e < kWalkWarps * 2; ++e) {
      const int r = w_row[e];
      if (r >= 0) { if (first_row < 0) first_row = r; last_row = r; }
    }
    bool first_partial = false, last_partial = false;
    if (first_row >= 0) {
      // rows of the first and last run: where do they begin and end?
      const int64_t fb = a.fiber_ptr[first_row];
      const int64_t le = a.fiber_ptr[last_row + 1];
      first_partial = a.nz_ptr[fb] < cta_p0;
      last_partial = a.nz_ptr[le] > cta_p1;
    }
    if (lane == 0) {
      a.carry_row[cta * 2] = -1;
      a.carry_row[cta * 2 + 1] = -1;
    }
    __syncwarp();
    merge_runs(w_row, w_val, kWalkWarps * 2, R, lane,
               [&](int row, const float (&run)[kMaxColsPerLane], bool first, bool last) {
                 const bool partial = (first && first_partial) || (last && last_partial);
                 if (!partial) {
#pragma unroll
                   for (int q = 0; q < kMaxColsPerLane; ++q) {
                     const int col = lane + 32 * q;
                     if (col < R) a.out[(int64_t)row * R + col] = run[q];
                   }
                 } else {
                   const int k = (first && first_partial) ? 0 : 1;
                   if (lane == 0) a.carry_row[cta * 2 + k] = row;
#pragma unroll
                   for (int q = 0; q < kMaxColsPerLane; ++q) {
                     const int col = lane + 32 * q;
                     if (col < R) a.carry[((int64_t)cta * 2 + k) * R + col] = run[q];
                   }
                 }
               });
  }
}

// Row of fiber q from row(M^r) alone: the largest r < dim_o with
// fiber_ptr[r] <= q (empty rows have fiber_ptr[r] == fiber_ptr[r + 1]).
__device__ __forceinline__ int row_of_fiber(const int64_t* fiber_ptr, int64_t dim_o, int64_t q) {
  int64_t lo = 0, hi = dim_o - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (fiber_ptr[mid] <= q) lo = mid; else hi = mid - 1;
  }
  return (int)lo;
}

// Row of fiber q given the row r0 of an earlier fiber (rows ascend with q).
__device__ __forceinline__ int row_after(const int64_t* fiber_ptr, int r0, int64_t q) {
  int r = r0;
  while (__ldg(fiber_ptr + r + 1) <= q) ++r;
  return r;
}

// kRowsFromPtr: take each fiber's row from fiber_ptr instead of the fiber_row
// array (for callers that pass only the CSR arrays of dfacto_csr_view).
template <typename T, int VEC, int G, bool kRowsFromPtr = false>
__global__ void __launch_bounds__(kWalkWarps * 32) mttkrp_walk(const MttkrpParams a) {
  constexpr int NG = 32 / G;
  constexpr int SEGS = kWalkWarps * NG;
  extern __shared__ float smem[];
  float* s_val = smem;                          // [SEGS * 2][R]
  float* w_val = smem + (size_t)SEGS * 2 * a.R; // [kWalkWarps * 2][R]
  __shared__ int32_t s_row[SEGS * 2];
  __shared__ int32_t w_row[kWalkWarps * 2];

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane / G, c = lane % G;
  const int gbase = g * G;
  const int col0 = c * VEC;
  const bool colok = col0 < a.R;
  const int sl = warp * NG + g;  // segment index inside the CTA
  const int64_t cta_p0 = (int64_t)blockIdx.x * SEGS * a.seg;
  const int64_t cta_p1 = min(cta_p0 + (int64_t)SEGS * a.seg, a.nnz);
  const int64_t p0 = cta_p0 + (int64_t)sl * a.seg;
  const int64_t p1 = min(p0 + a.seg, a.nnz);
  const bool active = p0 < a.nnz;
  const T* __restrict__ Fin = static_cast<const T*>(a.Fin);
  const T* __restrict__ Ff = static_cast<const T*>(a.Ff);
  const int R = a.R;

  float v[VEC], acc[VEC], ffc[VEC];
#pragma unroll
  for (int k = 0; k < VEC; ++k) { v[k] = 0.f; acc[k] = 0.f; ffc[k] = 0.f; }

  int64_t fib = 0, fend = 0, fend_next = 0;
  int row_cur = -1, row_next = -1, f_next = 0;
  if (active) {
    fib = a.seg_fib[(int64_t)blockIdx.x * SEGS + sl];
    fend = min(a.nz_ptr[fib + 1], p1);
    if constexpr (kRowsFromPtr) row_cur = row_of_fiber(a.fiber_ptr, a.dim_o, fib);
    else row_cur = a.fiber_row[fib];
    if (colok) VecIO<T, VEC>::load(Ff + (int64_t)a.fiber_idx[fib] * R + col0, ffc);
    if (fib + 1 < a.nfib) {
      fend_next = a.nz_ptr[fib + 2];
      f_next = a.fiber_idx[fib + 1];
      if constexpr (kRowsFromPtr) row_next = row_after(a.fiber_ptr, row_cur, fib + 1);
      else row_next = a.fiber_row[fib + 1];
    }
  }

  auto put_slot = [&](int k, int row, const float (&val)[VEC]) {
    if (c == 0) s_row[sl * 2 + k] = row;
    if (colok) {
#pragma unroll
      for (int q = 0; q < VEC; ++q) s_val[(size_t)(sl * 2 + k) * R + col0 + q] = val[q];
    }
  };
  bool head_open = true;

  for (int64_t base = p0; base < p0 + a.seg; base += G) {
    const int64_t pl = base + c;
    const bool okl = pl < p1;
    const int my_in = okl ? __ldg(a.nz_idx + pl) : 0;
    const float my_x = okl ? __ldg(a.nz_val + pl) : 0.f;
    // Row gathers are issued U at a time before any is used (memory-level
    // parallelism), U * VEC <= 32 registers.
    constexpr int U = (G < 32 / VEC) ? G : (32 / VEC);
#pragma unroll
    for (int u0 = 0; u0 < G; u0 += U) {
      float fin[U][VEC];
#pragma unroll
      for (int uu = 0; uu < U; ++uu) {
        const int in = __shfl_sync(kFull, my_in, gbase + u0 + uu);
        if (colok && base + u0 + uu < p1) {
          VecIO<T, VEC>::load(Fin + (int64_t)in * R + col0, fin[uu]);
        } else {
#pragma unroll
          for (int q = 0; q < VEC; ++q) fin[uu][q] = 0.f;
        }
      }
#pragma unroll
      for (int uu = 0; uu < U; ++uu) {
        const float x = __shfl_sync(kFull, my_x, gbase + u0 + uu);
        const int64_t p = base + u0 + uu;
        if (p < p1) {
#pragma unroll
          for (int q = 0; q < VEC; ++q) v[q] = fmaf(x, fin[uu][q], v[q]);
          if (p + 1 == fend) {  // the fiber (or its part in this segment) ends
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
              acc[q] = fmaf(v[q], ffc[q], acc[q]);
              v[q] = 0.f;
            }
            if (p + 1 < p1) {  // next fiber starts inside this segment
              ++fib;
              fend = min(fend_next, p1);
              if (row_next != row_cur) {
                if (head_open) {
                  put_slot(0, row_cur, acc);
                  head_open = false;
                } else if (colok) {
                  VecIO<float, VEC>::store(a.out + (int64_t)row_cur * R + col0, acc);
                }
#pragma unroll
                for (int q = 0; q < VEC; ++q) acc[q] = 0.f;
                row_cur = row_next;
              }
              if (colok) VecIO<T, VEC>::load(Ff + (int64_t)f_next * R + col0, ffc);
              if (fib + 1 < a.nfib) {
                fend_next = __ldg(a.nz_ptr + fib + 2);
                f_next = __ldg(a.fiber_idx + fib + 1);
                if constexpr (kRowsFromPtr) row_next = row_after(a.fiber_ptr, row_cur, fib + 1);
                else row_next = __ldg(a.fiber_row + fib + 1);
              }
            }
          }
        }
      }
    }
  }

  // Segment slots: 0 = head row partial, 1 = tail row partial (-1 = none).
  if (!active) {
    if (c == 0) { s_row[sl * 2] = -1; s_row[sl * 2 + 1] = -1; }
  } else if (head_open) {
    put_slot(0, row_cur, acc);
    if (c == 0) s_row[sl * 2 + 1] = -1;
  } else {
    put_slot(1, row_cur, acc);
  }
  __syncthreads();

  // Level 1: each warp merges its NG segments.  Runs strictly inside the
  // warp's range are complete rows.
  {
    if (lane == 0) { w_row[warp * 2] = -1; w_row[warp * 2 + 1] = -1; }
    __syncwarp();
    merge_runs(s_row + warp * NG * 2, s_val + (size_t)warp * NG * 2 * R, NG * 2, R, lane,
               [&](int row, const float (&run)[kMaxColsPerLane], bool first, bool last) {
                 const int k = first ? 0 : (last ? 1 : -1);
                 if (k < 0) {
#pragma unroll
                   for (int q = 0; q < kMaxColsPerLane; ++q) {
                     const int col = lane + 32 * q;
                     if (col < R) a.out[(int64_t)row * R + col] = run[q];
                   }
                 } else {
                   if (lane == 0) w_row[warp * 2 + k] = row;
#pragma unroll
                   for (int q = 0; q < kMaxColsPerLane; ++q) {
                     const int col = lane + 32 * q;
                     if (col < R) w_val[(size_t)(warp * 2 + k) * R + col] = run[q];
                   }
                 }
               });
  }
  __syncthreads();

  // Level 2: warp 0 merges the warps.  The CTA's first run may have started in
  // an earlier CTA, its last run may continue in a later one.
  if (warp == 0) {
    int first_row = -1, last_row = -1;
    for (int e = 0; e < kWalkWarps * 2; ++e) {
      const int r = w_row[e];
      if (r >= 0) { if (first_row < 0) first_row = r; last_row = r; }
    }
    bool first_partial = false, last_partial = false;
    if (first_row >= 0) {
      // rows of the first and last run: where do they begin and end?
      const int64_t fb = a.fiber_ptr[first_row];
      const int64_t le = a.fiber_ptr[last_row + 1];
      first_partial = a.nz_ptr[fb] < cta_p0;
      last_partial = a.nz_ptr[le] > cta_p1;
    }
    if (lane == 0) {
      a.carry_row[blockIdx.x * 2] = -1;
      a.carry_row[blockIdx.x * 2 + 1] = -1;
    }
    __syncwarp();
    merge_runs(w_row, w_val, kWalkWarps * 2, R, lane,
               [&](int row, const float (&run)[kMaxColsPerLane], bool first, bool last) {
                 const bool partial = (first && first_partial) || (last && last_partial);
                 if (!partial) {
#pragma unroll
                   for (int q = 0; q < kMaxColsPerLane; ++q) {
                     const int col = lane + 32 * q;
                     if (col < R) a.out[(int64_t)row * R + col] = run[q];
                   }
                 } else {
                   const int k = (first && first_partial) ? 0 : 1;
                   if (lane == 0) a.carry_row[blockIdx.x * 2 + k] = row;
#pragma unroll
                   for (int q = 0; q < kMaxColsPerLane; ++q) {
                     const int col = lane + 32 * q;
                     if (col < R) a.carry[((int64_t)blockIdx.x * 2 + k) * R + col] = run[q];
                   }
                 }
               });
  }
}

// ---------------------------------------------------------------------------
// mttkrp_walk2: the same sums in the same order with no branch on fiber
// metadata.  end_bits and row_bits mark the nonzeros that end a fiber and that
// start a row.  A group takes its segment in batches of B positions, whose
// (in, x) its lanes hold LPP each (loaded one batch ahead); the fiber of a
// position is the batch's first fiber plus the number of end bits before it,
// so each lane also holds f of its positions' fibers.  Per sub-batch of U
// positions the group gathers the U F_in rows and the F_f rows of the fibers
// that end there together, all independent of one another, and runs
//   v += x F_in;  at a fiber's last nonzero: acc += v (*) F_f, v = 0
// as predicated arithmetic; (in, x, f) are passed around by shuffles.  Batches
// in which no group of the warp starts a row (most of them on power-law
// tensors) skip the row tests.  The merge of rows shared between segments,
// warps and CTAs is the one of mttkrp_walk.
//
// What bounds it: the latency of the gathers against the registers that hold
// them.  The gathers mostly hit L1 and L2 (a bare probe of 128-byte rows reaches
// 140 G rows/s from L2 on this GPU, the walk 75 on 50M power-law nonzeros at
// R = 32), so what counts is how many are in flight and how few instructions
// stand between two rounds: the earlier form of this walk parked the fiber sums
// in shared memory and folded them in a second, dependent round of loads (18
// warp instructions per nonzero, now 8).  Per mode of 50M power-law nonzeros,
// before and now: R = 32 1.05 and 0.90 ms, R = 16 0.64 and 0.55, R = 8 0.59 and
// 0.40, R = 32 with BF16 factors 1.04 and 0.58.  Slower, all with segments of 256
// where this walk takes 0.86 ms at R = 32: the streams staged in shared memory by
// cp.async (0.87 ms, 12 instructions), the sum taken term by term without fibers
// (0.80 ms at R = 32 but 1.1 times slower at R = 12 to 16, and a gather more per
// nonzero), and eight FP32 columns per lane.
//
// nz_idx, nz_val and the bit words are allocated up to a multiple of 32
// nonzeros, zero past nnz: those positions read row 0, and as they end no
// fiber what they add to v is dropped.  fiber_idx has one entry more than
// fibers (the fiber "after" the last one, never gathered).  Lanes past column
// R walk column 0 and store nothing.
// ---------------------------------------------------------------------------

// VEC FP32 columns of a lane, two to a 64-bit register (one FFMA2 per pair).
template <int VEC>
struct Cols {
  uint64_t p[VEC / 2];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int e = 0; e < VEC / 2; ++e) p[e] = 0ull;
  }
  __device__ __forceinline__ void unpack(float (&o)[VEC]) const {
#pragma unroll
    for (int e = 0; e < VEC / 2; ++e) asm("mov.b64 {%0, %1}, %2;" : "=f"(o[2 * e]), "=f"(o[2 * e + 1]) : "l"(p[e]));
  }
  __device__ __forceinline__ void pack(const float (&v)[VEC]) {
#pragma unroll
    for (int e = 0; e < VEC / 2; ++e) asm("mov.b64 %0, {%1, %2};" : "=l"(p[e]) : "f"(v[2 * e]), "f"(v[2 * e + 1]));
  }
};
template <>
struct Cols<1> {
  float p[1];
  __device__ __forceinline__ void zero() { p[0] = 0.f; }
  __device__ __forceinline__ void unpack(float (&o)[1]) const { o[0] = p[0]; }
  __device__ __forceinline__ void pack(const float (&v)[1]) { p[0] = v[0]; }
};

// v += x w.
template <int VEC>
__device__ __forceinline__ void axpy_cols(float x, const Cols<VEC>& w, Cols<VEC>& v) {
  if constexpr (VEC == 1) {
    v.p[0] = fmaf(x, w.p[0], v.p[0]);
  } else {
    uint64_t xx;
    asm("mov.b64 %0, {%1, %1};" : "=l"(xx) : "f"(x));
#pragma unroll
    for (int e = 0; e < VEC / 2; ++e) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v.p[e]) : "l"(xx), "l"(w.p[e]));
  }
}

// If `on` is nonzero: acc += v w, v = 0 (predicated, no branch).
template <int VEC>
__device__ __forceinline__ void fold_cols_if(uint32_t on, const Cols<VEC>& w, Cols<VEC>& v, Cols<VEC>& acc) {
  if constexpr (VEC == 1) {
    asm("{.reg .pred q;\nsetp.ne.u32 q, %3, 0;\n@q fma.rn.f32 %0, %1, %2, %0;\n@q mov.f32 %1, 0f00000000;}"
        : "+f"(acc.p[0]), "+f"(v.p[0])
        : "f"(w.p[0]), "r"(on));
  } else {
#pragma unroll
    for (int e = 0; e < VEC / 2; ++e)
      asm("{.reg .pred q;\n.reg .f32 a0, a1, v0, v1, w0, w1;\nsetp.ne.u32 q, %3, 0;\n"
          "mov.b64 {a0, a1}, %0;\nmov.b64 {v0, v1}, %1;\nmov.b64 {w0, w1}, %2;\n"
          "@q fma.rn.f32 a0, v0, w0, a0;\n@q fma.rn.f32 a1, v1, w1, a1;\n"
          "@q mov.f32 v0, 0f00000000;\n@q mov.f32 v1, 0f00000000;\n"
          "mov.b64 %0, {a0, a1};\nmov.b64 %1, {v0, v1};}"
          : "+l"(acc.p[e]), "+l"(v.p[e])
          : "l"(w.p[e]), "r"(on));
  }
}

// VEC consecutive entries of a factor row as they are stored (widened at use).
template <typename T, int VEC>
struct RawCols;
template <int VEC>
struct RawCols<float, VEC> {
  Cols<VEC> v;
  __device__ __forceinline__ void load(const float* p) {
    if constexpr (VEC == 8) {
      asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];" : "=l"(v.p[0]), "=l"(v.p[1]), "=l"(v.p[2]), "=l"(v.p[3]) : "l"(p));
    } else if constexpr (VEC == 4) {
      asm("ld.global.nc.v2.b64 {%0, %1}, [%2];" : "=l"(v.p[0]), "=l"(v.p[1]) : "l"(p));
    } else if constexpr (VEC == 2) {
      asm("ld.global.nc.b64 %0, [%1];" : "=l"(v.p[0]) : "l"(p));
    } else {
      v.p[0] = __ldg(p);
    }
  }
  __device__ __forceinline__ Cols<VEC> get() const { return v; }
};
template <int VEC>
struct RawCols<__nv_bfloat16, VEC> {
  uint32_t w[(VEC + 1) / 2];
  __device__ __forceinline__ void load(const __nv_bfloat16* p) {
    if constexpr (VEC == 8) {
      const uint4 t = __ldg(reinterpret_cast<const uint4*>(p));
      w[0] = t.x; w[1] = t.y; w[2] = t.z; w[3] = t.w;
    } else if constexpr (VEC == 4) {
      const uint2 t = __ldg(reinterpret_cast<const uint2*>(p));
      w[0] = t.x; w[1] = t.y;
    } else if constexpr (VEC == 2) {
      w[0] = __ldg(reinterpret_cast<const unsigned int*>(p));
    } else {
      w[0] = __ldg(reinterpret_cast<const unsigned short*>(p));
    }
  }
  __device__ __forceinline__ Cols<VEC> get() const {
    Cols<VEC> o;
    if constexpr (VEC == 1) {
      o.p[0] = bf16_lo(w[0]);
    } else {
#pragma unroll
      for (int e = 0; e < VEC / 2; ++e)
        asm("mov.b64 %0, {%1, %2};" : "=l"(o.p[e]) : "f"(bf16_lo(w[e])), "f"(bf16_hi(w[e])));
    }
    return o;
  }
};

// Positions of the nonzero arrays a tensor of nnz nonzeros allocates.
__host__ __device__ constexpr int64_t walk_padded(int64_t nnz) { return (nnz + 31) / 32 * 32; }

// Dynamic shared memory of the walk at rank R: segment and warp partial rows
// for the merge.
inline size_t walk2_smem_bytes(int G, int R) {
  return sizeof(float) * (size_t)(2 * kWalkWarps * (32 / G) + 2 * kWalkWarps) * R;
}

template <typename T, int VEC, int G>
struct Walk2Shape {
  static constexpr int NG = 32 / G;
  static constexpr int SEGS = kWalkWarps * NG;
  // Positions per lane and batch, and per batch (divides 32).
  static constexpr int LPP = G >= 8 ? 1 : (G == 4 || VEC >= 8 ? 2 : 4);
  static constexpr int B = G * LPP;
  // Two buffers of U gathered rows and a budget of 128 registers (two CTAs per
  // SM): while one buffer is used the other is filled.  Eight lanes of four FP32
  // columns (R = 32) do better with one buffer at 80 registers and three CTAs.
  static constexpr int REGS = (VEC * (int)sizeof(T) + 3) / 4;  // registers of a row
  static constexpr int NBUF = REGS == 4 && VEC == 4 && G == 8 ? 1 : 2;
  static constexpr int MIN_BLOCKS = NBUF == 1 ? 3 : 2;
  static constexpr int U0 = REGS >= 8 ? 2 : (REGS >= 4 ? 4 : 8);
  static constexpr int U = NBUF * U0 <= B ? U0 : (B >= NBUF ? B / NBUF : 1);
  static_assert(B % (NBUF * U) == 0 && 32 % B == 0, "batch layout");
  static size_t smem_bytes(int R) { return walk2_smem_bytes(G, R); }
};

// LPP consecutive 32-bit words (the address is a multiple of their size).
template <int LPP>
__device__ __forceinline__ void ldg_words(const int32_t* p, int (&o)[LPP]) {
  if constexpr (LPP == 4) {
    const int4 t = __ldg(reinterpret_cast<const int4*>(p));
    o[0] = t.x; o[1] = t.y; o[2] = t.z; o[3] = t.w;
  } else if constexpr (LPP == 2) {
    const int2 t = __ldg(reinterpret_cast<const int2*>(p));
    o[0] = t.x; o[1] = t.y;
  } else {
    o[0] = __ldg(p);
  }
}

// The walk of CTA `cta` of one MTTKRP (shared by the single-tensor kernel and
// the batched one).  smem holds Walk2Shape::smem_bytes(R) bytes; s_row and
// w_row hold SEGS * 2 and kWalkWarps * 2 entries.
template <typename T, int VEC, int G>
__device__ __forceinline__ void walk2_cta(const MttkrpParams& a, int cta, float* smem,
                                          int32_t* s_row, int32_t* w_row) {
  using Shape = Walk2Shape<T, VEC, G>;
  constexpr int NG = Shape::NG, SEGS = Shape::SEGS, U = Shape::U, LPP = Shape::LPP, B = Shape::B;
  constexpr uint32_t kBatch = B == 32 ? 0xffffffffu : (1u << (B & 31)) - 1u;
  const int R = a.R;
  float* s_val = smem;                         // [SEGS * 2][R]
  float* w_val = smem + (size_t)SEGS * 2 * R;  // [kWalkWarps * 2][R]

  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int g = lane / G, c = lane % G;
  const int gbase = g * G;
  const int col0 = c * VEC;
  const bool colok = col0 < R;
  const int sl = warp * NG + g;
  // Positions fit in int: nnz <= kMaxNnz and seg <= kMaxSeg keep p0 + seg + 32
  // below 2^31 (the bounds are formed in 64 bits first).
  const int nnz = (int)a.nnz;
  const int npad = (int)walk_padded(a.nnz);
  const int cta_p0 = (int)min((int64_t)cta * SEGS * a.seg, a.nnz);
  const int cta_p1 = (int)min((int64_t)cta_p0 + (int64_t)SEGS * a.seg, a.nnz);
  const int p0 = (int)min((int64_t)cta * SEGS * a.seg + (int64_t)sl * a.seg, (int64_t)npad);
  const int p1 = min(p0 + a.seg, nnz);
  const bool active = p0 < nnz;
  // row t of the gathered factors from the lane's first column on
  const char* Fin = reinterpret_cast<const char*>(static_cast<const T*>(a.Fin) + (colok ? col0 : 0));
  const char* Ff = reinterpret_cast<const char*>(static_cast<const T*>(a.Ff) + (colok ? col0 : 0));
  const uint32_t stride = (uint32_t)(R * (int)sizeof(T));
  auto row_of = [&](const char* F, int t) {
    return reinterpret_cast<const T*>(F + (uint64_t)(uint32_t)t * stride);
  };

  Cols<VEC> v, acc;
  v.zero();
  acc.zero();
  int q = 0;  // fiber holding the batch's first position
  int row_cur = -1;
  uint32_t ew = 0u, rw = 0u;  // end and row-start bits from the batch's first position on
  if (active) {
    q = a.seg_fib[(int64_t)cta * SEGS + sl];
    row_cur = a.fiber_row[q];
    ew = __ldg(a.end_bits + (p0 >> 5));
    rw = __ldg(a.row_bits + (p0 >> 5)) & ~1u;  // the segment's first row is row_cur
  }
  // Segment slots: 0 = head row partial, 1 = tail row partial (-1 = none).  A
  // finished row goes to the output, the segment's first row to slot 0 (a
  // generic address either way).
  if (c == 0) s_row[sl * 2] = row_cur;
  float* head = s_val + (size_t)(sl * 2) * R + col0;  // null once the first row is in its slot
  auto put_row = [&](float* dst) {
    if (colok) {
      float val[VEC];
      acc.unpack(val);
      VecIO<float, VEC>::store(dst, val);
    }
  };
  // The lane's positions of the batch at p (past the arrays: of their last
  // batch, whose values are then not used).
  auto load_stream = [&](int p, int (&in)[LPP], int (&x)[LPP]) {
    const int pl = min(p, npad - B) + c * LPP;
    ldg_words<LPP>(a.nz_idx + pl, in);
    ldg_words<LPP>(reinterpret_cast<const int32_t*>(a.nz_val) + pl, x);
  };
  // f of the fibers of the lane's positions of a batch that starts in fiber qb.
  auto load_fibers = [&](int qb, uint32_t e, int (&f)[LPP]) {
#pragma unroll
    for (int j = 0; j < LPP; ++j)
      f[j] = __ldg(a.fiber_idx + (qb + __popc(e & ((1u << (c * LPP + j)) - 1u))));
  };

  // Gather the rows of positions u0 .. u0 + U - 1 of a batch (in, f, end bits).
  struct Rows {
    RawCols<T, VEC> fin[U], ff[U];
  };
  auto issue = [&](Rows& w, int u0, const int (&in)[LPP], const int (&f)[LPP], uint32_t e) {
#pragma unroll
    for (int uu = 0; uu < U; ++uu) {
      const int iu = G == 1 ? in[(u0 + uu) % LPP] : __shfl_sync(kFull, in[(u0 + uu) % LPP], gbase + (u0 + uu) / LPP);
      w.fin[uu].load(row_of(Fin, iu));
    }
#pragma unroll
    for (int uu = 0; uu < U; ++uu) {
      const int fu = G == 1 ? f[(u0 + uu) % LPP] : __shfl_sync(kFull, f[(u0 + uu) % LPP], gbase + (u0 + uu) / LPP);
      if (e & (1u << (u0 + uu))) w.ff[uu].load(row_of(Ff, fu));
    }
  };

  int in[LPP], x[LPP], f[LPP];
  load_stream(p0, in, x);
  load_fibers(q, ew, f);
  Rows buf[Shape::NBUF];
  if constexpr (Shape::NBUF == 2) issue(buf[0], 0, in, f, ew);
  for (int pb = p0; pb < p0 + a.seg; pb += 32) {
    uint32_t ewn = 0u, rwn = 0u;  // the next 32 positions' bits
    if (pb + 32 < p1) {
      ewn = __ldg(a.end_bits + ((pb + 32) >> 5));
      rwn = __ldg(a.row_bits + ((pb + 32) >> 5));
    }
#pragma unroll 1
    for (int k = 0; k < 32 / B; ++k) {
      const uint32_t eb = ew & kBatch, rb = rw & kBatch;
      const int qn = q + __popc(eb);
      if constexpr (B < 32) {
        ew = k == 32 / B - 1 ? ewn : ew >> (B & 31);
        rw = k == 32 / B - 1 ? rwn : rw >> (B & 31);
      } else {
        ew = ewn;
        rw = rwn;
      }
      int in_n[LPP], x_n[LPP], f_n[LPP];
      load_stream(pb + (k + 1) * B, in_n, x_n);
      load_fibers(qn, ew, f_n);
      const bool any = __any_sync(kFull, rb != 0u);
      auto batch = [&](auto with_rows) {
#pragma unroll
        for (int u0 = 0; u0 < B; u0 += U) {
          if constexpr (Shape::NBUF == 2) {
            // the next positions' rows are on their way while these are used
            if (u0 + U < B) issue(buf[((u0 / U) + 1) % 2], u0 + U, in, f, eb);
            else issue(buf[((u0 / U) + 1) % 2], 0, in_n, f_n, ew);
          } else {
            issue(buf[0], u0, in, f, eb);
          }
          const Rows& now = buf[(u0 / U) % Shape::NBUF];
#pragma unroll
          for (int uu = 0; uu < U; ++uu) {
            const int u = u0 + uu;
            const float xu = __int_as_float(G == 1 ? x[u % LPP] : __shfl_sync(kFull, x[u % LPP], gbase + u / LPP));
            if constexpr (decltype(with_rows)::value) {
              if ((rb >> u) & 1u) {
                put_row(head ? head : a.out + (int64_t)row_cur * R + col0);
                head = nullptr;
                acc.zero();
                row_cur = __ldg(a.fiber_row + (q + __popc(eb & ((1u << u) - 1u))));
              }
            }
            axpy_cols<VEC>(xu, now.fin[uu].get(), v);
            fold_cols_if<VEC>(eb & (1u << u), now.ff[uu].get(), v, acc);
          }
        }
      };
      if (any) batch(std::true_type{});
      else batch(std::false_type{});
      q = qn;
#pragma unroll
      for (int j = 0; j < LPP; ++j) {
        in[j] = in_n[j];
        x[j] = x_n[j];
        f[j] = f_n[j];
      }
    }
  }
  // The fiber open at the segment end (if its last nonzero lies beyond p1).
  if (active && !((__ldg(a.end_bits + ((p1 - 1) >> 5)) >> ((p1 - 1) & 31)) & 1u)) {
    RawCols<T, VEC> ff;
    ff.load(row_of(Ff, __ldg(a.fiber_idx + q)));
    fold_cols_if<VEC>(1u, ff.get(), v, acc);
  }

  if (c == 0) s_row[sl * 2 + 1] = head ? -1 : row_cur;
  if (active) put_row(s_val + (size_t)(sl * 2 + (head ? 0 : 1)) * R + col0);
  __syncthreads();
  mttkrp_merge_cta<SEGS, NG>(a, cta, s_row, s_val, w_row, w_val, lane, warp, cta_p0, cta_p1);
}

template <typename T, int VEC, int G>
__global__ void __launch_bounds__(kWalkWarps * 32, (Walk2Shape<T, VEC, G>::MIN_BLOCKS))
    mttkrp_walk2(const MttkrpParams a) {
  using Shape = Walk2Shape<T, VEC, G>;
  extern __shared__ __align__(16) float smem[];
  __shared__ int32_t s_row[Shape::SEGS * 2];
  __shared__ int32_t w_row[kWalkWarps * 2];
  walk2_cta<T, VEC, G>(a, blockIdx.x, smem, s_row, w_row);
}

// Launchers of the carry fix-up (mttkrp.cu) and of the segment-start search
// (build.cu), shared with the allocation-free entry point.
cudaError_t launch_mttkrp_fixup(const int32_t* carry_row, const float* carry,
                                const int64_t* fiber_ptr, const int64_t* nz_ptr, float* out, int R,
                                int64_t P, int64_t ncta, int64_t dim_o, int32_t* bad, bool serial,
                                cudaStream_t s);
cudaError_t launch_segment_starts(const int64_t* nz_ptr, int64_t nfib, int64_t nseg, int64_t seg,
                                  int32_t* seg_fib, cudaStream_t s);
// Zero end_bits and row_bits ((nnz + 31) / 32 words each) and set the bits of
// the last nonzero of every fiber and of the first nonzero of every row.
cudaError_t launch_walk_bits(const int64_t* nz_ptr, const int32_t* fiber_row, int64_t nfib, int64_t nnz,
                             uint32_t* end_bits, uint32_t* row_bits, cudaStream_t s);

// Launch one walk configuration (defined in the instantiation units).
template <typename T>
cudaError_t launch_walk(int vec, int G, const MttkrpParams& a, int64_t ncta, size_t smem,
                        cudaStream_t s);
template <typename T>
cudaError_t launch_walk2(int vec, int G, const MttkrpParams& a, int64_t ncta, cudaStream_t s);

}  // namespace dfacto
