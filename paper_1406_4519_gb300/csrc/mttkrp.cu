// mttkrp.cu -- host side of the MTTKRP: configuration, launch, and the carry
// fix-up kernel that finishes rows spanning several CTAs and zero-fills rows
// with no nonzeros.
#include <algorithm>
#include <type_traits>

#include "mttkrp.cuh"

namespace dfacto {
namespace {

constexpr int kFixThreads = 256;
constexpr int kFixWarps = kFixThreads / 32;
constexpr int kAheadCols = 32;  // carry values per lane a warp loads before adding them

// One block per CTA c (grid-stride): if c's last partial run belongs to a row r
// that starts inside c, add up r's partials from CTAs c .. c_last in a fixed
// order (eight warps take interleaved entries, a batch of them as a tree, then
// their FP64 sums are added in warp order) and store N[r, :].  Then all blocks
// zero the rows without fibers.  With SERIAL, the order of handles with BF16
// factors (see walk_segment), each warp adds its entries one after another and the
// warps' sums are added in warp order, all in FP32.
// `bad` (nullable) is set when a carry entry does not name the row it should.
// CPL = columns per lane (R <= 32 * CPL); a warp keeps 32 / CPL entries in
// flight, which bounds the time of the longest row (a heavy row of a
// power-law mode spans over a thousand CTAs).
template <int CPL, bool SERIAL>
__global__ void __launch_bounds__(kFixThreads) mttkrp_fixup(
    const int32_t* __restrict__ carry_row, const float* __restrict__ carry,
    const int64_t* __restrict__ fiber_ptr, const int64_t* __restrict__ nz_ptr, float* __restrict__ out,
    int R, int64_t P, int64_t ncta, int64_t dim_o, int32_t* __restrict__ bad) {
  using Acc = std::conditional_t<SERIAL, float, double>;
  __shared__ Acc part[kFixWarps][128];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t c = blockIdx.x; c < ncta; c += gridDim.x) {
    const int k = carry_row[2 * c + 1] >= 0 ? 1 : 0;
    const int r = carry_row[2 * c + k];
    if (r < 0) continue;
    const int64_t rb = nz_ptr[fiber_ptr[r]];
    if (rb < c * P) continue;  // r started in an earlier CTA, which owns it
    const int64_t re = nz_ptr[fiber_ptr[r + 1]];
    const int64_t clast = (re - 1) / P;
    const int64_t ne = clast - c + 1;
    Acc s[CPL];
#pragma unroll
    for (int q = 0; q < CPL; ++q) s[q] = 0;
    // Warp w adds entries w, w + 8, w + 16, ... in that order; kAhead of them
    // are loaded before the adds so that their loads overlap.
    constexpr int kAhead = kAheadCols / CPL;
    for (int64_t j0 = warp; j0 < ne; j0 += (int64_t)kAhead * kFixWarps) {
      float t[kAhead][CPL];
#pragma unroll
      for (int u = 0; u < kAhead; ++u) {
        const int64_t j = j0 + (int64_t)u * kFixWarps;
        const int64_t entry = (j == 0) ? (2 * c + k) : (2 * (c + j));
#pragma unroll
        for (int q = 0; q < CPL; ++q) {
          const int col = lane + 32 * q;
          t[u][q] = (j < ne && col < R) ? carry[entry * R + col] : 0.f;
        }
      }
      // A tree in FP32 over the batch, then one FP64 add: a heavy row's partials
      // are the longest chain of its sum, at the full magnitude of the result,
      // and FP64 instructions are slow (all of them in FP64: 25 us more per mode
      // of 50M nonzeros).  Entries past the end hold +0 and are added too.
      if constexpr (SERIAL) {
#pragma unroll
        for (int u = 0; u < kAhead; ++u)
#pragma unroll
          for (int q = 0; q < CPL; ++q) s[q] += t[u][q];
      } else {
#pragma unroll
        for (int w = kAhead / 2; w > 0; w >>= 1)
#pragma unroll
          for (int u = 0; u < w; ++u)
#pragma unroll
            for (int q = 0; q < CPL; ++q) t[u][q] += t[u + w][q];
#pragma unroll
        for (int q = 0; q < CPL; ++q) s[q] += (double)t[0][q];
      }
      if (lane < kAhead) {
        const int64_t j = j0 + (int64_t)lane * kFixWarps;
        if (bad && j > 0 && j < ne && carry_row[2 * (c + j)] != r) atomicOr(bad, 1);
      }
    }
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
      const int col = lane + 32 * q;
      if (col < R) part[warp][col] = s[q];
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
      for (int q = 0; q < CPL; ++q) {
        const int col = lane + 32 * q;
        if (col < R) {
          Acc t = part[0][col];
          for (int w = 1; w < kFixWarps && w < ne; ++w) t += part[w][col];
          out[(int64_t)r * R + col] = (float)t;
        }
      }
    }
    __syncthreads();
  }
  // 32 rows per warp: their empty ones as a mask, then the lanes over the rows'
  // consecutive columns (10M rows of 12 columns, the carries included: 241
  // us with a thread per row, 120 this way).
  const int R4 = R / 4;
  const bool quads = R % 4 == 0;
  const uint32_t inv = quads ? small_inv(R4) : small_inv(R);
  const int64_t stride = (int64_t)gridDim.x * kFixThreads;
  for (int64_t o = ((int64_t)blockIdx.x * kFixThreads + threadIdx.x) & ~(int64_t)31; o < dim_o; o += stride) {
    const int64_t row = o + lane;
    const unsigned empty = __ballot_sync(kFull, row < dim_o && fiber_ptr[row] == fiber_ptr[row + 1]);
    if (empty == 0u) continue;
    float* dst = out + o * R;
    if (quads) {
      for (int e = lane; e < 32 * R4; e += 32)
        if ((empty >> small_div(e, inv)) & 1u)
          reinterpret_cast<float4*>(dst)[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      for (int e = lane; e < 32 * R; e += 32)
        if ((empty >> small_div(e, inv)) & 1u) dst[e] = 0.f;
    }
  }
}

int next_pow2(int x) {
  int p = 1;
  while (p < x) p <<= 1;
  return p;
}

__device__ __forceinline__ float to_float(float x) { return x; }
__device__ __forceinline__ float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }

// Rows of an R-column matrix (storage type T) as FP32 rows of RP >= R columns
// (RP a multiple of four), the extra columns zero: 32 rows per warp, a lane per
// four columns of the result.
template <typename T>
__global__ void __launch_bounds__(256) pad_rows(const T* __restrict__ src, int64_t rows, int R, int RP,
                                                float* __restrict__ dst) {
  const int lane = threadIdx.x & 31, Q = RP / 4;
  const uint32_t inv = small_inv(Q);
  const int64_t stride = (int64_t)gridDim.x * 256;
  for (int64_t r0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) & ~(int64_t)31; r0 < rows; r0 += stride) {
    const int n = (int)min((int64_t)32, rows - r0) * Q;
    for (int e = lane; e < n; e += 32) {
      const int r = small_div(e, inv), c = 4 * (e - r * Q);
      const T* q = src + (r0 + r) * R + c;
      float4 v;
      v.x = to_float(q[0]);  // c < R: fewer than four columns are added
      v.y = c + 1 < R ? to_float(q[1]) : 0.f;
      v.z = c + 2 < R ? to_float(q[2]) : 0.f;
      v.w = c + 3 < R ? to_float(q[3]) : 0.f;
      reinterpret_cast<float4*>(dst + r0 * RP)[e] = v;
    }
  }
}

// The first R of every RP columns back to rows of R columns.
__global__ void __launch_bounds__(256) unpad_rows(const float* __restrict__ src, int64_t rows, int R, int RP,
                                                  float* __restrict__ dst) {
  const int lane = threadIdx.x & 31;
  const uint32_t inv = small_inv(R);
  const int64_t stride = (int64_t)gridDim.x * 256;
  for (int64_t r0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) & ~(int64_t)31; r0 < rows; r0 += stride) {
    const int n = (int)min((int64_t)32, rows - r0) * R;
    for (int e = lane; e < n; e += 32) {
      const int r = small_div(e, inv);
      dst[r0 * R + e] = src[(r0 + r) * RP + (e - r * R)];
    }
  }
}

unsigned rows_grid(int64_t n) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16));
}

}  // namespace

int walk_rank(int R, int vec_opt) {
  return (vec_opt == 0 && R > 2 && R % 4 != 0) ? (R + 3) / 4 * 4 : R;
}

cudaError_t pad_factor_rows(const void* src, int src_dtype, int64_t rows, int R, int RP, float* dst,
                            cudaStream_t s) {
  if (rows <= 0) return cudaSuccess;
  if (src_dtype == DFACTO_BF16)
    pad_rows<__nv_bfloat16><<<rows_grid(rows), 256, 0, s>>>(static_cast<const __nv_bfloat16*>(src),
                                                                   rows, R, RP, dst);
  else
    pad_rows<float><<<rows_grid(rows), 256, 0, s>>>(static_cast<const float*>(src), rows, R, RP, dst);
  DF_COUNT();
  return cudaGetLastError();
}

cudaError_t launch_mttkrp_fixup(const int32_t* carry_row, const float* carry,
                                const int64_t* fiber_ptr, const int64_t* nz_ptr, float* out, int R,
                                int64_t P, int64_t ncta, int64_t dim_o, int32_t* bad, bool serial,
                                cudaStream_t s) {
  const int64_t zero_blocks = (dim_o + kFixThreads - 1) / kFixThreads;
  const unsigned blocks =
      (unsigned)std::max<int64_t>(1, std::min<int64_t>(std::max(ncta, zero_blocks), 152 * 16));
  auto go = [&](auto kernel) {
    kernel<<<blocks, kFixThreads, 0, s>>>(carry_row, carry, fiber_ptr, nz_ptr, out, R, P, ncta, dim_o, bad);
  };
  if (R <= 32) serial ? go(mttkrp_fixup<1, true>) : go(mttkrp_fixup<1, false>);
  else if (R <= 64) serial ? go(mttkrp_fixup<2, true>) : go(mttkrp_fixup<2, false>);
  else serial ? go(mttkrp_fixup<kMaxColsPerLane, true>) : go(mttkrp_fixup<kMaxColsPerLane, false>);
  DF_COUNT();
  return cudaGetLastError();
}

// Segment length of a handle whose factors are stored as `dtype`, if none is
// asked for (0: by size).  BF16 factors round every updated entry to eight bits,
// so a last-bit change of a sum now and then moves an entry by 2^-9 and the next
// mode's weights by up to 1e-3.  A handle with BF16 factors therefore keeps one
// segment length and the fix-up's order of addition (SERIAL) at every size; a
// batch cuts the concatenated nonzeros of its jobs, at lengths of its own
// (batch.cu), so a job's sums are added in another order there.  Three modes of
// uniform nonzeros, R = 16: 100,000 115 us, 64 with segments of 32; 5M 361 us,
// 320 with 64.
int walk_segment(int dtype, int seg_opt) {
  return seg_opt > 0 ? seg_opt : dtype == DFACTO_BF16 ? 128 : 0;
}

WalkCfg choose_walk(int R, int dtype, int64_t nnz, int64_t nfib, int seg_opt, int vec_opt) {
  WalkCfg c;
  // Default: one 16-byte load per lane and factor row (4 FP32 or 8 BF16
  // columns), measured fastest on the 50M-nonzero power-law workload at
  // R = 16 and 32.
  int vec = vec_opt > 0 ? vec_opt : (dtype == DFACTO_BF16 ? 8 : 4);
  while (vec > 1 && (R % vec) != 0) vec >>= 1;
  int G = next_pow2((R + vec - 1) / vec);
  while (G > 32 && vec < 8 && (R % (vec * 2)) == 0) {
    vec *= 2;
    G = next_pow2((R + vec - 1) / vec);
  }
  c.vec = vec;
  c.G = G;
  c.kernel = 2;  // fiber ends from the end bitmask (faster on every measured shape)

  // Segment length: 128, or shorter where that leaves SMs without work: fewer
  // than a CTA per SM, or, with eight lanes per group and short fibers, than
  // four (such CTAs wait most and three are resident).  Never longer: a segment is
  // the longest FP32 chain of a row's sum (50M power-law nonzeros, R = 32: 860 us
  // per mode with 256 and 901 with 128, but 2.2e-7 from 64 bits and 1.8e-7).
  // Three modes with segments of 32, 64 and 128: uniform nonzeros 1M, R = 4: 103,
  // 146, 225 us; 8M, R = 4: 538, 463, 429; 2M, R = 16: 182, 147, 130; 2M in fibers
  // of 66, R = 16: 110, 92, 80; power-law nonzeros 2M, R = 32: 193, 178, 208.  Walk
  // 1 falls behind further with short ones (8M, R = 1: 1,569, 780, 755).
  const int segs = kWalkWarps * (32 / G);
  int seg = seg_opt;
  if (seg <= 0) {
    seg = 128;
    const int64_t ctas = 152 * (G >= 8 && nnz < 16 * nfib ? 4 : 1);
    while (seg > 32 && nnz < (int64_t)segs * seg * ctas) seg >>= 1;
  }
  seg = std::max(32, (seg + 31) / 32 * 32);
  c.seg = seg;
  return c;
}

void note_capture(dfacto_t* h) {
  if (h->recorded) return;
  cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(h->stream, &c) != cudaSuccess) cudaGetLastError();
  else h->recorded = c != cudaStreamCaptureStatusNone;
}

// The padded FP32 copy of factor m (rank RP), made when the factor changed, and
// at every call once a call on the handle was recorded into a graph.
dfacto_status ensure_padded(dfacto_t* h, int m) {
  const int RP = walk_rank(h->R, h->opt.vec);
  note_capture(h);
  if (h->pad_valid[m] && !h->recorded) return DFACTO_OK;
  dfacto_status st;
  if (!h->pad_F[m] &&
      (st = dalloc(h, reinterpret_cast<void**>(&h->pad_F[m]), sizeof(float) * (size_t)h->dims[m] * RP)) != DFACTO_OK)
    return st;
  DF_CUDA(h, pad_factor_rows(h->F[m], h->dtype, h->dims[m], h->R, RP, h->pad_F[m], h->stream));
  h->pad_valid[m] = true;
  return DFACTO_OK;
}

namespace {

// The walk and its fix-up.  At a rank that is not a multiple of four the walk
// runs on zero-padded FP32 copies of the two gathered factors at the padded
// rank RP (one 16-byte gather per lane: R = 10 walks 3 of 4 lanes per group
// instead of 5 of 8 with 8-byte gathers, measured 1.45x faster); an explicit
// lane width keeps the unpadded walk.  Both walks pad alike, so they still
// compute the same sums in the same order.  The result (rows of RP columns) goes
// to `wout`.
dfacto_status walk_rows(dfacto_t* h, int mode, float* wout) {
  ModeCSR& M = h->m[mode];
  const int RP = walk_rank(h->R, h->opt.vec);
  const bool padded = RP != h->R;
  const WalkCfg cfg = M.cfg;
  dfacto_status st = ensure_segments(h, mode);
  if (st != DFACTO_OK) return st;
  const int segs = kWalkWarps * (32 / cfg.G);
  const int64_t P = (int64_t)segs * cfg.seg;
  const int64_t ncta = (h->nnz + P - 1) / P;
  if (ncta > h->carry_cap || RP > h->carry_rank) {
    if (h->carry) dfree(h, h->carry, sizeof(float) * 2 * (size_t)h->carry_rank * h->carry_cap);
    if (h->carry_row) dfree(h, h->carry_row, sizeof(int32_t) * 2 * (size_t)h->carry_cap);
    h->carry = nullptr;
    h->carry_row = nullptr;
    const int64_t cap = std::max(ncta, h->carry_cap);
    const int rank = std::max(RP, h->carry_rank);
    h->carry_cap = 0;
    h->carry_rank = 0;
    st = dalloc(h, reinterpret_cast<void**>(&h->carry), sizeof(float) * 2 * (size_t)rank * cap);
    if (st == DFACTO_OK)
      st = dalloc(h, reinterpret_cast<void**>(&h->carry_row), sizeof(int32_t) * 2 * (size_t)cap);
    if (st != DFACTO_OK) return st;
    h->carry_cap = cap;
    h->carry_rank = rank;
  }
  const void* Fin = h->F[M.in];
  const void* Ff = h->F[M.f];
  if (padded) {
    if ((st = ensure_padded(h, M.in)) != DFACTO_OK) return st;
    if ((st = ensure_padded(h, M.f)) != DFACTO_OK) return st;
    Fin = h->pad_F[M.in];
    Ff = h->pad_F[M.f];
  }
  MttkrpParams a;
  a.fiber_ptr = M.fiber_ptr;
  a.fiber_idx = M.fiber_idx;
  a.fiber_row = M.fiber_row;
  a.nz_ptr = M.nz_ptr;
  a.nz_idx = M.nz_idx;
  a.nz_val = M.nz_val;
  a.seg_fib = M.seg_fib;
  a.end_bits = M.end_bits;
  a.row_bits = M.row_bits;
  a.Fin = Fin;
  a.Ff = Ff;
  a.out = wout;
  a.carry = h->carry;
  a.carry_row = h->carry_row;
  a.nnz = h->nnz;
  a.nfib = M.nfib;
  a.dim_o = M.dim_o;
  a.R = RP;
  a.seg = cfg.seg;
  if (ncta > 0) {
    const size_t smem = sizeof(float) * (size_t)(2 * segs + 2 * kWalkWarps) * RP;
    cudaError_t e;
    if (cfg.kernel == 2)
      e = (h->dtype == DFACTO_BF16 && !padded) ? launch_walk2<__nv_bfloat16>(cfg.vec, cfg.G, a, ncta, h->stream)
                                               : launch_walk2<float>(cfg.vec, cfg.G, a, ncta, h->stream);
    else
      e = (h->dtype == DFACTO_BF16 && !padded)
              ? launch_walk<__nv_bfloat16>(cfg.vec, cfg.G, a, ncta, smem, h->stream)
              : launch_walk<float>(cfg.vec, cfg.G, a, ncta, smem, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "mttkrp_walk launch");
  }
  DF_CUDA(h, launch_mttkrp_fixup(h->carry_row, h->carry, M.fiber_ptr, M.nz_ptr, wout, RP, P, ncta,
                                 M.dim_o, h->flags + kFlagInternal, h->dtype == DFACTO_BF16, h->stream));
  return DFACTO_OK;
}

dfacto_status ensure_pad_out(dfacto_t* h, int RP) {
  if (h->pad_out) return DFACTO_OK;
  const int64_t maxdim = std::max<int64_t>(h->dims[0], std::max<int64_t>(h->dims[1], h->dims[2]));
  return dalloc(h, reinterpret_cast<void**>(&h->pad_out), sizeof(float) * (size_t)maxdim * RP);
}

}  // namespace

dfacto_status mttkrp_launch(dfacto_t* h, int mode, float* out) {
  const int R = h->R, RP = walk_rank(R, h->opt.vec);
  if (RP == R) return walk_rows(h, mode, out);
  dfacto_status st = ensure_pad_out(h, RP);
  if (st == DFACTO_OK) st = walk_rows(h, mode, h->pad_out);
  if (st != DFACTO_OK) return st;
  const int64_t rows = h->m[mode].dim_o;
  unpad_rows<<<rows_grid(rows), 256, 0, h->stream>>>(h->pad_out, rows, R, RP, out);
  DF_COUNT();
  DF_CUDA(h, cudaGetLastError());
  return DFACTO_OK;
}

dfacto_status mttkrp_rows(dfacto_t* h, int mode, const float** N, int* ld) {
  const int RP = walk_rank(h->R, h->opt.vec);
  *ld = RP;
  *N = h->N;
  if (RP == h->R) return walk_rows(h, mode, h->N);
  const dfacto_status st = ensure_pad_out(h, RP);
  if (st != DFACTO_OK) return st;
  *N = h->pad_out;
  return walk_rows(h, mode, h->pad_out);
}

}  // namespace dfacto
