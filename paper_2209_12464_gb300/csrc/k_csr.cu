// Sparse (CSR) products of RU-QLP (Section III-D: with s nonzeros the method
// costs O(sd); the same passes over A as the dense path).
//
//   Y[rows x d] = A X    with A in CSR (rowptr, colidx, values)
//   Z[cols x d] = A^T Y  with the CSR of A^T (the CSC of A), built once per
//                        decomposition and kept in the workspace.
//
// SpMM: one warp per output row; lane l owns columns 4l..4l+3 (then +128, ...)
// of the d columns; for each nonzero the warp gathers the matching row of the
// skinny operand (L2-resident) with 128-bit loads.  Every output entry is a
// sum over the row's nonzeros in storage order, so the result is
// deterministic.  The transpose is made deterministic too: nonzeros are
// scattered to their column (atomic cursors), then each column's entries are
// sorted by row index, the unique order of the CSC.
#include <algorithm>

#include "../../include/ruqlp.h"
#include "internal.h"

namespace ruqlp {
namespace {

template <typename TV> __device__ __forceinline__ float val_f32(TV v);
template <> __device__ __forceinline__ float val_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float val_f32<__nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}

// (Up to 2^31 - 1 entries are accepted, and the last index plus a stride passes the
// end of int32: loops over a row's entries are unsigned, or end at a multiple of the
// stride.  64-bit indices take 5 to 10 % more on rows of a few entries.)
// flag bit 1: rowptr not a valid prefix (rowptr[0] != 0, decreasing, or
// rowptr[m] != nnz); bit 2: column index out of range or not strictly
// increasing inside a row.  The valid columns are counted on the way (counts,
// zeroed before): one warp per row, so the indices are read once, coalesced
// (20M nonzeros: 185 us as a thread per row and a counting pass).
__global__ void k_csr_validate(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx,
                               int64_t m, int64_t n, int64_t nnz, int* flag,
                               int32_t* __restrict__ counts) {
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i > m) return;
  if (i == 0 && lane == 0 && rowptr[0] != 0) atomicOr(flag, 1);
  if (i == m) {
    if (lane == 0 && (int64_t)rowptr[m] != nnz) atomicOr(flag, 1);
    return;
  }
  const int32_t a = rowptr[i], b = rowptr[i + 1];
  if (b < a || a < 0 || (int64_t)b > nnz) {
    if (lane == 0) atomicOr(flag, 1);
    return;
  }
  bool bad = false;
  int32_t before = -1;  // the last index of the chunk before
  for (uint32_t e0 = a; e0 < (uint32_t)b; e0 += 32) {
    const bool in = e0 + lane < (uint32_t)b;
    const int32_t c = in ? colidx[e0 + lane] : 0x7fffffff;
    int32_t prev = __shfl_up_sync(0xffffffffu, c, 1);
    if (lane == 0) prev = before;
    if (in) {
      if (c <= prev || c < 0 || (int64_t)c >= n) bad = true;
      else atomicAdd(&counts[c], 1);
    }
    before = __shfl_sync(0xffffffffu, c, 31);
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(flag, 2);
}

// Exclusive scan of counts[0..n) into ptr[0..n]: block sums of 1024 counts,
// then every block adds the sums before it and scans its own.  A single block (n <=
// 1024) needs no sums, and writes the scatter's cursors itself (300 x 200 with 6000
// nonzeros: 76 to 79 us a call with the general form's three steps, 68 to 73 so).
constexpr int SCAN_BLOCK = 1024;
__device__ __forceinline__ int32_t block_sum(int32_t v, int32_t* red) {  // 256 threads
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  int32_t s = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) s += red[w];
  __syncthreads();
  return s;
}
__global__ void __launch_bounds__(256) k_scan_sums(const int32_t* __restrict__ counts, int64_t n,
                                                   int32_t* __restrict__ sums) {
  __shared__ int32_t red[8];
  int32_t v = 0;
  for (int q = 0; q < 4; ++q) {
    const int64_t i = (int64_t)blockIdx.x * SCAN_BLOCK + q * 256 + threadIdx.x;
    if (i < n) v += counts[i];
  }
  v = block_sum(v, red);
  if (threadIdx.x == 0) sums[blockIdx.x] = v;
}
__global__ void __launch_bounds__(256) k_scan(const int32_t* __restrict__ counts,
                                              const int32_t* sums, int64_t n,
                                              int32_t* __restrict__ ptr,
                                              int32_t* cursor) {
  __shared__ int32_t red[8];
  int32_t v = 0;
  for (int i = threadIdx.x; i < (int)blockIdx.x; i += 256) v += sums[i];
  const int32_t base = block_sum(v, red);
  const int64_t i0 = (int64_t)blockIdx.x * SCAN_BLOCK + 4 * threadIdx.x;
  int32_t c[4], t = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    c[q] = i0 + q < n ? counts[i0 + q] : 0;
    t += c[q];
  }
  int32_t run = t;  // inclusive scan of the threads' sums
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t x = __shfl_up_sync(0xffffffffu, run, o);
    if (lane >= o) run += x;
  }
  if (lane == 31) red[w] = run;
  __syncthreads();
  run += base - t;
  for (int k = 0; k < w; ++k) run += red[k];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (i0 + q < n) {
      ptr[i0 + q] = run;
      if (cursor != nullptr) cursor[i0 + q] = run;
    }
    run += c[q];
    if (i0 + q + 1 == n) ptr[n] = run;
  }
}

template <typename TV>
__global__ void k_csc_scatter(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx,
                              const TV* __restrict__ vals, int64_t m, int32_t* cursor,
                              int32_t* __restrict__ rowidx, TV* __restrict__ cvals) {
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= m) return;
  const int32_t a = rowptr[warp], b = rowptr[warp + 1];
  for (uint32_t e = a + lane; e < (uint32_t)b; e += 32) {
    const int32_t pos = atomicAdd(&cursor[colidx[e]], 1);
    rowidx[pos] = (int32_t)warp;
    cvals[pos] = vals[e];
  }
}

// Sort each column's (row, value) entries by row, one warp per column, up to
// 1024 entries in shared memory (flag bit 4: a column holds more).  The rows
// (distinct) are dealt to 32 buckets between the column's least and largest
// row; an entry's place is its bucket's start plus the number of smaller rows
// in the bucket (6 of 200 on average: 748 -> 80 us for 100000 columns against
// the bitonic network, which stays for columns whose fullest bucket holds more
// than 64).
constexpr int SORT_MAX = 1024;
template <typename TV>
__global__ void __launch_bounds__(128)
k_csc_sort(const int32_t* __restrict__ colptr, int64_t n, int32_t* __restrict__ rowidx,
           TV* __restrict__ cvals, int* flag) {
  __shared__ int32_t keys[4][SORT_MAX];
  __shared__ TV sv[4][SORT_MAX];
  __shared__ int32_t s_at[4][32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t c = (int64_t)blockIdx.x * 4 + w;
  if (c >= n) return;
  const int32_t a = colptr[c], b = colptr[c + 1];
  const int len = b - a;
  if (len <= 1) return;
  if (len > SORT_MAX) {
    if (lane == 0) atomicOr(flag, 4);
    return;
  }
  {
    int32_t lo = 0x7fffffff, hi = 0;
    for (int i = lane; i < len; i += 32) {
      const int32_t k = rowidx[a + i];
      lo = min(lo, k);
      hi = max(hi, k);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    const float scale = 32.f / ((float)(hi - lo) + 1.f);  // (monotone in the row)
    auto bucket = [&](int32_t k) { return min(31, (int)((float)(k - lo) * scale)); };
    s_at[w][lane] = 0;
    __syncwarp();
    for (int i = lane; i < len; i += 32) atomicAdd(&s_at[w][bucket(rowidx[a + i])], 1);
    __syncwarp();
    const int cnt = s_at[w][lane];
    int end = cnt;  // inclusive scan
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += x;
    }
    if (__reduce_max_sync(0xffffffffu, cnt) <= 64) {
      s_at[w][lane] = end - cnt;
      __syncwarp();
      for (int i0 = 0; i0 < len; i0 += 32) {  // by bucket, in any order
        const int i = i0 + lane;
        if (i < len) {
          const int32_t k = rowidx[a + i];
          const int pos = atomicAdd(&s_at[w][bucket(k)], 1);
          keys[w][pos] = k;
          sv[w][pos] = cvals[a + i];
        }
      }
      __syncwarp();
      for (int i0 = 0; i0 < len; i0 += 32) {
        const int i = i0 + lane;
        const int32_t k = i < len ? keys[w][i] : lo;
        const int bk = bucket(k);
        const int e1 = __shfl_sync(0xffffffffu, end, bk);
        const int e0 = e1 - __shfl_sync(0xffffffffu, cnt, bk);
        if (i < len) {
          int r = e0;
          for (int j = e0; j < e1; ++j) r += keys[w][j] < k ? 1 : 0;
          rowidx[a + r] = k;
          cvals[a + r] = sv[w][i];
        }
      }
      return;
    }
    __syncwarp();
  }
  int p2 = 1;
  while (p2 < len) p2 <<= 1;
  int32_t* K = keys[w];
  TV* V = sv[w];
  for (int i = lane; i < p2; i += 32) {
    K[i] = (i < len) ? rowidx[a + i] : 0x7fffffff;
    V[i] = cvals[a + ((i < len) ? i : 0)];  // padding keys sort last, values unused
  }
  __syncwarp();
  for (int size = 2; size <= p2; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = lane; i < p2; i += 32) {
        const int j = i ^ stride;
        if (j > i) {
          const bool up = (i & size) == 0;
          const int32_t ki = K[i], kj = K[j];
          if ((ki > kj) == up) {
            K[i] = kj;
            K[j] = ki;
            const TV t = V[i];
            V[i] = V[j];
            V[j] = t;
          }
        }
      }
      __syncwarp();
    }
  }
  for (int i = lane; i < len; i += 32) {
    rowidx[a + i] = K[i];
    cvals[a + i] = V[i];
  }
}

// Y[r][0..d) = sum_e val[e] X[col[e]][0..d) for r in [0, rows); X, Y FP32.
template <typename TV>
__global__ void __launch_bounds__(256)
k_spmm(const int32_t* __restrict__ ptr, const int32_t* __restrict__ idx, const TV* __restrict__ vals,
       int64_t rows, const float* __restrict__ X, int64_t ldx, int d, float* __restrict__ Y,
       int64_t ldy) {
  const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (r >= rows) return;
  const int32_t a = ptr[r], b = ptr[r + 1], b4 = a + ((b - a) & ~3);
  const int nchunk = (d + 127) / 128;  // 128 columns per warp sweep (4 per lane)
  for (int ch = 0; ch < nchunk; ++ch) {
    const int c = ch * 128 + lane * 4;
    const bool on = c < d;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    int32_t e = a;
    for (; e < b4; e += 4) {  // four independent gathers in flight
      int32_t col[4];
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        col[u] = idx[e + u];
        v[u] = val_f32(vals[e + u]);
      }
      if (on) {
        float4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = *reinterpret_cast<const float4*>(X + (int64_t)col[u] * ldx + c);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          acc.x = fmaf(v[u], x[u].x, acc.x);
          acc.y = fmaf(v[u], x[u].y, acc.y);
          acc.z = fmaf(v[u], x[u].z, acc.z);
          acc.w = fmaf(v[u], x[u].w, acc.w);
        }
      }
    }
    for (; e < b; ++e) {
      const int32_t col = idx[e];
      const float v = val_f32(vals[e]);
      if (on) {
        const float4 x = *reinterpret_cast<const float4*>(X + (int64_t)col * ldx + c);
        acc.x = fmaf(v, x.x, acc.x);
        acc.y = fmaf(v, x.y, acc.y);
        acc.z = fmaf(v, x.z, acc.z);
        acc.w = fmaf(v, x.w, acc.w);
      }
    }
    if (on) *reinterpret_cast<float4*>(Y + r * ldy + c) = acc;
  }
}

// out[r][c] += t[r][c], r < rows, c < d (FP32).
__global__ void k_add_rows(float* __restrict__ out, int64_t ldo, const float* __restrict__ t,
                           int64_t ldt, int64_t rows, int d) {
  for (int64_t r = blockIdx.x; r < rows; r += gridDim.x)
    for (int c = threadIdx.x; c < d; c += blockDim.x) out[r * ldo + c] += t[r * ldt + c];
}

}  // namespace

cudaError_t add_rows_f32(float* out, int64_t ldo, const float* t, int64_t ldt, int64_t rows, int d,
                         cudaStream_t st) {
  if (rows <= 0 || d <= 0) return cudaSuccess;
  k_add_rows<<<(int)std::min<int64_t>(rows, 152 * 16), 128, 0, st>>>(out, ldo, t, ldt, rows, d);
  count_launch();
  return cudaGetLastError();
}

cudaError_t csr_validate(const int32_t* rowptr, const int32_t* colidx, int64_t m, int64_t n,
                         int64_t nnz, int* flag, int32_t* scratch, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(scratch, 0, (size_t)n * sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  k_csr_validate<<<ceil_div((m + 1) * 32, 256), 256, 0, st>>>(rowptr, colidx, m, n, nnz, flag,
                                                              scratch);
  count_launch();
  return cudaGetLastError();
}

cudaError_t csr_transpose(Ty tv, const int32_t* rowptr, const int32_t* colidx, const void* vals,
                          int64_t m, int64_t n, int64_t nnz, int32_t* colptr, int32_t* rowidx,
                          void* cvals, int32_t* scratch, int* flag, cudaStream_t st) {
  int32_t* counts = scratch;        // n, from csr_validate
  int32_t* cursor = scratch + n;    // n
  const int nblk = ceil_div(n, SCAN_BLOCK);
  const bool one = nblk == 1;
  if (!one) {
    k_scan_sums<<<nblk, 256, 0, st>>>(counts, n, cursor);
    count_launch();
  }
  k_scan<<<nblk, 256, 0, st>>>(counts, cursor, n, colptr, one ? cursor : nullptr);
  count_launch();
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && !one)
    e = cudaMemcpyAsync(cursor, colptr, (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return e;
  const int gw = ceil_div(m * 32, 256);
  const int gs = ceil_div(n, 4);
  if (tv == Ty::F32) {
    k_csc_scatter<float><<<gw, 256, 0, st>>>(rowptr, colidx, (const float*)vals, m, cursor, rowidx,
                                             (float*)cvals);
    count_launch();
    k_csc_sort<float><<<gs, 128, 0, st>>>(colptr, n, rowidx, (float*)cvals, flag);
    count_launch();
  } else if (tv == Ty::BF16) {
    k_csc_scatter<__nv_bfloat16><<<gw, 256, 0, st>>>(rowptr, colidx, (const __nv_bfloat16*)vals, m,
                                                     cursor, rowidx, (__nv_bfloat16*)cvals);
    count_launch();
    k_csc_sort<__nv_bfloat16><<<gs, 128, 0, st>>>(colptr, n, rowidx, (__nv_bfloat16*)cvals, flag);
    count_launch();
  } else {
    return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t spmm_csr(Ty tv, const int32_t* ptr, const int32_t* idx, const void* vals, int64_t rows,
                     const float* X, int64_t ldx, int d, float* Y, int64_t ldy, cudaStream_t st) {
  if (rows <= 0) return cudaSuccess;
  if ((ldx % 4) || (ldy % 4) || ((uintptr_t)X & 15) || ((uintptr_t)Y & 15))
    return cudaErrorInvalidValue;
  const int grid = ceil_div(rows * 32, 256);
  if (tv == Ty::F32)
    k_spmm<float><<<grid, 256, 0, st>>>(ptr, idx, (const float*)vals, rows, X, ldx, d, Y, ldy);
  else if (tv == Ty::BF16)
    k_spmm<__nv_bfloat16><<<grid, 256, 0, st>>>(ptr, idx, (const __nv_bfloat16*)vals, rows, X, ldx,
                                                d, Y, ldy);
  else
    return cudaErrorInvalidValue;
  count_launch();
  return cudaGetLastError();
}

}  // namespace ruqlp
