// SIMT (CUDA-core) products for RU-QLP: the FP64 and FP32 paths of the
// sketch / power-iteration products (Section III-D: A X and A^T Y, O(mnd)),
// and the tall-skinny Gram and R products of orth() (O(md^2)).
//
// One CTA of 256 threads computes a 64 x 64 output tile; each thread owns a
// 4 x 4 sub-tile.  K is walked in 16-wide slabs staged in shared memory.
// Out-of-range rows/columns are zero-filled on load and skipped on store, so
// any M, K, N works (ragged tails included).
#include <algorithm>
#include <type_traits>

#include "internal.h"

namespace ruqlp {
namespace {

constexpr int BM = 64, BN = 64, BK = 16, NT = 256;

template <Mul MODE> struct MulT;
template <> struct MulT<Mul::F64> { using mul = double; using acc = double; };
template <> struct MulT<Mul::F32> { using mul = float; using acc = float; };
template <> struct MulT<Mul::F32_ACC64> { using mul = float; using acc = double; };

template <typename T> __device__ __forceinline__ T zero() { return T(0); }

// TRANS_A = false: A is M x K (row-major, lda): C = A B.
// TRANS_A = true:  A is K x M (row-major, lda): C = A^T B.
// blockIdx.z selects a K slab [kz0, kz1); with PARTIAL the FP64 tile sums go to
// C + z*M*ldc (a [splits][M][ldc] FP64 buffer).
// ROUND_B: 1 = the B operand is rounded to BF16 as it is staged; 2 = to the
// sum of its two BF16 parts, h + bf16(b - h) (exact in FP32).
template <bool TRANS_A, typename TA, typename TB, typename TC, Mul MODE, bool PARTIAL,
          int ROUND_B = 0>
__device__ __forceinline__ void gemm_tile(const TA* __restrict__ A, int64_t lda,
                                          const TB* __restrict__ B, int64_t ldb,
                                          TC* __restrict__ C, int64_t ldc, int64_t M, int64_t K,
                                          int64_t N, int64_t kslab, int bx, int by, int bz) {
  using TM = typename MulT<MODE>::mul;
  using TAcc = typename MulT<MODE>::acc;
  __shared__ TM As[BK][BM + 4];
  __shared__ TM Bs[BK][BN + 4];
  const int t = threadIdx.x;
  const int tx = t & 15, ty = t >> 4;
  const int64_t m0 = (int64_t)bx * BM;
  const int64_t n0 = (int64_t)by * BN;
  const int64_t kz0 = (int64_t)bz * kslab;
  const int64_t kz1 = min(K, kz0 + kslab);

  TAcc acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = zero<TAcc>();

  for (int64_t k0 = kz0; k0 < kz1; k0 += BK) {
    // stage A (BM x BK) as As[k][m]
#pragma unroll
    for (int e = t; e < BM * BK; e += NT) {
      int r, c;
      if (TRANS_A) { r = e % BM; c = e / BM; }   // consecutive threads walk m (contiguous)
      else         { r = e / BK; c = e % BK; }   // consecutive threads walk k (contiguous)
      const int64_t gm = m0 + r, gk = k0 + c;
      TM v = zero<TM>();
      if (gm < M && gk < kz1) {
        v = Cvt<TM>::from(TRANS_A ? A[gk * lda + gm] : A[gm * lda + gk]);
      }
      As[c][r] = v;
    }
    // stage B (BK x BN) as Bs[k][n]
#pragma unroll
    for (int e = t; e < BK * BN; e += NT) {
      const int r = e / BN, c = e % BN;
      const int64_t gk = k0 + r, gn = n0 + c;
      TM v = zero<TM>();
      if (gk < kz1 && gn < N) {
        v = Cvt<TM>::from(B[gk * ldb + gn]);
        if constexpr (ROUND_B == 1) v = __bfloat162float(__float2bfloat16_rn(v));
        if constexpr (ROUND_B == 2) {
          const float h = __bfloat162float(__float2bfloat16_rn(v));
          v = h + __bfloat162float(__float2bfloat16_rn(v - h));
        }
      }
      Bs[r][c] = v;
    }
    __syncthreads();
    TM part[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) part[i][j] = zero<TM>();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      TM a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) part[i][j] = fma(a[i], b[j], part[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] += (TAcc)part[i][j];
    __syncthreads();
  }

  TC* Cz = PARTIAL ? C + (int64_t)bz * M * ldc : C;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t gm = m0 + ty * 4 + i;
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t gn = n0 + tx * 4 + j;
      if (gn < N) Cz[gm * ldc + gn] = Cvt<TC>::from(acc[i][j]);
    }
  }
}

// Whether a zero of the tile (bx, by) of C = A B (A^T B), formed by the
// tensor-core product, may stand for products that underflowed: both its row of A
// and its column of B hold a nonzero value, and one of them one below 2^-50.
// (Zero rows and columns, and sums that cancel among larger values, are exact.)
template <bool TRANS_A>
__device__ __forceinline__ bool zeros_suspect(const float* __restrict__ A, int64_t lda,
                                           const float* __restrict__ B, int64_t ldb,
                                           const float* __restrict__ C, int64_t ldc, int64_t M,
                                           int64_t K, int64_t N, int bx, int by) {
  constexpr int ZERO = 1, NONZERO = 2, SMALL = 4;
  __shared__ int s_row[BM], s_col[BN];  // bits: a zero result; operands met
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int64_t m0 = (int64_t)bx * BM, n0 = (int64_t)by * BN;
  auto kind = [](float x) {
    const uint32_t u = __float_as_uint(x) << 1;
    return u == 0u ? 0 : u < 2u * 0x26800000u ? NONZERO | SMALL : NONZERO;
  };
  auto is_zero = [&](int e) {
    const int64_t i = m0 + e / BN, j = n0 + e % BN;
    return i < M && j < N && C[i * ldc + j] == 0.f;
  };
  for (int e = t; e < BM + BN; e += NT) (e < BM ? s_row[e] : s_col[e - BM]) = 0;
  __syncthreads();
  bool any = false;
  for (int e = t; e < BM * BN; e += NT)
    if (is_zero(e)) {
      any = true;
      atomicOr(&s_row[e / BN], ZERO);
      atomicOr(&s_col[e % BN], ZERO);
    }
  if (!__syncthreads_or(any)) return false;
  // thread t: column t % 64 of a K x 64 panel, rows t / 64, + 4, ...
  auto panel = [&](const float* P, int64_t ld, int64_t c0, int64_t width, int* s) {
    const int c = t % 64;
    if (c0 + c >= width || !(s[c] & ZERO)) return;
    int f = 0;
#pragma unroll 8
    for (int64_t k = t / 64; k < K; k += NT / 64) f |= kind(P[k * ld + c0 + c]);
    atomicOr(&s[c], f);
  };
  panel(B, ldb, n0, N, s_col);
  if (TRANS_A) {
    panel(A, lda, m0, M, s_row);
  } else {
    for (int r = warp; r < BM; r += NT / 32) {
      if (!(s_row[r] & ZERO)) continue;
      int f = 0;
#pragma unroll 8
      for (int64_t k = lane; k < K; k += 32) f |= kind(A[(m0 + r) * lda + k]);
      atomicOr(&s_row[r], f);
    }
  }
  __syncthreads();
  any = false;
  for (int e = t; e < BM * BN; e += NT) {
    const int r = s_row[e / BN], c = s_col[e % BN];
    any |= (r & c & NONZERO) && ((r | c) & SMALL) && is_zero(e);
  }
  return __syncthreads_or(any);
}

// (80 registers in FP32: left to itself the compiler takes 74 beside the zeros' check,
// and the product 4 % longer; 0: the other types keep the compiler's choice)
template <bool TRANS_A, typename TA, typename TB, typename TC, Mul MODE, bool PARTIAL>
__global__ void __launch_bounds__(NT, MODE == Mul::F32 ? 3 : 0)
k_gemm(const TA* __restrict__ A, int64_t lda, const TB* __restrict__ B, int64_t ldb,
       TC* __restrict__ C, int64_t ldc, int64_t M, int64_t K, int64_t N, int64_t kslab,
       const int32_t* __restrict__ gate, const int32_t* __restrict__ redo) {
  if (gate != nullptr && *gate == 0) return;
  if (redo != nullptr && !range_redo(*redo)) {
    if constexpr (MODE == Mul::F32 && std::is_same_v<TA, float> && std::is_same_v<TB, float> &&
                  std::is_same_v<TC, float> && !PARTIAL) {
      if (!range_zeros(*redo) || !zeros_suspect<TRANS_A>(A, lda, B, ldb, C, ldc, M, K, N,
                                                         blockIdx.x, blockIdx.y))
        return;
    } else {
      return;
    }
  }
  gemm_tile<TRANS_A, TA, TB, TC, MODE, PARTIAL>(A, lda, B, ldb, C, ldc, M, K, N, kslab,
                                                blockIdx.x, blockIdx.y, blockIdx.z);
}

// Batched products over a problem table: tile t of the whole launch maps to
// matrix i = (prefix[i] <= t < prefix[i+1]) and a 64 x 64 output tile of it.
//   TRANS_A = false: buf[dst] (m x d) = A buf[src] (n x d)
//   TRANS_A = true:  buf[dst] (n x d) = A^T buf[src] (m x d)
// (two CTAs per SM at least in FP32: the zeros' check beside the product makes the
// compiler spill at three, 369 instead of 324 us for eight 2048 x 1024 A^T X at d = 72)
template <bool TRANS_A, typename TA, typename TB, int SPLIT2 = 0>
__global__ void __launch_bounds__(NT, std::is_same_v<TA, float> ? 2 : 0)
k_bgemm(const BMat* __restrict__ T, const int* __restrict__ prefix, int count, int src, int dst) {
  // FP32 items on the tensor cores come here only to be formed again
  const int t = blockIdx.x;
  int lo = 0, hi = count;  // largest i with prefix[i] <= t
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (prefix[mid] <= t) lo = mid; else hi = mid;
  }
  const BMat& b = T[prefix[count + 1 + lo]];  // the launch order's item lo
  const int local = t - prefix[lo];
  const int ntn = (b.d + BN - 1) / BN;
  const int64_t Mout = TRANS_A ? b.n : b.m, K = TRANS_A ? b.m : b.n;
  if constexpr (std::is_same_v<TA, float> && std::is_same_v<TB, float>) {
    if (b.flags & (TRANS_A ? BM_F32_ATY : BM_F32_AX)) {
      const int32_t range = b.status->range;
      if (range_redo(range)) {
        // no further attempts of this item (nothing reads the words in this launch)
        if (local == 0 && threadIdx.x == 0) {
          BMat& w = const_cast<BMat&>(b);
          w.f32_k[0] = w.f32_k[1] = 0;
        }
      } else if (!range_zeros(range) ||
                 !zeros_suspect<TRANS_A>((const float*)b.A, b.lda, bbuf(b, src), b.dp,
                                         bbuf(b, dst), b.dp, Mout, K, b.d, local / ntn,
                                         local % ntn)) {
        return;
      }
    }
  }
  // with BF16 A the skinny operand is rounded to BF16 (or to its two-part
  // BF16 sum) as it is staged, the product the single-matrix BF16 path computes
  constexpr int RB = std::is_same<TA, __nv_bfloat16>::value ? (SPLIT2 ? 2 : 1) : 0;
  gemm_tile<TRANS_A, TA, TB, float, Mul::F32, false, RB>(
      (const TA*)b.A, b.lda, (const TB*)bbuf(b, src), b.dp, bbuf(b, dst), b.dp, Mout, K, b.d,
      ((K + BK - 1) / BK) * BK, local / ntn, local % ntn, 0);
}

// FP64 products of one matrix with tiles fitted to the shape.  A CTA computes a
// BM x BN tile (BN any multiple of NI), each thread MI x NI of it: per entry FMA
// chains of BL rows of K, whose sums are added in turn.  (Measured against chains of
// 16, the 64 x 64 tiles' order: one chain over all of a slab has 1.2 to 1.6 times
// the rounding error in products of K <= 300, 1.1 at 8192, 1.2 to 1.5 in Grams;
// with these chains 1.00 at K <= 64, 0.7 at 544, 0.39 at 4096, 0.65 to 0.99 in
// Grams.  Chains of 32 halve the additions, 3 instead of 6 % of the FP64 work.)
// Products (PART = false): a cluster of S CTAs shares a tile; CTA s sums K slab
// s, and the slab sums are added in slab order through distributed shared
// memory.  Partial sums (PART = true, C = A^T B of a few columns): CTA (pair,
// slab) writes its tile of slab's M x N sum; tiles are the pairs (i, j) of
// equal column chunks, with sym only j >= i.
// The FP64 units do two DFMA per clock and SM, so an FP64 product is bound by
// them (1.19 TFLOP/s); neighbouring CTAs of an SM hide the loads.
struct FitShape {
  int bm, bn;     // tile
  int nch, nchm;  // column chunks, row chunks (partial sums)
  int64_t kslab;  // K per slab
  int S;          // slabs (products: CTAs per cluster)
  bool sym;
};
constexpr int FIT_BN = 64;       // widest tile of a product
constexpr int FIT_BN_PART = 44;  // ... of a partial sum (square tiles)
constexpr int FIT_BK = 32;       // K per staged block

template <int N>
__device__ __forceinline__ void fit_ld(const double* p, double (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; i += 2) {
    const double2 x = *reinterpret_cast<const double2*>(p + i);
    v[i] = x.x;
    v[i + 1] = x.y;
  }
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

template <bool TRANS_A, typename T, int MI, int NI, bool PART, int BL>
__global__ void __launch_bounds__(512)
k_fit(const T* __restrict__ A, int64_t lda, const T* __restrict__ B, int64_t ldb,
      double* __restrict__ C, int64_t ldc, int64_t M, int64_t K, int64_t N, FitShape f,
      const int32_t* __restrict__ gate) {
  constexpr int BK = FIT_BK, PAD = 2;  // rows stay on 16 bytes
  extern __shared__ __align__(16) unsigned char fit_smem[];
  if (gate != nullptr && *gate == 0) return;  // (the same for a whole cluster)
  const int bm = f.bm, bn = f.bn, t = threadIdx.x, nt = blockDim.x;
  const int pa = bm + PAD, pb = bn + PAD;
  double* As = reinterpret_cast<double*>(fit_smem);  // [BK][pa]
  double* Bs = As + BK * pa;                     // [BK][pb]
  // the block is a multiple of 32 threads: those past the tile only load
  const int nx = bn / NI;
  const bool live = t < (bm / MI) * nx;
  const int tx = live ? t % nx : 0, ty = live ? t / nx : 0;
  int64_t m0, n0;
  int slab;
  if (PART) {
    int i = 0, j = blockIdx.x;
    if (f.sym) {
      while (j >= f.nch - i) { j -= f.nch - i; ++i; }
      j += i;
    } else {
      i = j / f.nch;
      j -= i * f.nch;
    }
    m0 = (int64_t)i * bm;
    n0 = (int64_t)j * bn;
    slab = blockIdx.y;
  } else {
    m0 = (int64_t)(blockIdx.x / f.S) * bm;
    n0 = (int64_t)blockIdx.y * bn;
    slab = blockIdx.x % f.S;  // rank in the cluster
  }
  const int64_t kz0 = (int64_t)slab * f.kslab, kz1 = min(K, kz0 + f.kslab);
  const int warp = t >> 5, lane = t & 31, nw = nt >> 5;
  double acc[MI][NI];
#pragma unroll
  for (int i = 0; i < MI; ++i)
#pragma unroll
    for (int j = 0; j < NI; ++j) acc[i][j] = 0.0;
  for (int64_t k0 = kz0; k0 < kz1; k0 += BK) {
    if (TRANS_A) {  // a warp per k, lanes along m
#pragma unroll 4
      for (int c = warp; c < BK; c += nw)
        for (int r = lane; r < bm; r += 32)
          As[c * pa + r] = (m0 + r < M && k0 + c < kz1) ? (double)(A[(k0 + c) * lda + m0 + r])
                                                        : 0.0;
    } else {  // 16 consecutive k per row
      for (int e = t; e < bm * BK; e += nt) {
        const int r = e / BK, c = e % BK;
        As[c * pa + r] = (m0 + r < M && k0 + c < kz1) ? (double)(A[(m0 + r) * lda + k0 + c])
                                                      : 0.0;
      }
    }
#pragma unroll 4
    for (int c = warp; c < BK; c += nw)
      for (int r = lane; r < bn; r += 32)
        Bs[c * pb + r] = (n0 + r < N && k0 + c < kz1) ? (double)(B[(k0 + c) * ldb + n0 + r])
                                                      : 0.0;
    __syncthreads();
    if (live) {
#pragma unroll 1
      for (int kb = 0; kb < BK; kb += BL) {
        double part[MI][NI];
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
          for (int j = 0; j < NI; ++j) part[i][j] = 0.0;
#pragma unroll 16
        for (int kk = kb; kk < kb + BL; ++kk) {
          double a[MI], b[NI];
          fit_ld(As + kk * pa + ty * MI, a);
          fit_ld(Bs + kk * pb + tx * NI, b);
#pragma unroll
          for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int j = 0; j < NI; ++j) part[i][j] = fma(a[i], b[j], part[i][j]);
        }
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
          for (int j = 0; j < NI; ++j) acc[i][j] += part[i][j];
      }
    }
    __syncthreads();
  }
  if (PART || f.S == 1) {
    double* Cz = PART ? C + (int64_t)slab * M * ldc : C;
    if (!live) return;
#pragma unroll
    for (int i = 0; i < MI; ++i) {
      const int64_t gm = m0 + ty * MI + i;
#pragma unroll
      for (int j = 0; j < NI; ++j) {
        const int64_t gn = n0 + tx * NI + j;
        if (gm < M && gn < N) Cz[gm * ldc + gn] = acc[i][j];
      }
    }
    return;
  }
  // slab sums to shared memory; CTA s adds the entries s, s + S, ... of all slabs
  double* W = reinterpret_cast<double*>(fit_smem);
  if (live) {
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
      for (int j = 0; j < NI; ++j) W[(ty * MI + i) * bn + tx * NI + j] = acc[i][j];
  }
  cluster_barrier();
  const uint32_t w0 = (uint32_t)__cvta_generic_to_shared(W);
  for (int e = t * f.S + slab; e < bm * bn; e += nt * f.S) {
    const int r = e / bn, c = e - r * bn;
    if (m0 + r >= M || n0 + c >= N) continue;
    double v[8];
#pragma unroll
    for (int z = 0; z < 8; ++z) {
      v[z] = 0.0;
      if (z < f.S) {
        uint32_t p;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                     : "=r"(p)
                     : "r"(w0 + e * (uint32_t)sizeof(double)), "r"(z));
        asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[z]) : "r"(p) : "memory");
      }
    }
    double s = v[0];
#pragma unroll
    for (int z = 1; z < 8; ++z)
      if (z < f.S) s += v[z];
    C[(m0 + r) * ldc + n0 + c] = s;
  }
  cluster_barrier();  // no CTA leaves while others read its slab
}

size_t fit_smem_bytes(const FitShape& f, bool reduce) {
  const size_t stage = (size_t)FIT_BK * (f.bm + f.bn + 4) * sizeof(double);
  return reduce ? std::max(stage, (size_t)f.bm * f.bn * sizeof(double)) : stage;
}

// Chunks of N columns: equal, at most `widest`, multiples of ni.
void fit_columns(int64_t N, int ni, int widest, FitShape& f) {
  f.nch = ceil_div(N, widest);
  f.bn = ceil_div(ceil_div(N, f.nch), ni) * ni;
}

// Chain length over K rows.  In units of a product's rounding error squared, K
// rows in chains of L and S slabs add K L / 2 + K^2 / (2 L S) + K S / 2 (the
// chains, their sums, the slab sums; eight slabs at a time in a Gram: K S / 16):
// 32 is no worse than the 64 x 64 tiles' 16 (with one slab, or a Gram's few)
// from about 544 rows on in a product, 2048 in a Gram.
int fit_chain(int64_t K, bool gram) { return K >= (gram ? 2048 : 544) ? 32 : 16; }

int fit_threads(const FitShape& f, int mi, int ni) {
  return ceil_div((f.bm / mi) * (f.bn / ni), 32) * 32;
}

// A product: the tile rows and the K split are taken that leave the fullest SM
// the least work, the CTAs (ceil(M / bm) nch S of bm bn K / S multiply-adds)
// being dealt evenly.  8192 x 4096 at d = 72: 9.49 ms in 64 x 64 tiles of all K
// (128 padded columns), 4.41 ms in 64 x 36 tiles and 8 slabs (1.10 TFLOP/s of
// the 1.19 the FP64 units do, and the additions of the chains); 1000 x 800 at d = 30: 990 us (16 CTAs) to 76 us.
template <bool TRANS_A>
cudaError_t fit_launch(const double* A, int64_t lda, const double* B, int64_t ldb, double* C,
                       int64_t ldc, int64_t M, int64_t K, int64_t N, const int32_t* gate,
                       cudaStream_t st) {
  constexpr int MI = 4, NI = 2;
  if (M <= 0 || N <= 0) return cudaSuccess;
  FitShape f{};
  fit_columns(N, NI, FIT_BN, f);
  const int64_t P = sm_count();
  double best = 1e300;
  for (int b = 16 * MI; b >= 4 * MI; b /= 2) {
    for (int s = 1; s <= 8; s *= 2) {
      if (s > 1 && K < (int64_t)64 * s) break;
      const int64_t units = (int64_t)ceil_div(M, b) * f.nch * s;
      // shorter tiles load more per multiply-add (measured at 8192 x 4096, d =
      // 72, in 8 slabs: 4.26, 4.79 and 5.57 ms with 64, 32 and 16 rows); one CTA
      // per SM waits for its loads (1000 x 800, d = 30: 184 us with 128 CTAs of
      // 64 rows, 121 with 256 of 32)
      const double cost = (double)((units + P - 1) / P) * b / s *
                          (b == 16 * MI ? 1.0 : b == 8 * MI ? 1.11 : 1.3) *
                          (units <= P ? 1.5 : 1.0);
      if (cost < best * 0.999) {
        best = cost;
        f.bm = b;
        f.S = s;
      }
    }
  }
  f.kslab = ((K + f.S - 1) / f.S + FIT_BK - 1) / FIT_BK * FIT_BK;
  const size_t sm = fit_smem_bytes(f, f.S > 1);
  auto kern = fit_chain(K, false) == 32 ? k_fit<TRANS_A, double, MI, NI, false, 32>
                                        : k_fit<TRANS_A, double, MI, NI, false, 16>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(ceil_div(M, f.bm) * f.S), f.nch);
  cfg.blockDim = dim3(fit_threads(f, MI, NI));
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim = {(unsigned)f.S, 1, 1};
  cfg.attrs = attr;
  cfg.numAttrs = f.S > 1 ? 1 : 0;
  e = cudaLaunchKernelEx(&cfg, kern, A, lda, B, ldb, C, ldc, M, K, N, f, gate);
  count_launch();
  return e == cudaSuccess ? cudaGetLastError() : e;
}

// C[i][j] = sum_z P[z][i][j] in z order (deterministic), cast to TC.
// sym: only the entries with j >= i were formed.  TREE: eight slabs are added in
// pairs first (FP64 Grams, whose error many slabs added in turn would carry).
template <typename TC, bool TREE = false>
__global__ void k_reduce_partials(const double* __restrict__ P, int splits, int64_t M, int64_t N,
                                  TC* __restrict__ C, int64_t ldc,
                                  const int32_t* __restrict__ gate, bool sym = false) {
  if (gate != nullptr && *gate == 0) return;
  int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= M * N) return;
  const int64_t i = idx / N, j = idx % N;
  if (sym && j < i) idx = j * N + i;
  double s = 0.0;  // split order, eight independent loads in flight
  int z = 0;
  if constexpr (TREE) {
    for (; z < splits; z += 8) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = z + u < splits ? P[(int64_t)(z + u) * M * N + idx] : 0.0;
      s += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
  }
  for (; z + 8 <= splits; z += 8) {
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = P[(int64_t)(z + u) * M * N + idx];
#pragma unroll
    for (int u = 0; u < 8; ++u) s += v[u];
  }
  for (; z < splits; ++z) s += P[(int64_t)z * M * N + idx];
  C[i * ldc + j] = Cvt<TC>::from(s);
}

// C = A^T B (FP64 sums; M x N small) in `splits` K slabs, or its upper
// triangle's tiles mirrored when A = B: the square tiles' chunks fit N (one of
// 30 columns at d = 30, five of 44 at d = 220), half of the off-diagonal work
// is left out.
template <typename T, typename TC>
cudaError_t fit_partial(const void* A, int64_t lda, const void* B, int64_t ldb, void* C,
                        int64_t ldc, int64_t M, int64_t K, int64_t N, int splits, double* partial,
                        const int32_t* gate, cudaStream_t st) {
  FitShape f{};
  fit_columns(N, 2, FIT_BN_PART, f);
  f.bm = f.bn;
  f.nchm = ceil_div(M, f.bm);
  f.sym = A == B && lda == ldb && M == N;
  f.kslab = ((K + splits - 1) / splits + 15) / 16 * 16;
  f.S = (int)((K + f.kslab - 1) / f.kslab);
  const size_t sm = fit_smem_bytes(f, false);
  const int pairs = f.sym ? f.nch * (f.nch + 1) / 2 : f.nchm * f.nch;
  auto kern = fit_chain(K, true) == 32 ? k_fit<true, T, 2, 2, true, 32>
                                       : k_fit<true, T, 2, 2, true, 16>;
  kern<<<dim3(pairs, f.S), fit_threads(f, 2, 2), sm, st>>>((const T*)A, lda, (const T*)B, ldb,
                                                           partial, N, M, K, N, f, gate);
  count_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_reduce_partials<TC, true><<<ceil_div(M * N, 256), 256, 0, st>>>(partial, f.S, M, N, (TC*)C, ldc,
                                                                    gate, f.sym);
  count_launch();
  return cudaGetLastError();
}

template <bool TRANS_A, typename TA, typename TB, typename TC, Mul MODE>
cudaError_t launch(const void* A, int64_t lda, const void* B, int64_t ldb, void* C, int64_t ldc,
                   int64_t M, int64_t K, int64_t N, int splits, double* partial,
                   const int32_t* gate, cudaStream_t st, const int32_t* redo = nullptr) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (splits < 1) splits = 1;
  int64_t kslab = ((K + splits - 1) / splits + BK - 1) / BK * BK;
  if (kslab < BK) kslab = BK;
  splits = (int)((K + kslab - 1) / kslab);
  if (splits < 1) splits = 1;
  dim3 grid(ceil_div(M, BM), ceil_div(N, BN), splits);
  if (splits == 1) {
    k_gemm<TRANS_A, TA, TB, TC, MODE, false><<<grid, NT, 0, st>>>(
        (const TA*)A, lda, (const TB*)B, ldb, (TC*)C, ldc, M, K, N, kslab, gate, redo);
    count_launch();
    return cudaGetLastError();
  }
  k_gemm<TRANS_A, TA, TB, double, MODE, true><<<grid, NT, 0, st>>>(
      (const TA*)A, lda, (const TB*)B, ldb, partial, N, M, K, N, kslab, gate, redo);
    count_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int64_t tot = M * N;
  k_reduce_partials<TC><<<ceil_div(tot, 256), 256, 0, st>>>(partial, splits, M, N, (TC*)C, ldc, gate);
    count_launch();
  return cudaGetLastError();
}

}  // namespace

int tn_splits(int64_t M, int64_t K, int64_t N, int max_splits) {
  const int64_t tiles = (int64_t)ceil_div(M, BM) * ceil_div(N, BN);
  int64_t s = (4 * 152 + tiles - 1) / tiles;  // about four CTAs per SM
  const int64_t kmax = (K + BK - 1) / BK;     // at least 16 rows per slab
  if (s > kmax) s = kmax;
  if (s > max_splits) s = max_splits;
  if (s < 1) s = 1;
  return (int)s;
}

#define RUQLP_DISPATCH(TRANS, TA_, TB_, TC_, MODE_, CTA, CTB, CTC)                         \
  if (ta == TA_ && tb == TB_ && tc == TC_ && mul == MODE_)                                 \
    return launch<TRANS, CTA, CTB, CTC, MODE_>(A, lda, B, ldb, C, ldc, M, K, N, splits,    \
                                               partial, gate, st, redo);

cudaError_t simt_gemm_nn(Ty ta, Ty tb, Ty tc, Mul mul, const void* A, int64_t lda,
                         const void* B, int64_t ldb, void* C, int64_t ldc, int64_t M,
                         int64_t K, int64_t N, cudaStream_t st, const int32_t* redo) {
  const int splits = 1;
  double* partial = nullptr;
  const int32_t* gate = nullptr;
  if (ta == Ty::F64 && tb == Ty::F64 && tc == Ty::F64 && mul == Mul::F64)
    return fit_launch<false>((const double*)A, lda, (const double*)B, ldb, (double*)C, ldc, M, K, N,
                                                                     gate, st);
  RUQLP_DISPATCH(false, Ty::F32, Ty::F32, Ty::F32, Mul::F32, float, float, float)
  RUQLP_DISPATCH(false, Ty::BF16, Ty::F32, Ty::F32, Mul::F32, __nv_bfloat16, float, float)
  RUQLP_DISPATCH(false, Ty::BF16, Ty::BF16, Ty::F32, Mul::F32, __nv_bfloat16, __nv_bfloat16, float)
  RUQLP_DISPATCH(false, Ty::F32, Ty::F32, Ty::F32, Mul::F32_ACC64, float, float, float)
  return cudaErrorInvalidValue;
}

int bgemm_tiles(int64_t rows, int d) { return ceil_div(rows, BM) * ceil_div(d, BN); }

cudaError_t bgemm(bool trans, Ty ta, Ty tb, const BMat* T, const int* prefix, int total, int count,
                  int src, int dst, cudaStream_t st, bool split2) {
  if (total <= 0) return cudaSuccess;
  if (tb == Ty::F32) {
    if (ta == Ty::F32) {
      if (trans) k_bgemm<true, float, float><<<total, NT, 0, st>>>(T, prefix, count, src, dst);
      else k_bgemm<false, float, float><<<total, NT, 0, st>>>(T, prefix, count, src, dst);
    } else if (ta == Ty::BF16) {
      if (trans && split2)
        k_bgemm<true, __nv_bfloat16, float, 1><<<total, NT, 0, st>>>(T, prefix, count, src, dst);
      else if (trans) k_bgemm<true, __nv_bfloat16, float><<<total, NT, 0, st>>>(T, prefix, count, src, dst);
      else if (split2)
        k_bgemm<false, __nv_bfloat16, float, 1><<<total, NT, 0, st>>>(T, prefix, count, src, dst);
      else k_bgemm<false, __nv_bfloat16, float><<<total, NT, 0, st>>>(T, prefix, count, src, dst);
    } else {
      return cudaErrorInvalidValue;
    }
  } else {
    return cudaErrorInvalidValue;
  }
  count_launch();
  return cudaGetLastError();
}

cudaError_t simt_gemm_tn(Ty ta, Ty tb, Ty tc, Mul mul, const void* A, int64_t lda,
                         const void* B, int64_t ldb, void* C, int64_t ldc, int64_t M,
                         int64_t K, int64_t N, int splits, double* partial,
                         const int32_t* gate, cudaStream_t st, const int32_t* redo) {
  if (splits > 1 && partial == nullptr) return cudaErrorInvalidValue;
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (splits > 1 && mul == Mul::F64 && tc == Ty::F64 && ta == tb && ta != Ty::BF16)
    return ta == Ty::F64 ? fit_partial<double, double>(A, lda, B, ldb, C, ldc, M, K, N, splits,
                                                       partial, gate, st)
                         : fit_partial<float, double>(A, lda, B, ldb, C, ldc, M, K, N, splits,
                                                      partial, gate, st);
  if (ta == Ty::F64 && tb == Ty::F64 && tc == Ty::F64 && mul == Mul::F64)
    return fit_launch<true>((const double*)A, lda, (const double*)B, ldb, (double*)C, ldc, M, K, N,
                                                                    gate, st);
  RUQLP_DISPATCH(true, Ty::F32, Ty::F32, Ty::F32, Mul::F32, float, float, float)
  RUQLP_DISPATCH(true, Ty::BF16, Ty::F32, Ty::F32, Mul::F32, __nv_bfloat16, float, float)
  RUQLP_DISPATCH(true, Ty::BF16, Ty::BF16, Ty::F32, Mul::F32, __nv_bfloat16, __nv_bfloat16, float)
  RUQLP_DISPATCH(true, Ty::F32, Ty::F32, Ty::F64, Mul::F32_ACC64, float, float, double)
  RUQLP_DISPATCH(true, Ty::F32, Ty::F32, Ty::F64, Mul::F64, float, float, double)
  return cudaErrorInvalidValue;
}

}  // namespace ruqlp
