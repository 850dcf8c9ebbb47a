// FP32 products of RU-QLP on the tensor cores (Section III-D: the O(mnd)
// passes A X and A^T Y of an FP32 matrix):
//
//   out[m x dp] = A[m x n] X       (A K-major)
//   out[n x dp] = A^T[n x m] X     (A MN-major)
//
// Every FP32 value is split on the fly into three BF16 parts, x = h + m + l
// exactly (h and m rounded to nearest, l the rest: 8 + 8 + 7 significant bits),
// and a x is formed as the six part products
//   l h + h l + m m + m h + h m + h h
// (the dropped m l, l m, l l are below 2^-25 |a x|), accumulated in FP32.
//
// Accumulation: tcgen05.mma adds into TMEM with truncation (measured on the
// BF16 products: a relative bias of about 2e-8 per instruction that adds to a
// full-size accumulator), so a K-long accumulation there would lose FP32
// accuracy.  Each 32-row K block therefore gets a fresh accumulator, its small
// part products first and the two h h instructions last, and the epilogue
// warps add the block sums in FP32 (round to nearest) registers.
//
// One CTA per SM, four warpgroups:
//   warpgroup 0     warp 0: TMEM allocation and tcgen05.mma issue (one lane);
//                   warp 1: bulk copies of the split X (one lane);
//   warpgroups 1-2  copy FP32 blocks of A four ahead (cp.async), split them
//                   and write the parts into a swizzled shared-memory ring;
//   warpgroup 3     reads each block's accumulator (two TMEM buffers of 256
//                   columns) and adds it to 224 registers per thread.
// X is split once per product into an image of the X stages (k_f32_split) when
// the workspace has room for it (a handle without a memory budget); else the
// converters of every CTA split it too, with the same parts and result.
// Registers are moved from the first three warpgroups to the last one with
// setmaxnreg.  Output items are 128 rows x at most 224 columns; whole waves of
// items first, then the items of the last partial wave split along K into
// slabs summed in order by k_f32_fixup (the split is a function of the shape,
// so an item's result is the same alone and in a batch).
//
// Range: the split is exact for 2^-110 <= |x| < 2^127, and FP32 products and
// sums behave as on the CUDA cores while nothing comes near FP32's limits.
// The converters note values that are not finite, at least 2^60 or (nonzero)
// below 2^-100, and nonzero values below 2^-50; the epilogue notes nonzero
// results below 2^-70 and zeros.  The first, or the second and third together,
// make the CUDA-core kernel that follows form the product again; the second and
// the zeros together make it look at the zeros, whose row of A and column of X
// say whether products may have underflowed there, and form the tiles again in
// which they may (DevStatus::range; set-only bits, read after the launch, so the
// choice is deterministic).  8192 x 8192 with a zero row and an element of 2^-60
// elsewhere, d = 200: 4059 us for the call when a zero counted as a tiny result,
// 470 now (295 without the element; the CUDA cores alone 3785).
//
// Bound: at wide sketches the tensor cores and their operands' shared memory (a
// 32-deep block at 224 columns is 1344 clocks of tensor work and 132 KB of operand
// reads, beside the parts' writes; measured 1960 clocks a block at K = 20000; at K
// = 2048, launch and drain included, the tensor pipe is active 55 % and the LSU's
// shared-memory pipe 33 % of the time), HBM at narrow ones.  A^T X of a 20000 x
// 20000 matrix at d = 220: 0.66 ms (1.06 TFLOP of part products at 1.6 PFLOP/s)
// against 15.7 ms on the CUDA cores; the relative error against FP64 4.5e-7
// against 6.4e-7.  Measured slower: FP32
// blocks through registers (2.8k clocks a block whatever its width: the loads
// were waited for as soon as they were issued), X split by every CTA's
// converters (1.04 ms), eight accumulator columns per TMEM load (3.9k clocks of
// epilogue a block at 224 columns against 1.65k with sixteen).
#include <algorithm>

#include "internal.h"
#include "tcgen05.cuh"

namespace ruqlp {
namespace {

constexpr int FT_THREADS = 512;
constexpr int FT_CT = 256;                       // converter threads
constexpr int FT_CW = FT_CT / 32;                // converter warps
constexpr uint32_t FT_APART = F32_BM * F32_BK * 2;  // one part of an A block
constexpr uint32_t FT_BOX = F32_BOX;
constexpr int FT_NA = 2;                         // stages of split A blocks
constexpr int FT_NC = F32_WMAX / 16;             // accumulator chunks per thread
constexpr int FT_XV = F32_BK * F32_WMAX / 4 / FT_CT;  // X float4s per thread and block
constexpr int FT_AHEAD = 4;                      // A blocks in flight per CTA
constexpr uint32_t FT_RAW = F32_BM * F32_BK * 4; // one raw A block
constexpr int FT_SP = 20;                        // epilogue staging pitch (floats)
constexpr uint32_t FT_STG = 4 * 32 * FT_SP * 4;
constexpr int FT_REG_CTL = 56, FT_REG_CONV = 104, FT_REG_EPI = 248;

// One unit of work: a 128-row output tile, columns [col0, col0 + w), K blocks
// [kb0, kb1).
struct FtUnit {
  const float* A;
  int64_t lda, rows, K;  // A's row stride; output rows; contraction length
  const float* X;        // K x d, ld ldx
  int64_t ldx;
  const uint8_t* img;    // split X: the stage of K block 0 of this column chunk (or null)
  int d, xcols;          // columns; columns of X that may be read (a multiple of 4)
  int col0, w, xw, tile, kb0, kb1;  // xw: the chunk width (the image's stages)
  float* out;            // the tile's first row, first column
  int ocols;             // columns of the chunk that are stored
  int64_t ldo;
  bool vec;              // A's rows start on 16 bytes
  DevStatus* st;
};

struct FtParams {
  const float* A;
  int64_t lda, rows, K;
  const float* X;
  int64_t ldx;
  const uint8_t* img;
  float* out;
  int64_t ldo;
  float* frag;
  int d, xcols, ocols, dp, vec;
  F32Split sp;
  DevStatus* st;  // null: no range notes
  int* err;
};

__device__ __forceinline__ void ft_columns(const F32Split& sp, int item, int dp, FtUnit& u) {
  u.tile = item / sp.nch;
  u.col0 = (item - u.tile * sp.nch) * sp.w;
  u.w = min(sp.w, dp - u.col0);
  u.xw = sp.w;
}

// Single matrix: CTA c takes items c, c + P, ... of the whole waves, then one
// slab of a tail item.
struct FtSingle {
  const FtParams* p;
  static constexpr bool kEmpty = false;  // units without K blocks
  // A product that an operand outside the split's range sends to the CUDA cores is
  // given up where one is met, and by the other CTAs when they see the note.
  static constexpr bool kGiveUp = true;
  __device__ bool skip() const {
    return p->st != nullptr && range_redo(*(volatile int32_t*)&p->st->range);
  }
  __device__ int count() const {
    const F32Split& sp = p->sp;
    return sp.full_waves + ((int)blockIdx.x < sp.tail * sp.S ? 1 : 0);
  }
  __device__ FtUnit get(int i) const {
    const F32Split& sp = p->sp;
    const int c = blockIdx.x;
    FtUnit u;
    u.A = p->A;
    u.lda = p->lda;
    u.rows = p->rows;
    u.K = p->K;
    u.X = p->X;
    u.ldx = p->ldx;
    u.d = p->d;
    u.xcols = p->xcols;
    u.vec = p->vec != 0;
    u.st = p->st;
    int s = 0, S = 1, item = c + i * sp.P;
    if (i >= sp.full_waves) {
      S = sp.S;
      item = sp.full_waves * sp.P + c / S;
      s = c % S;
    }
    ft_columns(sp, item, p->dp, u);
    u.img = p->img == nullptr
                ? nullptr
                : p->img + (int64_t)(u.col0 / sp.w) * sp.KB * f32_xstage(sp.w);
    u.kb0 = (int)((int64_t)sp.KB * s / S);
    u.kb1 = (int)((int64_t)sp.KB * (s + 1) / S);
    u.ocols = u.w;
    if (S == 1) {
      u.out = p->out + (int64_t)u.tile * F32_BM * p->ldo + u.col0;
      u.ldo = p->ldo;
      u.ocols = min(u.w, p->ocols - u.col0);
    } else {
      u.out = p->frag + (int64_t)c * F32_BM * sp.w;
      u.ldo = sp.w;
    }
    return u;
  }
};

// An item's index among the tail items (past the whole waves of `sms` items).
__device__ __forceinline__ int tail_index_of(int64_t rows, int nch, int item, int sms) {
  const int items = (int)((rows + F32_BM - 1) / F32_BM) * nch;
  return item - items / sms * sms;
}

// Batch: CTA c takes entries c, c + P, ... of a host-built list.  An item of which a
// product was left to the CUDA cores whole has f32_k = 0 from then on: its units
// have no K blocks, so its later products cost no second attempt (eight 2048 x
// 1024 items with an element of 2^-110, d = 72, q = 2: 3580 us with one per
// product, 3000 now, 3040 on the CUDA cores alone).
struct FtBatch {
  const F32Tile* list;
  int n;
  const BMat* T;
  int src, dst, sms;
  bool trans;
  static constexpr bool kEmpty = true;
  static constexpr bool kGiveUp = false;  // (the CTA's next item may be another matrix)
  __device__ bool skip() const { return false; }
  __device__ int tail_index(int64_t rows, int nch, int item) const {
    return tail_index_of(rows, nch, item, sms);
  }
  __device__ int count() const {
    return (int)blockIdx.x < n ? (n - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  }
  __device__ FtUnit get(int i) const {
    const F32Tile e = list[blockIdx.x + (int64_t)i * gridDim.x];
    const BMat& b = T[e.mat()];
    FtUnit u;
    u.A = (const float*)b.A;
    u.lda = b.lda;
    u.rows = trans ? b.n : b.m;
    u.K = b.f32_k[trans];
    u.X = bbuf(b, src);
    u.ldx = b.dp;
    u.d = b.d;
    u.xcols = b.dp;
    u.vec = (b.lda & 3) == 0 && ((uintptr_t)b.A & 15) == 0;
    u.st = b.status;
    const F32Split sp = f32_columns(b.dp);
    const int KB = (int)((u.K + F32_BK - 1) / F32_BK);
    ft_columns(sp, e.item(), b.dp, u);
    u.img = b.Bt == nullptr
                ? nullptr
                : (const uint8_t*)b.Bt + (int64_t)(u.col0 / sp.w) * KB * f32_xstage(sp.w);
    const int s = e.s(), S = e.S();
    u.ocols = u.w;
    u.kb0 = (int)((int64_t)KB * s / S);
    u.kb1 = (int)((int64_t)KB * (s + 1) / S);
    if (S == 1) {
      u.out = bbuf(b, dst) + (int64_t)u.tile * F32_BM * b.dp + u.col0;
      u.ldo = b.dp;
    } else {
      u.out = (float*)b.partial + (int64_t)(tail_index(u.rows, sp.nch, e.item()) * S + s) * F32_BM * sp.w;
      u.ldo = sp.w;
    }
    return u;
  }
};

__device__ __forceinline__ void add2(float& a, float& b, float x, float y) {
  asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %3};\n\t"
      "add.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
      : "+f"(a), "+f"(b)
      : "f"(x), "f"(y));
}

// The three parts of four consecutive values at shared address a, a + pitch,
// a + 2 pitch (8 bytes each).
__device__ __forceinline__ void put4(uint32_t a, uint32_t pitch, const float4& v) {
  uint32_t h[2], m[2], l[2];
  split3(make_float2(v.x, v.y), h[0], m[0], l[0]);
  split3(make_float2(v.z, v.w), h[1], m[1], l[1]);
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(h[0]), "r"(h[1]) : "memory");
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a + pitch), "r"(m[0]), "r"(m[1])
               : "memory");
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a + 2 * pitch), "r"(l[0]), "r"(l[1])
               : "memory");
}

__device__ __forceinline__ void note(DevStatus* st, int32_t bits) {
  if (st != nullptr && (*(volatile int32_t*)&st->range & bits) != bits) atomicOr(&st->range, bits);
}
// Magnitudes met: the largest |x| (NaN kept) and the smallest nonzero one as
// twice its bits less one (zero wraps to the top, so it never counts as small).
struct Range {
  float hi = 0.f;
  uint32_t lo = 0xFFFFFFFFu;
  __device__ __forceinline__ static float top(float a, float b) {
    float r;
    asm("{\n\t.reg .f32 x;\n\tabs.f32 x, %2;\n\tmax.NaN.f32 %0, %1, x;\n\t}"
        : "=f"(r)
        : "f"(a), "f"(b));
    return r;
  }
  __device__ __forceinline__ static uint32_t key(float x) {
    const uint32_t u = __float_as_uint(x);
    return u + u - 1u;
  }
  __device__ __forceinline__ void add(const float4& v) {
    hi = top(top(top(top(hi, v.x), v.y), v.z), v.w);
    lo = min(lo, min(key(v.x), key(v.y)));
    lo = min(lo, min(key(v.z), key(v.w)));
  }
  // (returns whether a value outside the split's range was noted)
  __device__ __forceinline__ bool tell(DevStatus* st) const {
    const bool off = !(hi < 1.152921504606846976e18f) || lo < 2u * 0x0D800000u - 1u;
    if (off) note(st, RANGE_OFF);
    if (lo < 2u * 0x26800000u - 1u) note(st, RANGE_SMALL);
    return off && st != nullptr;
  }
};

// v = four values at p if `in`, else zeros (a predicated load: no branch whose
// merge would wait for the data).
__device__ __forceinline__ void load4_if(float4& v, const float* p, bool in) {
  v = make_float4(0.f, 0.f, 0.f, 0.f);
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %5, 0;\n\t"
      "@p ld.global.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
      : "+f"(v.x), "+f"(v.y), "+f"(v.z), "+f"(v.w)
      : "l"(p), "r"((int)in));
}

// The columns from d on of four values at column c are zero (an arena buffer's
// padding columns may hold anything).
__device__ __forceinline__ void mask4(float4& v, int c, int d) {
  if (c + 1 > d) v.x = 0.f;
  if (c + 2 > d) v.y = 0.f;
  if (c + 3 > d) v.z = 0.f;
  if (c + 4 > d) v.w = 0.f;
}

// Converter thread ct's place in an X block: row k, columns c + 32 q ...  A
// warp's four rows are 4 apart in pairs, so that its 8-byte stores cover both
// halves of the swizzled lines; off(q): the byte offset within a part.
struct XPlace {
  int k, c;
  __device__ __forceinline__ explicit XPlace(int ct) {
    const int cw = ct >> 5, lane = ct & 31;
    k = (cw & 3) + 8 * (cw >> 2) + 4 * ((lane >> 3) & 1) + 16 * (lane >> 4);
    c = (lane & 7) * 4;
  }
  __device__ __forceinline__ uint32_t off(int q) const {
    return f32_img_off(k, c + 32 * q);
  }
};

// X (K x d) split into the image of its stages: block (kb, chunk) writes the
// three parts of K block kb, columns [w chunk, w chunk + w) (zero past d and
// K).  Bandwidth-bound: 4 bytes read and 6 written per value.
__device__ __forceinline__ void split_block(const float* X, int64_t ldx, int64_t K, int d,
                                            int xcols, int kb, int col0, int w, uint8_t* img, DevStatus* st) {
  const XPlace xp(threadIdx.x);
  const int64_t row = (int64_t)kb * F32_BK + xp.k;
  const uint32_t part = f32_xstage(w) / 3;
  Range rx;
  for (int q = 0; 32 * q < (w + 63) / 64 * 64; ++q) {
    const int c = xp.c + 32 * q;
    float4 v;
    load4_if(v, X + row * ldx + col0 + c, row < K && c < w && col0 + c < xcols);
    mask4(v, col0 + c, d);
    rx.add(v);
    uint32_t h[2], m[2], l[2];
    split3(make_float2(v.x, v.y), h[0], m[0], l[0]);
    split3(make_float2(v.z, v.w), h[1], m[1], l[1]);
    uint8_t* o = img + xp.off(q);
    *reinterpret_cast<uint2*>(o) = make_uint2(h[0], h[1]);
    *reinterpret_cast<uint2*>(o + part) = make_uint2(m[0], m[1]);
    *reinterpret_cast<uint2*>(o + 2 * part) = make_uint2(l[0], l[1]);
  }
  rx.tell(st);
}

__global__ void __launch_bounds__(FT_CT) k_f32_split(const __grid_constant__ FtParams p) {
  pdl_launch();
  pdl_wait();
  const uint32_t xs = f32_xstage(p.sp.w);
  split_block(p.X, p.ldx, p.K, p.d, p.xcols, blockIdx.x, blockIdx.y * p.sp.w, p.sp.w,
              const_cast<uint8_t*>(p.img) + ((int64_t)blockIdx.y * p.sp.KB + blockIdx.x) * xs,
              p.st);
}

// Batch: block (x, i) takes K block x (and every gridDim.x after) of item i.
__global__ void __launch_bounds__(FT_CT) k_bf32_split(const BMat* __restrict__ T, int src) {
  const BMat& b = T[blockIdx.y];
  if (!(b.flags & (src == B_Y ? BM_F32_ATY : BM_F32_AX))) return;
  const F32Split sp = f32_columns(b.dp);
  const int64_t K = b.f32_k[src == B_Y];
  const int KB = (int)((K + F32_BK - 1) / F32_BK);
  for (int x = blockIdx.x; x < KB * sp.nch; x += gridDim.x) {
    const int ch = x / KB, kb = x - ch * KB;
    split_block(bbuf(b, src), b.dp, K, b.d, b.dp, kb, ch * sp.w, sp.w,
                (uint8_t*)b.Bt + (int64_t)x * f32_xstage(sp.w), b.status);
  }
}

// wmax sizes the X stages; each unit's own width sets its MMA N.  IMG: X comes
// split (u.img).
template <bool TRANS, bool IMG, class W>
__device__ __forceinline__ void ft_body(const W& w, int NX, int wmax, int* err) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - raw);
  // shared memory: split A stages, split X stages, raw A blocks, the epilogue's
  // staging, barriers
  // fa / ea (A full: converter warps; empty: MMA commit), fx / ex (X), tfull,
  // tempty, drain; then the TMEM address
  const uint32_t xstage = f32_xstage(wmax), xpart = xstage / 3;
  const uint32_t x_base = base + FT_NA * 3 * FT_APART;
  const uint32_t raw_base = x_base + NX * xstage;
  const uint32_t stg_base = raw_base + FT_AHEAD * FT_RAW;
  const uint32_t bar = stg_base + FT_STG;
  auto fa = [&](int i) { return bar + 8u * i; };
  auto ea = [&](int i) { return bar + 8u * (FT_NA + i); };
  auto fx = [&](int i) { return bar + 8u * (2 * FT_NA + i); };
  auto ex = [&](int i) { return bar + 8u * (2 * FT_NA + NX + i); };
  auto tfull = [&](int a) { return bar + 8u * (2 * FT_NA + 2 * NX + a); };
  auto tempty = [&](int a) { return bar + 8u * (2 * FT_NA + 2 * NX + 2 + a); };
  const uint32_t drain = bar + 8u * (2 * FT_NA + 2 * NX + 4);
  uint32_t* tmem_slot = (uint32_t*)(base_ptr + (drain + 8 - base));
  __shared__ int s_abort, s_skip;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, wg = warp >> 2;
  if (t == 0) {
    for (int i = 0; i < FT_NA; ++i) {
      mbar_init(fa(i), FT_CW);
      mbar_init(ea(i), 1);
    }
    for (int i = 0; i < NX; ++i) {
      mbar_init(fx(i), IMG ? 1 : FT_CW);
      mbar_init(ex(i), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull(a), 1);
      mbar_init(tempty(a), 4);
    }
    mbar_init(drain, 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                     smem_u32(tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  volatile int* abort_flag = &s_abort;
  // why the CTA's roles stop early: a wait ran out (the error word is set), or the
  // product is given up
  constexpr int TIMED_OUT = 1, GIVE_UP = 2;
  auto leave = [&]() {
    if (*abort_flag == 0) *abort_flag = TIMED_OUT;
  };
  pdl_launch();
  pdl_wait();
  // an earlier product of this run already asked for the CUDA cores (one thread
  // reads the word: other CTAs of this launch may be setting it)
  if (t == 0) s_skip = w.skip() ? 1 : 0;
  __syncthreads();
  const int nunits = s_skip ? 0 : w.count();

  if (wg == 0) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(FT_REG_CTL));
    if (warp == 0 && lane == 0) {
      // ---------------- MMA issuer ----------------
      bool ok = true;
      int sa = 0, sx = 0, it = 0;
      uint32_t pha = 0, phx = 0;
      // descriptors of the first A and X parts (offsets below 256 KB add to the
      // address field without carry).  K-major A: 64-byte rows, 64-byte
      // swizzle; MN-major: [32 k][64] boxes, 128-byte swizzle
      const uint64_t ad0 = TRANS ? sdesc(base, FT_BOX, 1024)
                                 : (sdesc(base, 16, 512) & ~(7ull << 61)) | (4ull << 61);
      const uint64_t xd0 = sdesc(x_base, FT_BOX, 1024);
      const uint64_t xstep = xpart >> 4;
      for (int i = 0; i < nunits && ok; ++i) {
        const FtUnit u = w.get(i);
        const uint32_t idesc = idesc_bf16(u.w, TRANS) | (1u << 16);  // X MN-major
        for (int kb = u.kb0; kb < u.kb1; ++kb, ++it) {
          const int acc = it & 1;
          if (!mbar_wait_inl(tempty(acc), (uint32_t)((it >> 1) & 1) ^ 1u, abort_flag) ||
              !mbar_wait_inl(fx(sx), phx, abort_flag) ||
              !mbar_wait_inl(fa(sa), pha, abort_flag)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t ad = ad0 + (uint64_t)((sa * 3 * FT_APART) >> 4);
          const uint64_t xd = xd0 + (uint64_t)((sx * xstage) >> 4);
          const uint32_t d = tmem_base + (uint32_t)(acc * 256);
          // small products first, h h last
          const int pa[6] = {2, 0, 1, 1, 0, 0}, px[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
          for (int q = 0; q < 6; ++q)
#pragma unroll
            for (int kk = 0; kk < F32_BK / 16; ++kk)
              mma_bf16(d, ad + ((pa[q] * FT_APART + kk * (TRANS ? 2048 : 32)) >> 4),
                       xd + px[q] * xstep + kk * (2048 >> 4), idesc,
                       (q > 0 || kk > 0) ? 1u : 0u);
          mma_commit(tfull(acc));
          mma_commit(ea(sa));
          mma_commit(ex(sx));
          if (++sa == FT_NA) { sa = 0; pha ^= 1u; }
          if (++sx == NX) { sx = 0; phx ^= 1u; }
        }
      }
      if (!ok) leave();
      // every MMA has completed before TMEM is freed
      mma_commit(drain);
      volatile int never = 0;
      mbar_wait_inl(drain, 0, &never);
    } else if (IMG && warp == 1 && lane == 0) {
      // ---------------- X producer ----------------
      bool ok = true;
      int sx = 0, issued = 0;
      uint32_t ph = 1;
      int32_t seen = 0;  // the run's range word as of the block before (not waited for)
      for (int i = 0; i < nunits && ok; ++i) {
        const FtUnit u = w.get(i);
        const uint32_t bytes = f32_xstage(u.xw);
        const uint32_t part = bytes / 3;
        const uint8_t* src = u.img + (int64_t)u.kb0 * bytes;
        for (int kb = u.kb0; kb < u.kb1; ++kb) {
          if (W::kGiveUp && (seen & RANGE_OFF)) {
            *abort_flag = GIVE_UP;
            ok = false;
            break;
          }
          if (W::kGiveUp && u.st != nullptr) seen = *(volatile int32_t*)&u.st->range;
          if (!mbar_wait_inl(ex(sx), ph, abort_flag)) {
            ok = false;
            break;
          }
          mbar_expect_tx(fx(sx), bytes);
#pragma unroll
          for (int q = 0; q < 3; ++q)
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes "
                "[%0], [%1], %2, [%3];" ::"r"(x_base + sx * xstage + q * xpart),
                "l"(src + q * part), "r"(part), "r"(fx(sx))
                : "memory");
          src += bytes;
          if (issued < NX) ++issued;
          if (++sx == NX) { sx = 0; ph ^= 1u; }
        }
      }
      if (!ok) leave();
      // the copies already issued land before the CTA gives up its shared memory
      // (also when none is left to issue: the other roles may stop before they use
      // them)
      for (; issued > 0; --issued) {
        if (sx == 0) { sx = NX; ph ^= 1u; }
        --sx;
        volatile int never = 0;
        mbar_wait_inl(fx(sx), ph ^ 1u, &never);
      }
    }
  } else if (wg < 3) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(FT_REG_CONV));
    // ---------------- converters ----------------
    const int ct = t - 128;
    // A: float4 q of a block is row (K-major) / k (MN-major) r0 + q * RS and
    // columns c0..c0+3 of it
    const int r0 = TRANS ? ct >> 5 : ct >> 3, c0 = TRANS ? (ct & 31) * 4 : (ct & 7) * 4;
    constexpr int RS = TRANS ? 8 : 32;
    // A's cursor runs FT_AHEAD blocks ahead of the one being converted, in a
    // ring of raw FP32 blocks that every thread fills with cp.async and reads
    // back itself (no barrier)
    const float *ap = nullptr, *a0 = nullptr;
    int64_t alda = 0;
    int anr = 0, anc = 0, akb = 0, akb1 = 0, ai = -1;  // rows / columns left from the block's first
    bool avec = false;
    const uint32_t raw_slot = raw_base + (uint32_t)ct * 16;
    // issue the next block's copies into a slot (one group per call, empty
    // past the end); zero-filled outside A
    auto fetch_a = [&](uint32_t slot) {
      bool any = true;
      if (akb == akb1) {
        if (++ai < nunits) {
          const FtUnit u = w.get(ai);
          akb = u.kb0;
          akb1 = u.kb1;
          alda = u.lda;
          avec = u.vec;
          const int m0 = u.tile * F32_BM, k0 = akb * F32_BK;
          a0 = u.A;
          ap = u.A + (int64_t)((TRANS ? k0 : m0) + r0) * u.lda + (TRANS ? m0 : k0) + c0;
          anr = (int)(TRANS ? u.K - k0 : u.rows - m0) - r0;
          anc = (int)(TRANS ? u.rows - m0 : u.K - k0) - c0;
          if (W::kEmpty) any = akb != akb1;  // (a unit without blocks takes a turn too)
        } else {
          any = false;
        }
      }
      if (any) {
        const uint32_t dst = raw_slot + slot * FT_RAW;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int in = q * RS < anr ? min(max(anc, 0), 4) : 0;
          const float* p = in > 0 ? ap + q * RS * alda : a0;
          if (avec) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                             dst + q * FT_CT * 16),
                         "l"(p), "r"(4 * in)
                         : "memory");
          } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                               dst + q * FT_CT * 16 + 4 * j),
                           "l"(j < in ? p + j : a0), "r"(j < in ? 4 : 0)
                           : "memory");
          }
        }
        ap += TRANS ? F32_BK * alda : F32_BK;
        (TRANS ? anr : anc) -= F32_BK;
        ++akb;
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    bool ok = true;
    int sa = 0, sx = 0;
    uint32_t pha = 1, phx = 1, slot = 0;
    const uint32_t aoff =
        TRANS ? (uint32_t)(c0 >> 6) * FT_BOX + (uint32_t)r0 * 128 +
                    ((uint32_t)(((c0 & 63) >> 3) ^ (r0 & 7)) << 4) + (uint32_t)((c0 & 7) * 2)
              : (uint32_t)r0 * 64 + ((uint32_t)((c0 >> 3) ^ ((r0 >> 1) & 3)) << 4) +
                    (uint32_t)((c0 & 7) * 2);
    for (uint32_t i = 0; i < FT_AHEAD; ++i) fetch_a(i);
    for (int i = 0; i < nunits && ok; ++i) {
      const FtUnit u = w.get(i);
      if (W::kEmpty && u.kb0 == u.kb1) {
        fetch_a(slot);
        slot = (slot + 1) % FT_AHEAD;
        continue;
      }
      for (int kb = u.kb0; kb < u.kb1; ++kb) {
        if (!__all_sync(0xffffffffu, mbar_wait_inl(ea(sa), pha, abort_flag))) {
          ok = false;
          break;
        }
        Range rg;
        float4 v[4];
        asm volatile("cp.async.wait_group %0;" ::"n"(FT_AHEAD - 1) : "memory");
#pragma unroll
        for (int q = 0; q < 4; ++q)
          asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                       : "=f"(v[q].x), "=f"(v[q].y), "=f"(v[q].z), "=f"(v[q].w)
                       : "r"(raw_slot + slot * FT_RAW + q * FT_CT * 16)
                       : "memory");
        const uint32_t a = base + sa * 3 * FT_APART + aoff;
#pragma unroll
        for (int q = 0; q < 4; ++q) {  // RS rows apart: the swizzle term does not change
          put4(a + q * RS * (TRANS ? 128 : 64), FT_APART, v[q]);
          rg.add(v[q]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(fa(sa));
        fetch_a(slot);
        const bool off = rg.tell(u.st);
        if (W::kGiveUp && __any_sync(0xffffffffu, off)) {
          *abort_flag = GIVE_UP;
          ok = false;
          break;
        }
        slot = (slot + 1) % FT_AHEAD;
        if (++sa == FT_NA) { sa = 0; pha ^= 1u; }
        if (!IMG) {
          if (!__all_sync(0xffffffffu, mbar_wait_inl(ex(sx), phx, abort_flag))) {
            ok = false;
            break;
          }
          Range rx;
          const XPlace xp(ct);
          const int64_t row = (int64_t)kb * F32_BK + xp.k;
#pragma unroll
          for (int q = 0; q < FT_XV; ++q) {
            if (32 * q >= u.w) break;
            const int c = u.col0 + xp.c + 32 * q;
            load4_if(v[q & 3], u.X + row * u.ldx + c, row < u.K && c < u.xcols);
            mask4(v[q & 3], c, u.d);
            put4(x_base + sx * xstage + xp.off(q), xpart, v[q & 3]);
            rx.add(v[q & 3]);
          }
          if (u.tile == 0) rx.tell(u.st);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(fx(sx));
          if (++sx == NX) { sx = 0; phx ^= 1u; }
        }
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (!ok) leave();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(FT_REG_EPI));
    // ---------------- epilogue ----------------
    const int g = warp & 3;  // TMEM lane quarter of this warp
    float* const stg = (float*)(base_ptr + (stg_base - base)) + g * 32 * FT_SP;
    const uint32_t lanes = (uint32_t)(g * 32) << 16;
    bool ok = true;
    int it = 0;
    for (int i = 0; i < nunits && ok; ++i) {
      const FtUnit u = w.get(i);
      float acc[FT_NC][16];
#pragma unroll
      for (int c = 0; c < FT_NC; ++c)
#pragma unroll
        for (int j = 0; j < 16; ++j) acc[c][j] = 0.f;
      for (int kb = u.kb0; kb < u.kb1; ++kb, ++it) {
        const int a = it & 1;
        if (!__all_sync(0xffffffffu, mbar_wait_inl(tfull(a), (uint32_t)((it >> 1) & 1), abort_flag))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t taddr = tmem_base + (uint32_t)(a * 256) + lanes;
#pragma unroll
        for (int c = 0; c < FT_NC; ++c) {
          if (c * 16 >= u.w) break;
          float v[16];
          tmem_ld16(taddr + c * 16, v);
#pragma unroll
          for (int j = 0; j < 16; j += 2) add2(acc[c][j], acc[c][j + 1], v[j], v[j + 1]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty(a));
      }
      if (!ok) break;
      // 16 columns at a time through a staging block, so that a store covers
      // whole 64-byte row segments (a lane storing its own row takes 32 of the
      // L1's cycles per instruction: 3600 clocks a tile at 112 columns)
      const int left = (int)min((int64_t)F32_BM, u.rows - (int64_t)u.tile * F32_BM) - g * 32;
      uint32_t lo = 0xFFFFFFFFu;  // (Range::key)
      bool zero = false;
#pragma unroll
      for (int c = 0; c < FT_NC; ++c) {
        if (c * 16 >= u.w) break;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<float4*>(stg + lane * FT_SP + 4 * j) = make_float4(
              acc[c][4 * j], acc[c][4 * j + 1], acc[c][4 * j + 2], acc[c][4 * j + 3]);
        __syncwarp();
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int rr = r * 8 + (lane >> 2), cc = (lane & 3) * 4;
          if (rr < left && c * 16 + cc < u.ocols)
            *reinterpret_cast<float4*>(u.out + (int64_t)(g * 32 + rr) * u.ldo + c * 16 + cc) =
                *reinterpret_cast<const float4*>(stg + rr * FT_SP + cc);
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (u.col0 + c * 16 + j < u.d) {
            lo = min(lo, Range::key(acc[c][j]));
            zero |= acc[c][j] == 0.f;
          }
      }
      if (lane < left && lo < 2u * 0x1C800000u - 1u) note(u.st, RANGE_TINY);  // 2^-70
      if (lane < left && zero) note(u.st, RANGE_ZERO);
    }
    if (!ok) leave();
  }
  __syncthreads();
  if (t == 0 && *abort_flag == TIMED_OUT) atomicExch(err, 1);
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base)
                 : "memory");
  }
}

template <bool TRANS, bool IMG>
__global__ void __launch_bounds__(FT_THREADS, 1)
k_f32_tc(const __grid_constant__ FtParams p, int stages) {
  const FtSingle w{&p};
  ft_body<TRANS, IMG>(w, stages, p.sp.w, p.err);
}

template <bool TRANS, bool IMG>
__global__ void __launch_bounds__(FT_THREADS, 1)
k_bf32_tc(const F32Tile* __restrict__ list, int n, const BMat* __restrict__ T, int src, int dst,
          int sms, int stages, int wmax, int* err) {
  const FtBatch w{list, n, T, src, dst, sms, TRANS};
  ft_body<TRANS, IMG>(w, stages, wmax, err);
}

// Sum the S slab fragments of tail item tt in slab order into the output:
// block (tt, y) adds rows 4 y .. 4 y + 3, a thread per 4 columns.
__device__ __forceinline__ void f32_fixup(const float* frag, int tt, int S, int sw, int w,
                                          int64_t rows, float* out, int64_t ldo) {
  const int r = blockIdx.y * 4 + threadIdx.x / 64, c = (threadIdx.x & 63) * 4;
  if (r >= rows || c >= w) return;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int i = 0; i < S; i += 8) {
    float4 v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (i + q < S)
        v[q] = *reinterpret_cast<const float4*>(
            frag + ((int64_t)(tt * S + i + q) * F32_BM + r) * sw + c);
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (i + q < S) {
        s.x += v[q].x;
        s.y += v[q].y;
        s.z += v[q].z;
        s.w += v[q].w;
      }
  }
  *reinterpret_cast<float4*>(out + (int64_t)r * ldo + c) = s;
}

__global__ void __launch_bounds__(256) k_f32_fixup(const __grid_constant__ FtParams p) {
  pdl_launch();
  pdl_wait();
  FtUnit u;
  ft_columns(p.sp, p.sp.full_waves * p.sp.P + (int)blockIdx.x, p.dp, u);
  f32_fixup(p.frag, blockIdx.x, p.sp.S, p.sp.w, min(u.w, p.ocols - u.col0), p.rows - (int64_t)u.tile * F32_BM,
            p.out + (int64_t)u.tile * F32_BM * p.ldo + u.col0, p.ldo);
}

// Batch: block x is the x-th split item of the list's fix-up entries.
__global__ void __launch_bounds__(256) k_bf32_fixup(const F32Tile* __restrict__ list,
                                                    const BMat* __restrict__ T, int dst,
                                                    bool trans, int sms) {
  const F32Tile e = list[blockIdx.x];
  const BMat& b = T[e.mat()];
  const int64_t rows = trans ? b.n : b.m;
  const F32Split sp = f32_columns(b.dp);
  FtUnit u;
  ft_columns(sp, e.item(), b.dp, u);
  f32_fixup((const float*)b.partial, tail_index_of(rows, sp.nch, e.item(), sms), e.S(), sp.w, u.w,
            rows - (int64_t)u.tile * F32_BM,
            bbuf(b, dst) + (int64_t)u.tile * F32_BM * b.dp + u.col0, b.dp);
}

size_t ft_smem(int nx, int w) {
  return 1024 + FT_NA * 3 * FT_APART + FT_AHEAD * FT_RAW + FT_STG + (size_t)nx * f32_xstage(w) +
         8 * (2 * FT_NA + 2 * nx + 5) + 16;
}
// X stages: as many as fit (2 at 224 columns), at most 6.
int ft_stages(int w) {
  int s = 6;
  while (s > 0 && ft_smem(s, w) > 226 * 1024) --s;
  return s;
}

// The register split needs every register a 128-register launch holds.
template <typename K>
cudaError_t ft_prepare(K kern, size_t smem) {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, kern);
  if (e != cudaSuccess) return e;
  if (a.numRegs * 4 < FT_REG_CTL + 2 * FT_REG_CONV + FT_REG_EPI) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

}  // namespace

// The split of a product: whole waves of items, then `tail` items in S slabs
// of at least 512 rows of the contraction, as many as the SMs and the Gram
// partials' buffer (free during a product; its size over this shape's row
// slabs, gram_slabs) hold.  A function of the shape and the device alone.
F32Split f32_split(int64_t rows, int64_t K, int64_t m, int64_t n, int d, int dp) {
  F32Split sp = f32_columns(dp);
  int64_t sl;
  const int64_t slabs = std::max(gram_slabs(m, 64, &sl), gram_slabs(n, 64, &sl));
  const int64_t cap = slabs * d * d * 8;
  const int64_t items = (int64_t)ceil_div(rows, F32_BM) * sp.nch;
  sp.P = sm_count();
  sp.KB = ceil_div(K, F32_BK);
  sp.full_waves = (int)(items / sp.P);
  sp.tail = (int)(items - (int64_t)sp.full_waves * sp.P);
  sp.S = 1;
  if (sp.tail > 0) {
    int64_t S = std::min<int64_t>(sp.P / sp.tail, K / 512);
    S = std::min(S, cap / ((int64_t)sp.tail * F32_BM * sp.w * 4));
    sp.S = (int)std::max<int64_t>(S, 1);
  }
  return sp;
}

// Whether a product over K rows runs on the tensor cores.  The CUDA-core
// kernel takes 47 us + 0.115 us K per call (its 64 x 64 tiles walk K one after
// another), this one 58 us + 0.035 us K with its three launches: they meet near
// K = 140 (256 x 256, d = 72: 72 against 58 us; 128 x 128, d = 30: 61 against
// 63; 64 x 64: 49 against 59).  The line is at 128 because a batch, which pays
// the launches anyway, gains from every item (a batch of 64: 1750 us with the
// items of K < 192 on the CUDA cores, 1640 without).
bool f32_tc_supported(int64_t K) { return K >= 128; }

cudaError_t f32_gemm_tc(bool trans, const float* A, int64_t lda, int64_t m, int64_t n,
                        const float* X, int64_t ldx, int xcols, int d, int dp, float* out,
                        int64_t ldo, int ocols, float* frag, void* img, DevStatus* st,
                        cudaStream_t stream) {
  if (ocols < d || ocols > dp || (ocols & 3) || xcols < d || xcols > ldx || (xcols & 3) ||
      (ldx & 3) || ((uintptr_t)X & 15) || (ldo & 3) || ((uintptr_t)out & 15))
    return cudaErrorInvalidValue;
  FtParams p{};
  p.A = A;
  p.lda = lda;
  p.rows = trans ? n : m;
  p.K = trans ? m : n;
  p.X = X;
  p.ldx = ldx;
  p.img = (const uint8_t*)img;
  p.out = out;
  p.ldo = ldo;
  p.ocols = ocols;
  p.frag = frag;
  p.d = d;
  p.xcols = xcols;
  p.dp = dp;
  p.vec = (lda & 3) == 0 && ((uintptr_t)A & 15) == 0;
  p.sp = f32_split(p.rows, p.K, m, n, d, dp);
  p.st = st;
  p.err = &st->timeout;
  const int stages = ft_stages(p.sp.w);
  const size_t smem = ft_smem(stages, p.sp.w);
  auto kern = img ? (trans ? k_f32_tc<true, true> : k_f32_tc<false, true>)
                  : (trans ? k_f32_tc<true, false> : k_f32_tc<false, false>);
  cudaError_t e = ft_prepare(kern, smem);
  if (e != cudaSuccess) return e;
  if (img) {
    e = launch_pdl(k_f32_split, dim3(p.sp.KB, p.sp.nch), dim3(FT_CT), 0, stream, p);
    count_launch();
    if (e != cudaSuccess) return e;
  }
  const int grid = p.sp.full_waves > 0 ? p.sp.P : p.sp.tail * p.sp.S;
  e = launch_pdl(kern, dim3(grid), dim3(FT_THREADS), smem, stream, p, stages);
  count_launch();
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess || p.sp.S == 1) return e;
  e = launch_pdl(k_f32_fixup, dim3(p.sp.tail, F32_BM / 4), dim3(256), 0, stream, p);
  count_launch();
  return e == cudaSuccess ? cudaGetLastError() : e;
}

cudaError_t f32_mul_img(const float* A, int64_t lda, int64_t M, int K, int dp, const void* img,
                        float* out, int64_t ldo, int* err, cudaStream_t stream) {
  if ((ldo & 3) || ((uintptr_t)out & 15) || K >= 512 || dp > F32_WMAX) return cudaErrorInvalidValue;
  FtParams p{};
  p.A = A;
  p.lda = lda;
  p.rows = M;
  p.K = K;
  p.img = (const uint8_t*)img;
  p.out = out;
  p.ldo = ldo;
  p.ocols = dp;
  p.d = K;
  p.dp = dp;
  p.vec = (lda & 3) == 0 && ((uintptr_t)A & 15) == 0;
  p.sp = f32_split(M, K, M, K, K, dp);  // (one slab: K < 512)
  p.err = err;
  const int stages = ft_stages(p.sp.w);
  const size_t smem = ft_smem(stages, p.sp.w);
  cudaError_t e = ft_prepare(k_f32_tc<false, true>, smem);
  if (e != cudaSuccess) return e;
  e = launch_pdl(k_f32_tc<false, true>, dim3(p.sp.full_waves > 0 ? p.sp.P : p.sp.tail),
                 dim3(FT_THREADS), smem, stream, p, stages);
  count_launch();
  return e == cudaSuccess ? cudaGetLastError() : e;
}

size_t f32_img_bytes(int64_t K, int dp) {
  const F32Split sp = f32_columns(dp);
  return (size_t)sp.nch * ceil_div(K, F32_BK) * f32_xstage(sp.w);
}

void f32_tiles(int mat, const F32Split& sp, std::vector<F32Tile>& list,
               std::vector<F32Tile>& fix) {
  const int whole = sp.full_waves * sp.P;
  for (int i = 0; i < whole; ++i) list.push_back(F32Tile::make(mat, i, 0, 1));
  for (int tt = 0; tt < sp.tail; ++tt) {
    for (int s = 0; s < sp.S; ++s) list.push_back(F32Tile::make(mat, whole + tt, s, sp.S));
    if (sp.S > 1) fix.push_back(F32Tile::make(mat, whole + tt, 0, sp.S));
  }
}

cudaError_t bf32_gemm_tc(bool trans, const BMat* T, const F32Tile* list, int n,
                         const F32Tile* fix, int nfix, int src, int dst, int wmax, int count,
                         bool img, int* err, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int stages = ft_stages(wmax);
  const size_t smem = ft_smem(stages, wmax);
  auto kern = img ? (trans ? k_bf32_tc<true, true> : k_bf32_tc<false, true>)
                  : (trans ? k_bf32_tc<true, false> : k_bf32_tc<false, false>);
  cudaError_t e = ft_prepare(kern, smem);
  if (e != cudaSuccess) return e;
  if (img) {
    k_bf32_split<<<dim3(32, count), FT_CT, 0, st>>>(T, src);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  kern<<<std::min(n, sm_count()), FT_THREADS, smem, st>>>(list, n, T, src, dst, sm_count(), stages,
                                                             wmax, err);
  count_launch();
  e = cudaGetLastError();
  if (e != cudaSuccess || nfix <= 0) return e;
  k_bf32_fixup<<<dim3(nfix, F32_BM / 4), 256, 0, st>>>(fix, T, dst, trans, sm_count());
  count_launch();
  return cudaGetLastError();
}

}  // namespace ruqlp
