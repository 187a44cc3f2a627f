// Offline side of the path: W' = R^T W (Eq. 1), the mixed-precision split of W'
// (Eq. 3, Section 3.3), and the conversions between the tiled layout the GEMM kernels
// read and the plain interchange layout.
//
// Everything that decides an integer code is written with explicit round-to-nearest
// intrinsics (__fmaf_rn, __fdiv_rn, ...) so that the compiler can neither contract nor
// reorder it: the codes must be reproducible bit for bit by a sequential IEEE fp32
// implementation.
#include <algorithm>

#include "rosaq_internal.cuh"
#include "cov_common.cuh"

namespace rosaq {

// =====================================================================================
// The fp32 chain.  out[i][n] = sum_k A[k][i] * B[k][n] as one fused multiply-add per term, k ascending, a single
// fp32 accumulator per output started at +0: the canonical order of W' = R^T W (and, with A = B = X, the Gram
// matrix of fp32 calibration activations).  A CTA of 128 threads computes a 128 x 128 tile, 8 x 16 outputs per
// thread, K stepped by kBK through two shared-memory buffers.  Zero padding is harmless: fma(0, 0, acc) = acc.
//
// Bound: the fp32 pipe (one multiply-add per lane and cycle, 128 lanes per SM) -- as long as the operands keep up.
// A 16-byte shared-memory load occupies the SM's load path for four cycles whatever it broadcasts, so an 8 x 8 thread
// tile (four loads per 64 multiply-adds) is bound by its loads; an 8 x 16 one (six per 128) is not.  Scalar
// multiply-adds then lose a quarter of their issue cycles to register-port stalls (3.27 ms in the example below);
// fma.rn.f32x2, two independent IEEE multiply-adds on register pairs, does not and leaves issue slots free.  (On registers alone
// two warps per scheduler reach 2.2 cycles per paired multiply-add, 63 TFLOP/s; one warp 2.2 to 3.0, by their order.)
// Steps of sixteen: 2.52 ms, of eight 2.65, of thirty-two 3.35 (the operands in flight no longer fit the registers).  The Gram kernel, whose
// operands are both fp32, gains from them where an SM has one CTA (4096 tokens x 512 channels 64.4 -> 59.9 us), and loses where two hide
// each other's barriers (x 2048: 382 -> 391).
// Measured at 4096 -> 4096 INT4, dense R, the rotation and the quantization: 3.41 ms (41 TFLOP/s; 8 x 8 scalar per
// thread, one buffer, W' through global memory) at first, 2.65 ms with the pairs, 2.52 ms (54 TFLOP/s) now.
// =====================================================================================
constexpr int kBM = 128, kBN = 128;
constexpr int kFmaThreads = 128;
constexpr int kTilePitch = 132;                                  // floats; the finished tile reuses the buffers
constexpr int kFmaSmemBytes = 128 * kTilePitch * 4;

// this thread's outputs: rows ty * 4 + {0..3} and 64 + ty * 4 + {0..3}; columns tx * 4 + {0..3} of each 32-column
// quarter.  A warp covers 4 x 8 of the 16 x 8 (ty, tx).
struct FmaThread {
  int ty, tx;
  __device__ FmaThread() {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    ty = warp * 4 + (lane >> 3);
    tx = lane & 7;
  }
  __device__ int row(int ia) const { return ia < 4 ? ty * 4 + ia : 64 + ty * 4 + ia - 4; }
};

__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
  return v;
}
__device__ __forceinline__ float4 unpack4(unsigned long long a, unsigned long long b) {
  float4 v;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(a));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(v.z), "=f"(v.w) : "l"(b));
  return v;
}
// two independent IEEE fp32 multiply-adds
__device__ __forceinline__ void fma2(unsigned long long &c, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

// Four values of one operand row as they come from memory.  They are converted when they are stored to shared memory,
// one K step after the load was issued: converted in place they would stall the warp for the whole latency.
template <typename T>
struct Raw4;
template <>
struct Raw4<float> {
  float4 v;
  __device__ __forceinline__ void zero() { v = make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ __forceinline__ void load4(const float *p) { v = *reinterpret_cast<const float4 *>(p); }
  __device__ __forceinline__ void set(int e, float x) { reinterpret_cast<float *>(&v)[e] = x; }
  __device__ __forceinline__ float4 expand() const { return v; }
};
template <>
struct Raw4<__half> {
  __half2 v[2];
  __device__ __forceinline__ void zero() { v[0] = v[1] = __float2half2_rn(0.f); }
  __device__ __forceinline__ void load4(const __half *p) { *reinterpret_cast<uint2 *>(v) = *reinterpret_cast<const uint2 *>(p); }
  __device__ __forceinline__ void set(int e, __half x) {
    if (e & 1) v[e >> 1].y = x;
    else v[e >> 1].x = x;
  }
  __device__ __forceinline__ float4 expand() const {
    const float2 a = __half22float2(v[0]), b = __half22float2(v[1]);
    return make_float4(a.x, a.y, b.x, b.y);
  }
};

// The K loop.  fetch_a(k, c, raw) / fetch_b(k, c, raw) deliver A[k][c .. c + 3] / B[k][c .. c + 3] (tile columns; 0 outside
// the operand, also for k >= K); with kScaled row k of B is multiplied by fetch_s(k), one rounding per product.
// acc[ia][2 q + e] is row(ia), columns 32 q + tx * 4 + 2 e, + 1.
template <int kBK, typename TA, typename TB, bool kScaled, typename FA, typename FB, typename FS>
__device__ __forceinline__ void fma_tile(float *smem, int K, const FmaThread &ft, FA fetch_a, FB fetch_b, FS fetch_s, unsigned long long acc[8][8]) {
#pragma unroll
  for (int ia = 0; ia < 8; ++ia)
#pragma unroll
    for (int ib = 0; ib < 8; ++ib) acc[ia][ib] = 0ull;
  constexpr int kFmaBufFloats = kBK * (kBM + kBN), kRows = kBK / 4;
  static_assert(2 * kFmaBufFloats * 4 <= kFmaSmemBytes, "two buffers");
  const int lr = threadIdx.x >> 5, lc = (threadIdx.x & 31) * 4;      // loader: rows lr, lr + 4, ... of the K step, four columns
  Raw4<TA> ra[kRows];
  Raw4<TB> rb[kRows];
  float rs[kRows];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int h = 0; h < kRows; ++h) {
      fetch_a(k0 + lr + 4 * h, lc, ra[h]);
      fetch_b(k0 + lr + 4 * h, lc, rb[h]);
      if (kScaled) rs[h] = fetch_s(k0 + lr + 4 * h);
    }
  };
  auto put = [&](float *buf) {
#pragma unroll
    for (int h = 0; h < kRows; ++h) {
      *reinterpret_cast<float4 *>(buf + (lr + 4 * h) * kBM + lc) = ra[h].expand();
      float4 b = rb[h].expand();
      if (kScaled) b = make_float4(__fmul_rn(rs[h], b.x), __fmul_rn(rs[h], b.y), __fmul_rn(rs[h], b.z), __fmul_rn(rs[h], b.w));
      *reinterpret_cast<float4 *>(buf + kBK * kBM + (lr + 4 * h) * kBN + lc) = b;
    }
  };
  fetch(0);
  put(smem);
  __syncthreads();
  int cur = 0;
  for (int k0 = 0; k0 < K; k0 += kBK) {
    const bool more = k0 + kBK < K;
    if (more) fetch(k0 + kBK);
    const float *as = smem + cur * kFmaBufFloats + ft.ty * 4, *bs = smem + cur * kFmaBufFloats + kBK * kBM + ft.tx * 4;
#pragma unroll
    for (int kk = 0; kk < kBK; ++kk) {
      __align__(16) float a[8];
      ulonglong2 b[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) *reinterpret_cast<float4 *>(a + 4 * h) = *reinterpret_cast<const float4 *>(as + kk * kBM + 64 * h);
#pragma unroll
      for (int q = 0; q < 4; ++q) b[q] = *reinterpret_cast<const ulonglong2 *>(bs + kk * kBN + 32 * q);
#pragma unroll
      for (int ia = 0; ia < 8; ++ia) {
        const unsigned long long aa = pack2(a[ia], a[ia]);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          fma2(acc[ia][2 * q], aa, b[q].x);
          fma2(acc[ia][2 * q + 1], aa, b[q].y);
        }
      }
    }
    if (more) put(smem + (cur ^ 1) * kFmaBufFloats);
    __syncthreads();
    cur ^= 1;
  }
}

__device__ __forceinline__ void store_tile_smem(float *tile, const FmaThread &ft, const unsigned long long acc[8][8]) {
#pragma unroll
  for (int ia = 0; ia < 8; ++ia)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      *reinterpret_cast<float4 *>(tile + ft.row(ia) * kTilePitch + 32 * q + ft.tx * 4) =
          unpack4(acc[ia][2 * q], acc[ia][2 * q + 1]);
}

// =====================================================================================
// Eq. 3 / Section 3.3: one 128 x 128 tile of W' in shared memory = one group of 128 output columns.  Salient rows ->
// fp16; other groups -> asymmetric min/max RTN codes, written straight into the tiled layout.  kParts
// threads per column (a CTA of 128 * kParts threads), each with its share of the rows; the parts' extremes are joined in
// row order through `ends`, so a tie between zeros of either sign falls as in one scan.
// =====================================================================================
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  return (uint32_t)__half_as_ushort(__float2half_rn(lo)) | ((uint32_t)__half_as_ushort(__float2half_rn(hi)) << 16);
}

template <int kBits, int kParts>
__device__ __forceinline__ void quant_tile(const float *tile, float2 *ends, const TiledOperand &t, int nt, int g) {
  constexpr int kRows = kGroup / kParts;
  static_assert(kRows % 32 == 0, "a part holds whole INT3 sets");
  const int nl = threadIdx.x & 127, part = threadIdx.x >> 7, k0 = part * kRows;
  const bool live = nt * kTileN + nl < t.d_out;
  uint8_t *out = t.blob + tile_offset(t, nt, g);
  const float *col = tile + k0 * kTilePitch + nl;
  if (g < t.g_fp16) {
    for (int k8 = 0; k8 < kRows; k8 += 8) {
      float v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = live ? col[(k8 + e) * kTilePitch] : 0.0f;
      *reinterpret_cast<uint4 *>(out + fp16_tile_byte(k0 + k8, nl)) =
          make_uint4(pack_half2(v[0], v[1]), pack_half2(v[2], v[3]), pack_half2(v[4], v[5]), pack_half2(v[6], v[7]));
    }
    return;
  }
  // The scan of a whole column starts with its first value and skips NaNs after it; a part that starts further down starts
  // with the empty range, so that a NaN there is skipped as well.
  const float inf = __int_as_float(0x7f800000);
  float lo = part == 0 ? col[0] : inf, hi = part == 0 ? col[0] : -inf;
#pragma unroll 16
  for (int k = 0; k < kRows; ++k) {
    const float w = col[k * kTilePitch];
    lo = w < lo ? w : lo;
    hi = w > hi ? w : hi;
  }
  if (kParts > 1) {
    ends[threadIdx.x] = make_float2(lo, hi);
    __syncthreads();
    lo = ends[nl].x, hi = ends[nl].y;
#pragma unroll
    for (int q = 1; q < kParts; ++q) {
      const float2 e = ends[q * 128 + nl];
      lo = e.x < lo ? e.x : lo;
      hi = e.y > hi ? e.y : hi;
    }
  }
  constexpr int kWords = (kBits == 4 ? 16 : 12) / kParts;
  uint32_t words[kWords];
#pragma unroll
  for (int w = 0; w < kWords; ++w) words[w] = 0;
  __half sh = __ushort_as_half(0), zh = __ushort_as_half(0);
  if (live) {
    const float qmax = (float)((1 << kBits) - 1);
    float range = __fsub_rn(hi, lo);
    if (range < 1e-5f) range = 1e-5f;
    unsigned short sb = __half_as_ushort(__float2half_rn(__fdiv_rn(range, qmax)));
    if (sb == 0x0000) sb = 0x0001;
    if (sb == 0x7c00) sb = 0x7bff;
    sh = __ushort_as_half(sb);
    const float sf = __half2float(sh);
    float z = -rintf(__fdiv_rn(lo, sf));
    if (z <= 0.0f) z = 0.0f;
    if (z > qmax) z = qmax;
    zh = __float2half_rn(z);
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      float q = __fadd_rn(rintf(__fdiv_rn(col[k * kTilePitch], sf)), z);
      if (q < 0.0f) q = 0.0f;
      if (q > qmax) q = qmax;
      put_code<kBits>(words, k, (uint32_t)q);
    }
  }
  if (kParts == 1) {
    store_quant_tile_column<kBits>(out, nl, words, sh, zh);
    return;
  }
  if (kBits == 4) {
#pragma unroll
    for (int j = 0; j < kWords / 4; ++j)
      *reinterpret_cast<uint4 *>(out + ((part * kWords / 4 + j) * kTileN + nl) * 16) =
          make_uint4(words[4 * j], words[4 * j + 1], words[4 * j + 2], words[4 * j + 3]);
  } else {
#pragma unroll
    for (int j = 0; j < kWords; ++j) *reinterpret_cast<uint32_t *>(out + int3_word_byte(part * kWords + j, nl)) = words[j];
  }
  if (part == 0)
    *reinterpret_cast<uint32_t *>(out + quant_code_bytes(kBits) + nl * 4) =
        (uint32_t)__half_as_ushort(sh) | ((uint32_t)__half_as_ushort(zh) << 16);
}

struct RotateArgs {
  const void *q;            // [n_blocks][dh][dh]
  const int32_t *perm;      // output row j takes column perm[j] of blockdiag(q), or NULL
  const int32_t *inv;       // its inverse (kSpill only), or NULL
  const __half *W;          // [d_in][d_out]
  const float *in_scale;    // [d_in]: the chain runs on the fp32 products in_scale[i] * W[i][n]; or NULL
  float *spill;             // kSpill: W' columns [n_base, n_base + spill_cols), row-major
  int d_in, d_out, dh, n_base, spill_cols;
};

// W' = R^T W for one 128 x 128 tile, then either quantized and packed from shared memory (kSpill = false: the tile is
// a whole group, so W' never reaches global memory), or, when the rows of a group come from different head blocks (a
// block-diagonal R with a column order), stored to a slab of W' that quant_tile_kernel reads.
template <typename TQ, int kBits, bool kSpill, bool kScaled, int kBK>
__global__ void __launch_bounds__(kFmaThreads, 2)
rotate_tile_kernel(const RotateArgs a, const TiledOperand t) {
  extern __shared__ __align__(16) float smem[];
  const FmaThread ft;
  // (kSpill: the row tiles, one and more per head block, in the grid's x: there may be more than 65535)
  const int nt = kSpill ? blockIdx.y : blockIdx.x, row = kSpill ? blockIdx.x : blockIdx.y, n0 = a.n_base + nt * kBN;
  // rows of the tile: output channels of group `row`, or (kSpill) source columns of one head block
  const int per_block = (a.dh + kBM - 1) / kBM;
  const int h = kSpill ? row / per_block : (a.perm ? 0 : row * kBM / a.dh);
  const int c0 = kSpill ? (row % per_block) * kBM : row * kBM - h * a.dh;   // first column inside the block
  const TQ *R = static_cast<const TQ *>(a.q) + (long long)h * a.dh * a.dh;
  const __half *W = a.W + (long long)h * a.dh * a.d_out;
  const int32_t *perm = kSpill ? nullptr : a.perm;
  int pc[4];                                                         // the four columns of R this thread loads
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int i = (threadIdx.x & 31) * 4 + e + c0;
    pc[e] = i >= a.dh ? -1 : (perm ? perm[i] : i);
  }
  // (W is 16-byte aligned; R may lie on any element)
  const bool a_vec = perm == nullptr && a.dh % 8 == 0 && reinterpret_cast<uintptr_t>(a.q) % (4 * sizeof(TQ)) == 0, b_vec = a.d_out % 8 == 0;
  auto fetch_a = [&](int k, int, Raw4<TQ> &raw) {
    if (k < a.dh && a_vec && pc[3] >= 0) {
      raw.load4(R + (long long)k * a.dh + pc[0]);
      return;
    }
    raw.zero();
    if (k < a.dh)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (pc[e] >= 0) raw.set(e, R[(long long)k * a.dh + pc[e]]);
  };
  auto fetch_b = [&](int k, int c, Raw4<__half> &raw) {
    const int n = n0 + c;
    if (k < a.dh && b_vec && n + 3 < a.d_out) {
      raw.load4(W + (long long)k * a.d_out + n);
      return;
    }
    raw.zero();
    if (k < a.dh)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (n + e < a.d_out) raw.set(e, W[(long long)k * a.d_out + n + e]);
  };
  const float *ds = kScaled ? a.in_scale + (long long)h * a.dh : nullptr;
  unsigned long long acc[8][8];
  fma_tile<kBK, TQ, __half, kScaled>(smem, a.dh, ft, fetch_a, fetch_b, [&](int k) { return k < a.dh ? ds[k] : 0.f; }, acc);
  if (!kSpill) {
    store_tile_smem(smem, ft, acc);                                  // (the K loop ends with a barrier)
    __syncthreads();
    quant_tile<kBits, 1>(smem, nullptr, t, nt, row);
  } else {
#pragma unroll
    for (int ia = 0; ia < 8; ++ia) {
      const int c = c0 + ft.row(ia);
      if (c >= a.dh) continue;
      const int p = h * a.dh + c, j = a.inv ? a.inv[p] : p;
      float *dst = a.spill + (long long)j * a.spill_cols + nt * kBN + ft.tx * 4;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4 *>(dst + 32 * q) = unpack4(acc[ia][2 * q], acc[ia][2 * q + 1]);
    }
  }
}

// Quantizes and packs tiles whose W' is already there: a slab of fp32 W' (spill), or no rotation at all, W or D W
// (one fp32 rounding per product).  Bound: HBM (2 bytes per weight in, half a byte out).
constexpr int kQuantParts = 4, kQuantThreads = 128 * kQuantParts;
constexpr int kQuantSmemBytes = kFmaSmemBytes + kQuantThreads * (int)sizeof(float2);

template <int kBits>
__global__ void __launch_bounds__(kQuantThreads, 3)
quant_tile_kernel(const float *__restrict__ spill, const __half *__restrict__ W, const float *__restrict__ in_scale, int nt0,
                  int spill_cols, const TiledOperand t) {
  extern __shared__ __align__(16) float tile[];
  const int nt = nt0 + blockIdx.x, g = blockIdx.y;
  const int lr = threadIdx.x >> 4, lc = (threadIdx.x & 15) * 8;      // 32 rows per step, eight columns per thread
  const int n = nt * kTileN + lc;
#pragma unroll
  for (int r0 = 0; r0 < kGroup; r0 += kQuantThreads / 16) {
    const long long i = (long long)g * kGroup + r0 + lr;
    float v[8];
    if (spill) {
      const float *src = spill + i * spill_cols + blockIdx.x * kTileN + lc;
      *reinterpret_cast<float4 *>(v) = *reinterpret_cast<const float4 *>(src);
      *reinterpret_cast<float4 *>(v + 4) = *reinterpret_cast<const float4 *>(src + 4);
    } else {
      if (t.d_out % 8 == 0 && n + 7 < t.d_out) {
        __align__(16) __half r[8];
        *reinterpret_cast<uint4 *>(r) = *reinterpret_cast<const uint4 *>(W + i * t.d_out + n);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = __half2float(r[e]);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = n + e < t.d_out ? __half2float(W[i * t.d_out + n + e]) : 0.f;
      }
      if (in_scale) {
        const float d = in_scale[i];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = __fmul_rn(d, v[e]);
      }
    }
    float *dst = tile + (r0 + lr) * kTilePitch + lc;
    *reinterpret_cast<float4 *>(dst) = *reinterpret_cast<const float4 *>(v);
    *reinterpret_cast<float4 *>(dst + 4) = *reinterpret_cast<const float4 *>(v + 4);
  }
  __syncthreads();
  quant_tile<kBits, kQuantParts>(tile, reinterpret_cast<float2 *>(tile + kGroup * kTilePitch), t, nt, g);
}

template <typename K>
static bool allow_smem(K kern, int bytes) {
  // (a per-device attribute; setting it again is a cheap no-op and these calls are offline)
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess) return true;
  (void)cudaGetLastError();
  return false;
}

template <typename TQ, int kBits, bool kScaled>
static int rotate_quantize_typed(const RotateArgs &args, int n_blocks, const TiledOperand &t, cudaStream_t s) {
  RotateArgs a = args;
  // (steps of sixteen for a dense R; head blocks of 128 channels are eight such steps, most of them start and end: 2048 channels 70.4 us
  // with steps of eight, 75.8 with sixteen)
  const auto fused = n_blocks == 1 ? rotate_tile_kernel<TQ, kBits, false, kScaled, 16> : rotate_tile_kernel<TQ, kBits, false, kScaled, 8>;
  const auto spilling = rotate_tile_kernel<TQ, kBits, true, kScaled, 8>;
  const auto quant = quant_tile_kernel<kBits>;
  if (!allow_smem(fused, kFmaSmemBytes) || !allow_smem(spilling, kFmaSmemBytes) || !allow_smem(quant, kQuantSmemBytes)) return ROSAQ_ERR_CUDA;
  const int groups = groups_per_tile(t);
  if (!a.q) {
    quant<<<dim3(t.n_tiles, groups), kQuantThreads, kQuantSmemBytes, s>>>(nullptr, a.W, a.in_scale, 0, 0, t);
  } else if (n_blocks == 1 || (a.perm == nullptr && a.dh % kGroup == 0)) {
    fused<<<dim3(t.n_tiles, groups), kFmaThreads, kFmaSmemBytes, s>>>(a, t);
  } else {
    const int tiles_max = a.spill_cols / kTileN, row_tiles = n_blocks * ((a.dh + kBM - 1) / kBM);
    for (int nt0 = 0; nt0 < t.n_tiles; nt0 += tiles_max) {
      const int nts = std::min(tiles_max, t.n_tiles - nt0);
      a.n_base = nt0 * kTileN;
      spilling<<<dim3(row_tiles, nts), kFmaThreads, kFmaSmemBytes, s>>>(a, t);
      quant<<<dim3(nts, groups), kQuantThreads, kQuantSmemBytes, s>>>(a.spill, nullptr, nullptr, nt0, a.spill_cols, t);
    }
  }
  return cudaGetLastError() == cudaSuccess ? ROSAQ_OK : ROSAQ_ERR_CUDA;
}

// Slab of W' that launch_rotate_quantize wants in `spill`: 16 MB of columns (L2-resident, whatever the weight's size), at
// least one column tile; 0 when the call needs none.
size_t rotate_quantize_spill_bytes(int d_in, int d_out, int n_blocks, bool perm) {
  if (n_blocks <= 1 || (!perm && d_in / n_blocks % kGroup == 0)) return 0;
  const size_t tile = sizeof(float) * (size_t)d_in * kTileN, most = size_t(16) << 20;
  const size_t tiles = most / tile < 1 ? 1 : most / tile, all = (size_t)(d_out + kTileN - 1) / kTileN;
  return tile * (tiles < all ? tiles : all);
}

int launch_rotate_quantize(const void *q, int q_is_f32, int n_blocks, const int32_t *perm, const int32_t *inv, const __half *W,
                           const float *in_scale, float *spill, size_t spill_bytes, const TiledOperand &t, cudaStream_t s) {
  RotateArgs a{};
  a.q = q, a.perm = perm, a.inv = inv, a.W = W, a.in_scale = in_scale, a.spill = spill;
  a.d_in = t.d_in, a.d_out = t.d_out, a.dh = q ? t.d_in / n_blocks : t.d_in;
  a.spill_cols = (int)(spill_bytes / (sizeof(float) * (size_t)t.d_in)) / kTileN * kTileN;
  auto run = [&](auto f32, auto f16) { return (q && !q_is_f32 ? f16 : f32)(a, n_blocks, t, s); };
  if (t.bits == 3)
    return in_scale ? run(rotate_quantize_typed<float, 3, true>, rotate_quantize_typed<__half, 3, true>)
                    : run(rotate_quantize_typed<float, 3, false>, rotate_quantize_typed<__half, 3, false>);
  return in_scale ? run(rotate_quantize_typed<float, 4, true>, rotate_quantize_typed<__half, 4, true>)
                  : run(rotate_quantize_typed<float, 4, false>, rotate_quantize_typed<__half, 4, false>);
}

// Gram matrix on CUDA cores (fp32 products, fp32 accumulate): exact-product path for fp32 calibration activations and
// the fallback for shapes the tensor-core kernel does not take.  Only tiles of the lower triangle are computed; an
// off-diagonal tile is also added, transposed, to the mirrored position (products commute and both chains run over the
// tokens in the same order, so the mirrored bits are those a tile of its own would produce).  With few tiles a cluster of up
// to eight CTAs shares the tokens of a tile and adds the partial tiles in order: a tile costs 128 cycles per token whatever the
// width (4096 tokens x 512 channels: 634 us with all tiles of both triangles and a CTA each, 67 so; x 2048: 1003 and 418).
template <typename T, int kBK>
__global__ void __launch_bounds__(kFmaThreads, 2)
gram_fma_kernel(const T *X, long long ldx, int dh, float *C, int n_tokens, int Z) {   // (X: not read-only while the kernel before may still write it)
  extern __shared__ __align__(16) float tile[];
  const FmaThread ft;
  int bi = 0;
  while ((bi + 1) * (bi + 2) / 2 <= (int)blockIdx.x) ++bi;
  const int bj = blockIdx.x - bi * (bi + 1) / 2;
  const int i0 = bi * kBM, n0 = bj * kBN;
  // split z of the tokens (a cluster shares the tile), cut at multiples of the K step
  const int z = blockIdx.z, steps = (n_tokens + kBK - 1) / kBK;
  const int t0 = (int)((long long)steps * z / Z) * kBK, K = min(n_tokens, (int)((long long)steps * (z + 1) / Z) * kBK) - t0;
  cov_grid_dep_wait();
  X += (long long)t0 * ldx + (long long)blockIdx.y * dh;
  C += (long long)blockIdx.y * dh * dh;
  auto fetch = [&](int k, int c, Raw4<T> &raw) {                     // (dh and ldx are multiples of 8, X is 16-byte aligned)
    if (k < K && c + 3 < dh) raw.load4(X + (long long)k * ldx + c);
    else raw.zero();
  };
  unsigned long long acc[8][8];
  fma_tile<kBK, T, T, false>(
      tile, K, ft, [&](int k, int c, Raw4<T> &raw) { fetch(k, i0 + c, raw); },
      [&](int k, int c, Raw4<T> &raw) { fetch(k, n0 + c, raw); }, [](int) { return 0.f; }, acc);
  cov_grid_dep_launch();
  store_tile_smem(tile, ft, acc);
  __syncthreads();
  const int r_begin = kBM * z / Z, r_end = kBM * (z + 1) / Z;        // rows of the tile that this CTA finishes
  if (Z > 1) {
    cov_cluster_sync();
    cov_sum_rows((uint32_t)__cvta_generic_to_shared(tile), tile, kTilePitch, kBN, r_begin, r_end, Z, 1, 0u, threadIdx.x, kFmaThreads);
    __syncthreads();
  }
  const int c4 = (threadIdx.x & 31) * 4, r_first = threadIdx.x >> 5;
  // C[row0 + r][col .. + 3] += value(r) for r = r0, r0 + step, ... < end: eight loads in flight, because a round trip to L2 costs
  // half a microsecond and a row at a time is 64 of them (64 tokens x 256 channels: 23.9 us, 17.0 so; 20 x 640 19.8 and 12.6)
  auto add_rows = [&](int row0, int col, int r0, int step, int end, auto value) {
    float *dst = C + (long long)row0 * dh + col;
    for (; r0 < end; r0 += 8 * step) {
      float4 old[8];
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (r0 + e * step < end) old[e] = *reinterpret_cast<const float4 *>(dst + (long long)(r0 + e * step) * dh);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int r = r0 + e * step;
        if (r >= end) break;
        const float4 v = value(r);
        *reinterpret_cast<float4 *>(dst + (long long)r * dh) = make_float4(__fadd_rn(old[e].x, v.x), __fadd_rn(old[e].y, v.y),
                                                                           __fadd_rn(old[e].z, v.z), __fadd_rn(old[e].w, v.w));
      }
    }
  };
  if (n0 + c4 < dh)
    add_rows(i0, n0 + c4, r_begin + r_first, 4, min(r_end, dh - i0),
             [&](int r) { return *reinterpret_cast<const float4 *>(tile + r * kTilePitch + c4); });
  // mirror: the share's rows, four at a time, x all columns
  const int n_quads = (r_end - r_begin) / 4, m4 = r_begin + 4 * (threadIdx.x % n_quads);
  if (bi != bj && i0 + m4 < dh)
    add_rows(n0, i0 + m4, threadIdx.x / n_quads, kFmaThreads / n_quads, min(kBN, dh - n0), [&](int r) {
      const float *tc = tile + m4 * kTilePitch + r;
      return make_float4(tc[0], tc[kTilePitch], tc[2 * kTilePitch], tc[3 * kTilePitch]);
    });
  if (Z > 1) cov_cluster_sync();                                     // nobody reads this CTA's tile any more
}

int launch_cov_fma(int sm_count, const void *X, int x_dtype, long long n_tokens, int d, long long ldx, int n_blocks, float *C,
                   cudaStream_t s) {
  const int dh = d / n_blocks, nb = (dh + kBM - 1) / kBM;
  const dim3 grid(nb * (nb + 1) / 2, n_blocks);
  if (!allow_smem(gram_fma_kernel<float, 8>, kFmaSmemBytes) || !allow_smem(gram_fma_kernel<float, 16>, kFmaSmemBytes) ||
      !allow_smem(gram_fma_kernel<__half, 16>, kFmaSmemBytes))
    return ROSAQ_ERR_CUDA;
  for (long long t0 = 0; t0 < n_tokens; t0 += 1ll << 30) {           // (the kernel counts tokens in 32 bits)
    const int n = (int)std::min(n_tokens - t0, 1ll << 30);
    // (two CTAs fit an SM; a split keeps at least 64 tokens)
    const int Z = cov_splits((long long)grid.x * grid.y, 2 * sm_count, n / 64, 8);
    const dim3 g(grid.x, grid.y, Z);
    auto launch = [&](auto kern, const auto *x) {
      return cov_launch(kern, g, kFmaThreads, kFmaSmemBytes, 1, Z, s, x + t0 * ldx, ldx, dh, C, n, Z);
    };
    // (clusters of eight double up on some SMs from about fifteen of them on: 14 blocks of 128 channels 41.6 -> 39.3 us, 16 of them 62.1 -> 65.3)
    const bool one_per_sm = (long long)g.x * g.y * g.z <= sm_count * 4 / 5;
    const int st = x_dtype != ROSAQ_F32 ? launch(gram_fma_kernel<__half, 16>, static_cast<const __half *>(X))
                   : one_per_sm         ? launch(gram_fma_kernel<float, 16>, static_cast<const float *>(X))
                                        : launch(gram_fma_kernel<float, 8>, static_cast<const float *>(X));
    if (st != ROSAQ_OK) return st;
  }
  return ROSAQ_OK;
}

// =====================================================================================
// tiled <-> interchange layout
// =====================================================================================
template <int kBits>
__global__ void __launch_bounds__(kTileN)
export_kernel(TiledOperand t, uint32_t *__restrict__ qw, __half *__restrict__ scales, __half *__restrict__ zeros,
              __half *__restrict__ salient) {
  const int nt = blockIdx.x, g = blockIdx.y, nl = threadIdx.x;
  const int n = nt * kTileN + nl;
  if (n >= t.d_out) return;
  const uint8_t *tile = t.blob + tile_offset(t, nt, g);
  if (g < t.g_fp16) {
    if (!salient) return;
    for (int k = 0; k < kGroup; ++k)
      salient[(long long)(g * kGroup + k) * t.d_out + n] =
          *reinterpret_cast<const __half *>(tile + fp16_tile_byte(k, nl));
    return;
  }
  constexpr int kWords = kBits == 4 ? 16 : 12;
  uint32_t words[kWords];
  __half sh, zh;
  load_quant_tile_column<kBits>(tile, nl, words, &sh, &zh);
  const int gq = g - t.g_fp16;
  if (scales) scales[(long long)gq * t.d_out + n] = sh;
  if (zeros) zeros[(long long)gq * t.d_out + n] = zh;
  if (!qw) return;
  if (kBits == 4) {
    for (int w = 0; w < 16; ++w) {
      uint32_t v = 0;
      for (int i = 0; i < 8; ++i) v |= get_code<4>(words, w * 8 + i) << (4 * i);
      qw[(long long)(gq * 16 + w) * t.d_out + n] = v;
    }
  } else {
    for (int blk = 0; blk < 4; ++blk) {
      uint32_t v[3] = {0, 0, 0};
      for (int i = 0; i < 32; ++i) {
        uint32_t c = get_code<3>(words, blk * 32 + i);
        for (int b = 0; b < 3; ++b) {
          int bit = 3 * i + b;
          v[bit >> 5] |= ((c >> b) & 1u) << (bit & 31);
        }
      }
      for (int w = 0; w < 3; ++w) qw[(long long)(gq * 12 + blk * 3 + w) * t.d_out + n] = v[w];
    }
  }
}

template <int kBits>
__global__ void __launch_bounds__(kTileN)
import_kernel(TiledOperand t, const uint32_t *__restrict__ qw, const __half *__restrict__ scales,
              const __half *__restrict__ zeros, const __half *__restrict__ salient) {
  const int nt = blockIdx.x, g = blockIdx.y, nl = threadIdx.x;
  const int n = nt * kTileN + nl;
  const bool live = n < t.d_out;
  uint8_t *tile = t.blob + tile_offset(t, nt, g);
  if (g < t.g_fp16) {
    for (int k = 0; k < kGroup; ++k)
      *reinterpret_cast<__half *>(tile + fp16_tile_byte(k, nl)) =
          live ? salient[(long long)(g * kGroup + k) * t.d_out + n] : __ushort_as_half(0);
    return;
  }
  constexpr int kWords = kBits == 4 ? 16 : 12;
  uint32_t words[kWords];
  for (int w = 0; w < kWords; ++w) words[w] = 0;
  __half sh = __ushort_as_half(0), zh = __ushort_as_half(0);
  if (live) {
    const int gq = g - t.g_fp16;
    sh = scales[(long long)gq * t.d_out + n];
    zh = zeros[(long long)gq * t.d_out + n];
    if (kBits == 4) {
      for (int w = 0; w < 16; ++w) {
        uint32_t v = qw[(long long)(gq * 16 + w) * t.d_out + n];
        for (int i = 0; i < 8; ++i) put_code<4>(words, w * 8 + i, (v >> (4 * i)) & 0xf);
      }
    } else {
      for (int blk = 0; blk < 4; ++blk) {
        uint32_t v[3];
        for (int w = 0; w < 3; ++w) v[w] = qw[(long long)(gq * 12 + blk * 3 + w) * t.d_out + n];
        for (int i = 0; i < 32; ++i) {
          uint32_t c = 0;
          for (int b = 0; b < 3; ++b) {
            int bit = 3 * i + b;
            c |= ((v[bit >> 5] >> (bit & 31)) & 1u) << b;
          }
          put_code<3>(words, blk * 32 + i, c);
        }
      }
    }
  }
  store_quant_tile_column<kBits>(tile, nl, words, sh, zh);
}

int launch_export(const TiledOperand &t, uint32_t *qw, __half *scales, __half *zeros, __half *salient,
                  cudaStream_t s) {
  dim3 grid(t.n_tiles, groups_per_tile(t));
  if (grid.y == 0) return ROSAQ_OK;
  if (t.bits == 3)
    export_kernel<3><<<grid, kTileN, 0, s>>>(t, qw, scales, zeros, salient);
  else
    export_kernel<4><<<grid, kTileN, 0, s>>>(t, qw, scales, zeros, salient);
  return cudaGetLastError() == cudaSuccess ? ROSAQ_OK : ROSAQ_ERR_CUDA;
}

int launch_import(const TiledOperand &t, const uint32_t *qw, const __half *scales, const __half *zeros,
                  const __half *salient, cudaStream_t s) {
  dim3 grid(t.n_tiles, groups_per_tile(t));
  if (grid.y == 0) return ROSAQ_OK;
  if (t.bits == 3)
    import_kernel<3><<<grid, kTileN, 0, s>>>(t, qw, scales, zeros, salient);
  else
    import_kernel<4><<<grid, kTileN, 0, s>>>(t, qw, scales, zeros, salient);
  return cudaGetLastError() == cudaSuccess ? ROSAQ_OK : ROSAQ_ERR_CUDA;
}

// =====================================================================================
// Online rotation operand: R (fp16, block-diagonal) re-tiled as fp16 tiles.  The "weight"
// of the rotation GEMM x . R is R itself: input channel k = row of the block, output
// column = column of the block-diagonal matrix (the permutation is applied when the
// result is stored).
// =====================================================================================
__global__ void __launch_bounds__(kTileN)
rotation_tiles_kernel(const __half *__restrict__ q, int dh, TiledOperand t) {
  // A column tile holds the groups of its (possibly merged) diagonal block: dm channels = block_groups * 128,
  // or all of d_in.  When two 128 x 128 head blocks are merged into one 256 x 256 block the off-diagonal
  // quarters are zero.
  const int nt = blockIdx.x, lg = blockIdx.y, nl = threadIdx.x;
  const int col = nt * kTileN + nl;          // column of blockdiag
  const int h = col / dh, c = col % dh;
  const int dm = t.block_groups > 0 ? t.block_groups * kGroup : t.d_in;
  const int k_base = (col / dm) * dm + lg * kGroup;             // first input channel of this group
  const __half *R = q + (long long)h * dh * dh;
  uint8_t *tile = t.blob + tile_offset(t, nt, lg);
  for (int k = 0; k < kGroup; ++k) {
    const int kg = k_base + k;
    *reinterpret_cast<__half *>(tile + fp16_tile_byte(k, nl)) = kg / dh == h ? R[(long long)(kg % dh) * dh + c] : __float2half(0.f);
  }
}

int launch_rotation_tiles(const __half *q, int d, int n_blocks, const TiledOperand &t, cudaStream_t s) {
  dim3 grid(t.n_tiles, groups_per_tile(t));
  rotation_tiles_kernel<<<grid, kTileN, 0, s>>>(q, d / n_blocks, t);
  return cudaGetLastError() == cudaSuccess ? ROSAQ_OK : ROSAQ_ERR_CUDA;
}

__global__ void invert_perm_kernel(const int32_t *__restrict__ perm, int d, int32_t *__restrict__ inv) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < d) {
    int p = perm[j];
    if (p >= 0 && p < d) inv[p] = j;
  }
}

// bad[0] = 1 when perm is not a permutation of 0..d-1: an entry out of range, or (inv still -1 somewhere
// after the scatter above) a value that never occurs, i.e. another one occurs twice
__global__ void check_perm_kernel(const int32_t *__restrict__ perm, const int32_t *__restrict__ inv, int d,
                                  int *__restrict__ bad) {
  int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < d && (perm[j] < 0 || perm[j] >= d || inv[j] < 0)) atomicExch(bad, 1);
}

// inv[perm[j]] = j.  Synchronizes the stream; ROSAQ_ERR_INVALID_ARG when perm is not a permutation (nothing
// that indexes with it has been launched then).  `bad` is a device word owned by the caller.
int launch_invert_perm(const int32_t *perm, int d, int32_t *inv, int *bad, cudaStream_t s) {
  if (cudaMemsetAsync(inv, 0xff, sizeof(int32_t) * (size_t)d, s) != cudaSuccess ||
      cudaMemsetAsync(bad, 0, sizeof(int), s) != cudaSuccess) {
    (void)cudaGetLastError();
    return ROSAQ_ERR_CUDA;
  }
  invert_perm_kernel<<<(d + 255) / 256, 256, 0, s>>>(perm, d, inv);
  check_perm_kernel<<<(d + 255) / 256, 256, 0, s>>>(perm, inv, d, bad);
  int host = 0;
  if (cudaGetLastError() != cudaSuccess || cudaMemcpyAsync(&host, bad, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    (void)cudaGetLastError();
    return ROSAQ_ERR_CUDA;
  }
  return host ? ROSAQ_ERR_INVALID_ARG : ROSAQ_OK;
}

}  // namespace rosaq
