// The GEMM stage  y = x' . W^  (Eq. 3; Eq. 6 for a block-diagonal rotation operand) for one to eight tokens.
//
// Why another kernel.  At a few tokens a launch of the tcgen05 kernel is bound by its latencies, not by the weight stream: every
// group is a chain through tensor memory (dequantise, store, barrier, eight MMAs, commit),
// and the splits of K meet in a cluster exchange of several microseconds before the next launch can begin.  Here
//   * a CTA owns a slice of 32 output columns and ALL of K, so nothing is exchanged between CTAs: its eight or sixteen warps take the
//     units of K in turn (a unit = a quantized group, or 32 channels of an fp16 group: 2 KB of a slice either way) and the
//     partial sums are added once, in shared memory, in warp order (the sums do not depend on timing);
//   * a warp streams its units on its own, with 16-byte asynchronous copies into a ring of its own: no barrier is shared with
//     another warp between x' and the sum.  x' itself is copied once per CTA (with the ring, per unit, the copies of x' cost
//     as many instructions as those of the weights: 17.1 us instead of 14.3 us for 4096 -> 2 x 11008 at one token);
//   * the products are warp-level mma.sync (m16n8k16) on weights dequantised in registers: A = 16 columns x 16 channels of
//     W^, B = 16 channels x 8 tokens;
//   * launches are chained with programmatic stream serialization: the rings of a launch fill under the tail of the one before;
//     x' and y are touched after griddepcontrol.wait.
// What bounds it: at 4096 -> 2 x 11008 the issue slots (362 instructions per unit of 2176 bytes, 0.57 issued per cycle and
// scheduler), at the smaller ones the last round of CTAs and the time to start.  Measured in a graph of distinct weights (us,
// INT4, one token; tcgen05 kernel / this one): 512 -> 512 3.3 / 1.6, 4096 -> 4096 7.7 / 4.4, 4096 -> 3 x 4096 13.9 / 9.2,
// 4096 -> 2 x 11008 19.9 / 14.3 (3.2 TB/s), 11008 -> 4096 13.1 / 8.6, rotations: dense 4096 9.9 / 6.8 (4.9 TB/s), head-wise
// 4096 4.1 / 1.95; eight tokens: 7.8 / 5.3, 14.1 / 12.9, 20.1 / 19.8, 13.3 / 11.6, 10.0 / 7.4, 4.7 / 3.0.
//
// Which channel sits in which k position of an MMA is free as long as both operands agree, so a thread feeds it the codes of
// the 16-byte chunk it loads: thread t of a quad takes channels 32 t .. 32 t + 31 of a quantized group (INT4: chunk t, INT3:
// words 3 t .. 3 t + 2), channels 8 t .. 8 t + 7 of an fp16 unit.  Rows of a slice lie 544 bytes apart in shared memory, so that
// the loads of a warp touch each bank once.
#include <algorithm>
#include <mutex>

#include "linear_common.cuh"

namespace rosaq {

namespace {

constexpr int kSmSlice = 32;                                     // output columns of a slice
constexpr int kSmRow = kSmSlice * 16 + 32;                       // bytes from one 16-byte row of a slice to the next
constexpr int kSmStage = 4 * kSmRow + kSmSlice * 4;              // 2304: rows, then scales and zero-points
constexpr int kSmWarps = 8;                                      // a multiple of 4: all fp16 units of a warp are the same quarter of a group
constexpr int kSmThreads = kSmWarps * 32;
constexpr int kSmWarpsLong = 16;                                 // of a CTA that has an SM and many units to itself
constexpr int kSmCtas = 3;                                       // resident CTAs per SM at most (80 registers)
constexpr int kSmSharedSm = 228 * 1024, kSmSharedCta = 1024;     // shared memory of an SM, and what the system takes of it per CTA
constexpr int kSmMaxProblems = 4;
constexpr int kSmMaxDevices = 64;
constexpr int kSmMaxSmem = 227 * 1024;

struct SmParams {
  int n_prob;
  int tile_start[kSmMaxProblems + 1];
  const uint8_t *blob[kSmMaxProblems];
  int d_out[kSmMaxProblems];
  __half *y[kSmMaxProblems];
  long long ldy[kSmMaxProblems];
  long long tile_stride;
  const __half *x;
  long long ldx;
  int u_fp16, n_units, block_groups;                             // units of fp16 groups, all units of a tile
  int M;
  const int32_t *col_map;
};

__device__ __forceinline__ void mma_16816(float *c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// fp16 pair p (channels 2 p, 2 p + 1) of an INT3 set of 32 channels in three words
__device__ __forceinline__ uint32_t int3_pair(const uint32_t *w, int p, uint32_t z1024, uint32_t z128, uint32_t z16, uint32_t s2) {
  if (p == 15) {
    const uint32_t tail = ((w[0] >> 15) & 0x00010001u) | ((w[1] >> 14) & 0x00020002u) | ((w[2] >> 13) & 0x00040004u);
    return h2_sub_mul(tail | 0x64006400u, z1024, s2);
  }
  const uint32_t q = w[p / 5];
  switch (p % 5) {
    case 0: return h2_sub_mul(lop_and_or(q, 0x00070007u, 0x64006400u), z1024, s2);
    case 1: return h2_sub_mul(lop_and_or(q, 0x00380038u, 0x58005800u), z128, s2);
    case 2: return h2_sub_mul(lop_and_or(q, 0x01c001c0u, 0x4C004C00u), z16, s2);
    case 3: return h2_sub_mul(lop_and_or(q >> 9, 0x00070007u, 0x64006400u), z1024, s2);
    default: return h2_sub_mul(lop_and_or(q >> 9, 0x00380038u, 0x58005800u), z128, s2);
  }
}

// Byte offset, in the row of token r, of the 16-byte chunk c of x'.  Eight lanes, rows r and r + 1 with t = 0 .. 3, read the chunks
// 4 t + v of a quantized group or t of an fp16 unit: they touch each bank once.
__device__ __forceinline__ uint32_t x_pos(int r, int c) {
  const int a = c >> 2, b = c & 3;
  return (a >> 1) * 128 + (((((a & 1) << 2) | ((a + b) & 3)) ^ ((r & 1) << 2)) << 4);
}

// acc[mt] += (columns 16 mt .. + 15) x (8 tokens), 16 channels: o[i] = two fp16 pairs of column 8 i + g, b = the same channels of
// token g
__device__ __forceinline__ void mul_pairs(const uint32_t (*o)[2], const uint4 &b, bool hi, float (*acc)[4]) {
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
    mma_16816(acc[mt], o[2 * mt][0], o[2 * mt + 1][0], o[2 * mt][1], o[2 * mt + 1][1], hi ? b.z : b.x, hi ? b.w : b.y);
}

// 32 fp16 channels; ws: this thread's position in the stage (row t, column g), b: channels 8 t .. 8 t + 7 of token g
__device__ __forceinline__ void unit_fp16(uint32_t ws, const uint4 &b, float (*acc)[4]) {
  uint4 w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) w[i] = lds128(ws + i * 128);
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    uint32_t o[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i][0] = e ? w[i].z : w[i].x, o[i][1] = e ? w[i].w : w[i].y;
    mul_pairs(o, b, e, acc);
  }
}

// a quantized group; xq[v]: address of channels 32 t + 8 v .. + 7 of token g in the first quantized group, x_unit: of this one
__device__ __forceinline__ void unit_int4(uint32_t ws, uint32_t scales, const uint32_t *xq, uint32_t x_unit, float (*acc)[4]) {
  uint32_t s2[4], z1024[4], z64[4];
  uint4 w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const ScaleZero c(lds32(scales + i * 32));
    s2[i] = c.s2, z1024[i] = c.z1024, z64[i] = c.z64;
    w[i] = lds128(ws + i * 128);
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const uint4 b = lds128(xq[v] + x_unit);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      uint32_t o[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t q0 = v == 0 ? w[i].x : v == 1 ? w[i].y : v == 2 ? w[i].z : w[i].w, q = e ? q0 >> 8 : q0;
        o[i][0] = h2_sub_mul(lop_and_or(q, 0x000f000fu, 0x64006400u), z1024[i], s2[i]);
        o[i][1] = h2_sub_mul(lop_and_or(q, 0x00f000f0u, 0x54005400u), z64[i], s2[i]);
      }
      mul_pairs(o, b, e, acc);
    }
  }
}

__device__ __forceinline__ void unit_int3(uint32_t stage, uint32_t scales, const uint32_t *xq, uint32_t x_unit, int g, int t, float (*acc)[4]) {
  uint32_t w[4][3], s2[4], z1024[4], z128[4], z16[4];
#pragma unroll
  for (int k = 0; k < 3; ++k) {                                  // words 3 t .. 3 t + 2 of four columns
    const uint32_t at = stage + ((3 * t + k) >> 2) * kSmRow + ((3 * t + k) & 3) * 4 + g * 16;
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i][k] = lds32(at + i * 128);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const ScaleZero c(lds32(scales + i * 32));
    s2[i] = c.s2, z1024[i] = c.z1024, z128[i] = c.z128, z16[i] = c.z16;
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const uint4 b = lds128(xq[v] + x_unit);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      uint32_t o[4][2];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 2; ++k) o[i][k] = int3_pair(w[i], 4 * v + 2 * e + k, z1024[i], z128[i], z16[i], s2[i]);
      mul_pairs(o, b, e, acc);
    }
  }
}

// A rotation and the linears that read it in one launch: the first CTAs are the slices of the rotation, the others copy its output
// as it appears.  The buffer between them announces its values itself: it is all ones, which no rounded value is, where nothing has been
// written yet.  The CTAs that wait need no order of starting: the launch has no more CTAs than the device has SMs, so each of them gets its
// room as soon as other launches leave it, whether the waiting ones hold theirs or not (a cooperative launch, which would say the same to the
// runtime, takes 6.2 us where this takes 4.3: 512 -> 512 at one token).
// (Aligned for its size: a launch takes the host 6.7 us with 408 or 416 bytes of parameters, 7.05 with 400, 424 or 440.)
struct alignas(32) SmPair {
  SmParams rot, lin;         // (lin.x: the values between)
  int n_rot;                 // CTAs of the rotation
  __half *other;             // the buffer of the launch before and of the one behind, kSmBetween values: emptied here
  int *status;
  long long wait_limit;
};
enum SmRole { kSmAlone, kSmProducer, kSmConsumer };

// some half of v is 0xffff
__device__ __forceinline__ uint32_t sm_missing(uint32_t v) {
  const uint32_t t = ~v;
  return (t - 0x00010001u) & ~t & 0x80008000u;
}

template <int kBits, int STAGES, int kWarps, SmRole kRole>
__device__ __forceinline__ void small_slice(uint8_t *smem, const SmParams &p, int block, const SmPair *pair) {
  constexpr int kThreads = kWarps * 32;
  static_assert(kWarps % 4 == 0 && kWarps >= kSmallTokens, "all fp16 units of a warp are the same quarter of a group; a token per warp");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  grid_dep_launch_dependents();

  const int u_fp16 = p.u_fp16, n_units = p.n_units, M = p.M;
  int prob = 0, tile = block >> 2;
  const int col = (block & 3) * kSmSlice;
  while (prob + 1 < p.n_prob && tile >= p.tile_start[prob + 1]) ++prob;
  tile -= p.tile_start[prob];
  if (tile * kTileN + col >= p.d_out[prob]) return;              // past the last column of a ragged last tile

  const int x_row = (u_fp16 * 32 + (n_units - u_fp16) * kGroup) * 2;
  const uint32_t x_smem = smem_u32(smem), ring = x_smem + M * x_row + warp * (STAGES * kSmStage), ring_end = ring + STAGES * kSmStage;

  // ---- this warp's units are warp, warp + kWarps, ...; the weights do not depend on the launches before
  constexpr int rows = kBits == 4 ? 4 : 3, quant_bytes = rows * kTileN * 16 + kScaleBytes;
  const uint8_t *const base16 = p.blob[prob] + (long long)tile * p.tile_stride + col * 16 + lane * 16;
  const uint8_t *const baseq = base16 + (long long)u_fp16 * kFp16SubBytes;
  auto fetch = [&](uint32_t st, int u) {
    const uint32_t dst = st + lane * 16;
    if (u < u_fp16) {
      const uint8_t *src = base16 + (uint32_t)u * kFp16SubBytes;
#pragma unroll
      for (int j = 0; j < 4; ++j) cp_async16(dst + j * kSmRow, src + j * (kTileN * 16));
    } else if (u < n_units) {
      const uint8_t *src = baseq + (uint32_t)(u - u_fp16) * quant_bytes;
#pragma unroll
      for (int j = 0; j < rows; ++j) cp_async16(dst + j * kSmRow, src + j * (kTileN * 16));
      if (lane < kSmSlice / 4)                                   // (the base counts 16 bytes per column; a scale pair has 4)
        cp_async16(dst + 4 * kSmRow, src + rows * (kTileN * 16) - col * 12);
    }
    cp_async_commit();
  };
  int f = warp;
#pragma unroll
  for (int s = 0; s < STAGES; ++s, f += kWarps) fetch(ring + s * kSmStage, f);

  grid_dep_wait();                                               // x may be the previous kernel's output, y its input
  if (kRole != kSmConsumer) {
    // block-diagonal operand: a tile multiplies its own channels
    const __half *xs = p.x + (p.block_groups > 0 ? (tile / p.block_groups) * p.block_groups * kGroup : 0) + threadIdx.x * 8;
    const int n_full = x_row >> 4;
    for (int r = 0; r < M; ++r, xs += p.ldx) {
      uint32_t dst = x_smem + r * x_row + x_pos(r, threadIdx.x);
      for (int c = threadIdx.x; c < n_full; c += kThreads, dst += kThreads * 16) cp_async16(dst, xs + (c - (int)threadIdx.x) * 8);
    }
  }
  if (kRole == kSmProducer) {                                    // (under the copies of x)
    uint4 *other = reinterpret_cast<uint4 *>(pair->other);
    for (int i = block * kThreads + threadIdx.x; i < kSmBetween / 8; i += pair->n_rot * kThreads) other[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
  }
  if (kRole == kSmConsumer) {
    int ok = 1;
    const int n_full = x_row >> 4, n_all = M * n_full;
    for (int i0 = threadIdx.x; i0 < n_all && ok; i0 += 4 * kThreads) {   // four chunks in flight
      uint4 v[4];
      for (long long it = 0;; ++it) {
        uint32_t missing = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int i = min(i0 + k * kThreads, n_all - 1);
          asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(v[k].x), "=r"(v[k].y), "=r"(v[k].z), "=r"(v[k].w)
                       : "l"(p.x + 8 * i)
                       : "memory");
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) missing |= sm_missing(v[k].x) | sm_missing(v[k].y) | sm_missing(v[k].z) | sm_missing(v[k].w);
        if (!missing) break;
        if (it >= pair->wait_limit) {
          ok = 0;
          break;
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = i0 + k * kThreads, r = i / n_full;
        if (i < n_all) *reinterpret_cast<uint4 *>(smem + r * x_row + x_pos(r, i - r * n_full)) = v[k];
      }
    }
    if (!__syncthreads_and(ok)) {
      if (threadIdx.x == 0) atomicExch(pair->status, (int)ROSAQ_ERR_TIMEOUT);
      asm volatile("cp.async.wait_all;" ::: "memory");
      return;
    }
  } else {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
  }

  // (rows past M repeat the last one, their products are dropped)
  const int x_tok = min(g, M - 1);
  const uint32_t x16 = x_smem + x_tok * x_row + x_pos(x_tok, (warp & 3) * 4 + t);
  uint32_t xq[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) xq[v] = x_smem + u_fp16 * 64 + x_tok * x_row + x_pos(x_tok, 4 * t + v);
  float acc[2][4] = {};
  uint32_t st = ring;
  int u = warp;
  auto next = [&] {
    __syncwarp();                                                // every lane has read the stage
    fetch(st, f);
    f += kWarps;
    st += kSmStage;
    if (st == ring_end) st = ring;
  };
  for (; u < u_fp16; u += kWarps) {
    cp_async_wait<STAGES - 1>();
    __syncwarp();
    unit_fp16(st + t * kSmRow + g * 16, lds128(x16 + (u >> 2) * (kGroup * 2)), acc);
    next();
  }
  for (; u < n_units; u += kWarps) {
    cp_async_wait<STAGES - 1>();
    __syncwarp();
    const uint32_t x_unit = (u - u_fp16) * (kGroup * 2), scales = st + 4 * kSmRow + g * 4;
    if (kBits == 4) unit_int4(st + t * kSmRow + g * 16, scales, xq, x_unit, acc);
    else unit_int3(st, scales, xq, x_unit, g, t, acc);
    next();
  }

  // ---- the partial sums [warp][token][column], each in its warp's ring; added in warp order
  float *const part = reinterpret_cast<float *>(smem + M * x_row);
  constexpr int part_stride = STAGES * kSmStage / 4;
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int tok = 2 * t + (e & 1);
      if (tok < M) part[warp * part_stride + tok * kSmSlice + mt * 16 + (e >> 1) * 8 + g] = acc[mt][e];
    }
  __syncthreads();
  const int nn = tile * kTileN + col + lane;
  if (warp < M && nn < p.d_out[prob]) {                          // (a token per warp)
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) v += part[w * part_stride + warp * kSmSlice + lane];
    __half *const at = p.y[prob] + warp * p.ldy[prob] + (p.col_map ? p.col_map[nn] : nn);
    if (kRole == kSmProducer) asm volatile("st.relaxed.gpu.global.u16 [%0], %1;" ::"l"(at), "h"(__half_as_ushort(__float2half_rn(v))) : "memory");
    else *at = __float2half_rn(v);
  }
}

template <int kBits, int STAGES, int kWarps>
__global__ void __launch_bounds__(kWarps * 32, kWarps == kSmWarps ? kSmCtas : 1)
linear_small_kernel(const __grid_constant__ SmParams p) {
  extern __shared__ __align__(128) uint8_t smem[];
  small_slice<kBits, STAGES, kWarps, kSmAlone>(smem, p, blockIdx.x, nullptr);
}

template <int kBits, int STAGES>
__global__ void __launch_bounds__(kSmThreads, kSmCtas)
rotate_linear_small_kernel(const __grid_constant__ SmPair p) {
  extern __shared__ __align__(128) uint8_t smem[];
  if ((int)blockIdx.x < p.n_rot) small_slice<4, STAGES, kSmWarps, kSmProducer>(smem, p.rot, blockIdx.x, &p);
  else small_slice<kBits, 2, kSmWarps, kSmConsumer>(smem, p.lin, blockIdx.x - p.n_rot, &p);
}

typedef void (*SmallKernel)(SmParams);
static_assert(sizeof(SmPair) == 416, "see there");
typedef void (*SmallPairKernel)(SmPair);
SmallPairKernel small_pair_pick(bool int3, int stages) {
  if (int3) return stages == 8 ? rotate_linear_small_kernel<3, 8> : stages == 4 ? rotate_linear_small_kernel<3, 4> : rotate_linear_small_kernel<3, 2>;
  return stages == 8 ? rotate_linear_small_kernel<4, 8> : stages == 4 ? rotate_linear_small_kernel<4, 4> : rotate_linear_small_kernel<4, 2>;
}
SmallKernel small_pick(bool int3, int stages, int warps) {
  if (warps == kSmWarpsLong) return int3 ? linear_small_kernel<3, 2, kSmWarpsLong> : linear_small_kernel<4, 2, kSmWarpsLong>;
  if (int3) return linear_small_kernel<3, 2, kSmWarps>;
  return stages == 8 ? linear_small_kernel<4, 8, kSmWarps> : stages == 4 ? linear_small_kernel<4, 4, kSmWarps> : linear_small_kernel<4, 2, kSmWarps>;
}

bool small_attrs() {
  bool ok = true;
  for (SmallKernel kern : {small_pick(true, 2, kSmWarps), small_pick(false, 2, kSmWarps), small_pick(false, 4, kSmWarps), small_pick(false, 8, kSmWarps),
                           small_pick(true, 2, kSmWarpsLong), small_pick(false, 2, kSmWarpsLong)})
    ok = ok && cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) == cudaSuccess &&
         cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmMaxSmem) == cudaSuccess;
  for (int i = 0; i < 6; ++i) {
    const SmallPairKernel kern = small_pair_pick(i & 1, 2 << (i >> 1));
    ok = ok && cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) == cudaSuccess &&
         cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmMaxSmem) == cudaSuccess;
  }
  if (!ok) (void)cudaGetLastError();
  return ok;
}

int small_bytes(int M, const TiledOperand &t, int stages, int warps = kSmWarps) {
  return M * groups_per_tile(t) * kGroup * 2 + warps * stages * kSmStage;
}
// A CTA that has an SM to itself issues 0.3 instructions per cycle and scheduler with two warps on each: a round of its warps (a unit each)
// takes 1300 cycles of which 724 are issue, with four warps 1800 of 1450.  Sixteen warps where that saves rounds: six rounds of eight and
// more (an INT3 unit is a longer chain: from five and a half).  us, eight / sixteen warps, one token: 11008 -> 4096 9.27 / 8.63 (INT3 9.75 /
// 8.75), 8192 -> 1024 6.8 / 6.1, 13824 -> 2048 10.2 / 9.3, 5504 -> 2048 5.35 / 5.10; up to the line 4096 -> 4096 4.78 / 5.05 (INT3 4.95 / 4.99),
// 512 -> 512 at eight tokens 2.37 / 2.62; twenty-four warps at 11008 -> 4096 9.09.  With two CTAs on an SM there are sixteen warps already.
int small_warps(const rosaq_ctx *ctx, int M, const TiledOperand &t, int tiles) {
  const int units = 4 * t.g_fp16 + t.g_quant;
  return 4 * tiles <= ctx->sm_count && t.g_quant > 0 && units > (t.bits == 3 ? 35 : 40) && small_bytes(M, t, 2, kSmWarpsLong) <= kSmMaxSmem
             ? kSmWarpsLong
             : kSmWarps;
}
int small_tiles(int n, const TiledOperand *const *ts) {
  int tiles = 0;
  for (int i = 0; i < n; ++i) tiles += ts[i]->n_tiles;
  return tiles;
}

}  // namespace

// Whether this kernel is the faster one, from its room: x' of M tokens and the rings of a CTA must leave space for a second CTA
// where the launch has more slices than SMs (5120 -> 5120 at six / eight tokens: 8.8 / 11.5 us here, 9.3 us on the tcgen05
// kernel), and for a third where it has many rounds of them (4096 -> 32000: four tokens 22.5 and 26.6 us, eight 28.0 and 26.6 us);
// and where the slices leave half of the SMs idle, where the tcgen05 kernel splits K, a CTA must not have a long K to itself
// (here, sixteen warps / there: 8192 -> 512 at four and eight tokens 6.3 / 6.4, 7.2 / 6.4, 8192 -> 1024 6.7 / 7.3, 7.55 / 7.3; 11008 -> 512 at
// three and six 7.8 / 7.75, 8.6 / 7.8; 13824 -> 2048 at two to five 9.6-10.5 / 11.9, at six, where the rings of sixteen warps have no room,
// 12.1 / 11.8; INT3 11008 -> 512 at three 8.1 / 8.0, 13824 -> 2048 at four 10.6 / 12.6).
bool linear_small_supported(const rosaq_ctx *ctx, int M, int n, const TiledOperand *const *ts) {
  const int G = groups_per_tile(*ts[0]);
  if (M > kSmallTokens || n < 1 || n > kSmMaxProblems || G <= 0) return false;
  const int bytes = small_bytes(M, *ts[0], 2), slices = 4 * small_tiles(n, ts), rounds = (slices + ctx->sm_count - 1) / ctx->sm_count;
  const int resident = rounds > 5 ? kSmCtas : std::min(rounds, 2);
  const bool int3 = ts[0]->g_quant > 0 && ts[0]->bits == 3, wide = small_warps(ctx, M, *ts[0], slices / 4) == kSmWarpsLong;
  if (2 * slices <= ctx->sm_count && M * G > std::max(int3 ? 180 : 260, wide ? (int3 ? 150 : 180) + 6 * slices : 0)) return false;
  return bytes <= kSmMaxSmem && resident * (bytes + kSmSharedCta) <= kSmSharedSm;
}

static int small_params(const __half *x, int M, long long ldx, int n, const TiledOperand *const *ts, const int32_t *col_map, __half *const *ys,
                        const long long *ldys, SmParams *out) {
  if (n < 1 || n > kSmMaxProblems || M < 1 || M > kSmallTokens) return ROSAQ_ERR_INVALID_ARG;
  const TiledOperand &t = *ts[0];
  SmParams &p = *out;
  p.n_prob = n;
  int tiles = 0;
  for (int i = 0; i < n; ++i) {
    const TiledOperand &ti = *ts[i];
    if (ti.d_in != t.d_in || ti.g_fp16 != t.g_fp16 || ti.g_quant != t.g_quant || ti.block_groups != t.block_groups ||
        (t.g_quant > 0 && ti.bits != t.bits))
      return ROSAQ_ERR_INVALID_ARG;
    p.tile_start[i] = tiles;
    p.blob[i] = ti.blob, p.d_out[i] = ti.d_out, p.y[i] = ys[i], p.ldy[i] = ldys[i];
    tiles += ti.n_tiles;
  }
  p.tile_start[n] = tiles;
  p.tile_stride = t.tile_stride;
  p.x = x, p.ldx = ldx;
  p.u_fp16 = 4 * t.g_fp16, p.n_units = p.u_fp16 + t.g_quant, p.block_groups = t.block_groups;
  p.M = M;
  p.col_map = col_map;
  return p.n_units <= 0 || small_bytes(M, t, 2) > kSmMaxSmem ? ROSAQ_ERR_UNSUPPORTED_SHAPE : ROSAQ_OK;
}

static int small_prepare(const rosaq_ctx *ctx) {
  static bool done[kSmMaxDevices] = {};                          // function attributes are per device
  static std::mutex mu;
  if (ctx->device < 0 || ctx->device >= kSmMaxDevices) return ROSAQ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lock(mu);
  if (!done[ctx->device]) {
    if (!small_attrs()) return ROSAQ_ERR_CUDA;
    done[ctx->device] = true;
  }
  return ROSAQ_OK;
}

template <typename K, typename P>
static int small_launch(K kern, const P &p, int ctas, int threads, int smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, kern, p) != cudaSuccess) {
    (void)cudaGetLastError();
    return ROSAQ_ERR_CUDA;
  }
  return ROSAQ_OK;
}

// n weights of identical geometry applied to the same activations in one launch
int launch_linear_small(const rosaq_ctx *ctx, const __half *x, int M, long long ldx, int n, const TiledOperand *const *ts,
                        const int32_t *col_map, __half *const *ys, const long long *ldys, cudaStream_t s) {
  const TiledOperand &t = *ts[0];
  SmParams p{};
  int st = small_params(x, M, ldx, n, ts, col_map, ys, ldys, &p);
  if (st == ROSAQ_OK) st = small_prepare(ctx);
  if (st != ROSAQ_OK) return st;
  const int tiles = p.tile_start[n];
  // Residency: no more CTAs per SM than the slices of this launch fill, because the CTAs of chained launches otherwise pile up
  // on some SMs while others idle (4096 -> 4096, one token, room for one / two / three CTAs: 4.4 / 6.2 / 7.5 us; 4096 -> 2 x
  // 11008 20.9 / 16.0 / 14.3 us).  Stages: two suffice for quantized groups (4096 -> 4096 4.4, with four 4.7 us); an all-fp16
  // operand has little arithmetic per byte and takes what fits (4096 dense, two / four / eight stages: 8.7 / 6.9 / 6.8 us).
  const int ctas = std::max(1, std::min(kSmCtas, (4 * tiles + ctx->sm_count - 1) / ctx->sm_count));
  const int room = std::min(kSmMaxSmem, kSmSharedSm / ctas - kSmSharedCta);
  int stages = 2;
  if (t.g_quant == 0)
    while (stages < 8 && small_bytes(M, t, 2 * stages) <= room) stages *= 2;
  const int warps = small_warps(ctx, M, t, tiles);
  // (more than a (ctas + 1)-th of an SM's shared memory)
  const int smem = std::max(small_bytes(M, t, stages, warps), ctas < kSmCtas ? (kSmSharedSm / (ctas + 1) - kSmSharedCta) / 128 * 128 + 128 : 0);
  return small_launch(small_pick(t.g_quant > 0 && t.bits == 3, stages, warps), p, 4 * tiles, warps * 32, smem, s);
}

// The rotation r of x and the n linears that read it in one launch, while every slice finds an SM of its own (4096 -> 4096 would take 13.8
// us instead of 9.4) and the values between are few: each reader copies all of them, and from 16384 on that takes longer than a second launch.
// us, two launches / one, behind a long kernel (a full queue: the device is the bound) and call by call (the host is):
//   512 -> 512    one token 4.35 / 3.9, 7.7 / 5.3     eight 5.7 / 4.8, 7.7 / 5.3
//   1024 -> 1024  one 4.95 / 4.35, 7.7 / 5.3          eight 6.4 / 5.5, 7.7 / 5.6
//   2048 -> 2048  one 6.3 / 5.9, 7.6 / 6.0            eight 7.7 / 7.6, 7.7 / 7.7
// past the line 2304 -> 1024 at eight 8.4 / 8.7, 3072 -> 1600 at six 8.8 / 9.35; 4096 -> 512 at four, on it, 11.4 / 11.6 (head-wise 6.8 / 7.1, call
// by call 7.7 / 7.2).
// A launch that is being captured costs the host nothing later, so captured calls stay two, and so do column orders, whose scatter the
// readers' polls disturb (1024 -> 3 x 1024 4.6 / 9.3).  The results are the same bits (linears whose sums sixteen warps share are not taken).
bool rotate_linear_small_supported(const rosaq_ctx *ctx, int M, const TiledOperand &r, const int32_t *col_map, int n, const TiledOperand *const *ts,
                                   cudaStream_t s) {
  const TiledOperand *rs[1] = {&r};
  if (col_map || (long long)M * r.d_out > kSmBetween || 4 * (r.n_tiles + small_tiles(n, ts)) > ctx->sm_count || !linear_small_supported(ctx, M, 1, rs) ||
      !linear_small_supported(ctx, M, n, ts) || small_warps(ctx, M, *ts[0], small_tiles(n, ts)) != kSmWarps)
    return false;
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) {
    (void)cudaGetLastError();
    return false;
  }
  return capture == cudaStreamCaptureStatusNone;
}

int launch_rotate_linear_small(rosaq_ctx *ctx, const __half *x, int M, long long ldx, const TiledOperand &r, int n,
                               const TiledOperand *const *ts, __half *const *ys, const long long *ldys, cudaStream_t s) {
  const TiledOperand &t = *ts[0];
  const TiledOperand *rs[1] = {&r};
  const long long ldxr = r.d_out;
  SmPair p{};
  // (launches of one context run in the order in which they are issued, one at a time; none of these is captured, to be run again later)
  __half *between = ctx->sm_between + (ctx->sm_turn ? kSmBetween : 0);
  p.other = ctx->sm_between + (ctx->sm_turn ? 0 : kSmBetween);
  int st = small_params(x, M, ldx, 1, rs, nullptr, &between, &ldxr, &p.rot);
  if (st == ROSAQ_OK) st = small_params(between, M, ldxr, n, ts, nullptr, ys, ldys, &p.lin);
  if (st == ROSAQ_OK) st = small_prepare(ctx);
  if (st != ROSAQ_OK) return st;
  p.n_rot = 4 * r.n_tiles;
  p.status = ctx->d_status;
  p.wait_limit = ctx->wait_limit;
  const int grid = p.n_rot + 4 * p.lin.tile_start[n], ctas = std::max(1, std::min(kSmCtas, (grid + ctx->sm_count - 1) / ctx->sm_count));
  const int room = std::min(kSmMaxSmem, kSmSharedSm / ctas - kSmSharedCta);
  int stages = 2;
  while (stages < 8 && small_bytes(M, r, 2 * stages) <= room) stages *= 2;
  const int need = std::max(small_bytes(M, r, stages), small_bytes(M, t, 2));
  const int smem = std::max(need, ctas < kSmCtas ? (kSmSharedSm / (ctas + 1) - kSmSharedCta) / 128 * 128 + 128 : 0);
  st = small_launch(small_pair_pick(t.g_quant > 0 && t.bits == 3, stages), p, grid, kSmThreads, smem, s);
  if (st == ROSAQ_OK) ctx->sm_turn ^= 1;
  return st;
}

}  // namespace rosaq
