// The GEMM stage  y = x . W^  (Eq. 3; x . R of Eq. 2 / Eq. 6 is the same contraction) for prefill-sized batches: more than
// 128 tokens.
//
// Why another kernel.  With a few hundred tokens the stage is bound by the tensor pipe, not by the weight
// stream, and what counts is how many tokens share one dequantisation of a weight tile and how often an
// operand byte is fetched from L2: a weight tile dequantised for 128 tokens costs as many instructions (317 cycles of an SM)
// as one dequantised for 256, next to 512 and 1024 cycles of MMAs, and a CTA that multiplies 128 columns with 256 tokens on its own
// pulls 64 KB of activations per 128-channel group.  Here two CTAs of a cluster (adjacent SMs) share a
// tile of 256 columns x NT <= 256 tokens as a cta_group::2 pair: rank r dequantises column tile 2 c + r into its own
// tensor memory (the A operand, 128 lanes each) and loads half of the token rows (its half of the B
// operand), the leader issues M = 256, N = NT MMAs for both, and each CTA ends up with the
// accumulator of its own 128 columns for all NT tokens.  A weight tile is dequantised once per 256 tokens.
// Several weights that multiply the same activations (q/k/v, gate/up) run in one launch, their column pairs side by side.
//
// All-fp16 operands (rotations) need no dequantisation: a fp16 tile lies in memory as the tensor core reads it (K-major,
// no swizzle), so both operands come straight from shared memory, the launch has no dequantisation warps, and the tensor
// memory they would fill holds a second accumulator.  (4096 -> 4096 dense rotation, 1900 tokens: 88 us through tensor
// memory, 57 so, 80 on the per-call kernel.)
//
// Work is cut in one of two ways (prefill_choose):
//   * S > 0: a cluster of S pairs per tile, each with 1 / S of the groups.  The partial rows meet in distributed shared memory
//     (two cluster barriers, 2-3 us).  Used while all clusters are resident at once.
//   * S = 0, equal shares: the list of (tile, 128-channel group) units, token blocks of one column pair
//     next to each other so that the second one finds the packed weights in L2, is cut into one contiguous range
//     of about equal cost per pair (a 13B projection at 512 tokens is 108 tiles for 74 pairs: whole tiles
//     would take two rounds, equal ranges take 1.46).  The first piece of a range can be the end of a tile; its partial tile
//     (fp32) goes to a workspace and a flag is raised.  The last piece can be a tile without its last groups: the pairs that
//     hold it so ("closers") each finish a share of its token rows: they store the other rows of their own partial tile, wait
//     for the flags of the other holders, fetch their rows with bulk copies and add them.  A flag counts the readers that
//     have yet to fetch; the last one puts it back to zero, so every launch, replays of a captured launch included, starts
//     from zero flags.  The launch is cooperative: closers wait for one another, so every pair must be resident.  A
//     handshake through L2 costs 3 us from the flag's store to the reader, the whole exchange about 8.
// In both, sums are added in a fixed order: the same bits on every run.
//
// Per CTA: warp 0 = weight-tile producer (bulk copies; one sub-ring of slots per dequantisation team; for an fp16 operand the
// producer of both operands), 1 = activation producer (TMA, bytes of both CTAs counted on the leader's barrier),
// 2 = MMA issuer (leader only; also owns the tensor memory), 4..19 = four dequantisation teams (group j of the CTA's stream
// goes to team and operand buffer j mod 4), the last eight = epilogue (two warps per TMEM lane quadrant, alternate blocks of
// sixteen tokens).  Tensor memory: accumulator in columns 0..255, four operand buffers of 64 columns behind it, so the
// accumulator of a quantized weight is single: the epilogue therefore rounds a finished tile into registers (64 of them, which
// setmaxnreg takes from the other warps), gives the accumulator back and only then stores.  Loads carry no cluster
// multicast.
// Every wait is bounded; a CTA that gives up records ROSAQ_ERR_TIMEOUT, lets its copies and MMAs in flight
// finish, frees its tensor memory and returns.
#include <cuda.h>

#include <algorithm>
#include <mutex>

#include "linear_common.cuh"

namespace rosaq {

namespace {

constexpr int kPfTmemCols = 512;
constexpr int kPfMaxTokens = 256;                   // most tokens per tile = N of the MMA
constexpr int kPfStages = 4;                        // operand buffers, each with its activation slot
constexpr int kPfTeams = 4;
constexpr int kPfFirstDequantWarp = 4, kPfFirstEpiWarp = kPfFirstDequantWarp + 4 * kPfTeams;
constexpr int kPfEpiThreads = 256;
constexpr int kPfThreads = kPfFirstEpiWarp * 32 + kPfEpiThreads;   // 896
// Registers: 72 per thread at launch; 128 x 40 + 512 x 64 + 256 x 104 = 896 x 72.
constexpr int kPfRegsLaunch = 72, kPfRegsRoles = 40, kPfRegsDequant = 64, kPfRegsEpi = 104;
static_assert(128 * kPfRegsRoles + kPfTeams * kTeamThreads * kPfRegsDequant + kPfEpiThreads * kPfRegsEpi == kPfThreads * kPfRegsLaunch,
              "the warpgroups share the registers of the launch");
constexpr int kPfMaxNW = 16;                        // weight slots (a multiple of the teams)
constexpr int kPfMaxSmemBytes = 227 * 1024;
constexpr int kPfMaxProblems = 4;
constexpr int kPfMaxPairs = 96;                     // of a launch cut into equal shares
constexpr int kPfMaxSplits = 4;                     // pairs in a cluster (eight CTAs: the portable limit)
constexpr int kDenseBits = 16;                      // an operand without quantized groups
constexpr int kPdEpiWarp = 4, kPdThreads = kPdEpiWarp * 32 + kPfEpiThreads;   // 384
constexpr int kPdMaxStages = 8;                     // stages of 64 channels
constexpr int kPdABytes = kFp16TileBytes / 2;       // 64 channels x 128 columns

struct alignas(64) PfParams {
  CUtensorMap xmap, xmap_last;                      // boxes of NT / 2 tokens, of NT_last / 2
  CUtensorMap wmap[kPfMaxProblems];                 // all-fp16 operands: the blob as rows of 128 bytes
  int n_prob;
  int pair_start[kPfMaxProblems + 1];
  const uint8_t *blob[kPfMaxProblems];
  __half *y[kPfMaxProblems];
  long long ldy[kPfMaxProblems];
  int d_out[kPfMaxProblems], n_tiles[kPfMaxProblems];
  long long tile_stride;
  int g_fp16, groups, block_groups;
  int n_tok_blocks, M;
  int NT;                     // tokens per tile (a multiple of 32); a CTA keeps NT / 2 rows of x in shared memory
  int NT_last;                // of the tiles of the last token block, which may hold fewer
  int NW;                     // weight slots; all-fp16 operands: stages
  int units;                  // (column pairs x token blocks) x groups
  int S;
  float *partials;            // [pair][2][rank][NT tokens][128 columns]: of the first and of the last piece of a range
  unsigned *flags;            // [pair][2][rank]: readers that still have to fetch from the slot
  int *status;
  long long wait_limit;
  int bounds[kPfMaxPairs + 1];   // S = 0: pair i holds the units [bounds[i], bounds[i + 1])
};

// whether work item wk is a tile of the last token block, and its tokens
__device__ __forceinline__ bool pf_last_block(const PfParams &p, int wk) { return (wk + 1) % p.n_tok_blocks == 0; }
__device__ __forceinline__ int pf_tokens(const PfParams &p, int wk) { return pf_last_block(p, wk) ? p.NT_last : p.NT; }
// next piece of the range [u, end): groups [g0, g1) of work item wk; false when the range is used up
__device__ __forceinline__ bool pf_next_piece(int &u, int end, int G, int &wk, int &g0, int &g1) {
  if (u >= end) return false;
  wk = u / G;
  g0 = u - wk * G;
  const int len = min(G - g0, end - u);
  g1 = g0 + len;
  u += len;
  return true;
}
// weight and column pair of work item wk
__device__ __forceinline__ int pf_problem(const PfParams &p, int wk, int &col_pair) {
  col_pair = wk / p.n_tok_blocks;
  int prob = 0;
  while (prob + 1 < p.n_prob && col_pair >= p.pair_start[prob + 1]) ++prob;
  col_pair -= p.pair_start[prob];
  return prob;
}
// the 256 epilogue threads agree on whether to go on (all of them always come here)
__device__ __forceinline__ bool pf_epi_vote(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.and.pred p, 1, 256, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ unsigned pf_ld_relaxed(const unsigned *ptr) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ptr) : "memory");
  return v;
}
template <int kRegs>
__device__ __forceinline__ void reg_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegs));
}
template <int kRegs>
__device__ __forceinline__ void reg_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegs));
}
// The fp16 tile of an operand (16-byte chunks of eight channels, column by column) is a K-major operand without swizzle:
// eight columns 128 bytes apart from the next eight, the next eight channels kTileN * 16 bytes further.
__device__ __forceinline__ uint64_t make_a_desc(uint32_t smem_addr) {
  return (uint64_t)((smem_addr >> 4) & 0x3fff) | ((uint64_t)(kTileN * 16 >> 4) << 16) | ((uint64_t)(128 >> 4) << 32) | (1ull << 46);
}
// four MMAs = 64 channels; A advances by two chunks (4096 bytes) per MMA, B by 32 bytes inside a swizzle row
__device__ __forceinline__ void tc_mma4_ss_pair(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q, e;\n\t.reg .b64 ta, tb;\n\t"
      "elect.sync _|e, 0xffffffff;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 q, 0, 0;\n\t"
      "@e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t"
      "add.u64 ta, %1, 256;\n\tadd.u64 tb, %2, 2;\n\t@e tcgen05.mma.cta_group::2.kind::f16 [%0], ta, tb, %3, q;\n\t"
      "add.u64 ta, %1, 512;\n\tadd.u64 tb, %2, 4;\n\t@e tcgen05.mma.cta_group::2.kind::f16 [%0], ta, tb, %3, q;\n\t"
      "add.u64 ta, %1, 768;\n\tadd.u64 tb, %2, 6;\n\t@e tcgen05.mma.cta_group::2.kind::f16 [%0], ta, tb, %3, q;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ uint32_t pf_pack(uint32_t lo, uint32_t hi) {          // two fp32 bit patterns, each rounded once
  __half2 r = __floats2half2_rn(__uint_as_float(lo), __uint_as_float(hi));
  return *reinterpret_cast<uint32_t *>(&r);
}
// Writes sixteen tokens t0 .. of 32 columns n0 .. (a warp): h[j] = tokens 2 j, 2 j + 1 of this lane's column.  When the
// warp's columns are all there, three rounds of exchange between lanes turn the columns into rows of eight, so that a
// lane writes 16 bytes twice instead of 2 bytes sixteen times.
__device__ __forceinline__ void pf_store_block(const uint32_t *h, __half *y, int n0, int d_out, int t0, int M, long long ldy, int lane) {
  if (n0 + 32 <= d_out) {
    uint32_t r[8];
    const bool b0 = lane & 1, b1 = lane & 2, b2 = lane & 4;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t o = __shfl_xor_sync(0xffffffffu, h[j], 1);
      r[j] = __byte_perm(h[j], o, b0 ? 0x3276 : 0x5410);       // token 2 j + b0, two columns
    }
    uint32_t e[4][2];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t o = __shfl_xor_sync(0xffffffffu, b1 ? r[2 * q] : r[2 * q + 1], 2);
      e[q][0] = b1 ? o : r[2 * q], e[q][1] = b1 ? r[2 * q + 1] : o;
    }
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      uint32_t o[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) o[k] = __shfl_xor_sync(0xffffffffu, b2 ? e[2 * m][k] : e[2 * m + 1][k], 4);
      const uint4 v = b2 ? make_uint4(o[0], o[1], e[2 * m + 1][0], e[2 * m + 1][1]) : make_uint4(e[2 * m][0], e[2 * m][1], o[0], o[1]);
      const int tok = t0 + 8 * m + (lane & 7);
      if (tok < M) *reinterpret_cast<uint4 *>(y + (long long)tok * ldy + n0 + (lane & 24)) = v;
    }
    return;
  }
  if (n0 + lane >= d_out) return;
  __half *yp = y + (long long)t0 * ldy + n0 + lane;
#pragma unroll
  for (int j = 0; j < 8; ++j, yp += 2 * ldy) {
    if (t0 + 2 * j < M) *yp = __ushort_as_half((unsigned short)(h[j] & 0xffffu));
    if (t0 + 2 * j + 1 < M) yp[ldy] = __ushort_as_half((unsigned short)(h[j] >> 16));
  }
}
// the two cluster barriers around the exchange of a split tile, for the warps that have no part in it
__device__ __forceinline__ void pf_join_exchange() {
  cluster_arrive();
  cluster_wait();
  cluster_arrive();
  cluster_wait();
}

// kBits: 3 or 4, or kDenseBits for an operand without quantized groups.
template <int kBits>
__global__ void __launch_bounds__(kBits == kDenseBits ? kPdThreads : kPfThreads, 1)
linear_prefill_kernel(const __grid_constant__ PfParams p) {
  constexpr bool kDense = kBits == kDenseBits;
  constexpr int kFirstEpi = kDense ? kPdEpiWarp : kPfFirstEpiWarp;
  constexpr int kAcc = kDense ? 2 : 1;                         // accumulators
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const int NT = p.NT, rows = NT >> 1, NW = p.NW;
  // quantized: kPfStages activation slots of a group (128 channels), then NW weight slots;
  // dense: NW stages of half a group, the weights' 64 channels x 128 columns and the activations' behind them
  const uint32_t x_slot_bytes = (uint32_t)rows * (kDense ? 128u : 256u);
  const uint32_t d_stage_bytes = kPdABytes + x_slot_bytes;
  const uint32_t x_ring = base;
  const uint32_t w_ring = x_ring + kPfStages * x_slot_bytes;
  const uint32_t ring_bytes = kDense ? NW * d_stage_bytes : kPfStages * x_slot_bytes;
  const uint32_t bars = kDense ? base + NW * d_stage_bytes : w_ring + NW * kWSlotBytes;
  const uint32_t bar_w_full = bars, bar_w_empty = bar_w_full + 8 * NW;     // dense: a stage's copies (leader's) / its MMAs done
  const uint32_t bar_a_full = bar_w_empty + 8 * NW;            // operand buffers written + activation slots landed (leader's)
  const uint32_t bar_s_empty = bar_a_full + 8 * kPfStages;     // stage consumed by its MMAs (both CTAs)
  const uint32_t bar_d_full = bar_s_empty + 8 * kPfStages;     // accumulators complete (both CTAs)
  const uint32_t bar_d_empty = bar_d_full + 16;                // accumulators drained by both CTAs (leader's)
  const uint32_t bar_drain = bar_d_empty + 16;
  const uint32_t bar_merge = bar_drain + 8;                    // partial tiles have landed in the ring
  const uint32_t misc = bar_merge + 8;                         // [0] TMEM base, [1] abort flag
  uint32_t *misc_ptr = reinterpret_cast<uint32_t *>(smem_raw + (misc - smem_u32(smem_raw)));

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t rank = blockIdx.x & 1u;                       // position in the pair; 0 = leader
  const bool is_lead = rank == 0;
  const int pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
  const int S = p.S, G = p.groups;
  const int split = S > 1 ? pair % S : 0;                      // this pair's position in its cluster
  const uint32_t lead = 2u * (uint32_t)split, pair_mask = 3u << lead;   // cluster rank of the pair's leader; its two CTAs
  int u_begin, u_end;
  if (S > 0) {
    const int wk0 = (pair / S) * G;
    u_begin = wk0 + G * split / S, u_end = wk0 + G * (split + 1) / S;
  } else {
    u_begin = p.bounds[pair], u_end = p.bounds[pair + 1];
  }
  const Abort ab{reinterpret_cast<volatile int *>(misc_ptr + 1), p.status, p.wait_limit};
  grid_dep_launch_dependents();

  if (threadIdx.x == 0) {
    for (int i = 0; i < NW; ++i) {
      mbar_init(bar_w_full + 8 * i, 1);
      mbar_init(bar_w_empty + 8 * i, kDense ? 1 : kTeamThreads);
    }
    for (int i = 0; i < kPfStages; ++i) {
      mbar_init(bar_a_full + 8 * i, 2 * (kTeamThreads / 32) + 1);   // a team's warps in both CTAs + the activation copies
      mbar_init(bar_s_empty + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_d_full + 8 * i, 1);
      mbar_init(bar_d_empty + 8 * i, 2 * (kPfEpiThreads / 32));     // one arrival per epilogue warp of both CTAs
    }
    mbar_init(bar_drain, 1);
    mbar_init(bar_merge, 1);
    misc_ptr[1] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) tmem_alloc_pair<kPfTmemCols>(misc);           // both CTAs of the pair, same warp index
  tc_fence_before();
  __syncthreads();
  cluster_arrive();                                            // the peer's barriers and tensor memory exist
  cluster_wait();
  tc_fence_after();
  const uint32_t tmem = misc_ptr[0];
  const uint32_t a_col0 = kPfMaxTokens;                        // operand buffers follow the accumulator

  // (what comes before the roles join again stays inside each role: the warps have different numbers of registers)
  if (warp < 4) {
    if (!kDense) reg_dec<kPfRegsRoles>();
    if (kDense && warp == 0) {
      // ---------------- dense producer: per stage this CTA's half of both operands, all bytes counted on the leader's barrier
      if (lane == 0) {
        grid_dep_wait();                                       // x may be the previous kernel's output
        int issued = 0;
        Ring rs{0, 0};
        bool live = true;
        int u = u_begin, wk, g0, g1;
        while (live && !ab.set() && pf_next_piece(u, u_end, G, wk, g0, g1)) {
          int col_pair;
          const int prob = pf_problem(p, wk, col_pair);
          const int my_tile = min(2 * col_pair + (int)rank, p.n_tiles[prob] - 1);
          const int a_row0 = (int)((long long)my_tile * p.tile_stride >> 7);     // rows of 128 bytes
          const int n_tok = pf_tokens(p, wk), tok0 = (wk % p.n_tok_blocks) * NT + (int)rank * (n_tok >> 1);
          const CUtensorMap *const xmap = n_tok == NT ? &p.xmap : &p.xmap_last;
          const uint32_t bytes = 2 * (kPdABytes + (uint32_t)(n_tok >> 1) * 128u);
          // block-diagonal operand: the pair of column tiles multiplies the channels of its own diagonal block
          const int g_block0 = p.block_groups > 0 ? (2 * col_pair / p.block_groups) * p.block_groups : 0;
          for (int h = 2 * g0; h < 2 * g1; ++h, ++issued, rs.advance(NW)) {
            if (!ab.wait(bar_w_empty + 8 * rs.idx, rs.lap ^ 1u)) {
              live = false;
              break;
            }
            if (is_lead) mbar_arrive_expect_tx(bar_w_full + 8 * rs.idx, bytes);
            const uint32_t bar = map_to_rank(bar_w_full + 8 * rs.idx, lead), dst = base + rs.idx * d_stage_bytes;
            tma_load_2d_pair(dst, &p.wmap[prob], bar, 0, a_row0 + h * (kPdABytes / 128));
            tma_load_3d_pair(dst + kPdABytes, xmap, bar, tok0, 2 * g_block0 + h);
          }
        }
        // (the leader's barriers count the copies of both CTAs, and the peer stays until the cluster barrier
        // at the end of the kernel, which the leader reaches after this drain: the last stage that it waits for, for as long as the
        // limit goes, is one that it has not posted, but the peer may have asked for)
        if (ab.set() && is_lead) {
          for (int back = min(NW, issued); back >= 0; --back) {
            const int k = issued - back;
            for (int it = 0; it < kDrainPolls; ++it)
              if (mbar_try_wait(bar_w_full + 8 * (k % NW), (k / NW) & 1)) break;
          }
        }
      }
    } else if (!kDense && warp == 0) {
      // ---------------- weight-tile producers
      if (lane < kPfTeams) {
        const int qbytes = quant_tile_bytes(kBits), team = lane;
        int u = u_begin, wk, j0 = 0, g = -kPfTeams, g_end = 0;
        const uint8_t *base = nullptr;
        feed_teams<kPfTeams, false>(ab, team, NW / kPfTeams, w_ring, bar_w_full, bar_w_empty, [&](WeightCopies &c) {
          g += kPfTeams;                             // the team's next group, in this piece or a later one
          while (g >= g_end) {
            int g0;
            if (!pf_next_piece(u, u_end, G, wk, g0, g_end)) return false;
            // (the second CTA of a pair on an odd last tile streams that tile again; its results are dropped)
            int col_pair;
            const int prob = pf_problem(p, wk, col_pair);
            const int my_tile = min(2 * col_pair + (int)rank, p.n_tiles[prob] - 1);
            base = p.blob[prob] + (long long)my_tile * p.tile_stride;
            g = g0 + ((team - j0) & (kPfTeams - 1));
            j0 += g_end - g0;
          }
          const bool f16 = g < p.g_fp16;
          c.src = base + (f16 ? (long long)g * kFp16TileBytes : (long long)p.g_fp16 * kFp16TileBytes + (long long)(g - p.g_fp16) * qbytes);
          c.bytes = f16 ? kFp16SubBytes : qbytes;
          c.left = f16 ? 3 : 0;
          return true;
        });
      }
    } else if (!kDense && warp == 1) {
      // ---------------- activation producer: this CTA's half of the token rows of every group (the whole warp, converged)
      {
        grid_dep_wait();                                       // x may be the previous kernel's output
        int gc = 0;
        Ring rs{0, 0};
        bool live = true;
        int u = u_begin, wk, g0, g1;
        while (live && !ab.set_all() && pf_next_piece(u, u_end, G, wk, g0, g1)) {
          const int n_tok = pf_tokens(p, wk), tok0 = (wk % p.n_tok_blocks) * NT + (int)rank * (n_tok >> 1);
          const CUtensorMap *const xmap = n_tok == NT ? &p.xmap : &p.xmap_last;
          for (int g = g0; g < g1; ++g, ++gc, rs.advance(kPfStages)) {
            const int slot = rs.idx;
            if (!ab.wait_all(bar_s_empty + 8 * slot, rs.lap ^ 1u)) {
              live = false;
              break;
            }
            // all bytes are counted on the leader's barrier
            if (elect_one()) {
              if (is_lead) mbar_arrive_expect_tx(bar_a_full + 8 * slot, (uint32_t)n_tok * 256u);
              tma_load_3d_pair(x_ring + slot * x_slot_bytes, xmap, map_to_rank(bar_a_full + 8 * slot, lead), tok0, 2 * g);
            }
            __syncwarp();
          }
        }
        if (lane == 0 && ab.set() && is_lead) {
          for (int back = min(kPfStages, gc); back >= 0; --back) {     // (as above)
            const int k = gc - back;
            for (int it = 0; it < kDrainPolls; ++it)
              if (mbar_try_wait(bar_a_full + 8 * (k % kPfStages), (k / kPfStages) & 1)) break;
          }
        }
      }
    } else if (warp == 2) {
      // ---------------- MMA issuer (leader): per group one wait, eight MMAs of 256 x NT x 16, one commit (dense: half a group)
      if (is_lead) {
        const uint64_t desc0 = make_b_desc(kDense ? base + kPdABytes : x_ring), adesc0 = make_a_desc(base);
        const uint32_t slot16 = (kDense ? d_stage_bytes : x_slot_bytes) >> 4;
        Ring rs{0, 0};
        int n_done = 0;
        bool live = true, issued = false;
        int u = u_begin, wk, g0, g1;
        for (; live && pf_next_piece(u, u_end, G, wk, g0, g1); ++n_done) {
          const int buf = kDense ? n_done & 1 : 0;
          if (!ab.wait_all(bar_d_empty + 8 * buf, (uint32_t)((n_done / kAcc) & 1) ^ 1u)) break;   // the last piece in it has been drained
          tc_fence_after();
          const uint32_t d_tmem = tmem + buf * kPfMaxTokens;
          const int n = (g1 - g0) * (kDense ? 2 : 1);
          // (n_tok comes straight from the parameters in either call, so the descriptors stay in uniform registers: selected, each MMA moved
          // them there, and launches of equal blocks were 2 to 5 % slower)
          auto run = [&](const int n_tok) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(n_tok >> 3) << 17) | (16u << 24), half16 = (uint32_t)n_tok * 4u;   // (n_tok / 2 rows of 128 bytes)
            uint32_t accumulate = 0;
            for (int i = 0; i < n; ++i, rs.advance(kDense ? NW : kPfStages)) {
              const int st = rs.idx;
              if (!ab.wait_all((kDense ? bar_w_full : bar_a_full) + 8 * st, rs.lap)) return false;
              tc_fence_after();
              const uint64_t b0 = desc0 + (uint64_t)(st * slot16);
              if (kDense) {
                tc_mma4_ss_pair(d_tmem, adesc0 + (uint64_t)(st * slot16), b0, idesc, accumulate);
                tc_commit_mc(bar_w_empty + 8 * st, pair_mask);   // frees the stage in both CTAs
              } else {
                tc_mma8_ts_pair(d_tmem, tmem + a_col0 + st * 64, b0, b0 + (uint64_t)half16, idesc, accumulate);
                tc_commit_mc(bar_s_empty + 8 * st, pair_mask);
              }
              accumulate = 1;
              issued = true;
            }
            return true;
          };
          live = pf_last_block(p, wk) ? run(p.NT_last) : run(p.NT);
          if (!live) break;
          tc_commit_mc(bar_d_full + 8 * buf, pair_mask);
        }
        if (ab.set_all() && issued) {  // MMAs already issued must retire before the tensor memory is given back
          tc_commit_mc(bar_drain, 1u << lead);
          for (int it = 0; it < kDrainPolls; ++it)
            if (mbar_try_wait(bar_drain, 0)) break;
        }
      }
    }
    __syncwarp();
    if (S > 1) pf_join_exchange();
  } else if (!kDense && warp < kFirstEpi) {
    // ---------------- dequantisation: group j of the CTA's stream goes to team and operand buffer j mod 4
    reg_dec<kPfRegsDequant>();
    const int quad = warp & 3;
    const int team = (warp - kPfFirstDequantWarp) >> 2;
    const int n = quad * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(quad * 32) << 16);
    const int NWT = NW / kPfTeams;
    const uint32_t my_ring = w_ring + team * NWT * kWSlotBytes, my_full = bar_w_full + 8 * team * NWT,
                   my_empty = bar_w_empty + 8 * team * NWT;
    const uint32_t a_addr = lane_addr + a_col0 + team * 64;
    const uint32_t my_s_empty = bar_s_empty + 8 * team, my_a_full = map_to_rank(bar_a_full + 8 * team, lead);
    Ring rw{0, 0};
    bool ok = true;
    int j0 = 0;                                      // position of the tile's first group in the CTA's stream
    uint32_t use = 0;                                // how often this team's buffer was used before
    int u = u_begin, wk, g0, g1;
    while (ok && pf_next_piece(u, u_end, G, wk, g0, g1)) {
      for (int g = g0 + ((team - j0) & (kPfTeams - 1)); g < g1 && ok; g += kPfTeams, ++use) {
        const bool f16 = g < p.g_fp16;
        const int nsub = f16 ? 4 : 1;
        bool got = ab.wait(my_s_empty, (use & 1u) ^ 1u);
        for (int sub = 0; sub < nsub && ok; ++sub, rw.advance(NWT)) {
          got = got && ab.wait(my_full + 8 * rw.idx, rw.lap);
          got = __all_sync(0xffffffffu, got);        // the TMEM instructions below need the whole warp
          if (!got) {
            ok = false;
            break;
          }
          tc_fence_after();
          dequant_unit<kDense ? 4 : kBits>(f16, my_ring + rw.idx * kWSlotBytes, n, a_addr, sub, my_empty + 8 * rw.idx);
        }
        tc_wait_st();
        if (!ok) break;
        tc_fence_before();
        __syncwarp();                                // one arrival per warp, on the leader's barrier
        if (lane == 0) mbar_arrive_cluster(my_a_full);
      }
      j0 += g1 - g0;
    }
    if (S > 1) pf_join_exchange();
  } else if (warp >= kFirstEpi) {
    // ---------------- epilogue: thread = (output column n of this CTA's tile = TMEM lane, every other block of sixteen
    // tokens = TMEM columns)
    if (!kDense) reg_inc<kPfRegsEpi>();
    const int quad = warp & 3;
    const int n = quad * 32 + lane;
    const int hf = (warp - kFirstEpi) >> 2;
    const bool epi_lead = threadIdx.x == kFirstEpi * 32;
    const long long slot_floats = (long long)NT * kTileN;                        // one CTA's partial tile
    auto slot_of = [&](int pr, int which) { return p.partials + ((long long)pr * 4 + which * 2 + (int)rank) * slot_floats; };
    auto flag_of = [&](int pr, int which) { return p.flags + pr * 4 + which * 2 + (int)rank; };
    uint32_t lane_addr = 0;
    // blocks [b0, b1) of the accumulator -> a partial tile
    auto store_partial = [&](float *slot, int b0, int b1) {
      for (int bk = b0 + hf; bk < b1; bk += 2) {
        uint32_t v[16];
        tmem_ld16(lane_addr + bk * 16, v);
        tc_wait_ld();
        float *dp = slot + (long long)bk * 16 * kTileN + n;
#pragma unroll
        for (int e = 0; e < 16; ++e) dp[e * kTileN] = __uint_as_float(v[e]);
      }
    };
    auto raise_flag = [&](unsigned *flag, int readers) {
      pf_epi_vote(true);                                       // all stores of the CTA are issued ...
      if (epi_lead) {
        __threadfence();                                       // ... and ordered before the flag (cumulative fence)
        asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(flag), "r"((unsigned)readers) : "memory");
      }
    };
    if (S <= 1) grid_dep_wait();   // y, the partial tiles and the flags may still be in use by the previous kernel
    int n_done = 0;
    int u = u_begin, wk, g0, g1;
    for (; S <= 1 && pf_next_piece(u, u_end, G, wk, g0, g1); ++n_done) {
      const int buf = kDense ? n_done & 1 : 0;
      lane_addr = tmem + ((uint32_t)(quad * 32) << 16) + buf * kPfMaxTokens;
      auto release = [&]() {                                   // the accumulator is free for the next piece but one (dense: two)
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_to_rank(bar_d_empty + 8 * buf, lead));
      };
      const bool have_d = ab.wait(bar_d_full + 8 * buf, (uint32_t)((n_done / kAcc) & 1));
      if (!pf_epi_vote(have_d && !ab.set())) break;
      tc_fence_after();
      int col_pair;
      const int prob = pf_problem(p, wk, col_pair);
      const int tile = 2 * col_pair + (int)rank;
      const int d_out = tile < p.n_tiles[prob] ? p.d_out[prob] : 0;              // (a tile that is not there writes nothing)
      const int n0 = tile * kTileN + quad * 32;
      __half *const y = p.y[prob];
      const long long ldy = p.ldy[prob];
      const int tok0 = (wk % p.n_tok_blocks) * NT;
      const int n_blk = (min(NT, p.M - tok0) + 15) >> 4;       // blocks of sixteen tokens in this tile
      // the pairs `first` .. `last` hold the tile's groups, ascending K
      int first = pair, last = pair;
      if (S == 0) {
        while (p.bounds[first] > wk * G) --first;
        while (p.bounds[last + 1] < (wk + 1) * G) ++last;
      }
      const int closers = last - first;                        // all holders but the last share the tile's token rows
      if (closers == 0) {
        // the whole tile is here: round it into registers, give the accumulator back, then store
        uint32_t h[8][8];
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
          uint32_t v[2][16];
#pragma unroll
          for (int k = 0; k < 2; ++k)
            if (hf + 2 * (i + k) < n_blk) tmem_ld16(lane_addr + (hf + 2 * (i + k)) * 16, v[k]);
          tc_wait_ld();
#pragma unroll
          for (int k = 0; k < 2; ++k)
#pragma unroll
            for (int j = 0; j < 8; ++j) h[i + k][j] = pf_pack(v[k][2 * j], v[k][2 * j + 1]);
        }
        release();
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (hf + 2 * i < n_blk) pf_store_block(h[i], y, n0, d_out, tok0 + (hf + 2 * i) * 16, p.M, ldy, lane);
        continue;
      }
      if (pair == last) {
        // the first piece of this range: its partial tile goes to the workspace
        store_partial(slot_of(pair, 0), 0, n_blk);
        release();
        raise_flag(flag_of(pair, 0), closers);
        continue;
      }
      int b0 = 0, b1 = n_blk;                                  // the blocks of token rows this pair finishes
      const int mine = pair - first;
      if (closers > 1) {
        b0 = n_blk * mine / closers, b1 = n_blk * (mine + 1) / closers;
        store_partial(slot_of(pair, 1), 0, b0);
        store_partial(slot_of(pair, 1), b1, n_blk);
        raise_flag(flag_of(pair, 1), closers - 1);
      }
      // This is the last piece of the range, so the ring is free: the other holders' rows come in as bulk copies, about a
      // whole tile in all (read straight from L2, sixteen loads at a time per thread, a tile took 6 us), and are added in
      // ascending order of the holders.
      const uint32_t share_bytes = (uint32_t)(b1 - b0) * 16 * kTileN * 4;
      const int fit = share_bytes > 0 ? (int)(ring_bytes / share_bytes) : closers;   // holders per round; the ring holds a whole tile
      bool alive = true;
      uint32_t phase = 0;
      for (int h0 = 0; h0 < closers && alive; h0 += fit) {
        const int h1 = min(closers, h0 + fit);                 // others: 0 .. closers - 1 = holders without `pair`
        if (warp == kFirstEpi) {
          // a lane per holder: the flags are polled and the copies issued side by side
          if (lane == 0) mbar_arrive_expect_tx(bar_merge, share_bytes * (uint32_t)(h1 - h0));
          __syncwarp();
          for (int o0 = h0; o0 < h1; o0 += 32) {
            const int o = o0 + lane, h = first + o + (o >= mine ? 1 : 0), which = h == last ? 0 : 1;
            bool got = o >= h1;
            for (long long it = 0; it < ab.limit; ++it) {
              if (!got) got = pf_ld_relaxed(flag_of(h, which)) != 0u;
              if (__all_sync(0xffffffffu, got)) break;         // (together: divergent lanes would fence and copy one after the other)
              if ((it & 15) == 15 && __any_sync(0xffffffffu, ab.set())) break;
            }
            if (!__all_sync(0xffffffffu, got)) {
              if (!got && !ab.set()) ab.raise();
              break;
            }
            __threadfence();                                   // acquires what the flags announce ...
            asm volatile("fence.proxy.async;" ::: "memory");   // ... written by generic stores, read by the copy engine
            if (o < h1 && share_bytes > 0)
              bulk_copy_g2s(base + (uint32_t)(o - h0) * share_bytes, slot_of(h, which) + (long long)b0 * 16 * kTileN, share_bytes, bar_merge);
          }
          __syncwarp();
        }
        const bool landed = ab.wait(bar_merge, phase);
        phase ^= 1u;
        if (warp == kFirstEpi && landed && !ab.set())
          for (int o = h0 + lane; o < h1; o += 32) {           // fetched: one reader less
            const int h = first + o + (o >= mine ? 1 : 0);
            atomicSub(flag_of(h, h == last ? 0 : 1), 1u);
          }
        if (!pf_epi_vote(landed && !ab.set())) {
          alive = false;
          break;
        }
        const bool final_round = h1 == closers;
        for (int bk = b0 + hf; bk < b1; bk += 2) {
          uint32_t v[16];
          tmem_ld16(lane_addr + bk * 16, v);
          tc_wait_ld();
          for (int o = 0; o < h1 - h0; ++o) {
            const uint32_t sp = base + (uint32_t)o * share_bytes + (uint32_t)(((bk - b0) * 16 * kTileN + n) * 4);
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = __float_as_uint(__fadd_rn(__uint_as_float(v[e]), __uint_as_float(lds32(sp + e * kTileN * 4))));
          }
          if (final_round) {
            uint32_t h[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) h[j] = pf_pack(v[2 * j], v[2 * j + 1]);
            pf_store_block(h, y, n0, d_out, tok0 + bk * 16, p.M, ldy, lane);
          } else {
            tmem_st16(lane_addr + bk * 16, v);
          }
        }
        if (!final_round) {
          tc_wait_st();
          pf_epi_vote(true);                                   // everybody has read the rows: the next ones may land
        }
      }
      if (!alive) break;
      release();
    }
    if (S > 1) {
      // The pairs of a cluster hold the same tile: each finishes the token blocks of its share.  Everybody sends the rows of
      // the others' shares into their shared memory (over the rings, hence the first barrier), then adds what came to its
      // own accumulator, in ascending order of the pairs.  All threads take the barriers whatever happened before.
      bool have = ab.wait(bar_d_full, 0);
      have = __all_sync(0xffffffffu, have && !ab.set());
      tc_fence_after();
      pf_next_piece(u, u_end, G, wk, g0, g1);
      int col_pair;
      const int prob = pf_problem(p, wk, col_pair);
      const int tok0 = (wk % p.n_tok_blocks) * NT;
      const int n_blk = (min(NT, p.M - tok0) + 15) >> 4;       // blocks of sixteen tokens
      const int max_blk = (n_blk + S - 1) / S;                 // blocks of the largest share
      lane_addr = tmem + ((uint32_t)(quad * 32) << 16);
      cluster_arrive();
      cluster_wait();
      if (have) {
        for (int bk = hf; bk < n_blk; bk += 2) {
          const int o = ((bk + 1) * S - 1) / n_blk;            // the pair that finishes block bk
          if (o == split) continue;
          const int from = split < o ? split : split - 1;
          const uint32_t dst = map_to_rank(base + (uint32_t)(((from * max_blk + bk - n_blk * o / S) * 16 * kTileN + n) * 4), 2u * (uint32_t)o + rank);
          uint32_t v[16];
          tmem_ld16(lane_addr + bk * 16, v);
          tc_wait_ld();
#pragma unroll
          for (int e = 0; e < 16; ++e) st_cluster_u32(dst + e * kTileN * 4, v[e]);
        }
      }
      cluster_arrive();                                        // releases my rows, acquires everybody's
      cluster_wait();
      if (have && !ab.set()) {
        grid_dep_wait();                                       // y may still be in use by the previous kernel
        const int tile = 2 * col_pair + (int)rank;
        const int d_out = tile < p.n_tiles[prob] ? p.d_out[prob] : 0;
        const int b0 = n_blk * split / S, b1 = n_blk * (split + 1) / S;
        for (int bk = b0 + hf; bk < b1; bk += 2) {
          uint32_t v[16];
          tmem_ld16(lane_addr + bk * 16, v);
          tc_wait_ld();
          for (int from = 0; from < S - 1; ++from) {
            const uint32_t sp = base + (uint32_t)(((from * max_blk + bk - b0) * 16 * kTileN + n) * 4);
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = __float_as_uint(__fadd_rn(__uint_as_float(v[e]), __uint_as_float(lds32(sp + e * kTileN * 4))));
          }
          uint32_t h[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) h[j] = pf_pack(v[2 * j], v[2 * j + 1]);
          pf_store_block(h, p.y[prob], tile * kTileN + quad * 32, d_out, tok0 + bk * 16, p.M, p.ldy[prob], lane);
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_arrive();     // the leader's MMAs write the peer's tensor memory, the peer arrives on the leader's barriers
  cluster_wait();
  if (warp == 2) {
    __syncwarp();
    tmem_dealloc_pair<kPfTmemCols>(tmem);
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn prefill_encode_fn() {
  static const EncodeTiledFn fn = [] {                       // thread-safe: initialised once
    void *sym = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      return reinterpret_cast<EncodeTiledFn>(sym);
    (void)cudaGetLastError();
    return static_cast<EncodeTiledFn>(nullptr);
  }();
  return fn;
}

typedef void (*PrefillKernel)(PfParams);

int prefill_set_attrs(PrefillKernel kern) {
  if (cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess ||
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kPfMaxSmemBytes) != cudaSuccess) {
    (void)cudaGetLastError();
    return ROSAQ_ERR_CUDA;
  }
  return ROSAQ_OK;
}

std::mutex g_pf_mu;
bool g_pf_attr_done[64] = {};                                // per device, all kernels at once

int prefill_prepare_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return ROSAQ_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_pf_mu);
  if (!g_pf_attr_done[dev]) {
    if (prefill_set_attrs(linear_prefill_kernel<4>) != ROSAQ_OK || prefill_set_attrs(linear_prefill_kernel<3>) != ROSAQ_OK ||
        prefill_set_attrs(linear_prefill_kernel<kDenseBits>) != ROSAQ_OK)
      return ROSAQ_ERR_CUDA;
    g_pf_attr_done[dev] = true;
  }
  return ROSAQ_OK;
}

size_t prefill_smem(bool dense, int NT, int NW) {
  const size_t rings = dense ? (size_t)NW * (kPdABytes + (NT / 2) * 128) : (size_t)kPfStages * (NT / 2) * 256 + (size_t)NW * kWSlotBytes;
  return 1024 + rings + 8 * (2 * NW + 2 * kPfStages + 6) + 16;
}

void prefill_config(cudaLaunchConfig_t *cfg, cudaLaunchAttribute *attr, int n_pairs, int S, int threads, size_t smem, cudaStream_t s) {
  cfg->gridDim = dim3(2 * n_pairs);
  cfg->blockDim = dim3(threads);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = S > 0 ? 2 * S : 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // the prologue runs under the previous kernel's tail
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  attr[2].id = cudaLaunchAttributeCooperative;               // equal shares: pairs wait for one another, all must be resident
  attr[2].val.cooperative = 1;
  cfg->attrs = attr;
  cfg->numAttrs = S > 0 ? 2 : 3;
}

// Clusters of S pairs that the device keeps resident at once (a cluster lives inside one GPC, so larger ones leave SMs over);
// 0 when the query fails
int prefill_clusters(rosaq_ctx *ctx, int S) {
  if (ctx->pf_clusters[S - 1] > 0) return ctx->pf_clusters[S - 1];
  if (prefill_prepare_device() != ROSAQ_OK) return 0;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[3];
  prefill_config(&cfg, attr, S * (ctx->sm_count / (2 * S)), S, kPfThreads, kPfMaxSmemBytes, nullptr);
  cfg.numAttrs = 1;                                          // (the cluster shape only)
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, linear_prefill_kernel<4>, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  clusters = std::min(clusters, ctx->sm_count / (2 * S));
  ctx->pf_clusters[S - 1] = clusters;
  return clusters;
}

}  // namespace

// Operands this kernel takes: any whose adjacent column tiles multiply the same channels; outputs in column order.
bool prefill_supported(const TiledOperand &t, const int32_t *col_map) {
  return t.block_groups % 2 == 0 && groups_per_tile(t) > 0 && (t.block_groups == 0 || t.g_quant == 0) && col_map == nullptr &&
         (t.bits == 3 || t.bits == 4);
}

// How a launch is cut, and about how long it takes (us) in a chain of launches.  A fit to the launches that linear_tc_estimate is
// fitted to, each cut measured by itself (clusters 4 % rms, equal shares 6 %): a launch and `token` us per token of a tile;
// `exchange` between the pairs of a cluster; a group of a pair 0.0021 us per token, and more the more pairs run (they share the L2
// and the power limit); `full` when more than half of the SMs are taken, so that the next launch has to wait for
// this one to end.  Equal shares: the exchange through L2, more of it the more pairs hold a tile (13824 -> 128 at 160
// tokens, 74 holders: 33 us; four pairs in a cluster 17; the per-call kernel 11.6).
PrefillCut prefill_choose(rosaq_ctx *ctx, int M, int n, const TiledOperand *const *ts) {
  struct Cluster { double launch, token, exchange[kPfMaxSplits + 1], group, group_token, full, crowd; };
  static constexpr Cluster kClusterQuant{3.493, 0.0166, {0, 0, 0.813, 1.16, 1.994}, 0.0236, 0.0022, 1.972, 0.2853};
  static constexpr Cluster kClusterDense{2.515, 0.0161, {0, 0, 1.683, 2.241, 2.838}, 0.0478, 0.0021, 0.615, 0.2883};
  struct Shares { double launch, token, group, group_token, holder, tile; };
  static constexpr Shares kSharesQuant{9.427, 0.0192, -0.0607, 0.0034, 0.2175, 2.462};
  static constexpr Shares kSharesDense{4.217, 0.028, 0.2805, 0.0021, 0.2613, 2.633};
  const bool dense = ts[0]->g_quant == 0;
  const int G = groups_per_tile(*ts[0]);
  long long col_pairs = 0;
  for (int i = 0; i < n; ++i) col_pairs += (ts[i]->n_tiles + 1) / 2;
  PrefillCut best;
  const int blocks = (M + kPfMaxTokens - 1) / kPfMaxTokens;
  best.NT = ((M + blocks - 1) / blocks + 31) / 32 * 32;
  best.n_tok_blocks = (M + best.NT - 1) / best.NT;
  best.NT_last = (M - (best.n_tok_blocks - 1) * best.NT + 31) / 32 * 32;
  const double NT = best.NT, tiles = (double)col_pairs * best.n_tok_blocks, half = ctx->sm_count / 4;
  const double whole = (double)col_pairs * (best.n_tok_blocks - 1 + best.NT_last / NT);   // tiles of NT tokens that are as much work
  {
    const Shares &f = dense ? kSharesDense : kSharesQuant;
    const double units = whole * G, pairs = std::max(1.0, std::min((double)prefill_clusters(ctx, 1), units));
    best.S = 0;
    best.us = f.launch + f.token * NT + units / pairs * (f.group + f.group_token * NT) + f.holder * std::max(0.0, pairs / tiles - 2) + f.tile * tiles / pairs;
  }
  const Cluster &f = dense ? kClusterDense : kClusterQuant;
  for (int S = 1; S <= kPfMaxSplits && S <= G; ++S) {
    const int res = prefill_clusters(ctx, S);
    if (res < 1 || tiles > res) continue;                    // (a second round of clusters costs more than equal shares)
    const double over = std::max(0.0, tiles * S / half - 1);
    const double us = f.launch + f.token * NT + f.exchange[S] + (over > 0 ? f.full : 0.0) + (double)((G + S - 1) / S) * (f.group + f.group_token * NT) * (1 + f.crowd * over);
    if (us < best.us) best.us = us, best.S = S;
  }
  return best;
}

// n weights of identical geometry applied to the same activations in one launch
int launch_linear_prefill(rosaq_ctx *ctx, const __half *x, int M, long long ldx, int n, const TiledOperand *const *ts,
                          __half *const *ys, const long long *ldys, const PrefillCut &cut, cudaStream_t s) {
  EncodeTiledFn encode = prefill_encode_fn();
  if (!encode) return ROSAQ_ERR_CUDA;
  if (n < 1 || n > kPfMaxProblems) return ROSAQ_ERR_INVALID_ARG;
  const TiledOperand &t = *ts[0];
  if (!prefill_supported(t, nullptr) || M < 1 || (n > 1 && t.block_groups > 0)) return ROSAQ_ERR_UNSUPPORTED_SHAPE;
  const int max_pairs = prefill_clusters(ctx, 1);
  if (max_pairs < 1) return ROSAQ_ERR_CUDA;
  PfParams p{};
  p.n_prob = n;
  int col_pairs = 0;
  for (int i = 0; i < n; ++i) {
    const TiledOperand &ti = *ts[i];
    if (ti.d_in != t.d_in || ti.g_fp16 != t.g_fp16 || ti.g_quant != t.g_quant || ti.block_groups != t.block_groups ||
        (t.g_quant > 0 && ti.bits != t.bits))
      return ROSAQ_ERR_INVALID_ARG;
    p.pair_start[i] = col_pairs;
    p.blob[i] = ti.blob, p.y[i] = ys[i], p.ldy[i] = ldys[i], p.d_out[i] = ti.d_out, p.n_tiles[i] = ti.n_tiles;
    col_pairs += (ti.n_tiles + 1) / 2;
  }
  p.pair_start[n] = col_pairs;
  p.tile_stride = t.tile_stride;
  p.g_fp16 = t.g_fp16;
  p.groups = groups_per_tile(t);
  p.block_groups = t.block_groups;
  p.M = M;
  p.NT = cut.NT;
  p.NT_last = cut.NT_last;
  p.n_tok_blocks = cut.n_tok_blocks;
  p.S = cut.S;
  const bool dense = t.g_quant == 0;
  const size_t budget = kPfMaxSmemBytes - 2048;
  if (dense) {
    p.NW = (int)std::min<size_t>(kPdMaxStages, budget / (kPdABytes + (p.NT / 2) * 128));
  } else {
    p.NW = std::min(kPfMaxNW, (int)((budget - kPfStages * (p.NT / 2) * 256) / kWSlotBytes) / kPfTeams * kPfTeams);
  }
  // {64 channels, tokens, 64-channel block} view of the row-major activations, box = a group (two blocks; dense: one) of
  // NT / 2 tokens; rows past M are zero-filled by the copy
  const cuuint64_t dims[3] = {64, (cuuint64_t)M, (cuuint64_t)(t.d_in / 64)};
  const cuuint64_t strides[2] = {(cuuint64_t)ldx * sizeof(__half), 128};
  const cuuint32_t box[3] = {64, (cuuint32_t)(p.NT / 2), dense ? 1u : 2u};
  const cuuint32_t estr[3] = {1, 1, 1};
  if (encode(&p.xmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half *>(x), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return ROSAQ_ERR_CUDA;
  const cuuint32_t box_last[3] = {64, (cuuint32_t)(p.NT_last / 2), box[2]};
  p.xmap_last = p.xmap;
  if (p.NT_last != p.NT &&
      encode(&p.xmap_last, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half *>(x), dims, strides, box_last, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return ROSAQ_ERR_CUDA;
  for (int i = 0; i < n && dense; ++i) {
    const cuuint64_t wdims[2] = {64, (cuuint64_t)(ts[i]->bytes / 128)}, wstrides[1] = {128};
    const cuuint32_t wbox[2] = {64, kPdABytes / 128}, west[2] = {1, 1};
    if (encode(&p.wmap[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, ts[i]->blob, wdims, wstrides, wbox, west, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return ROSAQ_ERR_CUDA;
  }
  const long long tiles = (long long)col_pairs * p.n_tok_blocks, units = tiles * p.groups;
  if (units < 1 || units > (1ll << 30)) return ROSAQ_ERR_UNSUPPORTED_SHAPE;
  p.units = (int)units;
  const int n_pairs = p.S > 0 ? (int)tiles * p.S : (int)std::min<long long>(units, std::min(max_pairs, kPfMaxPairs));
  // The cut into equal shares: pair i begins at the unit nearest to i n-ths of the cost.  A unit of the last token block
  // costs less when that block holds fewer tokens: 1900 are seven blocks of 256 and one of 108, which takes 128.  A unit costs what its tokens
  // do and about 100 tokens more.  us, all blocks of NT / this, in a loop: 4096 -> 3 x 4096 at 600 tokens 68.1 / 61.1, at 1570 145.8 / 139.9, at 1900 169.4 / 162.4;
  // 4096 -> 2 x 11008 at 900 153.5 / 145.1, at 1900 290.4 / 280.4; dense rotation of 5120 at 1900 104.0 / 99.0.  (No range may be empty, so each has
  // to be worth a unit.)
  // A range does not end with the first group or two of a tile (`snap`, for as little as a tenth of a range): the
  // epilogue still stores the tile before it then, and the exchange of this one begins only behind that.  us, with such ends / without: 1280 -> 10672 at 1782 tokens 63 / 53, 1408 -> 9000 at 1300 48 / 40, 1408 -> 3 x 6024 at
  // 569 44 / 37, INT3 4480 -> 3 x 4600 at 439 55 / 48; 330 launches of 200 to 2048 tokens 0.8 % on average.
  if (p.S == 0) {
    const int fixed = dense ? 4 : 3;                         // of a group, in 32 tokens
    long long cost = p.NT / 32 + fixed, cost_last = p.NT_last / 32 + fixed;
    const long long G = p.groups, nb = p.n_tok_blocks;
    if (col_pairs * G * ((nb - 1) * cost + cost_last) < n_pairs * cost) cost = cost_last = 1;
    const long long head = (nb - 1) * G * cost, per_col = head + G * cost_last;
    const long long snap = std::min(3ll, std::max(1ll, units / (10 * n_pairs)));
    for (int i = 0; i <= n_pairs; ++i) {
      const long long c = i * (col_pairs * per_col) / n_pairs, col = c / per_col, rest = c - col * per_col;
      long long at = col * G * nb + (rest <= head ? (2 * rest + cost) / (2 * cost) : (nb - 1) * G + (2 * (rest - head) + cost_last) / (2 * cost_last));
      const long long tail = at % G;
      if (i > 0 && i < n_pairs && tail <= snap && 2 * snap < G && at - tail > p.bounds[i - 1]) at -= tail;
      p.bounds[i] = (int)at;
    }
  }
  // two slots of 2 x NT x 128 floats per pair, (launches of one context do not overlap on the GPU)
  if (p.S == 0 && ctx->pf_partial_bytes < (size_t)n_pairs * 4 * p.NT * kTileN * sizeof(float)) return ROSAQ_ERR_ALLOC;
  p.partials = ctx->pf_partials;
  p.flags = ctx->pf_flags;
  p.status = ctx->d_status;
  p.wait_limit = ctx->wait_limit;
  const PrefillKernel kern = dense ? linear_prefill_kernel<kDenseBits> : (t.bits == 3 ? linear_prefill_kernel<3> : linear_prefill_kernel<4>);
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[3];
  prefill_config(&cfg, attr, n_pairs, p.S, dense ? kPdThreads : kPfThreads, prefill_smem(dense, p.NT, p.NW), s);
  if (cudaLaunchKernelEx(&cfg, kern, p) != cudaSuccess) {
    (void)cudaGetLastError();
    return ROSAQ_ERR_CUDA;
  }
  return ROSAQ_OK;
}

}  // namespace rosaq
