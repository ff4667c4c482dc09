// W4A16 projection for many tokens on the 5th-generation tensor cores
// (tcgen05): Y[n][r] = sum_k W[r][k] x[n][k] for S tokens, W in the shard's
// unit stream (kernels.h).  Used where the token count makes the projection
// a dense contraction -- a prompt's prefill (Section 3.4: the stateful cache
// is filled by running the prompt through the stage) -- where the per-token
// GEMV of the decode step would stream every weight once per 16 tokens.
//
// One CTA computes a tile of 128 weight rows (two row-blocks) by N tokens over
// all of K or a part of it, walking K one 128-input unit per step, with warp
// roles joined by mbarriers:
//   - warp 0 (producer): bulk-copies the step's two units (codes, scales,
//     zero points) and loads the token tile with two 2-D tensor copies (64
//     inputs x N tokens each, 128-byte swizzle), several stages ahead;
//   - warps 12..19 (dequantise): turn the codes into exact fp16 (q - z) and
//     store them to tensor memory, the A operand; two sets of four warps take
//     the steps in turn, 2 stages;
//   - warps 1, 2 (MMA): a thread each, steps in turn, issues tcgen05.mma
//     (kind::f16, M = 128, N tokens, K = 16 per instruction, A in tensor memory,
//     B in shared memory) into a ring of accumulators, one per quantisation
//     group and step, and commits to the step's mbarrier;
//   - warps 4..11 (epilogue): read the accumulators (tcgen05.ld; warp w owns
//     lanes 32 (w % 4) .. + 31 = tile rows, half the token columns each),
//     multiply by the row's fp32 group scale and add into registers; at the
//     end they write their rows' outputs.
// A in tensor memory: with A in shared memory too, a step of 128 x 128 x 128 moved
// 64 KB of operands through it beside 40 KB of arriving copies and 40 KB of
// dequantisation. The code words' fragment order (kernels.h) is the lane order
// of tcgen05.st's 16x256b shape, so a warp reads its words with conflict-free
// 16-byte loads and stores each word's four fp16 pairs as they are. The price is
// the order of the inputs: a lane's word holds inputs 8 t + 4 j .. + 3 of a
// 32-input block (t = lane % 4), so activations are kept with each block's
// 4-input chunks in the order 0 2 4 6 1 3 5 7 (act_pos).
// What bounds it is, in the K loop, the roles' own chains of barrier polls and
// short dependent work, ~1150 cycles a step against 512 of tensor time: leaving
// out, one at a time, the MMAs, the dequantisation's arithmetic, the epilogue's
// loads or the copies changes a step by 2-6 %. Before and behind the loop it is
// filling the rings and writing the tile out, which nothing overlaps with one CTA
// per SM: gate|up of 512 tokens at 8B width is 6 rounds of 32 steps, 72 % of its
// 148 us; o takes 25 us, down 71, q|k|v 42 (with three commits a step by one
// thread, one dequantise set and suspending waits, which with A in shared memory
// ran at the same ~1 us a step, and straight-line code for the outputs 225, 73 (o
// and down) and 61).
// The token tile sits in the canonical K-major layout with the 128-byte
// swizzle, as the tensor copy writes it. The
// arithmetic is the decode projection's: exact (q - z), fp32 sums per group,
// the fp16 scale applied in fp32.  Every wait is bounded; a wait that runs out
// sets the status word.  The TMEM columns are freed before the CTA exits.
#include <cuda.h>

#include <mutex>

#include "gemv_core.cuh"
#include "launch.cuh"

namespace shard {
namespace {

constexpr int kTcRows = 128;        // weight rows per CTA tile (two row-blocks)
constexpr int kTcWarps = 20;
constexpr int kTcThreads = kTcWarps * 32;
constexpr int kMmaWarp0 = 1, kMmaWarps = 2, kEpiWarp0 = 4, kEpiWarps = 8, kDqWarp0 = 12, kDqSets = 2;
constexpr int kUStages = 6, kBStages = 4, kAStages = 2;

// Accumulators in tensor memory for tiles of N tokens with g groups per step:
// what the columns hold, and no more than the completion barriers can tell apart.
constexpr int tc_accumulators(int N, int g) {
  const int fit = N == 128 ? 3 : N == 96 ? 4 : N == 64 ? 6 : 8;
  return fit < kBStages * g ? fit : kBStages * g;
}

template <int N, int GPU>
struct TcSmem {
  static constexpr size_t kUnit = Geom<GPU>::kUnitBytes;
  static constexpr size_t kUnits = 2 * kUnit;                          // the tile's two units
  static constexpr size_t kB = (size_t)N * 256;                        // 128 inputs x N tokens
  static constexpr size_t kBOff = 0;                                   // [kBStages][kB]
  static constexpr size_t kUOff = kBOff + kBStages * kB;               // [kUStages][kUnits]
  static constexpr int kHLd = 72;                                      // halves per token of the staged SwiGLU rows
  static constexpr size_t kTotal = kUOff + kUStages * kUnits + 1024;   // + alignment slack
  static_assert((size_t)N * (kTcRows * 4 + kHLd * 2) <= kBStages * kB, "staged sums");
  // tensor memory: two A stages of 64 columns behind the accumulator ring
  static constexpr int kDStages = tc_accumulators(N, GPU);
  static constexpr uint32_t kACol = kDStages * N;
  static constexpr uint32_t kCols = 512;
  static_assert(kACol + kAStages * 64 <= kCols, "tensor memory");
  // A parity wait tells a phase from its neighbours only: neither side of a
  // barrier may get two phases away from a waiter.
  // d_empty: two threads issue steps in turn and may be a step apart. A thread
  // that issues accumulator q has issued q - G - 1 or later before, so q - G -
  // 1 - kDStages has been read; q - 2 kDStages must be no later.
  static_assert(kDStages >= GPU + 1, "accumulator ring");
  // done: the epilogue warp that is furthest behind still waits for group q, and
  // the MMAs have gone on as far as the accumulators let them, up to group q +
  // kDStages - 1. The barrier's next phase is group q + kBStages G and must not be
  // among them. (Its other waiters cannot be overtaken: the phase takes a token
  // tile that the producer sends after its wait for the last one, and four
  // arrivals of the dequantise set that waits.)
  static_assert(kDStages <= kBStages * GPU, "completion barriers");
};

// Shared-memory matrix descriptor, K-major with the 128-byte swizzle: 8-row
// groups 1024 bytes apart (the byte offset between K-adjacent core matrices is
// implied by the swizzle); the start address may move by 32 bytes per K = 16
// inside a 64-input half.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;            // leading byte offset: unused with this swizzle
  d |= (uint64_t)(1024 >> 4) << 32;  // stride byte offset
  d |= 1ull << 46;                   // descriptor version for this architecture
  d |= 2ull << 61;                   // layout: 128-byte swizzle
  return d;
}

// Instruction descriptor, kind::f16: fp32 accumulator, fp16 A and B, both
// K-major, M = 128, N tokens.
template <int N>
__device__ __forceinline__ uint32_t instr_desc() {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kTcRows >> 4) << 24);
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// One lane of the converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

// A in tensor memory, B in shared memory.
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, bool acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"((uint32_t)acc)
      : "memory");
}

// 16 lanes x 32 columns: register 4 i + 2 h + e of a lane goes to row
// lane / 4 + 8 h, column 8 i + 2 (lane % 4) + e.
__device__ __forceinline__ void tc_st16x256x4(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

// Arrive on `bar` once every tcgen05 operation this thread issued so far is done.
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}

// 16 consecutive fp32 columns of this thread's tensor-memory lane; the registers
// are not to be read before tc_ld_wait.
__device__ __forceinline__ void tc_ld(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_ld_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) asm volatile("" : "+r"(r[i]));  // not read before the wait
}

// 2-D tensor copy of one box into shared memory, completion on `bar`.
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_addr(bar))
      : "memory");
}

// Kernel arguments: the projection and the tensor map of its activations
// (fp16 [S][act_ld] in act_pos order).
struct TcParams {
  GemmArgs a;
  CUtensorMap act_map;  // {K inputs, S tokens}, box 64 x N, 128-byte swizzle
};

template <int N, int GPU>
__global__ void __launch_bounds__(kTcThreads, 1) gemm_tc_kernel(const __grid_constant__ TcParams P) {
  const GemmArgs& a = P.a;
  using L = TcSmem<N, GPU>;
  constexpr int UB = Geom<GPU>::kUnitBytes;
  constexpr int G = GPU;                        // quantisation groups per unit
  constexpr int kMmaPerGroup = 8 / GPU;         // K = 16 per instruction
  constexpr int kPer = N / (kEpiWarps / 4);     // token columns per epilogue thread
  constexpr int kLd = 16;                       // of them, columns per load
  constexpr int kDStages = L::kDStages;
  constexpr uint32_t kHalfB = N * 128;          // bytes per 64-input half
  static_assert(kPer % kLd == 0, "columns per epilogue thread");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // u_*: a step's units; full: a step's A and B are in place; done: the MMAs up
  // to a step's group are; d_empty: an accumulator has been read
  __shared__ uint64_t u_full[kUStages], u_empty[kUStages], full[kBStages], done[kBStages * G], d_empty[kDStages];
  __shared__ uint32_t s_tmem;
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;  // warp: known uniform
  const int rb0 = 2 * blockIdx.x;   // the tile's first row-block
  const int n0 = blockIdx.y * N;    // the tile's first token
  const int k_begin = part_start(a.upr, blockIdx.z, gridDim.z);
  const int steps = part_start(a.upr, blockIdx.z + 1, gridDim.z) - k_begin;
  auto B_of = [&](int s) { return smem + L::kBOff + (size_t)s * L::kB; };
  auto U_of = [&](int s) { return smem + L::kUOff + (size_t)s * L::kUnits; };
  if (tid == 0) {
    for (int i = 0; i < kUStages; ++i) {
      mbar_init(&u_full[i], 1);
      mbar_init(&u_empty[i], 4 + kEpiWarps);  // the step's dequantise set; the epilogue takes the scales from the unit
    }
    for (int i = 0; i < kBStages; ++i) mbar_init(&full[i], 4 + 1);
    for (int i = 0; i < kBStages * G; ++i) mbar_init(&done[i], 1);
    for (int i = 0; i < kDStages; ++i) mbar_init(&d_empty[i], kEpiWarps);
    mbar_fence_init();
  }
  if (warp == kMmaWarp0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)),
                 "r"(L::kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  // false once a wait gave up: the role skips the rest of its waits. The producer
  // then copies nothing more and the MMA thread neither multiplies nor signals, so
  // that nothing they started is under way when the CTA ends: every copy is waited
  // for by a role whose waits hold, or was made a whole wait's limit ago.
  bool ok = true;
  // spinning: the suspending try_wait measured 8 % slower over the whole kernel
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (!ok) return;
    uint32_t it = 0;
    while (!mbar_test_wait(bar, parity))
      if (++it > (1u << 26)) {
        ok = false;
        break;
      }
  };
  // the MMAs of step k, up to group gq
  auto wait_done = [&](int k, int gq) { wait(&done[(k % kBStages) * G + gq], (k / kBStages) & 1); };

  auto load_units = [&](int k) {
    const int su = k % kUStages;
    mbar_arrive_expect_tx(&u_full[su], 2 * UB);
    for (int u = 0; u < 2; ++u) {
      const int rb = rb0 + u < a.n_rb ? rb0 + u : rb0;  // a missing second block repeats the first (unused)
      bulk_g2s(U_of(su) + (size_t)u * UB, a.units + ((size_t)rb * a.upr + k_begin + k) * UB, UB, &u_full[su]);
    }
  };
  // the weights are constant: the first units come in while the kernel before ends
  if (tid == 0)
    for (int k = 0; k < kUStages && k < steps; ++k) load_units(k);
  pdl_wait();
  pdl_launch_dependents();

  if (warp == 0) {
    // ---- producer: units and token tiles, kUStages / kBStages steps ahead ----
    if (lane == 0) {
      for (int k = 0; k < steps; ++k) {
        const int su = k % kUStages, sb = k % kBStages;
        if (k >= kUStages) {
          wait(&u_empty[su], ((k / kUStages) & 1) ^ 1);
          if (!ok) break;
          load_units(k);
        }
        if (k >= kBStages) wait_done(k - kBStages, G - 1);
        if (!ok) break;
        mbar_arrive_expect_tx(&full[sb], N * 256);
        for (int h = 0; h < 2; ++h)  // tokens past S read as zero
          tma_load_2d(B_of(sb) + (size_t)h * kHalfB, &P.act_map, (k_begin + k) * kUnitK + h * 64, n0, &full[sb]);
      }
    }
  } else if (warp >= kMmaWarp0 && warp < kMmaWarp0 + kMmaWarps) {
    // ---- MMA issue: one thread per warp, steps in turn ----
    // A step's issue is a chain of two barrier polls, 8 MMAs and a commit per
    // group, ~1150 cycles for a thread alone (more with a commit each for A, B
    // and the accumulator): two threads overlap it. Steps need no order among
    // themselves: each group starts a fresh accumulator.
    {
      const bool leader = elect_one();
      for (int k = warp - kMmaWarp0; k < steps; k += kMmaWarps) {
        const int sa = k % kAStages, sb = k % kBStages;
        const uint32_t aBase = tmem + L::kACol + (uint32_t)sa * 64u;
        const uint64_t bDesc = smem_desc_sw128(smem_addr(B_of(sb)));  // advanced by 16-byte units
        wait(&full[sb], (k / kBStages) & 1);
#pragma unroll
        for (int gq = 0; gq < G; ++gq) {
          const int q = k * G + gq, sd = q % kDStages;
          if (q >= kDStages) wait(&d_empty[sd], ((q / kDStages) & 1) ^ 1);
          tc_fence_after();
          if (ok && leader) {
#pragma unroll
            for (int i = 0; i < kMmaPerGroup; ++i) {
              const int kk = gq * kMmaPerGroup + i;          // K = 16: 8 columns of A, 32 bytes of a 64-input half of B
              tc_mma(tmem + (uint32_t)(sd * N), aBase + 8u * kk, bDesc + (((kk >> 2) * kHalfB + (kk & 3) * 32u) >> 4),
                     instr_desc<N>(), i > 0);
            }
            tc_commit(&done[sb * G + gq]);
          }
          __syncwarp();
        }
      }
    }
  } else if (warp >= kDqWarp0) {
    // ---- dequantise: exact fp16 (q - z) into the A stage ----
    // the warp's tensor-memory lanes are 32 (warp % 4) .. + 31: two 16-row
    // tiles of one unit
    const int quad = warp & 3, u = quad >> 1, gid = lane >> 2;
    for (int k = (warp - kDqWarp0) >> 2; k < steps; k += kDqSets) {
      const int su = k % kUStages, sa = k % kAStages;
      const uint8_t* U = U_of(su) + (size_t)u * UB;
      wait(&u_full[su], (k / kUStages) & 1);
#pragma unroll
      for (int kh = 0; kh < 2; ++kh) {  // 64 inputs at a time
        uint32_t r[2][16];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int rt = 2 * (quad & 1) + i;
          const uint4 w4 = *reinterpret_cast<const uint4*>(U + (kh * 4 + rt) * 512 + lane * 16);
          const uint32_t wv[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // word j: rows gid and gid + 8 at inputs 64 kh + 32 (j / 2) + 8 (lane % 4) + 4 (j % 2) .. + 3
            const uint32_t zz = *reinterpret_cast<const uint16_t*>(  // z of row gid, 16 z of row gid + 8
                U + kCodeBytes + ((64 * kh + 32 * (j >> 1)) / (kUnitK / G)) * kMetaBytesPerGroup + 128 + gid * 8 + rt * 2);
            const uint32_t zs = (0x6400u | (zz & 0xFFu)) * 0x00010001u;  // fp16x2 (1024 + z)
            const uint32_t zf = (0xD400u | (zz >> 8)) * 0x00010001u;     // fp16x2 -(64 + z)
            const uint32_t w = wv[j], w2 = w >> 8;
            r[i][4 * j] = hsub2_u32(lop3_and_or(w, 0x000F000Fu, 0x64006400u), zs);
            r[i][4 * j + 1] = hsub2_u32(lop3_and_or(w2, 0x000F000Fu, 0x64006400u), zs);
            r[i][4 * j + 2] = hfma2_u32(lop3_and_or(w, 0x00F000F0u, 0x64006400u), 0x2C002C00u, zf);
            r[i][4 * j + 3] = hfma2_u32(lop3_and_or(w2, 0x00F000F0u, 0x64006400u), 0x2C002C00u, zf);
          }
        }
        if (kh == 0 && k >= kAStages) wait_done(k - kAStages, G - 1);
        __syncwarp();
        if (kh == 0) tc_fence_after();
        const uint32_t at = tmem + ((uint32_t)(32 * quad) << 16) + L::kACol + (uint32_t)sa * 64u + 32u * kh;
        tc_st16x256x4(at, r[0]);
        tc_st16x256x4(at + (16u << 16), r[1]);
      }
      if (lane == 0) mbar_arrive(&u_empty[su]);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[k % kBStages]);
    }
  } else if (warp >= kEpiWarp0) {
    // ---- epilogue: scale and add each step's group sums ----
    const int quad = warp & 3;
    const int row = 32 * quad + lane;  // tile row = TMEM lane
    const int c0 = ((warp - kEpiWarp0) >> 2) * kPer;
    const int R = row & 63;
    const uint32_t lane_base = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)c0;
    const int sidx = (R & 7) * 8 + ((R >> 4) & 3) * 2 + ((R >> 3) & 1);
    float tot[kPer];
#pragma unroll
    for (int c = 0; c < kPer; ++c) tot[c] = 0.f;
    float sc[G];  // the step's scales; the next step's load behind its sums
    auto load = [&](int k) {
      const int su = k % kUStages;
      wait(&u_full[su], (k / kUStages) & 1);
#pragma unroll
      for (int gq = 0; gq < G; ++gq)
        sc[gq] = h2f(reinterpret_cast<const uint16_t*>(U_of(su) + (size_t)(row >> 6) * UB + kCodeBytes +
                                                      gq * kMetaBytesPerGroup)[sidx]);
      __syncwarp();
      if (lane == 0) mbar_arrive(&u_empty[su]);
    };
    load(0);
    int q = 0;
    for (int k = 0; k < steps; ++k) {
#pragma unroll
      for (int gq = 0; gq < G; ++gq, ++q) {
        const int sd = q % kDStages;
        wait_done(k, gq);
        __syncwarp();
        tc_fence_after();
        const uint32_t at = lane_base + (uint32_t)(sd * N);
        uint32_t v[2][kLd];
        tc_ld(at, v[0]);
#pragma unroll
        for (int i = 0; i < kPer / kLd; ++i) {
          tc_ld_wait(v[i & 1]);
          if (i + 1 < kPer / kLd) tc_ld(at + (i + 1) * kLd, v[(i & 1) ^ 1]);
#pragma unroll
          for (int c = 0; c < kLd; ++c) tot[i * kLd + c] = fmaf(sc[gq], __uint_as_float(v[i & 1][c]), tot[i * kLd + c]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&d_empty[sd]);
      }
      if (k + 1 < steps) load(k + 1);
    }
    // The sums go through shared memory (every copy into it is done: the last
    // accumulator is) into short loops: straight-line code for every column is
    // fetched for one use, which cost more than the work (4 layers at 8B width,
    // 77 tokens 621 -> 538 us, 512 tokens 1453 -> 1387; gate|up of 77 tokens 68 -> 49).
    float* ys = reinterpret_cast<float*>(smem);  // [N][128 rows]
#pragma unroll
    for (int c = 0; c < kPer; ++c) ys[(c0 + c) * kTcRows + row] = tot[c];
    const int live = min(N, a.S - n0);  // the tile's tokens
    if (a.h) {
      // SwiGLU: gate row 16 t + r and up row 16 t + r + 8 of a block give h index
      // 32 rb + 8 t + r; staged to go out in whole 16-byte pieces
      uint16_t* hs = reinterpret_cast<uint16_t*>(ys + N * kTcRows);
      const int et = tid - kEpiWarp0 * 32;
      const int u = (et >> 5) & 1, t = (et >> 3) & 3, r = et & 7;  // kEpiWarps * 32 threads: a multiple of 64
      const int gate = 64 * u + 16 * t + r, pos = 32 * u + act_pos(8 * t + r);
      named_bar_sync(1, kEpiWarps * 32);
#pragma unroll 4
      for (int c = et >> 6; c < live; c += kEpiWarps / 2)
        hs[c * L::kHLd + pos] = f2h(silu(ys[c * kTcRows + gate]) * ys[c * kTcRows + gate + 8]);
      named_bar_sync(1, kEpiWarps * 32);
      // positions past F (of the last, ragged block) stay as they are: zero
      for (int e = et; e < live * 8; e += kEpiWarps * 32) {
        const int c = e >> 3, j = 8 * (e & 7);
        const int blk = rb0 + (j >> 5);
        if (blk >= a.n_rb) continue;
        const uint16_t* src = hs + c * L::kHLd + j;
        uint16_t* dst = a.h + (size_t)(n0 + c) * a.h_ld + 32 * blk + (j & 31);
        if (32 * blk + 32 <= a.F) {
          *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
        } else {
          for (int i = 0; i < 8; ++i)
            if (32 * blk + act_unpos((j & 31) + i) < a.F) dst[i] = src[i];
        }
      }
    } else if (rb0 + (row >> 6) < a.n_rb) {
      // natural row order, [part of K][token][row]; each thread its own row
      const int nat = natural_row(a.dims, (rb0 + (row >> 6)) * kRowsPerBlock + R);
      float* y = a.y + (size_t)blockIdx.z * a.y_part + (size_t)n0 * a.y_ld + nat;
      const int c1 = min(c0 + kPer, live);
      if (nat >= 0)
#pragma unroll 4
        for (int c = c0; c < c1; ++c) y[(size_t)c * a.y_ld] = ys[c * kTcRows + row];
    }
  }
  if (!ok) atomicOr(a.status, ST_WAIT_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kMmaWarp0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(L::kCols) : "memory");
}

// cuTensorMapEncodeTiled, from the driver through the runtime (no link
// against the driver library).
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

template <int N, int GPU>
cudaError_t launch_tc(const GemmArgs& a, cudaStream_t s) {
  using L = TcSmem<N, GPU>;
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  // the activations: fp16 [S][act_ld] (16-byte aligned rows); box = 64
  // inputs (128 bytes) x N tokens; tokens past S read as zero
  if ((reinterpret_cast<uintptr_t>(a.act) & 15) || a.act_ld % 8 || a.upr * kUnitK > a.act_ld || a.S < 1)
    return cudaErrorInvalidValue;
  TcParams p;
  p.a = a;
  const cuuint64_t dims[2] = {(cuuint64_t)a.upr * kUnitK, (cuuint64_t)a.S};
  const cuuint64_t strides[1] = {(cuuint64_t)a.act_ld * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)N};
  const cuuint32_t estr[2] = {1, 1};
  if (enc(&p.act_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<uint16_t*>(a.act), dims, strides, box, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  const dim3 grid((a.n_rb + 1) / 2, (a.S + N - 1) / N, a.parts);
  return launch_behind(gemm_tc_kernel<N, GPU>, grid, kTcThreads, L::kTotal, s, p);
}

template <int N, int GPU>
cudaError_t setup_tc() {
  return cudaFuncSetAttribute(gemm_tc_kernel<N, GPU>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)TcSmem<N, GPU>::kTotal);
}

}  // namespace

cudaError_t gemm_tc_setup() {
  cudaError_t e;
  if ((e = setup_tc<32, 1>()) != cudaSuccess) return e;
  if ((e = setup_tc<32, 2>()) != cudaSuccess) return e;
  if ((e = setup_tc<32, 4>()) != cudaSuccess) return e;
  if ((e = setup_tc<64, 1>()) != cudaSuccess) return e;
  if ((e = setup_tc<64, 2>()) != cudaSuccess) return e;
  if ((e = setup_tc<64, 4>()) != cudaSuccess) return e;
  if ((e = setup_tc<96, 1>()) != cudaSuccess) return e;
  if ((e = setup_tc<96, 2>()) != cudaSuccess) return e;
  if ((e = setup_tc<128, 1>()) != cudaSuccess) return e;
  if ((e = setup_tc<128, 2>()) != cudaSuccess) return e;
  return cudaSuccess;
}

// Token tile: 128 for long prompts, or 96 where that makes no more tiles (65..96,
// 129..192 and 257..288 tokens: a quarter less of copies, MMAs and epilogue; 77
// tokens, 4 layers at 8B width 538 -> 523 us), smaller for short ones; at group 32
// (four accumulators per step) at most 64.
int gemm_tc_tile(int S, int group) {
  if (S <= 64 || group == 32) return S > 32 ? 64 : 32;
  return (S + 95) / 96 == (S + 127) / 128 ? 96 : 128;
}

void gemm_tc_rings(int tile, int group, int (&r)[6]) {
  r[0] = kUStages;
  r[1] = kBStages;
  r[2] = kAStages;
  r[3] = tc_accumulators(tile, kUnitK / group);
  r[4] = kMmaWarps;
  r[5] = kDqSets;
}

// Parts of K for a projection of n_rb row-blocks and upr units on `sms` SMs:
// the split whose last CTA finishes first, counting whole rounds of CTAs and,
// per CTA, about 6 steps' worth of filling the pipeline and writing the tile
// (o projection of 8B, 77 tokens: 32 CTAs of 32 steps -> 128 of 8).
int gemm_tc_parts(int n_rb, int upr, int S, int group, int sms) {
  const int N = gemm_tc_tile(S, group);
  const long long tiles = (long long)((n_rb + 1) / 2) * ((S + N - 1) / N);
  int best = 1;
  long long cost = 0;
  for (int ks = 1; ks <= kGemmMaxParts && 4 * ks <= upr; ++ks) {
    const long long c = (tiles * ks + sms - 1) / sms * ((upr + ks - 1) / ks + 6);
    if (ks == 1 || c < cost) best = ks, cost = c;
  }
  return best;
}

cudaError_t launch_gemm_tc(const GemmArgs& a, int group, cudaStream_t s) {
  const int N = gemm_tc_tile(a.S, group);
  if (N == 32) {
    if (group == 128) return launch_tc<32, 1>(a, s);
    if (group == 64) return launch_tc<32, 2>(a, s);
    if (group == 32) return launch_tc<32, 4>(a, s);
  } else if (N == 64) {
    if (group == 128) return launch_tc<64, 1>(a, s);
    if (group == 64) return launch_tc<64, 2>(a, s);
    if (group == 32) return launch_tc<64, 4>(a, s);
  } else if (N == 96) {
    if (group == 128) return launch_tc<96, 1>(a, s);
    if (group == 64) return launch_tc<96, 2>(a, s);
  } else if (N == 128) {
    if (group == 128) return launch_tc<128, 1>(a, s);
    if (group == 64) return launch_tc<128, 2>(a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace shard
